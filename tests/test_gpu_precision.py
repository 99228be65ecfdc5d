"""Precision that the fixed-point kernels keep where values of different size meet."""
import numpy as np
import pytest

from paper_1301_3460_gb300 import inputs, lgf

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_generated_links_are_rounded_to_the_nearest_double():
    """A generated link is an SU(3) matrix rounded to doubles.  Per row the rounding errors are
    half a unit of each entry's own last place: <row 0, row 1> of rough links is below 4.4e-17 rms
    (6.4e-17 with every entry on the grid 2^-53), and an entry of 2^-8 to 2^-4 lies on a
    multiple of 2^-53 with a chance of 1/8 at most."""
    L = (8, 8, 8, 8)
    with lgf.Lattice(L, track_gauge=False) as lat:
        lat.set_links(inputs.rough_gauge_field(L, 0.4, 81))
        lat.wilson_sweeps(6.0, 3, n_heatbath=1, n_overrelax=1)
        U = lat.get_links()
    r = U[..., :2, :]
    x = np.stack((r.real, r.imag)).ravel()
    x = x[(np.abs(x) > 2.0 ** -8) & (np.abs(x) < 2.0 ** -4)]
    assert x.size > 1000
    assert np.mean(x * 2.0 ** 53 % 1 == 0) < 0.15
    w = r.astype(np.clongdouble)
    ip = (w[..., 0, :].conj() * w[..., 1, :]).sum(-1)
    assert float(np.sqrt(np.mean(np.abs(ip) ** 2))) < 5e-17
    norm = (np.abs(w) ** 2).sum(-1) - 1
    assert float(np.sqrt(np.mean(norm ** 2))) < 1e-16


def _unit_with_cotangent(lat, V, big, small):
    """step_bwd at unit links (g = 1, so that colour components do not mix there): component
    01 of size big on even sites, 02 of size small on odd ones"""
    gen = torch.Generator(device="cuda").manual_seed(7)
    r = torch.randn((4, V, 2), dtype=torch.complex128, device="cuda", generator=gen)
    ct = torch.zeros((4, V, 3, 3), dtype=torch.complex128, device="cuda")
    ct[:, ::2, 0, 1] = big * r[:, ::2, 0]
    ct[:, 1::2, 0, 2] = small * r[:, 1::2, 1]
    lat.set_unit_links()
    return lat.step_bwd(ct)


@pytest.mark.parametrize("L", [(8, 8, 8, 8), (12, 6, 4, 48)])
def test_fields_of_different_size_keep_their_own_precision(L):
    """The backward step is linear and at unit links colour components stay apart, so a
    component gets what it gets alone, to its own rounding, however large another is: a few
    units of 2^-52 of its largest value, 64 covers the transforms' lengths."""
    V = int(np.prod(L))
    with lgf.Lattice(L, track_gauge=False) as lat:
        alone = _unit_with_cotangent(lat, V, 0.0, 1e-6)[..., 0, 2]
        both = _unit_with_cotangent(lat, V, 1.0, 1e-6)
        assert float(both[..., 0, 1].abs().max()) > 0.1
        assert float((both[..., 0, 2] - alone).abs().max()) < 64 * 2.0 ** -52 * float(alone.abs().max())


def test_subnormal_cotangents_count():
    """Cotangents in the subnormal range go through like others: with 2^-1074 as their last
    place and values near 2^-1040 each is known to 2^-35, and the step's sums multiply that by
    no more than a few hundred."""
    L = (6, 8, 4, 4)
    V = int(np.prod(L))
    gen = torch.Generator(device="cuda").manual_seed(8)
    ct = torch.randn((4, V, 3, 3), dtype=torch.complex128, device="cuda", generator=gen)
    with lgf.Lattice(L, track_gauge=False) as lat:
        lat.set_links(inputs.rough_gauge_field(L, 0.3, 82))
        one = lat.step_bwd(ct)
        tiny = lat.step_bwd(torch.view_as_complex(torch.view_as_real(ct) * 2.0 ** -1040))
        back = torch.view_as_complex(torch.view_as_real(tiny) * 2.0 ** 1000 * 2.0 ** 40)
    assert float((back - one).abs().max()) < 2.0 ** -26 * float(one.abs().max())
