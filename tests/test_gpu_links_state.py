"""What decides between the fixed-point and the FP64 kernels, and that neither answers for
links that are not its own: snapshots with a row 2 of their own, links that stopped being
finite, plain descent under the instrumentation, links that the generator has rewritten."""
import numpy as np
import pytest

from paper_1301_3460_gb300 import inputs, lgf

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def dag(m):
    return np.conj(np.swapaxes(m, -1, -2))


def one_step(lat, L, alpha=0.08):
    """rows 0,1 of the links after a step made of the FP64 stages"""
    W = lat.get_links()
    D, _, _ = lat.delta()
    g = lat.build_g(lat.accelerate(D), alpha)
    return np.stack([g @ W[mu] @ dag(g[inputs.neighbour(L, mu)]) for mu in range(4)])[..., :2, :]


def test_snapshot_of_18_reals_keeps_its_row_2():
    """Row 2 of an 18-real snapshot is read as it stands, also where rows 0,1 are SU(3)'s
    and it is not their product.  1e-13: the parity tests' bound after a step."""
    L = (8, 4, 6, 4)
    V = int(np.prod(L))
    U = inputs.rough_gauge_field(L, 0.4, 71)
    with lgf.Lattice(L, links18=True) as lat:
        lat.set_links(U)
        snap = lat.save_links()
        lat.fix(tol=0.0, max_iter=3)
        want = lat.get_links()
        lat.load_links(snap)  # a row 2 that is the product: the same kernels as after set_links
        lat.fix(tol=0.0, max_iter=3)
        assert np.array_equal(lat.get_links(), want)
        for err in (1e-6, 1e-12):
            odd = snap.clone().view(torch.float64).reshape(4, 9, V, 2)
            odd[:, 6:] *= 1 + err
            lat.load_links(odd.reshape(-1).view(torch.uint8))
            assert np.max(np.abs(lat.get_links()[..., 2, :] - U[..., 2, :])) > err / 4
            want2 = one_step(lat, L)
            lat.fix(tol=0.0, max_iter=1)
            assert np.max(np.abs(lat.get_links()[..., :2, :] - want2)) < 1e-13


def test_links_lost_under_the_instrumentation_stay_lost():
    """Kernels timed with a step that is not finite leave NaN links; a later fix says so."""
    L = (4, 6, 4, 4)
    U = inputs.rough_gauge_field(L, 0.3, 72)
    with lgf.Lattice(L) as lat:
        lat.set_links(U)
        lat.time_kernels(alpha=float("inf"), n_iter=1)
        assert np.isnan(lat.get_links()).any()
        assert lat.fix(check=False)["status"] == lgf.LGF_ERR_NAN
        lat.set_links(U)
        assert lat.fix(max_iter=2000)["converged"]


def test_kernels_timed_in_a_plain_context_are_the_accelerated_iteration():
    """Instrumentation of a context without Fourier acceleration runs the four kernels it
    names: the links move by an accelerated step."""
    L = (6, 8, 4, 6)
    U = inputs.rough_gauge_field(L, 0.3, 73)
    with lgf.Lattice(L) as lat:
        lat.set_links(U)
        lat.fix(tol=0.0, max_iter=2)
        want = lat.get_links()
    with lgf.Lattice(L, accelerate=False) as lat:
        lat.set_links(U)
        lat.time_kernels(n_iter=2)
        assert np.max(np.abs(lat.get_links() - want)) < 1e-13


@pytest.mark.parametrize("bits", [64, 32])
def test_rewritten_links_take_the_fixed_point_kernels(bits):
    """Sweeps rewrite every link into SU(3), so what follows them runs as after set_links,
    bit for bit, also when the chain started from a snapshot of other matrices."""
    L = (4, 6, 4, 8)
    U = inputs.rough_gauge_field(L, 0.4, 74)
    with lgf.Lattice(L) as lat, lgf.Lattice(L) as ref:
        lat.set_generator_precision(bits)
        lat.set_links(U)
        lat.load_links((lat.save_links().view(torch.float64) * 1.5).view(torch.uint8))
        lat.wilson_sweeps(6.0, 5, n_heatbath=1, n_overrelax=1)
        ref.set_links(lat.get_links())
        lat.fix(tol=0.0, max_iter=3)
        ref.fix(tol=0.0, max_iter=3)
        assert np.array_equal(lat.get_links(), ref.get_links())
        # a chain that begins with links out of range is the FP64 generator's
        lat.set_links(U)
        lat.load_links((lat.save_links().view(torch.float64) * 1.5).view(torch.uint8))
        lat.wilson_sweeps(6.0, 5, n_heatbath=0, n_overrelax=0)
        assert np.max(np.abs(lat.get_links()[..., :2, :] - 1.5 * U[..., :2, :])) < 1e-14
