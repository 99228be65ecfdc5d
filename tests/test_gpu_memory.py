"""Device memory of a context, and what shares it: the fixed-point links of a running loop, of a
sweep and of a derivative lie where idle arrays are, so that a context takes what its FP64
(and FP32) arrays take, and the stored links come back from their place unharmed."""
import numpy as np
import pytest

from paper_1301_3460_gb300 import inputs, lgf

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# bytes per site of the arrays: links, g, Delta, parts, Re Tr, multipliers in FP64, FP32 and
# fixed point; G; the FP32 phase (links twice, parts, Re Tr, G, g); the derivative's workspace
COMMON = 144 + 64 + 256 + 8 + 8 + 4 + 8
G = 96
FP32 = 2 * 192 + 128 + 4 + 48 + 72
DIFF = 16 * (3 * 36 + 6 + 2 * 4)
# allocations are rounded to 2 MiB; tables
SLACK = 40 << 20


def used(make):
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    lat = make()
    torch.cuda.synchronize()
    return lat, free


@pytest.mark.parametrize("form, links", [("fp64", 384), ("nogauge", 384), ("mixed", 384), ("links18", 576)])
def test_bytes_per_site(form, links):
    L = (32, 32, 32, 32)
    V = int(np.prod(L))
    kw = {"fp64": {}, "nogauge": dict(track_gauge=False), "mixed": dict(mixed=True), "links18": dict(links18=True)}[form]
    with lgf.Lattice((4, 4, 4, 4), **kw) as lat:  # code and driver state of the process
        lat.set_unit_links()
        lat.wilson_sweeps(6.0, 1, n_heatbath=1)
        lat.fix(max_iter=2, tol=0.0, check=False)
        lat.step_bwd(torch.zeros((4, 256, 3, 3), dtype=torch.complex128, device="cuda"))
    want = COMMON + links + (0 if form == "nogauge" else G) + (FP32 if form == "mixed" else 0)
    lat, free = used(lambda: lgf.Lattice(L, **kw))
    with lat:
        assert free - torch.cuda.mem_get_info()[0] < want * V + SLACK
        lat.set_unit_links()
        lat.wilson_sweeps(6.0, 1, n_heatbath=1)
        lat.fix(max_iter=2, tol=0.0, check=False)
        assert free - torch.cuda.mem_get_info()[0] < want * V + SLACK
        ct = torch.zeros((4, V, 3, 3), dtype=torch.complex128, device="cuda")
        lat.step_bwd(ct)
        lat.plaquette()
        del ct
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        assert free - torch.cuda.mem_get_info()[0] < (want + DIFF) * V + SLACK


@pytest.mark.parametrize("form", ["fp64", "links18", "links8", "mixed", "nogauge"])
def test_stored_links_survive_what_makes_no_update(form):
    """max_iter = 0, a tolerance above theta, the derivative, the autotuner and the stages leave the
    stored links bit for bit, entries far below the fixed-point grid among them."""
    L = (8, 6, 4, 8)
    V = int(np.prod(L))
    U = inputs.rough_gauge_field(L, 0.3, 95)
    # an SU(2) rotation by 2^-33 in two links: entries of 1e-10 with all their bits
    U[0, 3] = np.eye(3)
    t = 2.0 ** -33 * (1 + 2.0 ** -20 / 3)
    if form != "links8":  # (that form cannot hold links near 1)
        U[0, 3, :2, :2] = [[np.cos(t), np.sin(t)], [-np.sin(t), np.cos(t)]]
    else:
        U[0, 3] = U[0, 4]
    kw = dict(links18=form == "links18", links8=form == "links8", mixed=form == "mixed", track_gauge=form != "nogauge")
    with lgf.Lattice(L, **kw) as lat:
        lat.set_links(U)
        if form == "mixed":
            # the FP32 phase's projection rewrites the links by design; kept here by its own stop
            lat.set_switch_tol(1e300)
        snap = lat.save_links().clone()

        def same():
            return torch.equal(lat.save_links(), snap)

        if form != "mixed":
            lat.fix(max_iter=0, check=False)
            assert same()
            lat.fix(tol=1e6)
            assert same()
        lat.step_bwd(torch.ones((4, V, 3, 3), dtype=torch.complex128, device="cuda"))
        assert same()
        lat.autotune()
        lat.delta()
        assert same()
        lat.set_loop_bound(1)
        r = lat.fix(tol=0.0, max_iter=50, check=False)
        assert r["status"] == lgf.LGF_ERR_TIMEOUT
        lat.set_loop_bound(0)
        W = lat.get_links()
        assert np.max(np.abs(W @ np.conj(np.swapaxes(W, -1, -2)) - np.eye(3))) < (1e-9 if form == "links8" else 1e-13)
        lat.set_links(U)
        assert same()
