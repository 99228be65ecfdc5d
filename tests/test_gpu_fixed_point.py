"""The fixed-point kernels of the FP64 iterations, the generator and the derivative at
the sizes and values where a rule sends them another way, against the oracle or the
FP64 stage kernels.  Tolerances: 1e-13 on links and G after a few steps (the parity
tests' bound), a few roundings where two FP64 computations of one quantity are compared."""
import ctypes

import numpy as np
import pytest

from oracle import oracle as orc
from paper_1301_3460_gb300 import inputs
from paper_1301_3460_gb300 import lgf

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def dag(m):
    return np.conj(np.swapaxes(m, -1, -2))


# a thread per link up to 32768 sites, a thread per site above; blocks of 32 and 128
# sites that do not divide the volume; tiles that take 512 threads; split lines
@pytest.mark.parametrize("L", [(6, 6, 6, 6), (16, 16, 16, 8), (16, 12, 16, 12), (6, 6, 6, 48), (48, 64, 4, 4), (4, 4, 96, 64)])
@pytest.mark.parametrize("track", [True, False])
def test_steps_match_oracle(L, track):
    U = inputs.rough_gauge_field(L, 0.3, 61)
    ref = orc.fix(L, U, alpha=0.08, tol=0.0, max_iter=3)
    with lgf.Lattice(L, track_gauge=track) as lat:
        lat.set_links(U)
        r = lat.fix(tol=0.0, max_iter=3)
        assert r["iters"] == 3
        assert np.max(np.abs(lat.get_links() - ref["U"])) < 1e-13
        if track:
            assert np.max(np.abs(lat.get_gauge() - ref["G"])) < 1e-13
    assert r["theta"] == pytest.approx(ref["theta"], rel=1e-10)


@pytest.mark.parametrize("alpha", [1e-9, 0.08, 3.0, 300.0])
def test_step_sizes(alpha):
    """From a step that hardly moves a link to one beyond the integer Gram-Schmidt's
    range (alpha/2 Delta~ over 16, built in FP64): one step against the oracle."""
    L = (8, 6, 4, 8)
    U = inputs.rough_gauge_field(L, 0.4, 62)
    ref = orc.fix(L, U, alpha=alpha, tol=0.0, max_iter=1)
    with lgf.Lattice(L) as lat:
        lat.set_links(U)
        lat.fix(alpha=alpha, tol=0.0, max_iter=1)
        # X = 1 + alpha/2 Delta~ has condition number up to |X|: rounding errors of the
        # transforms, 1e-15 of Delta~, turn g by as much
        assert np.max(np.abs(lat.get_links() - ref["U"])) < 1e-13
        assert np.max(np.abs(lat.get_gauge() - ref["G"])) < 1e-13


def test_links_out_of_range_take_the_fp64_kernels():
    """A snapshot is stored unchecked; links that are not unitary are iterated by the FP64
    kernels: the same step as the stages, one by one."""
    L = (8, 4, 6, 4)
    V = int(np.prod(L))
    U = inputs.rough_gauge_field(L, 0.4, 63)
    with lgf.Lattice(L) as lat:
        lat.set_links(U)
        snap = lat.save_links()
        for scale in (1.0, 1.5):
            lat.load_links((snap.view(torch.float64) * scale).view(torch.uint8))
            W = lat.get_links()
            assert np.max(np.abs(W[..., :2, :] - scale * U[..., :2, :])) < 1e-15
            D, th, F = lat.delta()
            g = lat.build_g(lat.accelerate(D), 0.08)
            want = np.empty_like(W)
            for mu in range(4):
                want[mu] = g @ W[mu] @ dag(g[inputs.neighbour(L, mu)])
            r = lat.fix(tol=0.0, max_iter=0)
            assert r["theta"] == pytest.approx(th, rel=1e-13) and r["F"] == pytest.approx(F, rel=1e-13)
            lat.fix(tol=0.0, max_iter=1)
            assert np.max(np.abs(lat.get_links()[..., :2, :] - want[..., :2, :])) < 1e-13
        bad = snap.view(torch.float64).clone()
        bad[7] = float("nan")
        lat.load_links(bad.view(torch.uint8))
        assert lat.fix(check=False)["status"] == lgf.LGF_ERR_NAN
        lat.set_links(U)
        assert lat.fix(max_iter=2000)["converged"]
    assert V == U.shape[1]


def test_link_check_threshold_and_alignment():
    """Links are accepted up to 1e-12 of SU(3), whatever the array's alignment."""
    L = (4, 6, 4, 4)
    U = inputs.rough_gauge_field(L, 0.3, 64)
    lib = lgf.load()
    with lgf.Lattice(L) as lat:
        def status(W, shift):
            # a device copy that starts on a 16-byte boundary, or 8 bytes after one
            flat = torch.empty(W.size * 2 + 2, dtype=torch.float64, device="cuda")
            flat[shift:shift + W.size * 2] = torch.from_numpy(np.ascontiguousarray(W).view(np.float64).reshape(-1))
            torch.cuda.synchronize()
            return lib.lgf_set_links(lat._h, ctypes.c_void_p(flat.data_ptr() + 8 * shift), 1)

        for shift in (0, 1):
            assert status(U, shift) == lgf.LGF_OK
            got = lat.get_links()
            assert np.array_equal(got[..., :2, :], U[..., :2, :])
            for err, ok in ((0.4e-12, True), (0.7e-12, False), (1e-3, False), (1.0, False), (1e200, False)):
                W = U.copy()
                W[1, 3, 2] *= 1 + err  # the row's norm squared is off by 2 err
                assert (status(W, shift) == lgf.LGF_OK) == ok, (shift, err)
            for v in (np.nan, np.inf):
                W = U.copy()
                W[3, 100, 2, 1] = v
                assert status(W, shift) == lgf.LGF_ERR_NOT_SU3
            W = U.copy()
            W[2, 5] = W[2, 5][[1, 0, 2]]  # unitary with determinant -1
            assert status(W, shift) == lgf.LGF_ERR_NOT_SU3


def test_derivative_scales_exactly():
    """The backward step is linear in the cotangent: a power of two goes through exactly,
    zeros give zeros, and what is not finite gives NaN."""
    L = (6, 8, 4, 4)
    V = int(np.prod(L))
    U = torch.from_numpy(inputs.rough_gauge_field(L, 0.3, 65)).cuda()
    gen = torch.Generator(device="cuda").manual_seed(3)
    ct = torch.randn((4, V, 3, 3), dtype=torch.complex128, device="cuda", generator=gen)
    with lgf.Lattice(L, track_gauge=False) as lat:
        lat.set_links(U)
        one = lat.step_bwd(ct)
        for k in (-300, 5, 300):
            assert torch.equal(lat.step_bwd(ct * 2.0 ** k), one * 2.0 ** k)
        assert float(lat.step_bwd(ct * 0).abs().max()) == 0.0
        ct[2, 9, 1, 1] = float("inf")
        out = torch.view_as_real(lat.step_bwd(ct))
        assert bool(torch.isnan(out[..., :2, :, :]).all())


@pytest.mark.parametrize("alpha", [0.08, 40.0])
def test_fp32_g_builder_is_the_rounded_fp64_result(alpha):
    """The FP32 phase's g against the FP64 stage on the same field: rows 0,1 to FP32
    rounding of the transforms (the bound of the FP32 stage tests)."""
    L = (8, 8, 6, 4)
    Do, _, _ = orc.delta(L, inputs.rough_gauge_field(L, 0.4, 66))
    Dt = orc.accelerate(L, Do)
    with lgf.Lattice(L, mixed=True) as lat:
        g32, g64 = lat.build_g(Dt, alpha, precision=32), lat.build_g(Dt, alpha)
    assert np.max(np.abs(g32 - g64)) < 5e-6 * max(1.0, 0.5 * alpha * np.max(np.abs(Dt)))
    assert np.max(np.abs(g32 @ dag(g32) - np.eye(3))) < 2e-6
