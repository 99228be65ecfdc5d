"""Launch shapes that the autotuner keeps for the process: each for the kernels it was timed
on.  A context whose FP64 iterations run other kernels (FP32 accelerator, links out of the
fixed-point range, plain descent) must not take a later context of the same extents, or
itself after a switch back, off the integer transforms.  The FP64 transforms' TMA form wins by
a hair and not on every run, so several extents are tried where it has been seen to."""
import numpy as np
import pytest

from paper_1301_3460_gb300 import inputs, lgf

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def on_integers(lat, L, U):
    """whether three steps are, bit for bit, those of the integer transforms at the context's
    launch shape (the pencils' width enters their roundings; FP64 transforms differ in the
    last bits)"""
    def steps(x):
        x.set_links(U)
        x.fix(tol=0.0, max_iter=3)
        return x.get_links()

    sh = lat.get_shape(64)
    with lgf.Lattice(L) as ref:
        ref.set_shape(64, nt_xy=sh["nt_xy"], nt_zt=sh["nt_zt"], xw=sh["xw"], zt_form=0)
        return np.array_equal(steps(lat), steps(ref))


EXTENTS = [(32, 32, 8, 8), (12, 12, 12, 12), (32, 32, 12, 12), (24, 24, 8, 8), (24, 24, 12, 12), (16, 16, 12, 12),
           (32, 24, 8, 8), (48, 16, 8, 8), (32, 32, 8, 12), (12, 12, 8, 8)]


@pytest.mark.parametrize("L", EXTENTS)
@pytest.mark.parametrize("other", ["accel32", "wide", "plain"])
def test_other_kernels_leave_the_integer_transforms_alone(L, other):
    U = inputs.rough_gauge_field(L, 0.3, 91)
    with lgf.Lattice(L, mixed=other == "accel32", accelerate=other != "plain") as lat:
        lat.set_links(U)
        if other == "accel32":
            lat.set_accel_precision(32)
        if other == "wide":
            lat.load_links((lat.save_links().view(torch.float64) * 1.5).view(torch.uint8))
        lat.autotune()
        if other == "accel32":
            assert lat.get_shape(64)["zt_form"] == 0
            lat.set_accel_precision(64)
            assert lat.get_shape(64)["zt_form"] == 0
        if other == "wide":
            assert on_integers(lat, L, U)
    with lgf.Lattice(L) as lat:
        lat.set_links(U)
        lat.autotune()
        assert lat.get_shape(64)["zt_form"] == 0
        assert on_integers(lat, L, U)
        # asked for, the TMA form is taken; tuning returns to the integers
        lat.set_shape(64, nt_xy=128, nt_zt=64, xw=2, zt_form=1)
        assert not on_integers(lat, L, U)
        lat.autotune()
        assert lat.get_shape(64)["zt_form"] == 0
        assert on_integers(lat, L, U)
