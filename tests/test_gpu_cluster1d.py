"""The one-cluster advance of small 1D meshes against the three launches per
step (bitwise states, dt and time; totals to rounding), at the sizes where the
split over CTAs changes: one cell range, one CTA, a last CTA of one cell, two
warps a CTA, the largest mesh; every boundary rule, a force, and runs that reach
their end time inside a call."""
import numpy as np
import pytest

from paper_1207_3392_gb300 import hydro as H
from paper_1207_3392_gb300 import problems as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1207_3392_gb300 import build
    build.build()
    yield


def _run(pr, precision, one, calls, t_end=0.0):
    h = H.Hydro.from_problem(pr, precision=precision)
    h.set_one_launch(one)
    t = [h.advance(k, pr.cfl, t_end) for k in calls]
    h.step(h.compute_dt(0.1))
    out = h.get_conserved(), t, h.time, h.step_totals(), h.compute_dt(pr.cfl)
    h.close()
    return out


@pytest.mark.parametrize("precision", [H.FP64, H.FP32_MIXED])
@pytest.mark.parametrize("n", [2, 3, 8, 9, 16, 17, 129, 256, 481, 1024, 4088])
def test_cluster_advance_equals_three_launches(n, precision):
    for bc in (P.PERIODIC, P.REFLECT, P.OUTFLOW):
        pr = P.random_blocks(1, (n,), seed=n, bc=bc).with_(solver=H.HLL if n % 2 else H.HLLC)
        if n % 3 == 0:
            pr = pr.with_(grad_phi=(0.3, 0.0, 0.0))
        for calls, t_end in (((1, 2, 5), 0.0), ((7, 6), 4.5 * _first_dt(pr, precision))):
            a, b = (_run(pr, precision, one, calls, t_end) for one in (True, False))
            np.testing.assert_array_equal(a[0], b[0], err_msg=f"n={n} bc={bc}")
            assert a[1] == b[1] and a[2] == b[2] and a[4] == b[4]
            np.testing.assert_allclose(a[3], b[3], rtol=1e-12, atol=1e-12 * np.max(np.abs(b[3])))


def _first_dt(pr, precision):
    h = H.Hydro.from_problem(pr, precision=precision)
    dt = h.compute_dt(pr.cfl)
    h.close()
    return dt


@pytest.mark.parametrize("precision", [H.FP64, H.FP32_MIXED])
def test_cluster_advance_reports_a_bad_state(precision):
    pr = P.sod(100)
    pr.p[40] = -1.0
    h = H.Hydro.from_problem(pr, precision=precision)
    with pytest.raises(H.NonPhysicalState):
        h.advance(3, pr.cfl)
    h.close()
