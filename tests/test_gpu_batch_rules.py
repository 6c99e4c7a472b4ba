"""Which boxes share their launches in a batch, and with which shapes."""
import numpy as np
import pytest

from paper_2304_05494_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def s2():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2304_05494_gb300 import s2 as mod
    return mod


@pytest.mark.parametrize("mode", ["worklist", "worklist_all"])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("keeps", [(0, -1, 0, -1), (-1, 0, 0, 2)])
def test_split_form_and_keep_boxes_in_one_batch(s2, precision, mode, keeps):
    """Boxes with the split form and boxes with KEEP have other flux kernels
    and other tiles, whichever comes first: each box equals its solo run."""
    cases = [W.taylor_green(48, mach=0.3, seed=20 + i) for i in range(len(keeps))]
    kw = [dict(precision=precision, keep=k, threshold=0.1) for k in keeps]
    want = []
    for c, k in zip(cases, kw):
        c.weno_order = 5
        with s2.Solver.from_case(c, **k) as sv:
            sv.set_state(c.w0)
            sv.step(2)
            want.append(sv.get_state())
    solvers = [s2.Solver.from_case(c, **k) for c, k in zip(cases, kw)]
    for sv, c in zip(solvers, cases):
        sv.set_state(c.w0)
    with s2.Batch(solvers, mode=mode) as b:
        b.step(2)
        b.sync()
    got = [sv.get_state() for sv in solvers]
    for sv in solvers:
        sv.close()
    for k, g, w in zip(keeps, got, want):
        assert np.array_equal(g, w), k


def test_twelve_planes_are_what_is_asked_for(s2):
    """z_planes = 12 is a choice of its own, not the default: a forced channel
    of 12 planes sums its body force in one group with 12, 16 or 24 planes
    per CTA, and in several by default."""
    c = W.channel(40, 36, 12, seed=2)
    out = {}
    for z in (0, 12, 16, 24):
        with s2.Solver.from_case(c, cfl=0.8, threshold=0.05, precision="mixed") as sv:
            assert sv.get_tuning()["z_planes"] == 0 and sv.get_tuning()["weno_ctas_per_sm"] == 0
            sv.set_tuning(z_planes=z)
            sv.set_tuning(flux_ctas_per_sm=2)  # (leaves the others as they are)
            assert sv.get_tuning()["z_planes"] == z
            sv.set_state(c.w0)
            sv.step(3)
            out[z] = sv.get_state()
    assert np.array_equal(out[12], out[16]) and np.array_equal(out[12], out[24])
    assert not np.array_equal(out[12], out[0])


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_branch_mode_runs_the_solo_launches(s2, precision):
    """A member of a branch-mode batch has the launches of its solo step."""
    c = W.taylor_green(24, mach=0.3, seed=5)
    c.weno_order = 5
    with s2.Solver.from_case(c, precision=precision, threshold=0.2, cfl=0.0, dt_fixed=1e-3) as sv:
        sv.set_state(c.w0)
        sv.step(1)
        before = sv.stats()["launches"]
        sv.step(1)
        solo = sv.stats()["launches"] - before
        with s2.Batch([sv], mode="branches") as b:
            assert b.launches_per_step == solo
