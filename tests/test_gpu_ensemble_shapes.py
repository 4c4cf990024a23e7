"""Launch shapes of the ensemble, and reading states beside other work."""
import numpy as np
import pytest

import oracle
import paper_1311_0402_gb300 as dpd
import workloads
from gpu_util import force_error, need_gpu

pytestmark = pytest.mark.gpu


def _add(e, L, n, seed):
    x, v = workloads.uniform_fluid((L, L, L), n, 1.0, seed)[:2]
    return e.add((L, L, L), [[25.0]], 4.5, 1.0, 1.0, 1.0, 0.01, x, v, seed=seed)


def test_a_class_without_boxes_at_tuning_keeps_the_rule():
    """The tuner decides for the size classes it timed; boxes of another class
    that come later run as in an ensemble that was never tuned."""
    need_gpu()
    e, fresh = dpd.Ensemble(), dpd.Ensemble()
    _add(e, 5.0, 200, 1)
    e.step(1)
    e.sync()
    e.tune(steps=2)
    tuned = e.config()
    k = int(np.flatnonzero(tuned[0])[0])
    _add(e, 10.0, 3000, 2)
    _add(fresh, 10.0, 3000, 2)
    for h in (e, fresh):
        h.step(1)
        h.sync()
    got, want = e.config(), fresh.config()
    other = int(np.flatnonzero(want[0])[0])
    assert other != k
    assert (got[0][k], got[1][k]) == (tuned[0][k], tuned[1][k])
    assert (got[0][other], got[1][other]) == (want[0][other], want[1][other])
    e.close()
    fresh.close()


def test_config_reports_the_shapes_of_the_next_launch():
    need_gpu()
    e = dpd.Ensemble()
    for k in range(3):
        _add(e, 6.0, 600, k)
    _add(e, 10.0, 3000, 9)
    before = e.config()
    e.step(1)
    e.sync()
    assert e.config() == before
    e.close()


def test_reading_a_larger_box_does_not_wait_for_other_work():
    """The block states are read through does not grow while other streams
    run (page-locked memory taken or given back can wait for the device)."""
    need_gpu()
    e = dpd.Ensemble()
    ids = [_add(e, 4.0 + k, 100 * (k + 1), k) for k in range(4)]
    e.step(1)
    e.sync()
    e.state(ids[0])  # (the first launch of a kernel loads it, which waits)
    x, v = workloads.uniform_fluid((40.0, 40.0, 40.0), 192000, 1.0, 3)[:2]
    g = dpd.Sim((40.0, 40.0, 40.0), [[25.0]], 4.5, 1.0, 1.0, 1.0, 0.01)
    g.set_state(x, v)
    g.step(16)
    g.step_async(4000)  # a quarter of a second
    for i in ids:
        assert np.isfinite(e.state(i)[0]).all()
        assert not g.query()
    g.sync()
    g.close()
    e.close()


# more pairs than a lane notes; few particles; a box of 27 cells
@pytest.mark.parametrize("n,L,shape", [(2000, 4.5, (512, 2)), (17, 3.5, (128, 4)), (90, 3.01, (256, 8))])
def test_trajectories_of_sparse_and_dense_boxes(n, L, shape):
    need_gpu()
    box = (L, L + 0.3, L + 0.1)
    x, v = workloads.uniform_fluid(box, n, 1.0, n)[:2]
    a = [[2.0]]
    e = dpd.Ensemble(threads=shape[0], cluster=shape[1])
    i = e.add(box, a, 4.5, 1.0, 1.0, 0.5, 0.001, x, v, step=2, seed=7)
    x32, v32, _ = e.state(i)
    o = oracle.System(box, a, 4.5, 1.0, 1.0, 0.5, 0.001, seed=7, cut_fp32=True)
    f0, _ = o.forces(x32, v32, step=2)
    r = o.run(x32, v32, 3, step=2, f=f0)
    e.step(3)
    e.sync()
    xg, vg, step = e.state(i)
    assert step == r["step"] == 5
    d = xg - r["x"]
    d -= np.asarray(box) * np.round(d / np.asarray(box))
    assert np.abs(d).max() < 1e-5
    assert np.abs(vg - r["v"]).max() < 1e-3
    assert force_error(e.forces(i), r["f"])[0] < 1e-3
    e.close()
