"""The kernels' choices by size: group lists of 4, 8, 16 and 32 particles,
builder blocks per brick, the one-block sort -- each side of every line the
dispatch draws, against the oracle."""
import numpy as np
import pytest

import oracle
import paper_1311_0402_gb300 as dpd
import workloads
from gpu_util import force_error, need_gpu

pytestmark = pytest.mark.gpu

FORCE_TOL = 1e-4  # relative to the RMS force, max over particles/components


def _box_of(n, rho=3.0, aspect=(1.0, 1.0, 1.0)):
    k = (n / rho / np.prod(aspect)) ** (1.0 / 3.0)
    return tuple(float(k * a) for a in aspect)


# groups: 4 below 80,000 particles, 8 below 160,000, 16 below 320,000, else 32;
# the one-block sort up to 8,192 particles
@pytest.mark.parametrize("n,det,lam", [(200, 0, 0.5), (8192, 0, 0.65), (8193, 0, 0.5), (79999, 0, 0.5), (80000, 0, 0.5),
                                       (160001, 1, 0.5), (320000, 0, 0.5), (319999, 1, 0.65)])
def test_forces_and_step_each_side_of_the_size_rules(n, det, lam):
    need_gpu()
    c = workloads.CONFIGS["fluid_small"]
    box = _box_of(n, aspect=(1.0, 1.3, 0.8))
    x, v = workloads.uniform_fluid(box, n, 1.0, n)[:2]
    g = dpd.Sim(box, c["a"], c["gamma"], c["kT"], c["rc"], c["s"], c["dt"], lam=lam, deterministic=det)
    o = oracle.System(box, c["a"], c["gamma"], c["kT"], c["rc"], c["s"], c["dt"], lam=lam, cut_fp32=True)
    g.set_state(x, v, step=3)
    x32, v32, _ = g.state()
    f, _ = o.forces(x32, v32, step=3)
    assert force_error(g.forces(), f)[0] < FORCE_TOL
    if n <= 8193:
        assert np.array_equal(g.neighbors(), oracle.pairs_fp32(x32, box, 1.3))
    # the forces after a run that rebuilds several times, at the state it reached
    g.step(13)
    assert g.info()["rebuilds"] > 1
    g.build_neighbors()
    x1, v1, step = g.state()
    f1, _ = o.forces(x1, v1, step=step)
    assert force_error(g.forces(), f1)[0] < FORCE_TOL
    g.close()


def test_fixed_capacity_keeps_the_shared_capacity_of_32():
    """A capacity the caller sets is shared by groups of 32 particles: a box
    whose lists fit that way is still accepted when smaller groups would let
    one dense spot overflow."""
    need_gpu()
    c = workloads.CONFIGS["fluid_small"]
    box = (12.0, 12.0, 12.0)
    x, v = workloads.uniform_fluid(box, 3000, 1.0, 8)[:2]
    x[:12] = np.array([6.0, 6.0, 6.0]) + 0.05 * x[:12] / 12.0  # 12 particles in one spot
    def forces(cap):
        g = dpd.Sim(box, c["a"], c["gamma"], c["kT"], c["rc"], c["s"], c["dt"], nbr_capacity=cap)
        g.set_state(x, v, step=1)
        out = g.forces()
        g.close()
        return out
    a, b = forces(0), forces(24)
    assert force_error(a, b)[0] < FORCE_TOL
