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


# the one-launch sort up to 4,096 particles and cells; 8 lanes a particle up to
# 20,000, 4 up to 50,000, else 2; one, two and more cells along an axis; more
# pairs than a lane notes (rho = 24)
@pytest.mark.parametrize("n,box,s", [(1, (3.0, 4.0, 5.0), 1.0), (40, (2.1, 2.1, 2.1), 1.0), (98, (2.05, 3.1, 6.0), 0.5),
                                     (700, (4.5, 4.5, 4.5), 0.25), (3000, (5.0, 5.0, 5.0), 1.0),
                                     (4096, (11.0, 12.0, 10.0), 1.0), (4097, (11.0, 12.0, 10.0), 2.0),
                                     (1000, (17.0, 16.0, 16.0), 1.0), (20000, (20.0, 18.0, 19.0), 0.5),
                                     (20001, (20.0, 18.0, 19.0), 1.0), (50001, (26.0, 25.0, 25.5), 1.0),
                                     (131072, (35.2, 36.0, 34.3), 0.5), (60000, (40.0, 41.0, 39.9), 1.0)])
def test_static_forces_each_side_of_the_size_rules(n, box, s):
    need_gpu()
    import torch
    x, v = workloads.uniform_fluid(box, n, 1.0, n + 1)[:2]
    x32 = np.minimum(x.astype(np.float32), np.nextafter(np.asarray(box, np.float32), np.float32(0.0)))
    v32 = v.astype(np.float32)
    sp = np.random.default_rng(n).integers(0, 2, n).astype(np.int32)
    a = [[25.0, 40.0], [40.0, 30.0]]
    prm = dpd.dpd_static_params_from(box, a, 4.5, 1.0, 1.0, s, 0.01, seed=9, body_mode=2, body=(0.3, 0.0, -0.1))
    pos, vel = torch.zeros((n, 4)), torch.zeros((n, 4))
    pos[:, :3], vel[:, :3] = torch.from_numpy(x32), torch.from_numpy(v32)
    pos[:, 3] = torch.from_numpy(sp.view(np.float32))
    pos, vel, out = pos.cuda(), vel.cuda(), torch.full((n, 4), float("nan"), device="cuda")
    got = []
    for _ in range(2):
        dpd.dpd_forces_static(prm, n, pos.data_ptr(), vel.data_ptr(), None, 4, out.data_ptr(),
                              torch.cuda.current_stream().cuda_stream)
        got.append(out.cpu().numpy().copy())
    assert np.array_equal(got[0], got[1])  # fixed order: the same bits
    o = oracle.System(box, a, 4.5, 1.0, 1.0, s, 0.01, seed=9, body_mode=2, body=(0.3, 0.0, -0.1), cut_fp32=True)
    f, _ = o.forces(x32.astype(np.float64), v32.astype(np.float64), species=sp, step=4)
    assert force_error(got[0][:, :3].astype(np.float64), f)[0] < FORCE_TOL


# a table per warp up to 512 bins, fewer warps up to 4,096, each bin its own
# scan above; FP64 sums of FP32 values: 1e-12 of the largest sum is far above
# their rounding (n 2^-53)
@pytest.mark.parametrize("n,nbins", [(1, 1), (500, 3), (3000, 60), (30000, 512), (30000, 513), (9000, 4096), (9000, 4097)])
def test_profile_each_side_of_the_size_rules(n, nbins):
    need_gpu()
    c = workloads.CONFIGS["fluid_small"]
    box = (10.0, 11.0, 12.0)
    x, v = workloads.uniform_fluid(box, n, 1.0, n)[:2]
    g = dpd.Sim(box, c["a"], c["gamma"], c["kT"], c["rc"], c["s"], c["dt"])
    g.set_state(x, v)
    x32, v32, _ = g.state()
    for axis, comp in ((1, 0), (2, 2)):
        b = (x32[:, axis].astype(np.float32) * (np.float32(nbins) / np.float32(box[axis]))).astype(np.int64)
        b = np.clip(b, 0, nbins - 1)
        start = np.arange(nbins, dtype=np.float64)
        sums, counts = g.profile(axis, comp, nbins, start.copy(), start.copy())
        ref = np.bincount(b, weights=v32[:, comp], minlength=nbins)
        assert np.array_equal(counts - start, np.bincount(b, minlength=nbins))
        assert np.abs(sums - start - ref).max() < 1e-12 * max(np.abs(ref).max(), nbins, 1.0)
    g.close()


# more pairs than a lane notes (rho = 22); rows of the stencil that cross the
# boundary on both sides (three cells an axis); one particle; a box of few units
@pytest.mark.parametrize("n,L,lam,shape", [(2000, 4.5, 0.5, (128, 1)), (2000, 4.5, 0.65, (512, 2)), (90, 3.01, 0.5, (256, 8)),
                                           (1, 3.5, 0.5, (256, 2)), (17, 3.5, 0.5, (128, 4)), (3000, 10.0, 0.5, (512, 2))])
def test_ensemble_forces_of_sparse_and_dense_boxes(n, L, lam, shape):
    need_gpu()
    c = workloads.CONFIGS["fluid_small"]
    box = (L, L + 0.3, L + 0.1)
    x, v = workloads.uniform_fluid(box, n, 1.0, n)[:2]
    sp = np.random.default_rng(n).integers(0, 2, n).astype(np.int32)
    a = [[25.0, 40.0], [40.0, 30.0]]
    e = dpd.Ensemble(threads=shape[0], cluster=shape[1])
    i = e.add(box, a, c["gamma"], c["kT"], c["rc"], 0.5, c["dt"], x, v, species=sp, step=2, lam=lam, seed=7)
    x32, v32, _ = e.state(i)
    o = oracle.System(box, a, c["gamma"], c["kT"], c["rc"], 0.5, c["dt"], lam=lam, seed=7, cut_fp32=True)
    f, vir = o.forces(x32, v32, species=sp, step=2)
    got = e.forces(i)
    if n > 1:
        assert force_error(got, f)[0] < FORCE_TOL
        assert abs(e.observables(i)["virial"] - vir) < 1e-5 * abs(vir)
    else:
        assert np.array_equal(got, np.zeros((1, 3)))
    e.step(3)
    e.sync()
    assert np.isfinite(e.state(i)[0]).all()
    e.close()


def test_ensemble_runs_a_sparse_box_at_the_limit():
    """A box of few particles and many cells, the largest that is accepted,
    has a launch shape."""
    need_gpu()
    n, fits = 60, 0.0
    L = 25.0
    while dpd.dpd_ensemble_fits((L, 30.0, 30.0), [[25.0]], 4.5, 1.0, 1.0, 1.0, 0.01, n):
        fits, L = L, L + 1.01
    assert fits > 0.0
    box = (fits, 30.0, 30.0)
    x, v = workloads.uniform_fluid(box, n, 1.0, 3)[:2]
    e = dpd.Ensemble()
    i = e.add(box, [[25.0]], 4.5, 1.0, 1.0, 1.0, 0.01, x, v)
    e.step(2)
    e.sync()
    assert e.state(i)[2] == 2
    e.close()
