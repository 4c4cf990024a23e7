"""The packed neighbour lists: their capacity when a spot condenses, at load and
during a run, the top level of the cell scan, and what a few steps through them
give at each group size."""
import numpy as np
import pytest

import oracle
import paper_1311_0402_gb300 as dpd
import workloads
from gpu_util import force_error, need_gpu

pytestmark = pytest.mark.gpu

FORCE_TOL = 1e-4  # relative to the RMS force, max over particles/components


# groups of 4, 8 and 16 particles.  Counted with the builder's rules for these
# states: at the end a half list of 4 / 8 / 16 / 32 particles has up to 178 / 332
# / 601 / 958 entries, where 32 x 32 = 1,024 is what 32 particles share at this
# density; at the start, 36 / 61 / 91 / 144.
@pytest.mark.parametrize("n,L", [(1500, 24.0), (60000, 82.0), (200000, 122.0)])
def test_spots_that_condense_during_a_run_fit_the_lists(n, L):
    """24 spots of 45 free particles (no forces) contract to a seventh of their
    size while the handle steps: no list overflows, and every particle is
    where its free flight takes it."""
    need_gpu()
    rng = np.random.default_rng(n)
    spots, m, shrink, dt, steps = 24, 45, 0.14, 0.01, 200
    nc = int(L / (1.3 * (1 + 1e-4)))
    sites = np.stack(np.meshgrid(*[np.arange(2, nc - 2, 4)] * 3, indexing="ij"), -1).reshape(-1, 3)
    centre = (sites[rng.permutation(len(sites))[:spots]] + 0.5) * (L / nc)
    u = rng.normal(size=(spots, m, 3))
    u *= 2.2 * rng.random((spots, m, 1)) ** (1 / 3) / np.linalg.norm(u, axis=2, keepdims=True)
    rest = rng.random((n - spots * m, 3)) * L
    x = np.concatenate([(centre[:, None] + u).reshape(-1, 3), rest])
    v = np.concatenate([((shrink - 1.0) / (steps * dt) * u).reshape(-1, 3), 0.0 * rest])
    g = dpd.Sim((L, L, L), [[0.0]], 0.0, 0.0, 1.0, 1.0, dt)
    g.set_state(x % L, v)
    assert g.info()["nbr_capacity"] == 32
    r0 = g.info()["rebuilds"]
    g.step(steps)
    assert g.info()["rebuilds"] > r0 + 5
    xe, ve, _ = g.state()
    d = xe - (x + steps * dt * v)
    d -= L * np.round(d / L)
    # each step rounds the position and its increment: a unit in the last place of L
    assert np.abs(d).max() < steps * np.spacing(np.float32(L))
    assert np.array_equal(ve, v.astype(np.float32))
    g.close()


@pytest.mark.parametrize("det", [0, 1])
def test_a_spot_too_dense_for_small_groups_at_load(det):
    """A load whose densest spot overflows even 32 particles' share of a list of
    4 goes back to groups of 32 and grows those; the next load is again an
    ordinary one."""
    need_gpu()
    c = workloads.CONFIGS["fluid_small"]
    box = (12.0, 12.0, 12.0)
    x, v = workloads.uniform_fluid(box, 4000, 1.0, 8)[:2]
    dense = x.copy()
    dense[:900] = np.array([6.2, 6.2, 6.2]) + 0.4 * (x[:900] / 12.0 - 0.5)
    g = dpd.Sim(box, c["a"], c["gamma"], c["kT"], c["rc"], c["s"], c["dt"], deterministic=det)
    o = oracle.System(box, c["a"], c["gamma"], c["kT"], c["rc"], c["s"], c["dt"], cut_fp32=True)
    caps = []
    for state in (x, dense, x):
        g.set_state(state, v, step=2)
        x32, v32, _ = g.state()
        f, _ = o.forces(x32, v32, step=2)
        assert force_error(g.forces(), f)[0] < FORCE_TOL
        assert np.array_equal(g.neighbors(), oracle.pairs_fp32(x32, box, 1.3))
        caps.append(g.info()["nbr_capacity"])
    assert caps[0] == caps[2] < caps[1]
    g.close()


def test_a_list_that_cannot_grow_leaves_no_state(monkeypatch):
    """A rebuild whose lists have to grow and get no memory (refused on the host)
    leaves the handle without a state, not with the lists it gave back; the next
    load is an ordinary one."""
    need_gpu()
    box, n = (16.0, 16.0, 16.0), 1000
    x, v = workloads.uniform_fluid(box, n, 0.0, 4)[:2]
    c = np.array([8.3, 8.3, 8.3])
    u = 0.9 * (x[:60] / 16.0 - 0.5) * 4.0
    x[:60], v[:60] = c + u, -0.85 * u  # a spot that contracts within a time unit
    g = dpd.Sim(box, [[0.0]], 0.0, 0.0, 1.0, 1.0, 0.01)
    g.set_state(x, v)
    assert g.info()["nbr_capacity"] == 32
    g.step(100)
    monkeypatch.setenv("DPD_TEST_FAIL_ALLOC", "1")
    with pytest.raises(dpd.DPDError) as e:
        g.build_neighbors()
    assert e.value.status == 2  # DPD_ERR_OOM
    monkeypatch.delenv("DPD_TEST_FAIL_ALLOC")
    with pytest.raises(dpd.DPDError) as e:
        g.step(1)
    assert e.value.status == 7  # DPD_ERR_STATE
    g.set_state(x, v)
    g.step(100)
    g.build_neighbors()
    assert g.info()["nbr_capacity"] > 32
    x32, _, _ = g.state()
    assert np.array_equal(g.neighbors(), oracle.pairs_fp32(x32, box, 1.3))
    g.close()


def test_served_box_is_accepted_by_its_smallest_memory():
    """A budget that holds the box with lists of 32 particles a group is enough,
    and what is counted stays within it."""
    need_gpu()
    box = (10.0, 10.0, 10.0)
    x, v = workloads.uniform_fluid(box, 3000, 1.0, 5)[:2]
    cells = 7.0 ** 3
    need = 3000 * 320.0 + (3000 / 32.0 + cells / 64.0 + 2.0) * 32.0 * 72 * 4.0 + cells * 160.0 + 4.0 * 1024 * 1024
    for budget, ok in ((1.0001 * need, True), (0.9999 * need, False)):
        srv = dpd.Server(max_active=2, mem_budget_bytes=budget)
        if ok:
            t = srv.submit(box, [[25.0]], 4.5, 1.0, 1.0, 1.0, 0.01, x, v, 20)
            assert srv.counts()["mem_bytes"] <= budget
            assert srv.wait(t)["status"] == 0
        else:
            with pytest.raises(dpd.DPDError) as e:
                srv.submit(box, [[25.0]], 4.5, 1.0, 1.0, 1.0, 0.01, x, v, 20)
            assert e.value.status == 2
        srv.close()


def test_a_box_of_more_cells_than_one_level_of_the_scan():
    """Above 1,024 scan tiles (2.1 million cells) the tiles' totals are scanned
    by a kernel of their own: a sparse box of 132^3 cells with a fluid in its last
    corner, at load and after steps that rebuild."""
    need_gpu()
    L, corner, n = 172.0, 15.0, 14000
    rng = np.random.default_rng(5)
    x = rng.random((n, 3)) * L
    m = 3 * int(corner ** 3)
    x[:m] = L - corner * rng.random((m, 3))
    x[m:m + 200, :2] *= 0.01  # and a column along one edge
    v = rng.standard_normal((n, 3))
    box = (L, L, L)
    c = workloads.CONFIGS["fluid_small"]
    g = dpd.Sim(box, c["a"], c["gamma"], c["kT"], c["rc"], c["s"], c["dt"], rebuild_every=2)
    o = oracle.System(box, c["a"], c["gamma"], c["kT"], c["rc"], c["s"], c["dt"], cut_fp32=True)
    g.set_state(x, v, step=1)
    for _ in range(2):
        x32, v32, step = g.state()
        assert np.array_equal(g.neighbors(), oracle.pairs_fp32(x32, box, 1.3))
        f, _ = o.forces(x32, v32, step=step)
        assert force_error(g.forces(), f)[0] < FORCE_TOL
        g.step(5)
        g.build_neighbors()
    g.close()


# groups of 4 below 40,000 particles, 8 below 80,000, 16 below 320,000, else 32; the
# row layout has lists and a pair kernel of its own
@pytest.mark.parametrize("det", [0, 1])
@pytest.mark.parametrize("n", [3000, 39999, 40000, 100000, 200001, 330000])
def test_steps_that_rebuild_agree_with_the_row_layout(n, det):
    """Six steps with a rebuild every second one (before the third and the
    fifth).  The start is a jittered lattice (no near contacts).  A step rounds positions to a unit in the last
    place of L (3.8e-6 up to L = 48), which moves a force by some 240 per unit
    length and partner; a lost pair is a velocity error of 0.1 and more."""
    need_gpu()
    c = workloads.CONFIGS["fluid_small"]
    k = int(np.ceil(n ** (1 / 3)))
    L = (n / 3.0) ** (1 / 3)
    rng = np.random.default_rng(n)
    x = (np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)[rng.permutation(k ** 3)[:n]]
         + 0.5 + 0.2 * (rng.random((n, 3)) - 0.5)) * (L / k)
    v = rng.standard_normal((n, 3))
    out = []
    for kw in (dict(deterministic=det), dict(deterministic=1, list_layout=1)):
        g = dpd.Sim((L, L, L), c["a"], c["gamma"], c["kT"], c["rc"], c["s"], c["dt"], rebuild_every=2, **kw)
        g.set_state(x, v)
        r0 = g.info()["rebuilds"]
        g.step(6)
        assert g.info()["rebuilds"] >= r0 + 2
        out.append(g.state())
        g.close()
    d = out[0][0] - out[1][0]
    d -= L * np.round(d / L)
    assert np.abs(d).max() < 5e-5
    assert np.abs(out[0][1] - out[1][1]).max() < 2e-3
