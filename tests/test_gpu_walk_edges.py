"""Edges of the walks over flat lists that the ordinary cases do not reach."""
import numpy as np
import pytest

import oracle
from paper_2104_00537_gb300 import cases, sph
from tests.test_gpu_list_eval import check_step_eval

pytestmark = pytest.mark.gpu


def check_boundary(case, g):
    """Boundary values of an evaluated state (fixed walls) against the oracle's
    Eq 38-39 on it, with the tolerances of test_gpu_mdbc."""
    vel = g["vel"].astype(np.float64)
    rho, vel_o, dets = oracle.mdbc(case, g["pos"], vel, g["rho"].astype(np.float64),
                                   with_dets=True)
    b = case.ptype == 1
    ad = np.abs(dets)
    sel = b & (np.abs(ad / 1e-3 - 1.0) >= 1e-3)  # (at the threshold either branch)
    d = np.abs(g["rho"].astype(np.float64) - rho)
    assert d[sel & (ad < 1e-3)].max(initial=0) < 1e-3
    assert d[sel & (ad >= 1e-3) & (ad < 1e-2)].max(initial=0) < 0.1
    assert d[sel & (ad >= 1e-2)].max(initial=0) < 0.01
    vscale = max(np.abs(vel[~b]).max(), 1e-3)
    assert np.abs(g["vel"][sel] - vel_o[sel]).max() < 1e-5 * vscale


def lattice_at_ghosts(cell_mode):
    """An mDBC dam break on the bare lattice, with noise in velocity (0.1 m/s) and
    density (3 kg/m^3): the walls' mirror points fall on fluid particles.  Returns
    it and the number of ghost nodes that lie on one to within 1e-9 dp."""
    c = cases.dam_break(0.02, boundary_mode=1, mdbc_slip=1, cell_mode=cell_mode)
    f = c.ptype == 0
    dp = c.params["dp"]
    c.pos[f] = np.round(c.pos[f] / dp) * dp
    u = cases.uniform01(7, 4 * c.n_fluid).reshape(-1, 4) - 0.5
    c.vel[f] = (0.2 * u[:, :3]).astype(np.float32)
    c.rho[f] += (6.0 * u[:, 3]).astype(np.float32)
    site = lambda x: set(map(tuple, np.round(x / dp).astype(int)))
    b = ~f
    node = c.pos[b] + c.ghost[b]
    on = np.abs(node / dp - np.round(node / dp)).max(1) < 1e-9
    return c, len(site(node[on]) & site(c.pos[f]))


@pytest.mark.parametrize("cell_mode", [0, 1, 2])
@pytest.mark.parametrize("variant", [5, 4, 3])
def test_ghost_node_on_a_fluid_particle(variant, cell_mode):
    """A fluid particle exactly on a ghost node has the largest weight of Eq 38-39
    there: both evaluations of the first step against the oracle, and the nodes'
    lists by brute force."""
    c, hits = lattice_at_ghosts(cell_mode)
    assert hits > 100
    eng = sph.Engine.create(c)
    eng.set_options(pi_variant=variant, check_list=1)
    for stage in (0, 1):
        g = eng.eval_step(stage)
        check_boundary(c, g)
    eng.step(3)
    assert eng.list_info()["check_bad"] == 0
    eng.destroy()


@pytest.mark.parametrize("variant,pair_once", [(5, 0), (4, 0), (3, 0), (5, 1), (4, 1), (0, 0)])
@pytest.mark.parametrize("value", [-np.inf, np.inf, np.nan,
                                   np.uint32(0xffffdead).view(np.float32)])
def test_nonfinite_density_is_reported(variant, pair_once, value):
    """A density that is not finite makes the evaluation fail on every path, also
    the NaN that marks a record of a particle outside the domain."""
    c = cases.dam_break(0.04)
    f = np.nonzero(c.ptype == 0)[0]
    c.rho[f[len(f) // 2]] = value
    eng = sph.Engine.create(c)
    eng.set_options(pi_variant=variant, pair_once=pair_once)
    with pytest.raises(sph.SphError, match="NaN/Inf"):
        eng.eval_step(0)
    eng.destroy()


def walk_blocks(eng):
    """Threads per block of the list walk's launches in one evaluation, from its
    trace (the second session's: a process's first one misses launches, as does one
    in which the list is built, by a conditional graph)."""
    import json
    import os
    import tempfile
    import torch
    from torch.profiler import ProfilerActivity, profile
    for _ in range(2):
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            g = eng.eval_step(0)
            torch.cuda.synchronize()
    with tempfile.TemporaryDirectory() as d:
        path = os.path.join(d, "trace.json")
        prof.export_chrome_trace(path)
        with open(path) as f:
            events = json.load(f)["traceEvents"]
    kernels = [e for e in events if e.get("cat") == "kernel"]
    if not kernels:
        pytest.skip("no kernel trace on this machine")
    return g, {e["args"]["block"][0] for e in kernels if "k_interact_list" in e["name"]}


def test_pi_block_is_the_walk_s_block():
    """pi_block threads per block (0: 256), the same sums bit for bit."""
    eng = sph.Engine.create(cases.dam_break(0.03))
    ref = None
    for block in (0, 128, 256, 512, 1024):
        eng.set_options(pi_block=block)
        g, used = walk_blocks(eng)
        assert used == {block or 256}
        if ref is None:
            ref = g
        for k in ("acc", "drho", "mumax", "dt", "pairs"):
            assert np.array_equal(g[k], ref[k]), (block, k)
    eng.destroy()


def test_wide_records_takes_variant_3_to_4():
    """wide_records 1 changes one thing: pi_variant 3 runs as 4."""
    eng = sph.Engine.create(cases.dam_break(0.03))
    runs = {}
    for variant in (3, 4, 5):
        for wide in (0, 1):
            eng.set_options(pi_variant=variant, wide_records=wide)
            runs[variant, wide] = eng.eval_step(0)["acc"]
    assert np.array_equal(runs[3, 1], runs[4, 0])
    assert not np.array_equal(runs[3, 0], runs[4, 0])  # (sums in another order)
    for v in (4, 5):
        assert np.array_equal(runs[v, 1], runs[v, 0])
    eng.destroy()


def test_empty_case_keeps_its_time():
    """A pool whose only particles belong to a case just released still steps its
    case without particles: no pair bounds dt, so t advances by cfl h / cs0."""
    c = cases.dam_break(0.04)
    e = cases.dam_break(0.04)
    for k in ("pos", "vel", "rho", "ptype", "group", "ghost"):
        setattr(e, k, getattr(e, k)[:0])
    pool = sph.Engine.pool(50000, 400000, 2)
    a = pool.admit(c, t_end=1.0)
    b = pool.admit(e, t_end=1.0)
    pool.pool_step(1)
    t0 = pool.stats(b)["t"]
    assert t0 > 0
    pool.release(a)
    pool.pool_step(3)
    assert pool.stats(b)["t"] == pytest.approx(4 * t0, rel=1e-12)
    pool.destroy()
