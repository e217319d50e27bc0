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


def targets_per_group(n, lanes=8, sms=152):
    """The walk's rule: as many targets (at most the lanes) one after another as
    leave 128 warps per SM."""
    per = 1
    while per < lanes and n * lanes // 32 // (2 * per) >= sms * 128:
        per *= 2
    return per


@pytest.mark.parametrize("dp,per", [(0.0097, 1), (0.0095, 2), (0.0072, 4), (0.0055, 8)])
@pytest.mark.parametrize("pair_once", [0, 1])
def test_several_targets_per_group(dp, per, pair_once):
    """Either side of every size at which a lane group takes more targets: both
    evaluations against the oracle."""
    case = cases.dam_break(dp)
    assert targets_per_group(case.n) == per
    eng = sph.Engine.create(case)
    eng.set_options(use_graph=1, pair_once=pair_once)
    eng.step(2)
    for stage in (0, 1):
        check_step_eval(case, eng, stage, exact_pairs=False)
    eng.destroy()


@pytest.mark.parametrize("kw", [dict(visc_mode=1, nu0=1e-3), dict(ddt_mode=2),
                                dict(boundary_mode=1), dict(integrator=1)])
def test_several_targets_per_group_of_other_physics(kw):
    case = cases.dam_break(0.0085, **kw)
    assert targets_per_group(case.n) > 1
    eng = sph.Engine.create(case)
    eng.step(2)
    for stage in (0,) if "integrator" in kw else (0, 1):
        check_step_eval(case, eng, stage, exact_pairs=False)
    eng.destroy()


@pytest.mark.parametrize("lanes", [0, 4, 2, 1])
def test_groups_across_cases(lanes):
    """Groups whose targets belong to different cases (fluid and boundary ranges
    of 14 uneven cases, few of them a multiple of 32): every case bit for bit as alone,
    where its groups take one target each, with its own pair counts and dt."""
    cs = cases.batch_dam_breaks(14, seed=5, n_min=5000, n_max=60000)
    assert targets_per_group(sum(c.n for c in cs)) == 8
    assert all(targets_per_group(c.n) == 1 for c in cs)
    bat = sph.Engine.batch(cs)
    bat.set_options(use_graph=1, pi_lanes=lanes)
    once = sph.Engine.batch(cs)
    once.set_options(use_graph=1, pair_once=1, pi_lanes=lanes)
    first = [once.eval_step(0, i) for i in range(len(cs))]
    bat.step(4)
    for i, c in enumerate(cs):
        e = sph.Engine.create(c)
        e.set_options(use_graph=1, pi_lanes=lanes)
        g = e.eval_step(0)
        assert first[i]["pairs"] == g["pairs"], i
        assert first[i]["dt"] == pytest.approx(g["dt"], rel=1e-5), i
        scale = np.abs(g["acc"]).max()
        assert np.abs(first[i]["acc"] - g["acc"]).max() < 1e-5 * scale, i
        e.step(4)
        a, b = e.get_state(), bat.get_state(i)
        for k in ("pos", "vel", "rho", "t"):
            assert np.array_equal(a[k], b[k]), (i, k)
        sa, sb = e.stats(), bat.stats(i)
        for k in ("interactions", "interactions_fb", "interactions_bf", "last_dt", "flags"):
            assert sa[k] == sb[k], (i, k)
        e.destroy()
    bat.destroy()
    once.destroy()


def crowded_wall(cell_mode=1, **kw):
    """A dam break whose fluid near the middle of the x = 0 wall is drawn together:
    more candidates around it than a list segment holds as indices (256 at cells
    of 2h and h), so that fluid targets, and the ghost nodes of an mDBC wall, keep
    chunk records."""
    from scipy.spatial import cKDTree
    c = cases.dam_break(0.04, cell_mode=cell_mode, **kw)
    f = c.ptype == 0
    h = c.params["h"]
    mid = c.pos[f].mean(0)
    mid[0] = c.pos[f][:, 0].min()
    d = c.pos - mid
    near = f & (np.linalg.norm(d, axis=1) < 3.5 * h)
    c.pos[near] = mid + 0.62 * d[near]
    u = cases.uniform01(11, 3 * c.n_fluid).reshape(-1, 3) - 0.5
    c.vel[f] = (0.2 * u).astype(np.float32)
    tree = cKDTree(c.pos[f])
    where = c.pos[c.ptype == 1] + c.ghost[c.ptype == 1] if kw.get("boundary_mode") else c.pos[f]
    most = max(len(x) for x in tree.query_ball_point(where, 2.0 * h))
    assert most > 256, most
    return c


@pytest.mark.parametrize("cell_mode", [0, 1])
@pytest.mark.parametrize("kw", [dict(visc_mode=1, nu0=1e-3), dict(ddt_mode=2),
                                dict(boundary_mode=1, mdbc_slip=1), dict(integrator=1)])
def test_kept_records_of_other_physics(kw, cell_mode):
    """Targets that keep chunk records in the walks of laminar + SPS (with its
    strain pass), Fourtakas diffusion, mDBC (whose ghost nodes keep records too)
    and Verlet, against the oracle and by brute force."""
    c = crowded_wall(cell_mode, **kw)
    eng = sph.Engine.create(c)
    eng.set_options(pi_variant=5, check_list=1)
    for stage in (0,) if "integrator" in kw else (0, 1):
        g = check_step_eval(c, eng, stage)
        if "boundary_mode" in kw:
            check_boundary(c, g)
    eng.step(1)
    assert eng.list_info()["check_bad"] == 0
    eng.destroy()


@pytest.mark.parametrize("cell_mode", [0, 1])
@pytest.mark.parametrize("skin", [-1.0, 0.25])
def test_crowded_case_takes_the_same_steps_in_a_pool(cell_mode, skin):
    """A pool's list segments are larger than an engine's of the case alone.  Targets
    whose candidates fit only the larger one (257 to 384 of them) are summed in the
    same order in both: the same steps bit for bit."""
    from scipy.spatial import cKDTree
    c = cases.dam_break(0.04, cell_mode=cell_mode)
    f = c.ptype == 0
    h = c.params["h"]
    mid = c.pos[f].mean(0)
    d = c.pos - mid
    near = f & (np.linalg.norm(d, axis=1) < 3.0 * h)
    c.pos[near] = mid + 0.88 * d[near]
    most = max(map(len, cKDTree(c.pos).query_ball_point(c.pos[f], 2.16 * h)))  # 2h + skin
    assert 256 < most < 384, most
    pool = sph.Engine.pool(60000, 600000, 3)
    pool.set_options(list_skin=skin)
    pool.admit(cases.dam_break(0.04, seed=5, cell_mode=cell_mode), t_end=1.0)
    s = pool.admit(c, t_end=1.0)
    pool.pool_step(5)
    alone = sph.Engine.create(c)
    alone.set_options(list_skin=skin, check_list=1)
    alone.step(5)
    assert alone.list_info()["check_bad"] == 0
    a, b = alone.get_state(), pool.get_state(s)
    for k in ("pos", "vel", "rho"):
        assert np.array_equal(a[k], b[k]), k
    alone.destroy()
    pool.destroy()


@pytest.mark.parametrize("pooled", [0, 1])
def test_wide_skin_grows_the_list_segments(pooled):
    """list_skin above 0.1: longer list segments in the place of the first ones
    (4 bytes per candidate), kept when the skin narrows again; every pair is found
    and the evaluations match the oracle throughout."""
    import torch
    c = cases.dam_break(0.03)
    if pooled:
        eng = sph.Engine.pool(60000, 600000, 2)
        icase, slots = eng.admit(c, t_end=10.0), 60000
    else:
        eng, icase, slots = sph.Engine.create(c), 0, c.n
    bytes_of = torch.cuda.memory_allocated
    for skin in (-1.0, 0.25, 0.12, 0.0, -1.0):
        b0 = bytes_of()
        eng.set_options(list_skin=skin, check_list=1)
        grown = (bytes_of() - b0) / slots
        if skin == 0.25:
            # 480 entries instead of 256; a pool's (h up to 1.2 sqrt(3) dp) 800 of 384
            assert abs(grown - (4 * 416 if pooled else 4 * 224)) < 4 * 16, grown
        else:
            assert grown == 0
        eng.step(3)
        assert eng.list_info()["check_bad"] == 0
        for stage in (0, 1):
            check_step_eval(c, eng, stage, icase=icase)
    eng.destroy()
