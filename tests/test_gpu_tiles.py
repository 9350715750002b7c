"""The persistent path's tile engine (csrc/k_tiles.cu) against the plain path, bit for bit:
both field buffers, the cone state and the cone-update count.  The cases are the edges of its
range: one and several tiles per axis, rows that are not a multiple of 4 nodes, shifted last
tiles, one to sixteen steps per round, rounds cut short by the end of a run, a tile with more
cones than its shared-memory list, cones that all cross tile borders, walls, stops, rate maps
and the SNR rule."""
import math

import numpy as np
import pytest

from paper_1405_3331_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SNR = dict(gain=8.0, width=2.0, kd=1.5, c_min=0.05, c_max=50.0, turn=math.pi / 30)


@pytest.fixture(scope="module")
def cue():
    from paper_1405_3331_gb300 import build
    build.build()
    from paper_1405_3331_gb300 import cue as binding
    return binding


def _case(name):
    nx, ny = (int(v) for v in name.split("-")[0].split("x"))
    tags = name.split("-")[1:]
    n = next((int(t[:-5]) for t in tags if t.endswith("cones")), 500)
    w = W.make(name, 2, nx, ny, n_src=0 if "nosrc" in tags else 9, emit=(0.5, 2.0), n_axons=n, C0="smooth", seed=nx + ny,
               stop_radius=3.0 if "stop" in tags else 0.0, wall_mode=1 if "clamp" in tags else 0,
               src_map="random" if "map" in tags else False)
    if "crowd" in tags:                                  # all cones start in a square of 20 nodes
        rng = np.random.default_rng(nx)
        w.pos = (np.array([[nx * 0.4], [ny * 0.6]]) + rng.uniform(-10, 10, (2, n))).astype(np.float32)
    if "inactive" in tags:
        w.active[::3] = 0
    return w


def _run(cue, w, path, chunks, depth=0, snr=None):
    sim = cue.Simulation(w, path=path)
    if depth:
        sim.set_option(cue.CUE_OPT_TEMPORAL_DEPTH, depth)
    if snr:
        sim.set_steering(snr)
    for k in chunks:
        sim.sim_run(k)
    sim.check()
    out = [f.cpu().numpy() for f in (sim.fields[sim.state()[2]], sim.fields[sim.state()[2] ^ 1])]
    out += list(sim.snapshot()[1:]) + [sim.state()[2], sim.cone_updates()]
    info = sim.last_path(), sim.get_option(cue.CUE_INFO_GRID)
    sim.close()
    return out, info


def _assert_same(a, b):
    for k, (x, y) in enumerate(zip(a, b)):
        assert np.array_equal(x, y), f"output {k} differs"


@pytest.mark.parametrize("name,chunks", [
    ("512x300", [1]), ("512x300", [2, 0, 1, 40]), ("257x300-stop", [37]), ("258x300-clamp-map", [37]),
    ("1025x769-stop-4096cones", [45]), ("640x512-map-clamp-3000cones", [33]), ("1003x131-nosrc", [31]),
    ("520x400-crowd-clamp-5000cones", [50]), ("517x403-crowd-stop-2500cones", [50]),
    ("640x400-inactive-clamp", [21]), ("700x500-0cones", [26]),
])
def test_tile_engine_equals_plain_bitwise(cue, name, chunks):
    w = _case(name)
    a, _ = _run(cue, w, cue.CUE_PATH_PLAIN, chunks)
    b, (path, grid) = _run(cue, w, cue.CUE_PATH_AUTO, chunks)
    assert path == cue.CUE_PATH_PERSIST and grid > 1
    _assert_same(a, b)


def test_crowded_runs_go_to_another_path_and_come_back(cue):
    """4,000 cones in one tile: the run after the first is left to another path (the crowd read
    back from the first), later ones return; every run gives the plain path's values."""
    import torch
    w = _case("1024x640-crowd-clamp-4000cones")
    a, b = cue.Simulation(w, path=cue.CUE_PATH_PLAIN), cue.Simulation(w)
    paths = []
    for k in range(18):
        for s in (a, b):
            s.load(C=w.field0(), pos=w.pos, dir=w.dir, active=w.active, step=0)
            s.sim_run(5 + k % 3)
            s.check()
        paths.append(b.last_path())
        torch.cuda.synchronize()
        _assert_same(a.snapshot(), b.snapshot())
    assert paths[0] == cue.CUE_PATH_PERSIST and paths[1] == cue.CUE_PATH_FUSED
    assert cue.CUE_PATH_PERSIST in paths[2:]
    a.close()
    b.close()


@pytest.mark.parametrize("depth", [1, 2, 3, 5, 8, 16])
@pytest.mark.parametrize("name", ["512x384-clamp-2000cones", "263x301-map-stop"])
def test_any_number_of_steps_per_round(cue, name, depth):
    w = _case(name)
    a, _ = _run(cue, w, cue.CUE_PATH_PLAIN, [35])
    b, (path, _) = _run(cue, w, cue.CUE_PATH_AUTO, [35], depth=depth)
    assert path == cue.CUE_PATH_PERSIST
    _assert_same(a, b)


@pytest.mark.parametrize("name", ["512x384-clamp-2000cones", "301x263-stop"])
def test_snr_rule_on_tiles(cue, name):
    w = _case(name)
    a, _ = _run(cue, w, cue.CUE_PATH_PLAIN, [30], snr=SNR)
    b, (path, _) = _run(cue, w, cue.CUE_PATH_AUTO, [30], snr=SNR)
    assert path == cue.CUE_PATH_PERSIST
    _assert_same(a, b)


@pytest.mark.parametrize("nx,ny", [(512, 300), (261, 300)])
def test_adjoint_states_on_tiles_are_the_plain_path_s(cue, nx, ny):
    """The recomputed segments (trajectory mode) against the plain path's, state by state."""
    w = W.config_c5(seed=3, n=64, n_src=6, n_axons=300, nsteps=40)
    full = W.make("tr", 2, nx, ny, n_src=6, n_axons=300, wall_mode=1, seed=5, C0="ramp", src_map="zeros", targets=True)
    assert w.wall_mode == full.wall_mode
    got = []
    for path in (cue.CUE_PATH_PLAIN, cue.CUE_PATH_AUTO):
        sim = cue.Simulation(full, path=path)
        got.append(sim.adjoint(full.targets, 40, 12, trace=True))
        sim.check()
        sim.close()
    for k in ("trace_C", "trace_cone", "loss"):
        assert np.array_equal(got[0][k].cpu().numpy(), got[1][k].cpu().numpy()), k


# A strip of one tile row whose tile borders in x are known: W = 128 loaded columns, a halo of K + 1 nodes and the drift
# of K - 1 steps of 0.05 (one node), rounded up to whole float4 groups.
FLIP_TILES = range(3, 79, 5)


def _flip_case(depth, rate_map=False):
    """Tiles that hold 124 cones in their middle and 10 around their border, walking at random: their number
    rises above 128 (the cones a tile steps from registers), falls to 128 or below and rises again, for rounds of any number."""
    halo = (depth + 1 + (depth > 1) + 3) // 4 * 4
    first, inner = 128 - halo, 128 - 2 * halo
    n = 134 * len(FLIP_TILES)
    w = W.make("flip", 2, 9600, 16, n_src=9, emit=(0.5, 2.0), n_axons=n, C0="smooth", seed=40 + depth, wall_mode=1,
               src_map="random" if rate_map else False, targets=True, w=(0.0, 0.1, 1.0), step_len=0.05)
    rng = np.random.default_rng(depth)
    for i, k in enumerate(FLIP_TILES):
        left = first + (k - 1) * inner
        x = np.concatenate([left + rng.uniform(20, inner - 20, 124), left + rng.uniform(-0.2, 0.2, 10)])
        w.pos[0, 134 * i : 134 * (i + 1)] = x
        w.pos[1, 134 * i : 134 * (i + 1)] = rng.uniform(2, 13, 134)
    tile = lambda x: np.where(x < first, 0, 1 + (np.floor(x) - first) // inner)
    return w, lambda x: np.array([(tile(x) == k).sum() for k in FLIP_TILES])


def _returns(crowds):
    """How often a tile is crowded again after an odd number of rounds in which it was not."""
    found = 0
    for c in np.array(crowds).T > 128:
        at = np.flatnonzero(c)
        found += int(((np.diff(at) > 1) & (np.diff(at) % 2 == 0)).sum())
    return found


@pytest.mark.parametrize("depth,rate_map", [(1, False), (3, False), (5, True), (7, False), (8, False)])
def test_stored_states_of_tiles_that_are_crowded_now_and_then(cue, depth, rate_map):
    w, crowd = _flip_case(depth, rate_map)
    steps, got = max(26 * depth, 100), []
    for path in (cue.CUE_PATH_PLAIN, cue.CUE_PATH_AUTO):
        sim = cue.Simulation(w, path=path)
        sim.set_option(cue.CUE_OPT_TEMPORAL_DEPTH, depth)
        got.append(sim.adjoint(w.targets, steps, steps, trace=True))
        sim.check()
        sim.close()
    plain, tiles = ({k: g[k].cpu().numpy() for k in ("trace_cone", "trace_C", "loss")} for g in got)
    assert _returns([crowd(plain["trace_cone"][s, 0, 0]) for s in range(0, steps, depth)]) > 0
    for k in plain:
        assert np.array_equal(plain[k], tiles[k]), k


@pytest.mark.parametrize("name,depth,chunk", [
    ("512x300-clamp-4000cones", 0, 1), ("515x301-stop-4000cones", 5, 1), ("515x301-stop-4000cones", 1, 2),
    ("640x400-crowd-stop-5000cones", 0, 1), ("644x400-crowd-clamp-5000cones", 0, 3),
    ("640x400-crowd-clamp-5000cones", 1, 2), ("640x401-crowd-stop-5000cones", 4, 7),
])
def test_many_short_runs_find_every_cone_once(cue, name, depth, chunk):
    """The cones are found anew by every run, from arrays that the run's other blocks are about to write. Cones cross
    tile borders all the time; the caches are cold before each run, so that blocks load at different speeds."""
    import torch
    w = _case(name)
    w.w_grad, w.w_noise = 0.1, 0.5
    flush = torch.empty(96 << 20, dtype=torch.int32, device="cuda:0")
    a = cue.Simulation(w, path=cue.CUE_PATH_PLAIN)
    b = cue.Simulation(w, path=cue.CUE_PATH_AUTO if w.nx % 4 else cue.CUE_PATH_PERSIST)
    b.set_option(cue.CUE_OPT_TEMPORAL_DEPTH, depth)
    for k in range(60):
        a.sim_run(chunk)
        flush.fill_(k)
        b.sim_run(chunk)
        b.check()
        _assert_same(a.snapshot(), b.snapshot())
    assert b.get_option(cue.CUE_INFO_GRID) > 1 and a.cone_updates() == b.cone_updates()
    a.close()
    b.close()


@pytest.mark.parametrize("seed", [3, 14, 15, 92])
def test_long_runs_whose_cones_gather(cue, seed):
    """The large endpoint configuration: its cones gather at 32 sources, in tiles that hold 128 now and 129 then, over
    2,000 steps of 7 a round."""
    w = W.config_c5(seed=seed, n=1024, n_src=32, n_axons=4096, nsteps=2000)
    a, _ = _run(cue, w, cue.CUE_PATH_PLAIN, [2000])
    b, (path, _) = _run(cue, w, cue.CUE_PATH_AUTO, [2000])
    assert path == cue.CUE_PATH_PERSIST
    _assert_same(a, b)


@pytest.mark.parametrize("depth", [1, 2, 6])
@pytest.mark.parametrize("name", ["640x400-crowd-clamp-8000cones", "640x400-crowd-stop-3000cones"])
def test_a_crowd_that_marches_through_tiles(cue, name, depth):
    """All cones go the same way, from tile to tile: far more than a neighbour is posted, in lists that are longer than
    shared memory holds, so that every inbox on the way is filled, emptied and filled again."""
    w = _case(name)
    w.w_prev, w.w_grad, w.w_noise = 1.0, 0.0, 0.02
    w.dir[0], w.dir[1] = 0.6, -0.8
    a, _ = _run(cue, w, cue.CUE_PATH_PLAIN, [130])
    b, (path, _) = _run(cue, w, cue.CUE_PATH_PERSIST, [90, 40], depth=depth)
    assert path == cue.CUE_PATH_PERSIST
    _assert_same(a, b)


@pytest.mark.parametrize("name,steps,path", [
    ("1025x769-1000cones", 1, "PLAIN"), ("1025x769-1000cones", 64, "PERSIST"), ("1024x1024-0cones", 1, "FUSED"),
    ("1024x1024-0cones", 64, "PERSIST"), ("1024x1024-4000cones", 8, "PERSIST"), ("1700x1700-1000cones", 64, "FUSED"),
    ("1701x1701-1000cones", 64, "PLAIN"),
])
def test_the_library_s_choice_compares_whole_runs(cue, name, steps, path):
    """A run's modelled time against the path it would displace: short runs do not pay for the engine's start, nor
    grids for tiles too tall for it."""
    w = _case(name)
    a, _ = _run(cue, w, cue.CUE_PATH_PLAIN, [steps])
    b, (got, _) = _run(cue, w, cue.CUE_PATH_AUTO, [steps])
    assert got == getattr(cue, "CUE_PATH_" + path)
    _assert_same(a[:1] + a[2:], b[:1] + b[2:])           # (the fused path leaves an earlier step in the other buffer)


def test_crowds_on_rows_of_any_length_go_to_another_path_and_are_looked_at_again(cue):
    """As above for rows that are not whole float4 groups; while the crowd stays, the engine is tried again after
    15, 30, ... runs."""
    import torch
    w = _case("1025x769-crowd-clamp-4000cones")
    a, b = cue.Simulation(w, path=cue.CUE_PATH_PLAIN), cue.Simulation(w)
    paths = []
    for k in range(49):
        b.load(C=w.field0(), pos=w.pos, dir=w.dir, active=w.active, step=0)
        b.sim_run(20)
        b.check()
        paths.append(b.last_path())
        torch.cuda.synchronize()
    engine, other = cue.CUE_PATH_PERSIST, cue.CUE_PATH_PLAIN
    assert paths == [engine] + 15 * [other] + [engine] + 30 * [other] + [engine] + [other]
    a.sim_run(20)
    _assert_same(a.snapshot(), b.snapshot())
    a.close()
    b.close()


def test_a_wait_that_runs_out_is_reported_and_the_next_run_is_normal(cue):
    """Two looks at a neighbour's packets are too few: blocks give up, the others follow, the launch ends and the
    status says so; its tags, counts and abort word are no part of the next run."""
    w = _case("512x384-clamp-2000cones")
    sim = cue.Simulation(w, path=cue.CUE_PATH_PERSIST)
    for steps in (40, 100):
        sim.set_option(cue.CUE_OPT_WAIT_LIMIT, 1)
        sim.sim_run(steps)
        assert sim.status() == cue.CUE_ERR_TIMEOUT
        assert sim.status() == cue.CUE_OK                # cleared after reporting
    sim.set_option(cue.CUE_OPT_WAIT_LIMIT, 0)
    sim.load(C=w.field0(), pos=w.pos, dir=w.dir, active=w.active, step=0)
    sim.sim_run(31)
    sim.check()
    got = sim.snapshot()
    sim.close()
    ref = cue.Simulation(w, path=cue.CUE_PATH_PLAIN)
    ref.sim_run(31)
    _assert_same(ref.snapshot(), got)
    ref.close()


def test_device_side_problems_are_reported(cue):
    """Non-finite input is reported; sources outside the grid are skipped and reported."""
    w = _case("512x300")
    w.C0 = w.field0()
    w.C0[100, 300] = np.nan
    sim = cue.Simulation(w)
    sim.sim_run(3)
    assert sim.last_path() == cue.CUE_PATH_PERSIST
    assert sim.status() == cue.CUE_ERR_NONFINITE
    sim.close()
    w = _case("512x300")
    w.src_cell = np.array([5, 512 * 300 + 7, -3], np.int32)
    w.src_emit = np.ones(3, np.float32)
    sim = cue.Simulation(w)
    sim.status()
    sim.sim_run(3)
    assert sim.status() == cue.CUE_ERR_BOUNDS
    sim.close()
