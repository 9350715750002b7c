"""sim_adjoint (FP32 forward, FP64 adjoint field, through the C ABI) vs the FP64 oracle
adjoint and vs FP64 central finite differences of the oracle's forward loss.

How close an FP32 forward pass can bring the gradient to the FP64 one depends on the
problem, not only on the code: a cone that climbs to a cue maximum or reaches a point
source circles it, and there the gradient direction turns within a cell, so a rounding
difference of 1e-7 in a position grows by 10^3-10^4 over the circling and moves the
derivative of the endpoint loss by 1e-3 to 1e-1.  Each test therefore first measures, with
the oracle alone, how far its own gradients move when the inputs are perturbed at the size
of the rounding an FP32 run accumulates (``_spread``):

* well-conditioned cases (spread well under the bar) must match the oracle and central
  differences to ADJ_RTOL = 1e-4;
* the adjoint workload's own setting (cue front growing from C = 0, 200 steps) is compared
  within max(ADJ_RTOL, BAND x spread): the GPU must land inside the oracle's own band.  The
  kernels round each value a handful of times per step where the binary32-storage run of the
  oracle rounds it once; k independent roundings add up to about sqrt(k) times one, and
  k <= 25, hence BAND = 5.
"""
import numpy as np
import pytest

import oracle
from paper_1405_3331_gb300 import workloads as W
from parity import cone_of, grid_of

pytestmark = pytest.mark.gpu

ADJ_RTOL = 1e-4
U32 = 2.0 ** -24          # FP32 unit roundoff
BAND = 5.0


@pytest.fixture(scope="module")
def cue():
    from paper_1405_3331_gb300 import build
    build.build()
    from paper_1405_3331_gb300 import cue as binding
    return binding


def _copy64(seed=50, nsteps=200):
    """The adjoint workload's 64x64 copy: 2 sources, 64 cones, wall clamp, targets, C0 = 0."""
    return W.config_c5(seed=seed, n=64, n_src=2, n_axons=64, nsteps=nsteps)


def _ramp2d(seed=59):
    """2D cue field on a tilted plane (no interior maximum) with weak sources: no cone
    circles a critical point within 80 steps, so the derivative is well conditioned."""
    return W.make("adj2d-ramp", 2, 64, 48, n_src=3, emit=(0.02, 0.05), n_axons=64, C0="ramp",
                  seed=seed, wall_mode=1, src_map="zeros", targets=True)


def _gpu(cue, w, nsteps, k):
    sim = cue.Simulation(w)
    g = sim.adjoint(w.targets, nsteps, k)
    sim.check()
    out = {key: (None if v is None else v.cpu().numpy()) for key, v in g.items()}
    sim.close()
    return out


def _oracle(w, nsteps, pos=None, C0=None, D=None, lam=None, binary32=False):
    grid = oracle.Grid(w.dim, w.nx, w.ny, w.nz if w.dim == 3 else 1, h=w.h,
                       D=w.D if D is None else D, lam=w.lam if lam is None else lam, dt=w.dt)
    return oracle.adjoint(grid, cone_of(w), w.field0().astype(np.float64) if C0 is None else C0,
                          w.src_cell, w.src_emit, w.src_map, w.pos if pos is None else pos, w.dir,
                          w.targets, nsteps, state_binary32=binary32)


def _rel(a, b):
    return abs(a - b) / max(abs(b), 1e-30)


def _relmax(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-30))


KEYS = ("dD", "dlambda", "dsrc", "dmap")


def _spread(w, T, ref):
    """Largest relative change of each oracle gradient under perturbations of the size FP32
    makes: every forward state stored in binary32 (the oracle's ``state_binary32`` run), and
    the initial positions, the initial field, D and lambda perturbed by delta = sqrt(T) * u32
    relative (the rounding a T-step run accumulates if per-step errors add like a random walk)."""
    delta = np.sqrt(T) * U32
    pos0 = w.pos.astype(np.float64)
    C0 = w.field0().astype(np.float64)
    runs = [_oracle(w, T, binary32=True)]
    for s in range(2):
        rng = np.random.default_rng(1000 + s)
        runs.append(_oracle(w, T, pos=pos0 * (1 + delta * rng.standard_normal(pos0.shape)),
                            C0=C0 * (1 + delta * rng.standard_normal(C0.shape))))
    runs.append(_oracle(w, T, D=w.D * (1 + delta)))
    runs.append(_oracle(w, T, lam=w.lam * (1 + delta)))
    return {k: max(_relmax(r[i + 1], ref[i + 1]) for r in runs) for i, k in enumerate(KEYS)}


def _check_strict(g, ref):
    loss, gD, gl, gsrc, gmap = ref
    assert _rel(float(g["loss"]), loss) < 1e-5
    assert _rel(float(g["dD"]), gD) < ADJ_RTOL
    assert _rel(float(g["dlambda"]), gl) < ADJ_RTOL
    assert _relmax(g["dsrc"], gsrc) < ADJ_RTOL
    assert _relmax(g["dmap"], gmap) < ADJ_RTOL


def test_adjoint_2d_well_conditioned_matches_oracle(cue):
    w, T = _ramp2d(), 80
    ref = _oracle(w, T)
    spread = _spread(w, T, ref)
    assert max(spread.values()) < ADJ_RTOL / 3, spread       # precondition on the case
    _check_strict(_gpu(cue, w, T, 16), ref)


def test_adjoint_2d_matches_finite_differences(cue):
    """GPU gradients against central differences of the FP64 oracle's loss (relative steps
    inside the linear regime), on the well-conditioned 2D case: D, lambda, every emission,
    and the rate map at its largest-gradient node, at a source node and at a random node."""
    w, T = _ramp2d(), 80
    g = _gpu(cue, w, T, 16)
    c = cone_of(w)
    C0 = w.field0().astype(np.float64)

    def loss(D=w.D, lam=w.lam, emit=w.src_emit, smap=w.src_map):
        grid = oracle.Grid(2, w.nx, w.ny, h=w.h, D=D, lam=lam, dt=w.dt)
        return oracle.endpoint_loss(grid, c, C0, w.src_cell, emit, smap, w.pos, w.dir, w.targets, T)

    hD, hl = 1e-6 * w.D, 1e-5 * w.lam
    assert _rel(float(g["dD"]), (loss(D=w.D + hD) - loss(D=w.D - hD)) / (2 * hD)) < ADJ_RTOL
    assert _rel(float(g["dlambda"]), (loss(lam=w.lam + hl) - loss(lam=w.lam - hl)) / (2 * hl)) < ADJ_RTOL
    for k in range(w.n_src):
        e1, e2 = w.src_emit.astype(np.float64).copy(), w.src_emit.astype(np.float64).copy()
        h = 1e-5 * e1[k]
        e1[k] += h
        e2[k] -= h
        assert _rel(float(g["dsrc"][k]), (loss(emit=e1) - loss(emit=e2)) / (2 * h)) < ADJ_RTOL
    rng = np.random.default_rng(7)
    nodes = {int(np.argmax(np.abs(g["dmap"]))), int(w.src_cell[0]), int(rng.integers(w.n_cells))}
    for node in nodes:
        m1, m2 = w.src_map.astype(np.float64).copy(), w.src_map.astype(np.float64).copy()
        m1.flat[node] += 1e-4
        m2.flat[node] -= 1e-4
        fd = (loss(smap=m1) - loss(smap=m2)) / 2e-4
        assert abs(float(g["dmap"].flat[node]) - fd) <= ADJ_RTOL * np.abs(g["dmap"]).max(), node


@pytest.mark.parametrize("seed", [50, 51])
def test_adjoint_front_workload_within_the_oracle_band(cue, seed):
    """The adjoint workload's 64x64 copy over 200 steps: the loss to 1e-5; each gradient
    within max(ADJ_RTOL, BAND x the oracle's own spread).  With C0 = 0 and M = 0 the loss does
    not change when every emission is scaled alike, so sum_k e_k dL/de_k = 0 and dL/de is the
    small remainder of terms that cancel: its band is wider than that of dD.  In seed 51
    cones circle a source and every band is wide."""
    w, T = _copy64(seed=seed), 200
    ref = _oracle(w, T)
    spread = _spread(w, T, ref)
    g = _gpu(cue, w, T, 64)
    assert _rel(float(g["loss"]), ref[0]) < 1e-5
    for i, k in enumerate(KEYS):
        tol = max(ADJ_RTOL, BAND * spread[k])
        assert _relmax(g[k], ref[i + 1]) <= tol, (k, _relmax(g[k], ref[i + 1]), tol)
    for cell in w.src_cell:                          # source-node map entries, one by one
        tol = max(ADJ_RTOL, BAND * spread["dmap"] * np.abs(ref[4]).max() / abs(ref[4].flat[cell]))
        assert _rel(float(g["dmap"].flat[cell]), ref[4].flat[cell]) < tol


def test_adjoint_3d_matches_oracle(cue):
    w = W.make("adj3d", 3, 20, 16, 12, dt=0.15, n_src=3, n_axons=40, C0="smooth", seed=52, wall_mode=1,
               src_map=True, targets=True)
    T = 60
    ref = _oracle(w, T)
    spread = _spread(w, T, ref)
    assert max(spread.values()) < ADJ_RTOL / 3, spread
    _check_strict(_gpu(cue, w, T, 16), ref)


@pytest.mark.parametrize("k", [1, 7, 200])
def test_checkpoint_interval_does_not_change_the_gradients(cue, k):
    w = _copy64(seed=53, nsteps=100)
    ref = _gpu(cue, w, 100, 64)
    g = _gpu(cue, w, 100, k)
    for key in ("loss", "dD", "dlambda"):
        assert _rel(float(g[key]), float(ref[key])) < 1e-6
    assert np.abs(g["dmap"] - ref["dmap"]).max() <= 1e-6 * np.abs(ref["dmap"]).max()


def test_autograd_function_gives_the_adjoint_gradients(cue):
    import torch
    from paper_1405_3331_gb300.autograd import endpoint_loss
    w = _copy64(seed=54, nsteps=80)
    dev = torch.device("cuda:0")
    D = torch.tensor(w.D, dtype=torch.float32, device=dev, requires_grad=True)
    lam = torch.tensor(w.lam, dtype=torch.float32, device=dev, requires_grad=True)
    emit = torch.as_tensor(w.src_emit, device=dev).clone().requires_grad_(True)
    smap = torch.as_tensor(w.src_map, device=dev).clone().requires_grad_(True)
    L = endpoint_loss(D, lam, emit, smap, w, w.targets, 80, 16)
    (3.0 * L).backward()
    ref = _gpu(cue, w, 80, 16)
    assert _rel(float(L.detach()), float(ref["loss"])) < 1e-6
    assert _rel(float(D.grad), 3 * float(ref["dD"])) < 1e-5
    assert _rel(float(lam.grad), 3 * float(ref["dlambda"])) < 1e-5
    np.testing.assert_allclose(emit.grad.cpu().numpy(), 3 * ref["dsrc"], rtol=1e-5)
    np.testing.assert_allclose(smap.grad.cpu().numpy(), 3 * ref["dmap"], rtol=1e-5, atol=1e-12)


def test_autograd_problem_reuses_its_buffers_and_skips_the_adjoint_without_grad(cue):
    """An EndpointProblem called repeatedly gives the same loss and gradients bit for bit
    (its state is reset on the device each call), new parameter values take effect (D and
    lambda through cue_set_physics, emissions and map copied device to device), and under
    no_grad the forward alone (coupled steps + the loss kernel) gives the adjoint's loss."""
    import torch
    from paper_1405_3331_gb300.autograd import EndpointProblem
    w = _copy64(seed=57, nsteps=60)
    dev = torch.device("cuda:0")
    prob = EndpointProblem(w, w.targets, 60, 16, device=dev)
    D = torch.tensor(w.D, dtype=torch.float32, device=dev, requires_grad=True)
    lam = torch.tensor(w.lam, dtype=torch.float32, device=dev, requires_grad=True)
    emit = torch.as_tensor(w.src_emit, device=dev).clone().requires_grad_(True)
    smap = torch.as_tensor(w.src_map, device=dev).clone().requires_grad_(True)
    L1 = prob(D, lam, emit, smap)
    L1.backward()
    g1 = [t.grad.clone() for t in (D, lam, emit, smap)]
    for t in (D, lam, emit, smap):
        t.grad = None
    L2 = prob(D, lam, emit, smap)
    L2.backward()
    assert float(L1.detach()) == float(L2.detach())
    for a, t in zip(g1, (D, lam, emit, smap)):
        assert torch.equal(a, t.grad)
    ref = _gpu(cue, w, 60, 16)
    assert _rel(float(L1.detach()), float(ref["loss"])) < 1e-6
    assert _rel(float(g1[0]), float(ref["dD"])) < 1e-6
    with torch.no_grad():
        L0 = prob(D, lam, emit, smap)
    assert _rel(float(L0), float(ref["loss"])) < 1e-6
    # other parameter values: the same as a fresh handle built with them
    w2 = W.config_c5(seed=57, n=64, n_src=2, n_axons=64, nsteps=60)
    w2.D, w2.lam = 0.8, 0.02
    w2.src_emit = (w.src_emit * 1.5).astype(np.float32)
    ref2 = _gpu(cue, w2, 60, 16)
    D2 = torch.tensor(0.8, dtype=torch.float32, device=dev, requires_grad=True)
    lam2 = torch.tensor(0.02, dtype=torch.float32, device=dev, requires_grad=True)
    e2 = torch.as_tensor(w2.src_emit, device=dev).clone().requires_grad_(True)
    L3 = prob(D2, lam2, e2, smap)
    L3.backward()
    assert float(L3.detach()) == float(ref2["loss"])
    assert float(D2.grad) == float(ref2["dD"])
    np.testing.assert_array_equal(e2.grad.cpu().numpy(), ref2["dsrc"])
    prob.close()


def test_adjoint_refuses_runs_that_stop(cue):
    w = W.make("stop", 2, 32, 32, n_src=2, n_axons=8, C0="smooth", seed=55, targets=True)   # wall stop
    sim = cue.Simulation(w)
    with pytest.raises(cue.CueError) as e:
        sim.adjoint(w.targets, 10, 4)
    assert e.value.code == cue.CUE_ERR_ARG


def test_full_size_source_and_map_gradients_agree(cue):
    """The adjoint workload at its full size (1024^2, 4,096 cones, 2,000 steps, checkpoint
    every 64) is out of the oracle's reach; an identity that holds at any size is checked
    instead.  A point source adds e_k at its node every step and the rate map adds dt M
    there, so dL/de_k = dL/dM[cell_k] / dt.  The two sides are accumulated separately (one
    FP64 sum per source against the per-segment map sums), so a dropped step, a misplaced
    node or a wrong segment fold on either side shows."""
    w = W.config_c5()
    g = _gpu(cue, w, w.nsteps, 64)
    for key in ("loss", "dD", "dlambda"):
        assert np.isfinite(g[key]).all()
    de = g["dsrc"].astype(np.float64)
    via_map = g["dmap"].reshape(-1)[w.src_cell.astype(np.int64)].astype(np.float64) / w.dt
    scale = np.abs(de).max()
    assert scale > 0
    assert np.abs(de - via_map).max() <= 1e-4 * scale


def test_full_size_persistent_backward_equals_two_launch_backward(cue):
    """Same full-size workload through the persistent backward (one launch per segment) and
    through the two-launches-per-step backward: the forward trajectories agree bit for bit,
    the backward computes the same sums in another order, so every gradient agrees to
    rounding (relative to its largest entry)."""
    w = W.config_c5()
    a = _gpu(cue, w, w.nsteps, 64)
    sim = cue.Simulation(w, path=cue.CUE_PATH_PLAIN)
    gb = sim.adjoint(w.targets, w.nsteps, 64)
    sim.check()
    b = {key: (None if v is None else v.cpu().numpy()) for key, v in gb.items()}
    sim.close()
    assert a["loss"] == b["loss"]
    for key in ("dD", "dlambda", "dsrc", "dmap"):
        x, y = a[key].astype(np.float64), b[key].astype(np.float64)
        scale = max(np.abs(y).max(), 1e-30)
        assert np.abs(x - y).max() <= 1e-4 * scale, key


@pytest.mark.parametrize("nx,ny,n_axons,nsteps,k", [
    (132, 5, 40, 11, 4),          # a second strip one lane wide; fewer rows than warps
    (4, 3, 3, 7, 7),              # the smallest: every scatter folded at a wall
    (260, 900, 700, 9, 3),        # three strips, two rows a warp at most
    (128, 31000, 300, 5, 3),      # a dozen rows a warp
    (256, 192, 9000, 70, 64),     # more cones than one run of linearisations over the segment holds
])
def test_persistent_backward_equals_launches_per_step_at_odd_shapes(cue, nx, ny, n_axons, nsteps, k):
    """The persistent backward takes the cones' linearisations from a launch before it, for a
    bounded number of steps, and shares its rows out between warps; the launches per step do
    neither.  Same states, the same double-float sums in another order: the emission and map
    gradients agree to ADJ_RTOL of their largest entry.  (dD and dlambda are FP32 products over a
    smooth field whose large terms cancel; they are held to the FP64 oracle on the identical
    states below.)"""
    w = W.make("shape", 2, nx, ny, n_src=2, n_axons=n_axons, C0="smooth", seed=nx + ny, wall_mode=1,
               src_map="zeros", targets=True)
    out = []
    for path in (None, cue.CUE_PATH_PLAIN):
        sim = cue.Simulation(w) if path is None else cue.Simulation(w, path=path)
        g = sim.adjoint(w.targets, nsteps, k)
        sim.check()
        out.append({key: (None if v is None else v.cpu().numpy()) for key, v in g.items()})
        sim.close()
    a, b = out
    assert a["loss"] == b["loss"]
    for key in ("dsrc", "dmap"):
        x, y = a[key].astype(np.float64), b[key].astype(np.float64)
        scale = max(np.abs(y).max(), 1e-30)
        assert np.abs(x - y).max() <= ADJ_RTOL * scale, key


def test_adjoint_full_horizon_on_the_small_copy_is_reported(cue, record_property):
    """The adjoint workload's 64x64 copy over its full 2,000 steps (checkpoint every 64): the
    GPU gradients, the FP64 oracle's adjoint and FP64 central differences of the oracle's loss
    for D, lambda and each emission, recorded as relative differences.  Over this horizon
    the cones orbit the sources and the derivative is ill-conditioned (the oracle's own
    spread under FP32-sized perturbations is recorded beside it), so the numbers are a
    report, not a pass criterion; the run must stay finite and the loss must agree."""
    w, T = _copy64(seed=50), 2000
    g = _gpu(cue, w, T, 64)
    ref = _oracle(w, T)
    loss, gD, gl, gsrc, _ = ref
    c = cone_of(w)
    C0 = w.field0().astype(np.float64)

    def loss_at(D=w.D, lam=w.lam, emit=w.src_emit):
        grid = oracle.Grid(2, w.nx, w.ny, h=w.h, D=D, lam=lam, dt=w.dt)
        return oracle.endpoint_loss(grid, c, C0, w.src_cell, emit, w.src_map, w.pos, w.dir, w.targets, T)

    hD, hl = 1e-6 * w.D, 1e-5 * w.lam
    fd = {"dD": (loss_at(D=w.D + hD) - loss_at(D=w.D - hD)) / (2 * hD),
          "dlambda": (loss_at(lam=w.lam + hl) - loss_at(lam=w.lam - hl)) / (2 * hl)}
    fd_src = []
    for k in range(w.n_src):
        e1, e2 = w.src_emit.astype(np.float64).copy(), w.src_emit.astype(np.float64).copy()
        h = 1e-5 * e1[k]
        e1[k] += h
        e2[k] -= h
        fd_src.append((loss_at(emit=e1) - loss_at(emit=e2)) / (2 * h))
    for key in ("loss", "dD", "dlambda", "dsrc", "dmap"):
        assert np.isfinite(g[key]).all(), key
    assert _rel(float(g["loss"]), loss) < 1e-3
    record_property("gpu_vs_oracle_dD", _rel(float(g["dD"]), gD))
    record_property("gpu_vs_oracle_dlambda", _rel(float(g["dlambda"]), gl))
    record_property("gpu_vs_oracle_dsrc", _relmax(g["dsrc"], gsrc))
    record_property("oracle_vs_fd_dD", _rel(gD, fd["dD"]))
    record_property("oracle_vs_fd_dlambda", _rel(gl, fd["dlambda"]))
    record_property("oracle_vs_fd_dsrc", _relmax(gsrc, fd_src))
    record_property("gpu_vs_fd_dD", _rel(float(g["dD"]), fd["dD"]))
    record_property("gpu_vs_fd_dlambda", _rel(float(g["dlambda"]), fd["dlambda"]))
    record_property("gpu_vs_fd_dsrc", _relmax(g["dsrc"], fd_src))
    print("full-horizon 64x64 adjoint, relative differences:",
          {"gpu_vs_oracle": [_rel(float(g["dD"]), gD), _rel(float(g["dlambda"]), gl), _relmax(g["dsrc"], gsrc)],
           "oracle_vs_fd": [_rel(gD, fd["dD"]), _rel(gl, fd["dlambda"]), _relmax(gsrc, fd_src)]})


def _gpu_traced(cue, w, nsteps, k, path=None):
    sim = cue.Simulation(w) if path is None else cue.Simulation(w, path=path)
    g = sim.adjoint(w.targets, nsteps, k, trace=True)
    sim.check()
    out = {key: (None if v is None else v.cpu().numpy()) for key, v in g.items()}
    out["pos_end"] = sim.pos.cpu().numpy()
    sim.close()
    return out


@pytest.mark.parametrize("seed,path", [(50, None), (51, None), (50, "plain")])
def test_adjoint_backward_over_the_gpu_states_full_horizon(cue, seed, path):
    """The backward pass held to 1e-4 over the adjoint workload's whole horizon: the 64x64 copy,
    2,000 steps, checkpoint every 64.  The forward of an FP32 run and of the FP64 oracle part
    ways over this horizon (cones circle the sources; see the reported test above), so the
    backward kernels are compared on the identical states instead: the FP32 states the GPU
    recomputed from its checkpoints and walked back (cue_adjoint_trace) go into the oracle's
    backward pass alone (FP64), and the GPU gradients must match it -- dD, dlambda and every
    e_k to 1e-4 relative, every rate-map entry to 1e-4 of the largest, the loss to 1e-6.
    Run on the persistent backward (one launch per segment) and on the per-step launches."""
    w, T = _copy64(seed=seed), 2000
    g = _gpu_traced(cue, w, T, 64, path=cue.CUE_PATH_PLAIN if path == "plain" else None)
    Cs = g["trace_C"].astype(np.float64)
    Ps, Ds = g["trace_cone"][:, 0], g["trace_cone"][:, 1]
    # the trace is the run: it starts at the initial state and ends where the forward ended
    np.testing.assert_array_equal(g["trace_C"][0], w.field0())
    np.testing.assert_array_equal(Ps[0], w.pos)
    np.testing.assert_array_equal(Ds[0], w.dir)
    np.testing.assert_array_equal(Ps[-1], g["pos_end"])
    grid = oracle.Grid(2, w.nx, w.ny, h=w.h, D=w.D, lam=w.lam, dt=w.dt)
    loss, gD, gl, gsrc, gmap = oracle.adjoint_from_states(grid, cone_of(w), w.src_cell, w.targets, Cs, Ps, Ds)
    errs = {"loss": _rel(float(g["loss"]), loss), "dD": _rel(float(g["dD"]), gD),
            "dlambda": _rel(float(g["dlambda"]), gl), "dsrc": _relmax(g["dsrc"], gsrc),
            "dsrc_each": max(_rel(float(g["dsrc"][k]), gsrc[k]) for k in range(w.n_src)),
            "dmap": _relmax(g["dmap"], gmap)}
    print(f"identical-state backward, seed {seed}, {path or 'persistent'}: relative differences {errs}")
    assert _rel(float(g["loss"]), loss) < 1e-6
    assert _rel(float(g["dD"]), gD) < ADJ_RTOL, (float(g["dD"]), gD)
    assert _rel(float(g["dlambda"]), gl) < ADJ_RTOL, (float(g["dlambda"]), gl)
    for k in range(w.n_src):
        assert _rel(float(g["dsrc"][k]), gsrc[k]) < ADJ_RTOL, (k, float(g["dsrc"][k]), gsrc[k])
    assert _relmax(g["dmap"], gmap) < ADJ_RTOL


def test_adjoint_backward_over_the_gpu_states_3d(cue):
    """The same identical-state comparison in 3D (trilinear sample, 3-component noise), over
    600 steps with checkpoints every 50: gradients to 1e-4 of the oracle's backward pass."""
    w = W.make("adj3d-long", 3, 20, 16, 12, dt=0.15, n_src=3, n_axons=40, C0="smooth", seed=56, wall_mode=1,
               src_map=True, targets=True)
    T = 600
    g = _gpu_traced(cue, w, T, 50)
    Cs = g["trace_C"].astype(np.float64)
    Ps, Ds = g["trace_cone"][:, 0], g["trace_cone"][:, 1]
    np.testing.assert_array_equal(Ps[-1], g["pos_end"])
    grid = oracle.Grid(3, w.nx, w.ny, w.nz, h=w.h, D=w.D, lam=w.lam, dt=w.dt)
    loss, gD, gl, gsrc, gmap = oracle.adjoint_from_states(grid, cone_of(w), w.src_cell, w.targets, Cs, Ps, Ds)
    print("identical-state backward, 3D: relative differences",
          {"dD": _rel(float(g["dD"]), gD), "dlambda": _rel(float(g["dlambda"]), gl),
           "dsrc": _relmax(g["dsrc"], gsrc), "dmap": _relmax(g["dmap"], gmap)})
    assert _rel(float(g["loss"]), loss) < 1e-6
    assert _rel(float(g["dD"]), gD) < ADJ_RTOL
    assert _rel(float(g["dlambda"]), gl) < ADJ_RTOL
    assert _relmax(g["dsrc"], gsrc) < ADJ_RTOL
    assert _relmax(g["dmap"], gmap) < ADJ_RTOL
