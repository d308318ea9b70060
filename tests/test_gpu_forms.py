"""GPU tests of the forms that one call can take, at the edges of their ranges:
the FP64 symmetric sweep around its 128-disk blocks, the all-pairs force without
allocation around its thread and tile counts, the triangulation kernel as a grid,
as one cluster and with queued check passes, and the time step with its move in
the force's reduction or in a launch of its own.

Tolerances: forces as everywhere (1e-5 of the RMS force in FP32, 1e-12 in FP64);
trajectories of two forms agree to 1e-9 (they share every operation but the order
of the FP64 atomic additions of Algorithm 2, whose rounding is 2^-52 of a
correction and grows little in a few steps)."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1703_02484_gb300 as bd  # noqa: E402
from paper_1703_02484_gb300 import binding, workloads  # noqa: E402
from oracle import forces as oforces  # noqa: E402
from oracle import geometry  # noqa: E402

C2 = workloads.CONFIGS["c2"]


def stream():
    return torch.cuda.current_stream().cuda_stream


def lattice(n, L, seed):
    # n disks of radius 1 on a jittered square lattice: any n, no overlaps
    m = math.ceil(math.sqrt(n))
    rng = np.random.default_rng(seed)
    h = L / m
    ij = np.stack(np.meshgrid(np.arange(m), np.arange(m)), -1).reshape(-1, 2)[rng.permutation(m * m)[:n]]
    return (ij + 0.5) * h + rng.uniform(-1, 1, (n, 2)) * 0.49 * (h - 2.0)


def inputs(n, seed, periodic):
    L = float(np.float32(2.6 * math.ceil(math.sqrt(n))))
    rng = np.random.default_rng(seed + 1)
    sp = rng.integers(0, 2, n).astype(np.uint8)
    th = rng.uniform(0, 2 * math.pi, n).astype(np.float32)
    p = bd.params_from_config(C2, n=n)
    p.box_L = L
    if periodic:
        p.boundary = bd.BOUNDARY_PERIODIC
    return p, lattice(n, L, seed), sp, th, L


def rel_err(F, ref):
    return float(np.max(np.linalg.norm(F - ref, axis=1))) / math.sqrt(float(np.mean(np.sum(ref ** 2, axis=1))))


@pytest.mark.parametrize("n,periodic", [(3, False), (127, False), (128, True), (129, False), (129, True), (513, True),
                                        (1153, False)])
def test_fp64_sweep_edges(n, periodic):
    p, xy, sp, th, L = inputs(n, n, periodic)
    p.precision = 1
    s = bd.System(p, xy, sp, th, stream=stream())
    F = s.forces()
    grid = s.state(want_tri=False)["xy"]
    s.close()
    assert rel_err(F, oforces.long_range_numpy(grid, sp, C2.alpha, L=L if periodic else None)) <= 1e-12


@pytest.mark.parametrize("n", [1, 2, 63, 65, 127, 128, 129, 511, 513, 1025, 4097])
def test_noalloc_edges(n):
    _, xy, sp, _, _ = inputs(n, n, False)
    d_xy, d_sp = torch.from_numpy(xy).cuda(), torch.from_numpy(sp).cuda()
    d_F = torch.full((n + 1, 2), float("nan"), dtype=torch.float64, device="cuda")
    binding.forces_noalloc(n, d_xy.data_ptr(), d_sp.data_ptr(), C2.alpha, d_F.data_ptr(), stream())
    torch.cuda.synchronize()
    F = d_F.cpu().numpy()
    assert np.all(np.isnan(F[n]))            # nothing written past the end
    if n == 1:
        assert np.all(F[0] == 0.0)
    else:
        assert rel_err(F[:n], oforces.long_range_numpy(xy, sp, C2.alpha)) <= 1e-5


def crowded(monkeypatch, n, seed, periodic):
    # near-contact states: every step has corrections and flips.  The force sweep
    # is fixed: two sweeps that the autotuner may pick round differently.
    monkeypatch.setenv("BD_FORCE_VARIANT", "2")
    monkeypatch.setenv("BD_FORCE_TILES", "1")
    L = float(np.nextafter(np.float32(workloads.box_side(n, C2.rho)), np.float32(np.inf)))
    p = bd.params_from_config(C2, n=n)
    p.box_L = L
    if periodic:
        p.boundary = bd.BOUNDARY_PERIODIC
    xy = workloads.near_contact_state(n, L, C2.a, seed=seed)
    _, sp, th = workloads.initial_state(C2, n=n)
    return p, xy, sp, th


@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("n", [150, 1601, 3000])
def test_triangulation_forms_agree(monkeypatch, n, periodic):
    # the grid's kernel with an edge per thread, the same testing every triangle
    # in every pass, the queued passes, and the one cluster
    p, xy, sp, th = crowded(monkeypatch, n, 5, periodic)
    outs = []
    for env in ({"BD_TRI_CLUSTER": "0"}, {"BD_TRI_CLUSTER": "0", "BD_TRI_LISTS": "2"},
                {"BD_TRI_CLUSTER": "0", "BD_TRI_QUEUE": "0"}, {"BD_TRI_CLUSTER": "1000000"},
                {"BD_TRI_CLUSTER": "1000000", "BD_TRI_LISTS": "2"}):
        with monkeypatch.context() as m:
            for k, v in env.items():
                m.setenv(k, v)
            s = bd.System(p, xy, sp, th, stream=stream())
        st = s.step(12)
        assert st["steps_done"] == 12
        outs.append((env, s.state(), st))
        s.close()
    _, want, st0 = outs[0]
    assert st0["corr_iters"] > 0 and st0["flips"] > 0
    for env, o, st in outs[1:]:
        assert float(np.max(np.abs(o["xy"] - want["xy"]))) <= 1e-9, env
        assert np.array_equal(geometry.edges(o["tri"]), geometry.edges(want["tri"])), env
        assert st["corr_iters"] == st0["corr_iters"] and st["flips"] == st0["flips"], env


@pytest.mark.parametrize("form", ["cluster", "queue"])
def test_triangulation_forms_leave_at_a_timed_out_barrier(monkeypatch, form):
    if form == "cluster":
        monkeypatch.setenv("BD_TRI_CLUSTER", "1000000")
    else:
        monkeypatch.setenv("BD_TRI_CLUSTER", "0")
        monkeypatch.setenv("BD_TRI_QUEUE", "0")
    p, xy, sp, th = crowded(monkeypatch, 1601, 6, False)
    s = bd.System(p, xy, sp, th, stream=stream())
    free = bd.System(p, xy, sp, th, stream=stream())
    free.step(2)
    before = s.state()
    s.set_wait_limit(0.05, hold_barrier=3)
    st, code = s.step(2, raise_on_error=False)
    assert code == -7 and st["steps_done"] == 0
    after = s.state()
    assert np.array_equal(after["xy"], before["xy"]) and np.array_equal(after["tri"], before["tri"])
    s.set_wait_limit(2.0, hold_barrier=0)
    s.step(2)
    a, b = s.state(), free.state()
    assert float(np.max(np.abs(a["xy"] - b["xy"]))) <= 1e-9
    assert np.array_equal(geometry.edges(a["tri"]), geometry.edges(b["tri"]))
    s.close()
    free.close()


@pytest.mark.parametrize("n,variant,tiles,periodic,precision", [
    (3, 2, 1, False, 0), (511, 3, 1, True, 0), (513, 2, 1, False, 0), (3001, 3, 2, True, 0), (19000, 3, 4, False, 0),
    (3, 0, 1, False, 1), (129, 0, 1, True, 1), (1153, 0, 1, False, 1)])
def test_move_in_the_reduction(monkeypatch, n, variant, tiles, periodic, precision):
    # a timed single step keeps the force and the move in launches of their own
    if precision == 0:
        monkeypatch.setenv("BD_FORCE_VARIANT", str(variant))
        monkeypatch.setenv("BD_FORCE_TILES", str(tiles))
    p, xy, sp, th, L = inputs(n, n, periodic)
    p.precision = precision
    fused = bd.System(p, xy, sp, th, stream=stream())
    apart = bd.System(p, xy, sp, th, stream=stream())
    apart.force_timing(True)
    for _ in range(3):
        fused.step(1)
        apart.step(1)
    assert fused.last_launch_count() < apart.last_launch_count()
    a, b = fused.state(), apart.state()
    assert float(np.max(np.abs(a["xy"] - b["xy"]))) <= 1e-9
    assert np.array_equal(a["theta"], b["theta"])
    fused.close()
    apart.close()


@pytest.mark.parametrize("n", [257, 1601])
def test_rollout_passes_in_one_launch(monkeypatch, n):
    # the reverse pass (and its replay) with every correction pass as one launch
    # against two; they share all terms but the order of the additions to a disk,
    # whose last bits may round its FP32 multiplier (2^-24) in a later step
    p, xy, sp, th = crowded(monkeypatch, n, 7, False)
    out = []
    for pairs in ("1024", "-1"):
        monkeypatch.setenv("BD_ADJ_PAIRS", pairs)
        s = bd.System(p, xy, sp, th, stream=stream())
        loss, st = s.rollout(9, ckpt_every=4)
        assert st["corr_iters"] > 0
        out.append((loss, s.rollout_vjp()))
        s.close()
    assert out[0][0] == out[1][0]
    assert float(np.max(np.abs(out[0][1] - out[1][1]))) <= 1e-6 * float(np.max(np.abs(out[1][1])))
