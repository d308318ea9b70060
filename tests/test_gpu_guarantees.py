"""GPU tests of guarantees that no trajectory with noise shows by itself: image
shifts stay out of boxes with walls, and what follows below each heading."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1703_02484_gb300 as bd  # noqa: E402
from paper_1703_02484_gb300 import workloads  # noqa: E402


def stream():
    return torch.cuda.current_stream().cuda_stream


# ---------------------------------------------------------------- boxes of both kinds in one handle

@pytest.mark.parametrize("cluster", ["0", "1000000"])
def test_walled_boxes_take_no_image_shifts(monkeypatch, cluster):
    # the shift pass reads the re-entries of every triangle's corners, ghost
    # points among them: those of a box with walls never re-enter, whatever the
    # periodic boxes of the same handle do
    monkeypatch.setenv("BD_TRI_CLUSTER", cluster)
    cfgs = workloads.batch_configs(3, seed=31, n_lo=300, n_hi=900)
    params, xys, sps, ths = [], [], [], []
    for r, cfg in enumerate(cfgs):
        xy, sp, th = workloads.initial_state(cfg, seed=31 + r)
        p = bd.params_from_config(cfg)
        p.replica = r
        if r == 1:
            p.box_L = float(np.nextafter(np.float32(workloads.box_side(p.n, cfg.rho)), np.float32(np.inf)))
            p.boundary = bd.BOUNDARY_PERIODIC
            p.D = 25.0                                                  # (0.07 a step: a dozen re-enter)
            xy = np.mod(xy + np.array([0.3, 0.7]) * p.box_L, p.box_L)   # disks across the edges
        params.append(p)
        xys.append(xy)
        sps.append(sp)
        ths.append(th)
    b = bd.System(params, np.concatenate(xys), np.concatenate(sps), np.concatenate(ths), stream=stream())
    before = b.replica(1)["xy"]
    entered = 0
    for _ in range(20):
        assert b.step(2)["steps_done"] == 2
        now = b.replica(1)["xy"]
        entered += int(np.sum(np.abs(now - before) > 0.5 * params[1].box_L))
        before = now
        for r in (0, 2):
            assert not b.tri_shifts(r).any()
    assert entered > 0
    b.close()


# ---------------------------------------------------------------- pushes that cancel

FORMS = [{"BD_TRI_CLUSTER": "0"}, {"BD_TRI_CLUSTER": "0", "BD_TRI_LISTS": "2"},
         {"BD_TRI_CLUSTER": "0", "BD_TRI_QUEUE": "0"}, {"BD_TRI_CLUSTER": "1000000"},
         {"BD_TRI_CLUSTER": "1000000", "BD_TRI_LISTS": "2"}]
FORM_IDS = ["grid", "grid-all", "queue", "cluster", "cluster-all"]


def system_moving_to(target, dy, L, periodic, precision, **kw):
    # a handle whose next step ends at `target` before any correction: no force,
    # no noise, every disk driven up or down by about dy.  The move does not
    # depend on the positions, so it is read off a step of the same disks on a
    # wide jittered lattice; all coordinates are multiples of 2^-5, so nothing rounds
    n = len(target)
    theta = np.where(np.arange(n) % 2 == 0, 0.5 * math.pi, -0.5 * math.pi).astype(np.float32)

    def make(xy, side, **kw):
        p = bd.make_params(n, L=side, D=0.0, v0=dy / 0.125, dt=0.125, precision=precision,
                           boundary=bd.BOUNDARY_PERIODIC if periodic else bd.BOUNDARY_WALLS, **kw)
        return bd.System(p, xy, theta=theta, stream=stream())

    m = math.ceil(math.sqrt(n))
    wide = np.array([(4.0 * (k % m) + 3.0, 4.0 * (k // m) + 3.0) for k in range(n)])
    wide += np.random.default_rng(1).integers(-16, 17, wide.shape) / 32.0
    s = make(wide, max(L, 4.0 * m + 4.0))
    q0, _ = s.geometry()
    s.step(1)
    move = s.state()["xy"] - wide
    s.close()
    s = make(target - move, L, **kw)
    q1, _ = s.geometry()
    assert q1 <= q0      # the move is on the finer grid too
    start = s.state()["xy"]
    assert np.array_equal(start + move, target)
    return s, start


@pytest.mark.parametrize("env", FORMS, ids=FORM_IDS)
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("periodic", [False, True])
def test_overlap_between_disks_whose_pushes_cancel(monkeypatch, periodic, precision, env):
    # four disks in a row, each overlapping the next by 1/16: the inner two
    # are pushed equally from both sides, so the first pass moves the outer
    # two only and leaves the inner pair as it was
    from oracle import overlap
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    L = 30.0
    target = np.array([(10.0 + 1.9375 * k, 15.0) for k in range(4)]
                      + [(5.0 + 4 * k, y) for y in (4.0, 26.0) for k in range(6)]
                      + [(x, y) for x in (7.0, 12.90625, 19.0) for y in (11.0, 19.0)])
    s, _ = system_moving_to(target, 0.3, L, periodic, precision)
    st = s.step(1)
    ref = (overlap.correct_periodic if periodic else overlap.correct)(target, L, 1.0)
    assert ref[2] == 4 and not ref[4]
    out = s.state()["xy"]
    s.close()
    assert st["steps_done"] == 1 and st["corr_iters"] == 4
    assert float(np.max(np.abs(out - ref[0]))) <= 1e-9
    d = out[:4, None] - out[None, :4]
    assert float(np.min(np.hypot(d[..., 0], d[..., 1]) + 9.0 * np.eye(4))) >= 2.0 * (1 - 1e-12)


@pytest.mark.parametrize("env", FORMS, ids=FORM_IDS)
def test_closed_row_of_overlapping_disks_does_not_converge(monkeypatch, env):
    # a row round the periodic box, each disk pushed equally from both sides:
    # no pass moves any, and the step is undone with an error
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    L = 30.0
    target = np.array([(0.9375 + 1.875 * k, 15.0) for k in range(16)]
                      + [(1.5 + 3.0 * k, y) for y in (4.0, 10.0, 20.0, 26.0) for k in range(10)])
    s, start = system_moving_to(target, 0.35, L, True, 0, max_corr_iters=20)
    st, code = s.step(1, raise_on_error=False)
    assert code == -5 and st["fail_phase"] == 5 and st["steps_done"] == 0
    assert np.array_equal(s.state()["xy"], start)
    s.close()


# ---------------------------------------------------------------- one result however a step is launched

def test_step_is_the_same_bits_however_it_is_launched(monkeypatch):
    # a graph's replay, launches of their own, and the force timed apart from the
    # move.  16384 disks for 600 steps: about 2e7 force components, enough that
    # two orders of the partial sums (2^-46 apart, the move reads 2^-24) differ
    monkeypatch.setenv("BD_FORCE_VARIANT", "3")
    monkeypatch.setenv("BD_FORCE_TILES", "1")
    cfg = workloads.CONFIGS["c2"]
    n = 16384
    xy, sp, th = workloads.initial_state(cfg, n=n)
    out = []
    for form in ("graph", "plain", "timed"):
        with monkeypatch.context() as m:
            if form == "plain":
                m.setenv("BD_NO_GRAPH", "1")
            s = bd.System(bd.params_from_config(cfg, n=n), xy, sp, th, stream=stream())
        if form == "timed":
            s.force_timing(True)
        for _ in range(6):
            assert s.step(100)["steps_done"] == 100
        out.append(s.state())
        s.close()
    for o in out[1:]:
        assert np.array_equal(o["xy"], out[0]["xy"]) and np.array_equal(o["theta"], out[0]["theta"])
        assert np.array_equal(o["tri"], out[0]["tri"])


def test_plain_launches_are_those_of_the_graph(monkeypatch):
    cfg = workloads.CONFIGS["c2"]
    monkeypatch.setenv("BD_FORCE_VARIANT", "2")
    monkeypatch.setenv("BD_FORCE_TILES", "1")
    xy, sp, th = workloads.initial_state(cfg, n=3000)
    counts = []
    for off in (False, True):
        if off:
            monkeypatch.setenv("BD_NO_GRAPH", "1")
        s = bd.System(bd.params_from_config(cfg, n=3000), xy, sp, th, stream=stream())
        s.step(3)
        counts.append(s.last_launch_count())
        s.close()
    assert counts[0] == counts[1]


def test_fp32_rollout_replay_follows_the_recorded_run(monkeypatch):
    # without contacts (a wide lattice) the replay is the recorded moves from the
    # same forces, bit for bit; 16384 disks for 600 steps as above
    monkeypatch.setenv("BD_FORCE_VARIANT", "3")
    monkeypatch.setenv("BD_FORCE_TILES", "1")
    cfg = workloads.CONFIGS["c5"]
    m, h = 128, 8.0
    n = m * m
    rng = np.random.default_rng(5)
    xy = (np.stack(np.meshgrid(np.arange(m), np.arange(m)), -1).reshape(-1, 2) + 0.5) * h + rng.uniform(-1, 1, (n, 2))
    sp = rng.integers(0, 2, n).astype(np.uint8)
    th = rng.uniform(0, 2 * math.pi, n).astype(np.float32)
    p = bd.params_from_config(cfg, n=n)
    p.box_L = m * h
    s = bd.System(p, xy, sp, th, stream=stream())
    loss, st = s.rollout(600, ckpt_every=200)
    assert st["steps_done"] == 600 and st["corr_iters"] == 0
    end = s.state(want_tri=False)["xy"]
    assert s.rollout_replay() == loss
    assert np.array_equal(s.rollout_positions(1), end)
    s.close()


# ---------------------------------------------------------------- Verlet lists that run out of room

def dense_block(n, h, L):
    # n disks on a square lattice of spacing h in a corner of the box
    m = math.ceil(math.sqrt(n))
    k = np.arange(n)
    return np.stack([2.0 + h * (k % m), 2.0 + h * (k // m)], 1) + 0.5


@pytest.mark.parametrize("verlet", [False, True])
def test_list_overflow_is_an_error_each_time(verlet):
    # 400 disks 2.05 apart within reach 10.6: inner disks have some 80
    # neighbours, a list holds 64
    L = 90.0
    p = bd.make_params(400, L=L, law=bd.LAW_SHORT, r_cut=10.0, skin=0.6, D=0.01, dt=1e-4)
    if verlet:
        p.overlap_mode = bd.OVERLAP_VERLET
    s = bd.System(p, dense_block(400, 2.05, L), stream=stream())
    start = s.state()["xy"]
    for _ in range(3):
        st, code = s.step(2, raise_on_error=False)
        assert code == -10 and st["steps_done"] == 0
        with pytest.raises(bd.BDError) as e:
            s.forces()
        assert e.value.code == -10
    assert np.array_equal(s.state()["xy"], start)
    s.close()


def test_state_whose_lists_overflow_is_refused_whole():
    L = 90.0
    p = bd.make_params(400, L=L, law=bd.LAW_SHORT, r_cut=10.0, skin=0.6, D=0.01, Dr=0.1, v0=1.0, dt=1e-4)
    p.overlap_mode = bd.OVERLAP_VERLET
    wide = dense_block(400, 4.0, L)
    s = bd.System(p, wide, stream=stream())
    twin = bd.System(p, wide, stream=stream())
    s.step(3)
    twin.step(3)
    before = s.state()
    with pytest.raises(bd.BDError) as e:
        s.set_state(dense_block(400, 2.05, L), before["theta"] + np.float32(1.0))
    assert e.value.code == -10
    after = s.state()
    assert np.array_equal(after["xy"], before["xy"]) and np.array_equal(after["theta"], before["theta"])
    # and the handle goes on as if nothing had been asked (entries beyond the
    # cut-off, which a later rebuild may drop, add nothing to a force)
    s.step(3)
    twin.step(3)
    assert np.array_equal(s.state()["xy"], twin.state()["xy"])
    s.close()
    twin.close()


# ---------------------------------------------------------------- force shards without work items

def test_ranks_without_work_items_add_nothing(monkeypatch):
    # more ranks than the sweep has work items: a rank without any contributes a
    # force of 0 at every step, not what its arrays held before
    monkeypatch.setenv("BD_FORCE_VARIANT", "3")
    monkeypatch.setenv("BD_FORCE_TILES", "8")
    cfg = workloads.CONFIGS["c2"]
    n, world = 1024, 5
    xy, sp, th = workloads.initial_state(cfg, n=n)

    def make():
        return bd.System(bd.params_from_config(cfg, n=n), xy, sp, th, stream=stream())

    whole = make()
    assert whole.tuning()["n_items"] < world
    ranks = [make() for _ in range(world)]
    for r, h in enumerate(ranks):
        h.forces()                       # (the whole force is in every rank's arrays)
        h.set_force_shard(r, world)
    F = torch.empty(2 * whole.force_slots(), dtype=torch.float64, device="cuda")
    tot = torch.empty_like(F)
    for step in range(3):
        whole.step_begin(F.data_ptr())
        ref = F.clone()
        scale = float(torch.sqrt(torch.mean(ref.view(-1, 2).pow(2).sum(1))))
        tot.zero_()
        zero = 0
        for h in ranks:
            h.step_begin(F.data_ptr())
            zero += int(float(F.abs().max()) == 0.0)
            tot += F
        assert zero == world - whole.tuning()["n_items"]
        # (FP32 partial sums, split otherwise: a few roundings of 2^-46 apart)
        assert float((tot - ref).abs().max()) <= 1e-10 * scale
        for h in ranks:
            h.step_end(tot.data_ptr())
        whole.step_end(tot.data_ptr())
    for h in ranks + [whole]:
        h.close()


# ---------------------------------------------------------------- a tuning read back

@pytest.mark.parametrize("groups", [2, 4, 8, 24])
@pytest.mark.parametrize("variant", [2, 3])
def test_tuning_read_back_makes_the_same_sweep(monkeypatch, variant, groups):
    cfg = workloads.CONFIGS["c2"]
    n = 3001
    xy, sp, th = workloads.initial_state(cfg, n=n)
    monkeypatch.setenv("BD_FORCE_VARIANT", str(variant))
    monkeypatch.setenv("BD_FORCE_GROUPS", str(groups))
    a = bd.System(bd.params_from_config(cfg, n=n), xy, sp, th, stream=stream())
    t = a.tuning()
    assert t["variant"] == variant and t["groups_per_item"] == groups
    assert t["tiles_per_item"] == (groups + 7) // 8
    F = a.forces()
    a.close()
    monkeypatch.setenv("BD_FORCE_VARIANT", str(t["variant"]))
    monkeypatch.setenv("BD_FORCE_TILES", str(t["tiles_per_item"]))
    monkeypatch.setenv("BD_FORCE_GROUPS", str(t["groups_per_item"]))
    b = bd.System(bd.params_from_config(cfg, n=n), xy, sp, th, stream=stream())
    assert b.tuning() == t and np.array_equal(b.forces(), F)
    b.close()


def test_autotuned_sweep_can_be_asked_for_again(monkeypatch):
    for k in ("BD_FORCE_VARIANT", "BD_FORCE_TILES", "BD_FORCE_GROUPS", "BD_NCHUNK"):
        monkeypatch.delenv(k, raising=False)
    cfg = workloads.CONFIGS["c2"]
    for n in (777, 4096, 16384):
        xy, sp, th = workloads.initial_state(cfg, n=n)
        a = bd.System(bd.params_from_config(cfg, n=n), xy, sp, th, stream=stream())
        t, F = a.tuning(), a.forces()
        a.close()
        with monkeypatch.context() as m:
            m.setenv("BD_FORCE_VARIANT", str(t["variant"]))
            if t["variant"] >= 2:
                m.setenv("BD_FORCE_GROUPS", str(t["groups_per_item"]))
            else:
                m.setenv("BD_FORCE_TILES", str(t["tiles_per_item"]))
            b = bd.System(bd.params_from_config(cfg, n=n), xy, sp, th, stream=stream())
        assert b.tuning() == t and np.array_equal(b.forces(), F)
        b.close()
