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
