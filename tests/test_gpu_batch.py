"""Backbone launches over several agents whose split-K layers exchange their
slices through distributed shared memory.  On these grids a cluster of four CTAs
holds tiles of different agents in successive layers, so an agent that runs
ahead must not reach into an exchange that another agent's tile still reads.
Many frames, every agent's blocks and the head byte for byte against launches of
one agent each and against launches without clusters (no exchange)."""
import dataclasses

import pytest

import synth
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    return U.load()


def _cfg(w, h, agents, dtype):
    hx, hy = 0.2 * w, 0.2 * h
    return dataclasses.replace(
        synth.get_config("pp3"), n_agents=agents, grid_w=w, grid_h=h, x_min=-hx, x_max=hx, y_min=-hy,
        y_max=hy, pts_x=(-hx, hx), pts_y=(-hy, hy), n_uniform=40 * w, n_clusters=2, cluster_pts=200,
        max_pillars=w * h, dtype=dtype, cls_thresh=-1.0)


@pytest.mark.parametrize("w,h,agents,dtype", [
    (64, 64, 8, "fp16"), (64, 64, 5, "bf16"), (128, 64, 3, "bf16"), (176, 96, 2, "fp16")])
def test_batched_exchanges_keep_their_agents_apart(R, w, h, agents, dtype):
    cfg = _cfg(w, h, agents, dtype)
    frames = [[synth.points_for(cfg, f, k) for k in range(agents)] for f in range(3)]

    def outputs(ctx, f):
        boxes = U.run_frame(ctx, cfg, frames[f], [0.0] * agents, R.MODE_BARRIER)
        return [boxes.tobytes(), R.rtcc_get_head(ctx, cfg.feat_h, cfg.feat_w).tobytes()] + [
            R.rtcc_get_tensor(ctx, k, 1 + b).tobytes() for k in range(agents) for b in range(len(cfg.blocks))]

    want = None
    for flags, turns in ((R.FLAG_NO_BATCH, 1), (R.FLAG_NO_CLUSTERS, 1), (0, 20)):
        ctx, _ = U.make_ctx(cfg, flags=flags)
        try:
            got = [[outputs(ctx, f) for f in range(len(frames))] for _ in range(turns)]
            if flags == 0:
                info = R.rtcc_get_frame_info(ctx)
                assert info.n_backbone_launches == 1 and info.backbone_batch[0] == agents
        finally:
            R.rtcc_destroy(ctx)
        want = want or got[0]
        assert all(g == want for g in got)


def test_unbatched_branches_report_their_spans(R):
    """RTCC_FLAG_NO_BATCH: a branch released while another's backbone runs waits
    for it, and still reports its whole span."""
    cfg = _cfg(328, 184, 4, "fp16")
    pts = [synth.points_for(cfg, 0, k) for k in range(4)]
    ctx, _ = U.make_ctx(cfg, flags=R.FLAG_NO_BATCH | R.FLAG_TIMELINE)
    try:
        for mode in (R.MODE_BARRIER, R.MODE_RTCC):
            for f in range(5):
                U.run_frame(ctx, cfg, pts, [0.0] * 4, mode, frame_id=f)
                info = R.rtcc_get_frame_info(ctx)
                for k in range(4):
                    assert 0 < info.gpu_backbone_ms[k] < info.gpu_branch_ms[k] < 100
    finally:
        R.rtcc_destroy(ctx)
