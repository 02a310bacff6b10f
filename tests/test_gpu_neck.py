"""The post-join kernel that runs the deconv neck, the fusion over the agents and
the head from the blocks' outputs, against the path that stores the neck's maps
(RTCC_FLAG_KEEP_FUSED), for tiles that are ragged, single and narrow, one to
three blocks, absent agents and both storage types: the same sums, so the same
bytes; and the feature maps, which are then computed when they are read, and
how long the maps stand."""
import dataclasses
import time

import pytest

import synth
from paper_2608_08330_gb300 import rtcc as R0
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    return U.load()


def _cfg(w, h, agents, dtype="fp16", blocks=((1, 64, 2), (2, 128, 2), (1, 256, 2)), ups=(1, 2, 4), **kw):
    hx, hy = 0.2 * w, 0.2 * h
    base = synth.get_config("pp3")
    return dataclasses.replace(
        base, n_agents=agents, grid_w=w, grid_h=h, x_min=-hx, x_max=hx, y_min=-hy, y_max=hy,
        pts_x=(-hx, hx), pts_y=(-hy, hy), n_uniform=3 * w, n_clusters=1, cluster_pts=50,
        max_pillars=w * h, dtype=dtype, blocks=blocks, up_strides=ups, cls_thresh=-1.0, **kw)


CASES = [
    ("one tile of one pixel", _cfg(8, 8, 1), ()),
    ("one wide row", _cfg(1040, 8, 2), ()),
    ("one narrow column", _cfg(8, 1040, 2, "bf16"), ()),
    ("ragged, several positions a CTA", _cfg(328, 184, 3, "bf16"), (1,)),
    ("all agents, 25 rows", _cfg(704, 200, 8), ()),
    ("all but one absent", _cfg(72, 40, 8), (0, 1, 2, 3, 4, 6, 7)),
    ("one block", _cfg(40, 24, 3, blocks=((2, 128, 2),), ups=(1,)), ()),
    ("two blocks, strides 2 and 4", _cfg(48, 40, 2, blocks=((1, 64, 1), (1, 256, 2)), ups=(1, 2)), ()),
    ("multi-scale", _cfg(88, 56, 3, fusion="attn"), (2,)),
]


@pytest.mark.parametrize("cfg,absent", [c[1:] for c in CASES], ids=[c[0] for c in CASES])
def test_neck_max_head_matches_the_stored_maps(R, cfg, absent):
    scales = cfg.fusion == "attn"
    flags = R.FLAG_MULTISCALE if scales else 0
    pts = [synth.points_for(cfg, 0, k) for k in range(cfg.n_agents)]
    got = []
    for f in (flags, flags | R.FLAG_KEEP_FUSED):
        ctx, _ = U.make_ctx(cfg, flags=f)
        try:
            for mode in (R.MODE_RTCC, R.MODE_BARRIER):
                boxes = U.run_frame(ctx, cfg, pts, list(range(cfg.n_agents)), mode, absent=absent)
                maps = ([R.rtcc_get_tensor(ctx, 0, R.TENSOR_FUSED)] if scales else
                        [R.rtcc_get_tensor(ctx, k, R.TENSOR_FEAT) for k in range(cfg.n_agents) if k not in absent])
                got.append((R.rtcc_get_head(ctx, cfg.feat_h, cfg.feat_w).tobytes(), boxes.tobytes(),
                            [m.tobytes() for m in maps]))
        finally:
            R.rtcc_destroy(ctx)
    assert all(g == got[0] for g in got[1:])


ATTN = [
    ("one tile of one pixel, the ego alone", _cfg(8, 8, 1, fusion="attn"), ()),
    ("one narrow column", _cfg(8, 1040, 2, "bf16", fusion="attn"), ()),
    ("ragged, several positions a CTA", _cfg(328, 184, 3, "bf16", fusion="attn"), (1,)),
    ("all agents, 25 rows", _cfg(704, 200, 8, fusion="attn"), ()),
    ("all but the ego and one absent", _cfg(72, 40, 8, fusion="attn"), (1, 2, 3, 4, 6, 7)),
    ("one block", _cfg(40, 24, 3, blocks=((2, 128, 2),), ups=(1,), fusion="attn"), ()),
    ("two blocks, strides 2 and 4", _cfg(48, 40, 2, "bf16", blocks=((1, 64, 1), (1, 256, 2)), ups=(1, 2),
                                         fusion="attn"), ()),
    ("an odd number of cells", _cfg(42, 22, 5, "bf16", blocks=((1, 128, 2),), ups=(1,), fusion="attn"), (2,)),
]


@pytest.mark.parametrize("cfg,absent", [c[1:] for c in ATTN], ids=[c[0] for c in ATTN])
def test_neck_attention_head_matches_the_stored_maps(R, cfg, absent):
    # the path that stores the maps takes its sums in the same order
    pts = [synth.points_for(cfg, 0, k) for k in range(cfg.n_agents)]
    got = []
    for f in (0, R.FLAG_KEEP_FUSED):
        ctx, w = U.make_ctx(cfg, flags=f)
        try:
            for mode in (R.MODE_RTCC, R.MODE_BARRIER):
                boxes = U.run_frame(ctx, cfg, pts, list(range(cfg.n_agents)), mode, absent=absent)
                got.append((R.rtcc_get_head(ctx, cfg.feat_h, cfg.feat_w).tobytes(), boxes.tobytes(),
                            R.rtcc_get_tensor(ctx, 0, R.TENSOR_FUSED).tobytes(),
                            [R.rtcc_get_tensor(ctx, k, R.TENSOR_FEAT).tobytes()
                             for k in range(cfg.n_agents) if k not in absent]))
            # the last frame's fused map, also once the next frame has begun
            assert R.rtcc_frame_begin(ctx, 9, 0.0) == R.OK
            assert R.rtcc_get_tensor(ctx, 0, R.TENSOR_FUSED).tobytes() == got[-1][2]
        finally:
            R.rtcc_destroy(ctx)
    assert all(g == got[0] for g in got[1:])


@pytest.mark.parametrize("flags", [0, R0.FLAG_KEEP_FUSED], ids=["computed by the head's kernel", "stored slots"])
def test_fused_map_stands_until_the_next_post_join(R, flags):
    """The last frame's fused map, and the feature slots of agents that the open
    frame has not released, while the open frame's branches overwrite their
    blocks' outputs."""
    cfg = _cfg(328, 184, 3, "bf16", fusion="attn")
    old, new = ([synth.points_for(cfg, f, k) for k in range(3)] for f in (0, 1))
    ctx, _ = U.make_ctx(cfg, flags=flags)
    try:
        U.run_frame(ctx, cfg, old, [0.0, 0.0, 0.0], R.MODE_RTCC)
        fused = R.rtcc_get_tensor(ctx, 0, R.TENSOR_FUSED).tobytes()
        feat0 = R.rtcc_get_tensor(ctx, 0, R.TENSOR_FEAT).tobytes()
        block1 = R.rtcc_get_tensor(ctx, 1, 1).tobytes()
        assert R.rtcc_frame_begin(ctx, 1, 0.0) == R.OK
        for k in (1, 2):
            assert R.rtcc_payload_complete(ctx, k, new[k], 0.0) == R.OK
        end = time.monotonic() + 20                    # branch 1 has run
        while R.rtcc_get_tensor(ctx, 1, 1).tobytes() == block1:
            assert time.monotonic() < end
        for _ in range(20):
            assert R.rtcc_get_tensor(ctx, 0, R.TENSOR_FUSED).tobytes() == fused
            assert R.rtcc_get_tensor(ctx, 0, R.TENSOR_FEAT).tobytes() == feat0
        assert R.rtcc_payload_complete(ctx, 0, new[0], 1.0) == R.OK
        s, _, _ = R.rtcc_wait_detection(ctx, 60000)
        assert s == R.OK
        after = R.rtcc_get_tensor(ctx, 0, R.TENSOR_FUSED).tobytes()
        assert after != fused
        U.run_frame(ctx, cfg, new, [0.0, 0.0, 0.0], R.MODE_BARRIER)
        assert R.rtcc_get_tensor(ctx, 0, R.TENSOR_FUSED).tobytes() == after
    finally:
        R.rtcc_destroy(ctx)
