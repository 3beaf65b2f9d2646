"""Tiles of 176 keys under 65 to 128 text rows, whose last 16 columns are kept apart, and tiles with columns that
none of a warp's text rows sees, against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2411_10803_b200 import binding as md
from paper_2411_10803_b200 import build as md_build
from paper_2411_10803_b200 import synth

from parity_util import assert_scores_close, cfg, force, to_dev_bf16
from test_gpu_layers import run_ragged_layer
from test_gpu_parity import run_chain_and_check, small

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    md_build.build()


# keys that end in the last 16 columns (at 161, 169, 176), on their edge, in a tile of 160; the causal triangle in
# them, in front of them and across two CTAs; one head and more heads than buffers
@pytest.mark.parametrize("cluster,n_vis,n_txt,n_heads", [(1, 96, 65, 1), (1, 40, 128, 7), (2, 273, 65, 5), (2, 224, 128, 4),
                                                         (3, 400, 113, 6), (4, 576, 128, 9), (4, 530, 100, 3), (2, 200, 120, 3)])
@pytest.mark.parametrize("path", ["filter", "staged"])
def test_wide_tiles_match_the_oracle(cluster, n_vis, n_txt, n_heads, path, monkeypatch):
    force(monkeypatch, variant="fused", cluster=cluster)
    w = small(batch=2, n_vis=n_vis, n_txt=n_txt, n_heads=n_heads, hidden=128 * n_heads, vis_start=0, key_cnt=5, budget=n_vis // 3)
    f = md.Filter(cfg(w))
    tile = (-(-w.seq_len // cluster) + 15) // 16 * 16
    assert "cluster %d," % cluster in f.description and "%d keys per CTA" % tile in f.description
    f.close()
    run_chain_and_check(w, path=path)


# every cluster size holds tiles of 176 keys under more than 64 rows, with both readings of Eq. 10: the keys that
# fill them have a plan of one launch (seven and eight CTAs: two buffers; nine and more: two statistics slots)
@pytest.mark.parametrize("flags", [0, md.MUSTDROP_FLAG_PER_HEAD_MAX])
@pytest.mark.parametrize("cluster,n_txt", [(6, 65), (7, 128), (8, 100), (9, 128), (11, 70), (12, 66), (14, 128), (16, 65), (16, 128)])
def test_wide_tiles_in_large_clusters(cluster, n_txt, flags):
    w = small(batch=2, n_vis=cluster * 176 - n_txt, n_txt=n_txt, n_heads=5, hidden=640, vis_start=0)
    d = synth.make_batch(w, with_values=False)
    f = md.Filter(cfg(w, flags=flags, debug_score_variant=md.MUSTDROP_DEBUG_VARIANT_FUSED, debug_cluster=cluster))
    assert "cluster %d," % cluster in f.description and "176 keys per CTA" in f.description
    f.score(to_dev_bf16(d["q_text"]), to_dev_bf16(d["k"]))
    torch.cuda.synchronize()
    assert f.device_status() == (0, 0)
    G, I = (oracle.score_per_head if flags else oracle.score)(d["q_text"], d["k"], w.vis_start, w.n_vis, w.txt_start)
    assert_scores_close(f.g.cpu().numpy(), G, "G")
    assert_scores_close(f.i.cpu().numpy(), I, "I")
    f.close()


@pytest.mark.parametrize("batch,n_vis,n_txt", [(6, 2515, 119), (6, 2598, 96), (12, 1327, 114)])
def test_wide_tiles_with_few_slots_leave_one_head_to_grid_plans(batch, n_vis, n_txt):
    """(A tenth faster there; the clusters of nine and sixteen looked as fast.)"""
    w = small(batch=batch, n_vis=n_vis, n_txt=n_txt, n_heads=1, hidden=128, vis_start=0, n_salient=0, key_cnt=0, budget=n_vis // 7)
    f = md.Filter(cfg(w))
    assert "grid plan" in f.description
    f.close()


@pytest.mark.parametrize("flags", [0, md.MUSTDROP_FLAG_PER_HEAD_MAX])
@pytest.mark.parametrize("cluster,n_vis,n_txt,tail", [(2, 274, 78, 0), (3, 400, 120, 8), (9, 1484, 100, 0)])
def test_wide_tiles_without_a_mask(cluster, n_vis, n_txt, tail, flags):
    """Every row sees every key, those behind the text span among them."""
    w = small(batch=2, n_vis=n_vis, n_txt=n_txt, n_heads=5, hidden=640, vis_start=0)
    d = synth.make_batch(w, with_values=False)
    behind = synth.f32_to_bf16_bits(np.random.default_rng(4).standard_normal((2, 5, tail, 128), dtype=np.float32))
    k = np.concatenate([d["k"], behind], axis=2)
    f = md.Filter(cfg(w, flags=flags, causal=0, seq_len=w.seq_len + tail, debug_score_variant=md.MUSTDROP_DEBUG_VARIANT_FUSED,
                      debug_cluster=cluster))
    assert "176 keys per CTA" in f.description
    f.score(to_dev_bf16(d["q_text"]), to_dev_bf16(k))
    torch.cuda.synchronize()
    assert f.device_status() == (0, 0)
    G, I = (oracle.score_per_head if flags else oracle.score)(d["q_text"], k, w.vis_start, w.n_vis, w.txt_start, False)
    assert_scores_close(f.g.cpu().numpy(), G, "G")
    assert_scores_close(f.i.cpu().numpy(), I, "I")
    f.close()


@pytest.mark.parametrize("rebuild", [False, True])
@pytest.mark.parametrize("cluster,n_vis,n_txt,vis_cnt", [
    (4, 576, 128, [576, 400, 60, 33]),       # sequences that end with the last tile, the third, in the second, in the first's last 16
    (4, 600, 100, [429, 428, 251, 76]),      # ... one key into the last tile, on its edge, one short of two tiles, on the first's edge
])
def test_wide_tiles_that_a_short_sequence_never_reaches(cluster, n_vis, n_txt, vis_cnt, rebuild, monkeypatch):
    force(monkeypatch, variant="fused", cluster=cluster)
    w = small(batch=4, n_vis=n_vis, n_txt=n_txt, n_heads=5, hidden=640, vis_start=0, key_cnt=5, budget=30)
    f = md.Filter(cfg(w))
    assert "176 keys per CTA" in f.description
    f.close()
    run_ragged_layer(w, np.array(vis_cnt, np.int32), rebuild)


@pytest.mark.parametrize("flags", [0, md.MUSTDROP_FLAG_PER_HEAD_MAX])
@pytest.mark.parametrize("jump", [0, 150, 161, 170])
def test_logits_that_leave_the_range_in_the_last_columns(jump, flags):
    """From key `jump` of every CTA's tile on the logits lie 60 nats higher: the stabiliser moves while a chunk of the
    buffer, the last chunk, or both are under way (jump 0: never)."""
    w = small(batch=2, n_vis=284, n_txt=68, n_heads=5, hidden=640, n_salient=0, vis_start=0)
    d = synth.make_batch(w, with_values=False)
    q, k = synth.bf16_bits_to_f32(d["q_text"]), synth.bf16_bits_to_f32(d["k"])
    u = q.mean(axis=2, keepdims=True)
    u /= np.linalg.norm(u, axis=-1, keepdims=True)
    q = q + 8.0 * u
    step = (np.arange(w.seq_len) % 176 >= jump).astype(np.float32)[None, None, :, None]
    k = k + step * u * (60.0 * np.sqrt(128.0) / 8.0)
    qb, kb = synth.f32_to_bf16_bits(q.astype(np.float32)), synth.f32_to_bf16_bits(k.astype(np.float32))
    f = md.Filter(cfg(w, flags=flags, debug_score_variant=md.MUSTDROP_DEBUG_VARIANT_FUSED, debug_cluster=2))
    assert "176 keys per CTA" in f.description
    f.score(to_dev_bf16(qb), to_dev_bf16(kb))
    torch.cuda.synchronize()
    assert f.device_status() == (0, 0)
    G, I = (oracle.score_per_head if flags else oracle.score)(qb, kb, w.vis_start, w.n_vis, w.txt_start)
    g, i = f.g.cpu().numpy(), f.i.cpu().numpy()
    big = G > 1e-9
    assert big.sum() > 10
    assert_scores_close(g[big], G[big], "G")
    assert_scores_close(i[big], I[big], "I")
    f.close()
