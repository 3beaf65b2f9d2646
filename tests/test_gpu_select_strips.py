"""The selection at the sizes where its strips, its digits and its direct ranking change over, stand-alone
and inside the one-launch filter, against the CPU oracle (bit-exact on the same scores)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2411_10803_b200 import binding as md
from paper_2411_10803_b200 import build as md_build
from paper_2411_10803_b200 import synth

from parity_util import cfg, to_dev, to_dev_bf16
from test_gpu_parity import small

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    md_build.build()


def scores(kind, B, M, rng):
    if kind == "spread":            # decades apart: digits start at a high bit
        g = np.exp(rng.normal(0, 8, (B, M)))
    elif kind == "bulk":            # many tokens in one bin: further digits, then direct ranking
        g = 1.0 + 1e-4 * rng.random((B, M))
    elif kind == "ties":            # more equal scores than are ranked directly: the lowest indices win
        g = rng.integers(1, 4, (B, M)).astype(np.float64)
    else:                           # zeros and subnormals leave the quick division
        g = np.where(rng.random((B, M)) < 0.3, 0.0, np.exp(rng.normal(-95, 4, (B, M))))
    i = g * rng.choice([0.01, 0.5, 3.0], (B, M)) if kind != "ties" else g.copy()
    return g.astype(np.float32), i.astype(np.float32)


@pytest.mark.parametrize("M", [1, 31, 256, 257, 1023, 1024, 1025, 2049, 4096])
@pytest.mark.parametrize("kind", ["spread", "bulk", "ties", "tiny"])
def test_select_is_bit_exact_at_the_change_overs(M, kind):
    B, L, key_max = 2, M + 9, min(5, M)
    rng = np.random.default_rng(M)
    G, I = scores(kind, B, M, rng)
    key_idx = np.stack([np.sort(rng.choice(M, key_max, replace=False)) for _ in range(B)]).astype(np.int32)
    key_cnt = np.array([key_max, 0], np.int32)
    for budget in sorted({key_max, max(key_max, M // 7), max(key_max, M // 2), M}):
        ref_idx, ref_cnt, ref_s, _ = oracle.select(G, I, L, key_idx, key_cnt, budget=budget)
        w = small(batch=B, n_vis=M, n_txt=9, n_heads=1, hidden=128, key_cnt=key_max, budget=budget, vis_start=0)
        f = md.Filter(cfg(w))
        f.select(to_dev(key_idx), to_dev(key_cnt), g=to_dev(G), i=to_dev(I))
        torch.cuda.synchronize()
        cnt = f.kept_cnt.cpu().numpy()
        assert np.array_equal(cnt, ref_cnt)
        assert np.array_equal(f.s.cpu().numpy().view(np.uint32), ref_s.view(np.uint32))
        for b in range(B):
            assert np.array_equal(f.kept_idx.cpu().numpy()[b, :cnt[b]], ref_idx[b, :cnt[b]])
        f.close()


@pytest.mark.parametrize("M,variant", [(1000, 0), (1100, 0), (1100, md.MUSTDROP_DEBUG_VARIANT_GRID),
                                       (3000, md.MUSTDROP_DEBUG_VARIANT_GRID)])
def test_filter_selects_what_the_stand_alone_selection_does(M, variant):
    w = small(batch=2, n_vis=M, n_txt=20, n_heads=2, hidden=256, key_cnt=9, budget=M // 5, vis_start=3)
    d = synth.make_batch(w)
    q, k, v, hid = (to_dev_bf16(d[n]) for n in ("q_text", "k", "v", "hidden"))
    ki, kc = to_dev(d["key_idx"]), to_dev(d["key_cnt"])
    f = md.Filter(cfg(w, debug_score_variant=variant))
    assert f.filter_launches == 1
    f.filter(q, k, v, hid, ki, kc, want_s=True)
    one = [t.clone() for t in (f.kept_idx, f.kept_cnt, f.s)]
    f.select(ki, kc)
    torch.cuda.synchronize()
    assert f.device_status() == (0, 0)
    for a, b in zip(one, (f.kept_idx, f.kept_cnt, f.s)):
        assert torch.equal(a, b)
    f.close()
