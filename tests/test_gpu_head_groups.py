"""Plans that deal a request's heads out over groups of CTAs (one cluster per request, the groups'
head sums added through distributed shared memory at the end) against the CPU oracle."""
import re

import pytest
import torch

import oracle
from paper_2411_10803_b200 import binding as md
from paper_2411_10803_b200 import build as md_build
from paper_2411_10803_b200 import synth

from parity_util import assert_scores_close, cfg, to_dev_bf16
from test_gpu_parity import run_chain_and_check, small

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    md_build.build()


def groups_of(w, **kw):
    f = md.Filter(cfg(w, **kw))
    m = re.search(r"(\d+) head group", f.description)
    f.close()
    return int(m.group(1)) if m else 0


# heads that the groups do not divide, one head per group, 65 .. 128 text rows (one key range on all
# lanes), keys that end inside the last CTA's tile, one CTA per group, a share of the keys of zero columns
SHAPES = [dict(batch=1, n_vis=333, n_txt=21, n_heads=7, hidden=896, vis_start=2),
          dict(batch=2, n_vis=500, n_txt=64, n_heads=13, hidden=1664, vis_start=0),
          dict(batch=3, n_vis=290, n_txt=128, n_heads=9, hidden=1152, vis_start=1),
          dict(batch=2, n_vis=17, n_txt=3, n_heads=16, hidden=2048, vis_start=0),
          dict(batch=9, n_vis=250, n_txt=33, n_heads=6, hidden=768, vis_start=5)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "B%d_M%d_N%d_H%d" % (s["batch"], s["n_vis"], s["n_txt"], s["n_heads"]))
@pytest.mark.parametrize("path", ["filter", "staged"])
def test_head_groups_match_oracle(shape, path):
    w = small(key_cnt=min(9, shape["n_vis"] // 4), budget=max(5, shape["n_vis"] // 6), **shape)
    assert groups_of(w) > 1
    run_chain_and_check(w, path=path)


@pytest.mark.parametrize("shape", SHAPES[:3], ids=lambda s: "B%d_N%d" % (s["batch"], s["n_txt"]))
def test_head_groups_with_per_head_maxima(shape):
    w = small(key_cnt=0, budget=20, **shape)
    assert groups_of(w, flags=md.MUSTDROP_FLAG_PER_HEAD_MAX) > 1
    d = synth.make_batch(w)
    f = md.Filter(cfg(w, flags=md.MUSTDROP_FLAG_PER_HEAD_MAX))
    f.score(to_dev_bf16(d["q_text"]), to_dev_bf16(d["k"]))
    torch.cuda.synchronize()
    assert f.device_status() == (0, 0)
    G, I = oracle.score_per_head(d["q_text"], d["k"], w.vis_start, w.n_vis, w.txt_start)
    assert_scores_close(f.g.cpu().numpy(), G, "G")
    assert_scores_close(f.i.cpu().numpy(), I, "I")
    f.close()
