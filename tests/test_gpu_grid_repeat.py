"""Grid plans over many calls in a row: tiles whose keys end inside a warp, and a workspace that score calls
and filter calls share."""
import pytest
import torch

from paper_2411_10803_b200 import binding as md
from paper_2411_10803_b200 import build as md_build
from paper_2411_10803_b200 import synth

from parity_util import cfg, to_dev, to_dev_bf16
from test_gpu_parity import small

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    md_build.build()


def inputs(w, seed):
    d = synth.make_batch(w.with_(seed=seed))
    return [to_dev_bf16(d[n]) for n in ("q_text", "k", "v", "hidden")] + [to_dev(d["key_idx"]), to_dev(d["key_cnt"])]


@pytest.mark.parametrize("n_txt,ctas", [(74, 16), (40, 6), (64, 14)])
def test_many_grid_calls_in_a_row(n_txt, ctas):
    # 16 x 112 keys: the last of a tile's warps has keys for half of its lanes; 6 x 288, 14 x 128
    w = small(batch=9, n_vis=1631, n_txt=n_txt, n_heads=4, hidden=512, key_cnt=20, budget=200, vis_start=21)
    f = [md.Filter(cfg(w, debug_score_variant=md.MUSTDROP_DEBUG_VARIANT_GRID, debug_cluster=ctas)) for _ in range(2)]
    if "grid plan" not in f[0].description:
        pytest.skip("this split does not fit")
    x = [inputs(w, 5), inputs(w, 6)]
    for i in range(2):
        f[i].filter(*x[i])
    first = [[t.clone() for t in (y.g, y.i, y.kept_idx, y.k_out)] for y in f]
    for n in range(400):
        f[n % 2].filter(*x[n % 2])
    torch.cuda.synchronize()
    for y, want in zip(f, first):
        assert y.device_status() == (0, 0)
        for a, b in zip((y.g, y.i, y.kept_idx, y.k_out), want):
            assert torch.equal(a, b)
        y.close()


def test_score_and_filter_calls_share_a_grid_plan_s_workspace():
    w = small(batch=3, n_vis=700, n_txt=30, n_heads=3, hidden=384, key_cnt=5, budget=90, vis_start=0)
    force = dict(debug_score_variant=md.MUSTDROP_DEBUG_VARIANT_GRID, debug_cluster=6)
    f = md.Filter(cfg(w, **force))
    assert "grid plan" in f.description
    for n in range(1, 8):
        x = inputs(w, 100 + n)
        if n % 3 == 2:
            f.score(x[0], x[1])
            continue
        f.filter(*x)
        fresh = md.Filter(cfg(w, **force))
        fresh.filter(*x)
        torch.cuda.synchronize()
        assert f.device_status() == (0, 0)
        for a, b in ((f.g, fresh.g), (f.kept_idx, fresh.kept_idx), (f.hidden_out, fresh.hidden_out)):
            assert torch.equal(a, b)
        fresh.close()
    f.close()
