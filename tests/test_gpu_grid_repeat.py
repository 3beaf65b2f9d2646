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


@pytest.mark.parametrize("n_vis,n_txt,ctas", [(1631, 40, 6), (2048, 96, 16)])
def test_every_call_of_a_grid_plan_selects_from_its_own_scores(n_vis, n_txt, ctas):
    # Inputs change with every call and every output holds NaN bits before it, so that a score read before
    # it is stored shows: each CTA of a request selects for itself, and copies rows of its own list.  The
    # list must be the one the stand-alone selection makes of the call's own scores, the rows those of the
    # list, the scores those of a cluster plan (other orders of fp32 sums: 1e-5).
    w = small(batch=9, n_vis=n_vis, n_txt=n_txt, n_heads=2, hidden=256, key_cnt=20, budget=200, vis_start=21)
    f = md.Filter(cfg(w, debug_score_variant=md.MUSTDROP_DEBUG_VARIANT_GRID, debug_cluster=ctas))
    assert "grid plan" in f.description
    select = md.Filter(cfg(w))
    x = [inputs(w, 40 + n) for n in range(5)]
    want = []
    for y in x:
        r = md.Filter(cfg(w, debug_score_variant=md.MUSTDROP_DEBUG_VARIANT_TWO_PASS))
        r.score(y[0], y[1])
        want.append((r.g.clone(), r.i.clone()))
        r.close()
    outs = (f.g, f.i, f.kept_idx, f.kept_cnt, f.hidden_out, f.k_out, f.v_out)
    rows = torch.arange(w.batch, device="cuda")[:, None]
    wrong = torch.zeros(4, dtype=torch.int64, device="cuda")
    for n in range(300):
        q, k, v, hid, key_idx, key_cnt = x[n % 5]
        for t in outs:
            t.view(torch.uint8).fill_(0xFF)
        f.filter(q, k, v, hid, key_idx, key_cnt)
        select.g.copy_(f.g)
        select.i.copy_(f.i)
        select.select(key_idx, key_cnt)
        at = w.vis_start + f.kept_idx.long().clamp(0, w.n_vis - 1)
        for e, (a, b) in enumerate(zip((f.g, f.i), want[n % 5])):
            wrong[e] += (~((a - b).abs() <= 1e-5 * b.abs() + 1e-12)).sum()
        wrong[2] += (f.kept_idx != select.kept_idx).sum() + (f.kept_cnt != select.kept_cnt).sum()
        wrong[3] += (f.hidden_out.view(torch.int16) != hid[rows, at].view(torch.int16)).sum()
        for src, out in ((k, f.k_out), (v, f.v_out)):
            wrong[3] += (out.transpose(1, 2).view(torch.int16) != src.transpose(1, 2)[rows, at].view(torch.int16)).sum()
    assert wrong.tolist() == [0, 0, 0, 0]
    assert f.device_status() == (0, 0)
    f.close()
    select.close()


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


@pytest.mark.parametrize("n_vis,n_txt,ctas", [(300, 21, 2), (333, 64, 7), (500, 65, 6), (700, 128, 6), (1000, 40, 4)])
def test_per_head_maxima_of_a_small_grid_plan_are_fp32(n_vis, n_txt, ctas):
    """Grid plans take small calls from the two-pass kernel, whose per-head maxima are fp32.  The two kernels'
    sums run in other orders: 1e-5 covers both (a maximum rounded to 11 bits is off by up to 5e-4)."""
    w = small(batch=2, n_vis=n_vis, n_txt=n_txt, n_heads=3, hidden=384, key_cnt=0, budget=50, vis_start=3)
    per_head = dict(flags=md.MUSTDROP_FLAG_PER_HEAD_MAX)
    x = inputs(w, 77)
    got = []
    for force in (dict(debug_score_variant=md.MUSTDROP_DEBUG_VARIANT_GRID, debug_cluster=ctas),
                  dict(debug_score_variant=md.MUSTDROP_DEBUG_VARIANT_TWO_PASS)):
        f = md.Filter(cfg(w, **per_head, **force))
        assert ("grid plan" in f.description) == (len(got) == 0)
        f.score(x[0], x[1])
        scored = f.i.clone()
        f.filter(*x)
        torch.cuda.synchronize()
        assert f.device_status() == (0, 0) and torch.equal(scored, f.i)
        got.append(scored)
        f.close()
    assert ((got[0] - got[1]).abs() <= 1e-5 * got[1].abs()).all()
