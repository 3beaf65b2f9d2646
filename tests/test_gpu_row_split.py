"""Text rows scored by two launches: the second starts while the first one drains, on inputs that kernels
of the same stream have just written."""
import pytest
import torch

from paper_2411_10803_b200 import binding as md
from paper_2411_10803_b200 import build as md_build

from parity_util import cfg
from test_gpu_parity import small

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    md_build.build()


def bits(t):
    return t.contiguous().view(torch.uint8)


@pytest.mark.parametrize("cluster", [3, 8])
def test_two_layers_on_inputs_rewritten_in_the_stream(cluster):
    """Two pruning layers, each in two launches over the text rows with several rounds of clusters; the second
    layer reads the rebuilt keys and the counts of the first.  Queries, keys and counts are rewritten by
    kernels of the stream before every pass and nothing synchronises in between: every pass gives the bits of
    the same pass with a synchronisation after each call."""
    w = small(batch=90, n_vis=300, n_txt=80, n_heads=3, hidden=384, key_cnt=0, budget=130, vis_start=2)
    force = dict(debug_score_variant=md.MUSTDROP_DEBUG_VARIANT_ROW_SPLIT, debug_cluster=cluster, flags=md.MUSTDROP_FLAG_REBUILD_SEQUENCE)
    w2 = w.with_(n_vis=130, budget=50)
    first, second = md.Filter(cfg(w, **force)), md.Filter(cfg(w2, **force))
    for f in (first, second):
        assert "two launches" in f.description and f.filter_launches == 2
    gen = torch.Generator(device="cuda").manual_seed(8)

    def rand(*shape):
        return torch.randn(shape, generator=gen, device="cuda").to(torch.bfloat16)

    B, H, N = w.batch, w.n_heads, w.n_txt
    pool = [dict(q=rand(B, H, N, 128), k=rand(B, H, w.seq_len, 128), v=rand(B, H, w.seq_len, 128), hidden=rand(B, w.seq_len, w.hidden),
                 cnt=torch.randint(150, w.n_vis + 1, (B,), generator=gen, device="cuda").to(torch.int32)) for _ in range(3)]
    x = {n: torch.empty_like(t) for n, t in pool[0].items()}
    results = [(f, n) for f in (first, second) for n in ("g", "i", "kept_idx", "kept_cnt", "orig_out", "hidden_out", "k_out", "v_out")]

    def one_pass(n, wait):
        for f, name in results:
            bits(getattr(f, name)).fill_(0xFF if name in ("g", "i") else 0)
        for name, t in x.items():
            t.copy_(pool[n % 3][name])
        wait()
        first.filter_layer(x["q"], x["k"], x["v"], x["hidden"], vis_cnt=x["cnt"])
        wait()
        # (the keys, the caches and the counts that the launches just before have written)
        second.filter_layer(x["q"], first.k_out, first.v_out, first.hidden_out, vis_cnt=first.kept_cnt, orig_idx=first.orig_out)
        wait()

    want = []
    for n in range(3):
        one_pass(n, torch.cuda.synchronize)
        want.append([bits(getattr(f, name)).clone() for f, name in results])
    wrong = torch.zeros((), dtype=torch.int64, device="cuda")
    for n in range(60):
        one_pass(n, lambda: None)
        for (f, name), t in zip(results, want[n % 3]):
            wrong += (bits(getattr(f, name)) != t).sum()
    assert int(wrong) == 0
    for f in (first, second):
        assert f.device_status() == (0, 0)
        f.close()


def test_a_chain_of_score_calls_on_keys_rewritten_in_the_stream():
    """The score call alone in two launches, many in a row: each on the keys that a copy kernel just wrote."""
    w = small(batch=60, n_vis=500, n_txt=100, n_heads=2, hidden=256, key_cnt=0, budget=50, vis_start=0)
    f = md.Filter(cfg(w, debug_score_variant=md.MUSTDROP_DEBUG_VARIANT_ROW_SPLIT, debug_cluster=8))
    assert "two launches" in f.description
    gen = torch.Generator(device="cuda").manual_seed(9)
    pool = [(torch.randn((w.batch, w.n_heads, w.n_txt, 128), generator=gen, device="cuda").to(torch.bfloat16),
             torch.randn((w.batch, w.n_heads, w.seq_len, 128), generator=gen, device="cuda").to(torch.bfloat16)) for _ in range(2)]
    q, k = (torch.empty_like(t) for t in pool[0])
    want = []
    for a, b in pool:
        f.score(a, b)
        torch.cuda.synchronize()
        want.append((f.g.clone(), f.i.clone()))
    wrong = torch.zeros((), dtype=torch.int64, device="cuda")
    for n in range(100):
        q.copy_(pool[n % 2][0])
        k.copy_(pool[n % 2][1])
        f.score(q, k)
        wrong += (f.g != want[n % 2][0]).sum() + (f.i != want[n % 2][1]).sum()
    assert int(wrong) == 0 and f.device_status() == (0, 0)
    f.close()
