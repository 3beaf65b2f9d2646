"""The key set's reading of the keys at the head dimensions where the lanes that share a token's row, and the
vectors each of them reads, change over - and at token counts that end inside a trip, a unit and a CTA - and the
merge with numbers of CTAs per image that are no power of two, against the numpy oracle."""
import numpy as np
import pytest
import torch

from oracle import context
from paper_2411_10803_b200 import binding as md
from paper_2411_10803_b200 import build as md_build
from paper_2411_10803_b200 import synth

from parity_util import bf16_bits, to_dev_bf16

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    md_build.build()


# four lanes to a row with one, two and three vectors each, eight with two and four, whole and short rows, and a lane per
# vector: up to 16, and at 33 .. 64 where the batch fills the GPU (the last four)
@pytest.mark.parametrize("B,H,D,M", [(1, 2, 8, 33), (1, 2, 8, 700), (40, 2, 8, 100), (2, 3, 16, 577), (1, 2, 24, 400), (1, 2, 32, 200),
                                     (2, 3, 32, 640), (1, 2, 32, 641), (2, 3, 40, 130), (1, 2, 64, 64), (1, 2, 64, 1030), (2, 3, 72, 129),
                                     (1, 2, 88, 577), (1, 2, 96, 257), (1, 2, 104, 100), (2, 3, 128, 777), (1, 2, 136, 300),
                                     (2, 3, 192, 250), (1, 2, 248, 1031), (1, 1, 256, 70), (37, 2, 64, 272), (38, 1, 48, 300),
                                     (47, 2, 64, 256), (47, 1, 48, 300), (50, 2, 64, 330), (48, 1, 40, 577)])
def test_key_set_at_the_change_overs(B, H, D, M):
    qb, kb, _ = synth.make_cls_attention(7, B, H, D, M, min(M, 4))
    a = torch.zeros((B, M), dtype=torch.float32, device="cuda")
    mu = torch.zeros((B,), dtype=torch.float32, device="cuda")
    ki = torch.full((B, M), -1, dtype=torch.int32, device="cuda")
    kc = torch.zeros((B,), dtype=torch.int32, device="cuda")
    assert md.mustdrop_key_set(B, H, D, M, M, to_dev_bf16(qb), to_dev_bf16(kb), a, mu, ki, kc) == md.MUSTDROP_OK
    torch.cuda.synchronize()
    q, k = synth.bf16_bits_to_f64(qb), synth.bf16_bits_to_f64(kb)
    for b in range(B):
        _, ref_a = context.key_set(q[b], k[b])
        got_a = a.cpu().numpy()[b]
        assert np.allclose(got_a, ref_a, rtol=2e-5, atol=1e-12)          # fp32 dot products of D terms, exp2, M terms
        ref_mu = context.upper_fence(got_a)
        assert abs(float(mu[b]) - ref_mu) <= 1e-6 * abs(ref_mu)
        n = int(kc[b])
        assert np.array_equal(ki.cpu().numpy()[b, :n], np.nonzero(got_a > mu.cpu().numpy()[b])[0])


# on a B200, four, five and seven CTAs per image, three and six (the last three; with one vector of a token in flight at
# 16 channels, two at 264), vectors that end in the first and in the second of a lane's pair
@pytest.mark.parametrize("B,grid,C", [(3, 10, 512), (1, 12, 520), (2, 14, 776), (90, 24, 16), (111, 12, 264), (64, 24, 264)])
def test_spatial_merge_with_other_cluster_sizes(B, grid, C):
    bits = synth.make_vit_tokens(23, B, grid, C, merge_frac=0.4)
    n = grid * grid
    merged = torch.zeros((B, n, C), dtype=torch.bfloat16, device="cuda")
    slots = torch.full((B, n), -1, dtype=torch.int32, device="cuda")
    cnt = torch.zeros((B,), dtype=torch.int32, device="cuda")
    sims = torch.zeros((B, (grid // 2) ** 2), dtype=torch.float32, device="cuda")
    assert md.mustdrop_spatial_merge(B, grid, 2, C, 0.8, to_dev_bf16(bits), merged, slots, cnt, sims) == md.MUSTDROP_OK
    torch.cuda.synchronize()
    got, x = synth.bf16_bits_to_f64(bf16_bits(merged)), synth.bf16_bits_to_f64(bits)
    for b in range(B):
        rows, ref_slots, ref_sims = context.local_spatial_merge(x[b], grid, 2, 0.8, return_sims=True)
        assert np.allclose(sims.cpu().numpy()[b], ref_sims, rtol=0, atol=max(2e-6, C * 2.0 ** -24))   # fp32 sums of C products
        if np.any(np.abs(ref_sims - 0.8) <= 1e-3):
            continue                                                      # (a window too near the threshold decides either way)
        m = int(cnt[b])
        assert m == len(ref_slots) and np.array_equal(slots.cpu().numpy()[b, :m], ref_slots)
        assert np.all(np.abs(got[b, :m] - rows) <= 2.0 ** -8 * np.abs(rows) + 1e-30)      # one rounding to bf16
        assert not got[b, m:].any()
