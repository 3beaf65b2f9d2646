"""The vision-encoding kernels at the sizes where their shares, tiles and radix passes change over, against
the numpy oracle: odd channel counts and grids, tokens that the CTAs do not divide, more heads than fit a
CTA's shared memory at a time, values that share all but their lowest bits."""
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


@pytest.mark.parametrize("B,grid,C", [(1, 2, 8), (2, 4, 1032), (3, 10, 264), (2, 46, 40), (1, 24, 2056)])
def test_spatial_merge_shapes(B, grid, C):
    bits = synth.make_vit_tokens(19, B, grid, C, merge_frac=0.4)
    n = grid * grid
    merged = torch.zeros((B, n, C), dtype=torch.bfloat16, device="cuda")
    slots = torch.full((B, n), -1, dtype=torch.int32, device="cuda")
    cnt = torch.zeros((B,), dtype=torch.int32, device="cuda")
    sims = torch.zeros((B, (grid // 2) ** 2), dtype=torch.float32, device="cuda")
    assert md.mustdrop_spatial_merge(B, grid, 2, C, 0.8, to_dev_bf16(bits), merged, slots, cnt, sims) == md.MUSTDROP_OK
    torch.cuda.synchronize()
    got = synth.bf16_bits_to_f64(bf16_bits(merged))
    x = synth.bf16_bits_to_f64(bits)
    for b in range(B):
        rows, ref_slots, ref_sims = context.local_spatial_merge(x[b], grid, 2, 0.8, return_sims=True)
        assert np.all(np.abs(ref_sims - 0.8) > 1e-3)
        # fp32 sums of C products: C * 2^-24 relative at most
        assert np.allclose(sims.cpu().numpy()[b], ref_sims, rtol=0, atol=max(2e-6, C * 2.0 ** -24))
        m = int(cnt[b])
        assert m == len(ref_slots) and np.array_equal(slots.cpu().numpy()[b, :m], ref_slots)
        assert np.all(np.abs(got[b, :m] - rows) <= 2.0 ** -8 * np.abs(rows) + 1e-30)      # one rounding to bf16
        assert not got[b, m:].any()


@pytest.mark.parametrize("B,H,D,M", [(2, 1, 8, 1), (1, 3, 16, 7), (2, 5, 24, 63), (1, 12, 80, 577), (2, 64, 64, 130),
                                     (1, 40, 32, 4095), (1, 2, 248, 300)])
def test_key_set_shapes(B, H, D, M):
    qb, kb, _ = synth.make_cls_attention(5, B, H, D, M, min(M, 4))
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
        # quartiles and fence of the kernel's own fp32 values: order statistics are exact, the
        # interpolation rounds a handful of times
        ref_mu = context.upper_fence(got_a)
        assert abs(float(mu[b]) - ref_mu) <= 1e-6 * abs(ref_mu)
        n = int(kc[b])
        assert np.array_equal(ki.cpu().numpy()[b, :n], np.nonzero(got_a > mu.cpu().numpy()[b])[0])


@pytest.mark.parametrize("M", [64, 65, 300, 576, 3000])
def test_key_set_quartiles_among_equal_values(M):
    """Keys of three kinds only.  From 300 tokens on every order statistic sits in a run of equal values longer
    than the 64 that are ranked against each other, so all digits are resolved; 64 and 65 tokens have runs of
    about 21 and rank equal values."""
    B, H, D = 1, 2, 64
    rng = np.random.default_rng(M)
    q = rng.standard_normal((B, H, D)).astype(np.float32)
    kinds = np.stack([np.zeros(D), 0.02 * q[0, 0], 0.04 * q[0, 0]]).astype(np.float32)
    k = np.broadcast_to(kinds[rng.integers(0, 3, M)], (B, H, M, D))
    qb, kb = synth.f32_to_bf16_bits(q), synth.f32_to_bf16_bits(np.ascontiguousarray(k))
    a = torch.zeros((B, M), dtype=torch.float32, device="cuda")
    mu = torch.zeros((B,), dtype=torch.float32, device="cuda")
    ki = torch.full((B, M), -1, dtype=torch.int32, device="cuda")
    kc = torch.zeros((B,), dtype=torch.int32, device="cuda")
    assert md.mustdrop_key_set(B, H, D, M, M, to_dev_bf16(qb), to_dev_bf16(kb), a, mu, ki, kc) == md.MUSTDROP_OK
    torch.cuda.synchronize()
    got_a = a.cpu().numpy()[0]
    runs = np.unique(got_a, return_counts=True)[1]
    assert len(runs) == 3 and (runs.min() > 64) == (M >= 300)
    ref_mu = context.upper_fence(got_a)
    assert abs(float(mu[0]) - ref_mu) <= 1e-6 * ref_mu
