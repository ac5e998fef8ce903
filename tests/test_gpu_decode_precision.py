"""Precision of the decode steps behind the rounding of their outputs to 16 bits: inputs whose exact result is zero, so
that what comes out is the error of the kernel's own arithmetic.

Bounds.  A tensor core adds with 24 bits and cuts off: an MMA loses up to 2^-23 of the sum it leaves, 2^-24 on
average, towards zero.  Where a chain of MMAs adds zero-mean terms of deviation sigma over r rows, the sum grows to sigma sqrt(r),
and r / 16 MMAs lose about 2^-24 sigma sqrt(r) r / 16; divided by the r equal weights of the rows that is
2^-24 sigma sqrt(r) / 16 of a weight.  Scores: each of the D / 16 MMAs of a score loses up to 2^-23 of the
largest partial sum of the row."""
import numpy as np
import pytest
import torch

import oracle
from parity import to_np

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
CODE = {torch.bfloat16: 0, torch.float16: 2}


def quantised_step(z, k, v, q, n_hi, dtype):
    L, H, d = k.shape
    idx = torch.full((L,), -1, dtype=torch.int32, device=DEV)
    idx[:n_hi] = torch.arange(n_hi, dtype=torch.int32)
    cache = z.QuantCache(L, H, d, dtype, DEV, cap_hi=n_hi + 1, cap_lo=L - n_hi + 1)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    z.zipvl_quantize_kv(z.layer_desc(k, k), k.to(DEV), v.to(DEV), idx, torch.tensor([n_hi], dtype=torch.int32, device=DEV), L,
                        cache, status=st)
    desc = z.zipvl_decode_desc(1, q.shape[1], H, d, CODE[dtype], 0.0)
    out = to_np(z.zipvl_decode_quant(desc, q.to(DEV), None, None, cache, L, status=st))
    assert st.item() == 0
    return out[0]


def levels(shape, bits, g):
    """Odd whole numbers -(2^bits - 1) .. 2^bits - 1, both ends in every row: the quantiser's own grid (step 2)."""
    x = 2.0 * torch.randint(0, 1 << bits, shape, generator=g) - ((1 << bits) - 1)
    x[..., 0], x[..., 1] = (1 << bits) - 1, 1 - (1 << bits)
    return x


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
@pytest.mark.parametrize("d,G", [(128, 1), (64, 1), (128, 4)])
@pytest.mark.parametrize("bits", [4, 2])
def test_quantised_values_that_cancel(zipvl, dtype, d, G, bits):
    """Pairs of rows with one key and values v and -v: the exact output is zero."""
    H, n = 8, 2000
    g = torch.Generator().manual_seed(d + bits)
    k = torch.randn(n // 2, H, d, generator=g).repeat_interleave(2, 0).to(dtype)
    v = levels((n // 2, H, d), bits, g).repeat_interleave(2, 0)
    v[1::2] *= -1
    q = (0.1 * torch.randn(1, H * G, d, generator=g)).to(dtype)
    out = quantised_step(zipvl, k, v.to(dtype), q, n if bits == 4 else 0, dtype)
    sigma = np.sqrt((4.0 ** bits - 1) / 3)               # of the levels; no chain is longer than 512 rows
    assert np.sqrt(np.mean(out.astype(np.float64) ** 2)) < 2.0 ** -24 * sigma * np.sqrt(512) / 16


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
@pytest.mark.parametrize("d", [128, 64])
@pytest.mark.parametrize("bits", [4, 2])
def test_quantised_scores_that_agree(zipvl, dtype, d, bits):
    """Two rows whose keys are each other's mirror image over the channels, under a query that is its own: equal
    scores, values +1 and -1, an exact output of zero."""
    H = 64
    g = torch.Generator().manual_seed(3 * d + bits)
    k = levels((1, H, d), bits, g).to(dtype)
    k[..., -2:] = k[..., :2].flip(-1)                    # (both ends mirrored too)
    half = torch.randn(1, H, d // 2, generator=g)
    q = torch.cat([half, half.flip(-1)], -1).to(dtype)
    v = torch.ones(2, H, d, dtype=dtype)
    v[1] = -1
    out = quantised_step(zipvl, torch.cat([k, k.flip(-1)]), v, q, 2 if bits == 4 else 0, dtype)
    # partial sums of a score, in units of its exponent: centred codes times queries
    terms = to_np(q)[0].astype(np.float64) * to_np(k)[0] / np.sqrt(d) * np.log2(np.e)
    partial = np.abs(np.cumsum(terms, -1)).max(-1)
    # weights 2^s / (2^s + 2^s'): half the difference of the two scores, each off by D / 16 losses
    bound = np.log(2) * (d / 16) * 2.0 ** -24 * partial
    err = np.abs(out.astype(np.float64)).max(-1)
    assert np.sqrt(np.mean(err ** 2)) < np.sqrt(np.mean(bound ** 2))


def plain_step(z, q, k, v, dtype):
    """q [B, H, d] over caches k, v [B, L, H, d]; also the exact result."""
    B, L, H, d = k.shape
    off = torch.arange(B) * L * H * d
    n = torch.full((B,), L, dtype=torch.int32)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    desc = z.zipvl_decode_desc(B, H, H, d, CODE[dtype], 0.0)
    out = z.zipvl_decode(desc, q.to(DEV), None, None, k.to(DEV), v.to(DEV), off.to(DEV), n.to(DEV), n.to(DEV), L, status=st)
    assert st.item() == 0
    want = oracle.decode_step(to_np(q), None, None, to_np(k).ravel().copy(), to_np(v).ravel().copy(), off.numpy(), n.numpy().copy(), H)
    return to_np(out), want


@pytest.mark.parametrize("dtype,bits", [(torch.bfloat16, 8), (torch.float16, 11)])
@pytest.mark.parametrize("d", [64, 96, 128])
def test_small_weights_count(zipvl, dtype, bits, d):
    """Every sixteenth row has 2^26 times the weight of the others and a value of zero: the output is what the small
    weights add up to.  Bound: the output's rounding, and four units of the last of 24 bits."""
    L, H = 700, 3
    q = torch.ones(1, H, d, dtype=dtype)
    k = torch.zeros(1, L, H, d, dtype=dtype)
    v = torch.full((1, L, H, d), 30000.0).to(dtype)
    k[:, ::16] = 26 * np.log(2) / np.sqrt(d)
    v[:, ::16] = 0
    out, want = plain_step(zipvl, q, k, v, dtype)
    assert np.abs(out / want - 1).max() < 2.0 ** -bits + 4 * 2.0 ** -24 * 26


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
def test_sums_that_grow_and_cancel(zipvl, dtype):
    """The second half of a cache repeats the first with the values negated: sums over a warp's rows grow to half a value's
    size and go back to zero.  Rounded sums over its sixteen tiles are off by 2^-25 of that each, at random."""
    B, L, H, d = 16, 1024, 32, 128
    g = torch.Generator().manual_seed(5)
    k = torch.randn(B, L // 2, H, d, generator=g).repeat(1, 2, 1, 1).to(dtype)
    v = (1 + 0.1 * torch.randn(B, L // 2, H, d, generator=g)).to(dtype)
    q = (0.1 * torch.randn(B, H, d, generator=g)).to(dtype)
    out, _ = plain_step(zipvl, q, k, torch.cat([v, -v], 1), dtype)
    assert np.sqrt(np.mean(out.astype(np.float64) ** 2)) < np.sqrt(16) * 2.0 ** -25 * 0.5
