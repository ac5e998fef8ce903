"""Decode over mixed-precision caches at the ends of their chunks: blocks of whole chunks, one row more and less, an appended row
that opens a chunk, an empty block, lengths beyond max_len, requests of different lengths in one call."""
import numpy as np
import pytest
import torch

import oracle
from parity import check_attention, to_np

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def cache_of(z, n_hi, n_lo, Hkv, d, dtype, g):
    L = n_hi + n_lo
    k, v = (torch.randn(L, Hkv, d, generator=g).to(dtype) for _ in range(2))
    T = torch.sort(torch.randperm(L, generator=g)[:n_hi]).values
    idx = torch.full((L,), -1, dtype=torch.int32)
    idx[:n_hi] = T.to(torch.int32)
    c = z.QuantCache(L, Hkv, d, dtype, DEV, cap_hi=n_hi + 3, cap_lo=n_lo + 1)
    z.zipvl_quantize_kv(z.layer_desc(k, k), k.to(DEV), v.to(DEV), idx.to(DEV), torch.tensor([n_hi], dtype=torch.int32, device=DEV), L, c)
    return c, oracle.quantize_kv(to_np(k), to_np(v), T.numpy(), "f16" if dtype == torch.float16 else "bf16")


@pytest.mark.parametrize("blocks", [[(31, 32), (32, 31), (64, 96), (95, 1)], [(0, 64), (64, 0), (1, 1), (700, 129)],
                                    [(2047, 33), (2048, 32), (2049, 31), (5, 2075)]])
@pytest.mark.parametrize("Hq,Hkv,d,dtype", [(2, 2, 128, torch.bfloat16), (8, 2, 64, torch.float16), (10, 5, 128, torch.bfloat16)])
def test_ends_of_chunks(zipvl, blocks, Hq, Hkv, d, dtype):
    z, B = zipvl, len(blocks)
    storage, code = ("f16", z.ZIPVL_F16) if dtype == torch.float16 else ("bf16", z.ZIPVL_BF16)
    g = torch.Generator().manual_seed(sum(blocks[0]) + Hq)
    caches, refs = zip(*[cache_of(z, hi, lo, Hkv, d, dtype, g) for hi, lo in blocks])
    table, desc = z.quant_cache_table(caches, DEV), z.zipvl_decode_desc(B, Hq, Hkv, d, code, 0.0)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    for _ in range(3):
        q = torch.randn(B, Hq, d, generator=g).to(dtype)
        kn, vn = (torch.randn(B, Hkv, d, generator=g).to(dtype) for _ in range(2))
        out = to_np(z.zipvl_decode_quant_batch(desc, q.to(DEV), kn.to(DEV), vn.to(DEV), table, max(map(sum, blocks)) + 3, status=st))
        for b in range(B):
            want = oracle.decode_step_quant(to_np(q[b:b + 1]), to_np(kn[b:b + 1]), to_np(vn[b:b + 1]), refs[b], Hkv, storage)
            check_attention(out[b:b + 1], want, dtype)
    assert st.item() == 0 and [c.lens.tolist() for c in caches] == [[hi + 3, lo] for hi, lo in blocks]


@pytest.mark.parametrize("max_len", [700, 320, 299, 64, 1])
def test_rows_beyond_max_len(zipvl, max_len):
    """320 rows at 4 bits, 200 at 2, and max_len below their number: the first rows count, the call reports it, the appended
    row is stored all the same."""
    z, H, d, dtype = zipvl, 2, 128, torch.bfloat16
    g = torch.Generator().manual_seed(max_len)
    c, ref = cache_of(z, 320, 200, H, d, dtype, g)
    short, _ = cache_of(z, 320, 200, H, d, dtype, torch.Generator().manual_seed(max_len))
    desc = z.zipvl_decode_desc(1, H, H, d, z.ZIPVL_BF16, 0.0)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    q, kn, vn = (torch.randn(1, H, d, generator=g).to(dtype).to(DEV) for _ in range(3))
    out = z.zipvl_decode_quant(desc, q, kn, vn, c, max_len, status=st)
    assert (st.item() == z.DEV_CAPACITY) == (max_len < 521) and c.lens.tolist() == [321, 200]
    # the same rows as a cache of their own
    st.zero_()
    z.zipvl_decode_quant(desc, q, kn, vn, short, 521, status=st)
    n_hi = min(321, max_len)
    short.lens.copy_(torch.tensor([n_hi, min(200, max_len - n_hi)], dtype=torch.int32))
    want = z.zipvl_decode_quant(desc, q, None, None, short, max(max_len, 521), status=st)
    check_attention(to_np(out), to_np(want).astype(np.float64), dtype)
    for m in ("k_hi", "v_hi", "p_hi"):
        assert torch.equal(getattr(c, m)[:321], getattr(short, m)[:321])
