"""Infinities and NaN stay where they belong: a value reaches the outputs of the rows that see it, with its sign, and no
others."""
import numpy as np
import pytest
import torch

import oracle
from parity import to_np

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
CODE = {torch.bfloat16: 0, torch.float32: 1, torch.float16: 2}


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16, torch.float32])
@pytest.mark.parametrize("H,Hkv,d", [(2, 2, 128), (2, 2, 64), (3, 3, 96), (6, 2, 128), (12, 1, 96), (34, 2, 64)])
@pytest.mark.parametrize("L,row", [(37, 36), (37, 3), (64, 63), (1, 0), (129, 120)])
def test_infinite_value_in_a_cache(zipvl, dtype, H, Hkv, d, L, row):
    """In the last row of a cache that ends inside a tile, in full tiles and in the middle."""
    if dtype == torch.float32 and H // Hkv > 8:
        pytest.skip("fp32 takes up to 8 query heads per kv head")
    z = zipvl
    g = torch.Generator().manual_seed(L + row + H)
    q = torch.randn(1, H, d, generator=g).to(dtype)
    k, v = (torch.randn(L, Hkv, d, generator=g).to(dtype) for _ in range(2))
    clean = v.clone()
    v[row, :, 5], v[row, 0, 7] = float("inf"), -float("inf")
    n = torch.tensor([L], dtype=torch.int32, device=DEV)
    desc = z.zipvl_decode_desc(1, H, Hkv, d, CODE[dtype], 0.0)
    off = torch.zeros(1, dtype=torch.int64, device=DEV)
    run = lambda values: to_np(z.zipvl_decode(desc, q.to(DEV), None, None, k.to(DEV), values.to(DEV), off, n, n.clone(), L))[0]
    got, want = run(v), run(clean)
    want[:, 5], want[:H // Hkv, 7] = np.inf, -np.inf
    assert np.array_equal(got, want)


@pytest.mark.parametrize("d", [64, 96, 128])
@pytest.mark.parametrize("n,row", [(40, 32), (150, 96), (64, 48), (200, 176), (1000, 720)])
def test_infinite_value_in_a_prompt_fp32(zipvl, d, n, row):
    """Rows in front of the token do not see its value: their outputs are the bits they are without it.  (Rows that
    share its group of sixteen may meet it with weight zero; row is the first of one.)"""
    z, H = zipvl, 2
    g = torch.Generator().manual_seed(n + d)
    q, k, v = (torch.randn(n, H, d, generator=g).to(DEV) for _ in range(3))
    idx, count = torch.arange(n, dtype=torch.int32, device=DEV), torch.tensor([n], dtype=torch.int32, device=DEV)
    lay = z.layer_desc(q, k)
    want = z.zipvl_sparse_prefill(lay, q, k, v, idx, count, n).cpu()
    bad = v.clone()
    bad[row, :, 3] = float("inf")
    got = z.zipvl_sparse_prefill(lay, q, k, bad, idx, count, n).cpu()
    want[row:, :, 3] = float("inf")
    assert torch.equal(got, want)
