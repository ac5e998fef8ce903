"""The tensor-core attention at the edges of its query tiles: a single tile, a pair, an odd tile out, one row into
the next tile, full diagonal tiles, at each head_dim, with the compaction inside, against the oracle."""
import pytest
import torch

import oracle
from parity import check_attention, to_np

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n,Hq,Hkv,d,dtype", [(1, 2, 2, 128, torch.bfloat16), (128, 2, 2, 128, torch.bfloat16),
                                              (129, 2, 1, 64, torch.float16), (256, 2, 2, 96, torch.bfloat16),
                                              (257, 2, 1, 128, torch.float16), (384, 2, 2, 64, torch.bfloat16),
                                              (512, 2, 2, 128, torch.float16), (897, 4, 2, 96, torch.float16)])
def test_attention_and_compaction_at_the_edges_of_the_tiles(zipvl, n, Hq, Hkv, d, dtype):
    L = n + n // 4
    g = torch.Generator().manual_seed(n)
    q, k, v = (torch.randn(L, h, d, generator=g).to(dtype) for h in (Hq, Hkv, Hkv))
    T = torch.sort(torch.randperm(L, generator=g)[:n]).values
    idx = torch.full((L,), -1, dtype=torch.int32)
    idx[:n] = T.to(torch.int32)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    qd, kd, vd = q.to(DEV), k.to(DEV), v.to(DEV)
    kc, vc = torch.zeros_like(kd), torch.zeros_like(vd)
    out, length = zipvl.zipvl_sparse_prefill_compact(zipvl.layer_desc(qd, kd), qd, kd, vd, idx.to(DEV),
                                                     torch.tensor([n], dtype=torch.int32, device=DEV), L, kc, vc, L,
                                                     out=torch.full_like(qd, float("nan")), status=st)
    torch.cuda.synchronize()
    assert st.item() == 0 and length.item() == n
    ref = oracle.sparse_prefill(to_np(q), to_np(k), to_np(v), T.numpy())
    check_attention(to_np(out.cpu()[T]), ref, dtype)
    dropped = torch.ones(L, dtype=torch.bool)
    dropped[T] = False
    assert not out.cpu()[dropped].abs().sum().item()
    assert torch.equal(kc.cpu()[:n], k[T]) and torch.equal(vc.cpu()[:n], v[T])
