"""The fp32 kernels at the edges of their tiles and of their dispatch: 64-key score tiles (one, two or
four per CTA, and the two-sweep kernels behind them), 64-row query tiles shared by clusters of one to
eight CTAs, grouped heads, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2410_08584_b200 import workloads as W
from parity import check_attention, check_scores, to_np

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("L,Hq,Hkv,d,probes", [(1, 2, 2, 64, 1), (65, 2, 1, 128, 33), (512, 3, 3, 64, 64),
                                               (513, 2, 2, 96, 64), (1025, 4, 4, 128, 100), (2048, 2, 2, 64, 128),
                                               (2049, 2, 1, 64, 64), (700, 40, 8, 64, 64)])
def test_fp32_score_prefill_and_compaction(zipvl, L, Hq, Hkv, d, probes):
    g = torch.Generator().manual_seed(L)
    q, k, v = (torch.randn(L, h, d, generator=g) for h in (Hq, Hkv, Hkv))
    k[::7] *= 3
    probe = W.probe_positions(L, n_recent=probes // 2, n_random=probes - probes // 2, gen=g)
    desc = zipvl.layer_desc(q, k)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    qd, kd, vd = q.to(DEV), k.to(DEV), v.to(DEV)
    acc, norm = zipvl.zipvl_score(desc, qd, kd, probe.to(DEV), status=st)
    acc_ref, S = oracle.probe_scores(to_np(q), to_np(k), probe.numpy())
    norm_ref, _ = oracle.normalise(acc_ref, probe.numpy(), Hq)
    check_scores(acc.cpu().numpy(), norm.cpu().numpy(), acc_ref, norm_ref, S)

    T = torch.sort(torch.randperm(L, generator=g)[:max(1, L - L // 5)]).values
    n = len(T)
    idx = torch.full((L,), -1, dtype=torch.int32)
    idx[:n] = T.to(torch.int32)
    kc, vc = torch.zeros_like(kd), torch.zeros_like(vd)
    out, length = zipvl.zipvl_sparse_prefill_compact(desc, qd, kd, vd, idx.to(DEV),
                                                     torch.tensor([n], dtype=torch.int32, device=DEV), L, kc, vc, L,
                                                     out=torch.full_like(qd, float("nan")), status=st)
    torch.cuda.synchronize()
    assert st.item() == 0 and length.item() == n
    ref = oracle.sparse_prefill(to_np(q), to_np(k), to_np(v), T.numpy())
    check_attention(to_np(out.cpu()[T]), ref, torch.float32)
    dropped = torch.ones(L, dtype=torch.bool)
    dropped[T] = False
    assert not out.cpu()[dropped].abs().sum().item()
    assert torch.equal(kc.cpu()[:n], k[T]) and torch.equal(vc.cpu()[:n], v[T])
    assert not kc.cpu()[n:].abs().sum().item()
