"""zipvl_select at the edges of its dispatch (one CTA up to 4096 tokens, a cluster of eight with 4, 8 or 16
positions per thread up to 65536, the multi-CTA kernel beyond), for spread, tied and nearly equal scores,
single rows and batches, with and without the kept-mass output and the keep-last option."""
import numpy as np
import pytest
import torch

import oracle
from parity import check_select

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def scores(L, kind, g):
    if kind == "spread":
        return torch.rand(L, generator=g) ** 6
    if kind == "ties":
        return torch.randint(1, 9, (L,), generator=g).float() * 0.25
    if kind == "equal":
        return torch.full((L,), 0.5)
    return 1.0 + 2e-5 * torch.rand(L, generator=g)      # thousands of tokens in one bin of the first level


@pytest.mark.parametrize("L", [4096, 4097, 5003, 16384, 16385, 32769, 65536, 65537])
@pytest.mark.parametrize("kind", ["spread", "ties", "equal", "near"])
def test_select_sizes(zipvl, L, kind):
    g = torch.Generator().manual_seed(L)
    acc = scores(L, kind, g)
    norm = acc / torch.arange(L, 0, -1).float().clamp(max=64)
    a, n = acc.to(DEV), norm.to(DEV)
    a64, n64 = acc.double().numpy(), norm.double().numpy()
    kept = torch.zeros(1, device=DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    for tau, fk, last in ((0.95, 0, 0), (0.4, 0, 7), (1.0, 0, 0), (0.5, L // 3, 0)):
        k_dev, idx = zipvl.zipvl_select(a, n, tau, fixed_k=fk, mode=zipvl.keep_last(last), kept_mass=kept, status=st)
        k = int(k_dev.item())
        check_select(k, idx.cpu().numpy(), a64, n64, tau, fixed_k=fk, keep_last=last)
        T = idx[:k].cpu().numpy()
        assert abs(kept.item() - a64[T].sum() / a64.sum()) < 1e-5
    assert st.item() == 0


def test_select_batch_of_cluster_rows(zipvl):
    g = torch.Generator().manual_seed(3)
    L, B = 6001, 5                                      # (odd: the rows are not 16-byte aligned)
    acc = torch.stack([scores(L, k, g) for k in ("spread", "ties", "near", "equal", "spread")])
    norm = acc / torch.arange(L, 0, -1).float().clamp(max=64)
    k_dev, idx = zipvl.zipvl_select_batch(acc.to(DEV), norm.to(DEV), 0.9)
    for z in range(B):
        check_select(int(k_dev[z].item()), idx[z].cpu().numpy(), acc[z].double().numpy(), norm[z].double().numpy(), 0.9)
        one_k, one = zipvl.zipvl_select(acc[z].to(DEV), norm[z].to(DEV), 0.9)
        assert torch.equal(one, idx[z]) and one_k.item() == k_dev[z].item()
