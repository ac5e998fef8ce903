"""Prompts with more query tiles than a grid dimension other than x holds (65535 of 64 rows)."""
import pytest
import torch

import oracle
from parity import check_attention, to_np

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_fp32_attention_of_more_than_four_million_tokens(zipvl):
    """A bound of 65537 tiles, of which the kept tokens (from the end of the prompt) fill two."""
    L, H, d, n = 65537 * 64, 1, 64, 100
    g = torch.Generator(device=DEV).manual_seed(3)
    q, k, v = (torch.randn(L, H, d, generator=g, device=DEV) for _ in range(3))
    T = torch.arange(L - n, L)
    idx = torch.full((L,), -1, dtype=torch.int32, device=DEV)
    idx[:n] = T.to(torch.int32).to(DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    out = torch.full((L, H, d), 7.0, device=DEV)
    zipvl.zipvl_sparse_prefill(zipvl.layer_desc(q, k), q, k, v, idx, torch.tensor([n], dtype=torch.int32, device=DEV), L, out=out,
                               out_mode=zipvl.OUT_COMPACT, status=st)
    assert st.item() == 0 and bool((out[n:n + 1000] == 7).all())
    qs, ks, vs = (to_np(t[L - n:].cpu()) for t in (q, k, v))
    check_attention(to_np(out[:n].cpu()), oracle.sparse_prefill(qs, ks, vs, torch.arange(n).numpy()), torch.float32)
