"""Decode over grouped query heads at the edges of the kernel's head tiles (8, 16, 24 and 32 heads) and over single heads of 64
channels on either side of the lines between two kernels, on contiguous and paged caches, with appends, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from parity import check_attention, to_np

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
CODE = {torch.bfloat16: 0, torch.float32: 1, torch.float16: 2}


def check_steps(z, lens, Hq, Hkv, d, dtype, page, steps=2, seed=0):
    """Steps with an appended row each, on a paged cache (pages in random order) or a contiguous one."""
    g = torch.Generator().manual_seed(seed + Hq + d)
    B, row = len(lens), Hkv * d
    caps = [-(-(n + steps) // (page or 1)) * (page or 1) for n in lens]
    off = np.concatenate([[0], np.cumsum([c * row for c in caps[:-1]])]).astype(np.int64)
    kc, vc = (torch.randn(sum(caps) * row, generator=g).to(dtype) for _ in range(2))
    ko, vo, seqo = to_np(kc).copy(), to_np(vc).copy(), np.array(lens, np.int32)
    desc = z.zipvl_decode_desc(B, Hq, Hkv, d, CODE[dtype], 0.0)
    seq, cap = torch.tensor(lens, dtype=torch.int32, device=DEV), torch.tensor(caps, dtype=torch.int32, device=DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    if page:
        n_pages = sum(caps) // page
        where = torch.randperm(n_pages, generator=g)             # page i of the contiguous layout -> its place in the pool
        pools = []
        for c in (kc, vc):
            pool = torch.empty_like(c).view(n_pages, page, Hkv, d)
            pool[where] = c.view(n_pages, page, Hkv, d)
            pools.append(pool.to(DEV))
        table = torch.zeros(B, max(caps) // page, dtype=torch.int32)
        at = 0
        for b, c in enumerate(caps):
            table[b, :c // page] = where[at:at + c // page].to(torch.int32)
            at += c // page
        table = table.to(DEV)
    else:
        kd, vd, offd = kc.to(DEV), vc.to(DEV), torch.from_numpy(off).to(DEV)
    for _ in range(steps):
        q = torch.randn(B, Hq, d, generator=g).to(dtype)
        kn, vn = (torch.randn(B, Hkv, d, generator=g).to(dtype) for _ in range(2))
        if page:
            out = z.zipvl_decode_paged(desc, q.to(DEV), kn.to(DEV), vn.to(DEV), *pools, table, cap, seq, max(lens) + steps, status=st)
        else:
            out = z.zipvl_decode(desc, q.to(DEV), kn.to(DEV), vn.to(DEV), kd, vd, offd, cap, seq, max(lens) + steps, status=st)
        want = oracle.decode_step(to_np(q), to_np(kn), to_np(vn), ko, vo, off, seqo, Hkv)
        check_attention(to_np(out), want, dtype)
    assert st.item() == 0 and np.array_equal(seq.cpu().numpy(), seqo)


@pytest.mark.parametrize("G", [8, 9, 16, 17, 24, 25, 32])
@pytest.mark.parametrize("d,dtype", [(64, torch.float16), (96, torch.bfloat16), (128, torch.bfloat16)])
@pytest.mark.parametrize("page", [0, 16])
def test_heads_at_the_edges_of_the_tiles(zipvl, G, d, dtype, page):
    check_steps(zipvl, [15, 700, 63, 130], 2 * G, 2, d, dtype, page)


@pytest.mark.parametrize("G", [9, 17, 32])
def test_many_heads_on_more_than_a_wave(zipvl, G):
    """Chunks of 512 rows and more, lengths around their ends."""
    check_steps(zipvl, [509, 510, 511, 1021, 1022, 1023, 40, 0] * 5, 2 * G, 2, 64, torch.bfloat16, 0, steps=1)


@pytest.mark.parametrize("n,L,H", [(3, 1500, 16), (4, 1500, 16), (4, 1562, 16), (5, 1251, 16), (5, 1240, 16), (4, 63, 3), (7, 20, 1)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
@pytest.mark.parametrize("page", [0, 64])
def test_single_heads_of_64_channels(zipvl, n, L, H, dtype, page):
    """Either side of the lines between the two kernels: more than three requests, 100000 rows of heads, contiguous."""
    check_steps(zipvl, [L, 1, 17] + [max(0, L - 7 * i) for i in range(n - 3)], H, H, 64, dtype, page)


@pytest.mark.parametrize("G", [9, 17, 32])
@pytest.mark.parametrize("d,dtype", [(64, torch.float16), (96, torch.bfloat16), (128, torch.bfloat16)])
@pytest.mark.parametrize("page", [0, 16])
def test_rows_fetched_ahead(zipvl, G, d, dtype, page):
    """Chunks of 512 rows whose ends lie around the tiles that a step fetches for the step after the next."""
    check_steps(zipvl, [0, 127, 128, 129, 142, 143, 144, 145, 175, 192, 193, 511, 512, 513, 640, 641, 655] * 5, 2 * G, 2, d, dtype, page, steps=1)


@pytest.mark.parametrize("G", [9, 17, 32])
def test_page_outside_the_pool_ahead(zipvl, G):
    """Its rows are left out and reported, as the tile of a step and as one that a step fetches ahead."""
    z, B, L, d, page = zipvl, 80, 600, 64, 16
    g = torch.Generator().manual_seed(G)
    k, v = (torch.randn(L, 2, d, generator=g).to(torch.bfloat16) for _ in range(2))
    q = torch.randn(B, 2 * G, d, generator=g).to(torch.bfloat16)
    n = -(-L // page)
    pools = [torch.cat([c, c.new_zeros(n * page - L, 2, d)]).view(n, page, 2, d).to(DEV) for c in (k, v)]
    table = torch.arange(n, dtype=torch.int32).repeat(B, 1)
    gone = [8, 9, 20]
    table[:, gone] = torch.tensor([n, -1, n + 100000], dtype=torch.int32)
    seq = torch.full((B,), L, dtype=torch.int32, device=DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    desc = z.zipvl_decode_desc(B, 2 * G, 2, d, 0, 0.0)
    out = z.zipvl_decode_paged(desc, q.to(DEV), None, None, *pools, table.to(DEV), torch.full_like(seq, n * page), seq, L, status=st)
    rows = [r for r in range(L) if r // page not in gone]
    kept = [to_np(c)[rows].reshape(-1).copy() for c in (k, v)]
    want = oracle.decode_step(to_np(q), None, None, np.tile(kept[0], B), np.tile(kept[1], B),
                              np.arange(B, dtype=np.int64) * kept[0].size, np.full(B, len(rows), np.int32), 2)
    check_attention(to_np(out), want, torch.bfloat16)
    assert st.item() & z.DEV_BAD_INDEX
