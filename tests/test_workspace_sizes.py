"""zipvl_workspace_bytes never falls as a problem grows, so that a workspace sized for the longest prompt, the most probes, the
largest batch and the longest cache serves every smaller call."""
import ctypes as C

import pytest
import torch

import paper_2410_08584_b200 as z
from paper_2410_08584_b200 import build as zbuild

HEADS = [(1, 1, 128), (4, 4, 64), (32, 32, 128), (28, 4, 128), (14, 2, 64), (12, 4, 96), (64, 2, 128), (40, 40, 128)]
LENGTHS = sorted(set(list(range(1, 700, 13)) + [b + e for b in (1024, 1200, 1409, 2048, 2416, 2944, 4096, 8191, 24577, 65536, 131072, 1 << 20)
                                                for e in (-129, -65, -1, 0, 1, 63, 64, 65, 128, 640)]))


@pytest.fixture(scope="module")
def lib():
    zbuild.build()
    return z.load()


@pytest.mark.parametrize("Hq,Hkv,d", HEADS)
@pytest.mark.parametrize("dtype", [z.ZIPVL_BF16, z.ZIPVL_F32])
def test_score_workspace_grows(lib, Hq, Hkv, d, dtype):
    def need(L, P, n):
        lay = z.zipvl_layer(L, Hq, Hkv, d, dtype, 0, 0, 0, 0.0, 0)
        b = lib.zipvl_workspace_bytes_batch(z.OP_SCORE, C.byref(lay), P, n)
        assert n > 1 or b == z.zipvl_workspace_bytes(z.OP_SCORE, lay, P)
        return b

    probes, batches = [1, 31, 32, 33, 64, 96, 97, 127, 128, 129, 200, 512, 8192], [1, 2, 3, 5, 8, 9, 10, 40, 300]
    for P in probes:
        for n in batches:
            sizes = [need(L, P, n) for L in LENGTHS]
            assert sizes == sorted(sizes)
    for L in LENGTHS[::7] + [2047, 2048, 2049]:
        for n in batches:
            sizes = [need(L, P, n) for P in probes]
            assert sizes == sorted(sizes)
        for P in probes:
            sizes = [need(L, P, n) for n in batches]
            assert sizes == sorted(sizes)


@pytest.mark.parametrize("Hq,Hkv,d", HEADS)
@pytest.mark.parametrize("dtype", [z.ZIPVL_BF16, z.ZIPVL_F32])
def test_decode_workspace_grows(lib, Hq, Hkv, d, dtype):
    def need(B, L):
        return z.zipvl_workspace_bytes(z.OP_DECODE, z.zipvl_layer(L, Hq, Hkv, d, dtype, 0, 0, 0, 0.0, 0), 0, B)

    batches = list(range(1, 40)) + [48, 63, 64, 65, 100, 148, 149, 256, 1000]
    for B in batches:
        sizes = [need(B, L) for L in LENGTHS]
        assert sizes == sorted(sizes)
    for L in LENGTHS:
        sizes = [need(B, L) for B in batches]
        assert sizes == sorted(sizes)


@pytest.mark.gpu
@pytest.mark.parametrize("Hq,Hkv,d,dtype", [(32, 32, 128, torch.bfloat16), (28, 4, 128, torch.float16), (4, 4, 64, torch.float32)])
def test_one_workspace_for_every_step(zipvl, Hq, Hkv, d, dtype):
    """A workspace for four requests of 2416 rows takes every smaller step (1200 rows of one request need more partial
    results than 2416), and each gives the bits of a workspace of its own."""
    B, most = 4, 2416
    code = {torch.bfloat16: z.ZIPVL_BF16, torch.float16: z.ZIPVL_F16, torch.float32: z.ZIPVL_F32}[dtype]
    g = torch.Generator().manual_seed(1)
    k, v = (torch.randn(B * most, Hkv, d, generator=g).to(dtype).cuda() for _ in range(2))
    size = lambda n, L: z.zipvl_workspace_bytes(z.OP_DECODE, z.zipvl_layer(L, Hq, Hkv, d, code, 0, 0, 0, 0.0, 0), 0, n)
    ws = z.workspace(size(B, most), "cuda")
    for n in (1, 2, 3, 4):
        desc = z.zipvl_decode_desc(n, Hq, Hkv, d, code, 0.0)
        q = torch.randn(n, Hq, d, generator=g).to(dtype).cuda()
        off = (torch.arange(n) * most * Hkv * d).cuda()
        for L in (1, 63, 64, 65, 300, 777, 1200, 1216, 1217, 2000, 2416):
            lens = torch.full((n,), L, dtype=torch.int32, device="cuda")
            cap = torch.full((n,), most, dtype=torch.int32, device="cuda")
            a = z.zipvl_decode(desc, q, None, None, k, v, off, cap, lens, L, ws=ws)
            assert torch.equal(a, z.zipvl_decode(desc, q, None, None, k, v, off, cap, lens, L))


@pytest.mark.gpu
def test_one_workspace_for_every_score(zipvl):
    """fp32: a workspace for 2500 tokens and 200 probes takes 2048 tokens and 128 probes, which need more."""
    H, d = 16, 64
    lay = lambda L: z.zipvl_layer(L, H, H, d, z.ZIPVL_F32, 0, 0, 0, 0.0, 0)
    ws = z.workspace(z.zipvl_workspace_bytes(z.OP_SCORE, lay(2500), 200), "cuda")
    g = torch.Generator().manual_seed(2)
    q, k = (torch.randn(2500, H, d, generator=g).cuda() for _ in range(2))
    for L, P in ((2500, 200), (2048, 128), (2048, 129), (2049, 128), (700, 97), (64, 1)):
        probe = torch.arange(L - P, L, dtype=torch.int32, device="cuda")
        a, _ = z.zipvl_score(lay(L), q[:L], k[:L], probe, ws=ws)
        b, _ = z.zipvl_score(lay(L), q[:L], k[:L], probe)
        assert torch.equal(a, b)
