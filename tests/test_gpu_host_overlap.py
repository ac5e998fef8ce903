"""The host-buffer calls where copies and kernels overlap: pinned buffers, Q and the output in four, two and one groups of
heads, some of the buffers pageable, calls from two threads and one right behind another.  Every output is compared, bit for
bit, with the same steps called on device tensors."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
CODE = {torch.bfloat16: 0, torch.float32: 1, torch.float16: 2}


def inputs(L, Hq, Hkv, d, dtype, seed, pinned=("q", "k", "v", "probe", "qn", "kn", "vn")):
    g = torch.Generator().manual_seed(seed)
    x = {"q": torch.randn(L, Hq, d, generator=g), "k": torch.randn(L, Hkv, d, generator=g), "v": torch.randn(L, Hkv, d, generator=g),
         "qn": torch.randn(1, Hq, d, generator=g), "kn": torch.randn(1, Hkv, d, generator=g), "vn": torch.randn(1, Hkv, d, generator=g)}
    x["k"][::7] *= 3
    x = {m: t.to(dtype) for m, t in x.items()}
    P = min(L, 96)
    x["probe"] = torch.sort(torch.randperm(L, generator=g)[:P]).values.to(torch.int32)
    return {m: t.pin_memory() if m in pinned else t for m, t in x.items()}


def on_the_device(z, x, tau):
    q, k, v, probe, qn, kn, vn = (x[m].to(DEV) for m in ("q", "k", "v", "probe", "qn", "kn", "vn"))
    lay, L = z.layer_desc(q, k), q.shape[0]
    acc, norm = z.zipvl_score(lay, q, k, probe)
    count, idx = z.zipvl_select(acc, norm, tau)
    kc, vc = (torch.zeros(L + 1, *k.shape[1:], dtype=k.dtype, device=DEV) for _ in range(2))
    out, length = z.zipvl_sparse_prefill_compact(lay, q, k, v, idx, count, L, kc, vc, L)
    desc = z.zipvl_decode_desc(1, q.shape[1], k.shape[1], q.shape[2], CODE[q.dtype], 0.0)
    dec = z.zipvl_decode(desc, qn, kn, vn, kc, vc, torch.zeros(1, dtype=torch.int64, device=DEV),
                         torch.tensor([L + 1], dtype=torch.int32, device=DEV), length.clone(), L + 1)
    n = int(count.item())
    return n, idx.cpu(), out.cpu(), kc[:n].cpu(), vc[:n].cpu(), dec.cpu()


def from_the_host(z, x, tau, pinned_out=True):
    mk = lambda t: torch.full_like(t, 7).pin_memory() if pinned_out else torch.full_like(t, 7)
    L = x["q"].shape[0]
    idx = mk(torch.zeros(L, dtype=torch.int32))
    n, idx, out, kc, vc, dec = z.zipvl_layer_step_host(z.layer_desc(x["q"], x["k"]), x["q"], x["k"], x["v"], x["probe"], tau, x["qn"],
                                                       x["kn"], x["vn"], out=mk(x["q"]), k_cache=mk(x["k"]), v_cache=mk(x["v"]), idx=idx,
                                                       decode_out=mk(x["qn"]))
    assert bool((kc[n:] == 7).all()) and bool((vc[n:] == 7).all())      # rows past the set stay as they were
    return n, idx.clone(), out.clone(), kc[:n].clone(), vc[:n].clone(), dec.clone()


def same(a, b):
    assert a[0] == b[0]
    for x, y in zip(a[1:], b[1:]):
        assert torch.equal(x, y)


SHAPES = [(2945, 32, 32, 128, torch.bfloat16),      # four groups of eight heads
          (1301, 28, 4, 128, torch.float16),        # four groups of one kv head
          (5001, 12, 4, 96, torch.bfloat16),        # two groups (rows of a quarter would be under 1 KB)
          (4001, 14, 2, 64, torch.bfloat16), (7001, 10, 5, 64, torch.float16),      # one: 896-byte rows, five kv heads
          (333, 16, 16, 64, torch.float16), (65, 2, 1, 128, torch.bfloat16), (1024, 4, 4, 64, torch.float32)]


@pytest.mark.parametrize("L,Hq,Hkv,d,dtype", SHAPES)
def test_pinned_buffers(zipvl, L, Hq, Hkv, d, dtype):
    """Three calls with other inputs right behind one another, each on scratch that the one before gave back."""
    for seed in range(3):
        x = inputs(L, Hq, Hkv, d, dtype, seed)
        same(from_the_host(zipvl, x, 0.9), on_the_device(zipvl, x, 0.9))


@pytest.mark.parametrize("pinned", [("q", "probe"), ("k", "v", "qn"), ("q", "k", "v", "qn", "kn", "vn"), ("q", "k", "v", "probe")])
@pytest.mark.parametrize("pinned_out", [True, False])
def test_some_buffers_pageable(zipvl, pinned, pinned_out):
    x = inputs(1777, 32, 8, 128, torch.bfloat16, 4, pinned)
    same(from_the_host(zipvl, x, 0.95, pinned_out), on_the_device(zipvl, x, 0.95))


def test_two_threads(zipvl):
    """Calls of two threads share the library's pool, streams and events; neither sees the other's data."""
    sets = [[inputs(L, 16, 16, 64, torch.bfloat16, 10 * i + j) for j, L in enumerate((1948, 301, 2500))] for i in range(2)]
    want = [[on_the_device(zipvl, x, 0.9) for x in xs] for xs in sets]
    got, errors = [[], []], []

    def work(i):
        try:
            torch.cuda.set_device(0)
            for _ in range(3):
                got[i].append([from_the_host(zipvl, x, 0.9) for x in sets[i]])
        except Exception as e:          # (an assert in a thread would go unseen)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for i in range(2):
        for turn in got[i]:
            for a, b in zip(turn, want[i]):
                same(a, b)


def test_scratch_is_given_back(zipvl):
    """zipvl_release_host_scratch right behind a call leaves the device as much free memory as before the call."""
    x = inputs(2945, 32, 32, 128, torch.bfloat16, 1)
    from_the_host(zipvl, x, 0.9)
    zipvl.zipvl_release_host_scratch()
    before = torch.cuda.mem_get_info()[0]
    for _ in range(5):
        from_the_host(zipvl, x, 0.9)
        zipvl.zipvl_release_host_scratch()
        assert torch.cuda.mem_get_info()[0] >= before - (2 << 20)      # (the scratch is some 150 MB)


def test_more_calls_at_once_than_are_kept(zipvl):
    """Eight threads at a time, of which the library keeps the streams of four: the others' are made and destroyed."""
    x = inputs(700, 4, 4, 64, torch.bfloat16, 3)
    want, got = on_the_device(zipvl, x, 0.9), []
    gate = threading.Barrier(8)

    def work():
        torch.cuda.set_device(0)
        for _ in range(3):
            gate.wait(60)
            got.append(from_the_host(zipvl, x, 0.9))

    threads = [threading.Thread(target=work) for _ in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert len(got) == 24
    for r in got:
        same(r, want)
    zipvl.zipvl_release_host_scratch()
    same(from_the_host(zipvl, x, 0.9), want)
