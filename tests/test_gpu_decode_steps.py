"""Decode steps that end inside their kernel (at most one wave of thread blocks) and those that take the merge
kernel, around the line between them: lengths, heads and types at the edges of tiles and chunks, a workspace
full of arbitrary bytes, shared with other calls, and replays of a captured step."""
import numpy as np
import pytest
import torch

import oracle
from parity import check_attention, to_np

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
CODE = {torch.bfloat16: 0, torch.float32: 1, torch.float16: 2}


def make(lens, Hkv, d, dtype, extra, seed):
    g = torch.Generator().manual_seed(seed)
    cap = [n + extra for n in lens]
    row = Hkv * d
    off = np.concatenate([[0], np.cumsum([c * row for c in cap[:-1]])]).astype(np.int64)
    kc, vc = (torch.randn(sum(cap) * row, generator=g).to(dtype) for _ in range(2))
    return kc, vc, torch.from_numpy(off), torch.tensor(cap, dtype=torch.int32), g


def workspace(z, desc, max_len, fill):
    lay = z.zipvl_layer(max_len, desc.n_q_heads, desc.n_kv_heads, desc.head_dim, desc.dtype, 0, 0, 0, 0.0, 0)
    ws = z.workspace(z.zipvl_workspace_bytes(z.OP_DECODE, lay, 0, desc.batch), DEV)
    return ws.fill_(fill)


@pytest.mark.parametrize("lens,Hq,Hkv,d,dtype", [
    ([1], 2, 2, 64, torch.float32), ([63, 64, 65], 4, 4, 128, torch.bfloat16), ([2307], 32, 32, 128, torch.bfloat16),
    ([7000], 32, 32, 128, torch.float16), ([7200], 32, 32, 128, torch.float16),          # below and above one wave
    ([15, 16, 17, 0], 14, 2, 64, torch.bfloat16), ([3000, 1], 28, 4, 128, torch.float16),
    ([700, 33], 12, 4, 96, torch.bfloat16), ([1537, 90, 4000], 16, 1, 128, torch.bfloat16),
    ([500, 1200], 64, 2, 64, torch.float16), ([900], 17, 1, 96, torch.float16),
    ([300] * 40, 28, 4, 128, torch.bfloat16), ([200] * 13, 6, 3, 96, torch.float32)])
def test_decode_steps(zipvl, lens, Hq, Hkv, d, dtype):
    z, B, steps = zipvl, len(lens), 3
    kc, vc, off, cap, g = make(lens, Hkv, d, dtype, steps, sum(lens) + Hq)
    desc = z.zipvl_decode_desc(B, Hq, Hkv, d, CODE[dtype], 0.0)
    max_len = max(lens) + steps
    kd, vd, offd, capd = kc.to(DEV), vc.to(DEV), off.to(DEV), cap.to(DEV)
    seq = torch.tensor(lens, dtype=torch.int32, device=DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    ws = workspace(z, desc, max_len, 0xA5)
    ko, vo, seqo = to_np(kc).copy(), to_np(vc).copy(), np.array(lens, np.int32)
    for i in range(steps):
        q = torch.randn(B, Hq, d, generator=g).to(dtype)
        kn, vn = (torch.randn(B, Hkv, d, generator=g).to(dtype) for _ in range(2))
        append = i != 1
        args = (kn.to(DEV), vn.to(DEV)) if append else (None, None)
        out = z.zipvl_decode(desc, q.to(DEV), *args, kd, vd, offd, capd, seq, max_len, ws=ws, status=st)
        want = oracle.decode_step(to_np(q), to_np(kn) if append else None, to_np(vn) if append else None, ko, vo, off.numpy(),
                                  seqo, Hkv)
        check_attention(to_np(out), want, dtype)
        assert np.array_equal(seq.cpu().numpy(), seqo)
        again = z.zipvl_decode(desc, q.to(DEV), None, None, kd, vd, offd, capd, seq, max_len, ws=ws, status=st)
        if append:
            assert torch.equal(out, again)              # (the appended row is in the cache now)
    assert st.item() == 0
    assert np.array_equal(to_np(kd.cpu()), ko) and np.array_equal(to_np(vd.cpu()), vo)


@pytest.mark.parametrize("Hq,Hkv", [(32, 32), (28, 4)])
def test_replayed_step_next_to_other_work_in_the_same_workspace(zipvl, Hq, Hkv):
    """Steps captured once and replayed from the same lengths, the workspace rewritten in between in different
    ways (left alone, zeroed in part, other sizes of the same call): every replay gives the first one's bits."""
    z, d, dtype, n = zipvl, 128, torch.bfloat16, 1111
    kc, vc, off, cap, g = make([n, 5], Hkv, d, dtype, 4, 7)
    kd, vd, offd, capd = kc.to(DEV), vc.to(DEV), off.to(DEV), cap.to(DEV)
    desc = z.zipvl_decode_desc(2, Hq, Hkv, d, z.ZIPVL_BF16, 0.0)
    ws = workspace(z, desc, n + 4, 0xFF)
    lens0 = torch.tensor([n, 5], dtype=torch.int32, device=DEV)
    seq, st = lens0.clone(), torch.zeros(1, dtype=torch.int32, device=DEV)
    q = torch.randn(2, Hq, d, generator=g).to(dtype).to(DEV)
    kn, vn = (torch.randn(2, Hkv, d, generator=g).to(dtype).to(DEV) for _ in range(2))
    out = torch.empty_like(q)

    def step():
        seq.copy_(lens0)
        for _ in range(3):
            z.zipvl_decode(desc, q, kn, vn, kd, vd, offd, capd, seq, n + 4, out=out, ws=ws, status=st)

    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        step()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            step()
        graph.replay()
        side.synchronize()
        first = out.clone()
        one = z.zipvl_decode_desc(1, Hq, Hkv, d, z.ZIPVL_BF16, 0.0)
        for i in range(60):
            if i % 3 == 1:
                ws[:8 * (1 + i)].zero_()
            if i % 5 == 2:
                other = lens0[:1].clone()
                z.zipvl_decode(one, q[:1], None, None, kd, vd, offd[:1], capd[:1], other, n + 4, ws=ws, status=st)
            out.zero_()
            graph.replay()
            side.synchronize()
            assert torch.equal(out, first) and seq.tolist() == [n + 3, 8]
    assert st.item() == 0
