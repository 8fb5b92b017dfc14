"""Staging buffers of plans and work lists outlive the streams they were used on: streams that are destroyed with work
pending (which then still runs), and more uploads pending than there are buffers."""
import ctypes

import pytest
import torch

from paper_2604_13226_b200 import binding as kvp
from paper_2604_13226_b200 import inputs as gen
from paper_2604_13226_b200.session import Session

pytestmark = pytest.mark.gpu


def test_streams_destroyed_with_uploads_pending():
    cudart = ctypes.CDLL("libcudart.so.12")
    shape = gen.ModelShape(1, 8, 2, 128, "bf16", 500000.0, 0)
    # 200 short documents: a plan of more than 4 KB, which a kernel uploads
    wl = gen.make_workload(shape, [3 + p % 5 for p in range(200)], [[(p, 0) for p in range(200)]], q_len=4, seed=3)
    sess = Session(wl, max_assemblies=1)
    sess.assemble()
    qkv = sess.query_tensors(0)
    want, want_lse = sess.prefill(0, qkv=qkv)
    torch.cuda.synchronize()
    for _ in range(12):                                   # two plan buffers: every other assemble waits for one
        raw = ctypes.c_void_p()
        assert cudart.cudaStreamCreateWithFlags(ctypes.byref(raw), 1) == 0
        s = torch.cuda.ExternalStream(raw.value)
        with torch.cuda.stream(s):
            torch.cuda._sleep(2_000_000)
            out, lse = torch.zeros_like(want), torch.zeros_like(want_lse)
            aid, _ = sess.ctx.assemble(wl.items, kvp.REBASE)
            sess.ctx.query_prefill(aid, 0, *qkv, 4, out, lse)
            done = torch.cuda.Event()
            done.record(s)
        assert cudart.cudaStreamDestroy(raw) == 0         # its work still runs
        torch.cuda.current_stream().wait_event(done)
        torch.cuda.current_stream().synchronize()
        assert torch.equal(out, want) and torch.equal(lse, want_lse)
    sess.close()


def test_uploads_wait_for_destroyed_streams():
    cudart = ctypes.CDLL("libcudart.so.12")
    shape = gen.ModelShape(1, 8, 2, 128, "bf16", 500000.0, 0)
    wl = gen.make_workload(shape, [3 + p % 5 for p in range(200)], [[(p, 0) for p in range(200)]], q_len=4, seed=3)
    sess = Session(wl, max_assemblies=4)
    qkv = sess.query_tensors(0)
    raw = ctypes.c_void_p()
    assert cudart.cudaStreamCreateWithFlags(ctypes.byref(raw), 1) == 0
    outs, ids = [], []
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.ExternalStream(raw.value)):
        torch.cuda._sleep(100_000_000)                    # 50 ms: every upload behind it is pending
        for i in range(4):
            aid, _ = sess.ctx.assemble(wl.items, kvp.REBASE)
            out, lse = torch.zeros_like(qkv[0]), torch.zeros(1, 8, 4, device="cuda")
            sess.ctx.query_prefill(aid, 0, *qkv, 4, out, lse)
            outs.append(out)
    assert cudart.cudaStreamDestroy(raw) == 0
    # five plan buffers, four of them pending: the second assemble from here on waits until its buffer has been read
    for i in range(3):
        sess.assemble()
    torch.cuda.synchronize()
    want, _ = sess.prefill(0, qkv=qkv)
    torch.cuda.synchronize()
    assert sess.ctx.status_word() == 0
    assert all(torch.equal(o, want) for o in outs)
    sess.close()
