"""Many different calls queued up behind one another - launches overlap, each overwrites what the one before has read - give
the bits of the same calls made one at a time."""
import pytest
import torch

from paper_2604_13226_b200 import binding as kvp
from paper_2604_13226_b200 import inputs as gen
from paper_2604_13226_b200.session import Session

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d,hq,hkv,q_len,kind", [
    ("f32", 64, 4, 2, 20, "prefill"), ("f32", 128, 8, 2, 5, "steps"), ("bf16", 64, 32, 8, 31, "prefill"), ("bf16", 64, 8, 2, 3, "steps"),
    ("bf16", 128, 32, 8, 20, "prefill"), ("bf16", 128, 32, 8, 64, "prefill"), ("bf16", 128, 32, 8, 2, "steps"),
    ("bf16", 128, 8, 2, 20, "handover"), ("f32", 64, 4, 2, 9, "handover")])
def test_queued_calls(dtype, d, hq, hkv, q_len, kind):
    n = 24
    shape = gen.ModelShape(1, hq, hkv, d, dtype, 10000.0, 0)
    wl = gen.make_workload(shape, [700, 1024, 300], [[(0, 0), (1, 0)], [(1, 0), (2, -1), (0, 0)]], q_len=q_len, seed=q_len)
    sess = Session(wl, materialize=kind == "handover", max_query_tokens=q_len * (n if kind == "steps" else 1))
    base = sess.query_tensors(0)
    rng = torch.Generator(device="cuda")
    rng.manual_seed(1)
    sets = [tuple(torch.randn(t.shape, generator=rng, device="cuda", dtype=t.dtype) for t in base) for _ in range(n)]
    runs = []
    for queued in (False, True):
        got = []
        held = tuple(torch.zeros_like(t) for t in base)          # one set of buffers, as a serving loop keeps
        torch.cuda.synchronize()
        if queued:
            torch.cuda._sleep(40_000_000)
        aid, prefix = sess.assemble()
        for i, qkv in enumerate(sets):
            for to, x in zip(held, qkv):
                to.copy_(x)
            if kind == "handover" and i % 2 == 0:                # every other prefill over the same assembly
                aid, prefix = sess.assemble()
            flags = ((kvp.CONTINUE if i else 0) | kvp.ROPE_QUERY) if kind == "steps" else 0
            got += sess.prefill(0, flags, qkv=held)
            if kind == "handover":
                got += sess.ctx.export_cache(aid, 0, 1, prefix[1], q_len)
            if not queued:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert sess.ctx.status_word() == 0
        runs.append(got)
    assert all(torch.equal(a, b) for a, b in zip(*runs))
    sess.close()


@pytest.mark.parametrize("layers,kept", [(1, None), (4, 0.5)])
def test_queued_calls_with_lists_of_their_own(layers, kept):
    # Every call has a new work list, in the place of the one before: it comes along with the launch, one warp stores it and the
    # other CTAs release the merge and the next call before that; the same list again is read where it was stored.  Pairs (64
    # tokens), single CTAs (20) and one of several row blocks (100), layer after layer; `kept`: a list per layer.
    shape = gen.ModelShape(layers, 32, 8, 128, "bf16", 10000.0, 0)
    wl = gen.make_workload(shape, [700, 1024, 300], [[(0, -1), (1, -1)], [(1, -1), (2, -1), (0, -1)]], q_len=100, seed=3)
    if kept:
        gen.draw_kept(wl.packets, [kept] * 3, 4, layers, 8)
    sess = Session(wl)
    calls = [(l, n, again) for n in (64, 20, 100, 20, 64) for l in range(layers) for again in (0, 1)]
    qkv = [tuple(t[:, :n].contiguous() for t in sess.query_tensors(l)) for l, n, _ in calls]
    runs = []
    for queued in (False, True, True):
        got = []
        torch.cuda.synchronize()
        if queued:
            torch.cuda._sleep(40_000_000)
        sess.assemble()
        for (l, _, _), x in zip(calls, qkv):
            got += sess.prefill(l, qkv=x)
            if not queued:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert sess.ctx.status_word() == 0
        runs.append(got)
    for run in runs[1:]:
        assert all(torch.equal(a, b) for a, b in zip(runs[0], run))
    sess.close()
