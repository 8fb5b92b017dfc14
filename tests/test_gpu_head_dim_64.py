"""bf16 with head dimension 64: large calls run on the tcgen05 kernel (rotated Q and P in two bf16 numbers each),
small ones on the CUDA-core kernel.  Against the CUDA-core kernel on every row and against the oracle."""
import numpy as np
import pytest
import torch

from paper_2604_13226_b200 import binding as kvp
from paper_2604_13226_b200 import inputs as gen
from paper_2604_13226_b200.session import Session
from test_gpu_parity import check_attention

pytestmark = pytest.mark.gpu


# (q heads, kv heads, pairing, document lengths per request, q_len, CTAs of the work list): tile remainders of 1 and
# 127 keys, one and two query tiles per unit, odd tile counts, a unit's last tile of a few rows, split and whole units
CASES = [
    (32, 8, 0, [[1024, 129, 1, 2048], [700, 127]], 64, 0),
    (32, 8, 1, [[1024, 129, 1, 2048], [700, 127]], 64, 0),
    (32, 8, 0, [[2048] * 5, [3000, 17]], 16, 0),
    (32, 8, 0, [[1024] * 4], 129, 1),
    (28, 4, 1, [[511, 513, 2000], [128]], 150, 7),
    (8, 8, 0, [[4096, 300]], 257, 0),
]


@pytest.mark.parametrize("hq,hkv,pairing,docs,q_len,ctas", CASES)
def test_tensor_kernel_against_cuda_core_kernel_and_oracle(hq, hkv, pairing, docs, q_len, ctas):
    shape = gen.ModelShape(1, hq, hkv, 64, "bf16", 10000.0, pairing)
    lens, items = [], []
    for b, ds in enumerate(docs):
        items.append([(len(lens) + i, 0 if (b + i) % 3 < 2 else -1) for i in range(len(ds))])
        lens += ds
    wl = gen.make_workload(shape, lens, items, q_len=q_len, n_header=16, n_trailer=7, seed=q_len)
    sess = Session(wl)
    sess.assemble()
    if ctas:
        sess.ctx.tune(kvp.TUNE_SPLIT_TARGET_CTAS, ctas)
    qkv = sess.query_tensors(0)
    out, lse = sess.prefill(0, qkv=qkv)
    assert sess.ctx.status_word() == 0 and sess.ctx.last_launch()["kind"] == 1
    ref, ref_lse = sess.prefill(0, kvp.FORCE_SIMPLE, qkv=qkv)
    assert sess.ctx.last_launch()["kind"] == 0
    # q' = hi + rem leaves 2^-17 of each term of q.k: |q| |k| / sqrt(64) <= 12 * 12 / 8 here, so scores and lse move by
    # 2^-17 * 18 = 1.4e-4 at most; the probabilities' own split leaves 2^-17 relative.  Outputs: twice that times
    # max |v| (5.5) plus one bf16 rounding step of either side
    assert float((lse - ref_lse).abs().max()) <= 2e-4
    o, r = out.float(), ref.float()
    assert bool(((o - r).abs() <= 2.0 ** -8 * r.abs() + 1.6e-3).all()), float((o - r).abs().max())
    check_attention(wl, sess)
    sess.close()


def test_continuation_and_raw_query_on_the_tensor_kernel():
    # a prefill fed in two chunks, the library rotating q and k: together they equal one call over all tokens
    shape = gen.ModelShape(1, 32, 8, 64, "bf16", 10000.0, 0)
    wl = gen.make_workload(shape, [1500, 900], [[(0, 0), (1, 0)]], q_len=140, seed=5)
    sess = Session(wl)
    sess.assemble()
    q, k, v = sess.query_tensors(0)
    whole, lse = sess.prefill(0, kvp.ROPE_QUERY, qkv=(q, k, v))
    assert sess.ctx.last_launch()["kind"] == 1
    parts = []
    for i, (a, b) in enumerate(((0, 70), (70, 140))):
        cut = tuple(t[:, a:b].contiguous() for t in (q, k, v))
        parts.append(sess.prefill(0, kvp.ROPE_QUERY | (kvp.CONTINUE if i else 0), qkv=cut)[0])
        assert sess.ctx.last_launch()["kind"] == 1
    got = torch.cat(parts, dim=1).float()
    ref = whole.float()
    assert sess.ctx.status_word() == 0
    assert bool(((got - ref).abs() <= 2.0 ** -8 * ref.abs() + 1.6e-3).all())          # as above
    assert np.isfinite(lse.cpu().numpy()).all()
    sess.close()


@pytest.mark.parametrize("q_len,batch", [(31, 8), (27, 8), (95, 4)])        # 124, 108 and 124 rows in a unit's last tile
def test_the_same_bits_whatever_ran_before(q_len, batch):
    # the rows that a query tile has beyond the request's share warps with the request's last ones: their scores must not
    # depend on what shared memory held, or the probabilities next to them are taken apart into their two numbers again
    shape = gen.ModelShape(1, 32, 8, 64, "bf16", 10000.0, 0)
    lens = [2048, 1500, 900, 700]
    wl = gen.make_workload(shape, lens, [[(p, 0) for p in range(4)]] * batch, q_len=q_len, seed=q_len)
    sess = Session(wl)
    sess.assemble()
    q, k, v = sess.query_tensors(0)
    want, want_lse = sess.prefill(0, qkv=(q, k, v))
    for i in range(40):
        sess.prefill(0, qkv=(q * 2.0 ** (i % 12), k, v))
        out, lse = sess.prefill(0, qkv=(q, k, v))
        assert sess.ctx.last_launch()["kind"] == 1
        assert torch.equal(out, want) and torch.equal(lse, want_lse), i
    sess.close()
