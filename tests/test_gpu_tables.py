"""Plans and work lists on both sides of the sizes up to which they travel as kernel parameters (4 KB; 16 KB for a list per
layer): attention of both layers (the second reads the stored list) and the exported cache (which reads the stored plan)
against the oracle."""
import numpy as np
import pytest
import torch

from oracle import reference as orc
from paper_2604_13226_b200 import binding as kvp
from paper_2604_13226_b200 import inputs as gen
from paper_2604_13226_b200.session import Session, torch_to_np
from helpers import make_store
from test_gpu_compressed import compressed_small
from test_gpu_decode import check
from test_gpu_parity import check_attention

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_docs", [1, 60, 70, 74, 76, 78, 80, 160])    # a plan holds 52 bytes per document and some more
@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("bf16", 64), ("f32", 64)])
def test_plan_sizes(n_docs, dtype, d):
    shape = gen.ModelShape(2, 8, 2, d, dtype, 500000.0, 0)
    wl = gen.make_workload(shape, [3 + p % 11 for p in range(n_docs)], [[(p, 0) for p in range(n_docs)]], q_len=9, seed=n_docs)
    sess = Session(wl)
    aid, plen = sess.assemble()
    for layer in (0, 1):
        check_attention(wl, sess, layer=layer)
    plan = orc.compose(make_store(wl), wl.items[0], True)
    _, v_ref, _ = orc.composed_kv(make_store(wl), plan, 1, orc.inv_freq(shape.rope_theta, d), 0)
    _, v = sess.ctx.export_cache(aid, 1, 0, plen[0], 0)
    assert np.array_equal(orc.widen(torch_to_np(v, dtype), dtype), v_ref)
    sess.close()


@pytest.mark.parametrize("ctas", [1, 50, 58, 62, 66, 74, 148])          # a list holds 52 bytes per CTA and 32 per merged tile
@pytest.mark.parametrize("d", [128, 64])
def test_list_sizes(ctas, d):
    shape = gen.ModelShape(2, 32, 8, d, "bf16", 500000.0, 0)
    wl = gen.make_workload(shape, [1024, 700, 2048], [[(0, 0), (1, 0), (2, 0)]], q_len=20, seed=ctas)
    sess = Session(wl)
    sess.ctx.tune(kvp.TUNE_SPLIT_TARGET_CTAS, ctas)
    sess.assemble()
    for layer in (0, 1, 0):
        check_attention(wl, sess, layer=layer)
    sess.close()


@pytest.mark.parametrize("ctas", [1, 70, 148])
def test_list_per_layer(ctas):
    wl = compressed_small(q_len=130)
    sess = Session(wl)
    sess.ctx.tune(kvp.TUNE_SPLIT_TARGET_CTAS, ctas)
    sess.assemble()
    for layer in (0, 1, 0):
        out, lse = sess.prefill(layer)
        assert sess.ctx.status_word() == 0
        check(wl, out, lse, layer)
    sess.close()


@pytest.mark.parametrize("batch,start", [(1, 126), (3, 126), (6, 124)])
def test_lists_change_while_layers_follow_one_another(batch, start):
    # a decode over four layers, each step layer after layer: the list changes when the appended rows enter another 128-key
    # tile, in the place of the one before; the layers behind the first read it as that one's launch has stored it
    L, n = 4, 5
    shape = gen.ModelShape(L, 16, 2, 128, "bf16", 500000.0, 0)
    lens = [900, 300, 1500]
    wl = gen.make_workload(shape, lens, [[((b + i) % 3, 0) for i in range(1 + b % 3)] for b in range(batch)], q_len=start + n,
                           seed=batch)
    sess = Session(wl)
    for _ in range(2):                                        # the second time over the first one's lists
        sess.assemble()
        outs, lses = [[] for _ in range(L)], [[] for _ in range(L)]
        qkv = [sess.query_tensors(l) for l in range(L)]
        cuts = [(0, start)] + [(start + i, start + i + 1) for i in range(n)]
        parts = [[tuple(t[:, a:b].contiguous() for t in qkv[l]) for l in range(L)] for a, b in cuts]
        for i, layers in enumerate(parts):
            for l, x in enumerate(layers):
                o, z = sess.prefill(l, kvp.CONTINUE if i else 0, qkv=x)
                outs[l].append(o)
                lses[l].append(z)
        assert sess.ctx.status_word() == 0
        for l in range(L):
            check(wl, torch.cat(outs[l], dim=1), torch.cat(lses[l], dim=2), l)
    sess.close()
