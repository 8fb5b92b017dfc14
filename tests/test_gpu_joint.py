"""Joint units: short calls of several requests over shared documents, whose rows share one query tile.  Steps against the
oracle: batches of 2 to 32, groups of 1, 4 and 7, one and several tokens a step, a document that a request names twice,
documents of a single key and of ragged lengths, causal tiles that a step enters, offsets of either sign and none."""
import numpy as np
import pytest
import torch

from paper_2604_13226_b200 import binding as kvp
from paper_2604_13226_b200 import inputs as gen
from paper_2604_13226_b200.session import Session
from test_gpu_decode import check, run_chunks

pytestmark = pytest.mark.gpu


def joint_used(sess, n_kv):
    # n_kv units share the CTAs (otherwise batch * n_kv do): the largest has at least its even share of the pieces
    return sess.ctx.last_launch()["splits"] >= sess.ctx.last_launch()["ctas"] // n_kv


@pytest.mark.parametrize("hq,hkv,batch,chunks,flags", [
    (32, 8, 2, [(0, 9), (9, 10), (10, 11)], 0),
    (32, 8, 8, [(0, 3), (3, 4), (4, 5)], kvp.ROPE_QUERY),
    (28, 4, 4, [(0, 2), (2, 6), (6, 7)], 0),                # 4 x 7 x 4 = 112 rows, then 28
    (32, 8, 32, [(0, 1), (1, 2)], 0),                       # 128 rows: the tile is full
    (8, 8, 5, [(0, 120), (120, 127), (127, 129), (129, 131)], kvp.ROPE_QUERY),   # group 1; enters the second causal tile
])
@pytest.mark.parametrize("pairing", [0, 1])
def test_joint_steps(hq, hkv, batch, chunks, flags, pairing):
    shape = gen.ModelShape(1, hq, hkv, 128, "bf16", 500000.0, pairing)
    lens = [1500, 1, 900, 1029, 128, 700, 2100]
    items = [[((b + 2 * i) % 7, 0 if (b + i) % 3 else -1) for i in range(5)] for b in range(batch)]
    if batch == 2:
        items = [[(0, 0), (3, -1), (6, 0), (0, 0), (1, -1)], [(6, -1), (0, -1), (3, 0), (1, 0), (0, 0)]]
    wl = gen.make_workload(shape, lens, items, q_len=chunks[-1][1], seed=50 + batch, packet_pos0=[0, 3, 0, 5000, 1, 20, 700])
    sess = Session(wl)
    sess.assemble()
    out, lse = run_chunks(wl, sess, chunks, 0, flags)
    assert joint_used(sess, hkv)
    check(wl, out, lse, rope_query=bool(flags))
    sess.close()


def test_joint_only_where_it_saves():
    shape = gen.ModelShape(1, 32, 8, 128, "bf16", 500000.0, 0)
    for items, want in (([[(p, 0) for p in (0, 1, 2)], [(p, 0) for p in (3, 4, 5)]], False),
                        ([[(p, 0) for p in (0, 1, 2)], [(p, 0) for p in (2, 1, 0)]], True)):
        wl = gen.make_workload(shape, [2048] * 6, items, q_len=5, seed=3)
        sess = Session(wl)
        sess.assemble()
        out, lse = run_chunks(wl, sess, [(0, 4), (4, 5)])
        assert joint_used(sess, 8) == want
        check(wl, out, lse)
        sess.close()


@pytest.mark.parametrize("group,steps", [(4, 3), (1, 2), (7, 4)])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_one_requests_values_stay_with_it(group, steps, bad):
    # NaN or infinity among the values that only request 0 sees - a document of its own, rows it appends, a document it
    # shares with request 2 - leaves every other request's bits alone.  (Not in the first 15 rows of a document: the last
    # product over the document in front of it in the pool reaches that far, with weights of 0.)
    shape = gen.ModelShape(1, 2 * group, 2, 128, "bf16", 500000.0, 0)
    lens = [4096, 3000, 700, 130, 2048]
    items = [[(0, 0), (2, 0), (4, -1)], [(0, 0), (1, 0)], [(1, -1), (0, 0), (4, 0)], [(0, -1), (1, 0), (3, 0)], [(1, 0), (0, 0)]]
    outs = []
    for poison in (None, "document", "appended", "shared"):
        wl = gen.make_workload(shape, lens * 2, [it + [(p + 5, a) for p, a in it] for it in items], q_len=10 + steps, seed=9)
        word = gen.to_stored(np.array([bad], dtype=np.float32), "bf16")[0]
        if poison == "document":
            wl.packets[2].v[0, [20, 131, 699], :, :] = word
        elif poison == "shared":
            wl.packets[9].v[0, 1027, :, 17] = word
        elif poison == "appended":
            wl.v_new[0][0, [3, 11], :, 40:] = word
        sess = Session(wl)
        sess.assemble()
        outs.append(run_chunks(wl, sess, [(0, 10), (10, 10 + steps - 1), (10 + steps - 1, 10 + steps)])[0])
        assert joint_used(sess, 2)
        sess.close()
    clean, rest = outs[0][:, 10:], [o[:, 10:] for o in outs[1:]]
    assert torch.isfinite(clean).all()
    for o, hit in zip(rest, ([0], [0], [0, 2])):
        for b in range(5):
            assert torch.equal(o[b], clean[b]) == (b not in hit), b
            assert bool(torch.isfinite(o[b]).all()) == (b not in hit)


@pytest.mark.parametrize("group,batch,steps", [(4, 16, 2), (4, 8, 3), (7, 6, 3)])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), 3e38])
def test_one_requests_keys_stay_with_it(group, batch, steps, bad):
    # Scores of rows over documents that their request does not hold are not masked, and warps with no other rows leave them
    # where P would stand: NaN and infinity among the keys of request 0's own document and of one that it shares with the last
    # request, which lies in another warp, leave every other request's bits alone.
    shape = gen.ModelShape(1, 2 * group, 2, 128, "bf16", 500000.0, 0)
    lens = [4096, 2048, 300, 130]
    items = [[(0, 0), (1, 0)] for _ in range(batch)]
    items[0] = [(2, 0), (0, 0), (1, -1), (3, 0)]
    items[-1] = [(0, -1), (3, 0), (1, 0)]
    outs = []
    for poison in (None, 2, 3):
        wl = gen.make_workload(shape, lens, items, q_len=5 + steps, seed=19)
        if poison is not None:
            wl.packets[poison].k[0, 5::7, :, ::3] = gen.to_stored(np.array([bad], dtype=np.float32), "bf16")[0]
        sess = Session(wl)
        sess.assemble()
        outs.append(run_chunks(wl, sess, [(0, 5), (5, 5 + steps - 1), (5 + steps - 1, 5 + steps)])[0][:, 5:])
        assert joint_used(sess, 2)
        sess.close()
    assert torch.isfinite(outs[0]).all()
    for o, hit in zip(outs[1:], ([0], [0, batch - 1])):
        for b in range(batch):
            assert torch.equal(o[b], outs[0][b]) == (b not in hit), b
