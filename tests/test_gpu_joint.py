"""Joint units: short calls of several requests over shared documents, whose rows share one query tile.  Steps against the
oracle: batches of 2 to 32, groups of 1, 4 and 7, one and several tokens a step, a document that a request names twice,
documents of a single key and of ragged lengths, causal tiles that a step enters, offsets of either sign and none."""
import pytest

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
