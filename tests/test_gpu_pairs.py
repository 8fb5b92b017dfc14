"""The attention kernel on CTA pairs at the edges of its pipeline: pieces of one to four tiles (three S buffers), documents
of a single tile (a new Q buffer at every step), short tiles, remainders of rows in the second CTA, outliers that move the
reference maximum late in a piece - every row against the oracle, and the same bits when run again."""
import math

import numpy as np
import pytest
import torch

from paper_2604_13226_b200 import binding as kvp
from paper_2604_13226_b200 import inputs as gen
from paper_2604_13226_b200.session import Session
from test_gpu_parity import check_attention

pytestmark = pytest.mark.gpu


def on_pairs(sess, q_len):
    # an entry of a pair plan's list is two CTAs
    cta_begin = sess.ctx.export_schedule(sess.assembly_id, q_len)[0]
    launch = sess.ctx.last_launch()
    return launch["kind"] == 1 and launch["ctas"] == 2 * (len(cta_begin) - 1)


@pytest.mark.parametrize("lens,q_len,ctas,flags", [
    ([1], 64, 0, 0),                                   # two or three tiles in all
    ([128], 33, 2, 0),                                 # 132 rows: four in the second CTA; one pair walks everything
    ([100, 1, 128, 127, 31, 33, 64], 64, 0, 0),        # a document per tile
    ([100, 1, 128, 127, 31, 33, 64], 64, 4, kvp.PRECISE_QK),
    ([129, 257, 385, 513], 64, 148, 0),                # many pieces of two tiles
    ([640, 1024], 192, 6, kvp.PRECISE_QK),             # two causal tiles, several pieces per pair
    ([300, 200], 409, 0, 0),                           # six units of 256 rows and one of 100 per kv head
])
def test_pipeline_edges(lens, q_len, ctas, flags):
    shape = gen.ModelShape(1, 32, 8, 128, "bf16", 500000.0, 0)
    wl = gen.make_workload(shape, lens, [[(p, 0) for p in range(len(lens))]], q_len=q_len, seed=91 + q_len)
    sess = Session(wl)
    sess.assemble()
    if ctas:
        sess.ctx.tune(kvp.TUNE_SPLIT_TARGET_CTAS, ctas)
    check_attention(wl, sess, flags=flags)
    assert on_pairs(sess, q_len)
    qkv = sess.query_tensors(0)
    first, _ = sess.prefill(0, flags, qkv=qkv)
    for _ in range(20):
        assert torch.equal(first, sess.prefill(0, flags, qkv=qkv)[0])
    sess.close()


def test_reference_maximum_moves_late_in_a_piece():
    # keys grow from document to document, so that scores rise by more than 2^8 at tiles of both warpgroups: O and the
    # tile at hand are rescaled.  Scores reach +-40, so the rounding of the rotated Q (2^-9 relative per term) shows in the
    # probabilities: KVP_PRECISE_QK, whose outputs the shared bounds hold for
    shape = gen.ModelShape(1, 32, 8, 128, "bf16", 500000.0, 0)
    wl = gen.make_workload(shape, [300, 200, 130, 500, 90], [[(p, 0) for p in range(5)]], q_len=64, seed=7)
    for i, pk in enumerate(wl.packets):
        pk.k[:] = gen.to_stored(gen.bf16_bits_to_f32(pk.k) * np.float32(0.2 * 2.2 ** i), "bf16")
    for ctas in (2, 0):
        sess = Session(wl)
        sess.assemble()
        if ctas:
            sess.ctx.tune(kvp.TUNE_SPLIT_TARGET_CTAS, ctas)
        check_attention(wl, sess, flags=kvp.PRECISE_QK)
        assert on_pairs(sess, 64)
        sess.close()


@pytest.mark.parametrize("q_len", [64, 192])
def test_probabilities_are_rounded_once(q_len):
    # Without rotation the scores are those of bf16 numbers and a partial result is not narrowed: what separates it from
    # fp64 is the rounding of the probabilities to bf16.  The same sums with each probability rounded once, in torch: over
    # 10^5 and more outputs the two errors' 2-norms agree to a percent or two (chance - the probabilities are rounded against
    # another reference - and 1e-6 of fp32 sums); a second rounding of every third tile of a piece adds a sixth.
    shape = gen.ModelShape(1, 8, 2, 128, "bf16", 500000.0, 0)
    wl = gen.make_workload(shape, [640, 700, 1024], [[(0, -1), (1, -1), (2, -1)]], q_len=q_len, seed=17, rebase=False)
    sess = Session(wl)
    aid, (prefix,) = sess.assemble()
    q, k, v = sess.query_tensors(0)
    buf = torch.zeros(sess.ctx.partial_bytes(1, q_len) // 4, dtype=torch.float32, device=q.device)
    sess.ctx.query_prefill(aid, 0, q, k, v, q_len, buf, None, kvp.PARTIAL)
    assert sess.ctx.status_word() == 0
    tiles = 2 * (4 * q_len // 128)                                # kv heads x 128-row tiles: O [tile][32][128][4], (m, l) [tile][128][2]
    o = buf[:tiles * 16384].view(tiles, 32, 128, 4).permute(0, 2, 1, 3).reshape(2, q_len, 4, 128).double()
    l = buf[tiles * 16384:].view(tiles, 128, 2)[..., 1].reshape(2, q_len, 4, 1).double()
    K, V = (x.double().permute(1, 0, 2)[:, None] for x in sess.ctx.export_cache(aid, 0, 0, prefix, q_len))      # [kv head][1][row][128]
    s = q[0].view(q_len, 2, 4, 128).permute(1, 2, 0, 3).double() @ K.transpose(-1, -2) / math.sqrt(128)
    late = torch.arange(prefix + q_len, device=q.device) > prefix + torch.arange(q_len, device=q.device)[:, None]
    s = s.masked_fill(late, -math.inf) / math.log(2)
    p = torch.exp2(s - s.amax(-1, keepdim=True))
    want = (p @ V / p.sum(-1, keepdim=True)).permute(0, 2, 1, 3)
    once = (p.bfloat16().double() @ V / p.sum(-1, keepdim=True)).permute(0, 2, 1, 3)
    err, ideal = float((o / l - want).norm()), float((once - want).norm())
    assert err <= 1.06 * ideal, (err, ideal, err / ideal)
    sess.close()


def rounded_against_references(s, v, tiles):
    """sum of P V / sum of p over one piece by the rule that moves references (the comment at the head of the pair kernel), in
    float64 but for P, which is rounded to bf16 as often as there.  s: scores in powers of two [row][key], -inf where masked;
    tiles: (first key, keys) of each.  Returns (result, whether a reference of the row moved)."""
    bf16 = lambda x: x.bfloat16().double()
    rows = s.shape[0]
    m = [None, None]
    o = torch.zeros(rows, v.shape[1], dtype=torch.float64, device=s.device)
    moved = torch.zeros(rows, dtype=torch.bool, device=s.device)
    for k, (at, n) in enumerate(tiles):
        g = k & 1
        if k == 0:
            m[0] = m[1] = s[:, at:at + min(32, n)].amax(1)                # where a piece starts from
        p = torch.zeros(rows, 0, dtype=torch.float64, device=s.device)
        for c in range(at, at + n, 32):
            x = s[:, c:min(c + 32, at + n)]
            need = x.amax(1) - m[g] > 8
            new = torch.where(need, x.amax(1), m[g])
            p = torch.cat([bf16(p * torch.exp2(m[g] - new)[:, None]), bf16(torch.exp2(x - new[:, None]))], 1)
            m[g], moved = new, moved | need
        if k > 0:                                                         # against the one in force after the tile before
            raised = m[g] - in_force > 8
            p = torch.where(raised[:, None], p, bf16(p * torch.exp2(m[g] - in_force)[:, None]))
            o *= torch.where(raised, torch.exp2(in_force - m[g]), 1.0)[:, None]
            m[g] = torch.where(raised, m[g], in_force)
        in_force = m[g]
        o += p @ v[at:at + n]
    return o / torch.exp2(s - in_force[:, None]).sum(1, keepdim=True), moved


@pytest.mark.parametrize("loud,own", [(8, 1), (1, 6), (24, 1)])
def test_references_that_probabilities_are_rounded_against(loud, own):
    # Probabilities are rounded to bf16 against a reference: another one rounds others up or down, by 2^-9 of a value that is
    # many times the root mean square where a row attends to one key.  The reference is the maximum of a piece's first 32
    # keys, of the causal block to begin with, until a score exceeds it by 2^8.  `loud`: two channels of the documents' keys, at
    # 24 so much so that references move in later tiles, and O with them once P V of the tile before is done;  `own`: the query block's keys from the 40th on, so that references move in the first tile and the second one starts from
    # where the first did.  fp32 scores and exponentials put a few probabilities in 2,000 on the other side of a tie (a
    # twelfth of the rounding error of all); against another reference the results are 1.4 of it apart.
    q_len, lens = 64, [640, 700, 1024]
    shape = gen.ModelShape(1, 8, 2, 128, "bf16", 500000.0, 0)
    wl = gen.make_workload(shape, lens, [[(i, -1) for i in range(3)]], q_len=q_len, seed=29, rebase=False)
    for pk in wl.packets:
        x = gen.bf16_bits_to_f32(pk.k)
        x[..., [5, 77]] *= np.float32(loud)
        pk.k[:] = gen.to_stored(x, "bf16")
    x = gen.bf16_bits_to_f32(wl.k_new[0])
    x[:, 40:] *= np.float32(own)
    wl.k_new[0][:] = gen.to_stored(x, "bf16")
    sess = Session(wl)
    aid, (prefix,) = sess.assemble()
    sess.ctx.tune(kvp.TUNE_SPLIT_TARGET_CTAS, 2)                          # one pair: units in one piece
    q, k, v = sess.query_tensors(0)
    buf = torch.zeros(sess.ctx.partial_bytes(1, q_len) // 4, dtype=torch.float32, device=q.device)
    sess.ctx.query_prefill(aid, 0, q, k, v, q_len, buf, None, kvp.PARTIAL)
    assert sess.ctx.status_word() == 0 and sess.ctx.last_launch()["ctas"] == 2
    o = buf[:4 * 16384].view(2, 2, 32, 128, 4).permute(0, 1, 3, 2, 4).reshape(2, 4 * q_len, 128).double()
    l = buf[4 * 16384:].view(2, 2, 128, 2)[..., 1].reshape(2, 4 * q_len, 1).double()
    K, V = (x.double() for x in sess.ctx.export_cache(aid, 0, 0, prefix, q_len))                  # [row][kv head][128]
    token = torch.arange(4 * q_len, device=q.device) // 4                                         # packed row: token, head in group
    tiles = [(prefix, q_len)] + [(sum(lens[:i]) + t, min(128, n - t)) for i, n in enumerate(lens) for t in range(0, n, 128)]
    apart = ideal = some = 0.0
    for h in range(2):
        s = q[0, :, 4 * h:4 * h + 4].reshape(-1, 128).double() @ K[:, h].T / math.sqrt(128) / math.log(2)
        s = s.masked_fill(torch.arange(prefix + q_len, device=q.device) > prefix + token[:, None], -math.inf)
        rounded, moved = rounded_against_references(s, V[:, h], tiles)
        apart += float((o[h] / l[h] - rounded).square().sum())
        ideal += float((rounded - torch.softmax(s * math.log(2), 1) @ V[:, h]).square().sum())
        some += float(moved.double().mean()) / 2
    assert (some > 0.2) == ((loud, own) != (8, 1)), some
    assert apart <= 0.2 ** 2 * ideal, (apart / ideal) ** 0.5
    sess.close()


def test_same_bits_whenever_the_second_tile_arrives():
    # References move in the first tile of a piece (the query's own keys, from the 40th on).  The second one starts from where
    # the first did, also when its keys come from memory so late that the first is done by then: after a write of 256 MB,
    # and with them in L2.
    shape = gen.ModelShape(1, 32, 8, 128, "bf16", 500000.0, 0)
    wl = gen.make_workload(shape, [100, 128, 60, 300], [[(p, -1) for p in range(4)]], q_len=64, seed=31)
    x = gen.bf16_bits_to_f32(wl.k_new[0])
    x[:, 40:] *= np.float32(6)
    wl.k_new[0][:] = gen.to_stored(x, "bf16")
    sess = Session(wl)
    sess.assemble()
    sess.ctx.tune(kvp.TUNE_SPLIT_TARGET_CTAS, 8)
    qkv = sess.query_tensors(0)
    first, _ = sess.prefill(0, qkv=qkv)
    assert on_pairs(sess, 64)
    far = torch.empty(1 << 28, dtype=torch.uint8, device=first.device)
    for i in range(30):
        if i % 3:
            far.fill_(i)
        assert torch.equal(first, sess.prefill(0, qkv=qkv)[0])
    sess.close()


def test_a_long_request_among_short_ones():
    # 90 query tiles to be merged, of which those of the short requests have two parts and those of the long one five
    shape = gen.ModelShape(1, 32, 8, 128, "bf16", 500000.0, 0)
    wl = gen.make_workload(shape, [10000] + [1666] * 5, [[(p, -1)] for p in range(6)], q_len=64, seed=41)
    sess = Session(wl)
    sess.assemble()
    check_attention(wl, sess)
    merges = sess.ctx.export_schedule(sess.assembly_id, 64)[2]
    assert on_pairs(sess, 64) and len(merges) == 90 and merges[:, 4].min() == 2 and merges[:, 4].max() == 5
    sess.close()


@pytest.mark.parametrize("q_len", [64, 96, 150, 409])
def test_either_kernel_on_request(q_len):
    # KVP_TUNE_CTA_PAIRS: off, on again; 96 and 150 tokens (384 and 600 rows) have a narrow unit to one or two wide ones
    shape = gen.ModelShape(1, 32, 8, 128, "bf16", 500000.0, 0)
    wl = gen.make_workload(shape, [300, 700], [[(0, 0), (1, 0)]], q_len=q_len, seed=q_len)
    sess = Session(wl)
    sess.assemble()
    for pairs in (0, 1):
        sess.ctx.tune(kvp.TUNE_CTA_PAIRS, pairs)
        check_attention(wl, sess)
        assert on_pairs(sess, q_len) == (pairs == 1 and q_len in (64, 409))
    sess.close()


@pytest.mark.parametrize("lens,q_len,ctas", [([40], 33, 0), ([300, 500], 33, 2), ([300, 500], 64, 0), ([1500], 192, 4)])
def test_first_rows_see_few_keys(lens, q_len, ctas):
    # The first rows of the query block see one key, two, ... of it.  With those keys small and the documents' large, a
    # chunk's exponentials sum to more than 2^8 against such a start (33 tokens: three of the second CTA's warps have no rows).
    shape = gen.ModelShape(1, 32, 8, 128, "bf16", 500000.0, 0)
    wl = gen.make_workload(shape, lens, [[(p, 0) for p in range(len(lens))]], q_len=q_len, seed=23 + q_len)
    wl.k_new[0][:] = gen.to_stored(gen.bf16_bits_to_f32(wl.k_new[0]) * np.float32(0.05), "bf16")
    for i, pk in enumerate(wl.packets):
        pk.k[:] = gen.to_stored(gen.bf16_bits_to_f32(pk.k) * np.float32(1.5 + i), "bf16")
    sess = Session(wl)
    sess.assemble()
    if ctas:
        sess.ctx.tune(kvp.TUNE_SPLIT_TARGET_CTAS, ctas)
    check_attention(wl, sess, flags=kvp.PRECISE_QK)
    assert on_pairs(sess, q_len)
    sess.close()
