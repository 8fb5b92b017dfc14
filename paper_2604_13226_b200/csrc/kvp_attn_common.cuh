// What the two tcgen05 attention kernels share: parameters, PTX wrappers, work pieces and tiles, the Q producer's tile,
// the softmax of a 32-column chunk, the append.
#pragma once

#include <cuda_bf16.h>

#include <type_traits>

#include "kvp_internal.h"

namespace {

constexpr int kHalfBytes = KVP_TILE_KEYS * 64 * 2;       // 16 KB: one 64-column box of 128 rows
constexpr int kQBufBytes = 2 * kHalfBytes;               // a rotated-Q buffer

struct Params {
    kvp_plan_dev plan;
    uint32_t group_magic;                                     // ceil(2^32 / group): r / group = high word of r * magic
    int q_len, q_pos0, layer, n_q, n_kv, group, pairing;      // q_pos0: tail rows appended by earlier calls
    float scale, scale_log2;
    const int32_t *cta_begin;
    const kvp_work *works;
    const __nv_bfloat16 *q;
    __nv_bfloat16 *out;
    float *lse;
    float *partial_o;
    float2 *partial_ml;
    int32_t *status;
    // tail_direct: the query block's tiles come from k_new / v_new ([batch][q_len][Hkv][d], through their own
    // tensor maps) and the kernel copies those rows into the workspace rows (the append) itself
    int tail_direct;
    // precise: the counter-rotated query is kept as value + rounding remainder (two bf16 tiles per stream, one
    // epoch buffer instead of two) and Q K^T of a rotated tile takes both
    int precise;
    int fresh;                 // the work list was uploaded by the kernel in front, or comes along with this launch
    int plan_there;            // the plan was complete before the launch in front of this one was released
    uint32_t list_bytes, list_works;           // in the latter case: its size, where the pieces begin, and where it is stored for
    uint4 *list_dev;                           // the launches behind this one
    int joint_batch;           // joint units (kvp_joint): their requests, tiles and offsets
    const kvp_tile *joint_tiles;
    const int32_t *joint_ropes;
    // l2_prefetch: the K/V tiles of a unit are read by at most two units of the launch, i.e. they come from DRAM
    // rather than from L2: the TMA warp then asks L2 for each tile a few loads before it fetches it
    int l2_prefetch;
    const uint4 *k_new, *v_new;
    uint4 *ws_k, *ws_v;
    long long ws_rows;
};

// ---- PTX wrappers ---------------------------------------------------------------------------------

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// words of shared memory that several roles look at, by 32-bit address (a generic pointer costs two registers)
__device__ __forceinline__ uint32_t ld_shared(uint32_t a)
{
    uint32_t x;
    asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(x) : "r"(a) : "memory");
    return x;
}
__device__ __forceinline__ void st_shared(uint32_t a, uint32_t x)
{
    asm volatile("st.volatile.shared.u32 [%0], %1;" ::"r"(a), "r"(x) : "memory");
}
__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait.  Returns false when another role has aborted or after ~2 s (then the status word and
// the CTA's abort flag are set).  `code` identifies the wait.
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, uint32_t abort_flag,
                                            int32_t *status, int code)
{
    const uint64_t t0 = global_ns();
    uint32_t it = 0;
    while (true) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((++it & 63u) == 0) {
            if (ld_shared(abort_flag)) return false;
            if (global_ns() - t0 > 2000000000ull) {
                atomicCAS(status, 0, code);
                st_shared(abort_flag, 1);
                return false;
            }
        }
    }
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t abort_flag,
                                          int32_t *status, int code)
{
    if (mbar_try_wait(bar, parity)) return true;
    return mbar_wait_slow(bar, parity, abort_flag, status, code);
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *tm, int x, int y, int z, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(tm), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *tm, int x, int y, int z, int w, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
        ::"r"(dst), "l"(tm), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// The MMA warp runs convergently and one lane, elected once, issues every tcgen05.mma and tcgen05.commit (electing for each
// of them cost the warp issue slots that it shares with softmax warps).
__device__ __forceinline__ bool elect_one()
{
    uint32_t e;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
    return e != 0;
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }


// 64-bit shared-memory matrix descriptors are kept as a constant high word and a low word (start
// address and leading-dimension offset, in 16-byte units) that advances by an immediate per K-step.
__device__ __forceinline__ uint64_t desc64(uint32_t lo, uint32_t hi)
{
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(hi));
    return d;
}
#define KVP_R8(r, o) "=r"(r[o]), "=r"(r[o + 1]), "=r"(r[o + 2]), "=r"(r[o + 3]), "=r"(r[o + 4]), "=r"(r[o + 5]), "=r"(r[o + 6]), "=r"(r[o + 7])
#define KVP_W8(r, o) "r"(r[o]), "r"(r[o + 1]), "r"(r[o + 2]), "r"(r[o + 3]), "r"(r[o + 4]), "r"(r[o + 5]), "r"(r[o + 6]), "r"(r[o + 7])

// 32 TMEM lanes (this warp's) x 32 consecutive 32-bit columns -> 32 registers per thread
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t *r)
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : KVP_R8(r, 0), KVP_R8(r, 8), KVP_R8(r, 16), KVP_R8(r, 24)
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t *r)
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : KVP_R8(r, 0), KVP_R8(r, 8)
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t *r)
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), KVP_W8(r, 0), KVP_W8(r, 8), KVP_W8(r, 16), KVP_W8(r, 24)
        : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t *r)
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), KVP_W8(r, 0), KVP_W8(r, 8)
        : "memory");
}

// tcgen05.ld fills its destination registers asynchronously, until tcgen05.wait::ld.  This empty
// statement, placed after the wait, makes the compiler treat the 32 registers as written there, so that
// no copy of them taken between the load and the wait can be used afterwards.
#define KVP_RW8(r, o) "+r"(r[o]), "+r"(r[o + 1]), "+r"(r[o + 2]), "+r"(r[o + 3]), "+r"(r[o + 4]), "+r"(r[o + 5]), "+r"(r[o + 6]), "+r"(r[o + 7])
__device__ __forceinline__ void landed32(uint32_t *r)
{
    asm volatile("" : KVP_RW8(r, 0), KVP_RW8(r, 8), KVP_RW8(r, 16), KVP_RW8(r, 24)::"memory");
}

__device__ __forceinline__ void landed16(uint32_t *r)
{
    asm volatile("" : KVP_RW8(r, 0), KVP_RW8(r, 8)::"memory");
}

__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float fmax3(float a, float b, float c)
{
    float y;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
    return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// Shared-memory matrix descriptor, 128-byte swizzle, 8-row groups 1024 bytes apart.
//   K-major operand (Q, K): rows are 128-byte lines; the leading-dimension field is unused (1).
//   MN-major operand (V):   the second 64-column block lies `lbo_bytes` further on.
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);   // stride 1024 B, sm_100 version, SWIZZLE_128B
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr, uint32_t lbo_bytes)
{
    return ((addr & 0x3FFFFu) >> 4) | ((lbo_bytes >> 4) << 16);
}
// ---- work pieces and tiles ---------------------------------------------------------------------------

struct Work {
    int b, hk, row_base, mode, lo, n, slot0, slot1;
    int n_tail, tile_begin, tail_row0, plane;
    int steps0, steps1;
    int q_len;                 // query tokens of this request (the call's q_len unless the work record carries its own)
    int per;                   // joint units: causal tiles of each request
};

template <bool JOINT = false>
__device__ __forceinline__ Work load_work(const Params &p, const kvp_work *works, int wi)
{
    const int4 *w4 = reinterpret_cast<const int4 *>(works + wi);
    int4 a, c, e;
    if (p.list_bytes != 0) {                                  // this launch's own parameters
        a = w4[0]; c = w4[1]; e = w4[2];
    } else {                                                  // from L2: the launch in front may have stored the list
        a = __ldcg(w4); c = __ldcg(w4 + 1); e = __ldcg(w4 + 2);
    }
    Work w;
    w.b = a.x; w.hk = a.y; w.row_base = a.z; w.mode = a.w & 0xff;
    w.q_len = (a.w >> 8) ? (a.w >> 8) : p.q_len;
    w.lo = c.x; w.n = c.y; w.slot0 = c.z; w.slot1 = c.w;
    w.tile_begin = e.x;                                       // the plan item's entries, carried in the work record
    w.tail_row0 = e.y;
    if (JOINT) {
        w.per = (p.q_pos0 + p.q_len - 1) / KVP_TILE_KEYS + 1;
        w.n_tail = p.joint_batch * w.per;
    } else {
        const int n_rows = p.group * w.q_len;
        const int last = min(n_rows - 1, w.row_base + (w.mode ? KVP_TILE_ROWS : 2 * KVP_TILE_ROWS) - 1);
        w.n_tail = (p.q_pos0 + last / p.group) / KVP_TILE_KEYS + 1;
    }
    w.plane = p.layer * p.n_kv + w.hk;
    w.steps0 = w.mode ? (w.n + 1) >> 1 : w.n;
    w.steps1 = w.mode ? w.n >> 1 : w.n;
    return w;
}

struct Tile {
    int row0, n_keys, src, rope;
    uint32_t who;              // joint units: the requests that hold the tile, a bit each
};

// tile j of the unit's numbering.  Joint units: the causal tiles of request 0, 1, ..., then the joint prefix tiles, whose
// `rope` is the number of a document run - what makes a new Q tile, as the offset does elsewhere.
template <bool JOINT = false>
__device__ __forceinline__ Tile get_tile(const Params &p, const Work &w, int j)
{
    Tile t;
    if (JOINT && j < w.n_tail) {
        const int b = j / w.per, at = (j - b * w.per) * KVP_TILE_KEYS;
        t.row0 = p.plan.items[b].tail_row0 + at;
        t.n_keys = min(KVP_TILE_KEYS, p.q_pos0 + p.q_len - at);
        t.src = 1;
        t.rope = 0;
        t.who = 1u << b;
    } else if (j < w.n_tail) {
        t.row0 = p.tail_direct ? j * KVP_TILE_KEYS : w.tail_row0 + j * KVP_TILE_KEYS;
        t.n_keys = min(KVP_TILE_KEYS, p.q_pos0 + w.q_len - j * KVP_TILE_KEYS);
        t.src = p.tail_direct ? 2 : 1;               // 2: rows of the caller's k_new / v_new, by query token
        t.rope = 0;
    } else {
        const int4 g = *reinterpret_cast<const int4 *>((JOINT ? p.joint_tiles : p.plan.tiles + w.tile_begin) + (j - w.n_tail));
        t.row0 = g.x;
        t.n_keys = g.y & 0xFFFF;
        t.src = g.y >> 16;
        t.rope = g.z;
        t.who = (uint32_t)g.w;
    }
    return t;
}
// query token of packed row r
__device__ __forceinline__ int row_token(const Params &p, int r) { return p.group == 1 ? r : (int)__umulhi((uint32_t)r, p.group_magic); }

// ---- packed fp32 pairs (two lanes of the FMA pipe per instruction) --------------------------------------
__device__ __forceinline__ uint64_t pair(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpair(uint64_t r, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(r));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ float bf16_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }

// R(-Delta) on two partner chunks of a row (four words of bf16 pairs each); put(word, remainder word, x, y) takes the results.
template <typename Put>
__device__ __forceinline__ void rotate_chunks(int pairing, uint32_t *a, uint32_t *b, uint32_t *ar, uint32_t *br, const float4 *w4,
                                              const Put &put)
{
    if (pairing == 0) {
        // pairs (i, i + D/2): word j of chunk c holds elements 8c+2j, 8c+2j+1; partners in chunk c + kCh
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 w = w4[j];                      // cos, sin of pair 8c+2j; cos, sin of pair 8c+2j+1
            const uint64_t va = pair(bf16_lo(a[j]), bf16_hi(a[j])), vb = pair(bf16_lo(b[j]), bf16_hi(b[j]));
            const uint64_t cc = pair(w.x, w.z), ss = pair(w.y, w.w), ns = pair(-w.y, -w.w);
            float x, y;
            unpair(fma2(vb, ss, mul2(va, cc)), x, y);    // R(-Delta): cos same, sin negated
            put(a[j], ar[j], x, y);
            unpair(fma2(va, ns, mul2(vb, cc)), x, y);
            put(b[j], br[j], x, y);
        }
    } else {
        // pairs (2i, 2i+1): one word each; chunk c holds pairs 4c..4c+3 (w4[0], w4[1]), its partner w4[2], w4[3]
#pragma unroll
        for (int j = 0; j < 4; j += 2) {
            float4 w = w4[j >> 1];
            float x0 = bf16_lo(a[j]), y0 = bf16_hi(a[j]), x1 = bf16_lo(a[j + 1]), y1 = bf16_hi(a[j + 1]);
            put(a[j], ar[j], x0 * w.x + y0 * w.y, y0 * w.x - x0 * w.y);
            put(a[j + 1], ar[j + 1], x1 * w.z + y1 * w.w, y1 * w.z - x1 * w.w);
            w = w4[2 + (j >> 1)];
            x0 = bf16_lo(b[j]); y0 = bf16_hi(b[j]); x1 = bf16_lo(b[j + 1]); y1 = bf16_hi(b[j + 1]);
            put(b[j], br[j], x0 * w.x + y0 * w.y, y0 * w.x - x0 * w.y);
            put(b[j + 1], br[j + 1], x1 * w.z + y1 * w.w, y1 * w.z - x1 * w.w);
        }
    }
}

// The Q producer (128 threads) writes one 128-row query tile, counter-rotated by the offset of rope-table row
// `rope` - q' = R(-Delta) q, which leaves q'.k = q.(R(Delta) k), Eq. 1 moved onto Q - into a rotated-Q buffer
// in the K-major 128-byte-swizzled layout (two 64-column halves of 128 rows x 128 bytes).  Thread t owns
// the 16-byte chunks c = t & 7 and c + 8 (the rotation partners when pairs are (i, i + 64)) of rows
// t >> 3, + 16, + 32, ...  The raw rows go to their place in the buffer by asynchronous copies, all in flight
// together (one memory round trip for the tile, eight threads per 128-byte line); the thread then rotates
// its own chunks in place.
// With `qrem` (precise mode) the remainders r - bf16(r) of the rotated values go, as bf16, to the same places of
// a second tile: q' = hi + rem to about 2^-17, so that the rounding of the re-based operand leaves the scores.
// With D = 64 a row is one 128-byte line of eight chunks: thread t owns chunks c = t & 3 and c + 4 of rows t >> 2, + 32, ...
template <int D>
__device__ __forceinline__ void produce_q_tile(const Params &p, char *qbuf, char *qrem, int t, const __nv_bfloat16 *q_b, int hk,
                                               int row_base, int n_rows, int rope)
{
    constexpr int kCh = D / 16, kRows = 128 / kCh;            // chunks to the rotation partner; rows per pass
    const int c = t & (kCh - 1), r0 = t / kCh;
    const int at = r0 * 128 + ((c ^ (r0 & 7)) << 4);          // row & 7 == r0 & 7 for all of its rows
    char *mine = qbuf + at;
    const int hi_off = D == 128 ? kHalfBytes : (at ^ 64) - at;            // from a chunk to its partner's place
    float4 w4[4];
    if (rope != 0) {
        const float4 *cs = reinterpret_cast<const float4 *>(p.plan.rope + (size_t)rope * (D / 2));   // (cos, sin) pairs
#pragma unroll
        for (int j = 0; j < 4; ++j)
            w4[j] = *(p.pairing == 0 ? cs + c * 4 + j : cs + (c + kCh * (j >> 1)) * 2 + (j & 1));
    }
    pdl_wait();                                              // (plan and work list are there before; the query rows may not be)
#pragma unroll 1
    for (int i = 0; i < kCh; ++i) {
        const int r = row_base + r0 + kRows * i;
        char *lo = mine + i * (kRows * 128);
        if (r < n_rows) {
            const uint4 *src = reinterpret_cast<const uint4 *>(q_b) + ((long long)row_token(p, r) * (p.n_q - p.group) + hk * p.group + r) * (D / 8);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(lo)), "l"(src + c) : "memory");
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(lo + hi_off)), "l"(src + c + kCh) : "memory");
        } else {
            *reinterpret_cast<uint4 *>(lo) = make_uint4(0, 0, 0, 0);
            *reinterpret_cast<uint4 *>(lo + hi_off) = make_uint4(0, 0, 0, 0);
            if (qrem != nullptr) {                           // (scores of what lay there before would move the warp's references)
                char *rl = qrem + (lo - qbuf);
                *reinterpret_cast<uint4 *>(rl) = make_uint4(0, 0, 0, 0);
                *reinterpret_cast<uint4 *>(rl + hi_off) = make_uint4(0, 0, 0, 0);
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (rope == 0) return;
    // word = bf16 pair of (x, y); rem = bf16 pair of what the rounding of the word dropped
    auto rotate = [&](auto rem_c) {
        constexpr bool kRem = decltype(rem_c)::value;
        auto put = [&](uint32_t &word, uint32_t &rem, float x, float y) {
            word = pack_bf16(x, y);
            if (kRem) rem = pack_bf16(x - bf16_lo(word), y - bf16_hi(word));
        };
#pragma unroll 2
        for (int i = 0; i < kCh; ++i) {
            if (row_base + r0 + kRows * i >= n_rows) break;
            char *lo = mine + i * (kRows * 128);
            uint4 qa = *reinterpret_cast<uint4 *>(lo), qb = *reinterpret_cast<uint4 *>(lo + hi_off);
            uint32_t *a = reinterpret_cast<uint32_t *>(&qa);
            uint32_t *b = reinterpret_cast<uint32_t *>(&qb);
            uint4 ra, rb;                                        // remainders
            uint32_t *ar = reinterpret_cast<uint32_t *>(&ra);
            uint32_t *br = reinterpret_cast<uint32_t *>(&rb);
            rotate_chunks(p.pairing, a, b, ar, br, w4, put);
            *reinterpret_cast<uint4 *>(lo) = qa;
            *reinterpret_cast<uint4 *>(lo + hi_off) = qb;
            if (kRem) {
                char *rl = qrem + (lo - qbuf);
                *reinterpret_cast<uint4 *>(rl) = ra;
                *reinterpret_cast<uint4 *>(rl + hi_off) = rb;
            }
        }
    };
    if (qrem != nullptr) rotate(std::integral_constant<bool, true>{});
    else rotate(std::integral_constant<bool, false>{});
}

// The same for a joint unit: row r belongs to request r / (group * q_len) and takes that request's offset of document run
// `run` (0, or a run that the request does not hold: as it is - such rows are masked).
template <int D>
__device__ __forceinline__ void produce_q_joint(const Params &p, char *qbuf, int t, int hk, int run)
{
    constexpr int kCh = D / 16, kRows = 128 / kCh;
    const int c = t & (kCh - 1), r0 = t / kCh, per = p.group * p.q_len, n_rows = p.joint_batch * per;
    const int at = r0 * 128 + ((c ^ (r0 & 7)) << 4);
    const int hi_off = D == 128 ? kHalfBytes : (at ^ 64) - at;
    auto put = [](uint32_t &word, uint32_t &, float x, float y) { word = pack_bf16(x, y); };
#pragma unroll 1
    for (int i = 0; i < kCh; ++i) {
        const int r = r0 + kRows * i;
        uint4 qa = make_uint4(0, 0, 0, 0), qb = qa;
        if (r < n_rows) {
            const int b = r / per, rr = r - b * per, tok = row_token(p, rr);
            const int rope = run == 0 ? 0 : p.joint_ropes[(run - 1) * p.joint_batch + b];
            float4 w4[4];
            if (rope > 0) {
                const float4 *cs = reinterpret_cast<const float4 *>(p.plan.rope + (size_t)rope * (D / 2));
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    w4[j] = *(p.pairing == 0 ? cs + c * 4 + j : cs + (c + kCh * (j >> 1)) * 2 + (j & 1));
            }
            pdl_wait();
            const uint4 *src = reinterpret_cast<const uint4 *>(p.q) +
                               (((long long)b * p.q_len + tok) * p.n_q + hk * p.group + rr - tok * p.group) * (D / 8);
            qa = src[c];
            qb = src[c + kCh];
            if (rope > 0) {
                uint32_t *a = reinterpret_cast<uint32_t *>(&qa), *bb = reinterpret_cast<uint32_t *>(&qb);
                rotate_chunks(p.pairing, a, bb, a, bb, w4, put);
            }
        }
        char *lo = qbuf + at + i * (kRows * 128);
        *reinterpret_cast<uint4 *>(lo) = qa;
        *reinterpret_cast<uint4 *>(lo + hi_off) = qb;
    }
}

// ---- softmax of a chunk: one thread per query row, 32 scores in registers ----------------------------------
__device__ __forceinline__ float chunk_max(const uint32_t *v, float m)
{
    float m0 = m, m1 = m;
#pragma unroll
    for (int i = 0; i < 32; i += 4) {
        m0 = fmax3(m0, __uint_as_float(v[i]), __uint_as_float(v[i + 1]));
        m1 = fmax3(m1, __uint_as_float(v[i + 2]), __uint_as_float(v[i + 3]));
    }
    return fmaxf(m0, m1);
}
__device__ __forceinline__ void chunk_mask(uint32_t *v, int lim)
{
#pragma unroll
    for (int i = 0; i < 32; ++i)
        if (i >= lim) v[i] = 0xff800000u;                  // -inf
}
// A row's reference moves when a score lies more than 2^8 above it.  The sum of the chunk's 32 exponentials, which is formed
// anyway, is above 2^8 then, so up to this sum - below 2^8 by what rounding takes from either for references of 2^20 and less -
// the maximum need not be formed.  4 x 16 documents of 2048, 1024 query tokens: 2200 us, 2270 with 128 (a chunk of many scores
// somewhat above the reference reaches that), 2480 with a maximum of every chunk behind its exponentials; 20 x 8 documents, 28/4
// heads 820, 925, 909 - all three reading the scores from TMEM again; kept in registers they make 1 % of 8 layers over 4 x 10
// documents of 1024 (902 -> 893).
constexpr float kJumpSum = 240.f;
// p = exp2(s*c2 - mc) for 32 scores, packed as bf16 pairs into pk[0..15] (SPLIT: what that rounding dropped, as bf16
// pairs, into pk[16..31]); returns their fp32 sum.
// (Evaluating part of the exponentials by a polynomial on the FMA pipe was measured and lost: the
// extra issue slots cost more than the special-function unit saves.)
template <bool SPLIT>
__device__ __forceinline__ float chunk_exp(const uint32_t *v, float c2, float mc, uint32_t *pk)
{
    const uint64_t c2p = pair(c2, c2), nmc = pair(-mc, -mc);
    uint64_t la = pair(0.f, 0.f), lb = pair(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 32; i += 2) {
        float x0, x1;
        unpair(fma2(pair(__uint_as_float(v[i]), __uint_as_float(v[i + 1])), c2p, nmc), x0, x1);
        const float p0 = ex2(x0), p1 = ex2(x1);
        if (i & 2) lb = add2(lb, pair(p0, p1)); else la = add2(la, pair(p0, p1));
        pk[i >> 1] = pack_bf16(p0, p1);
        if (SPLIT) pk[16 + (i >> 1)] = pack_bf16(p0 - __uint_as_float(pk[i >> 1] << 16), p1 - __uint_as_float(pk[i >> 1] & 0xffff0000u));
    }
    float s0, s1;
    unpair(add2(la, lb), s0, s1);
    return s0 + s1;
}


// ---- append: query tokens whose first packed row is one of [row0, row0 + rows) of a unit ----------------------------
// Copied behind the prefix in the workspace by NT threads, for the unit's kv head; kVecs 16-byte words a row, up to four of
// K and of V in flight per thread.
template <int kVecs, int NT>
__device__ __forceinline__ void append_rows(const Params &p, const Work &w, int row0, int rows, int t)
{
    constexpr int U = 256 / NT;
    const int row_end = min(p.group * w.q_len, row0 + rows);
    const int i0 = (row0 + p.group - 1) / p.group, i1 = (row_end + p.group - 1) / p.group;         // tokens [i0, i1)
    const long long src0 = (((long long)w.b * p.q_len + i0) * p.n_kv + w.hk) * kVecs;
    const long long dst0 = ((long long)w.plane * p.ws_rows + w.tail_row0 + i0) * kVecs;
    const int n_words = (i1 - i0) * kVecs;
    for (int base = 0; base < n_words; base += NT * U) {
        uint4 k[U], v[U];
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const int i = base + j * NT + t;
            if (i < n_words) {
                const long long src = src0 + (long long)(i / kVecs) * p.n_kv * kVecs + i % kVecs;
                k[j] = p.k_new[src];
                v[j] = p.v_new[src];
            }
        }
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const int i = base + j * NT + t;
            if (i < n_words) {
                p.ws_k[dst0 + i] = k[j];
                p.ws_v[dst0 + i] = v[j];
            }
        }
    }
}

// A work list that comes along with the launch (a list in device memory costs a kernel of its own in front, 4 us on the way
// to the first tile) is stored for the launches behind by a warp of one CTA that has nothing to do yet.  That CTA releases
// them behind its store, all others at once; a grid releases when its last CTA has.
template <int LB>
__device__ __forceinline__ void store_list(const Params &p, const kvp_blob<LB> &list, int lane)
{
    pdl_wait();
    for (uint32_t i = lane; i < p.list_bytes / 16; i += 32) p.list_dev[i] = list.w[i];
    __threadfence();
    __syncwarp();
    pdl_launch_dependents();
}

// First of all a launch releases the ones behind it, unless its list is new ...
template <int LB>
__device__ __forceinline__ void release_at_once(const Params &p)
{
    if (LB == 0 && !p.fresh) pdl_launch_dependents();
}
// ... and before it reads tables it waits for those that may not be there, and releases then.  `storing`: this CTA stores the list.
template <int LB>
__device__ __forceinline__ void wait_for_tables(const Params &p, bool storing)
{
    if (LB > 0) {
        if (!p.plan_there) pdl_wait();
        if (!storing) pdl_launch_dependents();
    } else if (p.fresh) {
        pdl_wait();
        pdl_launch_dependents();
    }
}

inline Params make_params(const kvp_shape &sh, const kvp_attn2_args &a)
{
    Params p;
    p.plan = a.plan;
    p.q_len = a.q_len;
    p.q_pos0 = a.q_pos0;
    p.layer = a.layer;
    p.n_q = sh.n_q_heads;
    p.n_kv = sh.n_kv_heads;
    p.group = sh.group;
    p.group_magic = (uint32_t)((0x100000000ull + sh.group - 1) / sh.group);
    p.pairing = sh.pairing;
    p.scale = sh.scale;
    p.scale_log2 = sh.scale * 1.4426950408889634f;
    p.cta_begin = a.cta_begin;
    p.works = a.works;
    p.q = (const __nv_bfloat16 *)a.q;
    p.out = (__nv_bfloat16 *)a.out;
    p.lse = a.lse;
    p.partial_o = a.partial_o;
    p.partial_ml = a.partial_ml;
    p.status = a.status;
    p.tail_direct = a.tail_direct;
    p.precise = a.precise;
    p.fresh = a.fresh;
    p.plan_there = a.plan_there;
    p.list_bytes = a.list_bytes;
    p.list_works = a.list_works;
    p.list_dev = (uint4 *)a.list_dev;
    p.joint_batch = a.joint_batch;
    p.joint_tiles = a.joint_tiles;
    p.joint_ropes = a.joint_ropes;
    p.l2_prefetch = a.l2_prefetch;
    p.k_new = (const uint4 *)a.k_new;
    p.v_new = (const uint4 *)a.v_new;
    p.ws_k = (uint4 *)a.ws_k;
    p.ws_v = (uint4 *)a.ws_v;
    p.ws_rows = sh.ws_rows;
    return p;
}

}  // namespace
