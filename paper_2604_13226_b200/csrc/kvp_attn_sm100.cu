// bf16 composed-cache attention (head dimension 128, or 64) for sm_100a: TMA-staged K/V tiles, tcgen05 MMA with TMEM accumulators,
// two query streams per CTA so that the tensor pipe works on one stream while the other is in softmax.
//
// A persistent CTA (one per SM) walks a host-built list of work pieces.  A piece is a contiguous range
// of the key tiles of one unit (<= 256 packed query rows - query token i, head-in-group - of one
// request and kv head).  Key tiles are numbered per unit: the causal tiles of the query's own keys
// first, then the prefix tiles of the plan (staged adapter rows, then documents read in place from
// the pool).  The two streams of a piece are
//   mode 0: query rows [0,128) and [128,256) of the unit, both visiting every key tile of the range;
//   mode 1: the same 128 query rows twice, stream s visiting tiles lo+s, lo+s+2, ...; the two partial
//           results are combined inside the CTA at the end of the piece.
//
//   warps 0-3 / 4-7   softmax of stream 0 / 1: one thread per query row.  S = Q K^T arrives in TMEM;
//                     the thread takes the row max, forms p = exp2((s - m) * scale*log2e), sums it in
//                     fp32, writes P as bf16 back into TMEM over S, and rescales O in TMEM when the
//                     running max moved by more than 2^8.  Both warpgroups run the same compact code
//                     (rolled 32-column chunk loops) so that it stays in the instruction cache.  At the end of a piece it normalises O and
//                     writes the output rows (or an fp32 partial when the unit's keys are split).
//   warps 8-11        Q producer.  Documents keep the keys they were cached with: instead of rotating
//                     every key by Delta (Eq. 1) the 128-row Q tile of a stream is counter-rotated by
//                     -Delta once per document, which leaves every score q.k unchanged.  Each stream has
//                     two Q buffers, so the next document's Q is written while the current one is in use.
//   warp 12           MMA issuer and TMEM owner.  Per stream and step: O += P V of the previous tile,
//                     then S = Q K^T of the next one; the two streams alternate.
//   warp 13           TMA producer: K and V tiles into a 3-stage ring (two 64-column boxes each,
//                     128-byte swizzle), in the order the MMA warp consumes them.
//   warps 14-15       with tail_direct: copy the query block's K/V rows behind the prefix (the append).
//
// Every mbarrier wait is bounded: when it runs out the CTA records a code in the status word, drains
// what it has in flight, frees TMEM and returns.
#include "kvp_attn_common.cuh"

namespace {

constexpr int kThreads = 512;
constexpr int kTmemCols = 512;
constexpr uint32_t kColS = 0, kColO = 256;               // + 128 * stream

// Shared memory and barriers by head dimension D.  With D = 64 a tile is one box: the ring holds twice the stages, and
// the Q buffer's second half takes the rounding remainders of the rotated Q.
template <int D>
struct Cfg {
    static constexpr int kStages = D == 128 ? 3 : 6;
    static constexpr int kTileBytes = KVP_TILE_KEYS * D * 2;
    static constexpr int kOffQ = 0;                               // two rotated-Q buffers per stream: [stream][epoch & 1]
    static constexpr int kOffRing = 4 * kQBufBytes;
    static constexpr int kOffBar = kOffRing + kStages * kTileBytes;
    static constexpr int kOffMl = kOffBar + 256;                  // float2[128]: stream 1's (max, sum) in mode 1
    static constexpr int kSmemBytes = kOffMl + 1024 + 1024;       // + alignment slack
    static constexpr int kVecs = D / 8;                           // 16-byte words of a row
    static constexpr int kCols4 = D / 4;                          // float4 columns of a partial
    // D = 64 carries the rotated Q and P in two bf16 numbers each: the fp32 results of the CUDA-core kernel, which
    // serves this head dimension in small calls, hold for large ones too
    static constexpr bool kSplit = D == 64;
    enum BarIdx { kKvFull = 0, kKvEmpty = kStages, kQFull = 2 * kStages, kQFree = kQFull + 4, kSFull = kQFree + 4,   // Q: [2 * stream + buffer]
                  kPFull = kSFull + 2, kOFull = kPFull + 2, kOFree = kOFull + 2, kMlFull = kOFree + 2, kDrain = kMlFull + 1,
                  kNumBars = kDrain + 1 };
    static_assert(8 * kNumBars <= 248, "barrier block");
};

__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem]
template <int ACC>
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d), "l"(a), "l"(b), "r"(idesc), "n"(ACC)
        : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d), "r"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
// the same without the rows whose bit is set in (x, y, z, w), rows 0-31, 32-63, ...: they keep what they have
__device__ __forceinline__ void mma_ts_rows(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t acc, const uint4 &off)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, {%5, %6, %7, %8}, p;\n\t}"
        ::"r"(d), "r"(a), "l"(b), "r"(idesc), "r"(acc), "r"(off.x), "r"(off.y), "r"(off.z), "r"(off.w)
        : "memory");
}
template <int ACC>
__device__ __forceinline__ void mma_ts_c(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d), "r"(a), "l"(b), "r"(idesc), "n"(ACC)
        : "memory");
}

// Instruction descriptor: bf16 x bf16 -> fp32, M = 128, N = n, A K-major, B K-major or MN-major.
__device__ __forceinline__ uint32_t instr_desc(uint32_t n, uint32_t b_mn_major)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (b_mn_major << 16) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}

// unit tile number of step k of stream s
__device__ __forceinline__ int stream_tile(const Work &w, int s, int k) { return w.lo + (w.mode ? 2 * k + s : k); }

// Position of a K (kv = 0) or V (kv = 1) tile, r-th of the piece, in the piece's load order.
//   mode 0: K0 V0 K1 V1 ...        mode 1: K0 K1 V0 K2 V1 K3 V2 ... V(n-1)
__device__ __forceinline__ int load_seq(int mode, int n, int r, int kv)
{
    if (mode == 0) return 2 * r + kv;
    if (kv == 0) return r == 0 ? 0 : 2 * r - 1;
    return r <= n - 2 ? 2 * r + 2 : 2 * n - 1;
}

struct Cta {
    uint32_t smem_base, bar0, tmem;
    int item_begin, item_end;
    const kvp_work *works;
    __device__ __forceinline__ uint32_t bar(int i) const { return bar0 + 8u * i; }
    // behind the barriers: TMEM address and abort flag
    __device__ __forceinline__ uint32_t tmem_slot() const { return bar0 + 248; }
    __device__ __forceinline__ uint32_t abort_flag() const { return bar0 + 252; }
    __device__ __forceinline__ char *smem() const { return reinterpret_cast<char *>(__cvta_shared_to_generic(smem_base)); }
};

// ---- softmax / correction / epilogue of stream S -------------------------------------------------------
// One thread per query row.  S is read from TMEM in 32-column chunks, once; the chunk loop is rolled and
// shared by both streams so that the code stays resident in the instruction cache.
// Rare path of the softmax: the row's reference max moved up, so everything accumulated against the old
// one shrinks by alpha = 2^(old - new): O in TMEM (when a P V product has been accumulated) and the P
// chunks [0, n_chunks) of the current tile that were already written.  S of this step is complete, hence
// so is the P V product of the previous step: O is quiet.
template <int D>
__device__ __forceinline__ void rescale_row(uint32_t s_addr, uint32_t o_addr, float alpha, int n_chunks, bool with_o)
{
    uint32_t v[32];
    if (with_o) {
#pragma unroll 1
        for (int ch = 0; ch < D / 32; ++ch) {
            tmem_ld32(o_addr + ch * 32, v);
            tc_wait_ld();
            landed32(v);
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * alpha);
            tmem_st32(o_addr + ch * 32, v);
        }
    }
    if (n_chunks > 0) tc_wait_st();                  // the P chunks this thread stored are read back below
#pragma unroll 1
    for (int ch = 0; ch < n_chunks; ++ch) {          // 16 columns of packed bf16 pairs per chunk
        if (Cfg<D>::kSplit) {                        // and 16 of remainders
            tmem_ld32(s_addr + ch * 32, v);
            tc_wait_ld();
            landed32(v);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float x = (__uint_as_float(v[i] << 16) + __uint_as_float(v[16 + i] << 16)) * alpha;
                const float y = (__uint_as_float(v[i] & 0xffff0000u) + __uint_as_float(v[16 + i] & 0xffff0000u)) * alpha;
                v[i] = pack_bf16(x, y);
                v[16 + i] = pack_bf16(x - __uint_as_float(v[i] << 16), y - __uint_as_float(v[i] & 0xffff0000u));
            }
            tmem_st32(s_addr + ch * 32, v);
            continue;
        }
        tmem_ld16(s_addr + ch * 16, v);
        tc_wait_ld();
        landed16(v);
#pragma unroll
        for (int i = 0; i < 16; ++i)
            v[i] = pack_bf16(__uint_as_float(v[i] << 16) * alpha, __uint_as_float(v[i] & 0xffff0000u) * alpha);
        tmem_st16(s_addr + ch * 16, v);
    }
    tc_wait_st();
}

template <int D, bool JOINT>
__device__ __forceinline__ void softmax_role(const Params &p, const Cta &c, const int S, const int t)
{
    using C = Cfg<D>;
    const uint32_t lane_base = (uint32_t)((t >> 5) * 32) << 16;
    const uint32_t s_addr = c.tmem + lane_base + kColS + S * 128;
    const uint32_t o_addr = c.tmem + lane_base + kColO + S * 128;
    const float c2 = p.scale_log2;
    uint32_t ph = 0;                                            // parities: bit 0 S full, bit 1 O full, bit 2 (m, l) full
    uint32_t used = 0;                                          // joint units: pieces in which this stream had tiles
    bool ok = true;

    for (int wi = c.item_begin; wi < c.item_end && ok; ++wi) {
        // what the loop needs of the piece; the rest is read again at its end (registers are short here)
        int steps, first, stride, n_tail, n_total, limit;
        const kvp_tile *tiles;
        int row_b = 0, n_per = 1;                               // joint units: the row's request; causal tiles of each
        bool idle;                                              // none of this warp's rows exists
        {
            const Work w = load_work<JOINT>(p, c.works, wi);
            steps = S == 0 ? w.steps0 : w.steps1;
            first = stream_tile(w, S, 0);
            stride = w.mode ? 2 : 1;
            n_tail = w.n_tail;
            tiles = p.plan.tiles + w.tile_begin - n_tail;
            n_total = p.q_pos0 + w.q_len;
            const int r = w.row_base + (w.mode == 0 ? S * KVP_TILE_ROWS : 0) + t;
            idle = D == 128 && !JOINT && r - t + (t & ~31) >= p.group * w.q_len;
            if (JOINT) {
                tiles = p.joint_tiles - n_tail;
                n_per = w.per;
                row_b = t / (p.group * p.q_len);
                limit = p.q_pos0 + row_token(p, t - row_b * (p.group * p.q_len)) + 1;
            } else {
                limit = p.q_pos0 + (r < p.group * w.q_len ? row_token(p, r) : w.q_len - 1) + 1;     // causal keys this row sees
            }
        }
        if (steps == 0) continue;

        float m_ref = -1e30f, l = 0.f;
        // keys of tile j; joint units: with bit 8 set where the row's request holds the tile
        auto keys_of = [&](int j) {
            if (JOINT) {
                if (j < n_tail) return min(KVP_TILE_KEYS, n_total - j % n_per * KVP_TILE_KEYS) | (j / n_per == row_b ? 256 : 0);
                const int4 g = *reinterpret_cast<const int4 *>(tiles + j);
                return (g.y & 0xffff) | (row_b < 32 && ((uint32_t)g.w >> row_b & 1u) ? 256 : 0);
            }
            return j < n_tail ? min(KVP_TILE_KEYS, n_total - j * KVP_TILE_KEYS) : (int)tiles[j].n_keys;
        };
        int nk_next = keys_of(first);
#pragma unroll 1
        for (int k = 0; k < steps; ++k) {
            const int j = first + k * stride, n_keys = JOINT ? nk_next & 255 : nk_next;
            const bool mine = !JOINT || (nk_next & 256) != 0;
            if (k + 1 < steps) nk_next = keys_of(j + stride);
            ok = mbar_wait(c.bar(C::kSFull + S), ph & 1, c.abort_flag(), p.status, 30 + S);
            ph ^= 1;
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();

            const bool full = n_keys == KVP_TILE_KEYS && j >= n_tail;
            const int lim = j >= n_tail ? n_keys : min(n_keys, limit - (JOINT ? j % n_per : j) * KVP_TILE_KEYS);     // visible keys: [0, lim)
            if (JOINT && k == 0) {
                // P V leaves out the rows that do not hold a tile, so its first product does not set their O
                if (__any_sync(0xffffffffu, !mine && row_b < p.joint_batch)) {
                    if (used > 0) ok = mbar_wait(c.bar(C::kOFree + S), (used - 1) & 1, c.abort_flag(), p.status, 28 + S);   // the piece before has been read
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    tc_fence_after();
                    uint32_t zero[32] = {};
#pragma unroll 1
                    for (int ch = 0; ch < D / 32; ++ch) tmem_st32(o_addr + ch * 32, zero);
                }
                ++used;
            }

            // One pass over S, 32 columns at a time: the exponentials use the reference max carried over from earlier tiles;
            // a chunk's own max is reduced alongside and checked last, so that the two dependency chains overlap.  Only if it
            // exceeds the reference by more than 2^8 (first tile of a piece, or a rare jump) are l, O and the P chunks
            // already written rescaled.
            // a short tile (the end of a document, staged adapter rows) needs P only for the columns P V will read (a row that
            // does not see the tile writes P = 0).  Rows that do not exist have Q = 0, so S = 0, and that serves as P; what
            // stands as P of rows that do not hold a joint tile, P V leaves out.  Launches of few rows are at the power limit
            // like others: 16 tokens over 64 x 2048 (64 rows of 128) 115.4 -> 112.5 us; 16 decode steps of 4 requests over
            // documents of their own (4 rows of 128), 4 layers, 2755 -> 2690, of 8 4800 -> 4680 (7 rows of 28/4 heads 1782, 1788).
            const bool none = JOINT ? !__any_sync(0xffffffffu, mine) : idle;
            const int n_ch = none ? 0 : full ? 4 : max(1, (n_keys + 31) >> 5);
#pragma unroll 1
            for (int ch = 0; ch < n_ch; ++ch) {
                uint32_t v[32], pk[C::kSplit ? 32 : 16];
                auto load = [&] {
                    tmem_ld32(s_addr + ch * 32, v);
                    tc_wait_ld();
                    landed32(v);
                    if (!full && lim < ch * 32 + 32) chunk_mask(v, lim - ch * 32);
                };
                load();
                const float cm = chunk_max(v, -INFINITY);
                float ls = chunk_exp<C::kSplit>(v, c2, m_ref * c2, pk);
                const bool need = mine && (cm - m_ref) * c2 > 8.0f;
                if (__any_sync(0xffffffffu, need)) {
                    const float m_new = need ? cm : m_ref;
                    const float alpha = need ? ex2((m_ref - m_new) * c2) : 1.f;
                    rescale_row<D>(s_addr, o_addr, alpha, ch, k > 0);
                    l *= alpha;
                    m_ref = m_new;
                    load();                                     // this chunk's scores again (P so far lies below them)
                    ls = chunk_exp<C::kSplit>(v, c2, m_ref * c2, pk);
                }
                if (C::kSplit) tmem_st32(s_addr + ch * 32, pk);         // over this chunk's own scores
                else tmem_st16(s_addr + ch * 16, pk);
                if (mine) l += ls;
            }
            tc_wait_st();
            tc_fence_before();
            mbar_arrive(c.bar(C::kPFull + S));
        }
        if (!ok) break;

        // ---- end of the piece: O of this stream is complete once its last P V has landed ----------
        const Work w = load_work<JOINT>(p, c.works, wi);
        const int n_rows = p.group * w.q_len, req = JOINT ? t / n_rows : 0;
        const int r = JOINT ? t - req * n_rows : w.row_base + (w.mode == 0 ? S * KVP_TILE_ROWS : 0) + t;
        const bool valid = JOINT ? req < p.joint_batch : r < n_rows;
        const int qi = valid ? row_token(p, r) : w.q_len - 1, b = JOINT ? req : w.b;
        const int h = w.hk * p.group + (valid ? r - qi * p.group : 0);
        float2 *ml_smem = reinterpret_cast<float2 *>(c.smem() + C::kOffMl);
        ok = mbar_wait(c.bar(C::kOFull + S), (ph >> 1) & 1, c.abort_flag(), p.status, 32 + S);
        ph ^= 2;
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();

        if (w.mode == 1 && S == 1) {
            ml_smem[t] = make_float2(m_ref, l);
            mbar_arrive(c.bar(C::kMlFull));         // stream 0's warpgroup combines and writes
            continue;
        }
        float w0 = 1.f, w1 = 0.f;
        const bool both = (w.mode == 1) && (w.steps1 > 0);
        if (both) {
            ok = mbar_wait(c.bar(C::kMlFull), (ph >> 2) & 1, c.abort_flag(), p.status, 34);
            ph ^= 4;
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            const float2 o = ml_smem[t];
            const float M = fmaxf(m_ref, o.x);
            w0 = ex2((m_ref - M) * c2);
            w1 = ex2((o.x - M) * c2);
            l = w0 * l + w1 * o.y;
            m_ref = M;
        }
        const int slot = S == 0 ? w.slot0 : w.slot1;
        const bool direct = slot < 0;
        if (direct) {
            const float inv = 1.f / l;
            w0 *= inv;
            w1 *= inv;
        }
        // un-normalised (partial slot) or normalised (output rows) O = w0 O_s (+ w1 O_1)
        uint4 *orow_bf = (direct && valid) ? reinterpret_cast<uint4 *>(p.out + (((long long)b * p.q_len + qi) * p.n_q + h) * D) : nullptr;
        // partial slot layout: [D / 4 float4 columns][128 rows], so that a warp's store covers 512 contiguous bytes
        uint4 *orow_f = direct || !valid ? nullptr : reinterpret_cast<uint4 *>(p.partial_o) + (long long)slot * (C::kCols4 * KVP_TILE_ROWS) + t;
#pragma unroll 1
        for (int ch = 0; ch < D / 32; ++ch) {
            uint32_t a[32];
            tmem_ld32(o_addr + ch * 32, a);
            tc_wait_ld();
            landed32(a);
#pragma unroll
            for (int i = 0; i < 32; ++i) a[i] = __float_as_uint(__uint_as_float(a[i]) * w0);
            if (both) {
                uint32_t b2[32];
                tmem_ld32(o_addr + 128 + ch * 32, b2);
                tc_wait_ld();
                landed32(b2);
#pragma unroll
                for (int i = 0; i < 32; ++i) a[i] = __float_as_uint(fmaf(__uint_as_float(b2[i]), w1, __uint_as_float(a[i])));
            }
            if (orow_bf != nullptr) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    uint4 u;
                    u.x = pack_bf16(__uint_as_float(a[8 * i + 0]), __uint_as_float(a[8 * i + 1]));
                    u.y = pack_bf16(__uint_as_float(a[8 * i + 2]), __uint_as_float(a[8 * i + 3]));
                    u.z = pack_bf16(__uint_as_float(a[8 * i + 4]), __uint_as_float(a[8 * i + 5]));
                    u.w = pack_bf16(__uint_as_float(a[8 * i + 6]), __uint_as_float(a[8 * i + 7]));
                    orow_bf[ch * 4 + i] = u;
                }
            } else if (orow_f != nullptr) {
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    orow_f[(ch * 8 + i) * KVP_TILE_ROWS] = make_uint4(a[4 * i], a[4 * i + 1], a[4 * i + 2], a[4 * i + 3]);
            }
        }
        if (direct) {
            if (valid && p.lse != nullptr)
                p.lse[((long long)b * p.n_q + h) * p.q_len + qi] = m_ref * p.scale + logf(l);
        } else if (valid) {
            p.partial_ml[(long long)slot * KVP_TILE_ROWS + t] = make_float2(m_ref, l);
        }
        tc_fence_before();
        mbar_arrive(c.bar(C::kOFree + S));
        if (both) mbar_arrive(c.bar(C::kOFree + 1));
    }
}

// ---- Q producer -----------------------------------------------------------------------------------------
template <int D, bool JOINT>
__device__ __forceinline__ void producer_role(const Params &p, const Cta &c, const int t)
{
    using C = Cfg<D>;
    const bool one_buffer = !C::kSplit && p.precise;
    uint32_t nEp0 = 0, nEp1 = 0;
    bool ok = true;
    for (int wi = c.item_begin; wi < c.item_end && ok; ++wi) {
        const Work w = load_work<JOINT>(p, c.works, wi);
        const int n_rows = p.group * w.q_len;
        const int max_steps = max(w.steps0, w.steps1);
        int prev0 = 0, prev1 = 0;
        auto produce = [&](int s, int rope, uint32_t &nEp) {
            // two buffers per stream taken in turn; in precise mode one (value, remainder) pair, rewritten once
            // the last Q K^T of the epoch before has run
            const int buf = one_buffer ? 0 : (nEp & 1);
            const uint32_t back = one_buffer ? 1u : 2u;      // the epoch that used this buffer last
            if (nEp >= back) {
                const uint32_t par = one_buffer ? (nEp - 1) & 1 : ((nEp >> 1) - 1) & 1;
                ok = mbar_wait(c.bar(C::kQFree + 2 * s + buf), par, c.abort_flag(), p.status, 40 + s);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) return;
            }
            char *qb = c.smem() + C::kOffQ + (2 * s + buf) * kQBufBytes;
            char *qrem = C::kSplit ? qb + kHalfBytes : one_buffer ? qb + kQBufBytes : nullptr;
            if (JOINT) produce_q_joint<D>(p, qb, t, w.hk, rope);
            else produce_q_tile<D>(p, qb, qrem, t, p.q + (long long)w.b * p.q_len * p.n_q * D,
                           w.hk, w.row_base + (w.mode == 0 ? s * KVP_TILE_ROWS : 0), n_rows, rope);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive(c.bar(C::kQFull + 2 * s + buf));
            ++nEp;
        };
        for (int k = 0; k < max_steps && ok; ++k) {
            if (k < w.steps0) {
                const int rope = get_tile<JOINT>(p, w, stream_tile(w, 0, k)).rope;
                if (k == 0 || rope != prev0) produce(0, rope, nEp0);
                prev0 = rope;
            }
            if (ok && k < w.steps1) {
                const int rope = get_tile<JOINT>(p, w, stream_tile(w, 1, k)).rope;
                if (k == 0 || rope != prev1) produce(1, rope, nEp1);
                prev1 = rope;
            }
        }
    }
    pdl_wait();                                               // (a role that gave up early)
}

// ---- append (the two spare warps) -------------------------------------------------------------------------------
// With tail_direct the attention reads the query block's K/V from the caller's tensors; the rows are also copied
// behind the prefix in the workspace, for later calls.  Every unit copies the query tokens whose first packed row
// it holds (for its kv head), in the piece that starts the unit, so the copy is spread over all CTAs; four
// 16-byte words of K and of V are in flight per thread.  Nothing in this launch waits for the copy.
template <int D>
__device__ __forceinline__ void append_role(const Params &p, const Cta &c, const int t)
{
    if (!p.tail_direct) return;
    pdl_wait();
    for (int wi = c.item_begin; wi < c.item_end; ++wi) {
        const Work w = load_work(p, c.works, wi);
        if (w.lo == 0) append_rows<Cfg<D>::kVecs, 64>(p, w, w.row_base, w.mode ? KVP_TILE_ROWS : 2 * KVP_TILE_ROWS, t);
    }
}

// ---- TMA producer (whole warp; lane 0 issues) ----------------------------------------------------------
template <int D, bool JOINT>
__device__ __forceinline__ void tma_role(const Params &p, const Cta &c, const int lane, const CUtensorMap *tm_pool_k,
                                         const CUtensorMap *tm_pool_v, const CUtensorMap *tm_ws_k,
                                         const CUtensorMap *tm_ws_v, const CUtensorMap *tm_knew,
                                         const CUtensorMap *tm_vnew)
{
    using C = Cfg<D>;
    constexpr int kStages = C::kStages, kTileBytes = C::kTileBytes;
    uint32_t ring_n = 0;                                   // loads issued before this piece
    bool ok = true;
    for (int wi = c.item_begin; wi < c.item_end && ok; ++wi) {
        const Work w = load_work<JOINT>(p, c.works, wi);
        const int n_loads = 2 * w.n;
        for (int q0 = 0; q0 < n_loads && ok; q0 += 32) {
            // lane i looks up the tile of load q0 + i
            const int q = q0 + lane;
            int r = 0, kv = 0;
            if (w.mode == 0) { r = q >> 1; kv = q & 1; }
            else if (q == 0) { r = 0; kv = 0; }
            else if (q == n_loads - 1) { r = w.n - 1; kv = 1; }
            else if (q & 1) { r = (q + 1) >> 1; kv = 0; }
            else { r = (q - 2) >> 1; kv = 1; }
            int row0 = 0, src = 0;
            if (q < n_loads) {
                const Tile tl = get_tile<JOINT>(p, w, w.lo + r);
                row0 = tl.row0;
                src = tl.src;
            }
            // its lane issues each load when its turn comes (nothing is handed round: this warp shares its sub-partition's
            // issue slots with softmax warps)
            const CUtensorMap *tm = src == 2 ? (kv ? tm_vnew : tm_knew) : src == 0 ? (kv ? tm_pool_v : tm_pool_k) : (kv ? tm_ws_v : tm_ws_k);
            const int cnt = min(32, n_loads - q0);
            const bool ahead = p.l2_prefetch && w.mode == 0 && lane < cnt && src != 2;
            uint32_t stage = (ring_n + (uint32_t)q0) % kStages, use = (ring_n + (uint32_t)q0) / kStages;
#pragma unroll 1
            for (int i = 0; i < cnt && ok; ++i) {
                if (ahead && lane == i + 4) {              // tiles that come from DRAM: L2 is asked for the one four loads ahead
                    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(tm), "r"(0), "r"(row0), "r"(w.plane) : "memory");
                    if (D == 128)
                        asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(tm), "r"(64), "r"(row0), "r"(w.plane) : "memory");
                }
                if (lane == i) {
                    if (use > 0) ok = mbar_wait(c.bar(C::kKvEmpty + stage), (use - 1) & 1, c.abort_flag(), p.status, 10 + stage);
                    if (ok) {
                        const uint32_t dst = c.smem_base + C::kOffRing + stage * kTileBytes, full = c.bar(C::kKvFull + stage);
                        mbar_expect_tx(full, kTileBytes);
                        if (src != 0) pdl_wait();          // staged or appended rows: a kernel in front may have written them
                        if (src == 2) {
                            tma_load_4d(dst, tm, 0, w.hk, row0, w.b, full);
                            if (D == 128) tma_load_4d(dst + kHalfBytes, tm, 64, w.hk, row0, w.b, full);
                        } else {
                            tma_load_3d(dst, tm, 0, row0, w.plane, full);
                            if (D == 128) tma_load_3d(dst + kHalfBytes, tm, 64, row0, w.plane, full);
                        }
                    }
                }
                ok = __all_sync(0xffffffffu, ok);
                if (++stage == kStages) { stage = 0; ++use; }
            }
        }
        ring_n += (uint32_t)n_loads;
    }
}

// ---- MMA issuer (whole warp, convergent; one elected lane issues) ----------------------------------------------------------------------------
struct MmaStream {
    uint32_t nP, nEpoch, nItems, qbuf;
    int prev_rope, prev_keys;
    uint32_t prev_who;
    Tile cur, nxt;
};

template <int D, bool JOINT>
__device__ __forceinline__ void mma_role(const Params &p, const Cta &c)
{
    using C = Cfg<D>;
    constexpr int kStages = C::kStages, kTileBytes = C::kTileBytes;
    constexpr uint32_t kSteps = D / 16;                       // K-steps of Q K^T
    constexpr uint32_t kRem16 = (C::kSplit ? kHalfBytes : kQBufBytes) >> 4;      // from the rotated Q to its remainders
    const uint32_t idesc_pv = instr_desc(D, 1);
    const bool lead = elect_one();
    const bool one_buffer = !C::kSplit && p.precise, two_part = C::kSplit || p.precise;
    // P of 16 keys (K-step kk) in the score columns: packed pairs one after the other, or per 32 keys 16 columns of
    // pairs and 16 of remainders
    auto p_col = [](int kk) { return C::kSplit ? (kk >> 1) * 32 + (kk & 1) * 8 : kk * 8; };
    MmaStream st[2];
    st[0].nP = st[0].nEpoch = st[0].nItems = st[0].qbuf = 0;
    st[1].nP = st[1].nEpoch = st[1].nItems = st[1].qbuf = 0;
    uint32_t ring_n = 0;
    bool ok = true;

    // ---- mode 1: S_s = Q_s K^T of step k of piece wq (whose loads start at ring position `base`) ---------
    auto issue_qk = [&](auto s_c, const Work &wq, uint32_t base, int k) {
        constexpr int s = decltype(s_c)::value;
        MmaStream &ms = st[s];
        const int n_steps = s == 0 ? wq.steps0 : wq.steps1;
        if (k == 0) {
            ms.prev_rope = 0;
            ms.cur = get_tile<JOINT>(p, wq, stream_tile(wq, s, 0));
            ms.nxt = n_steps > 1 ? get_tile<JOINT>(p, wq, stream_tile(wq, s, 1)) : ms.cur;
        }
        const Tile tl = ms.cur;
        if (k == 0 || tl.rope != ms.prev_rope) {                  // first tile of a document: its own Q buffer
            ms.qbuf = one_buffer ? 0 : (ms.nEpoch & 1);
            ok = mbar_wait(c.bar(C::kQFull + 2 * s + ms.qbuf), (one_buffer ? ms.nEpoch : ms.nEpoch >> 1) & 1, c.abort_flag(), p.status, 20 + s);
            ++ms.nEpoch;
        }
        const int r = wq.mode ? 2 * k + s : k;
        const uint32_t g = base + (uint32_t)load_seq(wq.mode, wq.n, r, 0);
        const uint32_t stage = g % kStages, par = (g / kStages) & 1;
        if (ok) ok = mbar_wait(c.bar(C::kKvFull + stage), par, c.abort_flag(), p.status, 22);
        ok = __all_sync(0xffffffffu, ok);                         // the lanes stay together
        if (!ok) return;
        tc_fence_after();
        const bool last = (k + 1 == n_steps) || (ms.nxt.rope != tl.rope);
        if (lead) {
            const uint32_t n16 = max(16u, (uint32_t)(tl.n_keys + 15) & ~15u);
            const uint32_t idesc = instr_desc(n16, 0);
            const uint32_t q_lo = desc_lo(c.smem_base + C::kOffQ + (2 * s + ms.qbuf) * kQBufBytes, 16);
            const uint32_t k_lo = desc_lo(c.smem_base + C::kOffRing + stage * kTileBytes, 16);
            const uint32_t d = c.tmem + kColS + s * 128;
            mma_ss<0>(d, desc64(q_lo, kDescHi), desc64(k_lo, kDescHi), idesc);
#pragma unroll
            for (int kk = 1; kk < (int)kSteps; ++kk) {                         // 16 columns per step: 32 bytes, second half 16 KB on
                constexpr uint32_t kHalf16 = kHalfBytes >> 4;
                const uint32_t off = (kk >> 2) * kHalf16 + (kk & 3) * 2;
                mma_ss<1>(d, desc64(q_lo + off, kDescHi), desc64(k_lo + off, kDescHi), idesc);
            }
            if (two_part && tl.rope != 0) {                         // + (rounding remainder of the rotated Q) K^T
#pragma unroll
                for (int kk = 0; kk < (int)kSteps; ++kk) {
                    constexpr uint32_t kHalf16 = kHalfBytes >> 4;
                    const uint32_t off = (kk >> 2) * kHalf16 + (kk & 3) * 2;
                    mma_ss<1>(d, desc64(q_lo + kRem16 + off, kDescHi), desc64(k_lo + off, kDescHi), idesc);
                }
            }
            tc_commit(c.bar(C::kSFull + s));
            tc_commit(c.bar(C::kKvEmpty + stage));
            if (last) tc_commit(c.bar(C::kQFree + 2 * s + ms.qbuf));
        }
        __syncwarp();
        ms.prev_rope = tl.rope;
        ms.prev_keys = tl.n_keys;
        if (JOINT) ms.prev_who = tl.who;
        ms.cur = ms.nxt;
        if (k + 2 < n_steps) ms.nxt = get_tile<JOINT>(p, wq, stream_tile(wq, s, k + 2));
    };

    // ---- a piece in mode 0: both streams take every tile; loads arrive K(0) V(0) K(1) V(1) ... -----------------
    // This is the tensor-bound path, and the issuing warp's own instruction time is what bounds it, so
    // the loop is kept short: tile facts (key count, document) are fetched 32 tiles at a time, one per
    // lane, and handed round by shuffle; ring stages advance incrementally; all waits of a block come
    // first, with one vote and one fence.
    const int lane = threadIdx.x & 31;
    auto piece_mode0 = [&](const Work &w) {
        const int n = w.n;
        uint32_t stK = ring_n % kStages, parK = (ring_n / kStages) & 1;                 // K(k), used at step k
        uint32_t stV = (ring_n + 1) % kStages, parV = ((ring_n + 1) / kStages) & 1;     // V(k - 1), used at step k
        auto advance = [](uint32_t &st_, uint32_t &par_) {                              // two loads further on
            st_ += 2;
            if (st_ >= kStages) { st_ -= kStages; par_ ^= 1; }
        };
        int b0 = 0, nk_l = 0, rope_l = 0;
        auto refill = [&](int from) {
            b0 = from;
            if (from + lane < n) {
                const Tile t = get_tile<JOINT>(p, w, w.lo + from + lane);
                nk_l = t.n_keys;
                rope_l = t.rope;
            }
        };
        refill(0);
        int prev_nk = 0, prev_rope = 0;
        for (int k = 0; k <= n && ok; ++k) {
            if (k - b0 == 31) refill(k);                          // tile k + 1 stays inside the batch
            const int nk = __shfl_sync(0xffffffffu, nk_l, k - b0);
            const int rope = __shfl_sync(0xffffffffu, rope_l, k - b0);
            const int rope_n = __shfl_sync(0xffffffffu, rope_l, (k + 1 - b0) & 31);
            const bool newq = (k == 0) || rope != prev_rope;      // first tile of a document: its own Q buffer
            const bool lastq = (k + 1 >= n) || rope_n != rope;
            auto step = [&](auto s_c) {
                constexpr int s = decltype(s_c)::value;
                MmaStream &ms = st[s];
                // ---- waits of the block ---------------------------------------------------------
                if (s == 0) {                                 // the tiles first: they land while P is being formed
                    if (k >= 1) ok = mbar_wait(c.bar(C::kKvFull + stV), parV, c.abort_flag(), p.status, 23);
                    if (k < n && ok) ok = mbar_wait(c.bar(C::kKvFull + stK), parK, c.abort_flag(), p.status, 22);
                }
                if (k >= 1) {
                    if (ok) ok = mbar_wait(c.bar(C::kPFull + s), ms.nP & 1, c.abort_flag(), p.status, 24 + s);
                    ++ms.nP;
                    if (ok && k == 1 && ms.nItems > 0)
                        ok = mbar_wait(c.bar(C::kOFree + s), (ms.nItems - 1) & 1, c.abort_flag(), p.status, 26 + s);
                }
                if (k < n) {
                    if (newq) {
                        ms.qbuf = one_buffer ? 0 : (ms.nEpoch & 1);
                        if (ok) ok = mbar_wait(c.bar(C::kQFull + 2 * s + ms.qbuf), (one_buffer ? ms.nEpoch : ms.nEpoch >> 1) & 1, c.abort_flag(), p.status, 20 + s);
                        ++ms.nEpoch;
                    }
                }
                ok = __all_sync(0xffffffffu, ok);                 // the lanes stay together
                if (!ok) return;
                tc_fence_after();
                if (lead) {
                    if (k >= 1) {
                        // ---- O_s += P_s V of step k-1 ---------------------------------------------------
                        const uint32_t v_lo = desc_lo(c.smem_base + C::kOffRing + stV * kTileBytes, kHalfBytes);
                        const uint32_t pa = c.tmem + kColS + s * 128;
                        const uint32_t oa = c.tmem + kColO + s * 128;
                        if (prev_nk == KVP_TILE_KEYS && k > 1) {
#pragma unroll
                            for (int kk = 0; kk < 8; ++kk) {         // 16 keys per step: V advances 2048 bytes
                                mma_ts_c<1>(oa, pa + p_col(kk), desc64(v_lo + kk * 128, kDescHi), idesc_pv);
                                if (C::kSplit) mma_ts_c<1>(oa, pa + p_col(kk) + 16, desc64(v_lo + kk * 128, kDescHi), idesc_pv);
                            }
                        } else {
                            const int ksteps = max(1, (prev_nk + 15) >> 4);    // an empty tile still initialises O (P = 0)
                            for (int kk = 0; kk < ksteps; ++kk) {
                                mma_ts(oa, pa + p_col(kk), desc64(v_lo + kk * 128, kDescHi), idesc_pv, (k > 1 || kk > 0));
                                if (C::kSplit) mma_ts_c<1>(oa, pa + p_col(kk) + 16, desc64(v_lo + kk * 128, kDescHi), idesc_pv);
                            }
                        }
                        if (s == 1) tc_commit(c.bar(C::kKvEmpty + stV));
                        if (k == n) {
                            tc_commit(c.bar(C::kOFull + s));
                        }
                    }
                    if (k < n) {
                        // ---- S_s = Q_s K^T of step k ----------------------------------------------------
                        const uint32_t n16 = max(16u, (uint32_t)(nk + 15) & ~15u);   
                        const uint32_t idesc = instr_desc(n16, 0);
                        const uint32_t q_lo = desc_lo(c.smem_base + C::kOffQ + (2 * s + ms.qbuf) * kQBufBytes, 16);
                        const uint32_t k_lo = desc_lo(c.smem_base + C::kOffRing + stK * kTileBytes, 16);
                        const uint32_t d = c.tmem + kColS + s * 128;
                        mma_ss<0>(d, desc64(q_lo, kDescHi), desc64(k_lo, kDescHi), idesc);
#pragma unroll
                        for (int kk = 1; kk < (int)kSteps; ++kk) {             // 16 columns per step: 32 bytes, second half 16 KB on
                            constexpr uint32_t kHalf16 = kHalfBytes >> 4;
                            const uint32_t off = (kk >> 2) * kHalf16 + (kk & 3) * 2;
                            mma_ss<1>(d, desc64(q_lo + off, kDescHi), desc64(k_lo + off, kDescHi), idesc);
                        }
                        if (two_part && rope != 0) {                // + (rounding remainder of the rotated Q) K^T
#pragma unroll
                            for (int kk = 0; kk < (int)kSteps; ++kk) {
                                constexpr uint32_t kHalf16 = kHalfBytes >> 4;
                                const uint32_t off = (kk >> 2) * kHalf16 + (kk & 3) * 2;
                                mma_ss<1>(d, desc64(q_lo + kRem16 + off, kDescHi), desc64(k_lo + off, kDescHi), idesc);
                            }
                        }
                        tc_commit(c.bar(C::kSFull + s));
                        if (s == 1) tc_commit(c.bar(C::kKvEmpty + stK));
                        if (lastq) tc_commit(c.bar(C::kQFree + 2 * s + ms.qbuf));
                    }
                }
                __syncwarp();
                if (k == n) ++ms.nItems;
            };
            step(std::integral_constant<int, 0>{});
            if (ok) step(std::integral_constant<int, 1>{});
            if (k >= 1) advance(stV, parV);
            if (k < n) advance(stK, parK);
            prev_nk = nk;
            prev_rope = rope;
        }
    };

    for (int wi = c.item_begin; wi < c.item_end && ok; ++wi) {
        const Work w = load_work<JOINT>(p, c.works, wi);
        if (!JOINT && w.mode == 0) {
            piece_mode0(w);
            ring_n += 2u * (uint32_t)w.n;
            continue;
        }
        // Joint units: a row takes part in P V only where its request holds the tile.  P = 0 is not enough: one infinity or
        // NaN among another request's values would make it NaN.
        int req[4] = {};                                          // requests of the tile's rows lane, 32 + lane, ...
        if (JOINT)
            for (int i = 0; i < 4; ++i) req[i] = (32 * i + lane) / (p.group * p.q_len);
        auto not_held = [&](uint32_t who) {
            uint32_t m[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) m[i] = __ballot_sync(0xffffffffu, req[i] >= 32 || !(who >> (req[i] & 31) & 1u));
            return make_uint4(m[0], m[1], m[2], m[3]);
        };
        const int steps[2] = {w.steps0, w.steps1};
        const int max_steps = max(w.steps0, w.steps1);
        auto block = [&](auto s_c, int k) {
            constexpr int s = decltype(s_c)::value;
            MmaStream &ms = st[s];
            if (k >= 1 && k <= steps[s]) {
                // ---- O_s += P_s V of step k-1 -------------------------------------------------------
                const int r = w.mode ? 2 * (k - 1) + s : k - 1;
                const uint32_t g = ring_n + (uint32_t)load_seq(w.mode, w.n, r, 1);
                const uint32_t stage = g % kStages, par = (g / kStages) & 1;
                ok = mbar_wait(c.bar(C::kKvFull + stage), par, c.abort_flag(), p.status, 23);
                if (ok) ok = mbar_wait(c.bar(C::kPFull + s), ms.nP & 1, c.abort_flag(), p.status, 24 + s);
                ++ms.nP;
                if (ok && k == 1 && ms.nItems > 0)
                    ok = mbar_wait(c.bar(C::kOFree + s), (ms.nItems - 1) & 1, c.abort_flag(), p.status, 26 + s);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) return;
                tc_fence_after();
                const uint4 off = JOINT ? not_held(ms.prev_who) : uint4();
                if (lead) {
                    const uint32_t v_lo = desc_lo(c.smem_base + C::kOffRing + stage * kTileBytes, kHalfBytes);
                    const uint32_t pa = c.tmem + kColS + s * 128;
                    const uint32_t oa = c.tmem + kColO + s * 128;
                    if (JOINT) {
                        const int ksteps = (ms.prev_keys + 15) >> 4;
                        for (int kk = 0; kk < ksteps; ++kk)
                            mma_ts_rows(oa, pa + p_col(kk), desc64(v_lo + kk * 128, kDescHi), idesc_pv, (k > 1 || kk > 0), off);
                    } else if (ms.prev_keys == KVP_TILE_KEYS && k > 1) {
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk) {             // 16 keys per step: V advances 2048 bytes
                            mma_ts_c<1>(oa, pa + p_col(kk), desc64(v_lo + kk * 128, kDescHi), idesc_pv);
                            if (C::kSplit) mma_ts_c<1>(oa, pa + p_col(kk) + 16, desc64(v_lo + kk * 128, kDescHi), idesc_pv);
                        }
                    } else {
                        const int ksteps = max(1, (ms.prev_keys + 15) >> 4);   // an empty tile still initialises O (P = 0)
                        for (int kk = 0; kk < ksteps; ++kk) {
                            mma_ts(oa, pa + p_col(kk), desc64(v_lo + kk * 128, kDescHi), idesc_pv, (k > 1 || kk > 0));
                            if (C::kSplit) mma_ts_c<1>(oa, pa + p_col(kk) + 16, desc64(v_lo + kk * 128, kDescHi), idesc_pv);
                        }
                    }
                    tc_commit(c.bar(C::kKvEmpty + stage));
                    if (k == steps[s]) {
                        tc_commit(c.bar(C::kOFull + s));
                    }
                }
                __syncwarp();
                if (k == steps[s]) ++ms.nItems;
            }
            if (k < steps[s]) issue_qk(s_c, w, ring_n, k);
        };
        for (int k = 0; k <= max_steps && ok; ++k) {
            block(std::integral_constant<int, 0>{}, k);
            if (ok) block(std::integral_constant<int, 1>{}, k);
        }
        ring_n += 2u * (uint32_t)w.n;
    }
    __syncwarp();
    if (!ok) {                      // drain whatever was issued before giving TMEM back
        if (lead) tc_commit(c.bar(C::kDrain));
        const uint64_t t0 = global_ns();
        while (!mbar_try_wait(c.bar(C::kDrain), 0) && global_ns() - t0 < 100000000ull) {}
    }
}

template <int D, int LB, bool JOINT>
__global__ void __launch_bounds__(kThreads, 1)
attn_sm100_kernel(const __grid_constant__ CUtensorMap tm_pool_k, const __grid_constant__ CUtensorMap tm_pool_v,
                  const __grid_constant__ CUtensorMap tm_ws_k, const __grid_constant__ CUtensorMap tm_ws_v,
                  const __grid_constant__ CUtensorMap tm_knew, const __grid_constant__ CUtensorMap tm_vnew,
                  const Params p, const __grid_constant__ kvp_blob<LB> list)
{
    using C = Cfg<D>;
    extern __shared__ char smem_raw[];
    Cta c;
    c.smem_base = (smem_u32(smem_raw) + 1023) & ~1023u;
    c.bar0 = c.smem_base + C::kOffBar;
    release_at_once<LB>(p);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        for (int s = 0; s < C::kStages; ++s) {
            mbar_init(c.bar(C::kKvFull + s), 1);
            mbar_init(c.bar(C::kKvEmpty + s), 1);
        }
        for (int s = 0; s < 4; ++s) {
            mbar_init(c.bar(C::kQFull + s), 128);
            mbar_init(c.bar(C::kQFree + s), 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(c.bar(C::kSFull + s), 1);
            mbar_init(c.bar(C::kPFull + s), 128);
            mbar_init(c.bar(C::kOFull + s), 1);
            mbar_init(c.bar(C::kOFree + s), 128);
        }
        mbar_init(c.bar(C::kMlFull), 128);
        mbar_init(c.bar(C::kDrain), 1);
        st_shared(c.abort_flag(), 0);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 12) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(c.tmem_slot()),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    wait_for_tables<LB>(p, blockIdx.x == 0);
    // from here on: the Q producer, the append and the TMA warp (for anything but pool tiles) wait for the kernel in front;
    // everything else follows from what they deliver
    // (the work list gives every CTA at least one piece)
    const int32_t *cta_begin = p.cta_begin;
    c.works = p.works;
    if (LB > 0) {
        cta_begin = reinterpret_cast<const int32_t *>(&list);
        c.works = reinterpret_cast<const kvp_work *>(reinterpret_cast<const char *>(&list) + p.list_works);
    }
    const int32_t *range = cta_begin + blockIdx.x;
    c.item_begin = LB > 0 ? range[0] : __ldcg(range);
    c.item_end = LB > 0 ? range[1] : __ldcg(range + 1);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    c.tmem = ld_shared(c.tmem_slot());

    if (warp < 8) {
        softmax_role<D, JOINT>(p, c, warp >> 2, tid & 127);
    } else if (warp < 12) {
        producer_role<D, JOINT>(p, c, tid - 256);
    } else {
        if (warp == 12) {
            mma_role<D, JOINT>(p, c);
        } else if (warp == 13) {
            tma_role<D, JOINT>(p, c, lane, &tm_pool_k, &tm_pool_v, &tm_ws_k, &tm_ws_v, &tm_knew, &tm_vnew);
        } else {
            if (LB > 0 && blockIdx.x == 0 && warp == 15) store_list<LB>(p, list, lane);
            append_role<D>(p, c, tid - 448);
        }
    }

    // ---- teardown ------------------------------------------------------------------------------
    if (ld_shared(c.abort_flag())) {                    // let copies still in flight land before the CTA goes away
        const uint64_t t0 = global_ns();
        while (global_ns() - t0 < 200000ull) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 12) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(c.tmem), "r"(kTmemCols) : "memory");
    }
}

// ---- merge of partial results -------------------------------------------------------------------------------
// A partial holds, per 128-row query tile: un-normalised O (fp32, stored [D / 4 float4 columns][128 rows]), the
// running max m of the raw scores and the sum l of exp2((s - m) * c).  Block = 32 rows of one query tile; lanes
// run along rows while reading (coalesced).  The partials of a tile are `n` blocks `stride` apart (the slots of
// a unit cut into pieces: consecutive; the same tile on every rank of a prefix-sharded request: one rank buffer
// apart).  The result is either final - normalised, turned through shared memory so that bf16 output rows are
// written 256 contiguous bytes at a time - or again a partial, in the canonical order of a rank buffer
// [request][kv head][row tile] (KVP_PARTIAL: what a rank hands to the exchange).
struct MergeOut {
    __nv_bfloat16 *out;         // final: [batch][q_len][n_q][D]
    float *lse;
    float4 *part_o;             // or partial: [tiles][D / 4][128] float4 ...
    float2 *part_ml;            // ... and [tiles][128] (m, l)
};

// A block takes 32 rows and one of CS column parts of the tile; the parts of a tile are read U at a time, their O and
// (m, l) together, and folded in by the online rule, so that a tile of up to U parts costs one memory round trip.  CS > 1
// when a launch has few tiles (a short query over a long context: 8 tiles of 19 parts each took 22 us with 32 blocks that
// walked the parts one by one, twice).
template <int D, int CS, int U>
__device__ __forceinline__ void merge_tile(int b, int hk, int row_base, int item_q_len, int n_req, const float4 *po, const float2 *pml,
                                           int n, long long stride_o, long long stride_ml, int q_len, int n_q, int n_kv,
                                           int group, float scale, const MergeOut &mo)
{
    constexpr int kC = D / 32 / CS;                             // float4 columns per warp
    constexpr int kV = D / 64 / CS > 0 ? D / 64 / CS : 1;       // 16-byte words of a row this block writes per thread
    __shared__ uint2 tile[32][D / 4 / CS + 1];
    const int lane = threadIdx.x & 31, wv = threadIdx.x >> 5;
    const int row = blockIdx.y * 32 + lane;                     // row of the 128-row query tile
    const int col0 = CS > 1 ? blockIdx.z * (D / 4 / CS) : 0;    // first float4 column of this block
    // q_len stays the stride of the padded tensors; n_req > 1: the tile holds the rows of requests 0, 1, ... (kvp_joint)
    const int per = group * (item_q_len ? item_q_len : q_len), n_rows = n_req > 1 ? per * n_req : per;
    const float c2 = scale * 1.4426950408889634f;
    // rows behind the request's last one exist in no partial (a decode step fills 4 of 128): nothing to read or write
    if (row_base + (int)blockIdx.y * 32 >= n_rows) return;
    const bool valid = row_base + row < n_rows;
    if (!valid) n = 0;
    float M = -INFINITY;
    float L = 0.f;
    float4 o[kC];
#pragma unroll
    for (int j = 0; j < kC; ++j) o[j] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (int s0 = 0; s0 < n; s0 += U) {
        float2 ml[U];
        float4 a[U][kC];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            ml[u] = make_float2(0.f, 0.f);
            if (s0 + u < n) {
                ml[u] = pml[(s0 + u) * stride_ml + row];
#pragma unroll
                for (int j = 0; j < kC; ++j) a[u][j] = po[(s0 + u) * stride_o + (col0 + wv + 8 * j) * KVP_TILE_ROWS + row];
            }
        }
        float m_new = M;
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (ml[u].y > 0.f) m_new = fmaxf(m_new, ml[u].x);
        if (m_new > M) {
            const float alpha = exp2f((M - m_new) * c2);        // (0 while nothing has been added)
            L *= alpha;
#pragma unroll
            for (int j = 0; j < kC; ++j) { o[j].x *= alpha; o[j].y *= alpha; o[j].z *= alpha; o[j].w *= alpha; }
            M = m_new;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (!(ml[u].y > 0.f)) continue;                     // an empty partial: nothing was visible to this row
            const float w = exp2f((ml[u].x - M) * c2);
            L += w * ml[u].y;
#pragma unroll
            for (int j = 0; j < kC; ++j) {
                o[j].x += w * a[u][j].x; o[j].y += w * a[u][j].y; o[j].z += w * a[u][j].z; o[j].w += w * a[u][j].w;
            }
        }
    }
    if (mo.part_o != nullptr) {                                 // stays a partial: un-normalised, against the max M
        if (!valid) return;
        const long long c = ((long long)b * n_kv + hk) * ((group * q_len + KVP_TILE_ROWS - 1) / KVP_TILE_ROWS) + row_base / KVP_TILE_ROWS;
#pragma unroll
        for (int j = 0; j < kC; ++j) mo.part_o[(c * (D / 4) + col0 + wv + 8 * j) * KVP_TILE_ROWS + row] = o[j];
        if (wv == 0 && col0 == 0) mo.part_ml[c * KVP_TILE_ROWS + row] = make_float2(L > 0.f ? M : -1e30f, L);
        return;
    }
    const float inv = L > 0.f ? 1.f / L : 0.f;
#pragma unroll
    for (int j = 0; j < kC; ++j) {
        uint2 u;
        u.x = pack_bf16(o[j].x * inv, o[j].y * inv);
        u.y = pack_bf16(o[j].z * inv, o[j].w * inv);
        tile[lane][wv + 8 * j] = u;
    }
    const int r = row_base + row;
    if (wv == 0 && col0 == 0 && r < n_rows && mo.lse != nullptr) {
        const int rb = n_req > 1 ? r / per : b, rr = n_req > 1 ? r - rb * per : r;
        mo.lse[((long long)rb * n_q + hk * group + rr % group) * q_len + rr / group] = M * scale + logf(L);
    }
    __syncthreads();
    // 8 threads per output row (4 when the block's part of a row is 64 bytes)
    constexpr int kT = D / 8 / CS / kV;
    const int orow = threadIdx.x / kT, jt = threadIdx.x % kT;
    const int r2 = row_base + blockIdx.y * 32 + orow;
    if (orow < 32 && r2 < n_rows) {
        const int rb = n_req > 1 ? r2 / per : b, rr = n_req > 1 ? r2 - rb * per : r2;
        const int i = rr / group, h = hk * group + rr % group;
        uint4 *dst = reinterpret_cast<uint4 *>(mo.out + (((long long)rb * q_len + i) * n_q + h) * D) + col0 / 2 + kV * jt;
#pragma unroll
        for (int v = 0; v < kV; ++v) {
            const uint2 a0 = tile[orow][2 * (kV * jt + v)], a1 = tile[orow][2 * (kV * jt + v) + 1];
            dst[v] = make_uint4(a0.x, a0.y, a1.x, a1.y);
        }
    }
}

// The partial slots of the units of one launch.  Grid (merge item, 4, CS).
template <int D, int CS, int U>
__global__ void __launch_bounds__(256)
merge_list_kernel(const kvp_merge_item *__restrict__ merges, int list_there, int q_len, int n_q, int n_kv, int group, float scale,
                  const float *__restrict__ part_o, const float2 *__restrict__ part_ml, MergeOut mo)
{
    pdl_launch_dependents();
    if (!list_there) pdl_wait();                                // (no attention launch lies between the list's upload and this)
    PDL_AFTER(merges);
    kvp_merge_item mi;
    int4 *m4 = reinterpret_cast<int4 *>(&mi);                   // (from L2: stored while this launch was being set up)
    m4[0] = __ldcg(reinterpret_cast<const int4 *>(merges + blockIdx.x));
    m4[1] = __ldcg(reinterpret_cast<const int4 *>(merges + blockIdx.x) + 1);
    if (list_there) pdl_wait();
    PDL_AFTER(part_o); PDL_AFTER(part_ml);
    merge_tile<D, CS, U>(mi.b, mi.hk, mi.row_base, mi.pad[0], mi.pad[1], reinterpret_cast<const float4 *>(part_o) + (long long)mi.slot0 * (D / 4 * KVP_TILE_ROWS),
               part_ml + (long long)mi.slot0 * KVP_TILE_ROWS, mi.n_slots, D / 4 * KVP_TILE_ROWS, KVP_TILE_ROWS, q_len, n_q, n_kv,
               group, scale, mo);
}

// The rank buffers of a prefix-sharded request, `n_parts` of them `part_bytes` apart.  Grid (query tile, 4), query
// tiles in the canonical order [request][kv head][row tile].
__global__ void __launch_bounds__(256)
merge_ranks_kernel(const char *__restrict__ parts, int n_parts, long long part_bytes, long long ml_offset, int n_rt, int q_len,
                   int n_q, int n_kv, int group, float scale, MergeOut mo)
{
    const int c = blockIdx.x;
    const int rt = c % n_rt, hk = (c / n_rt) % n_kv, b = c / (n_rt * n_kv);
    merge_tile<128, 1, 4>(b, hk, rt * KVP_TILE_ROWS, 0, 1, reinterpret_cast<const float4 *>(parts) + (long long)c * (32 * KVP_TILE_ROWS),
               reinterpret_cast<const float2 *>(parts + ml_offset) + (long long)c * KVP_TILE_ROWS, n_parts, part_bytes / 16,
               part_bytes / 8, q_len, n_q, n_kv, group, scale, mo);
}

}  // namespace

template <int D>
static cudaError_t prepare()
{
    const cudaFuncAttribute what = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t rc = cudaFuncSetAttribute(attn_sm100_kernel<D, 0, false>, what, Cfg<D>::kSmemBytes);
    if (rc == cudaSuccess) rc = cudaFuncSetAttribute(attn_sm100_kernel<D, KVP_INLINE_SMALL, false>, what, Cfg<D>::kSmemBytes);
    if (rc == cudaSuccess) rc = cudaFuncSetAttribute(attn_sm100_kernel<D, KVP_INLINE_LARGE, false>, what, Cfg<D>::kSmemBytes);
    if (rc == cudaSuccess && D == 128) rc = cudaFuncSetAttribute(attn_sm100_kernel<128, 0, true>, what, Cfg<128>::kSmemBytes);
    return rc;
}
cudaError_t kvp_attn_sm100_prepare(int32_t head_dim) { return head_dim == 64 ? prepare<64>() : prepare<128>(); }

cudaError_t kvp_launch_attn_sm100(const kvp_shape &sh, const kvp_attn2_args &a, const CUtensorMap &tm_pool_k,
                                  const CUtensorMap &tm_pool_v, const CUtensorMap &tm_ws_k,
                                  const CUtensorMap &tm_ws_v, cudaStream_t st)
{
    const Params p = make_params(sh, a);
    // without tail_direct the two query maps are never dereferenced: any valid map will do
    const CUtensorMap &tk = a.tail_direct ? a.tm_knew : tm_ws_k, &tv = a.tail_direct ? a.tm_vnew : tm_ws_v;
    auto go = [&](auto *kernel, int smem, const auto &list) {
        return launch_pdl(kernel, a.n_ctas, kThreads, smem, st, tm_pool_k, tm_pool_v, tm_ws_k, tm_ws_v, tk, tv, p, list);
    };
    const auto *small = reinterpret_cast<const kvp_blob<KVP_INLINE_SMALL> *>(a.list);
    const auto *large = reinterpret_cast<const kvp_blob<KVP_INLINE_LARGE> *>(a.list);
    if (a.joint_batch > 0) return go(attn_sm100_kernel<128, 0, true>, Cfg<128>::kSmemBytes, kvp_blob<0>());
    const int size = !a.list ? 0 : a.list_bytes <= KVP_INLINE_SMALL ? 1 : 2;
    if (sh.head_dim == 64)
        return size == 0   ? go(attn_sm100_kernel<64, 0, false>, Cfg<64>::kSmemBytes, kvp_blob<0>())
               : size == 1 ? go(attn_sm100_kernel<64, KVP_INLINE_SMALL, false>, Cfg<64>::kSmemBytes, *small)
                           : go(attn_sm100_kernel<64, KVP_INLINE_LARGE, false>, Cfg<64>::kSmemBytes, *large);
    return size == 0   ? go(attn_sm100_kernel<128, 0, false>, Cfg<128>::kSmemBytes, kvp_blob<0>())
           : size == 1 ? go(attn_sm100_kernel<128, KVP_INLINE_SMALL, false>, Cfg<128>::kSmemBytes, *small)
                       : go(attn_sm100_kernel<128, KVP_INLINE_LARGE, false>, Cfg<128>::kSmemBytes, *large);
}

cudaError_t kvp_launch_merge_list(const kvp_shape &sh, int32_t q_len, int32_t n_merges, int32_t max_parts, int32_t sm_count, const kvp_merge_item *merges, bool list_there,
                                  const float *partial_o, const float2 *partial_ml, void *out, float *lse,
                                  void *part_out, int64_t part_tiles, cudaStream_t st)
{
    if (n_merges <= 0) return cudaSuccess;
    MergeOut mo;
    mo.out = (__nv_bfloat16 *)out;
    mo.lse = lse;
    mo.part_o = nullptr;
    mo.part_ml = nullptr;
    if (part_out != nullptr) {                                   // KVP_PARTIAL: `out` stays untouched
        mo.part_o = reinterpret_cast<float4 *>(part_out);
        mo.part_ml = reinterpret_cast<float2 *>((char *)part_out + (uint64_t)part_tiles * (32ull * KVP_TILE_ROWS * 16));
    }
    // whole rows per block when that gives two blocks per SM, else quarter rows (halves with head dimension 64).  Whole rows
    // take two parts per round trip, which leaves room for three blocks per SM (70 registers), where four leave it for two
    // (108): pruned documents 220.6 -> 218.2 us, ragged batches 818 -> 807, 4 x 10 x 1024 869 -> 864.  Units are cut into two or
    // three; a long request among short ones into up to seven, which two serve no worse: 10000 + 5 x 1666 tokens over 8
    // layers (five parts) 280.4 -> 279.4, 10000 + 6 x 1250 (six) 271.0 -> 267.9, 30000 + 4 x 5000 (seven) 589, 591.
    const bool few = n_merges * (KVP_TILE_ROWS / 32) < 2 * sm_count;
    auto go = [&](auto *kernel, int cs) {
        return launch_pdl(kernel, dim3(n_merges, KVP_TILE_ROWS / 32, cs), 256, 0, st, merges, (int)list_there, q_len, sh.n_q_heads, sh.n_kv_heads,
                          sh.group, sh.scale, partial_o, partial_ml, mo);
    };
    // 20 parts per round trip where a tile has more than 16 (a unit per kv head: 148 CTAs / 8; a decode layer 52 -> 50 us), 8
    // elsewhere: the longer code cost launches of a few parts 2-5 us, and still lost at 12 parts (63.7 us against 58.2).
    const bool many = max_parts > 16;
    if (sh.head_dim == 64)
        return !few ? go(merge_list_kernel<64, 1, 4>, 1) : many ? go(merge_list_kernel<64, 2, 20>, 2) : go(merge_list_kernel<64, 2, 8>, 2);
    return !few ? go(merge_list_kernel<128, 1, 2>, 1) : many ? go(merge_list_kernel<128, 4, 20>, 4) : go(merge_list_kernel<128, 4, 8>, 4);
}

cudaError_t kvp_launch_merge_ranks(const kvp_shape &sh, int32_t batch, int32_t q_len, const void *parts, int32_t n_parts,
                                   void *out, float *lse, cudaStream_t st)
{
    const int n_rt = (sh.group * q_len + KVP_TILE_ROWS - 1) / KVP_TILE_ROWS;
    const uint64_t tiles = (uint64_t)batch * sh.n_kv_heads * n_rt;
    MergeOut mo;
    mo.out = (__nv_bfloat16 *)out;
    mo.lse = lse;
    mo.part_o = nullptr;
    mo.part_ml = nullptr;
    merge_ranks_kernel<<<dim3((unsigned)tiles, KVP_TILE_ROWS / 32), 256, 0, st>>>(
        (const char *)parts, n_parts, (long long)(tiles * (32ull * KVP_TILE_ROWS * 16 + KVP_TILE_ROWS * 8)),
        (long long)(tiles * (32ull * KVP_TILE_ROWS * 16)), n_rt, q_len, sh.n_q_heads, sh.n_kv_heads, sh.group, sh.scale, mo);
    return cudaGetLastError();
}
