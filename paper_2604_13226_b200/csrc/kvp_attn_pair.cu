// bf16 composed-cache attention for sm_100a, head dimension 128, more than 128 packed query rows per (request, kv head):
// a pair of CTAs works on one unit of 256 rows, CTA r on rows [128 r, 128 r + 128), with tcgen05.mma over both
// (cta_group::2, M = 256).  Each CTA holds its own Q, S, P and O; of every K tile it loads half the keys, of every V tile
// half the columns, and the tensor cores of both read both halves.
//
// Why a pair: with both 128-row tiles of a unit in one CTA, TMEM (512 columns) is full with S and O of two streams, P lies
// over S, and per stream the steps form one chain - Q K^T, softmax, P V, and the next Q K^T only behind that P V - of
// about 3,900 cycles, in which tensor cores and special-function units are busy 2,048 each.  One tile per CTA leaves room
// for three S buffers beside O: Q K^T runs up to three tiles ahead, and the two softmax warpgroups take alternate tiles,
// so that the special-function unit's own 1,024 cycles per tile are what is left in the chain.  K and V traffic per SM
// stays what it was, because the pair shares every tile.
//
//   warps 0-3 / 4-7   softmax of the even / odd tiles of a piece: one thread per query row, exponentials against a
//                     reference maximum m, P as bf16 over S.  O is shared by both warpgroups, so tile k's P has to be
//                     relative to the reference that is in force after tile k - 1: the two warps of a row quadrant hand it
//                     over (mref, an mbarrier per warp).  It rarely changes (only by more than 2^8); then this tile's P
//                     or, once P V of tile k - 1 has landed, O is rescaled.  The second tile of a piece starts from
//                     the maximum of the first one's first 32 keys (another barrier): starting from its own, its P was always
//                     scaled at the hand-over, i.e. rounded twice, and the error of a piece of two or three tiles 1.15 times
//                     as large.
//   warps 8-11        Q producer: counter-rotates this CTA's rows once per document (as in the one-CTA kernel), and appends
//                     the query block's K/V rows
//   warp 12           CTA 0 of the pair: MMA issuer for both.  CTA 1: tells it of the Q tiles formed there.  TMEM owner in each.
//   warp 13           TMA producer of this CTA's halves; its bytes are counted on CTA 0's barriers
//
// Barriers that CTA 0's MMA warp waits for live in CTA 0 and are arrived at from both CTAs; those they signal
// (tcgen05.commit, multicast) exist in both.  Every wait is bounded: when it runs out the status word gets a code, both
// CTAs' abort flags are set and every role leaves.
#include "kvp_attn_common.cuh"

namespace {

constexpr int kThreads = 448;
constexpr int kStageBytes = 16384;                       // half a K or V tile
// Ring and Q buffers share 208 KB: two buffers of 32 KB (value) or 64 KB (value and remainder) and 9 or 5 stages.
constexpr int kMaxStages = 9;
constexpr int kOffBar = 208 * 1024;
constexpr int kOffMref = kOffBar + 512;                   // float[128]
constexpr int kOffStart = kOffMref + 512;                 // float[128]: the reference a piece starts from
constexpr int kOffMl = kOffStart + 512;                   // float2[2][128]: (m, l) of both warpgroups at the end of a piece
constexpr int kSmemBytes = kOffMl + 2048 + 1024;          // + alignment slack
constexpr uint32_t kColO = 384;                           // S buffer b: columns [128 b, 128 b + 128)
constexpr uint16_t kBoth = 3;

enum BarIdx { kKvFull = 0, kKvEmpty = kMaxStages, kQFull = 2 * kMaxStages, kQPeer = kQFull + 2, kQFree = kQPeer + 2, kSFull = kQFree + 2, kPFull = kSFull + 3,
              kOFull = kPFull + 3, kOFree, kMref, kEnd = kMref + 8, kStart = kEnd + 8, kDrain = kStart + 4,      // Mref, End: [4 * warpgroup + quadrant]; Start: [quadrant]
              kNumBars };
static_assert(8 * kNumBars <= 504, "barrier block");

struct Cta {
    uint32_t smem_base, bar0, lead0, tmem;                // lead0: CTA 0's barriers, as an address of the cluster's shared memory
    int rank, item_begin, item_end;
    const kvp_work *works;
    __device__ __forceinline__ uint32_t bar(int i) const { return bar0 + 8u * i; }
    __device__ __forceinline__ uint32_t lead(int i) const { return lead0 + 8u * i; }
    __device__ __forceinline__ uint32_t tmem_slot() const { return bar0 + 504; }
    __device__ __forceinline__ uint32_t abort_flag() const { return bar0 + 508; }
    __device__ __forceinline__ char *smem() const { return reinterpret_cast<char *>(__cvta_shared_to_generic(smem_base)); }
};

__device__ __forceinline__ uint32_t cluster_addr(uint32_t a, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Every warp arrives at the cluster's barrier once its own part of the set-up is done (warp 0: barriers, warp 12: TMEM) and
// waits there only when it has looked up its first piece and tile - the producers when they have formed the first Q tile.
// Pruned documents 240 us with all of it in front of the look-ups, so 230, both with Q released by its producers (the one-CTA
// kernel, where the look-ups lie behind one __syncthreads, lost 1 % with the same order).
__device__ __forceinline__ void begin(Cta &c)
{
    __syncwarp();
    cluster_wait();
    tc_fence_after();
    c.tmem = ld_shared(c.tmem_slot());
}
// For what lies in TMEM, which tcgen05.fence::before_thread_sync orders: a release to the cluster waits for everything the SM
// has in flight, 1,000 cycles and more per tile (it took half of the softmax warps' time).
__device__ __forceinline__ void remote_arrive(uint32_t cluster_bar)
{
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
// For shared memory that this CTA has written: wait_cluster acquires it.
__device__ __forceinline__ void remote_arrive_release(uint32_t cluster_bar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}

// the waits of this kernel; one that runs out also raises the other CTA's abort flag
__device__ __noinline__ bool wait_slow(uint32_t bar, uint32_t parity, uint32_t abort_flag, int rank, int32_t *status, int code)
{
    if (mbar_wait_slow(bar, parity, abort_flag, status, code)) return true;
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr(abort_flag, (uint32_t)(rank ^ 1))), "r"(1u) : "memory");
    return false;
}
__device__ __forceinline__ bool wait(const Params &p, const Cta &c, int i, uint32_t parity, int code)
{
    if (mbar_try_wait(c.bar(i), parity)) return true;
    return wait_slow(c.bar(i), parity, c.abort_flag(), c.rank, p.status, code);
}
// the same, and what the arrives released to the cluster is acquired (a complete phase stays so until this CTA goes on)
__device__ __forceinline__ bool wait_cluster(const Params &p, const Cta &c, int i, uint32_t parity, int code)
{
    if (!wait(p, c, i, parity, code)) return false;
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(c.bar(i)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ void load_3d(uint32_t dst, const CUtensorMap *tm, int x, int y, int z, uint32_t cluster_bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(tm), "r"(x), "r"(y), "r"(z), "r"(cluster_bar)
        : "memory");
}
__device__ __forceinline__ void load_4d(uint32_t dst, const CUtensorMap *tm, int x, int y, int z, int w, uint32_t cluster_bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%2, %3, %4, %5}], [%6];"
        ::"r"(dst), "l"(tm), "r"(x), "r"(y), "r"(z), "r"(w), "r"(cluster_bar)
        : "memory");
}

// arrives at the barrier of this place in both CTAs once the MMAs this thread has issued so far have run
__device__ __forceinline__ void commit_both(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar), "h"(kBoth)
                 : "memory");
}
template <int ACC>
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d), "l"(a), "l"(b), "r"(idesc), "n"(ACC)
        : "memory");
}
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d), "r"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
// bf16 x bf16 -> fp32, M = 256 over the pair, N = n, A K-major, B K-major or MN-major
__device__ __forceinline__ uint32_t instr_desc(uint32_t n, uint32_t b_mn_major)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (b_mn_major << 16) | ((n >> 3) << 17) | ((256u >> 4) << 24);
}
// N of a tile's Q K^T: its keys rounded up to what M = 256 takes; CTA r holds keys [r N / 2, (r + 1) N / 2)
__device__ __forceinline__ int qk_n(int n_keys) { return max(32, (n_keys + 31) & ~31); }

// Loads of a piece with n tiles in the order the MMA warp takes them: Q K^T runs three tiles ahead of P V, so
// K0 K1 K2 V0 K3 V1 K4 ... V(n-1).  Load q is tile r's K (kv = 0) or V (kv = 1).
__device__ __forceinline__ void load_at(int n, int q, int &r, int &kv)
{
    if (q < min(n, 3)) { r = q; kv = 0; }
    else if (q >= n + max(n - 3, 0)) { r = q - n; kv = 1; }
    else { kv = (q - 3) & 1 ? 0 : 1; r = (q - 3) / 2 + (kv ? 0 : 3); }
}
__device__ __forceinline__ int v_load(int n, int r) { return r < n - 3 ? 3 + 2 * r : n + r; }                // which load is tile r's V

// ---- softmax / epilogue of warpgroup G (tiles G, G + 2, ... of a piece) ------------------------------------
// Scales P of a tile (n_chunks x 16 columns of packed pairs) by alpha.
__device__ __forceinline__ void scale_p(uint32_t s_addr, float alpha, int n_chunks)
{
    tc_wait_st();                                         // the P chunks this thread stored are read back
#pragma unroll 1
    for (int ch = 0; ch < n_chunks; ++ch) {
        uint32_t v[16];
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
__device__ __forceinline__ void scale_o(uint32_t o_addr, float alpha)
{
#pragma unroll 1
    for (int ch = 0; ch < 4; ++ch) {
        uint32_t v[32];
        tmem_ld32(o_addr + ch * 32, v);
        tc_wait_ld();
        landed32(v);
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * alpha);
        tmem_st32(o_addr + ch * 32, v);
    }
    tc_wait_st();
}

__device__ __forceinline__ void softmax_role(const Params &p, Cta &c, const int G, const int t)
{
    const int quad = t >> 5;
    const bool lead_lane = (t & 31) == 0;
    const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
    uint32_t o_addr = 0;
    const float c2 = p.scale_log2;
    const uint32_t mref = c.smem_base + kOffMref + 4 * t;
    const int own = 4 * G + quad, other = 4 * (G ^ 1) + quad;         // hand-over barriers of this row quadrant's two warps
    uint32_t T0 = 0;                                      // tiles of the pieces before this one
    uint32_t seen = 0;                                    // the other warp's tiles up to the last one looked at
    uint32_t phO = 0;                                     // pieces
    bool ok = true;

    for (int wi = c.item_begin; wi < c.item_end && ok; ++wi) {
        int n, lo, n_tail, n_total, limit;
        bool idle;                                        // none of this warp's rows exists
        const kvp_tile *tiles;
        {
            const Work w = load_work(p, c.works, wi);
            n = w.n;
            lo = w.lo;
            n_tail = w.n_tail;
            tiles = p.plan.tiles + w.tile_begin - n_tail;
            n_total = p.q_pos0 + w.q_len;
            const int r = w.row_base + c.rank * KVP_TILE_ROWS + t;
            idle = r - t + (t & ~31) >= p.group * w.q_len;
            limit = p.q_pos0 + (r < p.group * w.q_len ? row_token(p, r) : w.q_len - 1) + 1;     // causal keys this row sees
        }
        float m = -1e30f, l = 0.f;
        auto keys_of = [&](int j) {                       // keys of tile j
            return j < n_tail ? min(KVP_TILE_KEYS, n_total - j * KVP_TILE_KEYS) : (int)tiles[j].n_keys;
        };
        int nk_next = G < n ? keys_of(lo + G) : 0;
        if (wi == c.item_begin) {
            begin(c);
            o_addr = c.tmem + lane_base + kColO;
        }
#pragma unroll 1
        for (int k = G; k < n; k += 2) {
            const int j = lo + k, n_keys = nk_next;
            if (k + 2 < n) nk_next = keys_of(j + 2);
            const uint32_t T = T0 + (uint32_t)k, use = T / 3, buf = T - 3 * use;
            const uint32_t s_addr = c.tmem + lane_base + buf * 128;
            ok = wait(p, c, kSFull + buf, use & 1, 30 + G);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            const int lim = j >= n_tail ? n_keys : min(n_keys, limit - j * KVP_TILE_KEYS);       // visible keys: [0, lim)
            // a short tile (the end of a document, staged adapter rows) needs P only for the columns P V will read; rows that
            // do not exist have Q = 0, so S = 0, and that serves as P
            const int n_ch = idle ? 0 : max(1, (n_keys + 31) >> 5);
            if (k < 2) {
                if (k == 0) {
                    // the reference a piece starts from: the maximum of its first 32 keys.  (That of the whole tile, and of the next
                    // one behind a causal block, moves less often: 28/4 heads with outlier channels 1180 -> 1120 us.  Not taken: it
                    // decides which way each probability is rounded, and single outputs moved by 0.14 of the root mean square.)
                    if (!idle) {
                        uint32_t v[32];
                        tmem_ld32(s_addr, v);
                        tc_wait_ld();
                        landed32(v);
                        if (lim < 32) chunk_mask(v, lim);
                        m = chunk_max(v, m);
                    }
                    // (in a place of its own: the second tile may look when this one's reference has moved on)
                    st_shared(mref + kOffStart - kOffMref, __float_as_uint(m));
                    __syncwarp();
                    if (lead_lane) mbar_arrive(c.bar(kStart + quad));
                } else {
                    ok = wait(p, c, kStart + quad, phO & 1, 38);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    m = __uint_as_float(ld_shared(mref + kOffStart - kOffMref));
                }
            }
            // One pass over S, 32 columns at a time, against the reference max this warpgroup knows.  Only if a chunk's max
            // exceeds the reference by more than 2^8 (a rare jump) does the reference move and the P written so far with it;
            // the max is formed only where the chunk's sum leaves room for that (kJumpSum).
#pragma unroll 1
            for (int ch = 0; ch < n_ch; ++ch) {
                uint32_t v[32], pk[16];
                tmem_ld32(s_addr + ch * 32, v);
                tc_wait_ld();
                landed32(v);
                if (lim < ch * 32 + 32) chunk_mask(v, lim - ch * 32);
                float ls = chunk_exp<false>(v, c2, m * c2, pk);
                if (__any_sync(0xffffffffu, !(ls <= kJumpSum))) {
                    const float cm = chunk_max(v, -INFINITY);
                    const bool need = (cm - m) * c2 > 8.0f;
                    if (__any_sync(0xffffffffu, need)) {
                        const float m_new = need ? cm : m;
                        const float alpha = need ? ex2((m - m_new) * c2) : 1.f;
                        scale_p(s_addr, alpha, ch);
                        l *= alpha;
                        m = m_new;
                        ls = chunk_exp<false>(v, c2, m * c2, pk);
                    }
                }
                tmem_st16(s_addr + ch * 16, pk);
                l += ls;
            }
            // the reference in force after tile k - 1
            if (k > 0) {
                ok = wait(p, c, kMref + other, seen & 1, 36);
                ++seen;
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                const float mp = __uint_as_float(ld_shared(mref));
                if (__any_sync(0xffffffffu, mp != m)) {
                    const bool raise = (m - mp) * c2 > 8.0f;              // O follows this tile; else this tile follows O
                    const float ap = raise ? 1.f : ex2((m - mp) * c2), ao = raise ? ex2((mp - m) * c2) : 1.f;
                    scale_p(s_addr, ap, n_ch);
                    l *= ap;
                    if (!raise) m = mp;
                    if (__any_sync(0xffffffffu, raise)) {
                        // O is quiet once P V of tile k - 1 is done, as the stage of that V being free shows: P V of tile k
                        // waits for this warp (so the stage, five or nine loads later in use again, is not free once more)
                        const uint32_t n_stages = p.precise ? 5 : 9, load = 2 * T0 + v_load(n, k - 1);
                        ok = wait(p, c, kKvEmpty + load % n_stages, (load / n_stages) & 1, 37);
                        ok = __all_sync(0xffffffffu, ok);
                        if (!ok) break;
                        tc_fence_after();
                        scale_o(o_addr, ao);
                    }
                }
            }
            st_shared(mref, __float_as_uint(m));
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lead_lane) {
                mbar_arrive(c.bar(kMref + own));
                remote_arrive(c.lead(kPFull + buf));
            }
        }
        T0 += (uint32_t)n;
        if (!ok) break;

        // ---- end of the piece: O is complete once its last P V has landed ----------
        const Work w = load_work(p, c.works, wi);
        ok = wait(p, c, kOFull, phO & 1, 32);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        float2 *ml = reinterpret_cast<float2 *>(c.smem() + kOffMl) + t;
        ml[128 * G] = make_float2(m, l);
        __syncwarp();
        if (lead_lane) mbar_arrive(c.bar(kEnd + own));
        seen += G == 0 ? n / 2 - (n - 1) / 2 : (n + 1) / 2 - n / 2;       // a last tile of the other warp that was not waited for
        ok = wait(p, c, kEnd + other, phO & 1, 34);
        ++phO;
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        const float2 o = ml[128 * (G ^ 1)];
        const float M = ((n - 1) & 1) == G ? m : o.x;     // O is relative to the last tile's reference
        l = l * ex2((m - M) * c2) + o.y * ex2((o.x - M) * c2);

        const int r = w.row_base + c.rank * KVP_TILE_ROWS + t;
        const bool valid = r < p.group * w.q_len;
        const int qi = valid ? row_token(p, r) : w.q_len - 1;
        const int h = w.hk * p.group + (valid ? r - qi * p.group : 0);
        const int slot = c.rank == 0 ? w.slot0 : w.slot1;
        const bool direct = slot < 0;
        const float w0 = direct ? 1.f / l : 1.f;
        // un-normalised (partial slot) or normalised (output rows) O, this warpgroup's half of the columns
        uint4 *orow_bf = (direct && valid) ? reinterpret_cast<uint4 *>(p.out + (((long long)w.b * p.q_len + qi) * p.n_q + h) * 128 + G * 64) : nullptr;
        // partial slot layout: [32 float4 columns][128 rows], so that a warp's store covers 512 contiguous bytes
        uint4 *orow_f = direct || !valid ? nullptr : reinterpret_cast<uint4 *>(p.partial_o) + ((long long)slot * 32 + G * 16) * KVP_TILE_ROWS + t;
#pragma unroll 1
        for (int ch = 0; ch < 2; ++ch) {
            uint32_t a[32];
            tmem_ld32(o_addr + G * 64 + ch * 32, a);
            tc_wait_ld();
            landed32(a);
#pragma unroll
            for (int i = 0; i < 32; ++i) a[i] = __float_as_uint(__uint_as_float(a[i]) * w0);
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
        tc_fence_before();
        __syncwarp();
        if (lead_lane && wi + 1 < c.item_end) remote_arrive(c.lead(kOFree));     // (nobody waits for the last one)
        if (G == 0) {
            if (direct) {
                if (valid && p.lse != nullptr) p.lse[((long long)w.b * p.n_q + h) * p.q_len + qi] = M * p.scale + logf(l);
            } else if (valid) {
                p.partial_ml[(long long)slot * KVP_TILE_ROWS + t] = make_float2(M, l);
            }
        }
    }
}

// ---- Q producer: this CTA's 128 rows, once per document; append ------------------------------------------------
__device__ __forceinline__ void producer_role(const Params &p, Cta &c, const int t)
{
    const uint32_t stride = p.precise ? 2 * kQBufBytes : kQBufBytes;
    uint32_t ep = 0;
    bool ok = true;
    for (int wi = c.item_begin; wi < c.item_end && ok; ++wi) {
        const Work w = load_work(p, c.works, wi);
        const int n_rows = p.group * w.q_len;
        int prev = 0;
        for (int k = 0; k < w.n && ok; ++k) {
            const int rope = get_tile(p, w, w.lo + k).rope;
            if (k > 0 && rope == prev) continue;
            prev = rope;
            const uint32_t buf = ep & 1;
            if (ep >= 2) {
                ok = wait(p, c, kQFree + buf, ((ep >> 1) - 1) & 1, 40);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
            }
            char *qb = c.smem() + buf * stride;
            produce_q_tile<128>(p, qb, p.precise ? qb + kQBufBytes : nullptr, t, p.q + (long long)w.b * p.q_len * p.n_q * 128, w.hk,
                                w.row_base + c.rank * KVP_TILE_ROWS, n_rows, rope);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            if (ep == 0) begin(c);                            // (the first tile is formed while barriers and TMEM are set up)
            __syncwarp();
            if ((t & 31) == 0) mbar_arrive(c.bar(kQFull + buf));
            ++ep;
            // the append (as in the one-CTA kernel): the tokens whose first packed row lies in this CTA's rows, behind the
            // piece's first Q tile
            if (k == 0 && w.lo == 0 && p.tail_direct) append_rows<16, 128>(p, w, w.row_base + c.rank * KVP_TILE_ROWS, KVP_TILE_ROWS, t);
        }
    }
    pdl_wait();                                               // (a role that gave up early)
    // the last arrive at each of this CTA's barriers, see the teardown (so far every one but the last has been waited for)
    for (uint32_t buf = 0; buf < 2 && ok; ++buf)
        if (ep > buf) ok = wait(p, c, kQFree + buf, ((ep - 1 - buf) >> 1) & 1, 41);
}

// ---- Q tiles of CTA 1 (its warp 12) ------------------------------------------------------------------------------
// Their MMAs are issued by a thread of CTA 0, so the tiles are released to the cluster, which takes 1,000 cycles and more: an
// arrive alone orders this CTA's threads only.  From here 4 x 20 documents of 100-200 tokens take 148 us, pruned documents
// 215; the producers themselves held up their next tile with it, 169 and 230.
// `first`: what else this warp has to do, behind the first one.
template <typename First>
__device__ __forceinline__ void peer_role(const Params &p, Cta &c, const int lane, const First &first)
{
    uint32_t ep = 0;
    bool ok = true;
    for (int wi = c.item_begin; wi < c.item_end && ok; ++wi) {
        const Work w = load_work(p, c.works, wi);
        for (int k0 = 0; k0 < w.n && ok; k0 += 32) {
            const int k = k0 + lane;
            const bool newq = k < w.n && (k == 0 || get_tile(p, w, w.lo + k).rope != get_tile(p, w, w.lo + k - 1).rope);
            int count = __popc(__ballot_sync(0xffffffffu, newq));
            if (ep == 0) begin(c);
            for (; count > 0 && ok; --count) {
                ok = wait(p, c, kQFull + (ep & 1), (ep >> 1) & 1, 42);
                ok = __all_sync(0xffffffffu, ok);
                if (ok && lane == 0) remote_arrive_release(c.lead(kQPeer + (ep & 1)));
                if (ep == 0) first();
                ++ep;
            }
        }
    }
}

// ---- TMA producer (whole warp): this CTA's half of every tile ---------------------------------------------------
__device__ __forceinline__ void tma_role(const Params &p, Cta &c, const int lane, const CUtensorMap *k_pool,
                                         const CUtensorMap *v_pool, const CUtensorMap *k_ws, const CUtensorMap *v_ws,
                                         const CUtensorMap *k_new, const CUtensorMap *v_new)
{
    const uint32_t n_stages = p.precise ? 5 : 9;
    const uint32_t ring = c.smem_base + (p.precise ? 4 : 2) * kQBufBytes;
    uint32_t stage = 0, use = 0;
    bool ok = true;
    for (int wi = c.item_begin; wi < c.item_end && ok; ++wi) {
        const Work w = load_work(p, c.works, wi);
        const int n_loads = 2 * w.n;
        for (int q0 = 0; q0 < n_loads && ok; q0 += 32) {
            // lane i looks up the tile of load q0 + i and issues it when its turn comes
            const int q = q0 + lane;
            int row0 = 0, src = 0, kv = 0, n_keys = 0;
            if (q < n_loads) {
                int r;
                load_at(w.n, q, r, kv);
                const Tile tl = get_tile(p, w, w.lo + r);
                row0 = tl.row0;
                src = tl.src;
                n_keys = tl.n_keys;
            }
            const CUtensorMap *tm = src == 2 ? (kv ? v_new : k_new) : src == 0 ? (kv ? v_pool : k_pool) : (kv ? v_ws : k_ws);
            const int x = kv ? 64 * c.rank : 0, y = kv ? row0 : row0 + c.rank * (qk_n(n_keys) / 2);
            const int cnt = min(32, n_loads - q0);
            const bool ahead = p.l2_prefetch && lane < cnt && src != 2;
            if (wi == c.item_begin && q0 == 0) begin(c);
#pragma unroll 1
            for (int i = 0; i < cnt && ok; ++i) {
                if (ahead && lane == i + 4) {             // tiles that come from DRAM: L2 is asked for the one four loads ahead
                    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(tm), "r"(x), "r"(y), "r"(w.plane) : "memory");
                    if (!kv)
                        asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(tm), "r"(64), "r"(y), "r"(w.plane) : "memory");
                }
                if (lane == i) {
                    if (use > 0) ok = wait(p, c, kKvEmpty + stage, (use - 1) & 1, 10);
                    if (ok) {
                        const uint32_t dst = ring + stage * kStageBytes, full = c.lead(kKvFull + stage);
                        if (c.rank == 0) mbar_expect_tx(c.bar(kKvFull + stage), 2 * kStageBytes);
                        if (src != 0) pdl_wait();         // staged or appended rows: a kernel in front may have written them
                        if (src == 2) {
                            load_4d(dst, tm, x, w.hk, y, w.b, full);
                            if (!kv) load_4d(dst + kStageBytes / 2, tm, 64, w.hk, y, w.b, full);
                        } else {
                            load_3d(dst, tm, x, y, w.plane, full);
                            if (!kv) load_3d(dst + kStageBytes / 2, tm, 64, y, w.plane, full);
                        }
                    }
                }
                ok = __all_sync(0xffffffffu, ok);
                if (++stage == n_stages) { stage = 0; ++use; }
            }
        }
    }
    // the last arrive at each of this CTA's barriers, see the teardown
    const uint32_t uses = use + ((uint32_t)lane < stage ? 1 : 0);
    if (ok && (uint32_t)lane < n_stages && uses > 0) wait(p, c, kKvEmpty + lane, (uses - 1) & 1, 11);
}

// ---- MMA issuer (one warp of CTA 0, convergent; one elected lane issues) ----------------------------------------
// Step k of a piece is O += P V of tile k - 3 and S = Q K^T of tile k, which takes over that tile's S buffer.  The MMAs
// wait in a queue that the sub-partition's special-function instructions go through too, so this warp's two softmax
// neighbours are slower than the others (3,000 cycles per tile against 2,400); three issuing warps on three sub-partitions
// in turn evened that out and did not help: the launch is then bound by power (1,000 W) or by the hand-over between them.
__device__ __forceinline__ void mma_role(const Params &p, Cta &c)
{
    const uint32_t n_stages = p.precise ? 5 : 9;
    const uint32_t q_stride = p.precise ? 2 * kQBufBytes : kQBufBytes;
    const uint32_t ring = c.smem_base + (p.precise ? 4 : 2) * kQBufBytes;
    const uint32_t idesc_pv = instr_desc(128, 1);
    const bool lead = elect_one();
    const int lane = threadIdx.x & 31;
    uint32_t stage = 0, par = 0;                          // ring position of the next load to be used
    uint32_t bufS = 0;                                    // S buffer of the next Q K^T
    uint32_t bufP = 0, parP = 0;                          // of the next P V
    uint32_t ep = 0, pieces = 0;
    bool ok = true;
    auto advance = [&] { if (++stage == n_stages) { stage = 0; par ^= 1; } };

    for (int wi = c.item_begin; wi < c.item_end && ok; ++wi) {
        const Work w = load_work(p, c.works, wi);
        const int n = w.n;
        // tile facts are fetched 32 at a time, one per lane, and handed round by shuffle
        int b0 = 0, nk_l = 0, rope_l = 0;
        auto refill = [&](int from) {
            b0 = from;
            if (from + lane < n) {
                const Tile t = get_tile(p, w, w.lo + from + lane);
                nk_l = t.n_keys;
                rope_l = t.rope;
            }
        };
        refill(0);
        if (wi == c.item_begin) begin(c);
        int nk1 = 0, nk2 = 0, nk3 = 0;                    // key counts of the last three tiles
        int prev_rope = 0;
        uint32_t qbuf = 0;
#pragma unroll 1
        for (int k = 0; k < n + 3; ++k) {
            // ---- waits: the tiles first, which land while P is being formed ------------------------------
            int nk = 0, rope = 0;
            bool lastq = false;
            uint32_t stK = stage;                         // K(k) lies behind V(k - 3) in the ring
            if (k >= 3) {
                ok = wait(p, c, kKvFull + stage, par, 23);
                if (++stK == n_stages) stK = 0;
            }
            if (k < n) {
                if (k - b0 == 31) refill(k);              // tile k + 1 stays inside the batch
                nk = __shfl_sync(0xffffffffu, nk_l, k - b0);
                rope = __shfl_sync(0xffffffffu, rope_l, k - b0);
                const int rope_n = __shfl_sync(0xffffffffu, rope_l, (k + 1 - b0) & 31);
                const bool newq = k == 0 || rope != prev_rope;   // first tile of a document: its own Q buffer
                lastq = k + 1 >= n || rope_n != rope;
                prev_rope = rope;
                if (ok) ok = wait(p, c, kKvFull + stK, stK < stage ? par ^ 1 : par, 22);
                if (newq) {
                    qbuf = ep & 1;
                    if (ok) ok = wait(p, c, kQFull + qbuf, (ep >> 1) & 1, 20);
                    if (ok) ok = wait_cluster(p, c, kQPeer + qbuf, (ep >> 1) & 1, 21);
                    ++ep;
                }
            }
            if (k >= 3) {
                if (ok) ok = wait(p, c, kPFull + bufP, parP, 24);
                if (ok && k == 3 && pieces > 0) ok = wait(p, c, kOFree, (pieces - 1) & 1, 26);
            }
            ok = __all_sync(0xffffffffu, ok);             // the lanes stay together
            if (!ok) break;
            tc_fence_after();
            if (k >= 3) {
                // ---- O += P V of tile k - 3 ---------------------------------------------------------
                if (lead) {
                    const uint32_t v_lo = desc_lo(ring + stage * kStageBytes, kHalfBytes);
                    const uint32_t pa = c.tmem + bufP * 128, oa = c.tmem + kColO;
                    if (nk3 == KVP_TILE_KEYS && k > 3) {
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk)           // 16 keys per step: P advances 8 columns, V 2048 bytes
                            mma_ts(oa, pa + kk * 8, desc64(v_lo + kk * 128, kDescHi), idesc_pv, 1);
                    } else {
                        const int ksteps = max(1, (nk3 + 15) >> 4);
                        for (int kk = 0; kk < ksteps; ++kk)
                            mma_ts(oa, pa + kk * 8, desc64(v_lo + kk * 128, kDescHi), idesc_pv, (k > 3 || kk > 0));
                    }
                    commit_both(c.bar(kKvEmpty + stage));
                    if (k == n + 2) commit_both(c.bar(kOFull));
                }
                __syncwarp();
                advance();
                if (++bufP == 3) { bufP = 0; parP ^= 1; }
            }
            if (k < n) {
                // ---- S = Q K^T of tile k ----------------------------------------------------------
                if (lead) {
                    const uint32_t idesc = instr_desc((uint32_t)qk_n(nk), 0);
                    const uint32_t q_lo = desc_lo(c.smem_base + qbuf * q_stride, 16);
                    const uint32_t k_lo = desc_lo(ring + stage * kStageBytes, 16);
                    const uint32_t d = c.tmem + bufS * 128;
                    // 16 columns per step: 32 bytes; the second 64 columns lie 16 KB (Q) and 8 KB (K) on
                    mma_ss<0>(d, desc64(q_lo, kDescHi), desc64(k_lo, kDescHi), idesc);
#pragma unroll
                    for (int kk = 1; kk < 8; ++kk)
                        mma_ss<1>(d, desc64(q_lo + (kk >> 2) * (kHalfBytes >> 4) + (kk & 3) * 2, kDescHi),
                                  desc64(k_lo + (kk >> 2) * (kStageBytes >> 5) + (kk & 3) * 2, kDescHi), idesc);
                    if (p.precise && rope != 0) {                // + (rounding remainder of the rotated Q) K^T
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk)
                            mma_ss<1>(d, desc64(q_lo + (kQBufBytes >> 4) + (kk >> 2) * (kHalfBytes >> 4) + (kk & 3) * 2, kDescHi),
                                      desc64(k_lo + (kk >> 2) * (kStageBytes >> 5) + (kk & 3) * 2, kDescHi), idesc);
                    }
                    commit_both(c.bar(kSFull + bufS));
                    commit_both(c.bar(kKvEmpty + stage));
                    if (lastq) commit_both(c.bar(kQFree + qbuf));
                }
                __syncwarp();
                advance();
                if (++bufS == 3) bufS = 0;
            }
            nk3 = nk2;
            nk2 = nk1;
            nk1 = nk;
        }
        ++pieces;
    }
    __syncwarp();
    if (!ok) {                      // drain whatever was issued before giving TMEM back
        if (lead) asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(c.bar(kDrain)) : "memory");
        const uint64_t t0 = global_ns();
        while (!mbar_try_wait(c.bar(kDrain), 0) && global_ns() - t0 < 100000000ull) {}
    }
}

template <int LB>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
attn_pair_kernel(const __grid_constant__ CUtensorMap k_pool, const __grid_constant__ CUtensorMap v_pool,
                 const __grid_constant__ CUtensorMap k_ws, const __grid_constant__ CUtensorMap v_ws,
                 const __grid_constant__ CUtensorMap k_new, const __grid_constant__ CUtensorMap v_new, const Params p,
                 const __grid_constant__ kvp_blob<LB> list)
{
    extern __shared__ char smem_raw[];
    Cta c;
    c.smem_base = (smem_u32(smem_raw) + 1023) & ~1023u;
    c.bar0 = c.smem_base + kOffBar;
    c.lead0 = cluster_addr(c.bar0, 0);
    c.rank = (int)(blockIdx.x & 1);
    release_at_once<LB>(p);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (warp == 0) {
        for (int i = lane; i < kNumBars; i += 32) {
            uint32_t count = 1;
            if (i >= kQFull && i < kQPeer) count = 4;                   // four producer warps
            else if (i >= kPFull && i < kOFull) count = 8;             // four softmax warps of both CTAs
            else if (i == kOFree) count = 16;                           // eight softmax warps of both CTAs
            mbar_init(c.bar(i), count);
        }
        if (lane == 0) st_shared(c.abort_flag(), 0);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 12) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(c.tmem_slot()) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    __syncwarp();
    tc_fence_before();
    cluster_arrive();
    wait_for_tables<LB>(p, blockIdx.x == 1);
    // from here on: the Q producer, the append and the TMA warp (for anything but pool tiles) wait for the kernel in front;
    // everything else follows from what they deliver
    const int32_t *cta_begin = p.cta_begin;
    c.works = p.works;
    if (LB > 0) {
        cta_begin = reinterpret_cast<const int32_t *>(&list);
        c.works = reinterpret_cast<const kvp_work *>(reinterpret_cast<const char *>(&list) + p.list_works);
    }
    const int32_t *range = cta_begin + (blockIdx.x >> 1);
    c.item_begin = LB > 0 ? range[0] : __ldcg(range);
    c.item_end = LB > 0 ? range[1] : __ldcg(range + 1);
    // (the work list gives every pair a piece; without one the roles would not get to it, and warps arrive twice)
    if (c.item_begin >= c.item_end) begin(c);

    if (warp < 8) {
        softmax_role(p, c, warp >> 2, tid & 127);
    } else if (warp < 12) {
        producer_role(p, c, tid - 256);
    } else if (warp == 12) {
        if (c.rank == 0) {
            mma_role(p, c);
        } else {
            peer_role(p, c, lane, [&] {
                if (LB > 0 && blockIdx.x == 1) store_list<LB>(p, list, lane);
            });
        }
    } else if (warp == 13) {
        tma_role(p, c, lane, &k_pool, &v_pool, &k_ws, &v_ws, &k_new, &v_new);
    }

    // ---- teardown: neither CTA leaves while the other may still reach into it -------------------------------
    if (ld_shared(c.abort_flag())) {        // let copies still in flight land
        const uint64_t t0 = global_ns();
        while (global_ns() - t0 < 200000ull) __nanosleep(1000);
    }
    __syncwarp();
    tc_fence_before();
    // (Every arrive at this CTA's barriers has been waited for, those of the MMAs' completion (kSFull and kOFull by the softmax,
    // kKvEmpty and kQFree to their last phase by the roles that use them) and, but for the last piece's kOFree, which is left
    // out, those of threads of the other CTA: none is under way when this CTA says so.  Relaxed: a release waits for the stores
    // of the partial results, 0.6 us, and nobody here reads them.  Question of 5 x 512 tokens 22.4 -> 22.0 us.)
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    cluster_wait();
    if (warp == 12) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(c.tmem) : "memory");
    }
}

}  // namespace

cudaError_t kvp_attn_pair_prepare(void)
{
    const cudaFuncAttribute what = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t rc = cudaFuncSetAttribute(attn_pair_kernel<0>, what, kSmemBytes);
    if (rc == cudaSuccess) rc = cudaFuncSetAttribute(attn_pair_kernel<KVP_INLINE_SMALL>, what, kSmemBytes);
    if (rc == cudaSuccess) rc = cudaFuncSetAttribute(attn_pair_kernel<KVP_INLINE_LARGE>, what, kSmemBytes);
    return rc;
}

cudaError_t kvp_launch_attn_pair(const kvp_shape &sh, const kvp_attn2_args &a, const CUtensorMap &k_pool, const CUtensorMap &v_pool,
                                 const CUtensorMap &k_ws, const CUtensorMap &v_ws, cudaStream_t st)
{
    // without tail_direct the two query maps are never dereferenced: any valid map will do
    const Params p = make_params(sh, a);
    auto go = [&](auto *kernel, const auto &list) {
        return launch_pdl(kernel, 2 * a.n_ctas, kThreads, kSmemBytes, st, k_pool, v_pool, k_ws, v_ws, a.tail_direct ? a.tm_knew : k_ws,
                          a.tail_direct ? a.tm_vnew : v_ws, p, list);
    };
    if (!a.list) return go(attn_pair_kernel<0>, kvp_blob<0>());
    if (a.list_bytes <= KVP_INLINE_SMALL)
        return go(attn_pair_kernel<KVP_INLINE_SMALL>, *reinterpret_cast<const kvp_blob<KVP_INLINE_SMALL> *>(a.list));
    return go(attn_pair_kernel<KVP_INLINE_LARGE>, *reinterpret_cast<const kvp_blob<KVP_INLINE_LARGE> *>(a.list));
}
