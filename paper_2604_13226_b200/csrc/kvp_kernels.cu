// CUDA-core kernels of the composed-cache path: packet registration (layout change), gather with
// RoPE re-basing (Eq. 1), query K/V append, cache export and an fp32 attention kernel that reads
// packets in place through the tile list.
#include <cuda_bf16.h>

#include <algorithm>

#include "kvp_internal.h"

namespace {

template <typename T> struct Elem;
template <> struct Elem<float> {
    static constexpr int kPerVec = 4;
    __device__ static float to_f32(float x) { return x; }
    __device__ static float from_f32(float x) { return x; }
};
template <> struct Elem<__nv_bfloat16> {
    static constexpr int kPerVec = 8;
    __device__ static float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }
    __device__ static __nv_bfloat16 from_f32(float x) { return __float2bfloat16_rn(x); }
};

template <typename T> union Vec16 {
    uint4 u;
    T e[Elem<T>::kPerVec];
};

// Eq. 1 for one pair: (a, b) -> (a cos - b sin, a sin + b cos), fp32.
__device__ __forceinline__ void rotate_pair(float &a, float &b, float c, float s)
{
    const float ra = a * c - b * s;
    const float rb = a * s + b * c;
    a = ra;
    b = rb;
}

// Rotate the two 16-byte vectors a thread owns.  Half-split pairing: lo holds elements
// [c*EV, c*EV+EV) and hi the partners d/2 further on; interleaved pairing: each vector holds its
// own pairs (2i, 2i+1).  cs points at the (cos, sin) row of this offset.
template <typename T>
__device__ __forceinline__ void rotate_vec_pair(Vec16<T> &lo, Vec16<T> &hi, const float2 *cs, int c, int half_vecs,
                                                int pairing)
{
    constexpr int EV = Elem<T>::kPerVec;
    if (pairing == 0) {
#pragma unroll
        for (int k = 0; k < EV; ++k) {
            const float2 w = cs[c * EV + k];
            float a = Elem<T>::to_f32(lo.e[k]), b = Elem<T>::to_f32(hi.e[k]);
            rotate_pair(a, b, w.x, w.y);
            lo.e[k] = Elem<T>::from_f32(a);
            hi.e[k] = Elem<T>::from_f32(b);
        }
    } else {
#pragma unroll
        for (int k = 0; k < EV; k += 2) {
            float2 w = cs[(c * EV + k) / 2];
            float a = Elem<T>::to_f32(lo.e[k]), b = Elem<T>::to_f32(lo.e[k + 1]);
            rotate_pair(a, b, w.x, w.y);
            lo.e[k] = Elem<T>::from_f32(a);
            lo.e[k + 1] = Elem<T>::from_f32(b);
            w = cs[((c + half_vecs) * EV + k) / 2];
            a = Elem<T>::to_f32(hi.e[k]);
            b = Elem<T>::to_f32(hi.e[k + 1]);
            rotate_pair(a, b, w.x, w.y);
            hi.e[k] = Elem<T>::from_f32(a);
            hi.e[k + 1] = Elem<T>::from_f32(b);
        }
    }
}

// ---- registration: [L][n][Hkv][d] -> plane (l, hk), rows dst_row0 + t ----------------------------
__global__ void store_rows_kernel(const uint4 *__restrict__ src, char *__restrict__ dst, int64_t plane_rows,
                                  int64_t dst_row0, int n_tokens, int n_layers, int n_kv, int vecs_per_row)
{
    const int64_t total = (int64_t)n_layers * n_tokens * n_kv * vecs_per_row;
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(idx % vecs_per_row);
        int64_t r = idx / vecs_per_row;
        const int hk = (int)(r % n_kv);
        r /= n_kv;
        const int t = (int)(r % n_tokens);
        const int l = (int)(r / n_tokens);
        const int64_t drow = ((int64_t)(l * n_kv + hk)) * plane_rows + dst_row0 + t;
        reinterpret_cast<uint4 *>(dst)[drow * vecs_per_row + c] = src[idx];
    }
}

// ---- upload of a plan or work list -------------------------------------------------------------------
// A copy engine's transfer of a few KB takes 3.5 us and leaves 2-3 us on either side of it in a stream of kernels; this
// kernel reads the pinned buffer (up to four 16-byte words per thread in flight) while its predecessor still runs and
// only the stores come after the wait.  5 x 512 tokens, one layer: two uploads, 47 -> 35 us per pass.
__global__ void __launch_bounds__(1024)
upload_kernel(const uint4 *__restrict__ host, uint4 *__restrict__ dst, int n_words, volatile uint32_t *flags, uint32_t seq)
{
    pdl_launch_dependents();
    const int per = (n_words + gridDim.x - 1) / gridDim.x;
    const int end = min(n_words, ((int)blockIdx.x + 1) * per);
    bool waited = false;
    for (int i0 = blockIdx.x * per; i0 < end; i0 += 4096) {
        uint4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * 1024 + threadIdx.x;
            if (i < end) v[u] = __ldcv(host + i);
        }
        if (!waited) pdl_wait();
        waited = true;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * 1024 + threadIdx.x;
            if (i < end) dst[i] = v[u];
        }
    }
    if (!waited) pdl_wait();
    __syncthreads();                             // every word of this block has been read
    if (threadIdx.x == 0) flags[blockIdx.x] = seq;
}

// ---- packets from pinned host memory into the pool, one layer ---------------------------------------------
// A run - one kv head of K or V of a packet - is contiguous on both sides; runs are cut into pieces of 4 KB and the blocks
// take pieces in turn, one thread each, with bulk copies host -> shared memory -> pool in a ring of three.  Bound by the
// host link: reads from the SMs reach 51.2 GB/s whatever the sizes, where a copy per packet, layer and K/V costs 4 us
// beside its transfer (1 MB each: 45.7 GB/s, 256 KB: 28.8; one copy of 128 MB: 55.2).  A block is one warp with 12 KB, so
// that the attention kernel on CTA pairs fits beside it (the one-CTA kernel, with 226 KB, does not).
constexpr int kLoadPiece = 4096, kLoadStages = 3;

__device__ __forceinline__ uint32_t shared_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint64_t now_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__global__ void __launch_bounds__(32)
load_kernel(const __grid_constant__ kvp_load_list list, int layer, int n_kv, int row_bytes, int64_t pool_rows,
            char *__restrict__ pool_k, char *__restrict__ pool_v, int32_t *status)
{
    __shared__ __align__(128) char buf[kLoadStages][kLoadPiece];
    __shared__ uint64_t bars[kLoadStages];
    if (threadIdx.x != 0) return;
    for (int i = 0; i < kLoadStages; ++i)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(shared_addr(&bars[i])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    const int mine = (list.n_pieces - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    int it = 0;                                              // packet of the next piece to fetch
    char *dst[kLoadStages];
    uint32_t size[kLoadStages];
    auto fetch = [&](int k, int stage) {
        const int piece = blockIdx.x + k * gridDim.x;
        while (it + 1 < list.n_items && piece >= list.item[it + 1].piece0) ++it;
        const kvp_load_item &x = list.item[it];
        const int64_t run = (int64_t)x.n * row_bytes;
        const int per_run = (int)((run + kLoadPiece - 1) / kLoadPiece);
        const int r = (piece - x.piece0) / per_run;
        const int64_t off = (int64_t)((piece - x.piece0) % per_run) * kLoadPiece;
        const int head = r % n_kv;
        const bool is_v = r >= n_kv;
        const char *src = (is_v ? x.v : x.k) + ((int64_t)layer * n_kv + head) * run + off;
        dst[stage] = (is_v ? pool_v : pool_k) + (((int64_t)layer * n_kv + head) * pool_rows + x.row0) * row_bytes + off;
        size[stage] = (uint32_t)min((int64_t)kLoadPiece, run - off);
        const uint32_t bar = shared_addr(&bars[stage]);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(size[stage]) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(shared_addr(buf[stage])),
                     "l"(src), "r"(size[stage]), "r"(bar)
                     : "memory");
    };
#pragma unroll
    for (int k = 0; k < kLoadStages; ++k)
        if (k < mine) fetch(k, k);
    bool ok = true;
    for (int k0 = 0; k0 < mine && ok; k0 += kLoadStages) {
#pragma unroll
        for (int s = 0; s < kLoadStages; ++s) {
            const int k = k0 + s;
            if (k >= mine || !ok) break;
            const uint64_t t0 = now_ns();
            uint32_t done = 0;
            while (!done && now_ns() - t0 < 2000000000ull)  // bounded: 2 s
                asm volatile(
                    "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                    : "=r"(done)
                    : "r"(shared_addr(&bars[s])), "r"((uint32_t)(k / kLoadStages) & 1u)
                    : "memory");
            if (!done) {
                atomicCAS(status, 0, 50);
                ok = false;
                break;
            }
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst[s]), "r"(shared_addr(buf[s])), "r"(size[s])
                         : "memory");
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            if (k + kLoadStages < mine) {
                asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");      // the buffer has been read
                fetch(k + kLoadStages, s);
            }
        }
    }
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (!ok)                                                 // let loads still in flight land before the block goes away
        for (const uint64_t t0 = now_ns(); now_ns() - t0 < 200000ull;) {}
}

// (cos, sin) of offset x theta, narrowed to fp32 once: the angle is formed in double precision in half turns (offsets
// reach 1e5 and more), which sincospi reduces exactly.
__device__ __forceinline__ float2 offset_cos_sin(int32_t offset, double half_turn)
{
    double s, c;
    sincospi((double)offset * half_turn, &s, &c);
    return make_float2((float)c, (float)s);
}

// ---- rope table + gather and re-base: pool rows -> workspace rows, all layers and kv heads -----------
// The first n_table blocks form the assembly's (cos, sin) table, 256 entries each; attention reads it.  (On the host it
// cost more than everything else in a call that composes many documents: 129 offsets x 64 angles, 0.2 ms.)  The other
// blocks gather: `groups` of them share a 32-row chunk and take every groups-th plane.  A gather block forms the 64
// angles of its chunk's offset itself, so it waits for no table block.  V is a byte copy, K is a byte copy when the
// offset is 0 and an fp32 rotation otherwise.  Bound by DRAM for a whole cache (materialised), by latency for adapter
// rows; a thread has the loads of two (row, plane) pairs in flight.
// With LB > 0 the plan comes along as a parameter: it is read from there, and block 0 stores it for everyone behind.  Then
// nothing that leads up to a block's first stores has to wait for the kernel in front: the angles and the rows of the pool
// are there by the time it ends (behind a registration, which writes them, the launch waits as a whole).
template <typename T, int LB>
__global__ void __launch_bounds__(256)
gather_kernel(kvp_plan_dev plan, const __grid_constant__ kvp_blob<LB> blob, int blob_words, uint4 *blob_dev, int n_table,
              int n_rope, int groups, const double *__restrict__ half_turns, float2 *__restrict__ table,
              const char *__restrict__ pool_k, const char *__restrict__ pool_v,
              char *__restrict__ ws_k, char *__restrict__ ws_v, int64_t pool_rows, int64_t ws_rows, int vecs_per_row,
              int half_dim, int pairing)
{
    pdl_launch_dependents();
    if (LB > 0) {
        const char *here = reinterpret_cast<const char *>(&blob), *there = reinterpret_cast<const char *>(blob_dev);
        plan.chunks = reinterpret_cast<const kvp_chunk *>(here + (reinterpret_cast<const char *>(plan.chunks) - there));
        plan.delta = reinterpret_cast<const int32_t *>(here + (reinterpret_cast<const char *>(plan.delta) - there));
    } else {
        pdl_wait();
        PDL_AFTER(pool_k); PDL_AFTER(pool_v); PDL_AFTER(plan.chunks); PDL_AFTER(plan.delta);
    }
    if ((int)blockIdx.x < n_table) {
        const int e = blockIdx.x * 256 + threadIdx.x;
        const bool word = LB > 0 && blockIdx.x == 0 && (int)threadIdx.x < blob_words;
        const uint4 mine = word ? blob.w[threadIdx.x] : uint4();
        float2 angle = make_float2(0.f, 0.f);
        if (e < n_rope * half_dim) angle = offset_cos_sin(plan.delta[e / half_dim], half_turns[e % half_dim]);
        if (LB > 0) pdl_wait();
        if (word) blob_dev[threadIdx.x] = mine;
        if (e < n_rope * half_dim) table[e] = angle;
        return;
    }
    __shared__ float2 cs[64];
    const int bi = blockIdx.x - n_table;
    const kvp_chunk ch = plan.chunks[bi / groups];
    const int half_vecs = vecs_per_row / 2;
    if (ch.rope != 0) {
        if ((int)threadIdx.x < half_dim) cs[threadIdx.x] = offset_cos_sin(plan.delta[ch.rope], half_turns[threadIdx.x]);
        __syncthreads();
    }
    const int per_plane = ch.n_rows * half_vecs;
    const int plane0 = bi % groups;
    const int n_items = (plan.n_planes - plane0 + groups - 1) / groups * per_plane;
    for (int w0 = threadIdx.x; w0 < n_items; w0 += 512) {
        Vec16<T> lo[2], hi[2];
        uint4 va[2], vb[2];
        int64_t dst[2];
        int c[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int w = w0 + 256 * u;
            if (w >= n_items) break;
            const int64_t plane = plane0 + (int64_t)(w / per_plane) * groups;
            const int r = w % per_plane;
            const int row = r / half_vecs;
            c[u] = r % half_vecs;
            const int64_t src = (plane * pool_rows + ch.src_row0 + row) * vecs_per_row + c[u];
            dst[u] = (plane * ws_rows + ch.dst_row0 + row) * vecs_per_row + c[u];
            const uint4 *sk = reinterpret_cast<const uint4 *>(pool_k) + src, *sv = reinterpret_cast<const uint4 *>(pool_v) + src;
            lo[u].u = __ldg(sk);
            hi[u].u = __ldg(sk + half_vecs);
            va[u] = __ldg(sv);
            vb[u] = __ldg(sv + half_vecs);
        }
        if (LB > 0 && w0 == (int)threadIdx.x) pdl_wait();
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (w0 + 256 * u >= n_items) break;
            if (ch.rope != 0) rotate_vec_pair<T>(lo[u], hi[u], cs, c[u], half_vecs, pairing);
            uint4 *dk = reinterpret_cast<uint4 *>(ws_k) + dst[u], *dv = reinterpret_cast<uint4 *>(ws_v) + dst[u];
            dk[0] = lo[u].u;
            dk[half_vecs] = hi[u].u;
            dv[0] = va[u];
            dv[half_vecs] = vb[u];
        }
    }
}

// ---- append: the query chunk's own K/V rows go behind the prefix (Section 3.2 step 4) --------------
// grid (batch*q_len); the rows go behind the q_pos0 rows appended earlier; with rope_query the raw
// k_new and q are first rotated to positions prefix_len + q_pos0 + i, angles formed in double precision.
// Latency is all there is (a decode step moves a few KB): a thread takes a pair of 16-byte words - the rotation partners -
// of K and V or of Q, the block is as wide as the token has pairs, and the angles are formed before the wait for the kernel
// in front (plan_there: the plan is complete by then - not so right behind the gather that stores it).  One element at a
// time with the angles first it took 9.4 us of a 75 us decode layer.
template <typename T>
__device__ __forceinline__ Vec16<T> load_vec(const T *p, bool aligned)
{
    Vec16<T> v;
    if (aligned) {
        v.u = *reinterpret_cast<const uint4 *>(p);
    } else {
#pragma unroll
        for (int e = 0; e < Elem<T>::kPerVec; ++e) v.e[e] = p[e];
    }
    return v;
}

template <typename T>
__global__ void __launch_bounds__(512)
append_kernel(kvp_plan_dev plan, int plan_there, int q_len, int q_pos0, const T *__restrict__ q, const T *__restrict__ k_new,
              const T *__restrict__ v_new, char *__restrict__ ws_k, char *__restrict__ ws_v,
              int64_t ws_rows, int layer, int n_q, int n_kv, int d, int pairing, int rope_query,
              const double *__restrict__ half_turns, T *__restrict__ q_rot)
{
    constexpr int EV = Elem<T>::kPerVec;
    __shared__ float2 cs[64];
    pdl_launch_dependents();
    if (!plan_there) pdl_wait();
    PDL_AFTER(plan.items);
    const int b = blockIdx.x / q_len, i = blockIdx.x % q_len;
    const kvp_item it = plan.items[b];
    const int half = d / 2, half_vecs = half / EV, vecs = 2 * half_vecs;
    if (rope_query && (int)threadIdx.x < half) cs[threadIdx.x] = offset_cos_sin(it.prefix_len + q_pos0 + i, half_turns[threadIdx.x]);
    __syncthreads();
    if (plan_there) pdl_wait();
    PDL_AFTER(q); PDL_AFTER(k_new); PDL_AFTER(v_new);
    const int64_t tok = (int64_t)b * q_len + i;
    const bool al_q = ((uintptr_t)q & 15) == 0, al_k = ((uintptr_t)k_new & 15) == 0, al_v = ((uintptr_t)v_new & 15) == 0;
    // keys and values: items [0, n_kv half_vecs); with rope_query the query rows behind them
    const int n_items = (n_kv + (rope_query ? n_q : 0)) * half_vecs;
    for (int w = threadIdx.x; w < n_items; w += blockDim.x) {
        Vec16<T> lo, hi, va, vb;
        const bool kv = w < n_kv * half_vecs;
        const int head = kv ? w / half_vecs : w / half_vecs - n_kv, c = w % half_vecs;
        const T *src = (kv ? k_new + (tok * n_kv + head) * d : q + (tok * n_q + head) * d) + c * EV;
        lo = load_vec<T>(src, kv ? al_k : al_q);
        hi = load_vec<T>(src + half, kv ? al_k : al_q);
        if (kv) {
            const T *vs = v_new + (tok * n_kv + head) * d + c * EV;
            va = load_vec<T>(vs, al_v);
            vb = load_vec<T>(vs + half, al_v);
        }
        if (rope_query) rotate_vec_pair<T>(lo, hi, cs, c, half_vecs, pairing);
        if (kv) {
            const int64_t drow = ((int64_t)(layer * n_kv + head)) * ws_rows + it.tail_row0 + q_pos0 + i;
            uint4 *dk = reinterpret_cast<uint4 *>(ws_k) + drow * vecs + c, *dv = reinterpret_cast<uint4 *>(ws_v) + drow * vecs + c;
            dk[0] = lo.u;
            dk[half_vecs] = hi.u;
            dv[0] = va.u;
            dv[half_vecs] = vb.u;
        } else {
            uint4 *dq = reinterpret_cast<uint4 *>(q_rot) + (tok * n_q + head) * vecs + c;
            dq[0] = lo.u;
            dq[half_vecs] = hi.u;
        }
    }
}

// ---- export of the logical composed cache of one (layer, request) ---------------------------------
// A block takes kExportRows rows of all kv heads: where each row lies is looked up once (prefix rows come from where
// attention reads them: the materialised cache or the staged adapter rows, already re-based, else the pool, rotated
// here), then every thread moves pairs of 16-byte words, two in flight.  The prefix lies there since before the launch (the
// caller sees to that with `early`); only blocks that reach the appended rows need loads that are coherent, which are slower
// (all blocks with them: a handover pass 182 -> 189 us).  Bound by DRAM: one element per thread and one
// row and head per block took 39 us for 9,000 rows of 8 heads of 128 (73 MB), 1.9 TB/s.
constexpr int kExportRows = 16;

template <typename T>
__device__ __forceinline__ void store_vec(T *p, const Vec16<T> &v, bool aligned)
{
    if (aligned) {
        *reinterpret_cast<uint4 *>(p) = v.u;
    } else {
#pragma unroll
        for (int e = 0; e < Elem<T>::kPerVec; ++e) p[e] = v.e[e];
    }
}

template <typename T>
__global__ void __launch_bounds__(256)
export_kernel(kvp_plan_dev plan, int b, int layer, int prefix_len, int n_rows, const char *__restrict__ pool_k,
              const char *__restrict__ pool_v, const char *__restrict__ ws_k,
              const char *__restrict__ ws_v, int64_t pool_rows, int64_t ws_rows, int n_kv, int d,
              int pairing, void *__restrict__ k_out, T *__restrict__ v_out, int k_as_f32)
{
    constexpr int EV = Elem<T>::kPerVec;
    __shared__ int s_row[kExportRows], s_rope[kExportRows], s_pool[kExportRows];
    pdl_launch_dependents();
    pdl_wait();
    PDL_AFTER(pool_k); PDL_AFTER(pool_v); PDL_AFTER(ws_k); PDL_AFTER(ws_v); PDL_AFTER(plan.rope);
    const int t0 = blockIdx.x * kExportRows;
    if (threadIdx.x < kExportRows && t0 + (int)threadIdx.x < n_rows) {
        const int t = t0 + threadIdx.x;
        const kvp_item it = plan.items[b];
        int row, rope = 0, pool = 0;
        if (t >= prefix_len) {
            row = it.tail_row0 + (t - prefix_len);
        } else if (it.cache_row0 >= 0) {
            row = it.cache_row0 + t;
        } else {
            int lo = it.seg_begin, hi = it.seg_end - 1;      // last segment with dst_pos0 <= t
            while (lo < hi) {
                const int mid = (lo + hi + 1) / 2;
                if (plan.segs[mid].dst_pos0 <= t) lo = mid; else hi = mid - 1;
            }
            const kvp_seg sg = plan.segs[lo];
            const int off = t - sg.dst_pos0;
            pool = sg.pad[0] < 0;                            // else staged in the workspace, already re-based
            row = (pool ? sg.src_row0 : sg.pad[0]) + off;
            if (pool) rope = sg.rope;
        }
        s_row[threadIdx.x] = row;
        s_rope[threadIdx.x] = rope;
        s_pool[threadIdx.x] = pool;
    }
    __syncthreads();
    const int half = d / 2, half_vecs = half / EV, vecs = 2 * half_vecs;
    const int n_items = min(kExportRows, n_rows - t0) * n_kv * half_vecs;
    const bool appended = t0 + kExportRows > prefix_len;     // rows that the launch in front may have written
    const bool al_k = ((uintptr_t)k_out & 15) == 0, al_v = ((uintptr_t)v_out & 15) == 0;
    for (int w0 = threadIdx.x; w0 < n_items; w0 += 512) {
        Vec16<T> lo[2], hi[2], va[2], vb[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int w = w0 + 256 * u;
            if (w >= n_items) break;
            const int c = w % half_vecs, hk = w / half_vecs % n_kv, r = w / (half_vecs * n_kv);
            const int64_t src = ((int64_t)(layer * n_kv + hk) * (s_pool[r] ? pool_rows : ws_rows) + s_row[r]) * vecs + c;
            const uint4 *ks = reinterpret_cast<const uint4 *>(s_pool[r] ? pool_k : ws_k) + src;
            const uint4 *vs = reinterpret_cast<const uint4 *>(s_pool[r] ? pool_v : ws_v) + src;
            if (appended) {
                lo[u].u = *ks;
                hi[u].u = *(ks + half_vecs);
                va[u].u = *vs;
                vb[u].u = *(vs + half_vecs);
            } else {
                lo[u].u = __ldg(ks);
                hi[u].u = __ldg(ks + half_vecs);
                va[u].u = __ldg(vs);
                vb[u].u = __ldg(vs + half_vecs);
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int w = w0 + 256 * u;
            if (w >= n_items) break;
            const int c = w % half_vecs, hk = w / half_vecs % n_kv, r = w / (half_vecs * n_kv);
            const int64_t o = ((int64_t)(t0 + r) * n_kv + hk) * d + c * EV;
            const float2 *cs = plan.rope + (size_t)s_rope[r] * half;
            if (k_as_f32) {                                  // the rotation's fp32 result, before narrowing
                float a[EV], x[EV];
#pragma unroll
                for (int e = 0; e < EV; ++e) {
                    a[e] = Elem<T>::to_f32(lo[u].e[e]);
                    x[e] = Elem<T>::to_f32(hi[u].e[e]);
                }
                if (s_rope[r] != 0) {
#pragma unroll
                    for (int e = 0; e < EV; ++e) {
                        if (pairing == 0) {
                            rotate_pair(a[e], x[e], cs[c * EV + e].x, cs[c * EV + e].y);
                        } else if (e % 2 == 0) {
                            const float2 p = cs[(c * EV + e) / 2], p2 = cs[(half + c * EV + e) / 2];
                            rotate_pair(a[e], a[e + 1], p.x, p.y);
                            rotate_pair(x[e], x[e + 1], p2.x, p2.y);
                        }
                    }
                }
                float *ko = reinterpret_cast<float *>(k_out) + o;
#pragma unroll
                for (int e = 0; e < EV; ++e) {
                    ko[e] = a[e];
                    ko[half + e] = x[e];
                }
            } else {
                if (s_rope[r] != 0) rotate_vec_pair<T>(lo[u], hi[u], cs, c, half_vecs, pairing);
                store_vec<T>(reinterpret_cast<T *>(k_out) + o, lo[u], al_k);
                store_vec<T>(reinterpret_cast<T *>(k_out) + o + half, hi[u], al_k);
            }
            store_vec<T>(v_out + o, va[u], al_v);
            store_vec<T>(v_out + o + half, vb[u], al_v);
        }
    }
}

// ---- fp32 attention over [tail tiles | prefix tiles] on the CUDA cores ------------------------------
// Any dtype and head dimension; every product, sum and exponential in fp32, keys still carrying an offset rotated here
// as Eq. 1 states it (on K, in fp32).  A CTA takes BM = 4 TY packed rows (query token i, head-in-group) of one (request,
// kv head) and a contiguous part of its 64-key blocks: split part `blockIdx.x % splits` of the range.  Thread (ty, tx)
// holds rows 4 ty .. + 3: of S the keys tx + TX j, of O the columns tx * V .. in V-wide pieces - 4 x 4 products per pair
// of 16-byte shared-memory words, so that the FMA pipe and not shared memory is the limit with BM = 64.  P takes the
// place of K once the scores are formed.  When the range is split the parts leave un-normalised rows in global memory,
// and the CTA that arrives last (a counter per row tile, which it clears again) combines them: one launch, no waiting.
// Why: 16 CTAs of one row tile each walked all keys in a serial chain, 80 us for 3 x 128 documents and 32 tokens.
struct CorePart {
    float *o;                  // [row tile][split][BM][D]
    float2 *ml;                // [row tile][split][BM]
    int32_t *arrived;          // [row tile], zero between launches
};

// packed fp32 pairs: two products per instruction, so that the FMA pipe is not held back by instruction issue
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
__device__ __forceinline__ uint64_t both(float x)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float2 halves(uint64_t r)
{
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(r));
    return f;
}

template <int N> struct VecOf;
template <> struct VecOf<2> { typedef float2 type; };
template <> struct VecOf<4> { typedef float4 type; };

template <typename T, int D, int TY, int TX>
__global__ void __launch_bounds__(TY *TX, 512 / (TY * TX))
attn_core_kernel(kvp_plan_dev plan, int q_len, int q_pos0, int layer, const T *__restrict__ q, const char *__restrict__ pool_k,
                 const char *__restrict__ pool_v, const char *__restrict__ ws_k, const char *__restrict__ ws_v,
                 const uint4 *__restrict__ k_new, const uint4 *__restrict__ v_new, char *__restrict__ ws_k_out,
                 char *__restrict__ ws_v_out, int64_t pool_rows, int64_t ws_rows, int n_q, int n_kv, int group, int pairing,
                 float scale, int splits, CorePart part, T *__restrict__ out, float *__restrict__ lse)
{
    constexpr int BM = 4 * TY, BN = 64, NT = TY * TX, HALF = D / 2, LD = D + 4, LP = BN + 4;
    constexpr int KN = BN / TX;                              // keys per thread
    constexpr int V = D / TX < 4 ? D / TX : 4;               // width of a piece of O's columns
    constexpr int PC = D / TX / V;                           // pieces per thread
    constexpr int EV = Elem<T>::kPerVec;
    typedef typename VecOf<V>::type VT;
    extern __shared__ float sm[];
    float *Qs = sm, *Ks = Qs + BM * LD, *Vs = Ks + BN * LD, *Ps = Ks;
    __shared__ int last_in;
    pdl_launch_dependents();
    pdl_wait();
    PDL_AFTER(q); PDL_AFTER(pool_k); PDL_AFTER(pool_v); PDL_AFTER(ws_k); PDL_AFTER(ws_v); PDL_AFTER(plan.rope);
    PDL_AFTER(k_new); PDL_AFTER(v_new);

    const int hk = blockIdx.y, b = blockIdx.z, rt = blockIdx.x / splits, sp = blockIdx.x % splits;
    const kvp_item it = plan.items[(layer * n_kv + hk) * plan.item_stride + b];
    const int n_rows = group * q_len, row0 = rt * BM;
    const int plane = layer * n_kv + hk;
    const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;

    if (((uintptr_t)q & 15) == 0) {
#pragma unroll
        for (int u = 0; u < BM * D / EV / NT; ++u) {
            const int w = threadIdx.x + u * NT, rr = row0 + w / (D / EV), c = w % (D / EV) * EV;
            Vec16<T> x;
            x.u = make_uint4(0, 0, 0, 0);
            if (rr < n_rows)
                x.u = *reinterpret_cast<const uint4 *>(q + (((int64_t)b * q_len + rr / group) * n_q + hk * group + rr % group) * D + c);
#pragma unroll
            for (int e = 0; e < EV; e += 4)
                *reinterpret_cast<float4 *>(Qs + (w / (D / EV)) * LD + c + e) =
                    make_float4(Elem<T>::to_f32(x.e[e]), Elem<T>::to_f32(x.e[e + 1]), Elem<T>::to_f32(x.e[e + 2]), Elem<T>::to_f32(x.e[e + 3]));
        }
    } else {                                                 // any element-aligned q is taken
        for (int w = threadIdx.x; w < BM * D; w += NT) {
            const int rr = row0 + w / D, c = w % D;
            float x = 0.f;
            if (rr < n_rows) x = Elem<T>::to_f32(q[(((int64_t)b * q_len + rr / group) * n_q + hk * group + rr % group) * D + c]);
            Qs[(w / D) * LD + c] = x;
        }
    }
    int lim[4];                                              // keys of the query block visible to row r: [0, lim)
#pragma unroll
    for (int r = 0; r < 4; ++r) lim[r] = q_pos0 + min(row0 + 4 * ty + r, n_rows - 1) / group + 1;

    // tail keys: rows appended earlier, then this call's, as far as this row tile sees them (the first one, which
    // appends, walks them all)
    const int i_max = k_new != nullptr && rt == 0 ? q_len - 1 : min(n_rows - 1, row0 + BM - 1) / group;
    const int n_tail = (q_pos0 + i_max) / KVP_TILE_KEYS + 1;
    const int n_blk = 2 * (n_tail + it.tile_end - it.tile_begin);
    const int blk0 = (int)((int64_t)n_blk * sp / splits), blk1 = (int)((int64_t)n_blk * (sp + 1) / splits);

    constexpr int AC = PC * V / 2;
    float m[4], l[4];
    uint64_t acc[4][AC];                                     // pairs of O's columns
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        m[r] = -1e30f;
        l[r] = 0.f;
#pragma unroll
        for (int e = 0; e < AC; ++e) acc[r][e] = 0;
    }

#pragma unroll 1
    for (int blk = blk0; blk < blk1; ++blk) {
        const int tt = blk >> 1;
        kvp_tile tl;
        int qoff = -1;
        if (tt < n_tail) {
            tl.row0 = it.tail_row0 + tt * KVP_TILE_KEYS;
            tl.n_keys = (int16_t)min(KVP_TILE_KEYS, q_pos0 + q_len - tt * KVP_TILE_KEYS);
            tl.src = 1;
            tl.rope = 0;
            qoff = tt * KVP_TILE_KEYS + (blk & 1) * BN;
        } else {
            tl = plan.tiles[it.tile_begin + tt - n_tail];
        }
        const int nk = min(BN, tl.n_keys - (blk & 1) * BN);
        if (nk <= 0) continue;
        const int64_t row = (tl.src == 0 ? (int64_t)plane * pool_rows : (int64_t)plane * ws_rows) + tl.row0 + (blk & 1) * BN;
        const T *kb = reinterpret_cast<const T *>(tl.src == 0 ? pool_k : ws_k) + row * D;
        const T *vb = reinterpret_cast<const T *>(tl.src == 0 ? pool_v : ws_v) + row * D;
        const float2 *cs = plan.rope + (size_t)tl.rope * HALF;

        // the query block's own rows: straight from the caller's tensors, and - by the first row tile - on to the cache
        const bool fresh = qoff >= 0 && k_new != nullptr;

        __syncthreads();                                     // the block before is done with K, P and V
        constexpr int CP = HALF / EV;                        // pairs of 16-byte chunks per row
        constexpr int PER = BN * CP / NT < 4 ? BN * CP / NT : 4;        // at most 16 words in flight per thread
        static_assert(BN * CP % (NT * PER) == 0, "whole rounds");
#pragma unroll 1
        for (int w0 = threadIdx.x; w0 < BN * CP; w0 += NT * PER) {
            Vec16<T> ka[PER], kc[PER], va[PER], vc[PER];
#pragma unroll
            for (int u = 0; u < PER; ++u) {
                const int w = w0 + u * NT, kk = w / CP, c = w % CP;
                ka[u].u = kc[u].u = va[u].u = vc[u].u = make_uint4(0, 0, 0, 0);
                if (kk < nk) {
                    const uint4 *kr = reinterpret_cast<const uint4 *>(kb + (int64_t)kk * D) + c;
                    const uint4 *vr = reinterpret_cast<const uint4 *>(vb + (int64_t)kk * D) + c;
                    if (fresh) {
                        const int64_t src = (((int64_t)b * q_len + qoff + kk) * n_kv + hk) * (2 * CP) + c;
                        kr = k_new + src;
                        vr = v_new + src;
                    }
                    ka[u].u = *kr;
                    kc[u].u = *(kr + CP);
                    va[u].u = *vr;
                    vc[u].u = *(vr + CP);
                    if (fresh && rt == 0) {
                        uint4 *kw = reinterpret_cast<uint4 *>(ws_k_out) + (row + kk) * (2 * CP) + c;
                        uint4 *vw = reinterpret_cast<uint4 *>(ws_v_out) + (row + kk) * (2 * CP) + c;
                        kw[0] = ka[u].u;
                        kw[CP] = kc[u].u;
                        vw[0] = va[u].u;
                        vw[CP] = vc[u].u;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < PER; ++u) {
                const int w = w0 + u * NT, kk = w / CP, c = w % CP;
                float a[EV], x[EV];
#pragma unroll
                for (int e = 0; e < EV; ++e) {
                    a[e] = Elem<T>::to_f32(ka[u].e[e]);
                    x[e] = Elem<T>::to_f32(kc[u].e[e]);
                }
                if (tl.rope != 0) {
                    if (pairing == 0) {
#pragma unroll
                        for (int e = 0; e < EV; ++e) {
                            const float2 r = *(cs + c * EV + e);
                            rotate_pair(a[e], x[e], r.x, r.y);
                        }
                    } else {
#pragma unroll
                        for (int e = 0; e < EV; e += 2) {
                            const float2 r = *(cs + (c * EV + e) / 2), r2 = *(cs + (c * EV + HALF + e) / 2);
                            rotate_pair(a[e], a[e + 1], r.x, r.y);
                            rotate_pair(x[e], x[e + 1], r2.x, r2.y);
                        }
                    }
                }
#pragma unroll
                for (int e = 0; e < EV; e += 4) {
                    *reinterpret_cast<float4 *>(Ks + kk * LD + c * EV + e) = make_float4(a[e], a[e + 1], a[e + 2], a[e + 3]);
                    *reinterpret_cast<float4 *>(Ks + kk * LD + HALF + c * EV + e) = make_float4(x[e], x[e + 1], x[e + 2], x[e + 3]);
                    *reinterpret_cast<float4 *>(Vs + kk * D + c * EV + e) =
                        make_float4(Elem<T>::to_f32(va[u].e[e]), Elem<T>::to_f32(va[u].e[e + 1]), Elem<T>::to_f32(va[u].e[e + 2]),
                                    Elem<T>::to_f32(va[u].e[e + 3]));
                    *reinterpret_cast<float4 *>(Vs + kk * D + HALF + c * EV + e) =
                        make_float4(Elem<T>::to_f32(vc[u].e[e]), Elem<T>::to_f32(vc[u].e[e + 1]), Elem<T>::to_f32(vc[u].e[e + 2]),
                                    Elem<T>::to_f32(vc[u].e[e + 3]));
                }
            }
        }
        __syncthreads();

        uint64_t s2[4][KN];                                  // sums over even and odd columns, side by side
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int j = 0; j < KN; ++j) s2[r][j] = 0;
#pragma unroll 4
        for (int c = 0; c < D; c += 4) {
            ulonglong2 qv[4], kv[KN];
#pragma unroll
            for (int r = 0; r < 4; ++r) qv[r] = *reinterpret_cast<const ulonglong2 *>(Qs + (4 * ty + r) * LD + c);
#pragma unroll
            for (int j = 0; j < KN; ++j) kv[j] = *reinterpret_cast<const ulonglong2 *>(Ks + (tx + TX * j) * LD + c);
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int j = 0; j < KN; ++j) {
                    s2[r][j] = fma2(qv[r].x, kv[j].x, s2[r][j]);
                    s2[r][j] = fma2(qv[r].y, kv[j].y, s2[r][j]);
                }
        }
        float s[4][KN];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int j = 0; j < KN; ++j) {
                const float2 h = halves(s2[r][j]);
                s[r][j] = h.x + h.y;
            }
        __syncthreads();                                     // everyone has read K: P goes there
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            float mx = -INFINITY;
#pragma unroll
            for (int j = 0; j < KN; ++j) {
                const int kk = tx + TX * j;
                const bool vis = kk < nk && (qoff < 0 || qoff + kk < lim[r]);
                s[r][j] = vis ? s[r][j] * scale : -INFINITY;
                mx = fmaxf(mx, s[r][j]);
            }
#pragma unroll
            for (int o = TX / 2; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            const float m_new = fmaxf(m[r], mx);
            const float alpha = expf(m[r] - m_new);
            float ps = 0.f;
#pragma unroll
            for (int j = 0; j < KN; ++j) {
                const float p = expf(s[r][j] - m_new);       // exp(-inf) = 0 for masked keys
                Ps[(4 * ty + r) * LP + tx + TX * j] = p;
                ps += p;
            }
            l[r] = l[r] * alpha + ps;                        // this thread's keys; added up over tx at the end
            m[r] = m_new;
            const uint64_t alpha2 = both(alpha);
#pragma unroll
            for (int e = 0; e < AC; ++e) acc[r][e] = mul2(acc[r][e], alpha2);
        }
        __syncwarp();                                        // a row's P is written and read by one warp
#pragma unroll 4
        for (int kk = 0; kk < BN; kk += 4) {
            float4 pv[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) pv[r] = *reinterpret_cast<const float4 *>(Ps + (4 * ty + r) * LP + kk);
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                union { VT v[PC]; uint64_t p[AC]; } vv;
#pragma unroll
                for (int y = 0; y < PC; ++y)
                    vv.v[y] = *reinterpret_cast<const VT *>(Vs + (kk + x) * D + y * (V * TX) + tx * V);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const uint64_t p = both(x == 0 ? pv[r].x : x == 1 ? pv[r].y : x == 2 ? pv[r].z : pv[r].w);
#pragma unroll
                    for (int e = 0; e < AC; ++e) acc[r][e] = fma2(p, vv.p[e], acc[r][e]);
                }
            }
        }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int o = TX / 2; o > 0; o >>= 1) l[r] += __shfl_xor_sync(0xffffffffu, l[r], o);

    if (splits == 1) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int row = row0 + 4 * ty + r;
            if (row >= n_rows) break;
            const float inv = 1.f / l[r];
            const int i = row / group, h = hk * group + row % group;
            T *dst = out + (((int64_t)b * q_len + i) * n_q + h) * D + tx * V;
#pragma unroll
            for (int e = 0; e < AC; ++e) {
                const float2 o = halves(acc[r][e]);
                dst[(2 * e / V) * (V * TX) + 2 * e % V] = Elem<T>::from_f32(o.x * inv);
                dst[(2 * e / V) * (V * TX) + 2 * e % V + 1] = Elem<T>::from_f32(o.y * inv);
            }
            if (lse != nullptr && tx == 0) lse[((int64_t)b * n_q + h) * q_len + i] = m[r] + logf(l[r]);
        }
        return;
    }
    const int unit = (b * n_kv + hk) * (gridDim.x / splits) + rt;
    const int64_t prow0 = (int64_t)unit * splits * BM;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int64_t pr = prow0 + sp * BM + 4 * ty + r;
#pragma unroll
        for (int y = 0; y < PC; ++y)
            *reinterpret_cast<VT *>(part.o + pr * D + y * (V * TX) + tx * V) = *reinterpret_cast<VT *>(acc[r] + y * (V / 2));
        if (tx == 0) part.ml[pr] = make_float2(m[r], l[r]);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last_in = atomicAdd(part.arrived + unit, 1) == splits - 1;
    __syncthreads();
    if (!last_in) return;
    __threadfence();
    if (threadIdx.x == 0) part.arrived[unit] = 0;
    // weights of the parts, per row, in shared memory (splits x BM pairs fit what K, V and Q took); then every thread
    // takes float4 columns of rows, four parts' loads in flight
    float2 *wl = reinterpret_cast<float2 *>(sm);
    for (int w = threadIdx.x; w < splits * BM; w += NT) wl[w] = __ldcg(part.ml + prow0 + w);
    __syncthreads();
    if (threadIdx.x < BM) {
        float M = -1e30f, L = 0.f;
        for (int z = 0; z < splits; ++z) M = fmaxf(M, wl[z * BM + threadIdx.x].x);
        for (int z = 0; z < splits; ++z) {
            const float2 ml = wl[z * BM + threadIdx.x];
            const float w = expf(ml.x - M);                  // a part without a visible key has l = 0 and O = 0
            wl[z * BM + threadIdx.x].x = w;
            L += w * ml.y;
        }
        const int row = row0 + threadIdx.x;
        wl[threadIdx.x].y = 1.f / L;
        if (lse != nullptr && row < n_rows)
            lse[((int64_t)b * n_q + hk * group + row % group) * q_len + row / group] = M + logf(L);
    }
    __syncthreads();
    constexpr int IT = BM * D / 4 / NT;                      // float4 columns per thread
    float4 o[IT];
#pragma unroll
    for (int u = 0; u < IT; ++u) o[u] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int z = 0; z < splits; ++z) {
#pragma unroll
        for (int u = 0; u < IT; ++u) {
            const int e = threadIdx.x + u * NT;
            const float4 t = __ldcg(reinterpret_cast<const float4 *>(part.o + (prow0 + z * BM) * D) + e);
            const float w = wl[z * BM + e / (D / 4)].x;
            o[u].x += w * t.x; o[u].y += w * t.y; o[u].z += w * t.z; o[u].w += w * t.w;
        }
    }
#pragma unroll
    for (int u = 0; u < IT; ++u) {
        const int e = threadIdx.x + u * NT, row = row0 + e / (D / 4);
        if (row >= n_rows) break;
        const float inv = wl[e / (D / 4)].y;
        T *dst = out + (((int64_t)b * q_len + row / group) * n_q + hk * group + row % group) * D + 4 * (e % (D / 4));
        dst[0] = Elem<T>::from_f32(o[u].x * inv);
        dst[1] = Elem<T>::from_f32(o[u].y * inv);
        dst[2] = Elem<T>::from_f32(o[u].z * inv);
        dst[3] = Elem<T>::from_f32(o[u].w * inv);
    }
}

// ---- attention mass per segment (diagnostic) ----------------------------------------------------------
// grid (batch * q_len, Hkv), 256 threads = 8 warps.  The block holds the group's q rows in fp32; each warp
// takes every eighth key of a segment, each lane two rotation pairs of the key (Eq. 1 in fp32, as the
// CUDA-core attention kernel does), scores by warp reduction, p = exp(scale * q.k' - lse) summed per head.
template <typename T, int D>
__global__ void __launch_bounds__(256)
segment_mass_kernel(kvp_plan_dev plan, int q_len, int q_pos0, int layer, const T *__restrict__ q,
                    const float *__restrict__ lse, const char *__restrict__ pool_k, const char *__restrict__ ws_k,
                    int64_t pool_rows, int64_t ws_rows, int n_q, int n_kv, int group, int pairing, float scale,
                    float *__restrict__ mass, int n_cols)
{
    constexpr int HALF = D / 2, PPL = HALF / 32;            // rotation pairs per lane
    extern __shared__ float sm[];                            // [group][D] q rows, [8][group] partial sums, [group] lse
    float *qs = sm, *part = sm + group * D, *ls = part + 8 * group;
    const int b = blockIdx.x / q_len, i = blockIdx.x % q_len, hk = blockIdx.y;
    const kvp_item it = plan.items[(layer * n_kv + hk) * plan.item_stride + b];
    const int plane = layer * n_kv + hk;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int w = threadIdx.x; w < group * D; w += blockDim.x)
        qs[w] = Elem<T>::to_f32(q[(((int64_t)b * q_len + i) * n_q + hk * group + w / D) * D + w % D]);
    for (int w = threadIdx.x; w < group; w += blockDim.x) ls[w] = lse[((int64_t)b * n_q + hk * group + w) * q_len + i];
    __syncthreads();
    float *out = mass + (((int64_t)b * q_len + i) * n_q + hk * group) * n_cols;
    const int n_seg = it.seg_end - it.seg_begin;
    for (int s = 0; s <= n_seg; ++s) {
        // segment s, or (s == n_seg) the query block: appended rows 0 .. q_pos0 + i
        const T *kb;
        int n_keys, rope = 0;
        if (s < n_seg) {
            const kvp_seg sg = plan.segs[it.seg_begin + s];
            kb = reinterpret_cast<const T *>(pool_k) + ((int64_t)plane * pool_rows + sg.src_row0) * D;
            n_keys = sg.pad[2] >= 0 ? plan.kept[sg.pad[2] * plan.n_planes + plane] : sg.len;
            rope = sg.rope;
        } else {
            kb = reinterpret_cast<const T *>(ws_k) + ((int64_t)plane * ws_rows + it.tail_row0) * D;
            n_keys = q_pos0 + i + 1;
        }
        const float2 *cs = plan.rope + (size_t)rope * HALF;
        float acc[8];
#pragma unroll
        for (int h = 0; h < 8; ++h) acc[h] = 0.f;
        for (int j = warp; j < n_keys; j += 8) {
            const T *kr = kb + (int64_t)j * D;
            float ka[PPL], kc[PPL];
            int ia[PPL], ib[PPL];
#pragma unroll
            for (int u = 0; u < PPL; ++u) {
                const int pr = lane + 32 * u;
                ia[u] = pairing ? 2 * pr : pr;
                ib[u] = pairing ? 2 * pr + 1 : pr + HALF;
                ka[u] = Elem<T>::to_f32(kr[ia[u]]);
                kc[u] = Elem<T>::to_f32(kr[ib[u]]);
                if (rope != 0) rotate_pair(ka[u], kc[u], cs[pr].x, cs[pr].y);
            }
            for (int h = 0; h < group; ++h) {
                float d = 0.f;
#pragma unroll
                for (int u = 0; u < PPL; ++u) d += qs[h * D + ia[u]] * ka[u] + qs[h * D + ib[u]] * kc[u];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
                if (h < 8) acc[h] += expf(d * scale - ls[h]);
            }
        }
        if (lane == 0)
            for (int h = 0; h < group && h < 8; ++h) part[warp * group + h] = acc[h];
        __syncthreads();
        if (threadIdx.x < group) {
            float t = 0.f;
            for (int w = 0; w < 8; ++w) t += part[w * group + threadIdx.x];
            out[(int64_t)threadIdx.x * n_cols + s] = t;
        }
        __syncthreads();
    }
    for (int w = threadIdx.x; w < group * (n_cols - n_seg - 1); w += blockDim.x)
        out[(int64_t)(w / (n_cols - n_seg - 1)) * n_cols + n_seg + 1 + w % (n_cols - n_seg - 1)] = 0.f;
}

}  // namespace

// ---- launchers ------------------------------------------------------------------------------------

cudaError_t kvp_launch_store_rows(const kvp_shape &sh, const void *src, char *dst_plane0, int64_t plane_rows,
                                  int64_t dst_row0, int32_t n_tokens, cudaStream_t st)
{
    const int vecs = sh.head_dim * sh.elem_bytes / 16;
    const int64_t total = (int64_t)sh.n_layers * n_tokens * sh.n_kv_heads * vecs;
    const int grid = (int)((total + 255) / 256 > 65535 * 8 ? 65535 * 8 : (total + 255) / 256);
    store_rows_kernel<<<grid, 256, 0, st>>>(reinterpret_cast<const uint4 *>(src), dst_plane0, plane_rows, dst_row0,
                                            n_tokens, sh.n_layers, sh.n_kv_heads, vecs);
    return cudaGetLastError();
}

cudaError_t kvp_launch_load(const kvp_shape &sh, kvp_load_list &list, int32_t layer, char *pool_k, char *pool_v, int32_t *status,
                            cudaStream_t st)
{
    const int row_bytes = sh.head_dim * sh.elem_bytes;
    int64_t pieces = 0;
    for (int i = 0; i < list.n_items; ++i) {
        list.item[i].piece0 = (int32_t)pieces;
        pieces += 2ll * sh.n_kv_heads * (((int64_t)list.item[i].n * row_bytes + kLoadPiece - 1) / kLoadPiece);
    }
    list.n_pieces = (int32_t)pieces;
    // 20 blocks have 240 KB in flight, just what the link's latency takes, and as few SMs as that needs: the one-CTA attention
    // kernel does not fit beside a block, and its CTAs there wait for the load to end.  Of 50.1 GB/s with 64 blocks: 12 blocks
    // 47.0, 16 49.9, 20 and more 50.0; four short layers over 10 x 1024 tokens on another stream meanwhile (85 us alone):
    // 64 blocks 495 us, 32 290, 20 200, 16 185.
    load_kernel<<<(int)std::min<int64_t>(20, pieces), 32, 0, st>>>(list, layer, sh.n_kv_heads, row_bytes, sh.pool_rows, pool_k, pool_v, status);
    return cudaGetLastError();
}

cudaError_t kvp_launch_upload(const void *host, void *dst, uint64_t bytes, volatile uint32_t *flags, uint32_t seq,
                              int32_t *blocks, cudaStream_t st)
{
    const int n_words = (int)((bytes + 15) / 16);
    const int n = std::min(KVP_UPLOAD_BLOCKS, (n_words + 1023) / 1024);
    *blocks = n;
    return launch_pdl(upload_kernel, n, 1024, 0, st, (const uint4 *)host, (uint4 *)dst, n_words, flags, seq);
}

cudaError_t kvp_launch_gather(const kvp_shape &sh, const kvp_plan_dev &plan, int32_t n_chunks, int32_t n_rope,
                              const double *half_turns, const char *pool_k, const char *pool_v, char *ws_k, char *ws_v,
                              const void *blob, uint32_t blob_bytes, char *blob_dev, bool early, cudaStream_t st)
{
    static_assert(KVP_INLINE_SMALL <= 256 * 16, "one word per thread of a block");
    const int vecs = sh.head_dim * sh.elem_bytes / 16, half = sh.head_dim / 2;
    const int planes = sh.n_layers * sh.n_kv_heads;
    const int n_table = (n_rope * half + 255) / 256;
    // Blocks per chunk: a block's angles cost about as much as moving one plane of its chunk, so a block takes several
    // planes once there are blocks enough to fill the chip (8 x 148), at least two rounds of its 256 threads.
    const int per_plane = KVP_CHUNK_ROWS * (vecs / 2);
    int groups = n_chunks > 0 ? (1184 + n_chunks - 1) / n_chunks : 1;
    const int most = (planes * per_plane + 511) / 512, least = (planes + 15) / 16;
    groups = groups < least ? least : groups;
    groups = groups > most ? most : groups;
    const int grid = n_table + n_chunks * groups;
    float2 *table = const_cast<float2 *>(plan.rope);
    auto go = [&](auto *kernel, const auto &b) {
        return launch_when(early, kernel, grid, 256, 0, st, plan, b, (int)((blob_bytes + 15) / 16), (uint4 *)blob_dev, n_table, n_rope, groups,
                          half_turns, table, pool_k, pool_v, ws_k, ws_v, sh.pool_rows, sh.ws_rows, vecs, half, sh.pairing);
    };
    const auto *small = reinterpret_cast<const kvp_blob<KVP_INLINE_SMALL> *>(blob);
    if (sh.dtype == KVP_DTYPE_BF16)
        return blob ? go(gather_kernel<__nv_bfloat16, KVP_INLINE_SMALL>, *small) : go(gather_kernel<__nv_bfloat16, 0>, kvp_blob<0>());
    return blob ? go(gather_kernel<float, KVP_INLINE_SMALL>, *small) : go(gather_kernel<float, 0>, kvp_blob<0>());
}

cudaError_t kvp_launch_append(const kvp_shape &sh, const kvp_plan_dev &plan, int32_t plan_there, int32_t batch, int32_t q_len,
                              int32_t q_pos0, const void *q, const void *k_new, const void *v_new, char *ws_k, char *ws_v,
                              int32_t layer, int32_t rope_query, const double *half_turns, void *q_rot,
                              cudaStream_t st)
{
    const int grid = batch * q_len;
    const int pairs = (sh.n_kv_heads + (rope_query ? sh.n_q_heads : 0)) * (sh.head_dim * sh.elem_bytes / 32);
    const int threads = pairs <= 64 ? 64 : pairs >= 512 ? 512 : (pairs + 31) / 32 * 32;     // (64: an angle each)
    if (sh.dtype == KVP_DTYPE_BF16)
        return launch_pdl(append_kernel<__nv_bfloat16>, grid, threads, 0, st, plan, plan_there, q_len, q_pos0, (const __nv_bfloat16 *)q,
                          (const __nv_bfloat16 *)k_new, (const __nv_bfloat16 *)v_new, ws_k, ws_v, sh.ws_rows, layer, sh.n_q_heads,
                          sh.n_kv_heads, sh.head_dim, sh.pairing, rope_query, half_turns, (__nv_bfloat16 *)q_rot);
    return launch_pdl(append_kernel<float>, grid, threads, 0, st, plan, plan_there, q_len, q_pos0, (const float *)q, (const float *)k_new,
                      (const float *)v_new, ws_k, ws_v, sh.ws_rows, layer, sh.n_q_heads, sh.n_kv_heads, sh.head_dim, sh.pairing,
                      rope_query, half_turns, (float *)q_rot);
}

cudaError_t kvp_launch_export(const kvp_shape &sh, const kvp_plan_dev &plan, int32_t b, int32_t layer,
                              int32_t prefix_len, int32_t n_query_rows, const char *pool_k, const char *pool_v,
                              const char *ws_k, const char *ws_v, void *k_out, void *v_out, int32_t k_as_f32, bool early,
                              cudaStream_t st)
{
    const int n_rows = prefix_len + n_query_rows;
    if (n_rows <= 0) return cudaSuccess;
    const int grid = (n_rows + kExportRows - 1) / kExportRows;
    if (sh.dtype == KVP_DTYPE_BF16)
        return launch_when(early, export_kernel<__nv_bfloat16>, grid, 256, 0, st, plan, b, layer, prefix_len, n_rows, pool_k, pool_v, ws_k,
                          ws_v, sh.pool_rows, sh.ws_rows, sh.n_kv_heads, sh.head_dim, sh.pairing, k_out, (__nv_bfloat16 *)v_out,
                          k_as_f32);
    return launch_when(early, export_kernel<float>, grid, 256, 0, st, plan, b, layer, prefix_len, n_rows, pool_k, pool_v, ws_k, ws_v,
                      sh.pool_rows, sh.ws_rows, sh.n_kv_heads, sh.head_dim, sh.pairing, k_out, (float *)v_out, k_as_f32);
}

cudaError_t kvp_launch_segment_mass(const kvp_shape &sh, const kvp_plan_dev &plan, int32_t batch, int32_t q_len,
                                    int32_t q_pos0, int32_t layer, const void *q, const float *lse, const char *pool_k,
                                    const char *ws_k, float *mass, int32_t n_cols, cudaStream_t st)
{
    const dim3 grid(batch * q_len, sh.n_kv_heads);
    const size_t smem = sizeof(float) * ((size_t)sh.group * sh.head_dim + 9 * sh.group);
#define KVP_MASS(T, D)                                                                                              \
    segment_mass_kernel<T, D><<<grid, 256, smem, st>>>(plan, q_len, q_pos0, layer, (const T *)q, lse, pool_k, ws_k,  \
                                                       sh.pool_rows, sh.ws_rows, sh.n_q_heads, sh.n_kv_heads,       \
                                                       sh.group, sh.pairing, sh.scale, mass, n_cols)
    if (sh.dtype == KVP_DTYPE_BF16) {
        if (sh.head_dim == 128) KVP_MASS(__nv_bfloat16, 128); else KVP_MASS(__nv_bfloat16, 64);
    } else {
        if (sh.head_dim == 128) KVP_MASS(float, 128); else KVP_MASS(float, 64);
    }
#undef KVP_MASS
    return cudaGetLastError();
}

namespace {

template <int D, int TY> constexpr int core_smem = 4 * (4 * TY * (D + 4) + 64 * (D + 4) + 64 * D);

template <typename T, int D>
cudaError_t prepare_core()
{
    const cudaError_t rc = cudaFuncSetAttribute(attn_core_kernel<T, D, 16, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, core_smem<D, 16>);
    if (rc != cudaSuccess) return rc;
    return cudaFuncSetAttribute(attn_core_kernel<T, D, 4, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, core_smem<D, 4>);
}

template <typename T, int D, int TY, int TX>
cudaError_t launch_core(const kvp_shape &sh, const kvp_plan_dev &plan, int batch, int q_len, int q_pos0, int layer, const void *q,
                        const char *pool_k, const char *pool_v, const char *ws_k, const char *ws_v, int n_tiles,
                        const kvp_core_ws &ws, void *out, float *lse, int32_t *ctas, cudaStream_t st)
{
    constexpr int BM = 4 * TY;
    static_assert(8 * 64 * BM <= core_smem<D, TY>, "the parts' weights fit");
    // Split the keys until the chip is full (two CTAs of 256 threads or four of 128 per SM), but never below one 64-key
    // block per part, and only as far as the partial rows and the counters reach.
    const int64_t row_tiles = (sh.group * (int64_t)q_len + BM - 1) / BM, units = row_tiles * sh.n_kv_heads * batch;
    const int64_t slots = (int64_t)ws.sm_count * (512 / (TY * TX));
    int64_t splits = (slots + units - 1) / units;
    splits = std::min<int64_t>(std::min<int64_t>(splits, 2 * n_tiles), 64);
    splits = std::min<int64_t>(splits, ws.max_rows / (units * BM));
    if (units > ws.max_units || splits < 1) splits = 1;
    const dim3 grid((unsigned)(row_tiles * splits), sh.n_kv_heads, batch);
    if (ctas) *ctas = (int32_t)(grid.x * grid.y * grid.z);
    const CorePart part = {ws.partial_o, ws.partial_ml, ws.arrived};
    return launch_pdl(attn_core_kernel<T, D, TY, TX>, grid, TY * TX, core_smem<D, TY>, st, plan, q_len, q_pos0, layer, (const T *)q, pool_k, pool_v, ws_k, ws_v,
                                    (const uint4 *)ws.k_new, (const uint4 *)ws.v_new, ws.ws_k, ws.ws_v, sh.pool_rows, sh.ws_rows,
                                    sh.n_q_heads, sh.n_kv_heads, sh.group, sh.pairing, sh.scale, (int)splits, part, (T *)out, lse);
}

}  // namespace

cudaError_t kvp_attn_core_prepare(const kvp_shape &sh)
{
    if (sh.dtype == KVP_DTYPE_BF16) return sh.head_dim == 128 ? prepare_core<__nv_bfloat16, 128>() : prepare_core<__nv_bfloat16, 64>();
    return sh.head_dim == 128 ? prepare_core<float, 128>() : prepare_core<float, 64>();
}

cudaError_t kvp_launch_attn_core(const kvp_shape &sh, const kvp_plan_dev &plan, int32_t batch, int32_t q_len, int32_t q_pos0,
                                 int32_t layer, const void *q, const char *pool_k, const char *pool_v, const char *ws_k,
                                 const char *ws_v, int32_t n_tiles, const kvp_core_ws &ws, void *out, float *lse, int32_t *ctas,
                                 cudaStream_t st)
{
    // 64-row tiles use the FMA pipe twice as well as 16-row ones (a shared-memory word feeds twice the products); 16-row
    // tiles when the rows would leave the larger ones half empty, or when even fully split 64-row tiles are fewer than SMs.
    const int64_t rows = sh.group * (int64_t)q_len;
    const int64_t most = (rows + 63) / 64 * sh.n_kv_heads * batch * 2 * n_tiles;
    const bool big = rows > 32 && most >= ws.sm_count;
#define KVP_CORE(T, D)                                                                                                   \
    return big ? launch_core<T, D, 16, 16>(sh, plan, batch, q_len, q_pos0, layer, q, pool_k, pool_v, ws_k, ws_v, n_tiles, \
                                           ws, out, lse, ctas, st)                                                      \
               : launch_core<T, D, 4, 32>(sh, plan, batch, q_len, q_pos0, layer, q, pool_k, pool_v, ws_k, ws_v, n_tiles,  \
                                          ws, out, lse, ctas, st)
    if (sh.dtype == KVP_DTYPE_BF16) {
        if (sh.head_dim == 128) KVP_CORE(__nv_bfloat16, 128); else KVP_CORE(__nv_bfloat16, 64);
    } else {
        if (sh.head_dim == 128) KVP_CORE(float, 128); else KVP_CORE(float, 64);
    }
#undef KVP_CORE
}
