// Internal declarations shared by the host planner and the CUDA kernels.
#pragma once

#include <cuda_runtime.h>
#include <cuda.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/kvp.h"

#define KVP_TILE_KEYS 128      // keys per attention tile (one TMA box of K or V rows)
#define KVP_TILE_ROWS 128      // packed query rows per CTA tile (MMA M)
#define KVP_CHUNK_ROWS 32      // rows per gather work item
#define KVP_MAX_SPLIT_UNITS 2048   // partial slots (128 query rows each) in the workspace
#define KVP_CORE_UNITS 2048        // row tiles the CUDA-core kernel may split
// Partial slots that every assembly has to itself: 320 hold what the CUDA-core kernel splits (148 x 2 CTAs of 64 rows, or 4
// of 16, and as many row tiles again), 640 also the four per CTA of the tensor kernel with head dimension 64.
#define KVP_OWN_SLOTS 320
#define KVP_OWN_SLOTS_64 640
#define KVP_SCHED_RING 8       // pinned staging buffers for work lists
// Plans and work lists up to the first size travel as parameters of the kernel that needs them first: an upload kernel in
// front costs 4 us on the way to the first tile, 4 KB of parameters next to nothing (one request of 5 documents x 512 tokens,
// one layer: 24.4 -> 18.8 us; 2 x 8 documents in fp32: 41 -> 37.5).  A launch with 12 KB costs the GPU as much as the upload
// does and saves host time only, so work lists up to the second size travel along where a list serves one launch (compressed
// packets, 4 layers: 244 -> 238 us; one layer, one call: 26.6 -> 24.8), not where it serves the launches of all layers (a
// 5 x 10 documents decode was 0.8 % slower with it).
#define KVP_INLINE_SMALL 4096
#define KVP_INLINE_LARGE 16384
#define KVP_UPLOAD_BLOCKS 16   // blocks of an upload, each with a completion flag of its own

// ---- device-visible plan records (written by the host planner, uploaded once per assembly) -----

struct kvp_tile {              // one run of <= 128 consecutive key rows sharing one rotation offset
    int32_t row0;              // first row, in the pool (src 0) or in the workspace rows (src 1)
    int16_t n_keys;            // 1..128
    int16_t src;               // 0 pool, 1 workspace
    int32_t rope;              // rope-table index of the offset still to be applied to these keys (0 = none)
    int32_t pad;
};

struct kvp_chunk {             // gather work item: <= 32 rows copied pool -> workspace, keys rotated
    int32_t src_row0;
    int32_t dst_row0;
    int32_t n_rows;
    int32_t rope;              // rope-table index (0 = identity: byte copy)
};

struct kvp_seg {               // one segment of a composed request (header, document or trailer)
    int32_t src_row0;
    int32_t len;
    int32_t dst_pos0;
    int32_t delta;
    int32_t rope;
    int32_t pad[3];
};

struct kvp_item {              // one request of the batch
    int32_t prefix_len;
    int32_t tile_begin, tile_end;      // its prefix tiles in the tile array
    int32_t seg_begin, seg_end;        // its segments
    int32_t tail_row0;                 // workspace row where its query K/V rows are appended
    int32_t cache_row0;                // workspace row of composed position 0 (materialised), else -1
    int32_t pad;
};

// One piece of work of the two-stream attention kernel: a contiguous range of one unit's key tiles.
// A unit is up to 256 packed query rows of one (request, kv head).  Its key tiles are numbered: the
// causal tiles of the query's own keys first, then the request's prefix tiles in plan order.
//   mode 0: two 128-row query tiles ("streams"), each visiting every key tile of the range;
//   mode 1: one 128-row query tile; the key tiles alternate between the two streams and the two
//           partial results are combined inside the CTA.
// slot >= 0: un-normalised fp32 partial written to that partial slot (the unit's key range is shared
// by several pieces); slot < 0: this piece covers the whole range and writes the output rows.
struct kvp_work {
    int32_t b, hk;
    int32_t row_base;          // first packed query row of the unit
    int32_t mode;
    int32_t tile_lo, n_tiles;  // range in the unit's tile numbering
    int32_t slot0, slot1;      // stream 0 / stream 1 (mode 1 uses slot0 only)
    // copied from the request's plan item, so that a CTA's first look-up is one memory round trip, not two
    int32_t tile_begin;        // first prefix tile of the (request, plane) in the plan's tile array
    int32_t tail_row0;         // workspace row where the request's query K/V rows are appended
    int32_t pad[2];
};
static_assert(sizeof(kvp_work) == 48, "three 16-byte words");

struct kvp_merge_item {        // 128 packed rows whose result is spread over n_slots partial slots
    int32_t b, hk;
    int32_t row_base;
    int32_t slot0, n_slots;
    int32_t pad[3];            // pad[0]: the request's own query length (0: the call's q_len); pad[1]: requests in the tile (0: one)
};

// Capacity of one plan blob (entries per array, bytes in all).
struct kvp_plan_layout {
    uint64_t total, upload;                // bytes on the device; bytes of the arrays that the host writes
    int32_t max_items, max_tiles, max_chunks, max_segs, max_rope;
};

// Offsets (bytes) of the arrays inside one plan blob, packed for the counts of the assembly it belongs to;
// identical on host and device.  [0, upload) is copied to the device; the rope table is formed there.
struct kvp_plan_offsets {
    uint64_t items = 0, tiles = 0, chunks = 0, segs = 0, kept = 0, delta = 0, upload = 0, rope = 0;
};

// Pointers into a device-resident plan, passed to kernels by value.
struct kvp_plan_dev {
    const kvp_item *items;
    const kvp_tile *tiles;
    const kvp_chunk *chunks;
    const kvp_seg *segs;
    const float2 *rope;        // [n_rope][head_dim/2] (cos, sin) of delta * theta_i
    const int32_t *delta;      // [n_rope] the offsets of the rope table's rows (0 first)
    const int32_t *kept;       // [compressed packets of the assembly][n_layers * n_kv_heads] kept rows per plane
    int32_t item_stride;       // 0: one item / tile list for all planes; batch: items[(layer * n_kv_heads + kv head) * batch + b]
    int32_t n_planes;
};

struct kvp_shape {
    int32_t n_layers, n_q_heads, n_kv_heads, head_dim, group, dtype, pairing, elem_bytes;
    float scale;               // softmax scale
    int64_t pool_rows;         // rows per (layer, kv head) plane in the pool
    int64_t ws_rows;           // rows per plane in one assembly's workspace rows
};

// One pinned staging buffer of the tables a call sends to the device.  The upload kernel reads it over the host link and
// then writes the number of the upload into its blocks' flags, which lie in the same pinned memory: whether the buffer is
// free again is a plain read for the host.
struct kvp_stage {
    char *host = nullptr;
    volatile uint32_t *flags = nullptr;    // [KVP_UPLOAD_BLOCKS]
    uint32_t seq = 0;                      // number of the last upload from here
    int32_t blocks = 0;                    // and its blocks
    bool recorded = false;                 // it was recorded into a graph, which reads the buffer whenever it is launched
};

// ---- host-side context -----------------------------------------------------------------------

struct kvp_segment_host {
    int32_t row0, n, pos0;             // first pool row, positions covered, position it was cached at
    std::vector<int32_t> kept;         // compressed packets: rows kept per plane (layer, kv head); else empty
};

// Short calls over documents that several requests share (decode steps, mostly): the rows of all requests lie in one query
// tile and every document is walked once.  Prefix tiles of all requests together, staged adapter rows first, documents by
// pool row; `rope` of a tile is the number of its document run (0: none), `pad` the requests that hold it, a bit each.
// ropes[(run - 1) * batch + b]: rope-table index of run `run` in request b (where it holds it).
struct kvp_joint {
    int32_t state = -1;                    // -1: not looked at; 0: not worth it; 1: made
    std::vector<kvp_tile> tiles;
    std::vector<int32_t> ropes;
};

struct kvp_assembly_host {
    int32_t id = -1;
    uint32_t flags = 0;
    int32_t batch = 0;
    std::vector<kvp_item> items;
    std::vector<kvp_seg> segs;
    std::vector<kvp_tile> tiles;
    std::vector<kvp_chunk> chunks;         // gather work
    std::vector<int32_t> delta;            // rope-table rows (row 0: no rotation)
    kvp_plan_offsets off;
    int32_t item_stride = 0;               // batch when the assembly has a tile list per (layer, kv head) (compressed packets)
    int32_t last_q_len = 0;
    std::vector<int32_t> appended;         // per layer: query rows appended so far (KVP_CONTINUE)
    bool shard = false;                    // made by kvp_assemble_at: positions start at a caller-given base
    bool ragged = false;                   // a kvp_query_prefill_ragged call has appended a different number of rows per request
    bool waits_loads = false;              // uses packets that came from host memory: wait for the layer's load event
    // work lists of the two-stream kernel (one, or one per layer when the tile lists differ per layer), each
    // built for q_len query tokens at offset q_pos0 (q_len 0 = none yet)
    struct sched_state { int32_t q_len = 0, q_pos0 = 0, ctas = 0, works = 0, merges = 0, slots = 0; uint32_t opts = 0, off_works = 0, off_merges = 0, off_joint = 0; std::vector<int32_t> q_lens; };
    std::vector<sched_state> sched;
    kvp_joint joint;
    bool settled = false;                  // an attention launch has waited for the plan
    // the stream (by its id, no handle is kept) whose calls use the assembly's scratch: its partial slots and counters and,
    // with head dimension 64, its work list
    bool owned = false;
    unsigned long long owner = 0;
};

// Work list of the two-stream kernel for one assembly and query length, with the scratch it is built in.
struct kvp_schedule {
    std::vector<int32_t> cta_begin;
    std::vector<kvp_work> works;
    std::vector<kvp_merge_item> merges;
    int32_t n_ctas = 0, n_slots = 0, max_pieces = 1;
    bool pair = false;                     // for CTA pairs: every unit in mode 0, n_ctas counts pairs
    struct unit { int32_t b, hk, row_base, mode, n_all, n_pieces, q_len, t_first, tile_begin, tail_row0, n_tail, slot; };
    struct cut { int32_t u, t; };
    std::vector<unit> units;
    std::vector<cut> cuts, model;
    std::vector<int64_t> after;
    std::vector<int32_t> order;            // emission order of the CTAs (indices into cuts)
    std::vector<int32_t> work_unit;        // unit of every piece
};

// Partial results of split key ranges, and the counters of the CUDA-core kernel's split row tiles.
struct kvp_scratch {
    float *partial_o;
    float2 *partial_ml;
    int32_t *arrived;
};

struct kvp_ctx {
    kvp_config cfg;
    kvp_shape shape;
    bool host_only = false;
    std::vector<double> inv_freq;
    std::vector<kvp_segment_host> packets;
    // packets whose K/V wait in host memory until a request uses them (parallel to `packets`, grown on demand)
    struct host_src { const char *k = nullptr, *v = nullptr; bool from_host = false, resident = true; };
    std::vector<host_src> packet_src;
    cudaStream_t load_stream = nullptr;             // host -> pool copies, layer by layer
    cudaEvent_t load_fence = nullptr;               // the caller's stream at the assemble that starts a load
    std::vector<cudaEvent_t> load_done;             // [layer]: the loads enqueued so far have landed for this layer
    bool loads_recorded = false;
    std::vector<kvp_segment_host> adapter_h, adapter_t;
    int64_t pool_rows_used = 0;
    // streams (compared, never used) that a registration was enqueued on and no assemble since
    std::vector<cudaStream_t> registered_on;
    bool registered_anywhere = false;               // more of them than are kept count of

    // device memory carved out of the caller's buffers
    char *pool_k = nullptr, *pool_v = nullptr;
    int32_t *status_dev = nullptr;
    kvp_plan_layout pl;
    std::vector<char *> slot_plan_dev;     // per assembly slot
    std::vector<char *> slot_k, slot_v;    // per assembly slot: workspace rows
    std::vector<kvp_scratch> slot_own;     // per assembly slot
    std::vector<char *> slot_sched_dev;    // per assembly slot: cta ranges, work list, merge list
    // pinned staging of the same: a ring, so that the layers of an assembly with a list each, or the steps of a
    // decode, do not wait for one another's upload (which lies behind the attention kernels enqueued before it)
    kvp_stage sched_ring[KVP_SCHED_RING];
    int sched_next = 0;
    const double *half_turns = nullptr;    // device [head_dim/2]: theta_i / pi (angles in half turns per position)
    uint64_t sched_bytes = 0;
    int32_t sched_max_works = 0, sched_max_merges = 0;
    // planning scratch: the large arrays of a call are kept from one to the next
    kvp_assembly_host build;
    std::vector<int32_t> rope_hash, kept_row_of;
    alignas(16) char list_inline[KVP_INLINE_LARGE], plan_inline[KVP_INLINE_SMALL];
    kvp_schedule plan;
    int32_t fused_append = 1;              // plain prefill: the attention kernel reads k_new / v_new itself and appends them
    void *encode_tiled = nullptr;          // cuTensorMapEncodeTiled
    void *pointer_attributes = nullptr;    // cuPointerGetAttributes
    // bf16 with head dimension 128, all assemblies together: [units][128][head_dim]; [units][128] (running max, running sum)
    float *partial_o = nullptr;
    float2 *partial_ml = nullptr;
    char *q_scratch = nullptr;

    char *staging = nullptr;               // the pinned block that all staging buffers and their flags lie in
    std::vector<kvp_stage> plan_ring;      // staging of plans: one more than assemblies alive
    int plan_next = 0;
    std::vector<kvp_assembly_host> slots;
    int32_t next_assembly = 0;

    // TMA descriptors (bf16, head_dim 128 only)
    bool have_tma = false;
    CUtensorMap tm_pool_k, tm_pool_v, tm_pool_k_half;       // _half: boxes of 64 rows, a CTA's part of a K tile in a pair
    std::vector<CUtensorMap> tm_ws_k, tm_ws_v, tm_ws_k_half;

    int32_t sm_count = 148;
    int32_t split_target_ctas = 0, force_splits = 0;
    bool pairs = true;                     // KVP_TUNE_CTA_PAIRS
    // optional CUDA-event timing of the attention (0) and gather (1) kernels, for roofline reports
    int32_t time_kernels = 0;             // 0: off; p >= 1: every p-th attention / gather kernel is bracketed by events
    int32_t tev_seen[2] = {0, 0};
    bool tev_open[2] = {false, false};
    std::vector<cudaEvent_t> tev[2][2];
    int32_t tev_n[2] = {0, 0};
    int32_t last_kind = -1, last_ctas = 0, last_splits = 0, last_launches = 0;
    std::string err;
};

// ---- launches that may begin before the kernel in front of them has ended ------------------------
// Every kernel of a call releases its successor at once and waits for its predecessor (griddepcontrol) before it reads what
// a kernel may have written just before or writes anything, so that launch latency and set-up - barriers, TMEM, filling
// the grid - lie under the predecessor's tail.  Some thread of every block waits before the block can end, so a grid that
// has ended implies that its predecessors have: later work in the stream needs no more than that.
// Readable without waiting: the pool - its writers (registration, host copies) never release a successor early, and between
// them and whatever reads their rows lies a launch that waits for them: the gather (right behind a registration on its
// stream it is launched in plain stream order; its successors start after it has) or a stream wait - and tables that a kernel further in front has waited for before it
// released anyone: the attention kernel behind a fresh work list waits first and releases then, so that the launches
// behind it find that list and the plan complete.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Loads the compiler may take for invariant (const __restrict__ parameters) could be moved in front of the wait, or made
// non-coherent; a pointer that passes through here cannot be used before this point.  What a kernel in front may have
// written is not read with __ldg either: that is for what nothing writes while the kernel is there, and it is there early.
#define PDL_AFTER(p) asm volatile("" : "+l"(p)::"memory")

template <typename T> struct as_given { typedef T type; };
template <typename... P>
cudaError_t launch_when(bool early, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, const typename as_given<P>::type &...args)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = early ? 1 : 0;
    void *ptrs[] = {(void *)&args...};
    return cudaLaunchKernelExC(&cfg, (const void *)kernel, ptrs);
}
template <typename... P>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, const typename as_given<P>::type &...args)
{
    return launch_when(true, kernel, grid, block, smem, st, args...);
}

// Tables that travel as a kernel's own parameters.  N = 0: none.
template <int N> struct kvp_blob { uint4 w[N ? N / 16 : 1]; };
#endif

// ---- kernel launchers (kvp_kernels.cu, kvp_attn_sm100.cu) ---------------------------------------

cudaError_t kvp_launch_store_rows(const kvp_shape &sh, const void *src, char *dst_plane0, int64_t plane_rows,
                                  int64_t dst_row0, int32_t n_tokens, cudaStream_t st);
// One layer of packets that wait in pinned host memory, into the pool.
struct kvp_load_item {
    const char *k, *v;         // device addresses of the host buffers, [n_layers][n_kv_heads][n][head_dim]
    int32_t n, row0;           // tokens; first pool row
    int32_t piece0;            // first of its pieces in the launch
    int32_t pad;
};
#define KVP_LOAD_ITEMS 48
struct kvp_load_list {
    int32_t n_items, n_pieces;
    kvp_load_item item[KVP_LOAD_ITEMS];
};
// fills in piece0 and n_pieces
cudaError_t kvp_launch_load(const kvp_shape &sh, kvp_load_list &list, int32_t layer, char *pool_k, char *pool_v, int32_t *status,
                            cudaStream_t st);
// `bytes` (rounded up to 16) from pinned host memory to the device; the blocks' flags receive `seq` once they have read
// their part.  Returns through *blocks how many there are.
cudaError_t kvp_launch_upload(const void *host, void *dst, uint64_t bytes, volatile uint32_t *flags, uint32_t seq,
                              int32_t *blocks, cudaStream_t st);
// the rope table of an assembly and the gather of its chunks, one launch; blob not null: the plan (blob_bytes) comes along and
// the launch stores it at blob_dev, where `plan` points.  early: it may begin before the kernel in front has ended
cudaError_t kvp_launch_gather(const kvp_shape &sh, const kvp_plan_dev &plan, int32_t n_chunks, int32_t n_rope,
                              const double *half_turns, const char *pool_k, const char *pool_v, char *ws_k, char *ws_v,
                              const void *blob, uint32_t blob_bytes, char *blob_dev, bool early, cudaStream_t st);
// plan_there: the plan was complete before the launch in front of this one was released
cudaError_t kvp_launch_append(const kvp_shape &sh, const kvp_plan_dev &plan, int32_t plan_there, int32_t batch, int32_t q_len,
                              int32_t q_pos0, const void *q, const void *k_new, const void *v_new, char *ws_k, char *ws_v,
                              int32_t layer, int32_t rope_query, const double *half_turns, void *q_rot,
                              cudaStream_t st);
// early: it may begin before the kernel in front has ended; the prefix was complete before that one released anyone
cudaError_t kvp_launch_export(const kvp_shape &sh, const kvp_plan_dev &plan, int32_t b, int32_t layer,
                              int32_t prefix_len, int32_t n_query_rows, const char *pool_k, const char *pool_v,
                              const char *ws_k, const char *ws_v, void *k_out, void *v_out, int32_t k_as_f32, bool early,
                              cudaStream_t st);
cudaError_t kvp_launch_segment_mass(const kvp_shape &sh, const kvp_plan_dev &plan, int32_t batch, int32_t q_len,
                                    int32_t q_pos0, int32_t layer, const void *q, const float *lse, const char *pool_k,
                                    const char *ws_k, float *mass, int32_t n_cols, cudaStream_t st);
// Where the CUDA-core attention kernel leaves the rows of a split key range.
struct kvp_core_ws {
    float *partial_o;
    float2 *partial_ml;
    int32_t *arrived;          // max_units counters, zero between launches
    int64_t max_rows, max_units;
    int32_t sm_count;
    // not null: the kernel reads the query block's rows from these ([batch][q_len][Hkv][d], 16-byte aligned) and copies
    // them behind the prefix (ws_k, ws_v) itself; null: they are there already
    const void *k_new, *v_new;
    char *ws_k, *ws_v;
};
cudaError_t kvp_attn_core_prepare(const kvp_shape &sh);
// n_tiles: most key tiles (causal and prefix) of any request
cudaError_t kvp_launch_attn_core(const kvp_shape &sh, const kvp_plan_dev &plan, int32_t batch, int32_t q_len, int32_t q_pos0,
                                 int32_t layer, const void *q, const char *pool_k, const char *pool_v, const char *ws_k,
                                 const char *ws_v, int32_t n_tiles, const kvp_core_ws &ws, void *out, float *lse, int32_t *ctas,
                                 cudaStream_t st);

struct kvp_attn2_args {
    kvp_plan_dev plan;
    int32_t q_len, q_pos0, layer, n_ctas;
    const int32_t *cta_begin;      // [n_ctas + 1] ranges into works
    const kvp_work *works;
    const void *q;
    void *out;
    float *lse;
    float *partial_o;
    float2 *partial_ml;
    int32_t *status;
    // tail_direct: the query block's K/V tiles are loaded from k_new / v_new ([batch][q_len][Hkv][d]) through
    // tm_knew / tm_vnew and the kernel copies those rows into the workspace rows itself
    int32_t tail_direct;
    int32_t precise;               // KVP_PRECISE_QK
    int32_t fresh;                 // the work list was uploaded just before, by a kernel this launch has to wait for
    int32_t plan_there;            // the plan was complete before the launch in front of this one was released
    // not null: the work list (list_bytes, padded to 16) comes along, works at list_works; the launch stores it at list_dev
    const void *list;
    uint32_t list_bytes, list_works;
    // joint_batch > 0: a unit is one kv head, its rows are those of all requests (kvp_joint), its prefix tiles these
    int32_t joint_batch;
    const kvp_tile *joint_tiles;
    const int32_t *joint_ropes;
    char *list_dev;
    int32_t l2_prefetch;           // the launch has at most two 256-row units per (request, kv head)
    const void *k_new, *v_new;
    char *ws_k, *ws_v;
    CUtensorMap tm_knew, tm_vnew;
};
cudaError_t kvp_attn_sm100_prepare(int32_t head_dim);
cudaError_t kvp_attn_pair_prepare(void);
// a.n_ctas counts CTA pairs; the K maps have boxes of 64 rows
cudaError_t kvp_launch_attn_pair(const kvp_shape &sh, const kvp_attn2_args &a, const CUtensorMap &k_pool, const CUtensorMap &v_pool,
                                 const CUtensorMap &k_ws, const CUtensorMap &v_ws, cudaStream_t st);
cudaError_t kvp_launch_attn_sm100(const kvp_shape &sh, const kvp_attn2_args &a, const CUtensorMap &tm_pool_k,
                                  const CUtensorMap &tm_pool_v, const CUtensorMap &tm_ws_k,
                                  const CUtensorMap &tm_ws_v, cudaStream_t st);
// part_out != nullptr: the merged tiles stay partials and go to a rank buffer of part_tiles query tiles
// list_there: the launch in front waited for the merge list before it released this one
cudaError_t kvp_launch_merge_list(const kvp_shape &sh, int32_t q_len, int32_t n_merges, int32_t max_parts, int32_t sm_count, const kvp_merge_item *merges, bool list_there,
                                  const float *partial_o, const float2 *partial_ml, void *out, float *lse,
                                  void *part_out, int64_t part_tiles, cudaStream_t st);
// n_parts rank buffers back to back -> final output rows
cudaError_t kvp_launch_merge_ranks(const kvp_shape &sh, int32_t batch, int32_t q_len, const void *parts, int32_t n_parts,
                                   void *out, float *lse, cudaStream_t st);
