// Internal declarations of the GB300 Polylla kernels (sm_103a).
//
// Layout of the work arrays in HBM (all sized at create, reused by every
// generate; nothing is allocated on the hot path):
//   le      [T]   uint8  local index of each triangle's longest half-edge
//   flags   [T]   uint8  bits 0-2 F1 (frontier after repair) of 3t+k,
//                        bits 3-5 walk-start marks (next and prev larger),
//                        bit 6 the triangle's longest half-edge is a seed
//   tips    [V]   int32  F0 half-edge leaving each barrier tip
//   chords  [V]   int32  chord half-edge leaving each barrier tip
//   tile_state, tile_pre [T/1024] u64  (polygons, length) total of each output
//                        tile, and their exclusive scan within groups of
//                        1024 tiles; group_tot, group_pre [T/2^20 + 1] u64 the
//                        groups' totals and their exclusive scan
//   poly_rec [T] u32     per polygon, at its output warp's first triangle on:
//                        its minimum within the warp's half-edges, its length
//                        and its chunk of the pool
//   cross_pool [cross_own_count(T) + cross_more_count(T)][16] i32  the half-edges that a polygon which
//                        leaves its tile visits from there on (in a batch, in
//                        the memory of the union origin and prev)
//   poly_wtot [T/64+66] u64  per output warp: its (polygons, length) total
//   seeds [T], offsets [T+1], he_list [3T], v_list [3T]   CSR output
//   ctrl          DevCtrl       counters and the device error word
// A batch context adds the union origin/twin/next/prev [H] (origin, prev and the
// border entries of twin are only filled by the layout check at create; every
// generate writes the interior twin entries from the meshes' own arrays), the
// per-mesh prefix sums and polygon ranges, and the input-check word.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace polylla {

// device error bits (ORed into DevCtrl::error)
enum : int32_t {
    DEV_ERR_NONTERMINATING = 1,
    DEV_ERR_CAPACITY = 2,
    DEV_ERR_TIMEOUT = 4,
    DEV_ERR_INPUT = 8,           // a batch mesh held an index outside its own range
};

struct DevCtrl {
    int32_t error;        // OR of DEV_ERR_* bits of this generate
    int32_t n_tips;       // barrier tips found by the relink
    int32_t n_polygons;   // P
    int32_t n_frontier;   // N_F
    int32_t scan_done;    // tile-scan blocks finished
    int32_t cross_used;   // chunks asked for from the common part of the crossing walks' pool
    int32_t pad[2];
};

struct MeshView {
    int32_t V, T, H;
    const double2 *xy;
    const int32_t *origin;
    const int32_t *twin;
    int32_t *next;
    int32_t *prev;
};

struct Work {
    uint8_t *le;
    uint8_t *flags;
    int32_t *tips;
    int32_t *chords;
    int32_t tip_cap;
    unsigned long long *tile_state; // (polygons, length) total per output tile [n_tile_max]
    unsigned long long *tile_pre;   // the totals' exclusive scan within groups of SCAN_THREADS tiles
    unsigned long long *group_tot;  // each group's total [n_tile_max / SCAN_THREADS + 1]
    unsigned long long *group_pre;  // their exclusive scan [n_tile_max / SCAN_THREADS + 1]
    uint32_t *poly_rec;             // per polygon: its minimum within its warp's half-edges, its length [T]
    unsigned long long *poly_wtot;  // per output warp: (polygons, length) of its range
    int32_t *cross_pool;            // chunks of 16 words: crossing walks' half-edges from their tile on
    int32_t cross_own;              // the tiles' own chunks, at the start of cross_pool
    int32_t cross_more;             // chunks after them, for the walks that need more than one
    int32_t n_tile_max;             // ceil(T / OUT_TILE_MIN)
    int32_t out_tile;               // output tile: triangles
    int32_t out_items;              // output kernel: triangles per thread
    int32_t rl_tile;                // relink: triangles per CTA
    int32_t rl_items;               // relink: triangles per thread
    int32_t *seeds;
    int32_t *offsets;
    int32_t *he_list;
    int32_t *v_list;
    DevCtrl *ctrl;
    int32_t max_rot;
    int32_t persistent_blocks;   // grid of the sparse (tip) kernels
    int32_t le_blocks;           // grid of the persistent longest-edge kernel
    int32_t le_items;            // longest edge: triangles per lane (2 or 4)
    int32_t le_batch_blocks;     // grid of the persistent longest-edge kernel on batches
    // batches: the emitted he_list / v_list are made mesh-local when set
    const int32_t *loc_t_off;    // [loc_n+1] triangle offset of each mesh
    const int32_t *loc_v_off;    // [loc_n+1] vertex offset of each mesh
    const int32_t *loc_h_off;    // [loc_n+1] half-edge offset of each mesh in the local arrays
    int32_t *loc_next;           // the meshes' own next/prev (local indices), written
    int32_t *loc_prev;           //   by the relink and repair kernels
    int32_t *loc_poly_off;       // [loc_n+1] first polygon of each mesh, P at the end
    int32_t loc_n;               // number of meshes (0: a single mesh)
    const int32_t *loc_seg;      // [T/256 + 1] mesh of triangle 256 g (SEG_SPAN)
    int32_t loc_aligned;         // loc_origin and loc_twin start on 16-byte boundaries (bulk copies allowed)
    const int32_t *loc_origin;   // the meshes' own origin and twin arrays (local indices),
    const int32_t *loc_twin;     //   read by the longest-edge and listing kernels
    int32_t *u_twin;             // union twin of interior half-edges, written by the longest-edge kernel
    int32_t *input_err;          // batches: set on an index outside its mesh, folded into
                                 //   the error word and cleared by the tile scan
};

// A batch of independent meshes, each in the single-mesh layout with its own
// (local) indices, concatenated; prefix sums locate mesh i.  The kernels run
// on the batch's union: one mesh whose interior half-edges are those of all
// meshes in order ([3 t_off[i], 3 t_off[i+1]) for mesh i), followed by all
// border half-edges ([3 T_tot + b_off[i], ...)), with global vertex ids.
struct BatchView {
    int32_t n;                   // meshes
    int32_t T_tot, H_tot;
    const int32_t *v_off;        // [n+1] device prefix sums of V_i
    const int32_t *t_off;        // [n+1] of T_i
    const int32_t *h_off;        // [n+1] of H_i
    const int32_t *b_off;        // [n+1] of H_i - 3 T_i (border half-edges)
    const int32_t *origin;       // local arrays [sum H_i]
    const int32_t *twin;
    int32_t *next;
    int32_t *prev;
};

// output kernel: tiles of out_tile triangles (1024, 2048 or 4096), out_items
// per thread; single-block scans (Lepp paths) with SCAN_THREADS threads
constexpr int OUT_TILE_MIN = 1024;
constexpr int OUT_TILE_MAX = 4096;
constexpr int OUT_ITEMS_MIN = 2;
constexpr int OUT_TILE_DEFAULT = 1024;
constexpr int OUT_ITEMS_DEFAULT = 4;
// output warps (of 32 triangles per thread at least OUT_ITEMS_MIN) for T
// triangles, any configuration
__host__ __device__ constexpr int64_t out_warp_count(int64_t T) { return (T + OUT_TILE_MAX) / (32 * OUT_ITEMS_MIN) + 2; }
// chunks of the crossing walks' pool: one per XQUOTA triangles for the tile
// that holds them (0.06 polygons per triangle leave a tile of 1,024 on
// grids, 0.02 on Delaunay meshes; the walks that find no chunk cost the
// listing kernel a chain of loads), then those for long walks
constexpr int XQUOTA = 8;
// (a tile's walks use at most 255 chunks, and at most one per triangle)
__host__ __device__ constexpr int64_t cross_own_count(int64_t T) { return T / XQUOTA + (T < 256 ? T : 256); }
__host__ __device__ constexpr int64_t cross_more_count(int64_t T) { return T / 32 + (T < 2048 ? T / 8 : 256); }
__host__ __device__ constexpr int64_t cross_bytes(int64_t T) { return 64 * (cross_own_count(T) + cross_more_count(T)); }
// A batch has the pool in the memory of its union origin and prev, which only the
// layout check at create uses: bytes of that block, and of each array's part
__host__ __device__ constexpr int64_t union_part(int64_t H) { return (4 * H + 255) / 256 * 256; }
__host__ __device__ constexpr int64_t union_block(int64_t T, int64_t H) {
    return union_part(H) + 4 * H > cross_bytes(T) ? union_part(H) + 4 * H : cross_bytes(T);
}
constexpr int SCAN_THREADS = 1024;

// longest-edge kernel: persistent warps, each with a two-stage ring of
// tiles of 32 x (2 or 4) triangles of origin bulk-copied (TMA) into shared
// memory
constexpr int LE_THREADS = 256;
constexpr int LE_ITEMS_DEFAULT = 2;

// relink kernel: rl_tile triangles per CTA, rl_items per thread
constexpr int RL_TILE_DEFAULT = 128;
constexpr int RL_ITEMS_DEFAULT = 1;

// meshes of up to so many triangles take one kernel of one block
constexpr int SMALL_MAX = 2048;

// bounded waits: iterations of an mbarrier try_wait loop before giving up
constexpr int MBAR_WAIT_LIMIT = 1 << 22;

// ---- launches that follow one another (programmatic dependent launch) --------
// The kernels of a generate each need all of the one before.  Launched plainly,
// each starts only when its predecessor has drained: 1 to 2 us of an idle chip
// per kernel, most of a small mesh's time.  A chained launch may be set up while
// its predecessor still runs: every kernel of the chain first lets its successor
// in (chain_next), whose blocks take what room is left on the SMs and wait there
// (chain_wait: until the predecessor has ended and its writes are visible).
// Every thread waits before it touches global memory, so a kernel has ended only
// after all kernels before it; without a chained launch both are no-ops.  A pass of
// 4 k triangles 87.8 -> 76.6 us, of 2 M 155.7 -> 146.6, of the 4096 grid 1,116 ->
// 1,110.  The waiting blocks do not hold up another stream's short kernels: requests
// of 20 k triangles in the server's lane beside back-to-back generates of 8.4 M took
// 0.270 ms (p99 0.298) with the chain, 0.280 (0.359) without it.
// A chained kernel is resident while the kernels before it still write, so only
// what no kernel of its chain writes may be read through the read-only path
// (__ldg, const __restrict__): the caller's mesh arrays (coords, origin, twin) and
// a batch's tables.  next, prev, labels, flags, lists, records, the chunk pool,
// polygon ranges and a batch's union twins take ordinary loads.
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// an ordinary load of what an earlier kernel of the chain wrote and this one does not
// write, behind chain_wait (volatile keeps it there; without the compiler's aliasing
// rules it takes no more registers than __ldg: written as m.next[x] the listing
// spilled, and the 4096 grid took 1,058 us against 1,052)
__device__ __forceinline__ int32_t ld_chain(const int32_t *p) {
    int32_t v;
    asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
// chained only directly behind a kernel of the chain on the same stream
template <typename... P, typename... A>
cudaError_t launch_kernel(void (*kernel)(P...), int64_t blocks, int threads, size_t smem, cudaStream_t s, bool chained,
                   const A &...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);  // an error also stays pending
}

// ---- bulk copies (TMA engine) and mbarriers, inline PTX --------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
// 1-D bulk copy global -> shared; dst, src 16-byte aligned, bytes % 16 == 0
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// wait for the phase of the given parity; false after MBAR_WAIT_LIMIT tries
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity) {
    for (int i = 0; i < MBAR_WAIT_LIMIT; i++)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// batches: the mesh table holds the mesh of every SEG_SPAN-th triangle
constexpr int SEG_SPAN = 256;
__host__ __device__ constexpr int64_t seg_count(int64_t T) { return T / SEG_SPAN + 1; }

// largest i in [0, n) with off[i] <= x, for ascending prefix sums off[0..n]
// with off[0] <= x < off[n]
__device__ __forceinline__ int32_t seg_of(const int32_t *off, int32_t n, int32_t x) {
    int32_t lo = 0, hi = n - 1;
    while (lo < hi) {
        const int32_t mid = (lo + hi + 1) >> 1;
        if (__ldg(off + mid) <= x) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// the mesh of union triangle t of a batch: from the mesh table's entry at
// or before t, stepping over the meshes that end by t
__device__ __forceinline__ int32_t mesh_of(const int32_t *seg, const int32_t *t_off, int32_t n, int32_t t) {
    int32_t j = __ldg(seg + t / SEG_SPAN);
    while (j + 1 < n && __ldg(t_off + j + 1) <= t) j++;
    return j;
}

// ---- float32 filters of float64 decisions -----------------------------------
// v truncated to float32: the top 23 significand bits, so |v^ - v| <= 2^-23
// |v^| and |v^| <= |v|, by bit manipulation (no float64 instruction).  A
// magnitude outside [2^-126, 2^61) (zero included) sets bad: the caller then
// takes its exact float64 path.
// trunc_to_f32_far leaves the test to the caller, once for several values: far
// collects the largest distance of their exponents from the range's lower end,
// and all lie inside it iff far < TRUNC_SPAN.
constexpr uint32_t TRUNC_SPAN = (1084u - 897u) << 21;
__device__ __forceinline__ float trunc_to_f32_far(double v, uint32_t &far) {
    const uint32_t hi = (uint32_t)__double2hiint(v);
    const uint32_t lo = (uint32_t)__double2loint(v);
    // biased float64 exponent must lie in [897, 1083]: |v| in [2^-126, 2^61)
    // (doubling drops the sign)
    far = max(far, 2u * hi - (897u << 21));
    // (hi:lo) << 3 puts the low 9 exponent bits at 31..23 and the top 23
    // significand bits at 22..0; subtracting 384 from that 9-bit field
    // rebiases 1023 -> 127 for exponents in range
    const uint32_t bits = __funnelshift_l(lo, hi, 3) - (384u << 23);
    return __uint_as_float(bits | (hi & 0x80000000u));
}
__device__ __forceinline__ float trunc_to_f32(double v, uint32_t &bad) {
    uint32_t far = 0;
    const float f = trunc_to_f32_far(v, far);
    bad |= (uint32_t)(far >= TRUNC_SPAN);
    return f;
}

// ---- implicit triangle layout (paper Section 4.2) -------------------------
__device__ __forceinline__ int32_t tri_of(int32_t e) { return e / 3; }
__device__ __forceinline__ int32_t loc_of(int32_t e) { return e - 3 * (e / 3); }
__device__ __forceinline__ int32_t nx_of(int32_t e) {
    int32_t b = 3 * (e / 3);
    int32_t k = e - b;
    return b + (k == 2 ? 0 : k + 1);
}
__device__ __forceinline__ int32_t pv_of(int32_t e) {
    int32_t b = 3 * (e / 3);
    int32_t k = e - b;
    return b + (k == 0 ? 2 : k - 1);
}

// launchers (each enqueues one kernel on stream; chained: behind a kernel of
// the chain, see launch_kernel)
void launch_validate(const MeshView &m, int32_t *bad, cudaStream_t s);
void launch_longest_edge(const MeshView &m, const Work &w, cudaStream_t s, bool chained);
int longest_edge_blocks_per_sm(int32_t items);
int longest_edge_batch_blocks_per_sm();
// the whole generate of a single mesh of at most SMALL_MAX triangles (kernels_small.cu)
void launch_small(const MeshView &m, const Work &w, cudaStream_t s);
int small_configure();  // its shared memory on the current device; 0 on success
void launch_label_relink(const MeshView &m, const Work &w, cudaStream_t s, bool chained);
// allows the relink kernels their shared memory on the current device (once
// per device before the first launch); 0 on success
int relink_configure();
bool relink_config_valid(int32_t tile, int32_t items);
void launch_chords(const MeshView &m, const Work &w, cudaStream_t s, bool chained);
void launch_chord_links(const MeshView &m, const Work &w, cudaStream_t s, bool chained);
void launch_chord_links_list(const MeshView &m, const Work &w, const int32_t *list, const int32_t *count,
                             int32_t cap, cudaStream_t s, bool chained);
// convexification (kernels_convex.cu)
// two kernels: the reflex corners into reflex (count n_reflex), then their
// chords into list (count count); both lists hold at most cap entries
void launch_convex_chords(const MeshView &m, const Work &w, int32_t *reflex, int32_t *n_reflex, int32_t *list,
                          int32_t *count, int32_t cap, cudaStream_t s, bool chained);
void launch_convex_mark(const MeshView &m, const Work &w, const int32_t *list, const int32_t *count, int32_t cap,
                        cudaStream_t s, bool chained);
void launch_poly_count(const MeshView &m, const Work &w, cudaStream_t s, bool chained);
void launch_tile_scan(const MeshView &m, const Work &w, cudaStream_t s, bool chained);
void launch_poly_list(const MeshView &m, const Work &w, cudaStream_t s, bool chained);
// allows the output kernels their shared memory on the current device (once
// per device before the first launch); 0 on success
int polygons_configure();
bool polygons_config_valid(int32_t tile, int32_t items);
int polygons_blocks_per_sm(int32_t tile, int32_t items);
cudaError_t launch_ctrl_out(const Work &w, DevCtrl *host, cudaStream_t s);  // host: pinned
// exclusive scan of n u64 values by one block; *grand gets the sum
void launch_scan_u64(const unsigned long long *in, unsigned long long *out, int32_t n, unsigned long long *grand,
                     cudaStream_t s);
// Lepp (kernels_lepp.cu)
void launch_lepp_terminal(const MeshView &m, const Work &w, int32_t *terminal, int32_t *length, int32_t *err,
                          cudaStream_t s);
void launch_lepp_paths(const MeshView &m, const Work &w, const int32_t *tri, int32_t n, int32_t *offsets,
                       int32_t *paths, int64_t capacity, unsigned long long *blk, unsigned long long *blk_pre,
                       unsigned long long *total, int32_t *err, cudaStream_t s);
// batches (kernels_batch.cu)
void launch_batch_pack(const BatchView &b, int32_t *u_origin, int32_t *u_twin, int32_t *u_next, int32_t *u_prev,
                       int32_t *bad, int32_t *input_err, cudaStream_t s);
void launch_batch_seg(const int32_t *t_off, int32_t n, int32_t T, int32_t *seg, cudaStream_t s);
void launch_batch_meta(const BatchView &b, const Work &w, const int32_t *poly_off, int32_t *local_offsets,
                       int32_t *meta, cudaStream_t s, bool chained);

}  // namespace polylla
