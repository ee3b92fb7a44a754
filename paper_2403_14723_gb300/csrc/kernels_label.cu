// Label-phase kernels: mesh layout check, longest edge per triangle
// (stage 1), and the fused frontier / seed / relink pass (stages 2-4).
#include "longest_edge.cuh"
#include "polylla_internal.cuh"

namespace polylla {

// ===========================================================================
// Layout check (create only).  One thread per half-edge; any violation sets
// *bad.  Checks the contract the hot path relies on instead of re-reading
// next/prev: the implicit triangle layout of interior half-edges, a twin
// involution without fixed points, consistent border links, indices in
// range, target consistency and finite coordinates.
// ===========================================================================
__global__ void k_validate(MeshView m, int32_t *bad) {
    const int32_t HI = 3 * m.T;
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int32_t fail = 0;
    if (i < m.V) {
        double2 p = m.xy[i];
        fail |= !isfinite(p.x) || !isfinite(p.y);
    }
    if (i < m.H) {
        int32_t e = (int32_t)i;
        int32_t t = m.twin[e];
        int32_t o = m.origin[e];
        int32_t n = m.next[e];
        int32_t p = m.prev[e];
        fail |= t < 0 || t >= m.H || t == e;
        fail |= o < 0 || o >= m.V;
        fail |= n < 0 || n >= m.H || p < 0 || p >= m.H;
        if (!fail) {
            fail |= m.twin[t] != e;
            fail |= m.prev[n] != e;
            // target(e) = origin(twin e) = origin(next e)
            fail |= m.origin[n] != m.origin[t];
            if (e < HI) {
                fail |= n != nx_of(e) || p != pv_of(e);
            } else {
                fail |= t >= HI || n < HI || p < HI;
            }
        }
    }
    if (fail) atomicOr(bad, 1);
}

void launch_validate(const MeshView &m, int32_t *bad, cudaStream_t s) {
    int64_t n = m.H > m.V ? m.H : m.V;
    int blocks = (int)((n + 255) / 256);
    k_validate<<<blocks, 256, 0, s>>>(m, bad);
}

// ===========================================================================
// Stage 1 on a mesh: longest_of (longest_edge.cuh) for every triangle.
// ===========================================================================

// Bound by latency and issue together (grid 2048 under ncu: 47 us, issue 62 %,
// 28 warps per SM, 55 % of the measured copy rate, float64 pipe 34 %): whole
// generate of the 4096 grid 1,121 -> 1,108 us with one bound for three edges,
// 1,076 -> 1,058 with the twins read for ties only; 5 or 6 CTAs per SM (fewer
// registers) and the next set's coordinates in flight during a label gained nothing.
// Persistent warps walk tiles of 32 PER triangles.  Each warp owns a
// two-stage shared-memory ring: lane 0 bulk-copies (TMA engine,
// cp.async.bulk + mbarrier) the origin triples of the warp's next tile while
// the warp computes the current one, so the HBM stream of origin never waits
// on the coordinate gathers and no warp waits for another (no block
// barrier).  Each lane takes PER triangles (lane, lane + 32, ..., so a
// warp's gathers and byte stores stay contiguous) and issues their 3 PER
// coordinate loads together.
template <int PER>
__global__ void __launch_bounds__(LE_THREADS, PER == 2 ? 4 : 2) k_longest_edge(MeshView m, Work w) {
    constexpr int NW = LE_THREADS / 32;
    constexpr int LE_TILE = 32 * PER;
    __shared__ __align__(128) int32_t s_org[NW][2][3 * LE_TILE];
    __shared__ __align__(8) uint64_t s_bar[NW][2];
    chain_next();
    chain_wait();
    // reset this generate's control block (error word, tip count, totals)
    // and the output tiles' totals
    const int32_t gtid = blockIdx.x * blockDim.x + threadIdx.x;
    if (gtid < (int32_t)(sizeof(DevCtrl) / sizeof(int32_t))) reinterpret_cast<int32_t *>(w.ctrl)[gtid] = 0;
    for (int32_t i = gtid; i < w.n_tile_max; i += gridDim.x * blockDim.x) w.tile_state[i] = 0ull;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t n_tiles = (m.T + LE_TILE - 1) / LE_TILE;
    uint64_t *bar = s_bar[warp];
    if (lane == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
    }
    __syncwarp();
    // the copy rounds the tail up to 16 bytes: at most 3 ints past 3T,
    // inside origin because H >= 3T + 3 (checked at create)
    auto issue = [&](int32_t tile, int st) {
        const int32_t t0 = tile * LE_TILE;
        const int32_t nt = min(LE_TILE, m.T - t0);
        const uint32_t bytes = ((uint32_t)(12 * nt) + 15u) & ~15u;
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(&bar[st], bytes);
        bulk_load(s_org[warp][st], m.origin + 3 * (int64_t)t0, bytes, &bar[st]);
    };
    const int32_t nwarps = gridDim.x * NW;
    int32_t tile = blockIdx.x * NW + warp;
    if (lane == 0 && tile < n_tiles) issue(tile, 0);
    uint32_t parity = 0u;  // bit st = parity to wait for on stage st
    for (int it = 0; tile < n_tiles; it++, tile += nwarps) {
        const int st = it & 1;
        const int32_t nxt = tile + nwarps;
        if (lane == 0 && nxt < n_tiles) issue(nxt, st ^ 1);
        const bool ok = mbar_wait(&bar[st], (parity >> st) & 1u);
        if (__any_sync(0xffffffffu, !ok)) {
            // give up: record it, wait (bounded) for this warp's copies in
            // flight so no bulk copy lands after the warp has left, return
            if (lane == 0) atomicOr(&w.ctrl->error, DEV_ERR_TIMEOUT);
            mbar_wait(&bar[st], (parity >> st) & 1u);
            if (nxt < n_tiles) mbar_wait(&bar[st ^ 1], (parity >> (st ^ 1)) & 1u);
            return;
        }
        parity ^= 1u << st;
        const int32_t t0 = tile * LE_TILE;
        const int32_t *so = s_org[warp][st];
        double2 p[PER][3];
#pragma unroll
        for (int q = 0; q < PER; q++) {
            const int32_t lt = lane + 32 * q;
            if (t0 + lt < m.T) {
                p[q][0] = __ldg(m.xy + so[3 * lt]);
                p[q][1] = __ldg(m.xy + so[3 * lt + 1]);
                p[q][2] = __ldg(m.xy + so[3 * lt + 2]);
            }
        }
#pragma unroll
        for (int q = 0; q < PER; q++) {
            const int32_t lt = lane + 32 * q;
            const int32_t t = t0 + lt;
            const int32_t *__restrict__ twin = m.twin + 3 * t;
            if (t < m.T)
                w.le[t] = (uint8_t)longest_of(p[q][0], p[q][1], p[q][2], 3 * t,
                                              [twin](int k) { return __ldg(twin + k); });
        }
        __syncwarp();  // stage st is refilled next iteration
    }
}

// ===========================================================================
// Stage 1 on a batch, straight from the meshes' own arrays (no packing
// pass).  Persistent warps with a two-stage ring as in k_longest_edge; a
// warp's tile of 32 PER triangles that lies inside one mesh has its origin
// and twin entries contiguous in the mesh's local arrays (local half-edge
// 3 (t - t_off) + k of triangle t of mesh j sits at h_off + 3 (t - t_off)
// + k), so lane 0 bulk-copies both from that start rounded down to 16
// bytes (r entries early) to 16 bytes past the end, which stays inside the
// mesh's entries since at least 3 border half-edges follow its interior
// ones.  A tile across meshes, or arrays that do not start on a 16-byte
// boundary, are read with plain loads.  The mesh comes from the batch's
// mesh table (the mesh of every 256th triangle).  Every origin and twin is
// range-checked against its mesh: an index outside it is replaced by one
// inside it (vertex 0; the mesh's first border half-edge, which stops
// rotations) and the run is flagged, so no later kernel reads outside the
// mesh.  Each lane writes its triangles' union twins (interior: 3 t_off +
// y; border: 3 T + b_off + (y - 3 T_j)), which the later stages walk, and
// the longest edge as on a single mesh, from the coordinates at the mesh's
// vertex offset.
// ===========================================================================
// what a triangle of a mesh needs of the batch's tables: the mesh's first and
// number of interior union half-edges, local entries, vertices, and the shift
// of its border half-edges into the union
struct MeshRow {
    int32_t t3, ti3, h0, hi, v0, vi, bo;
};
__device__ __forceinline__ MeshRow mesh_row(const Work &w, int32_t j, int32_t HI) {
    MeshRow r;
    r.t3 = 3 * __ldg(w.loc_t_off + j);
    r.ti3 = 3 * __ldg(w.loc_t_off + j + 1) - r.t3;
    r.h0 = __ldg(w.loc_h_off + j);
    r.hi = __ldg(w.loc_h_off + j + 1) - r.h0;
    r.v0 = __ldg(w.loc_v_off + j);
    r.vi = __ldg(w.loc_v_off + j + 1) - r.v0;
    r.bo = HI + (r.h0 - r.t3) - r.ti3;
    return r;
}

template <int PER>
__global__ void __launch_bounds__(LE_THREADS, PER == 2 ? 4 : 2) k_longest_edge_batch(MeshView m, Work w) {
    constexpr int NW = LE_THREADS / 32;
    constexpr int LE_TILE = 32 * PER;
    constexpr int SPAN = 3 * LE_TILE + 4;  // a stage's entries, 4 to spare for an unaligned start
    static_assert(SPAN % 4 == 0, "stages start on 16-byte boundaries");
    __shared__ __align__(128) int32_t s_org[NW][2][SPAN];
    __shared__ __align__(128) int32_t s_tw[NW][2][SPAN];
    __shared__ __align__(8) uint64_t s_bar[NW][2];
    __shared__ int32_t s_r[NW][2];        // per stage: start offset (-1: plain loads)
    __shared__ MeshRow s_row[NW][2];      // and the mesh of a bulk-copied tile
    chain_next();
    chain_wait();
    const int32_t gtid = blockIdx.x * blockDim.x + threadIdx.x;
    if (gtid < (int32_t)(sizeof(DevCtrl) / sizeof(int32_t))) reinterpret_cast<int32_t *>(w.ctrl)[gtid] = 0;
    for (int32_t i = gtid; i < w.n_tile_max; i += gridDim.x * blockDim.x) w.tile_state[i] = 0ull;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t HI = 3 * m.T;
    const int32_t n_tiles = (m.T + LE_TILE - 1) / LE_TILE;
    uint64_t *bar = s_bar[warp];
    if (lane == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
    }
    __syncwarp();
    auto issue = [&](int32_t tile, int st) {
        const int32_t t0 = tile * LE_TILE;
        const int32_t nt = min(LE_TILE, m.T - t0);
        const int32_t j = mesh_of(w.loc_seg, w.loc_t_off, w.loc_n, t0);
        const int32_t t3 = 3 * __ldg(w.loc_t_off + j);
        const bool one = w.loc_aligned && 3 * __ldg(w.loc_t_off + j + 1) >= 3 * (t0 + nt);
        fence_proxy_async_smem();
        if (one) {
            const MeshRow row = mesh_row(w, j, HI);
            s_row[warp][st] = row;
            const int32_t L0 = row.h0 + (3 * t0 - t3);
            const int32_t r = L0 & 3;
            const uint32_t bytes = ((uint32_t)(r + 3 * nt) * 4u + 15u) & ~15u;
            s_r[warp][st] = r;
            mbar_arrive_expect_tx(&bar[st], 2 * bytes);
            bulk_load(s_org[warp][st], w.loc_origin + (L0 - r), bytes, &bar[st]);
            bulk_load(s_tw[warp][st], w.loc_twin + (L0 - r), bytes, &bar[st]);
        } else {
            s_r[warp][st] = -1;
            mbar_arrive_expect_tx(&bar[st], 0u);  // nothing to copy: the phase completes now
        }
    };
    const int32_t nwarps = gridDim.x * NW;
    int32_t tile = blockIdx.x * NW + warp;
    if (lane == 0 && tile < n_tiles) issue(tile, 0);
    uint32_t parity = 0u;
    bool bad = false;
    for (int it = 0; tile < n_tiles; it++, tile += nwarps) {
        const int st = it & 1;
        const int32_t nxt = tile + nwarps;
        if (lane == 0 && nxt < n_tiles) issue(nxt, st ^ 1);
        const bool ok = mbar_wait(&bar[st], (parity >> st) & 1u);
        if (__any_sync(0xffffffffu, !ok)) {
            if (lane == 0) atomicOr(&w.ctrl->error, DEV_ERR_TIMEOUT);
            mbar_wait(&bar[st], (parity >> st) & 1u);
            if (nxt < n_tiles) mbar_wait(&bar[st ^ 1], (parity >> (st ^ 1)) & 1u);
            return;
        }
        parity ^= 1u << st;
        const int32_t t0 = tile * LE_TILE;
        const int32_t r = s_r[warp][st];
        const int32_t *so = s_org[warp][st] + (r > 0 ? r : 0);
        const int32_t *stw = s_tw[warp][st] + (r > 0 ? r : 0);
        double2 p[PER][3];
        int32_t tw[PER][3];
        MeshRow row{};
        if (r >= 0) row = s_row[warp][st];
#pragma unroll
        for (int q = 0; q < PER; q++) {
            const int32_t lt = lane + 32 * q;
            const int32_t t = t0 + lt;
            if (t >= m.T) continue;
            if (r < 0) row = mesh_row(w, mesh_of(w.loc_seg, w.loc_t_off, w.loc_n, t), HI);
            const int32_t g = row.h0 + (3 * t - row.t3);
            int32_t o[3];
#pragma unroll
            for (int k = 0; k < 3; k++) {
                o[k] = r >= 0 ? so[3 * lt + k] : __ldg(w.loc_origin + g + k);
                tw[q][k] = r >= 0 ? stw[3 * lt + k] : __ldg(w.loc_twin + g + k);
            }
#pragma unroll
            for (int k = 0; k < 3; k++) {
                if ((uint32_t)o[k] >= (uint32_t)row.vi) { o[k] = 0; bad = true; }
                if ((uint32_t)tw[q][k] >= (uint32_t)row.hi) { tw[q][k] = row.ti3; bad = true; }
                tw[q][k] += tw[q][k] < row.ti3 ? row.t3 : row.bo;
                p[q][k] = __ldg(m.xy + row.v0 + o[k]);
            }
        }
        // the union twins go out from the stage's own buffer, in whole 16-byte
        // words (every lane has read its local ones)
        __syncwarp();
        int32_t *ut = s_tw[warp][st];
#pragma unroll
        for (int q = 0; q < PER; q++) {
            const int32_t lt = lane + 32 * q;
#pragma unroll
            for (int k = 0; k < 3; k++) ut[3 * lt + k] = tw[q][k];
        }
        __syncwarp();
        if (t0 + LE_TILE <= m.T) {
#pragma unroll
            for (int i = lane; i < 3 * LE_TILE / 4; i += 32)
                reinterpret_cast<int4 *>(w.u_twin + 3 * (int64_t)t0)[i] = reinterpret_cast<const int4 *>(ut)[i];
        } else {
            for (int32_t i = lane; i < 3 * (m.T - t0); i += 32) w.u_twin[3 * (int64_t)t0 + i] = ut[i];
        }
#pragma unroll
        for (int q = 0; q < PER; q++) {
            const int32_t t = t0 + lane + 32 * q;
            const int32_t *twq = tw[q];
            if (t < m.T)
                w.le[t] = (uint8_t)longest_of(p[q][0], p[q][1], p[q][2], 3 * t, [twq](int k) { return twq[k]; });
        }
        // stage st is refilled next iteration: every lane's writes of its twins come
        // before the copy engine's
        fence_proxy_async_smem();
        __syncwarp();
    }
    if (bad) atomicOr(w.input_err, 1);
}

int longest_edge_blocks_per_sm(int32_t items) {
    int n = 0;
    const cudaError_t e = items == 4
        ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_longest_edge<4>, LE_THREADS, 0)
        : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_longest_edge<2>, LE_THREADS, 0);
    if (e != cudaSuccess) n = 1;
    return n > 0 ? n : 1;
}

int longest_edge_batch_blocks_per_sm() {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_longest_edge_batch<2>, LE_THREADS, 0) != cudaSuccess) n = 1;
    return n > 0 ? n : 1;
}

void launch_longest_edge(const MeshView &m, const Work &w, cudaStream_t s, bool chained) {
    const int32_t tile = 32 * (w.le_items == 4 && w.loc_n == 0 ? 4 : 2);  // batches: 2 per lane
    const int32_t n_tiles = (m.T + tile - 1) / tile;
    const int32_t want = (n_tiles + LE_THREADS / 32 - 1) / (LE_THREADS / 32);  // one tile per warp
    const int32_t grid = w.loc_n > 0 ? w.le_batch_blocks : w.le_blocks;  // persistent: every CTA resident
    const int blocks = want < grid ? want : grid;
    // the control-block reset needs >= 8 threads: any grid >= 1 works
    if (w.loc_n > 0) launch_kernel(k_longest_edge_batch<2>, blocks, LE_THREADS, 0, s, chained, m, w);
    else if (w.le_items == 4) launch_kernel(k_longest_edge<4>, blocks, LE_THREADS, 0, s, chained, m, w);
    else launch_kernel(k_longest_edge<2>, blocks, LE_THREADS, 0, s, chained, m, w);
}


// ===========================================================================
// Stages 2-4 fused: frontier labels (Algorithm 3 / 9), seeds (Algorithm 4 /
// 10) and the relink of every frontier half-edge (Section 4.2; the per-half-
// edge form of Algorithm 12).  A CTA of NT threads takes NT * IPT
// consecutive triangles, IPT per thread (strided: triangle t0 + q NT + tid);
// with BATCH (a batch's union) it also writes every link in the meshes' own
// indices and arrays.
//
//   F0[e] = border(e) or (not LE[e] and not LE[twin e])
//   seed  = the triangle's longest half-edge e when it is the smaller half of
//           a terminal edge (LE[e] and LE[twin e]) or lies on the border
//   next[e] for frontier e: x = next(e); while not F0[x]: x = CW(x) =
//           next(twin x); then next[e] = x, prev[x] = e.  Non-frontier e get
//           their triangle links.  A rotation that comes back to twin(e)
//           means target(e) has one frontier edge: a barrier tip, recorded
//           with the frontier half-edge twin(e) leaving it.
//
// F0 of a half-edge in another triangle is evaluated on the fly from the
// longest-edge bytes (L2-resident) and that half-edge's twin, which the
// rotation loads anyway, so the twin array is read from HBM once and no
// frontier array is needed.  Twin values are split into (triangle, corner)
// once, so a rotation step costs one twin and one byte load, and the next
// step's twin is fetched together with the current step's byte.
// next and prev of the CTA's triangles are assembled in shared memory and
// stored coalesced; only prev[x] for an x outside them is stored directly.
// In place is race-free: the rotation reads only twin and le; each next[e]
// is written once (by e's thread, or by the lane that ran e's rotation) and
// each prev[x] once, for the unique e with next[e] = x (or by x's own
// thread when x is not frontier).
//
// Rotations are compacted per warp.  Each thread labels its triangles and
// links the frontier half-edges whose successor is the next half-edge of the
// same triangle; the others (the successor lies across a non-frontier edge)
// become tasks that the warp's lanes then take one each, so a warp runs its
// rotations side by side instead of once per local half-edge.  (Staging the
// CTA's twin and longest-edge bytes in shared memory by bulk copies measured
// slower: on row-major grids half of each vertex fan lies in the next row,
// outside any tile narrower than a row.)
// ===========================================================================
// the twin of interior half-edge e: a batch's union twins are written by the
// kernel before this one, a mesh's own are the caller's input (see chain_wait)
template <bool BATCH, typename I>
__device__ __forceinline__ int32_t twin_of(const MeshView &m, I e) {
    return BATCH ? ld_chain(m.twin + e) : __ldg(m.twin + e);
}

__device__ __forceinline__ int32_t div3(int32_t x) { return (int32_t)((uint32_t)x / 3u); }

// A rotation came back to its tip's only frontier half-edge f, steps steps past
// CW^2(f): the tip has degree steps + 2, which k_chords reads in the chord's
// place (choosing the chord here, by walking half of the rotation again, made
// the relink of Delaunay meshes 5 % slower: a tip in every fourth warp).
__device__ __forceinline__ void add_tip(const Work &w, int32_t f, int32_t steps) {
    const int32_t sl = atomicAdd(&w.ctrl->n_tips, 1);
    if (sl < w.tip_cap) {
        w.tips[sl] = f;
        w.chords[sl] = steps + 2;
    } else {
        atomicOr(&w.ctrl->error, DEV_ERR_CAPACITY);
    }
}

template <int NT, int IPT, bool BATCH>
__global__ void __launch_bounds__(NT, 2048 / NT / IPT) k_label_relink(MeshView m, Work w) {
    constexpr int TT = NT * IPT;  // triangles per CTA
    static_assert(IPT >= 1 && IPT <= 4, "a thread's flag bytes fit one 32-bit word");
    __shared__ __align__(16) int32_t s_nx[3 * TT];
    __shared__ __align__(16) int32_t s_pv[3 * TT];
    __shared__ int4 s_task[NT / 32][96 * IPT];
    __shared__ int32_t s_m0;  // batches: the mesh of the CTA's first triangle
    chain_next();
    chain_wait();
    const int32_t t0 = blockIdx.x * TT;
    const int32_t nT = min(TT, m.T - t0);
    const int32_t eb = 3 * t0;
    const int32_t nE = 3 * nT;
    const int32_t HI = 3 * m.T;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t below = (1u << lane) - 1u;
    if (BATCH && threadIdx.x == 0) s_m0 = mesh_of(w.loc_seg, w.loc_t_off, w.loc_n, t0);
    uint32_t fls = 0;  // byte q: flags of triangle t0 + q NT + tid
    uint32_t total = 0;
#pragma unroll
    for (int q = 0; q < IPT; q++) {
        const int32_t lt = q * NT + (int32_t)threadIdx.x;
        const bool live = lt < nT;
        const int32_t t = t0 + lt;
        const int32_t e0 = 3 * t;
        const int32_t lb = 3 * lt;
        uint32_t pend = 0;
        int32_t tw[3], ttri[3];
        uint32_t tloc[3], lnb[3];
        if (live) {
            tw[0] = twin_of<BATCH>(m, e0);
            tw[1] = twin_of<BATCH>(m, e0 + 1);
            tw[2] = twin_of<BATCH>(m, e0 + 2);
            const uint32_t ltl = w.le[t];
            uint32_t F = 0, twle = 0;
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const bool b = tw[k] >= HI;
                ttri[k] = b ? 0 : div3(tw[k]);
                tloc[k] = (uint32_t)(tw[k] - 3 * ttri[k]);
                lnb[k] = b ? 3u : (uint32_t)w.le[ttri[k]];
                const bool tl = !b && lnb[k] == tloc[k];
                F |= (uint32_t)(b || ((uint32_t)k != ltl && !tl)) << k;
                twle |= (uint32_t)tl << k;
            }
            const int32_t twl = ltl == 0u ? tw[0] : (ltl == 1u ? tw[1] : tw[2]);
            const bool seed = (twl >= HI) || (((twle >> ltl) & 1u) && (e0 + (int32_t)ltl) < twl);
            fls |= (F | ((uint32_t)seed << 6)) << (8 * q);
            // own slots: non-frontier half-edges keep their triangle links,
            // frontier ones wait for their predecessor (-1 until then)
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const int j = k == 2 ? 0 : k + 1;
                const bool f = (F >> k) & 1u;
                s_pv[lb + k] = f ? -1 : e0 + (k == 0 ? 2 : k - 1);
                if (!f || ((F >> j) & 1u)) s_nx[lb + k] = e0 + j;
                else pend |= 1u << k;
            }
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const int j = k == 2 ? 0 : k + 1;
                if (((F >> k) & 1u) && ((F >> j) & 1u)) s_pv[lb + j] = e0 + k;  // successor in the triangle
            }
        }
        // compact the warp's pending rotations (the order of the tasks does
        // not matter: each writes its own slots)
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const bool mine = (pend >> k) & 1u;
            const uint32_t bal = __ballot_sync(0xffffffffu, mine);
            if (mine) {
                const int j = k == 2 ? 0 : k + 1;
                s_task[wid][total + __popc(bal & below)] =
                    make_int4(e0 + k, tw[k], ttri[j], (int32_t)(tloc[j] | (lnb[j] << 2)));
            }
            total += __popc(bal);
        }
    }
    __syncthreads();  // every slot initialised before the rotations write prev
    for (uint32_t i = lane; i < total; i += 32) {
        const int4 tk = s_task[wid][i];
        const int32_t e = tk.x;
        int32_t ty = tk.z;
        uint32_t ly = (uint32_t)tk.w & 3u;
        uint32_t ley = ((uint32_t)tk.w >> 2) & 3u;
        uint32_t lx = ly == 2u ? 0u : ly + 1u;
        int32_t x = 3 * ty + (int32_t)lx;
        int32_t tx = twin_of<BATCH>(m, x);
        int32_t steps = 0;
        while (true) {
            if (tx >= HI) break;                     // border edge: frontier
            const int32_t ttx = div3(tx);
            const uint32_t ltx = (uint32_t)(tx - 3 * ttx);
            const uint32_t lxn = ltx == 2u ? 0u : ltx + 1u;
            const int32_t xn = 3 * ttx + (int32_t)lxn;
            const uint32_t lex = w.le[ttx];
            const int32_t txn = twin_of<BATCH>(m, xn);
            if (ley != lx && lex != ltx) break;      // neither half longest: frontier
            ley = lex;
            x = xn;
            lx = lxn;
            tx = txn;
            if (++steps > w.max_rot) {
                atomicOr(&w.ctrl->error, DEV_ERR_NONTERMINATING);
                break;
            }
        }
        s_nx[e - eb] = x;
        const uint32_t dx = (uint32_t)(x - eb);
        if (dx < (uint32_t)nE) s_pv[dx] = e;
        else {
            if (!BATCH) m.prev[x] = e;
            else {  // e, x lie in one mesh, at or after the CTA's first
                int32_t mj = s_m0;
                while (mj + 1 < w.loc_n && 3 * __ldg(w.loc_t_off + mj + 1) <= e) mj++;
                const int32_t sh = 3 * __ldg(w.loc_t_off + mj);
                w.loc_prev[__ldg(w.loc_h_off + mj) + (x - sh)] = e - sh;
            }
        }
        if (x == tk.y) add_tip(w, tk.y, steps);
    }
    __syncthreads();
    // walk-start marks: frontier, next and prev larger (prev unknown: set
    // by another CTA, counted as larger)
#pragma unroll
    for (int q = 0; q < IPT; q++) {
        const int32_t lt = q * NT + (int32_t)threadIdx.x;
        if (lt >= nT) break;
        uint32_t fl = (fls >> (8 * q)) & 0xffu;
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const int32_t e = eb + 3 * lt + k;
            const int32_t pv = s_pv[3 * lt + k];
            if (((fl >> k) & 1u) && s_nx[3 * lt + k] > e && (pv < 0 || pv > e)) fl |= 8u << k;
        }
        w.flags[t0 + lt] = (uint8_t)fl;
    }
    int4 *dn = reinterpret_cast<int4 *>(m.next + eb);
    for (int i = threadIdx.x; 4 * i < nE; i += NT) {
        if (4 * i + 3 < nE) {
            dn[i] = reinterpret_cast<const int4 *>(s_nx)[i];
        } else {
            for (int c = 0; c < 4; c++)
                if (4 * i + c < nE) m.next[eb + 4 * i + c] = s_nx[4 * i + c];
        }
    }
    // (a batch's union prev is never read: its links go to the meshes' own
    // prev only)
    for (int i = threadIdx.x; i < nE && !BATCH; i += NT) {
        const int32_t v = s_pv[i];
        if (v >= 0) m.prev[eb + i] = v;
    }
    // in a batch, the links in the meshes' own indices and arrays (the CTA's
    // half-edges are consecutive in a mesh's local arrays between mesh
    // boundaries, so these stores stay coalesced)
    if (BATCH) {
        // mesh mj spans union half-edges [sh, nb); its local entry of union
        // x is x + gsh
        int32_t mj = s_m0;
        int32_t sh = 3 * __ldg(w.loc_t_off + mj);
        int32_t nb = 3 * __ldg(w.loc_t_off + mj + 1);
        int32_t gsh = __ldg(w.loc_h_off + mj) - sh;
        for (int i = threadIdx.x; i < nE; i += NT) {
            const int32_t x = eb + i;
            while (x >= nb && mj + 1 < w.loc_n) {
                mj++;
                sh = nb;
                nb = 3 * __ldg(w.loc_t_off + mj + 1);
                gsh = __ldg(w.loc_h_off + mj) - sh;
            }
            const int32_t g = x + gsh;
            w.loc_next[g] = s_nx[i] - sh;
            const int32_t v = s_pv[i];
            if (v >= 0) w.loc_prev[g] = v - sh;
        }
    }
}

// ===========================================================================
// Stages 2-4 fused, one triangle per thread (the same labels, seeds, links
// and tips as k_label_relink).  A triangle's frontier half-edges form at most
// one cyclic run among its three (one run, or none, or all three), and only
// the last half-edge of a run has a successor across a non-frontier edge: a
// triangle has at most one rotation.  With one triangle per thread, each
// thread runs its own rotation: a warp's lanes run their rotations side by
// side without any task list, and every next entry is set by its own thread.
// prev goes through shared memory (a rotation sets prev[x] for an x of another
// thread); each warp stores the next and prev of its 32 triangles as
// contiguous, coalesced runs and shares nothing with the others, so there is no
// block barrier.  Only the lowest frontier half-edge of a triangle can carry
// the walk-start mark.
// Bound by instruction issue together with the latency of its chains of loads
// (twin, label, twin, label): on the 2048 grid 93 M warp instructions at 3.1 a
// cycle, 57 of 64 warps per SM; with at most 48 (40 registers) 0.428 ms on the 4096
// grid, with 40 0.520 ms, against 0.376 ms here and 0.387 ms with block barriers and a mark
// test for every half-edge.  Loads without branches (clamped indices past the
// border) measured 0.407 ms.
// ===========================================================================
template <int NT, bool BATCH>
__global__ void __launch_bounds__(NT, 2048 / NT) k_label_relink1(MeshView m, Work w) {
    static_assert(NT % 32 == 0, "whole warps");
    __shared__ int32_t s_pv[3 * NT];
    __shared__ __align__(16) int32_t s_nx[3 * NT];
    chain_next();
    chain_wait();
    // a warp's 32 triangles and their links are its own: no block barrier
    const int lane = threadIdx.x & 31;
    const int32_t t0 = blockIdx.x * NT + ((int32_t)threadIdx.x & ~31);
    const int32_t eb = 3 * t0;
    const int32_t nE = 3 * min(32, m.T - t0);  // negative past the mesh's end
    const uint32_t HI = 3u * (uint32_t)m.T;
    const int32_t lb = 3 * (int32_t)threadIdx.x;
    const int32_t t = t0 + lane;
    const bool live = t < m.T;
    const int32_t e0 = 3 * t;
    const int32_t ws = 3 * ((int32_t)threadIdx.x & ~31);  // the warp's first slot
    uint32_t F = 0, fl = 0;
    uint32_t kt = 3;          // the local index of the rotating half-edge (3: none)
    uint32_t kf = 3;          // that of the run's first half-edge (3: no frontier, or all of it)
    int32_t twk = 0;          // the rotating half-edge's twin (coming back to it finds a tip)
    uint32_t x = 0, lx = 0, ley = 0;  // the rotation: half-edge, its local index, its triangle's longest
    uint32_t tw[3] = {0, 0, 0}, ltl = 0;
    if (live) {
        tw[0] = (uint32_t)twin_of<BATCH>(m, e0);
        tw[1] = (uint32_t)twin_of<BATCH>(m, e0 + 1);
        tw[2] = (uint32_t)twin_of<BATCH>(m, e0 + 2);
        ltl = w.le[t];
    }
    // batches (looked up while the twins are on their way; with the fast stores
    // below and the longest-edge kernel's table rows 789 -> 757 us for 512 meshes):
    // the mesh of the warp's first triangle (m0) and the thread's, its
    // first union half-edge (sh), and from a union half-edge to its entry in the
    // local arrays (gsh).  Most warps lie inside one mesh.
    int32_t m0 = 0, sh = 0, gsh = 0;
    bool one = true;
    if (BATCH && t0 < m.T) {
        m0 = mesh_of(w.loc_seg, w.loc_t_off, w.loc_n, t0);
        int32_t mj = m0;
        one = nE == 96 && eb + 96 <= 3 * __ldg(w.loc_t_off + m0 + 1);
        if (!one && live)
            while (mj + 1 < w.loc_n && __ldg(w.loc_t_off + mj + 1) <= t) mj++;
        sh = 3 * __ldg(w.loc_t_off + mj);
        gsh = __ldg(w.loc_h_off + mj) - sh;
    }
    if (live) {
        uint32_t ttri[3], tloc[3], lnb[3];
        uint32_t twle = 0;
#pragma unroll
        for (uint32_t k = 0; k < 3; k++) {
            const bool b = tw[k] >= HI;
            ttri[k] = b ? 0u : tw[k] / 3u;
            tloc[k] = tw[k] - 3u * ttri[k];
            lnb[k] = b ? ~0u : (uint32_t)w.le[ttri[k]];
            const bool tl = lnb[k] == tloc[k];
            F |= (uint32_t)(b || (k != ltl && !tl)) << k;
            twle |= (uint32_t)tl << k;
        }
        const uint32_t twl = ltl == 0u ? tw[0] : (ltl == 1u ? tw[1] : tw[2]);
        const bool seed = (twl >= HI) || (((twle >> ltl) & 1u) && (uint32_t)e0 + ltl < twl);
        fl = F | ((uint32_t)seed << 6);
        // the run's last half-edge (its successor in the triangle is not
        // frontier) rotates; the first one's predecessor is a rotation's.  One
        // bit at most: 1, 2 or 4 -> k = bit >> 1 (0 stays 0: told by F)
        const uint32_t last = F & ~((F >> 1) | (F << 2)), head = F & ~((F << 1) | (F >> 2));
        s_pv[lb] = head & 1u ? -1 : e0 + 2;
        s_pv[lb + 1] = head & 2u ? -1 : e0;
        s_pv[lb + 2] = head & 4u ? -1 : e0 + 1;
        if (last) {
            kt = last >> 1;
            kf = head >> 1;
            twk = (int32_t)(kt == 0u ? tw[0] : (kt == 1u ? tw[1] : tw[2]));
            // x = CW(next e) = next(twin(next e)), j = next e's local index
            const uint32_t txj = kt == 2u ? tw[0] : (kt == 0u ? tw[1] : tw[2]);
            const uint32_t ly = kt == 2u ? tloc[0] : (kt == 0u ? tloc[1] : tloc[2]);
            ley = kt == 2u ? lnb[0] : (kt == 0u ? lnb[1] : lnb[2]);
            x = ly == 2u ? txj - 2u : txj + 1u;
            lx = ly == 2u ? 0u : ly + 1u;
        }
    }
    __syncwarp();  // every prev slot initialised before rotations write them
    if (kt < 3u) {
        // while x is not frontier, x = CW(x).  The next step's twin is fetched
        // with this step's label.
        const int32_t e = e0 + (int32_t)kt;
        uint32_t tx = (uint32_t)twin_of<BATCH>(m, x);
        int32_t steps = 0;
        while (tx < HI) {                            // a border edge is frontier
            const uint32_t ttx = tx / 3u;
            const uint32_t ltx = tx - 3u * ttx;
            const uint32_t xn = ltx == 2u ? tx - 2u : tx + 1u;
            const uint32_t lex = w.le[ttx];
            const uint32_t txn = (uint32_t)twin_of<BATCH>(m, xn);
            if (ley != lx && lex != ltx) break;      // neither half longest: frontier
            ley = lex;
            x = xn;
            lx = xn - 3u * ttx;
            tx = txn;
            if (++steps > w.max_rot) {
                atomicOr(&w.ctrl->error, DEV_ERR_NONTERMINATING);
                break;
            }
        }
        const uint32_t dx = x - (uint32_t)eb;
        if (dx < 96u) s_pv[ws + (int32_t)dx] = e;  // (past the end of the mesh there is no x)
        else if (!BATCH) m.prev[x] = e;
        else w.loc_prev[(int32_t)x + gsh] = e - sh;  // e and x lie in one mesh
        if ((int32_t)x == twk) add_tip(w, twk, steps);
    }
    __syncwarp();  // every prev slot is final
    // the walk-start mark: next and prev larger (prev -1: set by another warp,
    // counted as larger).  Only the lowest frontier half-edge can be a
    // polygon's minimum: links inside the triangle ascend, but for the one from
    // its third half-edge to its first.
    if (live) {
        if (F) {
            const uint32_t kl = F & 1u ? 0u : F >> 1 & 1u ? 1u : 2u;
            const uint32_t el = (uint32_t)e0 + kl;
            const uint32_t pk = (uint32_t)s_pv[lb + (int32_t)kl];  // -1 is the largest
            if ((kl != kt || x > el) && (kl != kf || pk > el)) fl |= 8u << kl;
        }
        const int32_t xi = (int32_t)x;
        s_nx[lb] = kt == 0u ? xi : e0 + 1;
        s_nx[lb + 1] = kt == 1u ? xi : e0 + 2;
        s_nx[lb + 2] = kt == 2u ? xi : e0;
        w.flags[t] = (uint8_t)fl;
    }
    __syncwarp();
    // each warp stores the links of its 96 half-edges in place, coalesced
    // (in a batch, also in the meshes' own indices and arrays; a batch's
    // union prev is never read, so it is not written)
    if (nE == 96 && one) {
        if (lane < 24)
            reinterpret_cast<int4 *>(m.next + eb)[lane] = reinterpret_cast<const int4 *>(s_nx + ws)[lane];
        const int32_t *ps = s_pv + ws + lane, *ns = s_nx + ws + lane;
        if (BATCH) {
            int32_t *nd = w.loc_next + (eb + gsh) + lane;
#pragma unroll
            for (int i = 0; i < 96; i += 32) nd[i] = ns[i] - sh;
        }
        int32_t *pd = BATCH ? w.loc_prev + (eb + gsh) + lane : m.prev + eb + lane;
#pragma unroll
        for (int i = 0; i < 96; i += 32)
            if (ps[i] >= 0) pd[i] = ps[i] - sh;
        return;
    }
    int32_t bj = m0;
    for (int i = lane; i < nE; i += 32) {
        const int32_t xe = eb + i;
        const int32_t nv = s_nx[ws + i];
        const int32_t pv = s_pv[ws + i];
        m.next[xe] = nv;
        if (!BATCH) {
            if (pv >= 0) m.prev[xe] = pv;
        } else {
            while (bj + 1 < w.loc_n && 3 * __ldg(w.loc_t_off + bj + 1) <= xe) bj++;
            const int32_t shj = 3 * __ldg(w.loc_t_off + bj);
            const int32_t g = __ldg(w.loc_h_off + bj) + (xe - shj);
            w.loc_next[g] = nv - shj;
            if (pv >= 0) w.loc_prev[g] = pv - shj;
        }
    }
}

// launch configurations: (triangles per CTA, triangles per thread); one per
// thread runs k_label_relink1, more run k_label_relink
#define RELINK1_CONFIGS(X) \
    X(64)                  \
    X(128)                 \
    X(256)
#define RELINK_CONFIGS(X) \
    X(128, 2)             \
    X(64, 4)

bool relink_config_valid(int32_t tile, int32_t items) {
#define X(N) \
    if (tile == N && items == 1) return true;
    RELINK1_CONFIGS(X)
#undef X
#define X(N, I) \
    if (tile == N * I && items == I) return true;
    RELINK_CONFIGS(X)
#undef X
    return false;
}

int relink_configure() { return 0; }  // static shared memory only

void launch_label_relink(const MeshView &m, const Work &w, cudaStream_t s, bool chained) {
#define X(N)                                                                         \
    if (w.rl_tile == N && w.rl_items == 1) {                                         \
        if (w.loc_n > 0) launch_kernel(k_label_relink1<N, true>, (m.T + N - 1) / N, N, 0, s, chained, m, w); \
        else launch_kernel(k_label_relink1<N, false>, (m.T + N - 1) / N, N, 0, s, chained, m, w);       \
        return;                                                                      \
    }
    RELINK1_CONFIGS(X)
#undef X
#define X(N, I)                                                                      \
    if (w.rl_tile == N * I && w.rl_items == I) {                                     \
        if (w.loc_n > 0) launch_kernel(k_label_relink<N, I, true>, (m.T + N * I - 1) / (N * I), N, 0, s, chained, m, w);  \
        else launch_kernel(k_label_relink<N, I, false>, (m.T + N * I - 1) / (N * I), N, 0, s, chained, m, w);        \
        return;                                                                      \
    }
    RELINK_CONFIGS(X)
#undef X
    if (w.loc_n > 0) launch_kernel(k_label_relink1<128, true>, (m.T + 127) / 128, 128, 0, s, chained, m, w);
    else launch_kernel(k_label_relink1<128, false>, (m.T + 127) / 128, 128, 0, s, chained, m, w);
}

}  // namespace polylla
