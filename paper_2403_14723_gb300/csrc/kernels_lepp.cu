// Longest-edge propagation paths (Definition 1, Section 3.1) as a device
// primitive over the longest edges of the last generate.  Section 1 lists a
// data-parallel Lepp among the paper's contributions, as a building block
// for Lepp-based refinement and optimisation.
//
// Lepp(t0) = t0, t1, ...: t_i is the neighbour of t_{i-1} across the longest
// edge of t_{i-1}; the path ends at the terminal edge, the longest edge of
// both of its triangles (both are listed), or at a longest edge on the
// border.  The terminal edge is reported by its seed half-edge: the smaller
// half of an interior terminal edge, the interior half of a border one.
// Every step is a dependent load of twin then of the neighbour's longest-
// edge byte; one thread per path.
#include "polylla_internal.cuh"

namespace polylla {

// one step bound: under the strict (length, edge id) order a path never
// revisits a triangle, so T + 1 steps are never reached on a valid mesh
__device__ __forceinline__ int32_t lepp_chase(const MeshView &m, const uint8_t *le, int32_t t, int32_t max_steps,
                                              int32_t *path, int64_t path_cap, int32_t *terminal, bool *ok) {
    const int32_t HI = 3 * m.T;
    int32_t n = 1;
    if (path && 0 < path_cap) path[0] = t;
    uint32_t l = le[t];
    for (;;) {
        const int32_t e = 3 * t + (int32_t)l;
        const int32_t tw = __ldg(m.twin + e);
        if (tw >= HI) {
            *terminal = e;
            break;
        }
        const int32_t t1 = (int32_t)((uint32_t)tw / 3u);
        const uint32_t l1 = le[t1];
        if (path && n < path_cap) path[n] = t1;
        n++;
        if ((int32_t)l1 == tw - 3 * t1) {
            *terminal = e < tw ? e : tw;
            break;
        }
        t = t1;
        l = l1;
        if (n > max_steps) {
            *ok = false;
            break;
        }
    }
    return n;
}

// Every triangle's terminal edge and path length.  Most paths end at their
// first step (three in four on the grids, whose mean is 2.3 triangles), so a
// warp takes LT_ITEMS x 32 consecutive triangles, does everyone's first step with
// the loads of a lane's LT_ITEMS triangles in flight together, and then gathers
// the paths that go on and follows those in full rounds of 32 lanes.  One
// path per lane to its end (13 chains of 3 to 6 loads one after the other per
// lane, each warp as long as its longest path) took 55.0 us a call on 8.4 M
// triangles, this 38.9 us, against 25 us for the 20 bytes a triangle it cannot do
// without.
constexpr int LT_THREADS = 256;
constexpr int LT_ITEMS = 4;
__global__ void __launch_bounds__(LT_THREADS) k_lepp_terminal(MeshView m, const uint8_t *__restrict__ le,
                                                              int32_t max_steps, int32_t *terminal, int32_t *length,
                                                              int32_t *err) {
    constexpr int WT = 32 * LT_ITEMS;  // triangles of a warp
    __shared__ uint2 s_open[LT_THREADS / 32][WT];  // (triangle, 4 times the neighbour + its longest edge)
    const int lane = threadIdx.x & 31;
    uint2 *open = s_open[threadIdx.x >> 5];
    const uint32_t below = (1u << lane) - 1u;
    const int32_t HI = 3 * m.T;
    const int64_t stride = (int64_t)gridDim.x * (LT_THREADS / 32) * WT;
    for (int64_t t0 = ((int64_t)blockIdx.x * (LT_THREADS / 32) + (threadIdx.x >> 5)) * WT; t0 < m.T; t0 += stride) {
        const int32_t tb = (int32_t)t0 + lane;
        int32_t e[LT_ITEMS], tw[LT_ITEMS];
        uint32_t l1[LT_ITEMS];
#pragma unroll
        for (int q = 0; q < LT_ITEMS; q++)
            e[q] = 32 * q < m.T - tb ? 3 * (tb + 32 * q) + (int32_t)__ldg(le + tb + 32 * q) : -1;
#pragma unroll
        for (int q = 0; q < LT_ITEMS; q++) tw[q] = e[q] >= 0 ? __ldg(m.twin + e[q]) : HI;
#pragma unroll
        for (int q = 0; q < LT_ITEMS; q++) l1[q] = tw[q] < HI ? (uint32_t)__ldg(le + (uint32_t)tw[q] / 3u) : 0u;
        uint32_t n_open = 0;
#pragma unroll
        for (int q = 0; q < LT_ITEMS; q++) {
            const int32_t t = tb + 32 * q;
            const uint32_t t1 = (uint32_t)tw[q] / 3u;
            const bool border = tw[q] >= HI;
            const bool ends = border || 3u * t1 + l1[q] == (uint32_t)tw[q];
            if (e[q] >= 0 && ends) {
                terminal[t] = border || e[q] < tw[q] ? e[q] : tw[q];
                if (length) length[t] = border ? 1 : 2;
            }
            const uint32_t bal = __ballot_sync(0xffffffffu, e[q] >= 0 && !ends);
            if (e[q] >= 0 && !ends) open[n_open + __popc(bal & below)] = make_uint2((uint32_t)t, 4u * t1 + l1[q]);
            n_open += __popc(bal);
        }
        __syncwarp();
        for (uint32_t i = lane; i < n_open; i += 32) {
            const uint2 o = open[i];
            uint32_t t = o.y >> 2, l = o.y & 3u;
            int32_t n = 2, term = -1;
            while (true) {
                const int32_t ee = (int32_t)(3u * t + l);
                const int32_t tt = __ldg(m.twin + ee);
                if (tt >= HI) {
                    term = ee;
                    break;
                }
                t = (uint32_t)tt / 3u;
                l = __ldg(le + t);
                n++;
                if (3u * t + l == (uint32_t)tt) {
                    term = ee < tt ? ee : tt;
                    break;
                }
                if (n > max_steps) {
                    atomicOr(err, DEV_ERR_NONTERMINATING);
                    break;
                }
            }
            terminal[o.x] = term;
            if (length) length[o.x] = n;
        }
        __syncwarp();  // the list is the next round's
    }
}

// paths, pass 1: the length of each query's path into offsets[i]
__global__ void k_lepp_len(MeshView m, const uint8_t *le, const int32_t *tri, int32_t n, int32_t max_steps,
                           int32_t *offsets, int32_t *err) {
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int32_t t = tri[i];
        if (t < 0 || t >= m.T) {
            atomicOr(err, DEV_ERR_INPUT);
            offsets[i] = 0;
            continue;
        }
        int32_t term;
        bool ok = true;
        const int32_t len = lepp_chase(m, le, t, max_steps, nullptr, 0, &term, &ok);
        if (!ok) atomicOr(err, DEV_ERR_NONTERMINATING);
        offsets[i] = len;
    }
}

// paths, pass 2: exclusive scan of the lengths per block of LP_THREADS,
// block totals into blk
constexpr int LP_THREADS = 1024;
__global__ void __launch_bounds__(LP_THREADS) k_lepp_scan_local(int32_t *offsets, int32_t n, unsigned long long *blk) {
    __shared__ int32_t s_w[LP_THREADS / 32];
    const int32_t i = blockIdx.x * LP_THREADS + threadIdx.x;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int32_t v = i < n ? offsets[i] : 0;
    int32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) s_w[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        const int32_t x = s_w[lane];
        int32_t xi = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t u = __shfl_up_sync(0xffffffffu, xi, o);
            if (lane >= o) xi += u;
        }
        s_w[lane] = xi - x;
        if (lane == 31) blk[blockIdx.x] = (unsigned long long)xi;
    }
    __syncthreads();
    if (i < n) offsets[i] = s_w[wid] + inc - v;
}

// paths, pass 3 (after the block totals are scanned): add the block's
// prefix; offsets[n] = total; paths written where they fit the capacity
__global__ void k_lepp_write(MeshView m, const uint8_t *le, const int32_t *tri, int32_t n, int32_t max_steps,
                             int32_t *offsets, const unsigned long long *blk_pre, const unsigned long long *total,
                             int32_t *paths, int64_t capacity, int32_t *err) {
    const int32_t i = blockIdx.x * LP_THREADS + threadIdx.x;
    if (i == 0) {
        if ((long long)*total > (long long)INT32_MAX) atomicOr(err, DEV_ERR_CAPACITY);
        offsets[n] = (int32_t)min(*total, (unsigned long long)INT32_MAX);
        if ((long long)*total > capacity) atomicOr(err, DEV_ERR_CAPACITY);
    }
    if (i >= n) return;
    const int64_t off = (int64_t)offsets[i] + (int64_t)blk_pre[blockIdx.x];
    offsets[i] = (int32_t)min(off, (int64_t)INT32_MAX);
    const int32_t t = tri[i];
    if (t < 0 || t >= m.T || off >= capacity) return;
    int32_t term;
    bool ok = true;
    lepp_chase(m, le, t, max_steps, paths + off, capacity - off, &term, &ok);
}

void launch_lepp_terminal(const MeshView &m, const Work &w, int32_t *terminal, int32_t *length, int32_t *err,
                          cudaStream_t s) {
    const int64_t want = ((int64_t)m.T + LT_THREADS * LT_ITEMS - 1) / (LT_THREADS * LT_ITEMS);
    const int64_t most = 16 * (int64_t)w.persistent_blocks;
    k_lepp_terminal<<<(int)(want < most ? want : most), LT_THREADS, 0, s>>>(m, w.le, m.T + 1, terminal, length, err);
}

void launch_lepp_paths(const MeshView &m, const Work &w, const int32_t *tri, int32_t n, int32_t *offsets,
                       int32_t *paths, int64_t capacity, unsigned long long *blk, unsigned long long *blk_pre,
                       unsigned long long *total, int32_t *err, cudaStream_t s) {
    const int32_t nb = (n + LP_THREADS - 1) / LP_THREADS;
    k_lepp_len<<<w.persistent_blocks * 4, 256, 0, s>>>(m, w.le, tri, n, m.T + 1, offsets, err);
    k_lepp_scan_local<<<nb, LP_THREADS, 0, s>>>(offsets, n, blk);
    launch_scan_u64(blk, blk_pre, nb, total, s);
    k_lepp_write<<<nb, LP_THREADS, 0, s>>>(m, w.le, tri, n, m.T + 1, offsets, blk_pre, total, paths, capacity, err);
}

}  // namespace polylla
