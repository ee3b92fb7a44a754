// Output kernels (stages 5b-5d): find every polygon, key it by its smallest
// half-edge, and write the scan-compacted CSR in ascending seed order.
//
// A frontier half-edge e is its polygon's minimum iff walking next from e
// comes back to e without meeting a smaller half-edge.  A minimum is smaller
// than both its neighbours along the polygon, so only half-edges carrying
// the relink's walk-start mark (next and prev both larger, a superset kept
// by the repair) walk.  This finds every cycle of the relink exactly once,
// keyed by the canonical seed the paper's Algorithm 14 keeps, without a seed
// list; listing each minimum's cycle from the minimum, minima in ascending
// order, is the canonical CSR (Section 6.8's scan-and-compact output).
//
// The stage works on tiles of consecutive triangles.  Meshes come in a
// spatially coherent order, so about nine polygons in ten lie inside the
// tile that holds their minimum, and two kernels stream the tiles through
// shared memory (bulk copies by the TMA engine, one mbarrier per CTA):
//   k_poly_count  walks the starts of its tile, writes one word per minimum
//                 (half-edge and length) and, for the polygons that cross the
//                 tile, the half-edges they visit from there on; totals the
//                 (count, length) pairs per listing warp and per tile;
//   k_tile_scan   scans the tile totals per group of 1024 tiles;
//   k_poly_list   gives every lane one word, so one polygon, places the
//                 polygons by a warp scan of the lengths and lists them through
//                 a staging buffer that goes out with coalesced stores.
// The count is bound by instruction issue and latency, the listing by its bytes: on
// the 2048 grid (8.4 M triangles, under ncu) the count issues 35.1 M warp
// instructions at 2.5 a cycle and moves 140 MB in 49 us, 43 % of the measured copy
// rate (6,696 GB/s), the listing 51.3 M at 2.4 and 358 MB in 72 us, 74 %.  Against a lane per 4
// triangles that walked and listed whatever minima it held, each polygon that
// left the tile stalling its lane's warp once in either kernel: count 0.168 ->
// 0.172 ms, listing 0.395 -> 0.267 ms on the 4096 grid; 51 -> 33 and 49 -> 14 us
// on 200 k random points, whose hull polygons of 100 and more half-edges are a
// chain of loads (now one, in the count only).
// No warp waits for another warp.  Two designs that did were slower: a
// single kernel whose tiles looked back for the totals of tiles still being
// walked (every CTA in flight waited for the slowest walk before it), and a
// listing kernel whose tiles looked back for the prefixes of tiles still
// being listed (each look-back summed back over the tiles started during
// its own round trip to L2).
#include "polylla_internal.cuh"

namespace polylla {

__device__ __forceinline__ unsigned long long warp_incl_scan(unsigned long long v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// exclusive block scan of one value per thread (blockDim.x a multiple of
// 32, at most 1024); returns the exclusive prefix, *total gets the block
// total.  s_warp holds 32 + 1 entries.
__device__ unsigned long long block_excl_scan(unsigned long long v, unsigned long long *s_warp,
                                              unsigned long long *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const unsigned long long inc = warp_incl_scan(v, lane);
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        // one warp scans the warp totals: s_warp[q] becomes the exclusive
        // prefix of warp q, s_warp[32] the block total
        const unsigned long long x = lane < nw ? s_warp[lane] : 0ull;
        const unsigned long long xi = warp_incl_scan(x, lane);
        if (lane < nw) s_warp[lane] = xi - x;
        if (lane == 31) s_warp[32] = xi;
    }
    __syncthreads();
    const unsigned long long wb = s_warp[warp];
    *total = s_warp[32];
    __syncthreads();  // s_warp may be reused by the caller
    return wb + inc - v;
}

// ===========================================================================
// k_scan_blocks: one block, exclusive scan of n 64-bit values; *grand
// receives the sum.  Rounds of blockDim.x coalesced entries with a running
// carry.  (Used by the Lepp paths.)
// ===========================================================================
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_blocks(const unsigned long long *in, unsigned long long *out,
                                                              int32_t n, unsigned long long *grand) {
    __shared__ unsigned long long s_warp[33];
    unsigned long long carry = 0;
    for (int32_t b = 0; b < n; b += SCAN_THREADS) {
        const int32_t i = b + threadIdx.x;
        const unsigned long long v = i < n ? in[i] : 0ull;
        unsigned long long total;
        const unsigned long long ex = block_excl_scan(v, s_warp, &total);
        if (i < n) out[i] = carry + ex;
        carry += total;
    }
    if (threadIdx.x == 0) *grand = carry;
}

void launch_scan_u64(const unsigned long long *in, unsigned long long *out, int32_t n, unsigned long long *grand,
                     cudaStream_t s) {
    k_scan_blocks<<<1, SCAN_THREADS, 0, s>>>(in, out, n, grand);
}

// ---- polygon records of the count pass ----------------------------------------
// A triangle lies in one polygon, so a warp's WT consecutive triangles hold
// at most WT minima.  Per minimum, in ascending order from the warp's first
// triangle's slot, one 32-bit word: bits 0-9 the minimum's half-edge within
// the warp's 3 WT (WT <= 256), bits 10-17 its walk's chunk + 1 among the tile's
// (0: none), bits 18-31 the polygon's length.  Lengths
// from REC_LEN_MAX on are recorded as REC_LEN_MAX: the listing kernel measures
// those polygons again.
constexpr int REC_X_SHIFT = 10;
constexpr int REC_LEN_SHIFT = 18;
constexpr uint32_t REC_E_MASK = (1u << REC_X_SHIFT) - 1u;
constexpr uint32_t REC_X_MASK = (1u << (REC_LEN_SHIFT - REC_X_SHIFT)) - 1u;
constexpr uint32_t REC_LEN_MAX = (1u << (32 - REC_LEN_SHIFT)) - 1u;

// Walks that leave their tile: the count gathers a tile's (further ones are
// walked where they are met) and writes every half-edge from the first
// outside the tile on into a chunk of the pool, so that the listing kernel
// copies them instead of following a chain of global loads.  A chunk is 16
// words: XCHUNK half-edges and the chunk that goes on with the walk.  Every
// tile owns TILE / XQUOTA chunks; a long walk takes further ones from the
// pool's common part (ctrl.cross_used).
constexpr int XCHUNK = 15;
constexpr int LIST_CROSS = 16;
template <int TILE>
constexpr int count_cross() { return TILE / XQUOTA < (int)REC_X_MASK ? TILE / XQUOTA : (int)REC_X_MASK; }

__device__ __forceinline__ int32_t lds_i32(uint32_t addr) {
    int32_t v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

// ---- tiles -----------------------------------------------------------------
// A tile is TILE consecutive triangles (3 TILE half-edges); its copies start
// on 16-byte boundaries (TILE is a multiple of 16) and round their length up
// to 16 bytes: at most 3 ints past 3T, inside next/origin because
// H >= 3T + 3, and flags is allocated to a multiple of 16 bytes.
__device__ __forceinline__ uint32_t tile_bytes(int32_t nt, int32_t bytes_per_triangle) {
    return ((uint32_t)(bytes_per_triangle * nt) + 15u) & ~15u;
}

// ===========================================================================
// k_poly_count<TILE, IPT>: one CTA per tile, for the listing kernel's warps of
// WT = 32 IPT triangles; a warp here counts for two of them (2 WT consecutive
// triangles: its rounds of 32 walks are fuller, and half the threads per tile
// leave room for more tiles on an SM).  Thread 0 bulk-copies the tile's next
// and flags into shared memory; then
//   - every warp gathers its starts (at most one a triangle: a minimum is its
//     triangle's lowest frontier half-edge, since the links inside a triangle
//     ascend) into a list, so that every lane walks one;
//   - each start walks next inside the tile until a smaller half-edge or back
//     to itself; the walks that leave the tile upwards (downwards is smaller)
//     are gathered for the whole CTA and then run side by side in full warps,
//     their global loads in flight together;
//   - every warp writes its minima's words (half-edge, chunk, length) in
//     ascending order, stores the (count, length) totals and adds them to the
//     tile's total (zeroed by the first kernel of the generate).
// ===========================================================================
template <int TILE, int IPT>
__global__ void __launch_bounds__(TILE / (2 * IPT)) k_poly_count(MeshView m, Work w) {
    constexpr int NT = TILE / (2 * IPT);
    constexpr int E = 3 * TILE;
    constexpr int WT = 32 * IPT;           // triangles of a listing warp
    constexpr int CT = 2 * WT;             // triangles of a warp here
    constexpr int NW = TILE / WT;          // listing warps
    constexpr int NX = count_cross<TILE>();
    static_assert(TILE % NT == 0 && 3 * CT <= (1 << REC_X_SHIFT) && E < (1 << 16), "records and queue entries hold the half-edge");
    static_assert(TILE % 16 == 0, "tile copies start on 16-byte boundaries");
    extern __shared__ __align__(128) unsigned char smem[];
    int32_t *s_nx = reinterpret_cast<int32_t *>(smem);              // [E]
    int2 *s_cross = reinterpret_cast<int2 *>(s_nx + E);             // [NX] walks that left the tile
    uint32_t *s_ent = reinterpret_cast<uint32_t *>(s_cross + NX + (NX & 1));  // [TILE] starts, then records
    uint8_t *s_fl = reinterpret_cast<uint8_t *>(s_ent + TILE);      // [TILE]
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ uint32_t s_ncross;
    const uint32_t HI = 3u * (uint32_t)m.T;
    const int32_t tile = blockIdx.x;
    const int32_t t0 = tile * TILE;
    const int32_t nt = min(TILE, m.T - t0);
    const int32_t eb = 3 * t0;
    const uint32_t ne = (uint32_t)(3 * nt);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t below = (1u << lane) - 1u;
    chain_next();
    chain_wait();
    if (threadIdx.x == 0) {
        mbar_init(&s_bar, 1);
        fence_mbar_init();
        const uint32_t be = tile_bytes(nt, 12), bf = tile_bytes(nt, 1);
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(&s_bar, be + bf);
        bulk_load(s_nx, m.next + eb, be, &s_bar);
        bulk_load(s_fl, w.flags + t0, bf, &s_bar);
        s_ncross = 0;
    }
    __syncthreads();
    unsigned long long *wtot = w.poly_wtot + (int64_t)tile * NW + 2 * wid;
    if (__syncthreads_or(!mbar_wait(&s_bar, 0))) {
        // copies not seen in time: record it; the tile stays empty.  A CTA
        // leaves only after its bulk copies landed (bounded wait).
        if (lane < 2) wtot[lane] = 0ull;
        if (threadIdx.x == 0) {
            atomicOr(&w.ctrl->error, DEV_ERR_TIMEOUT);
            mbar_wait(&s_bar, 0);
        }
        return;
    }
    // the warp's starts, in ascending order
    uint32_t *ent = s_ent + wid * CT;
    uint32_t ns = 0;
#pragma unroll
    for (int q = 0; q < 2 * IPT; q++) {
        const int32_t lt = wid * CT + 32 * q + lane;
        const uint32_t f = lt < nt ? s_fl[lt] : 0u;
        const uint32_t st = (f >> 3) & f & (0u - (f & 7u)) & 7u;  // the mark of the lowest frontier half-edge
        const uint32_t bal = __ballot_sync(0xffffffffu, st != 0u);
        if (st) ent[ns + __popc(bal & below)] = (uint32_t)(3 * (32 * q + lane)) + (st >> 1);
        ns += __popc(bal);
    }
    __syncwarp();
    const int32_t wb = eb + 3 * CT * wid;                     // the warp's first half-edge
    const uint32_t nxa = smem_u32(s_nx) - 4u * (uint32_t)eb;  // shared address of next[0]
    uint32_t over0 = 0, over1 = 0;  // length of the lane's minima that their records do not hold
    bool runaway = false;
    for (uint32_t r = 0; r < ns; r += 32) {
        const uint32_t i = r + lane;
        int32_t x = -1, e = 0;
        uint32_t L = 1;
        if (i < ns) {
            // one comparison for "above e and inside the tile"
            e = wb + (int32_t)ent[i];
            const uint32_t span = (uint32_t)(eb - e - 1) + ne;
            x = lds_i32(nxa + 4u * (uint32_t)e);
            while ((uint32_t)(x - e - 1) < span && L <= ne) {
                x = lds_i32(nxa + 4u * (uint32_t)x);
                L++;
            }
            if (L > ne) {  // more steps than half-edges in the tile
                runaway = true;
                x = -1;
            }
            if (x == e) ent[i] |= L << REC_LEN_SHIFT;
        }
        const bool out = x > e;
        const uint32_t bal = __ballot_sync(0xffffffffu, out);
        if (bal) {
            uint32_t slot = 0;
            if (lane == 0) slot = atomicAdd(&s_ncross, (uint32_t)__popc(bal));
            slot = __shfl_sync(0xffffffffu, slot, 0) + __popc(bal & below);
            if (out && slot < NX) {
                s_cross[slot] = make_int2(x, (int32_t)((uint32_t)(e - eb) | (L << 16)));
                ent[i] |= (slot + 1) << REC_X_SHIFT;
            } else if (out) {
                while (x > e) {
                    const uint32_t d = (uint32_t)(x - eb);
                    x = d < ne ? s_nx[d] : ld_chain(m.next + x);
                    if (++L > HI) {
                        runaway = true;
                        x = -1;
                    }
                }
                if (x == e) {
                    const uint32_t held = min(L, REC_LEN_MAX);
                    ent[i] |= held << REC_LEN_SHIFT;
                    if (e - wb < 3 * WT) over0 += L - held;
                    else over1 += L - held;
                }
            }
        }
    }
    __syncthreads();
    // the tile's crossing walks; the result, in place of the exit: the length
    // (0: not a minimum) and bit 31 if the walk's chunk does not hold it all
    const uint32_t ncross = min(s_ncross, (uint32_t)NX);
    for (uint32_t r = threadIdx.x; r < ncross; r += NT) {
        const int2 c = s_cross[r];
        int32_t x = c.x;
        const int32_t e = eb + (int32_t)((uint32_t)c.y & 0xffffu);
        uint32_t L = (uint32_t)c.y >> 16;
        int32_t *p = w.cross_pool + 16 * (int64_t)(t0 / XQUOTA + (int32_t)r);
        bool held = true;
        while (true) {
            // a chunk's worth of steps, all through global memory: a warp
            // waits for its slowest lane, which is outside the tile
            int32_t j = 0;
            do {
                const int32_t y = ld_chain(m.next + x);
                if (held) p[j] = x;
                x = y;
            } while (++j < XCHUNK && x > e);
            L += (uint32_t)j;
            if (x <= e) break;
            if (L > HI) {
                runaway = true;
                break;
            }
            const int32_t more = held ? atomicAdd(&w.ctrl->cross_used, 1) : -1;
            held = more >= 0 && more < w.cross_more;  // else the pool is used up
            if (held) {
                p[XCHUNK] = w.cross_own + more;
                p = w.cross_pool + 16 * (int64_t)(w.cross_own + more);
            }
        }
        s_cross[r].x = x == e ? (int32_t)(L | (held ? 0u : 0x80000000u)) : 0;
    }
    if (runaway) atomicOr(&w.ctrl->error, DEV_ERR_NONTERMINATING);
    __syncthreads();
    // the words of both halves (the first half's starts come first)
    uint32_t *out = w.poly_rec + t0 + CT * wid;
    uint32_t k = 0, k0 = 0, len0 = over0, len1 = over1;
    for (uint32_t r = 0; r < ns; r += 32) {
        const uint32_t i = r + lane;
        uint32_t v = i < ns ? ent[i] : 0u;
        uint32_t L = v >> REC_LEN_SHIFT;
        const uint32_t slot1 = (v >> REC_X_SHIFT) & REC_X_MASK;
        if (slot1) {
            const uint32_t R = (uint32_t)s_cross[slot1 - 1].x;
            L = R & 0x7fffffffu;
            v = (v & ((R >> 31) ? REC_E_MASK : (1u << REC_LEN_SHIFT) - 1u)) | (min(L, REC_LEN_MAX) << REC_LEN_SHIFT);
        }
        const bool half = (v & REC_E_MASK) >= 3u * WT;
        const uint32_t bal = __ballot_sync(0xffffffffu, L != 0u);
        k0 += __popc(bal & __ballot_sync(0xffffffffu, !half));
        if (L) {
            const uint32_t at = k + __popc(bal & below);
            if (half) out[WT + at - k0] = v - 3u * WT;
            else out[at] = v;
        }
        k += __popc(bal);
        len0 += half ? 0u : L;
        len1 += half ? L : 0u;
    }
    len0 = __reduce_add_sync(0xffffffffu, len0);
    len1 = __reduce_add_sync(0xffffffffu, len1);
    if (lane == 0) {
        wtot[0] = ((unsigned long long)k0 << 32) | len0;
        wtot[1] = ((unsigned long long)(k - k0) << 32) | len1;
        const unsigned long long tot = ((unsigned long long)k << 32) + len0 + len1;
        if (tot) atomicAdd(w.tile_state + tile, tot);
    }
}

// ===========================================================================
// k_tile_scan: one block per group of SCAN_THREADS tiles: the exclusive scan
// of the tiles' (polygons, length) totals within the group (tile_pre) and
// the group's total (group_tot).  The last block to finish (a counter in
// the control block) scans the group totals into group_pre and ends the
// output: P, N_F and offsets[P].  A tile's place in the output is then
// tile_pre[tile] + group_pre[its group], and no block waits for another.
// ===========================================================================
__global__ void __launch_bounds__(SCAN_THREADS) k_tile_scan(MeshView m, Work w, int32_t n) {
    __shared__ unsigned long long s_warp[33];
    __shared__ int s_last;
    chain_next();
    chain_wait();
    const int32_t i = blockIdx.x * SCAN_THREADS + threadIdx.x;
    const unsigned long long v = i < n ? w.tile_state[i] : 0ull;
    unsigned long long total;
    const unsigned long long ex = block_excl_scan(v, s_warp, &total);
    if (i < n) w.tile_pre[i] = ex;
    if (threadIdx.x == 0) {
        w.group_tot[blockIdx.x] = total;
        __threadfence();  // the total is visible before the count says so
        s_last = atomicAdd(&w.ctrl->scan_done, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    unsigned long long carry = 0;
    for (int32_t b = 0; b < (int32_t)gridDim.x; b += SCAN_THREADS) {
        const int32_t g = b + threadIdx.x;
        const unsigned long long x = g < (int32_t)gridDim.x ? __ldcg(w.group_tot + g) : 0ull;
        unsigned long long t;
        const unsigned long long e = block_excl_scan(x, s_warp, &t);
        if (g < (int32_t)gridDim.x) w.group_pre[g] = carry + e;
        carry += t;
    }
    if (threadIdx.x != 0) return;
    int64_t P = (int64_t)(carry >> 32);
    const int64_t NF = (int64_t)(carry & 0xffffffffull);
    if (P > (int64_t)m.T || NF > 3 * (int64_t)m.T) {
        atomicOr(&w.ctrl->error, DEV_ERR_CAPACITY);
        P = P > m.T ? m.T : P;
    }
    w.offsets[P] = (int32_t)NF;
    w.ctrl->n_polygons = (int32_t)P;
    w.ctrl->n_frontier = (int32_t)NF;
    // in a batch, P closes the ranges (and starts the meshes without triangles
    // at the end, which no lane holds)
    for (int32_t j = w.loc_n; w.loc_n > 0 && j >= 0 && __ldg(w.loc_t_off + j) >= m.T; j--) w.loc_poly_off[j] = (int32_t)P;
    // a batch mesh with an index outside its range (found by the longest-edge
    // kernel) fails the run; the word is cleared for the next one
    if (w.input_err && *w.input_err) {
        atomicOr(&w.ctrl->error, DEV_ERR_INPUT);
        *w.input_err = 0;
    }
}

// ===========================================================================
// k_poly_list<TILE, IPT, BATCH>: one CTA per tile (BATCH: the mesh is a
// batch's union, whose seeds, lists and per-mesh polygon ranges are written
// in each mesh's own indices).  Thread 0 bulk-copies the tile's
// next and origin (BATCH: next only when the tile spans meshes; the block
// then reads origin from the meshes' own arrays, which hold local vertex ids,
// into shared memory).  Then every warp works on its own: its first polygon
// and entry are the scanned total of the tiles before its tile plus the
// totals of the warps before it in the tile; its polygon words, one per lane,
// give every polygon's place by a warp scan of the lengths (seeds and offsets
// go out coalesced).  Each lane lists one polygon from its minimum along next
// into the warp's staging buffer (entries past it go out directly); a polygon
// that leaves the tile goes to a list with its place so far, and its chunks are
// then copied half a warp at a time.  The warp stores its staged range of
// he_list coalesced and reads each half-edge's origin (shared memory, or global
// memory outside the tile) as it does, for v_list.
// Six CTAs of 256 threads per SM (40 registers, 37 KB) measured 0.267 ms on the
// 4096 grid, five (48 registers) 0.342 ms.
// ===========================================================================
template <int IPT>
constexpr int list_stage() { return 72 * IPT; }  // CSR entries a warp stages: 2.25 per triangle

template <int TILE, int IPT, bool BATCH>
__global__ void __launch_bounds__(TILE / IPT, TILE == 1024 && IPT == 4 ? 6 : 1) k_poly_list(MeshView m, Work w) {
    constexpr int NT = TILE / IPT;
    constexpr int E = 3 * TILE;
    constexpr int NW = NT / 32;
    constexpr int WT = 32 * IPT;    // triangles per warp
    constexpr int WCAP = list_stage<IPT>();
    extern __shared__ __align__(128) unsigned char smem[];
    int32_t *s_nx = reinterpret_cast<int32_t *>(smem);  // [E]
    int32_t *s_org = s_nx + E;                          // [E + 4]
    int32_t *s_stage = s_org + E + 4;                   // [NW][WCAP]
    int4 *s_cross = reinterpret_cast<int4 *>(s_stage + NW * WCAP);  // [NW][LIST_CROSS]
    __shared__ __align__(8) uint64_t s_bar;
    const int32_t HI = 3 * m.T;
    const int32_t tile = blockIdx.x;
    const int32_t t0 = tile * TILE;
    const int32_t nt = min(TILE, m.T - t0);
    const int32_t eb = 3 * t0;
    const uint32_t ne = (uint32_t)(3 * nt);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // batches: the mesh of the tile's first triangle, and where the tile's
    // origins start in s_org (-1: not bulk-copied, loaded below)
    __shared__ int32_t s_j0, s_r;
    chain_next();
    chain_wait();
    if (threadIdx.x == 0) {
        mbar_init(&s_bar, 1);
        fence_mbar_init();
        const uint32_t be = tile_bytes(nt, 12);
        fence_proxy_async_smem();
        if (!BATCH) {
            mbar_arrive_expect_tx(&s_bar, 2 * be);
            bulk_load(s_nx, m.next + eb, be, &s_bar);
            bulk_load(s_org, m.origin + eb, be, &s_bar);
            s_r = 0;
        } else {
            // a tile inside one mesh has its origins contiguous in the local
            // array, from entry L0: bulk-copy from L0 rounded down to 16 bytes
            // (r entries early) to 16 bytes past the end, which stays inside
            // the mesh's entries since at least 3 border half-edges follow
            // its interior ones
            const int32_t j = mesh_of(w.loc_seg, w.loc_t_off, w.loc_n, t0);
            s_j0 = j;
            const bool one = w.loc_aligned && 3 * __ldg(w.loc_t_off + j + 1) >= eb + (int32_t)ne;
            const int32_t L0 = eb + __ldg(w.loc_h_off + j) - 3 * __ldg(w.loc_t_off + j);
            const int32_t r = L0 & 3;
            const uint32_t bo = ((uint32_t)(r + (int32_t)ne) * 4u + 15u) & ~15u;
            mbar_arrive_expect_tx(&s_bar, one ? be + bo : be);
            bulk_load(s_nx, m.next + eb, be, &s_bar);
            if (one) bulk_load(s_org, w.loc_origin + (L0 - r), bo, &s_bar);
            s_r = one ? r : -1;
        }
    }
    __syncthreads();
    if (BATCH && s_r < 0) {
        // origin from the meshes' own arrays (already local vertex ids): union
        // half-edge x of mesh j is local entry x + h_off[j] - 3 t_off[j].  All
        // of a thread's addresses first, then all its loads, then the stores,
        // so its loads are in flight together.
        constexpr int NK = E / NT;
        static_assert(E % NT == 0, "whole rounds of the tile's half-edges");
        int32_t j = s_j0;
        int32_t jn = 3 * __ldg(w.loc_t_off + j + 1);
        int32_t sb = __ldg(w.loc_h_off + j) - 3 * __ldg(w.loc_t_off + j);
        int32_t at[NK];
#pragma unroll
        for (int k = 0; k < NK; k++) {
            const uint32_t d = threadIdx.x + (uint32_t)(k * NT);
            const int32_t x = eb + (int32_t)d;
            at[k] = -1;
            if (d < ne) {
                while (x >= jn && j + 1 < w.loc_n) {
                    j++;
                    jn = 3 * __ldg(w.loc_t_off + j + 1);
                    sb = __ldg(w.loc_h_off + j) - 3 * __ldg(w.loc_t_off + j);
                }
                at[k] = x + sb;
            }
        }
#pragma unroll
        for (int k = 0; k < NK; k++) at[k] = at[k] >= 0 ? __ldg(w.loc_origin + at[k]) : 0;
#pragma unroll
        for (int k = 0; k < NK; k++) {
            const uint32_t d = threadIdx.x + (uint32_t)(k * NT);
            if (d < ne) s_org[d] = at[k];
        }
        __syncthreads();
    }
    const int32_t *so = s_org + (s_r > 0 ? s_r : 0);  // the tile's origins
    // the warps before this one in the tile, and this warp's own total
    const unsigned long long wt = lane <= wid ? w.poly_wtot[(int64_t)tile * NW + lane] : 0ull;
    const unsigned long long wbase =
        ((unsigned long long)__reduce_add_sync(0xffffffffu, lane < wid ? (uint32_t)(wt >> 32) : 0u) << 32) |
        __reduce_add_sync(0xffffffffu, lane < wid ? (uint32_t)wt : 0u);
    const unsigned long long wtot = __shfl_sync(0xffffffffu, wt, wid);
    // the tiles before this one: those of the groups before its group, then
    // those before it in its group
    const unsigned long long tbase = w.group_pre[tile / SCAN_THREADS] + w.tile_pre[tile];
    // the warp's words, the first round of 32 while the tile's copy is under way
    const int32_t nwords = (int32_t)(wtot >> 32);
    const uint32_t *recs = w.poly_rec + t0 + WT * wid;
    uint32_t first = lane < nwords ? recs[lane] : 0u;
    if (!__all_sync(0xffffffffu, mbar_wait(&s_bar, 0))) {
        if (lane == 0) {
            atomicOr(&w.ctrl->error, DEV_ERR_TIMEOUT);
            if (wid == 0) mbar_wait(&s_bar, 0);
        }
        return;
    }
    const unsigned long long base = tbase + wbase;  // this warp's first polygon and entry
    const int64_t P0 = (int64_t)(base >> 32);
    const int64_t NF0 = (int64_t)(base & 0xffffffffull);
    const int64_t wlen = (int64_t)(wtot & 0xffffffffull);
    if (P0 + (int64_t)(wtot >> 32) > (int64_t)m.T || NF0 + wlen > (int64_t)HI) {
        if (lane == 0) atomicOr(&w.ctrl->error, DEV_ERR_CAPACITY);
        return;  // warp-uniform
    }
    int32_t *he_out = w.he_list + NF0;
    int32_t *v_out = w.v_list + NF0;
    int32_t *st = s_stage + wid * WCAP;  // half-edges (of the union), until they go out
    int4 *cross = s_cross + wid * LIST_CROSS;
    const int32_t tw0 = t0 + WT * wid;  // the warp's first triangle
    // in a batch, the mesh of the warp's first triangle (from the mesh
    // table); each lane steps forward from it to the mesh of its polygon
    int32_t mi = 0;
    if (BATCH) {
        mi = __shfl_sync(0xffffffffu, lane == 0 ? mesh_of(w.loc_seg, w.loc_t_off, w.loc_n, min(tw0, m.T - 1)) : 0, 0);
        // the warp holding a mesh's first triangle writes the mesh's first
        // polygon: its own first polygon plus its minima before the mesh
        const int32_t te = min(tw0 + WT, t0 + nt);
        int32_t j = mi;
        while (j < w.loc_n && __ldg(w.loc_t_off + j) < tw0) j++;
        for (; j < w.loc_n; j++) {
            const int32_t tj = __ldg(w.loc_t_off + j);
            if (tj >= te) break;
            int32_t before = 0;
            for (int32_t r = 0; r < nwords; r += 32) {
                const uint32_t v = r + lane < nwords ? recs[r + lane] : ~0u;
                const bool b = v != ~0u && tw0 + (int32_t)((v & REC_E_MASK) / 3u) < tj;
                before += __popc(__ballot_sync(0xffffffffu, b));
            }
            if (lane == 0) w.loc_poly_off[j] = (int32_t)P0 + before;
        }
    }
    const int32_t *origin = BATCH ? w.loc_origin : m.origin;
    // entry pos of the warp's range: half-edge x; she, sb: from a union
    // half-edge to its mesh's own half-edge and to its entry in the local
    // arrays (used past the staging buffer only)
    auto emit = [&](int32_t pos, int32_t x, int32_t she, int32_t sb) {
        if (pos < WCAP) {
            st[pos] = x;
        } else {
            const uint32_t d = (uint32_t)(x - eb);
            he_out[pos] = x - she;
            v_out[pos] = d < ne ? so[d] : __ldg(origin + x + sb);
        }
    };
    // the k half-edges from x on, in and out of the tile
    auto list_on = [&](int32_t x, int32_t pos, int32_t k, int32_t she, int32_t sb) {
        for (; k > 0; k--, pos++) {
            emit(pos, x, she, sb);
            const uint32_t d = (uint32_t)(x - eb);
            x = d < ne ? s_nx[d] : ld_chain(m.next + x);
        }
    };
    auto mesh_shift = [&](int32_t j, int32_t &she, int32_t &sb) {
        she = 3 * __ldg(w.loc_t_off + j);
        sb = __ldg(w.loc_h_off + j) - she;
    };
    const uint32_t below = (1u << lane) - 1u;
    const uint32_t nxa = smem_u32(s_nx) - 4u * (uint32_t)eb;  // shared address of next[0]
    const int32_t mw = mi;  // in a batch, the mesh of the warp's first triangle
    int32_t pos0 = 0;  // within the warp's range
    uint32_t ncross = 0;
    for (int32_t r = 0; r < nwords; r += 32) {
        const uint32_t v = first;
        first = r + 32 + lane < nwords ? recs[r + 32 + lane] : 0u;  // the next round's
        int32_t k = (int32_t)(v >> REC_LEN_SHIFT);
        const int32_t ch = (int32_t)((v >> REC_X_SHIFT) & REC_X_MASK);
        int32_t x = eb + 3 * WT * wid + (int32_t)(v & REC_E_MASK);
        if (k == (int32_t)REC_LEN_MAX) {  // or longer: measure it
            int32_t y = x;
            k = 0;
            do {
                y = ld_chain(m.next + y);
                k++;
            } while (y != x && k < HI);
        }
        int32_t inc = k;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        int32_t pos = pos0 + inc - k;
        pos0 += __shfl_sync(0xffffffffu, inc, 31);
        if (k > 0) {
            const int64_t p = P0 + r + lane;
            int32_t she = 0, sb = 0;
            if (BATCH) {
                while (mi + 1 < w.loc_n && __ldg(w.loc_t_off + mi + 1) <= x / 3) mi++;
                mesh_shift(mi, she, sb);
            }
            w.seeds[p] = x - she;
            w.offsets[p] = (int32_t)NF0 + pos;
            if (pos + k <= WCAP) {
                do {  // inside the tile
                    st[pos++] = x;
                    x = lds_i32(nxa + 4u * (uint32_t)x);
                } while (--k > 0 && (uint32_t)(x - eb) < ne);
            } else {
                do {
                    emit(pos++, x, she, sb);
                    x = lds_i32(nxa + 4u * (uint32_t)x);
                } while (--k > 0 && (uint32_t)(x - eb) < ne);
            }
        }
        // the rest of a crossing polygon comes later, from its chunks or, if
        // none holds its walk, from x on
        const uint32_t bal = __ballot_sync(0xffffffffu, k > 0);
        if (k > 0) {
            const uint32_t slot = ncross + __popc(bal & below);
            if (slot < LIST_CROSS) {
                cross[slot] = make_int4(ch ? -ch : x, pos, k, mi);
            } else {
                int32_t she = 0, sb = 0;
                if (BATCH) mesh_shift(mi, she, sb);
                list_on(x, pos, k, she, sb);
            }
        }
        ncross = min(ncross + __popc(bal), (uint32_t)LIST_CROSS);
    }
    __syncwarp();
    // crossing polygons: half a warp copies a chunk, four pairs of chunks in
    // flight
    const int32_t cown = t0 / XQUOTA - 1;  // the tile's chunks, from 1 on
    const int hl = lane & 15;
    const uint32_t hmask = 0xffffu << (lane & 16);
    for (uint32_t q0 = 0; q0 < ncross; q0 += 8) {
        int4 c[4];
        int32_t h[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const uint32_t q = q0 + 2 * j + (lane >> 4);
            c[j] = q < ncross ? cross[q] : make_int4(0, 0, 0, 0);
            h[j] = c[j].x < 0 ? ld_chain(w.cross_pool + 16 * (int64_t)(cown - c[j].x) + hl) : 0;
        }
#pragma unroll
        for (int j = 0; j < 4; j++) {
            if (c[j].x >= 0) continue;
            int32_t pos = c[j].y, k = c[j].z, y = h[j], she = 0, sb = 0;
            if (BATCH && pos + k > WCAP) mesh_shift(c[j].w, she, sb);
            while (true) {
                if (hl < min(k, XCHUNK)) emit(pos + hl, y, she, sb);
                k -= XCHUNK;
                if (k <= 0) break;
                pos += XCHUNK;
                y = ld_chain(w.cross_pool + 16 * (int64_t)__shfl_sync(hmask, y, 15, 16) + hl);
            }
        }
    }
    if ((uint32_t)lane < ncross) {
        const int4 c = cross[lane];
        if (c.x >= 0) {
            int32_t she = 0, sb = 0;
            if (BATCH) mesh_shift(c.w, she, sb);
            list_on(c.x, c.y, c.z, she, sb);
        }
    }
    __syncwarp();
    const int32_t nb = (int32_t)min(wlen, (int64_t)WCAP);
    // the staged half-edges of the range with the vertices they leave, up to
    // four loads of a lane in flight
    int32_t mo = mw, oshe = 0, osb = 0, oend = 0;
    if (BATCH) {
        oshe = 3 * __ldg(w.loc_t_off + mo);
        oend = 3 * __ldg(w.loc_t_off + mo + 1);
        osb = __ldg(w.loc_h_off + mo) - oshe;
    }
    for (int32_t k0 = lane; k0 < nb; k0 += 128) {
        int32_t x[4], v[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int32_t k = k0 + 32 * j;
            if (k >= nb) continue;
            x[j] = st[k];
            if (BATCH) {  // the meshes ascend along the range
                while (x[j] >= oend && mo + 1 < w.loc_n) {
                    mo++;
                    oshe = oend;
                    oend = 3 * __ldg(w.loc_t_off + mo + 1);
                    osb = __ldg(w.loc_h_off + mo) - oshe;
                }
            }
            const uint32_t d = (uint32_t)(x[j] - eb);
            v[j] = d < ne ? so[d] : __ldg(origin + x[j] + osb);
            x[j] -= oshe;
        }
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int32_t k = k0 + 32 * j;
            if (k < nb) {
                he_out[k] = x[j];
                v_out[k] = v[j];
            }
        }
    }
}

// The control block into pinned host memory.  A kernel's store and not a copy:
// copies of one direction go through one engine in order, so the 32-byte copy of
// polylla_generate_host waited behind the links on their way out (0.5 M triangles:
// 272 us a call, 264 with the store); after a generate alone it took 2 us longer.
__global__ void k_ctrl_out(const int32_t *ctrl, int32_t *host) {
    if (threadIdx.x < sizeof(DevCtrl) / sizeof(int32_t)) host[threadIdx.x] = ctrl[threadIdx.x];
}

cudaError_t launch_ctrl_out(const Work &w, DevCtrl *host, cudaStream_t s) {
    return launch_kernel(k_ctrl_out, 1, 32, 0, s, false, reinterpret_cast<const int32_t *>(w.ctrl),
                         reinterpret_cast<int32_t *>(host));
}

// ---- launch configurations (tile triangles, triangles per thread) ------------
template <int TILE, int IPT>
constexpr size_t count_smem() {
    // next and flags of the tile, a word per triangle, and its crossing walks
    return (size_t)3 * TILE * sizeof(int32_t) + TILE + TILE * sizeof(uint32_t) +
           (size_t)(count_cross<TILE>() + (count_cross<TILE>() & 1)) * sizeof(int2);
}
template <int TILE, int IPT>
constexpr size_t list_smem() {
    // next and origin of the tile (origin with 4 entries to spare for an
    // unaligned start), and per warp its staged entries and its crossing
    // polygons
    return (size_t)(2 * 3 * TILE + 4 + TILE / IPT / 32 * list_stage<IPT>()) * sizeof(int32_t) + TILE / IPT / 32 * LIST_CROSS * sizeof(int4);
}

#define POLYGON_CONFIGS(X) \
    X(1024, 4)             \
    X(1024, 2)             \
    X(2048, 4)             \
    X(2048, 2)             \
    X(4096, 4)

bool polygons_config_valid(int32_t tile, int32_t items) {
#define X(TL, N) \
    if (tile == TL && items == N) return true;
    POLYGON_CONFIGS(X)
#undef X
    return false;
}

int polygons_configure() {
#define X(TL, N)                                                                                             \
    if (cudaFuncSetAttribute(k_poly_count<TL, N>, cudaFuncAttributeMaxDynamicSharedMemorySize,               \
                             (int)count_smem<TL, N>()) != cudaSuccess ||                                        \
        cudaFuncSetAttribute(k_poly_list<TL, N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,         \
                             (int)list_smem<TL, N>()) != cudaSuccess ||                                         \
        cudaFuncSetAttribute(k_poly_list<TL, N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,          \
                             (int)list_smem<TL, N>()) != cudaSuccess)                                           \
        return -1;
    POLYGON_CONFIGS(X)
#undef X
    return 0;
}

// resident CTAs per SM of the listing kernel (the larger of the two)
int polygons_blocks_per_sm(int32_t tile, int32_t items) {
    int nb = 0;
#define X(TL, N)                                                                                          \
    if (tile == TL && items == N) {                                                                  \
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_poly_list<TL, N, false>, TL / N, list_smem<TL, N>()) != \
            cudaSuccess)                                                                                  \
            nb = 0;                                                                                       \
    }
    POLYGON_CONFIGS(X)
#undef X
    return nb;
}

// the two kernels of the output stage (an unknown configuration takes the
// default one: the tuning entry points accept only valid ones)
void launch_poly_count(const MeshView &m, const Work &w, cudaStream_t s, bool chained) {
#define X(TL, N)                                                                            \
    if (w.out_tile == TL && w.out_items == N) {                                        \
        launch_kernel(k_poly_count<TL, N>, (m.T + TL - 1) / TL, TL / (2 * N), count_smem<TL, N>(), s, chained, m, w);         \
        return;                                                                             \
    }
    POLYGON_CONFIGS(X)
#undef X
    constexpr int TL = OUT_TILE_DEFAULT, N = OUT_ITEMS_DEFAULT;
    launch_kernel(k_poly_count<TL, N>, (m.T + TL - 1) / TL, TL / (2 * N), count_smem<TL, N>(), s, chained, m, w);
}

void launch_tile_scan(const MeshView &m, const Work &w, cudaStream_t s, bool chained) {
    const int32_t tile = polygons_config_valid(w.out_tile, w.out_items) ? w.out_tile : OUT_TILE_DEFAULT;
    const int32_t n = (m.T + tile - 1) / tile;
    launch_kernel(k_tile_scan, (n + SCAN_THREADS - 1) / SCAN_THREADS, SCAN_THREADS, 0, s, chained, m, w, n);
}

void launch_poly_list(const MeshView &m, const Work &w, cudaStream_t s, bool chained) {
#define X(TL, N)                                                                            \
    if (w.out_tile == TL && w.out_items == N) {                                        \
        if (w.loc_n > 0) launch_kernel(k_poly_list<TL, N, true>, (m.T + TL - 1) / TL, TL / N, list_smem<TL, N>(), s, chained, m, w); \
        else launch_kernel(k_poly_list<TL, N, false>, (m.T + TL - 1) / TL, TL / N, list_smem<TL, N>(), s, chained, m, w);      \
        return;                                                                             \
    }
    POLYGON_CONFIGS(X)
#undef X
    constexpr int TL = OUT_TILE_DEFAULT, N = OUT_ITEMS_DEFAULT;
    if (w.loc_n > 0) launch_kernel(k_poly_list<TL, N, true>, (m.T + TL - 1) / TL, TL / N, list_smem<TL, N>(), s, chained, m, w);
    else launch_kernel(k_poly_list<TL, N, false>, (m.T + TL - 1) / TL, TL / N, list_smem<TL, N>(), s, chained, m, w);
}

}  // namespace polylla
