// A whole generate of a small mesh in one kernel of one block: every stage of
// kernels_label.cu, kernels_repair.cu and kernels_output.cu on the mesh's twins,
// links and labels in shared memory, with block barriers between the stages.
#include "longest_edge.cuh"
#include "polylla_internal.cuh"

namespace polylla {

// What bounds a small mesh is not its work but the seven launches and the chains
// of loads in each kernel (twin, label, twin, ... through L2).  Here one launch
// does it, and every chain after the first loads runs in shared memory.  Only one
// SM works, so the time grows with the mesh while the staged kernels' does not.
// Generates back to back, this kernel against the staged ones: 8 against 20 us at
// 91 triangles of random points, 12 against 28 at 1,019, 18 against 32 at 2,022,
// 29 against 34 at 3,103, 35 against 34 at 3,982; on jittered grids 12 against 26
// at 882, 18 against 22 at 1,800, 23 against 24 at 2,450, 25 against 24 at 2,888.
// SMALL_MAX lies below where the grids meet.
constexpr int SM_THREADS = 1024;

__device__ __forceinline__ bool small_f1(const uint32_t *s_fl, int32_t e, int32_t HI) {
    return e >= HI || ((s_fl[tri_of(e)] >> loc_of(e)) & 1u);
}

__global__ void __launch_bounds__(SM_THREADS) k_small(MeshView m, Work w) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int32_t T = m.T, HI = 3 * T, HP = (HI + 3) & ~3;
    int32_t *s_tw = reinterpret_cast<int32_t *>(smem);           // [3T] twins
    int32_t *s_nx = s_tw + HP;                                   // [3T] next
    int32_t *s_pv = s_nx + HP;                                   // [3T] prev
    uint32_t *s_fl = reinterpret_cast<uint32_t *>(s_pv + HP);    // [T] flags
    uint8_t *s_le = reinterpret_cast<uint8_t *>(s_fl + T);       // [T] longest edges
    __shared__ int32_t s_tips, s_err;
    __shared__ unsigned long long s_warp[SM_THREADS / 32 + 1];
    const int32_t tid = threadIdx.x, NT = blockDim.x;
    const int lane = tid & 31, wid = tid >> 5;
    if (tid == 0) s_tips = s_err = 0;
    int32_t err = 0;
    // stage 1
    for (int32_t t = tid; t < T; t += NT) {
        int32_t v[3], tw[3];
#pragma unroll
        for (int k = 0; k < 3; k++) v[k] = __ldg(m.origin + 3 * t + k);
#pragma unroll
        for (int k = 0; k < 3; k++) s_tw[3 * t + k] = tw[k] = __ldg(m.twin + 3 * t + k);
        const double2 p0 = __ldg(m.xy + v[0]), p1 = __ldg(m.xy + v[1]), p2 = __ldg(m.xy + v[2]);
        const uint32_t l = longest_of(p0, p1, p2, 3 * t, [&tw](int k) { return tw[k]; });
        s_le[t] = (uint8_t)l;
        w.le[t] = (uint8_t)l;
    }
    __syncthreads();
    // stages 2 and 3, and the links inside the triangles
    for (int32_t t = tid; t < T; t += NT) {
        const uint32_t l = s_le[t];
        uint32_t F = 0, twle = 0;
#pragma unroll
        for (uint32_t k = 0; k < 3; k++) {
            const int32_t tw = s_tw[3 * t + k];
            const bool b = tw >= HI;
            const bool tl = !b && (int32_t)s_le[tri_of(tw)] == loc_of(tw);
            F |= (uint32_t)(b || (k != l && !tl)) << k;
            twle |= (uint32_t)tl << k;
            s_nx[3 * t + k] = 3 * t + (k == 2 ? 0 : k + 1);
            s_pv[3 * t + k] = 3 * t + (k == 0 ? 2 : k - 1);
        }
        const int32_t e = 3 * t + (int32_t)l, tw = s_tw[e];
        const bool seed = tw >= HI || (((twle >> l) & 1u) && e < tw);
        s_fl[t] = F | ((uint32_t)seed << 6) | (F << 8);  // bits 8-10: F0, which no chord changes
    }
    __syncthreads();
    // stage 4: the triangle's one rotation (the last half-edge of its run); a
    // barrier tip's chord (stage 5a) is chosen here: everything in this stage
    // reads the stage-2 labels (s_le, bits 8-10), the chords set bits 0-2
    for (int32_t t = tid; t < T; t += NT) {
        const uint32_t F0 = (s_fl[t] >> 8) & 7u;
        const uint32_t last = F0 & ~((F0 >> 1) | (F0 << 2));
        if (!last) continue;
        const int32_t e = 3 * t + (int32_t)(last >> 1);
        int32_t x = nx_of(e), steps = -1;
        while (true) {
            const int32_t tx = s_tw[x];
            if (tx >= HI) break;
            const int32_t ttx = tri_of(tx);
            if ((int32_t)s_le[tri_of(x)] != loc_of(x) && (int32_t)s_le[ttx] != tx - 3 * ttx) break;
            x = nx_of(tx);
            if (++steps > w.max_rot) {
                err |= DEV_ERR_NONTERMINATING;
                break;
            }
        }
        s_nx[e] = x;
        s_pv[x] = e;
        const int32_t f = s_tw[e];
        if (x != f) continue;
        // the tip of degree steps + 2 left by its only frontier half-edge f
        const int32_t slot = atomicAdd(&s_tips, 1), d = steps + 2;
        if (slot >= w.tip_cap) {
            err |= DEV_ERR_CAPACITY;
            continue;
        }
        int32_t y = f, ty = s_tw[f];
        bool ok = d <= w.max_rot && ty < HI;  // a border twin: not a valid mesh (as in k_chords)
        for (int32_t r = 0; ok && r < (d - 1) / 2 + 1; r++) {
            y = nx_of(ty);
            ty = s_tw[y];
            ok = ty < HI;
        }
        if (ok) {
            atomicOr(s_fl + tri_of(y), 1u << loc_of(y));
            atomicOr(s_fl + tri_of(ty), 1u << loc_of(ty));
        } else {
            err |= DEV_ERR_NONTERMINATING;
            y = -1;
        }
        w.tips[slot] = f;
        w.chords[slot] = y;
    }
    __syncthreads();
    // the links around the chords' ends, four threads a chord
    const int32_t n_tips = min(s_tips, w.tip_cap);
    for (int32_t i = tid; i < 4 * n_tips; i += NT) {
        const int32_t c0 = w.chords[i >> 2];
        if (c0 < 0) continue;
        const int32_t t0 = s_tw[c0], c = i & 1 ? t0 : c0, tc = i & 1 ? c0 : t0;
        int32_t a, b, steps = 0;
        bool ok = true;
        if (i & 2) {
            a = tc;
            b = nx_of(tc);
            while (ok && !small_f1(s_fl, b, HI)) {
                b = nx_of(s_tw[b]);
                ok = ++steps <= w.max_rot;
            }
        } else {
            b = c;
            a = pv_of(c);
            while (ok && !small_f1(s_fl, s_tw[a], HI)) {
                a = pv_of(s_tw[a]);
                ok = ++steps <= w.max_rot;
            }
        }
        if (!ok) {
            err |= DEV_ERR_NONTERMINATING;
            continue;
        }
        s_nx[a] = b;
        s_pv[b] = a;
    }
    __syncthreads();
    // next and prev go out while the polygons are walked
    {
        const int32_t n4 = HI / 4;
        for (int32_t i = tid; i < n4; i += NT) {
            reinterpret_cast<int4 *>(m.next)[i] = reinterpret_cast<const int4 *>(s_nx)[i];
            reinterpret_cast<int4 *>(m.prev)[i] = reinterpret_cast<const int4 *>(s_pv)[i];
        }
        for (int32_t i = 4 * n4 + tid; i < HI; i += NT) {
            m.next[i] = s_nx[i];
            m.prev[i] = s_pv[i];
        }
    }
    // the polygons, NT triangles at a time: (polygons, length) so far
    unsigned long long base = 0;
    for (int32_t tb = 0; tb < T; tb += NT) {
        const int32_t t = tb + tid;
        int32_t e = 0, L = 0;
        if (t < T) {
            uint32_t fl = s_fl[t];
            const uint32_t F = fl & 7u;
            if (F) {
                // only the lowest frontier half-edge can be a polygon's minimum
                const int32_t k = F & 1u ? 0 : F >> 1 & 1u ? 1 : 2;
                e = 3 * t + k;
                if (s_nx[e] > e && s_pv[e] > e) {
                    fl |= 8u << k;
                    int32_t x = s_nx[e];
                    L = 1;
                    while (x > e && L <= HI) {
                        x = s_nx[x];
                        L++;
                    }
                    if (L > HI) err |= DEV_ERR_NONTERMINATING;
                    if (x != e || L > HI) L = 0;
                }
            }
            w.flags[t] = (uint8_t)fl;
        }
        const unsigned long long mine = L ? (1ull << 32) | (uint32_t)L : 0ull;
        unsigned long long inc = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        if (lane == 31) s_warp[wid] = inc;
        __syncthreads();
        if (wid == 0) {
            const unsigned long long q = lane < NT / 32 ? s_warp[lane] : 0ull;
            unsigned long long qi = q;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long u = __shfl_up_sync(0xffffffffu, qi, o);
                if (lane >= o) qi += u;
            }
            if (lane < NT / 32) s_warp[lane] = qi - q;
            if (lane == 31) s_warp[SM_THREADS / 32] = qi;
        }
        __syncthreads();
        const unsigned long long at = base + s_warp[wid] + inc - mine;
        base += s_warp[SM_THREADS / 32];
        const int64_t p = (int64_t)(at >> 32), n = (int64_t)(at & 0xffffffffull);
        if (L && (p >= T || n + L > HI)) {
            err |= DEV_ERR_CAPACITY;
        } else if (L) {
            w.seeds[p] = e;
            w.offsets[p] = (int32_t)n;
            int32_t x = e;
            for (int32_t j = 0; j < L; j++) {
                w.he_list[n + j] = x;
                w.v_list[n + j] = __ldg(m.origin + x);
                x = s_nx[x];
            }
        }
        __syncthreads();  // s_warp is the next round's
    }
    if (err) atomicOr(&s_err, err);
    __syncthreads();
    if (tid == 0) {
        const int64_t P = (int64_t)(base >> 32), NF = (int64_t)(base & 0xffffffffull);
        const bool over = P > T || NF > HI;
        DevCtrl c{};
        c.error = s_err | (over ? DEV_ERR_CAPACITY : 0);
        c.n_tips = s_tips;
        c.n_polygons = (int32_t)(P > T ? T : P);
        c.n_frontier = (int32_t)NF;
        w.offsets[c.n_polygons] = (int32_t)NF;
        *w.ctrl = c;
    }
}

static size_t small_smem(int32_t T) { return 3 * (size_t)((3 * T + 3) & ~3) * sizeof(int32_t) + 5 * (size_t)T + 16; }

int small_configure() {
    return cudaFuncSetAttribute(k_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)small_smem(SMALL_MAX)) ==
                   cudaSuccess
               ? 0
               : -1;
}

void launch_small(const MeshView &m, const Work &w, cudaStream_t s) {
    const int threads = m.T < SM_THREADS ? (m.T + 31) / 32 * 32 : SM_THREADS;
    launch_kernel(k_small, 1, threads, small_smem(m.T), s, false, m, w);
}

}  // namespace polylla
