// Convexification of the Polylla mesh (post-processing).  Section 4.2 keeps
// every half-edge of the triangulation, relinking instead of deleting, so
// that a later step can turn non-convex polygons into convex ones; the
// paper gives no method.  This one splits every reflex corner with the
// fewest edges of the triangulation itself:
//   - the corner of a polygon at a frontier half-edge e is (e, x = next[e])
//     at v = target(e); directions leave v, dir(h) = target(h) - v, and the
//     corner's first side is twin(e), dir = origin(e) - v;
//   - cross(a, b) = a.x b.y - a.y b.x, every operation in binary64 rounded
//     to nearest on its own (no FMA); b lies within a half turn clockwise of
//     a iff cross(a, b) <= 0; the corner is reflex iff cross(dir twin e,
//     dir x) > 0;
//   - the corner's interior half-edges, clockwise: y1 = the triangle's next
//     of e, then y = CW(y) = next(twin y), up to x (the relink's rotation);
//     from cur = twin(e) the last of them within a half turn of cur becomes
//     a chord and the new cur, until x is within a half turn of cur.
// Both halves of every chord join the frontier; the links around the chord
// ends are redone exactly as the repair's, and the output stage lists the
// new polygons.  Every turn test first tries a certified float32 filter
// (cross_sign) and computes the binary64 expression only when the filter
// cannot decide, so the decisions are those of binary64 throughout.
#include "polylla_internal.cuh"

namespace polylla {

__device__ __forceinline__ double cross_rn(double ax, double ay, double bx, double by) {
    return __dsub_rn(__dmul_rn(ax, by), __dmul_rn(ay, bx));
}

// A vertex: its id and the float32 truncations of its coordinates (the
// binary64 path reloads the coordinates themselves).
struct Pt {
    float x, y;
    uint32_t bad;  // a coordinate the filter cannot take
    int32_t v;
};

__device__ __forceinline__ Pt load_pt(const double2 *__restrict__ xy, int32_t v) {
    Pt r;
    const double2 p = __ldg(xy + v);
    r.bad = 0;
    r.x = trunc_to_f32(p.x, r.bad);
    r.y = trunc_to_f32(p.y, r.bad);
    r.v = v;
    return r;
}

// Sign (+1, 0, -1) of the binary64 expression cross(a - v, b - v) =
// fl(fl(ux wy) - fl(uy wx)), ux = fl(a.x - v.x), ... (every operation
// rounded to nearest, no FMA): the turn test of the convexification.
//
// Float32 filter (u = 2^-24).  Truncated coordinates satisfy |x - x^| <=
// 2u|x^|, so a float32 difference d^ = fl32(a^ - v^) is within
// e = 3uS of the exact a - v, S = |a^| + |v^|.  For the products,
// |ux wy - ux^ wy^| <= e_ux|wy^| + |ux^|e_wy + e_ux e_wy, plus u|p^| for the
// rounding of p^ = fl32(ux^ wy^); the final difference adds u|c^|.  So the
// exact cross c lies within
//   B = sum over both products (e1|f2| + |f1|e2 + e1 e2 + u|p|) + u|c^|
// of c^.  The binary64 value is within 2^-50 (|p1| + |p2|) of c, far below
// the 1 % margin added to B (with an absolute 2^-120 for float32 underflow);
// so |c^| > B gives the binary64 sign, and a nonzero one.  Otherwise, or
// for coordinates the truncation cannot take, the binary64 expression
// decides, computed exactly as the oracle does.
__device__ int cross_sign(const double2 *__restrict__ xy, const Pt &a, const Pt &b, const Pt &v) {
    if (!(a.bad | b.bad | v.bad)) {
        const float u = 5.9604644775390625e-08f;  // 2^-24
        const float ux = __fsub_rn(a.x, v.x), uy = __fsub_rn(a.y, v.y);
        const float wx = __fsub_rn(b.x, v.x), wy = __fsub_rn(b.y, v.y);
        const float e_ux = 3.001f * u * (fabsf(a.x) + fabsf(v.x)), e_uy = 3.001f * u * (fabsf(a.y) + fabsf(v.y));
        const float e_wx = 3.001f * u * (fabsf(b.x) + fabsf(v.x)), e_wy = 3.001f * u * (fabsf(b.y) + fabsf(v.y));
        const float p1 = __fmul_rn(ux, wy), p2 = __fmul_rn(uy, wx);
        const float c = __fsub_rn(p1, p2);
        float B = e_ux * fabsf(wy) + fabsf(ux) * e_wy + e_ux * e_wy + u * fabsf(p1);
        B += e_uy * fabsf(wx) + fabsf(uy) * e_wx + e_uy * e_wx + u * fabsf(p2);
        B = 1.01f * (B + u * fabsf(c)) + 7.5e-37f;
        if (c > B) return 1;
        if (c < -B) return -1;
    }
    const double2 pa = __ldg(xy + a.v), pb = __ldg(xy + b.v), pv = __ldg(xy + v.v);
    const double c = cross_rn(__dsub_rn(pa.x, pv.x), __dsub_rn(pa.y, pv.y), __dsub_rn(pb.x, pv.x),
                              __dsub_rn(pb.y, pv.y));
    return c > 0.0 ? 1 : (c < 0.0 ? -1 : 0);
}

// A slot at the end of a list shared by the whole grid for every lane of the
// (whole) warp that asks for one: one atomic per warp and call.  List order is
// free: every consumer of these lists treats them as sets.
__device__ __forceinline__ int32_t warp_slot(int32_t *count, bool want) {
    const uint32_t bal = __ballot_sync(0xffffffffu, want);
    const int lane = (int)(threadIdx.x & 31u);
    int32_t base = 0;
    if (lane == 0 && bal) base = atomicAdd(count, __popc(bal));
    return __shfl_sync(0xffffffffu, base, 0) + __popc(bal & ((1u << lane) - 1u));
}

// ===========================================================================
// The corners: for a frontier half-edge e = 3t + k, v = target(e) is the
// triangle's vertex k + 1, origin(e) its vertex k, and the corner's other
// side is x = next[e].  k_convex_reflex tests every corner; k_convex_chords
// chooses a reflex corner's chords (appended to the list; the frontier bits are
// set by the next kernel, so every thread reads the frontier of the Polylla
// mesh).
// ===========================================================================
// k_convex_reflex: one thread per triangle; the reflex corners go to a list, so
// that the chord search (a chain of dependent loads) runs one reflex corner per
// thread in k_convex_chords instead of holding up a warp of mostly convex
// corners.  A corner whose successor is the next half-edge of its own triangle
// is a triangle's angle, less than a half turn: only the last half-edge of the
// triangle's cyclic run of frontier half-edges has a link across an edge, so a
// triangle holds at most one reflex corner.  The list's counter takes one atomic
// per block of CR_THREADS triangles: with one per warp and local half-edge (94 k
// on 1 M triangles, one after the other in L2) the kernel took 64 us there; generate
// and convexify together went from 280 to 217 us.
constexpr int CR_THREADS = 512;
__global__ void __launch_bounds__(CR_THREADS) k_convex_reflex(MeshView m, Work w, int32_t *reflex, int32_t *n_reflex,
                                                              int32_t cap) {
    constexpr int NW = CR_THREADS / 32;
    __shared__ uint32_t s_n[NW];
    __shared__ int32_t s_base;
    chain_next();
    chain_wait();
    const int lane = (int)(threadIdx.x & 31u), wid = (int)(threadIdx.x >> 5);
    for (int64_t b = (int64_t)blockIdx.x * CR_THREADS; b < m.T; b += (int64_t)gridDim.x * CR_THREADS) {
        const int64_t t = b + threadIdx.x;
        const uint32_t F = t < m.T ? w.flags[t] & 7u : 0u;
        int32_t e = 0;
        bool is_reflex = false;
        const uint32_t last = F & ~((F >> 1) | (F << 2));  // one bit at most: 1, 2 or 4
        if (last) {
            const int32_t e0 = 3 * (int32_t)t, k = (int32_t)(last >> 1);
            e = e0 + k;
            const int32_t x = m.next[e];
            const Pt pa = load_pt(m.xy, __ldg(m.origin + e));                      // origin(e)
            const Pt pv = load_pt(m.xy, __ldg(m.origin + e0 + (k == 2 ? 0 : k + 1)));  // target(e)
            const Pt pw = load_pt(m.xy, __ldg(m.origin + nx_of(x)));               // target(x)
            is_reflex = cross_sign(m.xy, pa, pw, pv) > 0;
        }
        const uint32_t bal = __ballot_sync(0xffffffffu, is_reflex);
        if (lane == 0) s_n[wid] = (uint32_t)__popc(bal);
        __syncthreads();
        if (wid == 0) {
            const uint32_t n = lane < NW ? s_n[lane] : 0u;
            uint32_t inc = n;
#pragma unroll
            for (int o = 1; o < NW; o <<= 1) {
                const uint32_t u = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += u;
            }
            if (lane < NW) s_n[lane] = inc - n;
            if (lane == NW - 1) s_base = inc ? atomicAdd(n_reflex, (int32_t)inc) : 0;
        }
        __syncthreads();
        if (is_reflex) {
            const int32_t slot = s_base + (int32_t)s_n[wid] + __popc(bal & ((1u << lane) - 1u));
            if (slot < cap) reflex[slot] = e;
            else atomicOr(&w.ctrl->error, DEV_ERR_CAPACITY);
        }
        __syncthreads();  // s_n and s_base are the next round's
    }
}

// k_convex_chords: one thread per reflex corner e: its chords.  A warp's lanes
// search a chord each and then take their slots together: one atomic per warp
// and chord.
__global__ void __launch_bounds__(256) k_convex_chords(MeshView m, Work w, const int32_t *reflex,
                                                       const int32_t *n_reflex, int32_t cap_reflex, int32_t *list,
                                                       int32_t *count, int32_t cap) {
    chain_next();
    chain_wait();
    int32_t n = *n_reflex;
    if (n > cap_reflex) n = cap_reflex;
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x; b < n; b += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = b + threadIdx.x;
        bool open = i < n;  // the corner left of cur is still reflex
        int32_t x = 0, y = 0, steps = 0;
        Pt pv{}, cur{}, pw{};
        if (open) {
            const int32_t e = reflex[i];
            x = m.next[e];
            y = nx_of(e);
            pv = load_pt(m.xy, __ldg(m.origin + y));           // target(e)
            cur = load_pt(m.xy, __ldg(m.origin + e));          // origin(e)
            pw = load_pt(m.xy, __ldg(m.origin + nx_of(x)));    // target(x)
        }
        // (the first test is the one that put the corner on the list)
        while (__any_sync(0xffffffffu, open)) {
            int32_t best = -1;
            if (open) {
                Pt bp = cur;
                while (y != x) {
                    const int32_t ty = __ldg(m.twin + y);
                    const Pt pd = load_pt(m.xy, __ldg(m.origin + nx_of(y)));  // target(y)
                    if (cross_sign(m.xy, cur, pd, pv) > 0) break;             // beyond a half turn
                    best = y;
                    bp = pd;
                    y = nx_of(ty);                                            // CW(y)
                    if (++steps > w.max_rot) {
                        atomicOr(&w.ctrl->error, DEV_ERR_NONTERMINATING);
                        break;
                    }
                }
                if (steps > w.max_rot) best = -1;
                cur = bp;
            }
            const int32_t slot = warp_slot(count, best >= 0);
            if (best >= 0) {
                if (slot < cap) list[slot] = best;
                else atomicOr(&w.ctrl->error, DEV_ERR_CAPACITY);
            }
            // without a candidate the corner is left reflex
            open = best >= 0 && cross_sign(m.xy, cur, pw, pv) > 0;
        }
    }
}

// both halves of every listed chord join the frontier (F bits of flags)
__global__ void __launch_bounds__(256) k_convex_mark(MeshView m, Work w, const int32_t *list, const int32_t *count,
                                                     int32_t cap) {
    chain_next();
    chain_wait();
    int32_t n = *count;
    if (n > cap) n = cap;
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < 2 * n; i += gridDim.x * blockDim.x) {
        const int32_t c0 = list[i >> 1];
        const int32_t c = (i & 1) ? __ldg(m.twin + c0) : c0;
        const int32_t t = tri_of(c);
        unsigned int *word = reinterpret_cast<unsigned int *>(w.flags) + (t >> 2);
        atomicOr(word, 1u << (8 * (t & 3) + loc_of(c)));
    }
}

void launch_convex_chords(const MeshView &m, const Work &w, int32_t *reflex, int32_t *n_reflex, int32_t *list,
                          int32_t *count, int32_t cap, cudaStream_t s, bool chained) {
    const int64_t want = ((int64_t)m.T + CR_THREADS - 1) / CR_THREADS;
    const int64_t most = 16 * (int64_t)w.persistent_blocks;
    launch_kernel(k_convex_reflex, want < most ? want : most, CR_THREADS, 0, s, chained, m, w, reflex, n_reflex, cap);
    launch_kernel(k_convex_chords, 8 * w.persistent_blocks, 256, 0, s, true, m, w, reflex, n_reflex, cap, list, count,
                  cap);
}

void launch_convex_mark(const MeshView &m, const Work &w, const int32_t *list, const int32_t *count, int32_t cap,
                        cudaStream_t s, bool chained) {
    launch_kernel(k_convex_mark, w.persistent_blocks, 256, 0, s, chained, m, w, list, count, cap);
}

}  // namespace polylla
