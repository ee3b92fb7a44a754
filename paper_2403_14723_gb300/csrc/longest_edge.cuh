// The longest edge of a triangle, shared by the kernels that label triangles.
#pragma once

#include "polylla_internal.cuh"

namespace polylla {

// ===========================================================================
// Stage 1: longest edge of each triangle (Algorithm 2 / Algorithm 8).
//
// The reference value is the float64 squared length
//     d = fl(fl(dx*dx) + fl(dy*dy)),  dx = fl(xb - xa),  dy = fl(yb - ya),
// and the longest edge is the largest d, equal d going to the smaller edge id
// min(e, twin e).  GB300 issues float64 at a small fraction of its float32
// rate, so the argmax is first decided by a certified float32 filter and
// only triangles the filter cannot decide take the float64 path.
//
// Filter.  Each coordinate x is truncated to float32 (x^ keeps the top 23
// significand bits, so |x^ - x| <= 2^-23 |x| = 2u|x| with u = 2^-24, and
// |x^| <= |x|) by bit manipulation (no float64 instruction); coordinates
// outside [2^-126, 2^61) in magnitude (zero included) send the triangle to
// the float64 path.  With S = |x^a| + |x^b| the float32 difference
// dx^ = fl32(x^b - x^a) satisfies |dx^ - dx| <= 3.0001 u Sx, hence an edge's
// D^ = fl32(dx^ dx^ + fl32(dy^ dy^)) lies within
//   6.0003u (Sx|dx^| + Sy|dy^|) + 9.0007u^2 (Sx^2 + Sy^2) + 2.0002u D^
//   + (float64 rounding of d, < 2^-50 d)
// of d.  One bound serves the three edges: with X, Y the largest |x^|, |y^| of
// the triangle, DX, DY the largest |dx^|, |dy^| and D the largest D^,
//   B = 12.3u (X DX + Y DY) + 36.5u^2 (X^2 + Y^2) + 4.5u D + 2^-118
// (S <= 2X; 2.5 % over 12.0006 and 1 % over 36.003 for B's own roundings, 2.5u D
// for that of the comparison, an absolute term for float32 underflow).  If the
// largest D^ exceeds the second by more than 2B, the float64 argmax is the same
// edge and has no tie.  A bound for each edge was tighter (0.35 % of jittered grid
// cells' triangles to the float64 path against 0.48 %) but took half of the filter's
// instructions.
// ===========================================================================

__device__ __forceinline__ double sq_len_f64(double2 a, double2 b) {
    double dx = __dsub_rn(b.x, a.x);
    double dy = __dsub_rn(b.y, a.y);
    return __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
}

// The edges of the largest float64 length, a bit each (several: a tie).  out is an
// edge known to be shorter (3: none): its length is left out, since float64 is what
// this path spends its time on.
static __device__ __noinline__ uint32_t longest_exact(double2 p0, double2 p1, double2 p2, uint32_t out) {
    // from the vertex after it on: edges a, b and (perhaps out) c
    const uint32_t a = out == 0u ? 1u : (out == 1u ? 2u : 0u), b = a == 2u ? 0u : a + 1u;
    const double2 pa = a == 0u ? p0 : (a == 1u ? p1 : p2);
    const double2 pb = a == 0u ? p1 : (a == 1u ? p2 : p0);
    const double2 pc = a == 0u ? p2 : (a == 1u ? p0 : p1);
    const double da = sq_len_f64(pa, pb), db = sq_len_f64(pb, pc);
    uint32_t best = (db > da ? 0u : 1u << a) | (db >= da ? 1u << b : 0u);
    if (out > 2u) {  // a is 0, b is 1, c is 2
        const double dc = sq_len_f64(pc, pa), d = db > da ? db : da;
        best = (dc > d ? 0u : best) | (dc >= d ? 4u : 0u);
    }
    return best;
}

// TW: the twins of the triangle's half-edges for the exact path, as
// tw(k) (read only when the filter cannot decide)
template <typename TW>
__device__ __forceinline__ uint32_t longest_of(double2 p0, double2 p1, double2 p2, int32_t e0, TW tw) {
    uint32_t far = 0;
    const float x0 = trunc_to_f32_far(p0.x, far), y0 = trunc_to_f32_far(p0.y, far);
    const float x1 = trunc_to_f32_far(p1.x, far), y1 = trunc_to_f32_far(p1.y, far);
    const float x2 = trunc_to_f32_far(p2.x, far), y2 = trunc_to_f32_far(p2.y, far);
    const float ax = __fsub_rn(x1, x0), ay = __fsub_rn(y1, y0);
    const float bx = __fsub_rn(x2, x1), by = __fsub_rn(y2, y1);
    const float cx = __fsub_rn(x0, x2), cy = __fsub_rn(y0, y2);
    const float d0 = fmaf(ax, ax, __fmul_rn(ay, ay));
    const float d1 = fmaf(bx, bx, __fmul_rn(by, by));
    const float d2 = fmaf(cx, cx, __fmul_rn(cy, cy));
    const float hi01 = fmaxf(d0, d1), lo01 = fminf(d0, d1);
    const float dm = fmaxf(hi01, d2), second = fmaxf(lo01, fminf(hi01, d2));
    uint32_t k = d1 > d0 ? 1u : 0u;
    if (d2 > hi01) k = 2u;
    const float X = fmaxf(fmaxf(fabsf(x0), fabsf(x1)), fabsf(x2)), Y = fmaxf(fmaxf(fabsf(y0), fabsf(y1)), fabsf(y2));
    const float DX = fmaxf(fmaxf(fabsf(ax), fabsf(bx)), fabsf(cx)), DY = fmaxf(fmaxf(fabsf(ay), fabsf(by)), fabsf(cy));
    const float u = 5.9604644775390625e-08f;  // 2^-24
    // 2B
    const float b2 = fmaf(24.6f * u, fmaf(X, DX, Y * DY),
                          fmaf(73.0f * u * u, fmaf(X, X, Y * Y), fmaf(9.0f * u, dm, 6.0e-36f)));
    const bool sure = far < TRUNC_SPAN && __fsub_rn(dm, second) > b2;
    if (!sure) {
        // the shortest edge, where the filter is sure of it
        const float least = fminf(lo01, d2);
        uint32_t out = least == d2 ? 2u : (least == d0 ? 0u : 1u);
        if (!(far < TRUNC_SPAN && __fsub_rn(dm, least) > b2)) out = 3u;
        // equal lengths go to the smaller edge id min(e, twin e).  Only they read
        // the twins: every triangle of this path waited for three loads from memory.
        const uint32_t ties = longest_exact(p0, p1, p2, out);
        k = ties >> 1;  // of one bit: 1, 2 or 4
        if (ties & (ties - 1u)) {
            int32_t least_id = INT32_MAX;
#pragma unroll
            for (int j = 0; j < 3; j++) {
                if (!((ties >> j) & 1u)) continue;
                const int32_t id = min(e0 + j, tw(j));
                if (id < least_id) {
                    least_id = id;
                    k = (uint32_t)j;
                }
            }
        }
    }
    return k;
}

}  // namespace polylla
