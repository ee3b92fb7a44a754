// Repair-phase kernels (stage 5a): the chords of the barrier tips join the
// frontier, and the links around their endpoints are redone.  Both run over the
// (short) tip list in a grid-stride loop, so a mesh without tips costs two tiny
// launches.
#include "polylla_internal.cuh"

namespace polylla {

__device__ __forceinline__ bool f1_of(const uint8_t *flags, int32_t e, int32_t HI) {
    if (e >= HI) return true;  // border half-edges are always frontier
    return (flags[tri_of(e)] >> loc_of(e)) & 1u;
}

__device__ __forceinline__ void set_flag_bit(uint8_t *flags, int32_t e, int shift) {
    const int32_t t = tri_of(e);
    unsigned int *word = reinterpret_cast<unsigned int *>(flags) + (t >> 2);
    atomicOr(word, 1u << (8 * (t & 3) + shift + loc_of(e)));
}
// F1 bit (bits 0-2) and walk-start mark (bits 3-5) of half-edge e
__device__ __forceinline__ void set_f1(uint8_t *flags, int32_t e) { set_flag_bit(flags, e, 0); }
__device__ __forceinline__ void set_start(uint8_t *flags, int32_t e) { set_flag_bit(flags, e, 3); }

// ===========================================================================
// Chords (Algorithm 6 first part / Algorithm 11).  For the tip b of degree d
// (counted by the relink's rotation around it) left by the unique stage-2
// frontier half-edge f, the chord is m = CW^r(f) with r = floor((d-1)/2) + 1
// (the inclusive loop "for 0 to (degree-1)/2"), CW(y) = next(twin y).  Both
// halves of m join the frontier (F1).  Tips come only from the stage-2 labels,
// so the result does not depend on the order in which tips are processed.
// One chain of r + 1 loads per tip: 12 us, when every tip also counted its
// degree here, to 8 us on 1 M random points (16.8 k tips).
// ===========================================================================
__global__ void __launch_bounds__(256) k_chords(MeshView m, Work w) {
    chain_next();
    chain_wait();
    const int32_t HI = 3 * m.T;
    int32_t n = w.ctrl->n_tips;
    if (n > w.tip_cap) n = w.tip_cap;
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int32_t d = w.chords[i];
        int32_t y = w.tips[i];
        int32_t ty = ld_chain(m.twin + y);
        // around a tip every edge is interior.  A mesh that was not validated can
        // have a border twin here: the links of the border are not the layout's
        // (and a batch's union holds none), so the walk ends with an error.
        bool ok = d <= w.max_rot && ty < HI;
        for (int32_t s = 0; ok && s < (d - 1) / 2 + 1; s++) {
            y = nx_of(ty);
            ty = ld_chain(m.twin + y);
            ok = ty < HI;
        }
        if (!ok) {
            atomicOr(&w.ctrl->error, DEV_ERR_NONTERMINATING);
            w.chords[i] = -1;
            continue;
        }
        w.chords[i] = y;
        set_f1(w.flags, y);
        set_f1(w.flags, ty);
    }
}

// Blocks of a kernel over a list of unknown length: one per `per` triangles (a
// list longer than that takes the kernel's loop more often), at most the chip
// full.  608 blocks were too many for a small mesh (8 us a launch for nothing) and
// too few for a convexification's chords (several rounds of chains).
static int list_blocks(const MeshView &m, const Work &w, int32_t per) {
    const int64_t want = m.T / per + 1, most = 2 * (int64_t)w.persistent_blocks;
    return (int)(want < most ? want : most);
}

void launch_chords(const MeshView &m, const Work &w, cudaStream_t s, bool chained) {
    launch_kernel(k_chords, list_blocks(m, w, 8192), 256, 0, s, chained, m, w);  // random meshes: a tip per 120 triangles
}

// ===========================================================================
// Links around chord endpoints.  Around a vertex the relink pairs each
// frontier half-edge o leaving it with the next frontier half-edge leaving
// it in clockwise order: next[twin o] = that half-edge.  A chord half-edge c
// inserts itself into that order, so only the two links touching c change:
//   after c : y = first F1 half-edge clockwise from c  -> next[twin c] = y
//   before c: z = first F1 half-edge counter-clockwise from c (CCW(z) =
//             twin(prev z)) -> next[twin z] = c
// Every other link keeps its stage-4 value.  Two chords at one vertex write
// the link between them with the same value, so no ordering is needed.
// Every half-edge whose next or prev changes gets the walk-start mark (the
// polygon kernel needs the marks to be a superset of the polygon minima).
// ===========================================================================
// in a batch, a union link a -> b (both interior, one mesh) in the mesh's own
// next/prev as well
struct LocalLinks {
    int32_t sh, ho;  // 3 t_off and h_off of the mesh; ho < 0: a single mesh
    __device__ void link(const Work &w, int32_t a, int32_t b) const {
        if (ho < 0) return;
        w.loc_next[ho + (a - sh)] = b - sh;
        w.loc_prev[ho + (b - sh)] = a - sh;
    }
};

// one chord half-edge c with twin tc: the link after it (cw) or before it.  A
// step's label and the next step's twin are fetched together.
__device__ __forceinline__ void relink_around(const MeshView &m, const Work &w, int32_t c, int32_t tc, bool cw,
                                              int32_t HI) {
    LocalLinks loc{0, -1};
    if (w.loc_n > 0) {
        const int32_t mj = mesh_of(w.loc_seg, w.loc_t_off, w.loc_n, tri_of(c));
        loc.sh = 3 * __ldg(w.loc_t_off + mj);
        loc.ho = __ldg(w.loc_h_off + mj);
    }
    int32_t a, b;  // the link a -> b
    int32_t steps = 0;
    if (cw) {
        // clockwise neighbour: the twin of y is read before y's label is known
        // (y is interior: next of an interior half-edge)
        a = tc;
        b = nx_of(tc);
        while (true) {
            const int32_t tb = ld_chain(m.twin + b);
            if (f1_of(w.flags, b, HI)) break;
            b = nx_of(tb);
            if (++steps > w.max_rot) { atomicOr(&w.ctrl->error, DEV_ERR_NONTERMINATING); return; }
        }
    } else {
        // counter-clockwise neighbour; reaching a border half-edge z means the
        // interior half-edge before it, a, is twin(z)
        b = c;
        a = pv_of(c);
        int32_t z = ld_chain(m.twin + a);
        while (z < HI) {
            const int32_t pz = pv_of(z);
            const int32_t nz = ld_chain(m.twin + pz);
            if (f1_of(w.flags, z, HI)) break;
            a = pz;
            z = nz;
            if (++steps > w.max_rot) { atomicOr(&w.ctrl->error, DEV_ERR_NONTERMINATING); return; }
        }
    }
    m.next[a] = b;
    if (loc.ho < 0) m.prev[b] = a;  // a batch's union prev is never read
    loc.link(w, a, b);
    set_start(w.flags, a);
    set_start(w.flags, b);
}

// over a list of chords (*count of them, at most cap; negative entries are
// skipped): the repair's chords, or the convexification's.  Four threads per
// chord, one per half and direction (the directions in different warps): every
// thread follows one chain of loads.
__global__ void __launch_bounds__(256) k_chord_links(MeshView m, Work w, const int32_t *list, const int32_t *count,
                                                     int32_t cap) {
    chain_next();
    chain_wait();
    const int32_t HI = 3 * m.T;
    int32_t n = *count;
    if (n > cap) n = cap;
    for (int64_t i = blockIdx.x * blockDim.x + threadIdx.x; i < 4 * (int64_t)n; i += gridDim.x * blockDim.x) {
        const bool cw = i < 2 * (int64_t)n;
        const int64_t q = cw ? i : i - 2 * (int64_t)n;
        const int32_t c0 = list[q >> 1];
        if (c0 < 0) continue;
        const int32_t t0 = ld_chain(m.twin + c0);
        relink_around(m, w, q & 1 ? t0 : c0, q & 1 ? c0 : t0, cw, HI);
    }
}

void launch_chord_links(const MeshView &m, const Work &w, cudaStream_t s, bool chained) {
    launch_kernel(k_chord_links, list_blocks(m, w, 2048), 256, 0, s, chained, m, w, w.chords, &w.ctrl->n_tips, w.tip_cap);
}

void launch_chord_links_list(const MeshView &m, const Work &w, const int32_t *list, const int32_t *count,
                             int32_t cap, cudaStream_t s, bool chained) {
    launch_kernel(k_chord_links, list_blocks(m, w, 512), 256, 0, s, chained, m, w, list, count, cap);  // a chord per 10 to 25 triangles
}

}  // namespace polylla
