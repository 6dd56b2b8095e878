// Per-piece images of every selected piece from one march per ray, for
// sm_103a (the paper's per-rank local images, Sec. 4.1-4.2, all ranks' pieces
// on one GPU).
//
// A ray meets every lattice point once, in depth order; the point's unit
// (brick, leaf or tet) names its piece.  The lane keeps the running sums of
// the piece it is in and changes them when the piece changes: the old sums go
// to that piece's image, the new piece's come back from its image (zero at its
// first sample: the images are cleared before the launch).  Sums are stored
// in float32 as they stand in registers, so a piece that a ray leaves and
// enters again goes on exactly where it stopped, and every image equals the
// one its own march (k_pass1_piece, k_pass2_piece) gives, bit for bit.
// Trigonometric moment slabs hold 16-bit quotients, which cannot be taken up
// again: their pass 1 keeps one march per piece.
//
// One march per piece costs K launches, each of which visits every ray tile,
// finds the piece's box and skips the other pieces' units one by one; one
// march for all pieces costs one launch, one walk of the volume and the
// piece changes (16 to 20 bytes out and in per change, mostly L2 hits).  256^3
// grid in 16 pieces, 1024^2 view (193 M samples), passes 1 and 2 with the
// clearing of the images: 2.85 + 3.31 ms as own marches, 0.81 + 1.16 ms as
// one.  What bounds it is issue (72 % of the slots in pass 1, 81 % in pass 2, with
// the windows' shared-memory reads at 67 and 58 % of the L1 pipe), one point at
// a time with the brick of each sample: 103 and 170 warp instructions per
// 32 samples, where the frame's passes take 72 and 56 (two points at a time,
// pass 2 from the sample cache).  The images' traffic does not show: DRAM 2 %,
// 92 % of the L2 reads hit.  Lists of one or two pieces may be better off with
// marches of their own (one_march).
#pragma once
#include "mboit_grid.cuh"
#include "mboit_pieces.h"
#include "mboit_units.cuh"

namespace mb {
namespace {

// Pass-1 sums of the current piece, and its moment slab.
template <int MS>
struct MomentPieces {
    typename Bodies<MS>::Moment b;
    const GridD& g;
    const ViewSlot& S;
    char* base;
    int64_t slab;
    int pix;
    __device__ __forceinline__ void put(int slot) {
        b.store(g, base, S, S.moment_off + slot * slab, pix);   // base is the first view's first slab
    }
    __device__ __forceinline__ void get(int slot) {
        const char* p = base + S.moment_off + slot * slab;
        const float m0 = reinterpret_cast<const float*>(p)[pix];
        const float4 q = reinterpret_cast<const float4*>(p + (size_t)4 * S.plane)[pix];
        if constexpr (MS == 0) {
            b.m0 = m0;
            b.m12 = make_float2(q.x, q.y);
            b.m34 = make_float2(q.z, q.w);
        } else {
            b.m[0] = m0;
            b.m[1] = q.x; b.m[2] = q.y; b.m[3] = q.z; b.m[4] = q.w;
            if constexpr (MS == 6) {
                const float2 r = reinterpret_cast<const float2*>(p + (size_t)20 * S.plane)[pix];
                b.m[5] = r.x; b.m[6] = r.y;
            } else {
                const float4 r = reinterpret_cast<const float4*>(p + (size_t)20 * S.plane)[pix];
                b.m[5] = r.x; b.m[6] = r.y; b.m[7] = r.z; b.m[8] = r.w;
            }
        }
    }
};

// Pass-2 sums of the current piece, and its colour image.
template <int MS>
struct BlendPieces {
    typename Bodies<MS>::Blend b;
    float4* img;      // the view's first image
    int64_t npix;
    int pix;
    __device__ __forceinline__ void put(int slot) { img[slot * npix + pix] = b.C; }
    __device__ __forceinline__ void get(int slot) { b.C = img[slot * npix + pix]; }
};

// The body of the marches: follows the piece of the sample's unit.
template <class Sums>
struct PieceBody {
    Sums s;
    const int32_t* __restrict__ pou;   // piece of unit (-1: none)
    const SlotMap& map;
    int unit = -1, slot = -1;
    // Takes up the sums of unit u's piece; false when the piece is not wanted.
    __device__ __forceinline__ bool enter(int u) {
        if (u != unit) {
            unit = u;
            const int p = __ldg(pou + u);
            const int j = p < 0 ? -1 : map.n ? (int)map.slot[p] : p;
            if (j != slot) {
                leave();
                slot = j;
                if (j >= 0) s.get(j);
            }
        }
        return slot >= 0;
    }
    __device__ __forceinline__ void leave() {
        if (slot >= 0) s.put(slot);
    }
    __device__ __forceinline__ void operator()(float t, float xt, float ws = 1.0f) { s.b(t, xt, ws); }
};

template <class S> struct TakesUnits<PieceBody<S>> : std::true_type {};

// Grid: the marches of the fused passes (windows of the field in shared
// memory, direct loads where the rays spread too far), each point's brick
// looked up.
template <class Cfg, class Body>
__device__ __forceinline__ void march_pieces(const GridD& g, float* __restrict__ win, const float o[3], const float d[3],
                                             int k0, int k1, Body& body) {
    march_fused<Cfg, false, Body>(g, nullptr, win, o, d, k0, k1, body);
}

// Octree: fixed or adaptive step, the leaf kept while the ray stays in it.
template <class Body>
__device__ __forceinline__ void march_pieces(const AmrD& a, const float o[3], const float d[3], int k0, int k1, Body& body) {
    const GridD& g = a.g;
    const bool adaptive = (g.flags & kFlagAdaptiveStep) != 0;
    const int tmask = adaptive ? tag_mask(a.max_level) : 0;
    LeafCache lc;
    for (int k = k0; k <= k1; ++k) {
        const float t = lattice_t(k, g.step);
        const float p[3] = {ffma(t, d[0], o[0]), ffma(t, d[1], o[1]), ffma(t, d[2], o[2])};
        const int u = lc.find<false>(a, nullptr, p);
        if (u < 0 || !body.enter(u)) continue;
        if (!adaptive) {
            body(t, tf_x(g, leaf_value(a, p, u, lc.lo, lc.inv_h)));
        } else if (!(k & ((1 << lc.shift) - 1))) {
            body(t, tag_shift(tf_x(g, leaf_value(a, p, u, lc.lo, lc.inv_h)), lc.shift, tmask), (float)(1 << lc.shift));
        }
    }
}

// Mesh: the walk of the fused passes.
template <bool kNarrow, class Body>
__device__ __forceinline__ void march_pieces(const TetT<kNarrow>& m, const float o[3], const float d[3], int k0, int k1,
                                             Body& body) {
    march_unit<false>(m, nullptr, o, d, k0, k1, body);
}

template <class V> struct PieceMinBlocks { static constexpr int value = 3; };
template <> struct PieceMinBlocks<AmrD> { static constexpr int value = 4; };

template <class V, class Cfg, int MS>
__global__ void __launch_bounds__(256, MS == 0 ? PieceMinBlocks<V>::value : 2)
    k_pass1_pieces(const __grid_constant__ V vol, const float4* __restrict__ tf, const int32_t* __restrict__ pou,
                   const __grid_constant__ ViewTable vt, const __grid_constant__ SlotMap map, int n_slots,
                   char* moments, Counters* __restrict__ ctr) {
    if (tables_bad(vol)) return;
    constexpr bool kGrid = std::is_same<V, GridD>::value;
    const GridD& g = common(vol);
    __shared__ float2 s_sig[256];
    __shared__ __align__(16) float s_win[kGrid ? kFusedWarps : 1][kGrid ? Cfg::Floats : 4];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) {
        const float s0 = tf[i].w;
        s_sig[i] = make_float2(s0, i < 255 ? tf[i + 1].w - s0 : 0.0f);
    }
    __syncthreads();
    int vi, px, py, tile;
    while (next_tile<MS == 0>(vt, &ctr->tile_next[0], vi, px, py, tile)) {
        const ViewSlot& S = vt.s[vi];
        const bool valid = px < S.v.width && py < S.v.height;
        float o[3], d[3];
        int k0, k1;
        ray_range(g, S.v, valid, px, py, o, d, k0, k1);
        PieceBody<MomentPieces<MS>> body{{make_moment_body<MS>(s_sig, g, S.v), g, S,
                                          moments + S.moment_off * (n_slots - 1), slab_bytes(g, S.plane),
                                          valid ? py * S.v.width + px : 0},
                                         pou, map};
        if constexpr (kGrid)
            march_pieces<Cfg>(vol, s_win[threadIdx.x >> 5], o, d, k0, k1, body);
        else
            march_pieces(vol, o, d, k0, k1, body);
        body.leave();
        warp_add_u64(&ctr->samples[0], body.s.b.n);
    }
}

template <class V, class Cfg, int MS>
__global__ void __launch_bounds__(256, MS == 0 ? PieceMinBlocks<V>::value : 2)
    k_pass2_pieces(const __grid_constant__ V vol, const float4* __restrict__ tf, const int32_t* __restrict__ pou,
                   const __grid_constant__ ViewTable vt, const __grid_constant__ SlotMap map, int n_slots,
                   const char* __restrict__ moments, float* color, Counters* __restrict__ ctr) {
    if (tables_bad(vol)) return;
    constexpr bool kGrid = std::is_same<V, GridD>::value;
    const GridD& g = common(vol);
    __shared__ float4 s_tf[512];
    __shared__ __align__(16) float s_win[kGrid ? kFusedWarps : 1][kGrid ? Cfg::Floats : 4];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) {
        const float4 e0 = tf[i], e1 = i < 255 ? tf[i + 1] : tf[i];
        s_tf[2 * i] = e0;
        s_tf[2 * i + 1] = make_float4(e1.x - e0.x, e1.y - e0.y, e1.z - e0.z, e1.w - e0.w);
    }
    __syncthreads();
    int vi, px, py, tile;
    while (next_tile<MS == 0>(vt, &ctr->tile_next[1], vi, px, py, tile)) {
        const ViewSlot& S = vt.s[vi];
        const bool valid = px < S.v.width && py < S.v.height;
        const int pix = valid ? py * S.v.width + px : 0;
        float o[3], d[3];
        int k0, k1;
        ray_range(g, S.v, valid, px, py, o, d, k0, k1);
        PieceBody<BlendPieces<MS>> body{{make_blend_body<MS>(s_tf, g, S, moments, S.moment_off, pix, valid),
                                         reinterpret_cast<float4*>(color + S.color_off * n_slots),
                                         (int64_t)S.v.width * S.v.height, pix},
                                        pou, map};
        if constexpr (kGrid)
            march_pieces<Cfg>(vol, s_win[threadIdx.x >> 5], o, d, k0, k1, body);
        else
            march_pieces(vol, o, d, k0, k1, body);
        body.leave();
        warp_add_u64(&ctr->samples[1], body.s.b.n);
    }
}

}  // namespace
}  // namespace mb
