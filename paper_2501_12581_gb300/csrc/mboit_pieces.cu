// One-march per-piece passes: kernel selection and launchers (the kernels and
// their design are in mboit_pieces.cuh).
#include "mboit_pieces.cuh"

namespace mb {

// The kernels of the other moment sets (mboit_pieces_sets.cu).
const void* pieces_set_fn(int vkind, int pass, int ms);

namespace {

int moment_variant(const GridD& g) { return g.trig.sel; }
int moment_variant(const AmrD& a) { return a.g.trig.sel; }
int moment_variant(const TetD& m) { return m.g.trig.sel; }

// vec: configuration 3's window (grids with 16-byte rows), else configuration 0's.
template <class V>
const void* pieces_fn(int vkind, int pass, int ms, bool vec) {
    if (ms != 0) return pieces_set_fn(vkind, pass, ms);
    if constexpr (std::is_same<V, GridD>::value)
        if (vec)
            return pass == 1 ? (const void*)k_pass1_pieces<V, Stage3, 0> : (const void*)k_pass2_pieces<V, Stage3, 0>;
    return pass == 1 ? (const void*)k_pass1_pieces<V, Stage0, 0> : (const void*)k_pass2_pieces<V, Stage0, 0>;
}

template <class V>
cudaError_t launch1(int vkind, const V& vol, bool vec, const float4* tf, const int32_t* pou, const ViewTable& vt,
                    const SlotMap& map, int32_t n_slots, void* moments, Counters* ctr, cudaStream_t s) {
    const int ms = moment_variant(vol);
    const ViewSlot& last = vt.s[vt.n - 1];
    const int64_t bytes = last.moment_off + (int64_t)(4 + 4 * (ms ? ms : 4)) * last.plane;
    cudaError_t e = cudaMemsetAsync(moments, 0, (size_t)(bytes * n_slots), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(&ctr->tile_next[0], 0, sizeof(int32_t), s);
    if (e != cudaSuccess) return e;
    const void* fn = pieces_fn<V>(vkind, 1, ms, vec);
    char* m = static_cast<char*>(moments);
    int ns = n_slots;
    void* args[] = {(void*)&vol, (void*)&tf, (void*)&pou, (void*)&vt, (void*)&map, (void*)&ns, (void*)&m, (void*)&ctr};
    return cudaLaunchKernel(fn, dim3(persistent_blocks(fn, 256, 0)), dim3(256), args, 0, s);
}

template <class V>
cudaError_t launch2(int vkind, const V& vol, bool vec, const float4* tf, const int32_t* pou, const ViewTable& vt,
                    const SlotMap& map, int32_t n_slots, const void* moments, float* color, Counters* ctr,
                    cudaStream_t s) {
    const ViewSlot& last = vt.s[vt.n - 1];
    const int64_t floats = last.color_off + (int64_t)4 * last.v.width * last.v.height;
    cudaError_t e = cudaMemsetAsync(color, 0, (size_t)(floats * n_slots) * sizeof(float), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(&ctr->tile_next[1], 0, sizeof(int32_t), s);
    if (e != cudaSuccess) return e;
    const void* fn = pieces_fn<V>(vkind, 2, moment_variant(vol), vec);
    const char* m = static_cast<const char*>(moments);
    int ns = n_slots;
    void* args[] = {(void*)&vol, (void*)&tf, (void*)&pou, (void*)&vt, (void*)&map, (void*)&ns, (void*)&m, (void*)&color,
                    (void*)&ctr};
    return cudaLaunchKernel(fn, dim3(persistent_blocks(fn, 256, 0)), dim3(256), args, 0, s);
}

template <bool kN>
TetT<kN> as_tet(const TetD& m) {
    TetT<kN> t;
    static_cast<TetD&>(t) = m;
    return t;
}

}  // namespace

cudaError_t prepare_piece_kernels() {
    for (int ms : {0, 3, 4, 6, 8})
        for (int pass = 1; pass <= 2; ++pass) {
            if (pass == 1 && (ms == 3 || ms == 4)) continue;
            const void* fns[] = {pieces_fn<GridD>(0, pass, ms, false), pieces_fn<GridD>(0, pass, ms, true),
                                 pieces_fn<AmrD>(1, pass, ms, false), pieces_fn<TetT<true>>(2, pass, ms, false),
                                 pieces_fn<TetT<false>>(3, pass, ms, false)};
            for (const void* f : fns) {
                cudaFuncAttributes a;
                const cudaError_t e = cudaFuncGetAttributes(&a, f);
                if (e != cudaSuccess) return e;
                persistent_blocks(f, 256, 0);
            }
        }
    return cudaSuccess;
}

cudaError_t launch_pass1_pieces(const GridD& g, const float4* tf, const int32_t* pou, const ViewTable& vt,
                                const SlotMap& map, int32_t n_slots, void* moments, Counters* ctr, cudaStream_t s) {
    return launch1(0, g, stage_config_eligible(g, 3), tf, pou, vt, map, n_slots, moments, ctr, s);
}

cudaError_t launch_pass1_pieces(const AmrD& a, const float4* tf, const int32_t* pou, const ViewTable& vt,
                                const SlotMap& map, int32_t n_slots, void* moments, Counters* ctr, cudaStream_t s) {
    return launch1(1, a, false, tf, pou, vt, map, n_slots, moments, ctr, s);
}

cudaError_t launch_pass1_pieces(const TetD& m, const float4* tf, const int32_t* pou, const ViewTable& vt,
                                const SlotMap& map, int32_t n_slots, void* moments, Counters* ctr, cudaStream_t s) {
    return m.narrow ? launch1(2, as_tet<true>(m), false, tf, pou, vt, map, n_slots, moments, ctr, s)
                    : launch1(3, as_tet<false>(m), false, tf, pou, vt, map, n_slots, moments, ctr, s);
}

cudaError_t launch_pass2_pieces(const GridD& g, const float4* tf, const int32_t* pou, const ViewTable& vt,
                                const SlotMap& map, int32_t n_slots, const void* moments, float* color, Counters* ctr,
                                cudaStream_t s) {
    return launch2(0, g, stage_config_eligible(g, 3), tf, pou, vt, map, n_slots, moments, color, ctr, s);
}

cudaError_t launch_pass2_pieces(const AmrD& a, const float4* tf, const int32_t* pou, const ViewTable& vt,
                                const SlotMap& map, int32_t n_slots, const void* moments, float* color, Counters* ctr,
                                cudaStream_t s) {
    return launch2(1, a, false, tf, pou, vt, map, n_slots, moments, color, ctr, s);
}

cudaError_t launch_pass2_pieces(const TetD& m, const float4* tf, const int32_t* pou, const ViewTable& vt,
                                const SlotMap& map, int32_t n_slots, const void* moments, float* color, Counters* ctr,
                                cudaStream_t s) {
    return m.narrow ? launch2(2, as_tet<true>(m), false, tf, pou, vt, map, n_slots, moments, color, ctr, s)
                    : launch2(3, as_tet<false>(m), false, tf, pou, vt, map, n_slots, moments, color, ctr, s);
}

}  // namespace mb
