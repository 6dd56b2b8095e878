// The one-march per-piece kernels of the moment sets other than four power
// moments (templates in mboit_pieces.cuh), compiled in parallel with the rest.
#include "mboit_pieces.cuh"

namespace mb {
namespace {

template <class V>
const void* pieces_fn(int pass, int ms) {
    if (pass == 1) return ms == 6 ? (const void*)k_pass1_pieces<V, Stage0, 6> : (const void*)k_pass1_pieces<V, Stage0, 8>;
    switch (ms) {
        case 3: return (const void*)k_pass2_pieces<V, Stage0, 3>;
        case 4: return (const void*)k_pass2_pieces<V, Stage0, 4>;
        case 6: return (const void*)k_pass2_pieces<V, Stage0, 6>;
        default: return (const void*)k_pass2_pieces<V, Stage0, 8>;
    }
}

}  // namespace

// vkind: 0 grid, 1 octree, 2 narrow mesh, 3 wide mesh; pass 1 (6 / 8 power moments) or 2.
const void* pieces_set_fn(int vkind, int pass, int ms) {
    switch (vkind) {
        case 0: return pieces_fn<GridD>(pass, ms);
        case 1: return pieces_fn<AmrD>(pass, ms);
        case 2: return pieces_fn<TetT<true>>(pass, ms);
        default: return pieces_fn<TetT<false>>(pass, ms);
    }
}

}  // namespace mb
