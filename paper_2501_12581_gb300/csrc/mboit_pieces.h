// One march for the per-piece images of every selected piece: the launches'
// parameters (kernels in mboit_pieces.cuh).
#pragma once
#include "mboit_internal.h"

namespace mb {

// Image slot of each piece (-1: not wanted); n = 0: slot = piece.
constexpr int kMaxSlotPieces = 256;
struct SlotMap {
    int32_t n;
    int16_t slot[kMaxSlotPieces];
};

// Clears the images and marches every ray once.  The slabs / images are laid
// out as by the one-piece launches.  Trigonometric sets have no such pass 1.
cudaError_t launch_pass1_pieces(const GridD& g, const float4* tf, const int32_t* pou, const ViewTable& vt,
                                const SlotMap& map, int32_t n_slots, void* moments, Counters* ctr, cudaStream_t s);
cudaError_t launch_pass1_pieces(const AmrD& a, const float4* tf, const int32_t* pou, const ViewTable& vt,
                                const SlotMap& map, int32_t n_slots, void* moments, Counters* ctr, cudaStream_t s);
cudaError_t launch_pass1_pieces(const TetD& m, const float4* tf, const int32_t* pou, const ViewTable& vt,
                                const SlotMap& map, int32_t n_slots, void* moments, Counters* ctr, cudaStream_t s);
cudaError_t launch_pass2_pieces(const GridD& g, const float4* tf, const int32_t* pou, const ViewTable& vt,
                                const SlotMap& map, int32_t n_slots, const void* moments, float* color, Counters* ctr,
                                cudaStream_t s);
cudaError_t launch_pass2_pieces(const AmrD& a, const float4* tf, const int32_t* pou, const ViewTable& vt,
                                const SlotMap& map, int32_t n_slots, const void* moments, float* color, Counters* ctr,
                                cudaStream_t s);
cudaError_t launch_pass2_pieces(const TetD& m, const float4* tf, const int32_t* pou, const ViewTable& vt,
                                const SlotMap& map, int32_t n_slots, const void* moments, float* color, Counters* ctr,
                                cudaStream_t s);
cudaError_t prepare_piece_kernels();

}  // namespace mb
