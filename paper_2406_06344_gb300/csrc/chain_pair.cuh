// The factor chain on pairs of SMs (chain_pair.cu): the default tensor-core kernel of the kind::f16
// forms with d >= 2, where the ranks fit it.
#pragma once

#include "pttk_internal.cuh"

namespace pttk {

// Per-handle core images of one form.
struct PairImages {
  uint8_t* buf = nullptr;
  size_t off[2][2] = {};
  float in_scale[2][2] = {}, out_scale[2][2] = {};
};

bool pair_form(const pttk_tt* tt, pttk_prec prec);
// Lays out the images (synchronises).
pttk_status pair_prepare(const pttk_tt* tt, pttk_prec prec, PairImages& im, cudaStream_t s);
pttk_status pair_build(const pttk_tt* tt, pttk_prec prec, const PairImages& im, const float* X, int64_t N_s,
                       const float* Y, int64_t N_t, float* U, float* V, int* d_status, cudaStream_t s);

}  // namespace pttk
