// Angular sweeps (sweeps_angular.cu).  Each call launches one kernel on `st`;
// the arrays are those of the workspace, S rows of (l_max + 1)^2 - 1
// components per channel.
#pragma once
#include <cuda_runtime.h>

#include "gnep_internal.h"

namespace gnep {

// Atoms of one block of the angular sweeps (four warps, a group of atoms each).
int ang_block_atoms(const Shape& s);
// Blocks of the c-gradient sweep per SM: what its registers are bounded for, and its grid.
constexpr int ang_cgrad_per_sm(int lmax) { return lmax > 4 ? 3 : 4; }

template <class C>
int ang_setup();
// sweep 1: S_nlm and the angular descriptor columns of G
template <class C>
int ang_descriptors(const gnep_model* m, const gnep_nlist* nl, cudaStream_t st, float* S, float* G);
// sweep 3: Sdot, the angular columns of Gdot and the tangent directions w_ij
template <class C>
int ang_tangent(const gnep_model* m, const gnep_nlist* nl, cudaStream_t st, const float4* a, const float* Bs,
                const float* S, float* Sd, float* Gd, float4* wij);
// sweep 2: the angular pair forces dE_i/dr_ij into dA
template <class C>
int ang_force(const gnep_model* m, const gnep_nlist* nl, cudaStream_t st, const float* S, const float* Ep,
              float4* dA);
// sweep 4: the angular part of dL/dc into cpart[block][c^R + c^A] for nb blocks
template <class C>
int ang_cgrad(const gnep_model* m, const gnep_nlist* nl, cudaStream_t st, int nb, const float4* wij, const float* S,
              const float* Sd, const float* Gb, const float* Ep, float* cpart);

}  // namespace gnep
