// Shape-specialised sweeps of one training step over a packed batch.
//
//   sweep 1  descriptors  q_n (Eqs. 5-6), S_nlm and q_nl (Eqs. 7-8), 4-body q4_n
//   network  (network.cu) E_i, E'_i, per-atom radial contraction chat_i
//   sweep 2  dE_i/dr_ij (C3.6), forces (Eq. 3), per-atom virial (Eq. 4)
//   sweep 3  tangent  Gdot_i = sum_j dG_i/dr_ij . u_ij
//   network  (network.cu) tangent and reverse pass, adjoints Gbar_i
//   sweep 4  dL/dc^R and dL/dc^A
//
// Gradient route.  With a_i = dL/dF_i and B_s = dL/dW_s held fixed (Eqs. 11-12),
//   sum_i a_i.F_i + sum_s B_s:W_s = - sum_i sum_j u_ij . dE_i/dr_ij,
//   u_ij = (a_j - a_i) + B_s r_ij,
// because F_i = sum_j (dE_i/dr_ij - dE_j/dr_ji) (Eq. 3) and W_s = -sum r_ij (x) dE_i/dr_ij
// (Eq. 4 summed).  Hence the force and virial parts of dL/dtheta (Eqs. 15-16 with
// the mixed derivatives of App. C3 and D1.11-D1.17) equal -d/dtheta sum_i E'_i.Gdot_i:
// one forward-mode sweep (3) and one reverse sweep (4) instead of explicit second
// derivative tensors.
//
// Thread mappings.  Radial sweeps: RL consecutive lanes per atom, each taking
// every RL-th pair, combined by warp shuffles; RL is 4 for batches that give
// every SM several blocks, 8 or 16 for smaller ones, where the per-lane pair
// loop (one dependent global load per pair) sets the kernel's length.
// Angular sweeps: sweeps_angular.cu.  No float atomics anywhere: fixed
// summation order.
#include <cstdio>
#include <mutex>
#include <string>

#include "device_math.cuh"
#include "gnep_internal.h"
#include "network.cuh"
#include "shape.cuh"
#include "sweeps_angular.cuh"

namespace gnep {

namespace {

template <int NS, int K>
__device__ __forceinline__ void acc_row(float (&acc)[NS][K], int J, const float (&v)[K], float w) {
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    const float ws = (s == J) ? w : 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) acc[s][k] = fmaf(ws, v[k], acc[s][k]);
  }
}

template <int NS, int K>
__device__ __forceinline__ float dot_row(const float (&c)[NS][K], int J, const float (&v)[K]) {
  float r = 0.f;
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) t = fmaf(c[s][k], v[k], t);
    r = (s == J) ? t : r;
  }
  return r;
}

__device__ __forceinline__ float3 sym_apply(const float* b, float3 r) {  // b = xx yy zz xy yz zx
  return make_float3(b[0] * r.x + b[3] * r.y + b[5] * r.z, b[3] * r.x + b[1] * r.y + b[4] * r.z,
                     b[5] * r.x + b[4] * r.y + b[2] * r.z);
}

template <int RL, int NS, int K>
__device__ __forceinline__ void lane_reduce(float (&acc)[NS][K]) {
#pragma unroll
  for (int o = 1; o < RL; o <<= 1)
#pragma unroll
    for (int s = 0; s < NS; ++s)
#pragma unroll
      for (int k = 0; k < K; ++k) acc[s][k] += __shfl_xor_sync(0xffffffffu, acc[s][k], o);
}

}  // namespace

// ------------------------------------------------------------- sweep 1

// Radial descriptors: per-atom basis sums FR[J][k] = sum_{j in J} f_k(r_ij) and
// q_n = sum_J sum_k c^R_nk^{IJ} FR[J][k]  (Eqs. 5-6).
template <class C, int RL>
__global__ void __launch_bounds__(128) k_desc_radial(int N, DevModel dm, const int* __restrict__ type,
                                                     const int* __restrict__ off, const float4* __restrict__ rij,
                                                     float* __restrict__ FR, float* __restrict__ G) {
  GNEP_PDL_START();
  __shared__ float cR[C::NCR];
  for (int q = threadIdx.x; q < C::NCR; q += blockDim.x) cR[q] = dm.params[dm.off_cR + q];
  __syncthreads();
  const int gt = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = gt / RL, lane = gt % RL;
  const bool ok = i < N;
  float acc[C::NS][C::KR];
#pragma unroll
  for (int s = 0; s < C::NS; ++s)
#pragma unroll
    for (int k = 0; k < C::KR; ++k) acc[s][k] = 0.f;
  if (ok) {
    const int p1 = off[i + 1];
    int p = off[i] + lane;
    float4 rn = p < p1 ? rij[p] : make_float4(1.f, 0.f, 0.f, 0.f);  // the pair after the current one
    for (; p < p1; p += RL) {
      const float4 r = rn;
      if (p + RL < p1) rn = rij[p + RL];
      const float rr = sqrtf(r.x * r.x + r.y * r.y + r.z * r.z);
      float f[C::KR];
      radial_basis<C::KR>(rr, dm.rcr_inv, f);
      acc_row<C::NS, C::KR>(acc, (int)r.w, f, 1.f);
    }
  }
  lane_reduce<RL>(acc);
  if (!ok) return;
  const int I = type[i];
  float* fr = FR + (size_t)i * C::NS * C::KR;
#pragma unroll
  for (int s = 0; s < C::NS; ++s)
#pragma unroll
    for (int k = 0; k < C::KR; ++k)
      if ((s * C::KR + k) % RL == lane) fr[s * C::KR + k] = acc[s][k];
#pragma unroll
  for (int n = 0; n < C::NQR; ++n) {
    if (n % RL != lane) continue;
    float q = 0.f;
#pragma unroll
    for (int s = 0; s < C::NS; ++s)
#pragma unroll
      for (int k = 0; k < C::KR; ++k) q = fmaf(cR[((I * C::NS + s) * C::NQR + n) * C::KR + k], acc[s][k], q);
    G[(size_t)i * C::NDES + n] = q;
  }
}

// ------------------------------------------------------------- sweep 2

// Forces and per-atom virials, RL lanes per atom.
//   radial pairs: d_ij - d_ji = (chat_i[J] . f'(r) + chat_j[I] . f'(r)) r_ij / r
//                 (C1.1, C3.6 with the per-atom contraction chat = sum_n E'_n c^R_n)
//   angular pairs: d_ij - d_rev(ij) from the pair forces of the angular force sweep (Eq. 3)
//   virial: -sum_j r_ij (x) d_ij, symmetrised (Eq. 4 summed over atoms).
// With `early` (the angular force sweep is the previous kernel) the radial pairs,
// which read the lists and the network's chat, run beside that sweep, ahead of
// the wait for its pair forces.
template <class C, int RL>
__global__ void __launch_bounds__(128) k_force_atoms(int N, DevModel dm, const int* __restrict__ type,
                                                     const int* __restrict__ offR, const int* __restrict__ jR,
                                                     const float4* __restrict__ rijR, const float* __restrict__ chat,
                                                     const int* __restrict__ offA, const int* __restrict__ revA,
                                                     const float4* __restrict__ rijA, const float4* __restrict__ dA,
                                                     float* __restrict__ F, float* __restrict__ Wat, bool early) {
  if (!early) GNEP_PDL_START();
  const int gt = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = gt / RL, lane = gt % RL;
  const bool ok = i < N;
  float v[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // F (3), W (6)
  if (ok) {
    const int I = type[i];
    float ci[C::NS][C::KR];
#pragma unroll
    for (int s = 0; s < C::NS; ++s)
#pragma unroll
      for (int k = 0; k < C::KR; ++k) ci[s][k] = chat[((size_t)i * C::NS + s) * C::KR + k];
    const int p1 = offR[i + 1];
    int p = offR[i] + lane;
    float4 rn = p < p1 ? rijR[p] : make_float4(1.f, 0.f, 0.f, 0.f);  // the pair after the current one
    int jn = p < p1 ? jR[p] : 0;
    for (; p < p1; p += RL) {
      const float4 r = rn;
      const int j = jn;
      if (p + RL < p1) {
        rn = rijR[p + RL];
        jn = jR[p + RL];
      }
      const float* cj = chat + ((size_t)j * C::NS + I) * C::KR;
      const float rr = sqrtf(r.x * r.x + r.y * r.y + r.z * r.z);
      float f[C::KR], fp[C::KR];
      radial_basis_d<C::KR>(rr, dm.rcr_inv, f, fp);
      const float dij = dot_row<C::NS, C::KR>(ci, (int)r.w, fp);
      float dji = 0.f;
#pragma unroll
      for (int k = 0; k < C::KR; ++k) dji = fmaf(cj[k], fp[k], dji);
      const float s1 = (dij + dji) / rr, s0 = dij / rr;
      v[0] += s1 * r.x;
      v[1] += s1 * r.y;
      v[2] += s1 * r.z;
      v[3] -= s0 * r.x * r.x;
      v[4] -= s0 * r.y * r.y;
      v[5] -= s0 * r.z * r.z;
      v[6] -= s0 * r.x * r.y;
      v[7] -= s0 * r.y * r.z;
      v[8] -= s0 * r.z * r.x;
    }
    if (early) GNEP_PDL_START();
    const int q1 = offA[i + 1];
    for (int p = offA[i] + lane; p < q1; p += RL) {
      const float4 d = dA[p], b = dA[revA[p]], r = rijA[p];
      v[0] += d.x - b.x;
      v[1] += d.y - b.y;
      v[2] += d.z - b.z;
      v[3] -= r.x * d.x;
      v[4] -= r.y * d.y;
      v[5] -= r.z * d.z;
      v[6] -= 0.5f * (r.x * d.y + r.y * d.x);
      v[7] -= 0.5f * (r.y * d.z + r.z * d.y);
      v[8] -= 0.5f * (r.z * d.x + r.x * d.z);
    }
  } else if (early) {
    GNEP_PDL_START();
  }
#pragma unroll
  for (int o = 1; o < RL; o <<= 1)
#pragma unroll
    for (int q = 0; q < 9; ++q) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
  if (!ok || lane != 0) return;
  F[3 * (size_t)i] = v[0];
  F[3 * (size_t)i + 1] = v[1];
  F[3 * (size_t)i + 2] = v[2];
#pragma unroll
  for (int q = 0; q < 6; ++q) Wat[6 * (size_t)i + q] = v[3 + q];
}

// E_s = sum_i E_i and W_s = sum_i w_i, one block per structure (Eqs. 1, 4): each
// thread sums its few atoms in FP32 (128 threads, 1,024 where the structures
// average above 512 atoms), the warps combine their lanes as FP32 pairs without
// rounding (F2) and the warp sums are added in FP64 in order.  It also leaves the
// results in the caller's device buffers (NULL: not wanted), instead of a copy for
// each.
template <int T>
__global__ void __launch_bounds__(T) k_struct_sum(const int* __restrict__ soff, const float* __restrict__ Eatom,
                                                  const float* __restrict__ Wat, const float* __restrict__ F,
                                                  double* __restrict__ Es, double* __restrict__ Ws,
                                                  float* __restrict__ oE, float* __restrict__ oF,
                                                  double* __restrict__ oEs, double* __restrict__ oWs) {
  GNEP_PDL_START();
  const int s = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int a0 = soff[s], a1 = soff[s + 1];
  float acc[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  for (int i = a0 + threadIdx.x; i < a1; i += T) {
    const float e = Eatom[i];
    if (oE) oE[i] = e;
    acc[0] += e;
#pragma unroll
    for (int q = 0; q < 6; ++q) acc[1 + q] += Wat[6 * (size_t)i + q];
  }
  if (oF)
    for (int q = 3 * a0 + threadIdx.x; q < 3 * a1; q += T) oF[q] = F[q];
  __shared__ float2 wsum[T / 32][7];
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    const F2 v = f2_warp_sum(F2{acc[q], 0.f});
    if (lane == 0) wsum[warp][q] = make_float2(v.hi, v.lo);
  }
  __syncthreads();
  if (threadIdx.x >= 7) return;
  double v = 0.0;
#pragma unroll
  for (int w = 0; w < T / 32; ++w) v += (double)wsum[w][threadIdx.x].x + (double)wsum[w][threadIdx.x].y;
  const int q = 6 * s + threadIdx.x - 1;
  if (threadIdx.x == 0) {
    Es[s] = v;
    if (oEs) oEs[s] = v;
  } else {
    Ws[q] = v;
    if (oWs) oWs[q] = v;
  }
}

// ------------------------------------------------------------- sweep 3

// Radial tangent: FRd[J][k] = sum_{j in J} f_k'(r_ij) (u_hat . u_ij),
// qdot_n = sum_J sum_k c^R_nk^{IJ} FRd[J][k].
template <class C, int RL>
__global__ void __launch_bounds__(128) k_tangent_radial(int N, DevModel dm, const int* __restrict__ type,
                                                        const int* __restrict__ atom_struct, const int* __restrict__ off,
                                                        const int* __restrict__ jj, const float4* __restrict__ rij,
                                                        const float4* __restrict__ a, const float* __restrict__ Bs,
                                                        float* __restrict__ FRd, float* __restrict__ Gd) {
  __shared__ float cR[C::NCR];
  for (int q = threadIdx.x; q < C::NCR; q += blockDim.x) cR[q] = dm.params[dm.off_cR + q];
  GNEP_PDL_START();
  __syncthreads();
  const int gt = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = gt / RL, lane = gt % RL;
  const bool ok = i < N;
  float acc[C::NS][C::KR];
#pragma unroll
  for (int s = 0; s < C::NS; ++s)
#pragma unroll
    for (int k = 0; k < C::KR; ++k) acc[s][k] = 0.f;
  if (ok) {
    const float4 ai = a[i];
    float b[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) b[q] = Bs[6 * atom_struct[i] + q];
    const int p1 = off[i + 1];
    int p = off[i] + lane;
    // the pair after the current one, and its neighbour's tangent
    float4 rn = p < p1 ? rij[p] : make_float4(1.f, 0.f, 0.f, 0.f);
    float4 an = p < p1 ? a[jj[p]] : ai;
    for (; p < p1; p += RL) {
      const float4 r = rn, aj = an;
      if (p + RL < p1) {
        rn = rij[p + RL];
        an = a[jj[p + RL]];
      }
      const float3 br = sym_apply(b, make_float3(r.x, r.y, r.z));
      const float ux = aj.x - ai.x + br.x, uy = aj.y - ai.y + br.y, uz = aj.z - ai.z + br.z;
      const float rr = sqrtf(r.x * r.x + r.y * r.y + r.z * r.z);
      const float ru = (r.x * ux + r.y * uy + r.z * uz) / rr;
      float f[C::KR], fp[C::KR];
      radial_basis_d<C::KR>(rr, dm.rcr_inv, f, fp);
      acc_row<C::NS, C::KR>(acc, (int)r.w, fp, ru);
    }
  }
  lane_reduce<RL>(acc);
  if (!ok) return;
  float* fr = FRd + (size_t)i * C::NS * C::KR;
#pragma unroll
  for (int s = 0; s < C::NS; ++s)
#pragma unroll
    for (int k = 0; k < C::KR; ++k)
      if ((s * C::KR + k) % RL == lane) fr[s * C::KR + k] = acc[s][k];
  const int I = type[i];
#pragma unroll
  for (int n = 0; n < C::NQR; ++n) {
    if (n % RL != lane) continue;
    float q = 0.f;
#pragma unroll
    for (int s = 0; s < C::NS; ++s)
#pragma unroll
      for (int k = 0; k < C::KR; ++k) q = fmaf(cR[((I * C::NS + s) * C::NQR + n) * C::KR + k], acc[s][k], q);
    Gd[(size_t)i * C::NDES + n] = q;
  }
}

// ------------------------------------------------------------- sweep 4

// dL/dc^R: each atom contributes dL/dc^R_nk^{IJ} += Gbar_n FR[J][k] - E'_n FRd[J][k]
// (the angular part is sweeps_angular.cu's).
// Radial part: one block per contiguous range of atoms, lane = column (J, k),
// warp r takes the range's atoms r, r + 16, ... (four per iteration, loads
// first); the block folds its warps in order and writes cpart[block][c^R].
// It is a few dependent rounds of loads, so what counts is warps and loads in
// flight: an atom's Gbar_n and E'_n come in one load, a lane each, and are
// passed round by shuffles (18 loads and registers an atom otherwise, which held
// the SM to one block), 64 registers let two blocks share an SM, and the grid
// is the two blocks per SM that fit (55,200 atoms: 19.7 -> 11.2 us;
// 92 registers and 608 blocks, one per SM at a time, before).
constexpr int kCgRadialWarps = 16;

// acc[I][n] += Gbar_n FR - E'_n FRd, with Gbar_n and E'_n in lanes n and 16 + n of
// x; I is the same for the whole warp.  The statement without instructions keeps
// the branches apart: merged, they would index acc by I, in local memory.
template <int S, int NS, int NQ>
__device__ __forceinline__ void add_channels(float (&acc)[NS][NQ], int I, float x, float fr, float frd) {
  if constexpr (S < NS) {
    if (I == S) {
      asm volatile("// species %0" ::"n"(S));
#pragma unroll
      for (int n = 0; n < NQ; ++n)
        acc[S][n] += __shfl_sync(0xffffffffu, x, n) * fr - __shfl_sync(0xffffffffu, x, 16 + n) * frd;
    } else {
      add_channels<S + 1>(acc, I, x, fr, frd);
    }
  }
}

template <class C>
__global__ void __launch_bounds__(32 * kCgRadialWarps, 2) k_cgrad_radial(int N, const int* __restrict__ type,
                                                                       const float* __restrict__ Gb,
                                                                       const float* __restrict__ Ep,
                                                                       const float* __restrict__ FR,
                                                                       const float* __restrict__ FRd,
                                                                       float* __restrict__ cpart) {
  GNEP_PDL_START();
  constexpr int NCOL = C::NS * C::KR, NW = kCgRadialWarps, U = 4;
  static_assert(NCOL <= 32 && C::NQR <= 16, "one lane per radial column, half a warp per set of channels");
  __shared__ float red[NW][C::NS][C::NQR][32];
  const int lane = threadIdx.x & 31, r = threadIdx.x >> 5;
  const int per = (N + gridDim.x - 1) / gridDim.x;
  const int lo = min(N, (int)blockIdx.x * per), hi = min(N, lo + per);
  const float* src = lane < 16 ? Gb : Ep;  // lanes n and 16 + n hold Gbar_n and E'_n
  const int ch = lane & 15;
  float acc[C::NS][C::NQR];
#pragma unroll
  for (int s = 0; s < C::NS; ++s)
#pragma unroll
    for (int n = 0; n < C::NQR; ++n) acc[s][n] = 0.f;
  for (int i = lo + r; i < hi; i += U * NW) {
    int I[U];
    float fr[U], frd[U], x[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int iu = i + u * NW;
      const bool ok = iu < hi;
      I[u] = ok ? type[iu] : -1;
      x[u] = ok && ch < C::NQR ? src[(size_t)iu * C::NDES + ch] : 0.f;
      fr[u] = ok && lane < NCOL ? FR[(size_t)iu * NCOL + lane] : 0.f;
      frd[u] = ok && lane < NCOL ? FRd[(size_t)iu * NCOL + lane] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) add_channels<0>(acc, I[u], x[u], fr[u], frd[u]);
  }
#pragma unroll
  for (int s = 0; s < C::NS; ++s)
#pragma unroll
    for (int n = 0; n < C::NQR; ++n) red[r][s][n][lane] = acc[s][n];
  __syncthreads();
  for (int q = threadIdx.x; q < C::NCR; q += blockDim.x) {
    const int k = q % C::KR, n = (q / C::KR) % C::NQR, J = (q / (C::KR * C::NQR)) % C::NS,
              I = q / (C::KR * C::NQR * C::NS);
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) v += red[w][I][n][J * C::KR + k];
    cpart[(size_t)blockIdx.x * (C::NCR + C::NCA) + q] = v;
  }
}

// ------------------------------------------------------------- launchers

// Launch CALL (which names RL) with RL = the radial sweeps' lanes per atom.
// The radial sweep of a phase beside its angular sweep: the radial kernel goes
// to the list's second stream, which first waits for the caller's stream (fork)
// and which the caller's stream waits for before the phase's consumer (join).
// The two kernels write disjoint columns of G, Gdot and the c-gradient
// partials.  Per-stage timing keeps them in turn.  *rs is the radial stream.
static int radial_fork(gnep_nlist* nl, cudaStream_t st, cudaStream_t* rs) {
  *rs = st;
  if (g_prof.on || !nl->side || !radial_beside(nl)) return GNEP_OK;
  GNEP_CUDA(cudaEventRecord(nl->fork_ev, st));
  GNEP_CUDA(cudaStreamWaitEvent(nl->side, nl->fork_ev, 0));
  *rs = nl->side;
  return GNEP_OK;
}
static int radial_join(gnep_nlist* nl, cudaStream_t st, cudaStream_t rs) {
  if (rs == st) return GNEP_OK;
  GNEP_CUDA(cudaEventRecord(nl->join_ev, rs));
  GNEP_CUDA(cudaStreamWaitEvent(st, nl->join_ev, 0));
  return GNEP_OK;
}

#define GNEP_RADIAL_LANES(RLV, CALL)  \
  switch (RLV) {                      \
    case 16: {                        \
      constexpr int RL = 16;          \
      CALL;                           \
    } break;                          \
    case 8: {                         \
      constexpr int RL = 8;           \
      CALL;                           \
    } break;                          \
    default: {                        \
      constexpr int RL = 4;           \
      CALL;                           \
    }                                 \
  }

namespace {

template <class C>
struct Runner {
  // Network forward/backward in the model's precision: plain FP32 tiles, or
  // tensor-core tiles with TF32 or BF16 operands.
  static int network_forward(const gnep_model* m, gnep_nlist* nl, cudaStream_t st) {
    if (C::LMAX > 4 || m->precision == GNEP_PREC_FP32) {
      switch (hidden_pad(m->shape.H)) {
        case 32: return mlp_forward<C::NDES, 32, C::NS, C::NQR, C::KR>(m, nl, st);
        case 64: return mlp_forward<C::NDES, 64, C::NS, C::NQR, C::KR>(m, nl, st);
        default: return mlp_forward<C::NDES, 128, C::NS, C::NQR, C::KR>(m, nl, st);
      }
    }
    if constexpr (C::LMAX > 4) {
      return set_error(GNEP_ERR_UNSUPPORTED, "l_max > 4 runs the FP32 network only");
    } else {
      const bool tf = m->precision == GNEP_PREC_TF32;
      switch (hidden_pad_tc(m->shape.H)) {
        case 32:
          return tf ? mlp_forward_tc<true, C::NDES, 32, C::NS, C::NQR, C::KR>(m, nl, st)
                    : mlp_forward_tc<false, C::NDES, 32, C::NS, C::NQR, C::KR>(m, nl, st);
        case 64:
          return tf ? mlp_forward_tc<true, C::NDES, 64, C::NS, C::NQR, C::KR>(m, nl, st)
                    : mlp_forward_tc<false, C::NDES, 64, C::NS, C::NQR, C::KR>(m, nl, st);
        default:
          return tf ? mlp_forward_tc<true, C::NDES, 112, C::NS, C::NQR, C::KR>(m, nl, st)
                    : mlp_forward_tc<false, C::NDES, 112, C::NS, C::NQR, C::KR>(m, nl, st);
      }
    }
  }

  static int network_backward(const gnep_model* m, gnep_nlist* nl, cudaStream_t st) {
    if (C::LMAX > 4 || m->precision == GNEP_PREC_FP32) {
      switch (hidden_pad(m->shape.H)) {
        case 32: return mlp_backward<C::NDES, 32>(m, nl, st);
        case 64: return mlp_backward<C::NDES, 64>(m, nl, st);
        default: return mlp_backward<C::NDES, 128>(m, nl, st);
      }
    }
    if constexpr (C::LMAX > 4) {
      return set_error(GNEP_ERR_UNSUPPORTED, "l_max > 4 runs the FP32 network only");
    } else {
      const bool tf = m->precision == GNEP_PREC_TF32;
      switch (hidden_pad_tc(m->shape.H)) {
        case 32:
          return tf ? mlp_backward_tc<true, C::NDES, 32>(m, nl, st) : mlp_backward_tc<false, C::NDES, 32>(m, nl, st);
        case 64:
          return tf ? mlp_backward_tc<true, C::NDES, 64>(m, nl, st) : mlp_backward_tc<false, C::NDES, 64>(m, nl, st);
        default:
          return tf ? mlp_backward_tc<true, C::NDES, 112>(m, nl, st)
                    : mlp_backward_tc<false, C::NDES, 112>(m, nl, st);
      }
    }
  }

  static int descriptors(const StepArgs& A, bool with_mlp) {
    const gnep_model* m = A.m;
    gnep_nlist* nl = A.nl;
    Workspace& w = nl->ws;
    const DevModel dm = m->dev();
    const int N = nl->n_atoms;
    if (N == 0) return GNEP_OK;
    cudaStream_t rs;
    if (int rc = radial_fork(nl, A.st, &rs)) return rc;
    GNEP_RADIAL_LANES(radial_lanes(nl), ((void)launch_on(rs == A.st, k_desc_radial<C, RL>,
                                             blocks_for((int64_t)N * RL, 128), 128, 0, rs,
                                             N, dm, nl->type, nl->L[0].off, nl->L[0].rij, w.FR, w.G)));
    stage("desc_radial");
    if (int rc = ang_descriptors<C>(m, nl, A.st, w.S, w.G)) return rc;
    stage("desc_angular");
    if (int rc = radial_join(nl, A.st, rs)) return rc;
    GNEP_CHECK_LAUNCH("descriptor sweep");
    if (with_mlp) {
      if (int rc = network_forward(m, nl, A.st)) return rc;
      stage("mlp_fwd");
    }
    return GNEP_OK;
  }

  static int forward(const StepArgs& A) {
    const gnep_model* m = A.m;
    gnep_nlist* nl = A.nl;
    Workspace& w = nl->ws;
    const DevModel dm = m->dev();
    const int N = nl->n_atoms;
    if (N == 0) return GNEP_OK;
    if (nl->L[1].n > 0) {
      if (int rc = ang_force<C>(m, nl, A.st, w.S, w.Ep, w.dA)) return rc;
      stage("force_angular");
    }
    GNEP_RADIAL_LANES(radial_lanes(nl), ((void)launch_pdl(k_force_atoms<C, RL>, blocks_for((int64_t)N * RL, 128), 128, 0, A.st, 
                                             N, dm, nl->type, nl->L[0].off, nl->L[0].j, nl->L[0].rij, w.chat,
                                             nl->L[1].off, nl->L[1].rev, nl->L[1].rij, w.dA, w.F, w.Wat,
                                             nl->L[1].n > 0 && (int64_t)N * RL <= (int64_t)kPdlThreads)));
    stage("force_atoms");
    if (!A.loss_follows) {  // otherwise the loss kernel forms these sums
      const bool wide = N > 512 * (int64_t)nl->n_struct;
      (void)launch_pdl(wide ? k_struct_sum<1024> : k_struct_sum<128>, nl->n_struct, wide ? 1024 : 128, 0, A.st,
                       nl->struct_off, w.Eatom, w.Wat, w.F, w.Es, w.Ws, A.out.Eatom, A.out.F, A.out.Es, A.out.Ws);
      stage("struct_sum");
    }
    GNEP_CHECK_LAUNCH("force sweep");
    return GNEP_OK;
  }

  static int backward(const StepArgs& A) {
    const gnep_model* m = A.m;
    gnep_nlist* nl = A.nl;
    Workspace& w = nl->ws;
    const DevModel dm = m->dev();
    const int N = nl->n_atoms;
    if (N == 0) return GNEP_OK;
    cudaStream_t rs;
    if (int rc = radial_fork(nl, A.st, &rs)) return rc;
    GNEP_RADIAL_LANES(radial_lanes(nl),
                      ((void)launch_on(rs == A.st, k_tangent_radial<C, RL>, blocks_for((int64_t)N * RL, 128), 128, 0,
                          rs, N, dm, nl->type, nl->atom_struct, nl->L[0].off, nl->L[0].j, nl->L[0].rij, w.a, w.Bs,
                          w.FRd, w.Gd)));
    stage("tangent_radial");
    if (int rc = ang_tangent<C>(m, nl, A.st, w.a, w.Bs, w.S, w.Sd, w.Gd, w.wij)) return rc;
    stage("tangent_angular");
    if (int rc = radial_join(nl, A.st, rs)) return rc;
    if (int rc = network_backward(m, nl, A.st)) return rc;
    stage("mlp_bwd");
    const int nb = cgrad_blocks(nl);
    if (int rc = radial_fork(nl, A.st, &rs)) return rc;
    (void)launch_on(rs == A.st, k_cgrad_radial<C>, cgrad_radial_blocks(nl), 32 * kCgRadialWarps, 0, rs, N, nl->type, w.Gb, w.Ep, w.FR,
                    w.FRd, w.cpart);
    stage("cgrad_radial");
    if (int rc = ang_cgrad<C>(m, nl, A.st, nb, w.wij, w.S, w.Sd, w.Gb, w.Ep, w.cpart)) return rc;
    stage("cgrad");
    if (int rc = radial_join(nl, A.st, rs)) return rc;
    GNEP_CHECK_LAUNCH("backward sweeps");
    return GNEP_OK;
  }
};

}  // namespace

// Shapes with compiled kernels: (species, n_max+1, basis+1 radial; same angular; 4-body; l_max).
#define GNEP_SHAPES(X)            \
  X(2, 5, 9, 5, 9, false, 4)      \
  X(2, 9, 13, 9, 13, true, 4)     \
  X(2, 9, 13, 9, 13, false, 4)    \
  X(2, 5, 9, 5, 9, false, 6)      \
  X(2, 5, 9, 5, 9, true, 8)

#define GNEP_MATCH(P_NS, P_NQR, P_KR, P_NQA, P_KA, P_FB, P_LM)                                                \
  (s.ns == P_NS && s.nqr == P_NQR && s.kr == P_KR && s.nqa == P_NQA && s.ka == P_KA && (s.fb != 0) == P_FB && \
   s.lmax == P_LM)

bool shape_supported(const Shape& s) {
#define X(P_NS, P_NQR, P_KR, P_NQA, P_KA, P_FB, P_LM) \
  if (GNEP_MATCH(P_NS, P_NQR, P_KR, P_NQA, P_KA, P_FB, P_LM)) return true;
  GNEP_SHAPES(X)
#undef X
  return false;
}

namespace {
template <class C>
int setup_shape() {
  if (int rc = ang_setup<C>()) return rc;
  int rc = mlp_setup<C::NDES, 32, C::NS, C::NQR, C::KR>();
  if (!rc) rc = mlp_setup<C::NDES, 64, C::NS, C::NQR, C::KR>();
  if (!rc) rc = mlp_setup<C::NDES, 128, C::NS, C::NQR, C::KR>();
  if constexpr (C::LMAX <= 4) {
    if (!rc) rc = mlp_setup_tc<false, C::NDES, 32, C::NS, C::NQR, C::KR>();
    if (!rc) rc = mlp_setup_tc<false, C::NDES, 64, C::NS, C::NQR, C::KR>();
    if (!rc) rc = mlp_setup_tc<false, C::NDES, 112, C::NS, C::NQR, C::KR>();
    if (!rc) rc = mlp_setup_tc<true, C::NDES, 32, C::NS, C::NQR, C::KR>();
    if (!rc) rc = mlp_setup_tc<true, C::NDES, 64, C::NS, C::NQR, C::KR>();
    if (!rc) rc = mlp_setup_tc<true, C::NDES, 112, C::NS, C::NQR, C::KR>();
  }
  return rc;
}
}  // namespace

int shape_setup(const Shape& s) {
#define X(P_NS, P_NQR, P_KR, P_NQA, P_KA, P_FB, P_LM) \
  if (GNEP_MATCH(P_NS, P_NQR, P_KR, P_NQA, P_KA, P_FB, P_LM)) \
    return setup_shape<Sh<P_NS, P_NQR, P_KR, P_NQA, P_KA, P_FB, P_LM>>();
  GNEP_SHAPES(X)
#undef X
  return set_error(GNEP_ERR_UNSUPPORTED, "no kernel for this shape");
}

int run_descriptors(const StepArgs& A, bool with_mlp) {
  const Shape& s = A.m->shape;
#define X(P_NS, P_NQR, P_KR, P_NQA, P_KA, P_FB, P_LM) \
  if (GNEP_MATCH(P_NS, P_NQR, P_KR, P_NQA, P_KA, P_FB, P_LM)) \
    return Runner<Sh<P_NS, P_NQR, P_KR, P_NQA, P_KA, P_FB, P_LM>>::descriptors(A, with_mlp);
  GNEP_SHAPES(X)
#undef X
  return set_error(GNEP_ERR_UNSUPPORTED, "no kernel for this shape");
}

int run_forward(const StepArgs& A) {
  const Shape& s = A.m->shape;
#define X(P_NS, P_NQR, P_KR, P_NQA, P_KA, P_FB, P_LM) \
  if (GNEP_MATCH(P_NS, P_NQR, P_KR, P_NQA, P_KA, P_FB, P_LM)) \
    return Runner<Sh<P_NS, P_NQR, P_KR, P_NQA, P_KA, P_FB, P_LM>>::forward(A);
  GNEP_SHAPES(X)
#undef X
  return set_error(GNEP_ERR_UNSUPPORTED, "no kernel for this shape");
}

int run_backward(const StepArgs& A) {
  const Shape& s = A.m->shape;
#define X(P_NS, P_NQR, P_KR, P_NQA, P_KA, P_FB, P_LM) \
  if (GNEP_MATCH(P_NS, P_NQR, P_KR, P_NQA, P_KA, P_FB, P_LM)) \
    return Runner<Sh<P_NS, P_NQR, P_KR, P_NQA, P_KA, P_FB, P_LM>>::backward(A);
  GNEP_SHAPES(X)
#undef X
  return set_error(GNEP_ERR_UNSUPPORTED, "no kernel for this shape");
}

// SMs of this GPU (looked up once).
int sm_count() {
  static int sms = 0;
  if (!sms) {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        n < 1)
      n = 1;
    sms = n;
  }
  return sms;
}

// Lanes per atom of the radial sweeps: the tuned value, else 4 while that
// gives every SM at least four blocks of 128 threads, and 8 or 16 below.
int radial_lanes(const gnep_nlist* nl) {
  if (nl->tune.radial_lanes > 0) return nl->tune.radial_lanes;
  const int64_t full = 4LL * 128 * sm_count();  // threads of four blocks per SM
  const int64_t N = nl->n_atoms;
  return 4 * N >= full ? 4 : 8 * N >= full ? 8 : 16;
}

// The radial sweeps run beside the angular ones when tuned so, and by default
// while the batch has fewer than 8 x 32 atoms per SM (and 8 x 256 angular pairs).  The
// sweeps of both kinds are chains of dependent loads and products with idle
// issue slots: on a small batch neither fills the GPU and the two at once hide
// the shorter one; up to a few tiles per SM the radial warps still fill issue
// slots the angular warps leave (on the 256-structure workload, 375
// atoms per SM, the two placements time the same).  Above l_max 4 the angular
// sweeps hold fewer warps per SM and leave room at every size (l_max 8, the same
// workload: 525 us in turn, 508 us beside).
bool radial_beside(const gnep_nlist* nl) {
  if (nl->tune.beside > 0) return nl->tune.beside == 2;
  if (nl->shape.lmax > 4) return true;
  const int64_t most = 8LL * sm_count();
  return nl->n_atoms < 32 * most && nl->L[1].n < 256 * most;
}

// Persistent blocks of the c-gradient sweep: enough warps for every atom group
// up to the default (or tuned) count, at most kCgBlocksMax (the size of the
// partial buffer).  The default is what the SMs hold.
int cgrad_blocks(const gnep_nlist* nl) {
  const int per = ang_block_atoms(nl->shape), need = (nl->n_atoms + per - 1) / per;
  int cap = nl->tune.cg_blocks > 0 ? nl->tune.cg_blocks : ang_cgrad_per_sm(nl->shape.lmax) * sm_count();
  if (cap > kCgBlocksMax) cap = kCgBlocksMax;
  return need < cap ? (need > 0 ? need : 1) : cap;
}

// Rows of the coefficient partials whose radial part is written: the radial
// c-gradient's two resident blocks per SM.
int cgrad_radial_blocks(const gnep_nlist* nl) {
  const int nb = cgrad_blocks(nl), fit = 2 * sm_count();
  return nb < fit ? nb : fit;
}

// What gnep_tuning_get reports for the values 0 to 3 by default: the tile limits of
// earlier angular sweeps ([0] 32 atoms and 256 pairs, [1] 128 / channels and 128
// pairs).  The present ones cut no tiles.
void angular_tile_limits(const Shape& s, int which, int* na, int* ch) {
  const int nq = s.nqr > s.nqa ? s.nqr : s.nqa;
  if (which == 0) {
    *na = 32;
    *ch = 256;
  } else {
    *na = 128 / nq;
    *ch = 128;
  }
}

}  // namespace gnep

// ---------------------------------------------------------------------------
// Descriptors without any device allocation.
//
// Some callers must not allocate device memory at the point where they need
// descriptors: hosts whose device memory is reserved up front by another
// allocator or a fixed pool (a cudaMalloc there fails or fragments the pool),
// and per-step hooks of simulation engines that forbid allocation in their hot
// loop (cudaMalloc and cudaFree may synchronise the device).  For them the
// descriptor sweep can use this fixed scratch array, which every GPU that
// loads the library holds until the process exits, instead of workspace
// memory.  Calls share the array; calls that overlap on the GPU race.
namespace gnep {
namespace {

constexpr size_t kStaticScratchFloats = size_t(1) << 21;  // 8 MiB
static __device__ __align__(256) float g_static_scratch[kStaticScratchFloats];
constexpr int kMaxDevices = 64;
std::mutex g_static_mu;
float* g_static_ptr[kMaxDevices] = {nullptr};

// Device address of the scratch array on the current device, looked up once per
// device (host code must not use the symbol itself as a device pointer).
int static_scratch(float** out) {
  int dev = 0;
  GNEP_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return set_error(GNEP_ERR_INVALID_ARG, "device ordinal out of range");
  std::lock_guard<std::mutex> lock(g_static_mu);
  if (!g_static_ptr[dev]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess) return cuda_error(e, "cudaGetSymbolAddress(static scratch)");
    g_static_ptr[dev] = static_cast<float*>(p);
  }
  *out = g_static_ptr[dev];
  return GNEP_OK;
}

template <class C>
int descriptors_static(const StepArgs& A, float* G) {
  const gnep_model* m = A.m;
  const gnep_nlist* nl = A.nl;
  const int64_t N = nl->n_atoms;
  const int64_t fr = N * C::NS * C::KR;
  const int64_t sa = N * C::NQA * C::NLX;
  const int64_t fr_padded = (fr + 63) / 64 * 64;
  if (fr_padded + sa > (int64_t)kStaticScratchFloats)
    return set_error(GNEP_ERR_INVALID_ARG,
                     "batch too large for the fixed descriptor scratch (needs " + std::to_string(fr_padded + sa) +
                         " floats, holds " + std::to_string(kStaticScratchFloats) + ")");
  float* scratch = nullptr;
  int rc = static_scratch(&scratch);
  if (rc) return rc;
  if (N == 0) return GNEP_OK;
  const DevModel dm = m->dev();
  // Both kernels overwrite every scratch element they later read, so the
  // array needs no clearing between calls.
  GNEP_RADIAL_LANES(radial_lanes(nl), ((void)launch_pdl(k_desc_radial<C, RL>, blocks_for(N * RL, 128), 128, 0, A.st, 
                                           (int)N, dm, nl->type, nl->L[0].off, nl->L[0].rij, scratch, G)));
  if ((rc = ang_descriptors<C>(m, nl, A.st, scratch + fr_padded, G))) return rc;
  GNEP_CHECK_LAUNCH("descriptor sweep (static scratch)");
  return GNEP_OK;
}

}  // namespace

int run_descriptors_static(const StepArgs& A, float* G) {
  const Shape& s = A.m->shape;
#define X(P_NS, P_NQR, P_KR, P_NQA, P_KA, P_FB, P_LM) \
  if (GNEP_MATCH(P_NS, P_NQR, P_KR, P_NQA, P_KA, P_FB, P_LM)) \
    return descriptors_static<Sh<P_NS, P_NQR, P_KR, P_NQA, P_KA, P_FB, P_LM>>(A, G);
  GNEP_SHAPES(X)
#undef X
  return set_error(GNEP_ERR_UNSUPPORTED, "no kernel for this shape");
}

}  // namespace gnep
