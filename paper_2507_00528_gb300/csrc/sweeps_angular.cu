// Angular sweeps of one training step for every l_max (4, 6, 8): descriptors
// (Eqs. 7-8, 4-body), pair forces, the tangent and the coefficient gradient.  See angular.cuh for the thread map
// and sweeps.cu for the gradient route.
#include "angular.cuh"
#include "sweeps_angular.cuh"

namespace gnep {

namespace {

// Shared memory of a block: the coefficient rows, then per warp CP pair rows
// of RS floats, [B | g] or (tangent) [B | D | (g, ga) pairs], and the atom
// records of the tangent (a_i, B_s).
template <class C, bool TAN>
struct DescRow {
  using A = Ang<C>;
  static constexpr int G = TAN ? 2 * A::NLX : A::NLX;  // first channel value
  static constexpr int RS = odd4(G + (TAN ? 2 : 1) * A::NQ);
  static constexpr int REC = TAN ? 12 * A::AW : 0;
  static constexpr size_t warp_floats = (size_t)A::CP * RS + REC;
  static constexpr size_t smem = sizeof(float) * ((size_t)A::NS * A::NS * A::CST + kAngW * warp_floats);
};

// N values to a 16-byte aligned place in 16-byte words (the rows' stride is odd in
// those, so a warp's stores meet no bank twice; single words would, fourfold).
template <int N>
__device__ __forceinline__ void store_row(float* o, const float (&v)[N]) {
#pragma unroll
  for (int q = 0; q + 4 <= N; q += 4)
    *reinterpret_cast<float4*>(o + q) = make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
  if constexpr (N % 4 == 1) o[N - 1] = v[N - 1];
  if constexpr (N % 4 >= 2) *reinterpret_cast<float2*>(o + N / 4 * 4) = make_float2(v[N / 4 * 4], v[N / 4 * 4 + 1]);
  if constexpr (N % 4 == 3) o[N - 1] = v[N - 1];
}

// The geometry of one pair into its row: basis sums g_n (and the tangent's
// ga_n = g_n' (u . w)), harmonics B and D = grad B . w.
template <class C, bool TAN>
__device__ __forceinline__ void write_pair_row(float* row, const float* cIJ, float4 r, float3 w, float rca_inv) {
  using A = Ang<C>;
  float rr, ri;
  bond_length(r, rr, ri);
  const float ux = r.x * ri, uy = r.y * ri, uz = r.z * ri;
  float f[C::KA], fu[C::KA], g[C::NQA], ga[C::NQA];
  const float ru = ux * w.x + uy * w.y + uz * w.z;
  if (TAN) {
    radial_basis_d<C::KA>(rr, rca_inv, f, fu);
#pragma unroll
    for (int k = 0; k < C::KA; ++k) fu[k] *= ru;
  } else {
    radial_basis<C::KA>(rr, rca_inv, f);
  }
  channel_sums<C, TAN>(cIJ, f, fu, g, ga);
  {
    constexpr int NG = (TAN ? 2 : 1) * C::NQA;
    float v[NG];
#pragma unroll
    for (int n = 0; n < C::NQA; ++n) {
      v[TAN ? 2 * n : n] = g[n];
      if (TAN) v[TAN ? 2 * n + 1 : n] = ga[n];
    }
    store_row(row + DescRow<C, TAN>::G, v);
  }
  float B[A::NLX], D[TAN ? A::NLX : 1];
  // 16-byte stores as soon as four components are known
  auto flush = [&](auto q0, auto q1) {
#pragma unroll
    for (int q = decltype(q0)::value / 4 * 4; q + 4 <= decltype(q1)::value; q += 4) {
      *reinterpret_cast<float4*>(row + q) = make_float4(B[q], B[q + 1], B[q + 2], B[q + 3]);
      if constexpr (TAN)
        *reinterpret_cast<float4*>(row + A::NLX + q) = make_float4(D[q], D[q + 1], D[q + 2], D[q + 3]);
    }
  };
  {
    float B4[NLM], D4[NLM];
    if constexpr (TAN)
      harmonics_dir(ux, uy, uz, ri, w.x, w.y, w.z, B4, D4);
    else
      harmonics(ux, uy, uz, B4);
#pragma unroll
    for (int q = 0; q < NLM; ++q) {
      B[q] = B4[q];
      if constexpr (TAN) D[q] = D4[q];
    }
    flush(std::integral_constant<int, 0>{}, std::integral_constant<int, NLM>{});
  }
  if constexpr (C::LMAX > 4) {
    solid_levels<C::LMAX>(ux, uy, uz, [&](auto lc, const auto& R, const auto& L) {
      constexpr int l = decltype(lc)::value, q0 = l * l - 1;
#pragma unroll
      for (int k = 0; k <= 2 * l; ++k) B[q0 + k] = solid_comp(R, k);
      if constexpr (TAN) {  // grad B . w = grad R . (w - (u . w) u) / r
        float d[2 * l + 1];
        solid_dir<l>(L, (w.x - ru * ux) * ri, (w.y - ru * uy) * ri, (w.z - ru * uz) * ri, d);
#pragma unroll
        for (int k = 0; k <= 2 * l; ++k) D[q0 + k] = d[k];
      }
      flush(std::integral_constant<int, q0>{}, std::integral_constant<int, q0 + 2 * l + 1>{});
    });
  }
}

// Degree sums over the atom lanes of one channel: lane qg holds t[e] = C_q x_q y_q
// of the components q = 8 qg + e.  With the degrees starting at q = 0, 3, 8, 15,
// 24, 35, 48, 63 a lane's components belong to one degree (A), or to the end of
// one and the start of the next (B, from e = cut on); sums that span lanes are
// passed up: q_4 = B_1 + A_2, q_5 = A_3 + A_4, q_6 = B_4 + A_5, q_7 = A_6 + A_7,
// q_8 = B_7 + A_8 + A_9.  emit(l, value) runs on the lane that ends a degree.
template <class C, class F>
__device__ __forceinline__ void degree_sums(const float (&t)[8], int qg, F&& emit) {
  const float s0 = (t[0] + t[1]) + t[2], s3 = (t[3] + t[4]) + (t[5] + t[6]);
  const bool cut3 = qg == 0 || qg == 4, cut7 = qg == 1 || qg == 7;
  const float B = cut3 ? s3 + t[7] : cut7 ? t[7] : 0.f;
  float A = cut3 ? s0 : s0 + s3 + (cut7 ? 0.f : t[7]);
  const float up = __shfl_up_sync(0xffffffffu, qg == 3 || qg == 6 ? A : B, 1);
  if (qg == 2 || qg == 4 || qg == 5 || qg == 7 || qg == 8) A += up;
  if constexpr (C::LMAX > 6) {
    const float up2 = __shfl_up_sync(0xffffffffu, A, 1);
    if (qg == 9) A += up2;
  }
  constexpr unsigned long long kDeg = 0x8070650431ull;  // degree that lane qg ends (0: none)
  const int l = (int)(kDeg >> (4 * qg)) & 15;
  if (l > 0) emit(l, A);
  if (qg == 0) emit(2, B);
}

// Sweep 1 (TAN = false): S_nq = sum_j g_n(r_ij) B_q (Eq. 8), q_nl = sum_m C S^2
// (Eq. 7), q4_n.  Sweep 3 (TAN = true): with w_ij = (a_j - a_i) + B_s r_ij
// (stored for sweep 4) Sdot_nq = sum_j [g_n' (u . w) B_q + g_n D_q],
// qdot_nl = 2 sum_m C S Sdot and the 4-body tangent.
// Bound by shared-memory bandwidth and the latency of a warp's alternating
// phases (ncu: 64 to 68% of the wavefront slots, a third of the issue slots used).  Three atoms a
// warp, because their 25 pairs and 27 summing lanes fill both mappings; a summing
// lane's 3 x 8 tile reads 11 values for 24 products (one channel of all 24
// components: 25 for 24).  On the 256-structure batch (55,200 atoms, 460,534
// angular pairs, n_max 8, l_max 4) the descriptors take 35 us and the tangent 61
// us (one channel per lane: 40 and 65; per-atom split-TF32 tensor-core tiles: 68
// and 106); at l_max 8 43 and 102 us (61 and 121; lanes summing one (n,
// component) each over the pairs: 464 and 711).
// Blocks per SM: the register bound at which a thread spills at most 104 bytes; one
// block more spills 108 to 288 bytes in the tangent, and 20 to 60 in the descriptors
// (but for l_max 6), where now at most 4 do.
template <class C, bool TAN>
__global__ void __launch_bounds__(32 * kAngW, TAN ? (C::LMAX > 4 || C::NQA < 9 ? 3 : 4) : (C::LMAX > 4 ? 4 : 5))
    k_ang_desc(int N, DevModel dm, const int* __restrict__ type, const int* __restrict__ atom_struct,
               const int* __restrict__ off, const int* __restrict__ jj, const float4* __restrict__ rij,
               const float4* __restrict__ av, const float* __restrict__ Bs, const float* __restrict__ Sin,
               float* __restrict__ Sout, float* __restrict__ Gout, float4* __restrict__ wij) {
  using A = Ang<C>;
  using R = DescRow<C, TAN>;
  constexpr int AW = A::AW, NQ = A::NQ, NLX = A::NLX, CP = A::CP, RS = R::RS, TN = A::TN;
  extern __shared__ float4 smraw[];
  float* cA = reinterpret_cast<float*>(smraw);
  const bool room = (int)gridDim.x * kAngW * A::AW >= N;
  if (!TAN) GNEP_PDL_START_IF(room);  // the previous kernel may have updated the parameters
  load_ang_coef<C>(dm, cA);
  if (TAN) GNEP_PDL_START_IF(room);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* rows = cA + A::NS * A::NS * A::CST + warp * R::warp_floats;
  float* rec = rows + CP * RS;  // [AW][12]: a_i (3), B_s (6)
  const int a = lane / A::TPA, n0 = lane % A::TPA / A::QG * TN, qg = lane % A::QG;  // summing lane
  const int ngrp = (N + AW - 1) / AW, stride = gridDim.x * kAngW;
  int grp = blockIdx.x * kAngW + warp;
  if (grp >= ngrp) return;
  float wt[8];  // C_q of the lane's components
#pragma unroll
  for (int e = 0; e < 8; ++e) wt[e] = ang_weight_at(8 * qg + e);
  int offl, typl;
  group_fetch<C>(grp, N, off, type, lane, offl, typl);
  for (; grp < ngrp; grp += stride) {
    const int i0 = grp * AW, i = i0 + a;
    const bool mine = a < AW && i < N;
    const int p0 = __shfl_sync(0xffffffffu, offl, 0), p1 = __shfl_sync(0xffffffffu, offl, AW);
    const int q0 = __shfl_sync(0xffffffffu, offl, min(a, AW)), q1 = __shfl_sync(0xffffffffu, offl, min(a + 1, AW));
    int offn = offl, typn = typl;
    if (grp + stride < ngrp) group_fetch<C>(grp + stride, N, off, type, lane, offn, typn);
    const size_t srow = ((size_t)(mine ? i : 0) * NQ + n0) * NLX + 8 * qg;  // the lane's first row of S
    float x[TAN ? TN : 1][8];  // the tangent's S rows, read ahead of the pair loop
    if constexpr (TAN) {
      if (lane < AW && i0 + lane < N) {
        const float4 ai = av[i0 + lane];
        const float* b = Bs + 6 * atom_struct[i0 + lane];
        float* o = rec + 12 * lane;
        o[0] = ai.x; o[1] = ai.y; o[2] = ai.z;
#pragma unroll
        for (int q = 0; q < 6; ++q) o[3 + q] = b[q];
      }
#pragma unroll
      for (int n = 0; n < TN; ++n) load8(Sin + srow + n * NLX, x[n]);
      __syncwarp();
    }
    float2 acc[TN][4];
#pragma unroll
    for (int n = 0; n < TN; ++n)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[n][q] = make_float2(0.f, 0.f);
    for (int cs = p0; cs < p1; cs += CP) {
      const int ce = min(cs + CP, p1);
#pragma unroll
      for (int u = 0; u < CP / 32; ++u) {
        const int p = cs + 32 * u + lane;
        const int sl = pair_slot<C>(p, offl);
        const int I = __shfl_sync(0xffffffffu, typl, sl);
        if (p < ce) {
          const float4 r = rij[p];
          float3 w = make_float3(0.f, 0.f, 0.f);
          if constexpr (TAN) {
            const float4 aj = av[jj[p]];
            const float* o = rec + 12 * sl;
            w.x = aj.x - o[0] + (o[3] * r.x + o[6] * r.y + o[8] * r.z);
            w.y = aj.y - o[1] + (o[6] * r.x + o[4] * r.y + o[7] * r.z);
            w.z = aj.z - o[2] + (o[8] * r.x + o[7] * r.y + o[5] * r.z);
            wij[p] = make_float4(w.x, w.y, w.z, 0.f);
          }
          write_pair_row<C, TAN>(rows + (32 * u + lane) * RS, cA + (I * A::NS + (int)r.w) * A::CST, r, w, dm.rca_inv);
        }
      }
      __syncwarp();
      if (mine) {
        const int s1 = min(q1, ce) - cs;
        for (int s = max(q0, cs) - cs; s < s1; ++s) {
          const float* row = rows + s * RS;
          const float4 b0 = *reinterpret_cast<const float4*>(row + 8 * qg), b1 = *reinterpret_cast<const float4*>(row + 8 * qg + 4);
          if constexpr (TAN) {
            const float4 d0 = *reinterpret_cast<const float4*>(row + NLX + 8 * qg),
                         d1 = *reinterpret_cast<const float4*>(row + NLX + 8 * qg + 4);
#pragma unroll
            for (int n = 0; n < TN; ++n) {
              const float2 gg = *reinterpret_cast<const float2*>(row + R::G + 2 * (n0 + n));
              const float2 g = dup2(gg.x), ga = dup2(gg.y);
              acc[n][0] = fma2(ga, lo2(b0), fma2(g, lo2(d0), acc[n][0]));
              acc[n][1] = fma2(ga, hi2(b0), fma2(g, hi2(d0), acc[n][1]));
              acc[n][2] = fma2(ga, lo2(b1), fma2(g, lo2(d1), acc[n][2]));
              acc[n][3] = fma2(ga, hi2(b1), fma2(g, hi2(d1), acc[n][3]));
            }
          } else {
#pragma unroll
            for (int n = 0; n < TN; ++n) {
              const float2 g = dup2(row[R::G + n0 + n]);
              acc[n][0] = fma2(g, lo2(b0), acc[n][0]);
              acc[n][1] = fma2(g, hi2(b0), acc[n][1]);
              acc[n][2] = fma2(g, lo2(b1), acc[n][2]);
              acc[n][3] = fma2(g, hi2(b1), acc[n][3]);
            }
          }
        }
      }
      __syncwarp();  // the rows are read before the next chunk (or group) replaces them
    }
    float* gi = Gout + (size_t)i * C::NDES;
    float y[TN][8];
#pragma unroll
    for (int n = 0; n < TN; ++n) {
      float t[8];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        y[n][2 * q] = acc[n][q].x;
        y[n][2 * q + 1] = acc[n][q].y;
      }
      if (mine) store8(Sout + srow + n * NLX, y[n]);
#pragma unroll
      for (int e = 0; e < 8; ++e) t[e] = wt[e] * (TAN ? x[TAN ? n : 0][e] : y[n][e]) * y[n][e];
      degree_sums<C>(t, qg, [&](int l, float v) {
        if (mine) gi[C::vang(n0 + n, l)] = TAN ? 2.f * v : v;
      });
    }
    if constexpr (C::FB) {
      static_assert(A::QG >= TN, "a lane per row of the tile");
      float y2[5], v;
      spread_moments<C>(y, lane, qg, y2);
      if constexpr (TAN) {
        float x2[5], g4[5];
        spread_moments<C>(x, lane, qg, x2);
        q4_grad(x2, g4);
        v = 0.f;
#pragma unroll
        for (int m = 0; m < 5; ++m) v = fmaf(g4[m], y2[m], v);
      } else {
        v = q4_value(y2);
      }
      if (mine && qg < TN) gi[C::v4b(n0 + qg)] = v;
    }
    offl = offn;
    typl = typn;
  }
}

// ------------------------------------------------------------- sweep 2

// Rows of the group's atoms that the pair lanes contract: components of degree
// up to 4 as [n][24 W] rows (W values per component), above as [q - 24][HW]
// with the channels side by side, since those harmonics appear one by one.
template <class C, int W>
struct AtomRows {
  using A = Ang<C>;
  static constexpr int L = odd4(A::NQ * NLM * W);
  static constexpr int HW = W == 1 ? (A::NQ + 3) / 4 * 4 : 4 * ((A::NQ + 1) / 2);  // [s] or [s | t] padded to pairs
  static constexpr int H = C::LMAX > 4 ? odd4((A::NLX - NLM) * HW) : 0;
  static constexpr int floats = A::AW * (L + H);
  static_assert(HW % 4 == 0, "16-byte channel rows");
};

template <class C>
struct ForceRow {
  using A = Ang<C>;
  using R = AtomRows<C, 1>;
  static constexpr size_t smem = sizeof(float) * ((size_t)A::NS * A::NS * A::CST + kAngW * (size_t)R::floats);
};

// Calls f(integral base) with the first component of half h of a channel.
template <class C, class F>
__device__ __forceinline__ void with_half(int h, F&& f) {
  if (Ang<C>::SPL == 1 || h == 0)
    f(std::integral_constant<int, 0>{});
  else
    f(std::integral_constant<int, Ang<C>::SPL == 1 ? 0 : Ang<C>::NQL>{});
}

template <int N4>
__device__ __forceinline__ void load_row4(const float* p, float (&x)[4 * N4]) {
#pragma unroll
  for (int q = 0; q < N4; ++q) {
    const float4 v = reinterpret_cast<const float4*>(p)[q];
    x[4 * q] = v.x; x[4 * q + 1] = v.y; x[4 * q + 2] = v.z; x[4 * q + 3] = v.w;
  }
}

// Pair forces dE_i/dr_ij = P u + (I - u u^T) v / r  (C2.1, C2.3, C3.6) with
//   P = sum_q ghat'_q B_q,  v = sum_q ghat_q grad p_q  (p_q the polynomial of B_q),
//   ghat_q = sum_n g_n Shat_nq,  ghat'_q = sum_n g_n' Shat_nq,
//   Shat_nq = dE_i/dS_nq = 2 C_q E'_{n l} S_nq (+ E'_4b,n dq4/dS_n2m).
// Channel lanes form Shat in shared memory, pair lanes contract it.  Bound by
// shared-memory bandwidth (216 row values and 120 coefficients per pair at
// n_max 8).  256 structures: 42 us at n_max 8, l_max 4, against 48 us with block
// tiles and the gradient of every component projected; 73 us at l_max 8 against
// 480 us with three lanes per pair running the recurrence in dual numbers.
template <class C>
__global__ void __launch_bounds__(32 * kAngW)
    k_ang_force(int N, DevModel dm, const int* __restrict__ type, const int* __restrict__ off,
                const float4* __restrict__ rij, const float* __restrict__ S, const float* __restrict__ Ep,
                float4* __restrict__ dA) {
  using A = Ang<C>;
  using R = AtomRows<C, 1>;
  constexpr int AW = A::AW, NQ = A::NQ, NQL = A::NQL, NLX = A::NLX, KA = C::KA;
  extern __shared__ float4 smraw[];
  float* cA = reinterpret_cast<float*>(smraw);
  load_ang_coef<C>(dm, cA);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* aL = cA + A::NS * A::NS * A::CST + warp * R::floats;  // [AW][R::L]
  float* aH = aL + AW * R::L;                                   // [AW][R::H]
  const int a = lane / A::LPA, n = (lane % A::LPA) / A::SPL, h = lane % A::SPL;
  const int ngrp = (N + AW - 1) / AW, stride = gridDim.x * kAngW;
  int grp = blockIdx.x * kAngW + warp;
  if (grp >= ngrp) {
    GNEP_PDL_START_IF((int)gridDim.x * kAngW * AW >= N);
    return;
  }
  int offl, typl;
  group_fetch<C>(grp, N, off, type, lane, offl, typl);
  GNEP_PDL_START_IF((int)gridDim.x * kAngW * AW >= N);
  for (; grp < ngrp; grp += stride) {
    const int i0 = grp * AW, i = i0 + a;
    const int p0 = __shfl_sync(0xffffffffu, offl, 0), p1 = __shfl_sync(0xffffffffu, offl, AW);
    int offn = offl, typn = typl;
    if (grp + stride < ngrp) group_fetch<C>(grp + stride, N, off, type, lane, offn, typn);
    if (a < AW && i < N) {
      float x[NQL];
      load_row4<NQL / 4>(S + ((size_t)i * NQ + n) * NLX + h * NQL, x);
      const float* ep = Ep + (size_t)i * C::NDES;
      with_half<C>(h, [&](auto bc) {
        constexpr int base = decltype(bc)::value, lb = ang_deg(base);
        float e[C::LMAX + 1];
#pragma unroll
        for (int l = lb; l <= ang_deg(base + NQL - 1); ++l) e[l] = 2.f * ep[C::vang(n, l)];
        float g4[5], e4 = 0.f;
        if constexpr (C::FB && base == 0) {
          q4_grad(&x[3], g4);
          e4 = ep[C::v4b(n)];
        }
#pragma unroll
        for (int q = 0; q < NQL; ++q) x[q] *= ang_weight(base + q) * e[ang_deg(base + q)];
        if constexpr (C::FB && base == 0) {
#pragma unroll
          for (int m = 0; m < 5; ++m) x[3 + m] = fmaf(e4, g4[m], x[3 + m]);
        }
        if constexpr (base < NLM) {
          float4* o = reinterpret_cast<float4*>(aL + a * R::L + n * NLM + base);
#pragma unroll
          for (int q = 0; q < (NLM - base < NQL ? NLM - base : NQL) / 4; ++q)
            o[q] = make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
        }
#pragma unroll
        for (int q = (base < NLM ? NLM - base : 0); q < NQL; ++q)
          aH[a * R::H + (base + q - NLM) * R::HW + n] = x[q];
      });
    }
    __syncwarp();
    for (int cs = p0; cs < p1; cs += 32) {
      const int p = cs + lane;
      const int sl = pair_slot<C>(p, offl);
      const int I = __shfl_sync(0xffffffffu, typl, sl);
      if (p < p1) {
        const float4 r = rij[p];
        float rr, ri;
        bond_length(r, rr, ri);
        const float ux = r.x * ri, uy = r.y * ri, uz = r.z * ri;
        float f[KA], fp[KA], g[NQ], gp[NQ];
        radial_basis_d<KA>(rr, dm.rca_inv, f, fp);
        channel_sums<C, true>(cA + (I * A::NS + (int)r.w) * A::CST, f, fp, g, gp);
        float P = 0.f, vx = 0.f, vy = 0.f, vz = 0.f;
        {
          float2 gh[NLM / 2], ghp[NLM / 2];
#pragma unroll
          for (int q = 0; q < NLM / 2; ++q) gh[q] = ghp[q] = make_float2(0.f, 0.f);
          const float4* s4 = reinterpret_cast<const float4*>(aL + sl * R::L);
#pragma unroll
          for (int m = 0; m < NQ; ++m) {
            const float2 gm = dup2(g[m]), gpm = dup2(gp[m]);
#pragma unroll
            for (int q = 0; q < NLM / 4; ++q) {
              const float4 v = s4[m * (NLM / 4) + q];
              gh[2 * q] = fma2(gm, lo2(v), gh[2 * q]);
              ghp[2 * q] = fma2(gpm, lo2(v), ghp[2 * q]);
              gh[2 * q + 1] = fma2(gm, hi2(v), gh[2 * q + 1]);
              ghp[2 * q + 1] = fma2(gpm, hi2(v), ghp[2 * q + 1]);
            }
          }
          float B[NLM], gx[NLM], gy[NLM], gz[NLM];
          harmonics_grad(ux, uy, uz, B, gx, gy, gz);
#pragma unroll
          for (int q = 0; q < NLM; ++q) {
            const float s = q & 1 ? gh[q / 2].y : gh[q / 2].x, sp = q & 1 ? ghp[q / 2].y : ghp[q / 2].x;
            P = fmaf(sp, B[q], P);
            vx = fmaf(s, gx[q], vx);
            vy = fmaf(s, gy[q], vy);
            vz = fmaf(s, gz[q], vz);
          }
        }
        if constexpr (C::LMAX > 4) {
          const float* hr = aH + sl * R::H;
          solid_levels<C::LMAX>(ux, uy, uz, [&](auto lc, const auto& Rl, const auto& Ll) {
            constexpr int l = decltype(lc)::value;
            static_for<0, 2 * l + 1>([&](auto kc) {
              constexpr int k = decltype(kc)::value;
              float s[R::HW];
              load_row4<R::HW / 4>(hr + (l * l - 1 + k - NLM) * R::HW, s);
              float gh = 0.f, ghp = 0.f;
#pragma unroll
              for (int m = 0; m < NQ; ++m) {
                gh = fmaf(g[m], s[m], gh);
                ghp = fmaf(gp[m], s[m], ghp);
              }
              const float3 d = solid_grad<l, k>(Ll);
              P = fmaf(ghp, solid_comp(Rl, k), P);
              vx = fmaf(gh, d.x, vx);
              vy = fmaf(gh, d.y, vy);
              vz = fmaf(gh, d.z, vz);
            });
          });
        }
        const float uv = ux * vx + uy * vy + uz * vz;
        dA[p] = make_float4(fmaf(P, ux, (vx - uv * ux) * ri), fmaf(P, uy, (vy - uv * uy) * ri),
                            fmaf(P, uz, (vz - uv * uz) * ri), 0.f);
      }
    }
    __syncwarp();  // the atom rows are read before the next group replaces them
    offl = offn;
    typl = typn;
  }
}

// ------------------------------------------------------------- sweep 4

// Angular coefficient gradient: per pair
//   P_n = sum_q Sbar_nq B_q + Sdbar_nq D_q,  R_n = sum_q Sdbar_nq B_q,
//   dL/dc^A_nk^{IJ} += P_n f_k + R_n fu_k,   fu_k = f_k' (u . w_ij),
//   Sbar_nq  = 2 C_q (Gbar_nl S_nq - E'_nl Sdot_nq) (+ 4-body terms),
//   Sdbar_nq = -2 C_q E'_nl S_nq                    (+ 4-body term).
// Channel lanes form [Sbar | Sdbar], pair lanes contract it to (P, R) and leave
// them with (f, fu) in shared memory, and output lanes (n, group of k) add the
// pairs' products into registers per species pair.  The accumulators stay in
// registers over all of a warp's groups; the block folds its warps in order and
// writes cpart[block][c^A] once.  Bound by shared-memory bandwidth (each pair
// lane reads its atom's 432 row values, 27 output lanes 12 values per pair).
// 256 structures: 91 us at n_max 8, l_max 4 (71% of the wavefront slots), against
// 125 us as split-TF32 tensor-core products in block tiles; 143 us at n_max 4,
// l_max 8, against 770 us with a pair per lane and scalar row loads.
template <class C>
struct CgradRow {
  using A = Ang<C>;
  using R = AtomRows<C, 2>;
  static constexpr int KG = 3, KW = (C::KA + KG - 1) / KG;  // groups of k, k per group
  static constexpr int GW = (2 * KW + 3) / 4 * 4;           // floats of a group: (f, fu) pairs
  static constexpr int PR = KG * GW;                        // (P, R) pairs follow
  static constexpr int RS = odd4(PR + 2 * A::NQ);
  static constexpr int NOUT = A::NQ * KG;                   // output lanes
  static constexpr int PARS = 32 / NOUT;                    // pairs taken at once
  static constexpr int warp_floats = R::floats + 32 * RS + 32;
  static constexpr size_t smem = sizeof(float) * ((size_t)kAngW * warp_floats);
  static_assert(kAngW * C::NCA <= kAngW * warp_floats, "the fold fits the rows");
};

template <class C>
__global__ void __launch_bounds__(32 * kAngW, ang_cgrad_per_sm(C::LMAX))
    k_ang_cgrad(int N, DevModel dm, const int* __restrict__ type, const int* __restrict__ off,
                const float4* __restrict__ rij, const float4* __restrict__ wij, const float* __restrict__ S,
                const float* __restrict__ Sd, const float* __restrict__ Gb, const float* __restrict__ Ep,
                float* __restrict__ cpart) {
  using A = Ang<C>;
  using R = AtomRows<C, 2>;
  using Q = CgradRow<C>;
  constexpr int AW = A::AW, NQ = A::NQ, NQL = A::NQL, NLX = A::NLX, KA = C::KA, NS = A::NS, KW = Q::KW;
  extern __shared__ float4 smraw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* aL = reinterpret_cast<float*>(smraw) + warp * Q::warp_floats;  // [AW][R::L]
  float* aH = aL + AW * R::L;                                            // [AW][R::H]
  float* rows = aL + R::floats;                                          // [32][RS]
  int* cls = reinterpret_cast<int*>(rows + 32 * Q::RS);                  // [32] species pair
  const int a = lane / A::LPA, n = (lane % A::LPA) / A::SPL, h = lane % A::SPL;
  const int on = lane % Q::NOUT / Q::KG, og = lane % Q::KG, par = lane / Q::NOUT;  // output lane
  const int ngrp = (N + AW - 1) / AW, stride = gridDim.x * kAngW;
  float acc[NS * NS][KW];
#pragma unroll
  for (int c = 0; c < NS * NS; ++c)
#pragma unroll
    for (int k = 0; k < KW; ++k) acc[c][k] = 0.f;
  int grp = blockIdx.x * kAngW + warp;
  int offl = 0, typl = 0;
  if (grp < ngrp) group_fetch<C>(grp, N, off, type, lane, offl, typl);
  GNEP_PDL_START_IF((int)gridDim.x * kAngW * AW >= N);
  for (; grp < ngrp; grp += stride) {
    const int i0 = grp * AW, i = i0 + a;
    const int p0 = __shfl_sync(0xffffffffu, offl, 0), p1 = __shfl_sync(0xffffffffu, offl, AW);
    int offn = offl, typn = typl;
    if (grp + stride < ngrp) group_fetch<C>(grp + stride, N, off, type, lane, offn, typn);
    if (a < AW && i < N) {
      float s[NQL], d[NQL];
      load_row4<NQL / 4>(S + ((size_t)i * NQ + n) * NLX + h * NQL, s);
      load_row4<NQL / 4>(Sd + ((size_t)i * NQ + n) * NLX + h * NQL, d);
      const float* gb = Gb + (size_t)i * C::NDES;
      const float* ep = Ep + (size_t)i * C::NDES;
      with_half<C>(h, [&](auto bc) {
        constexpr int base = decltype(bc)::value, lb = ang_deg(base);
        float e[C::LMAX + 1], b[C::LMAX + 1];
#pragma unroll
        for (int l = lb; l <= ang_deg(base + NQL - 1); ++l) {
          b[l] = 2.f * gb[C::vang(n, l)];
          e[l] = 2.f * ep[C::vang(n, l)];
        }
        float g4[5], h4[5], gb4 = 0.f, ep4 = 0.f;
        if constexpr (C::FB && base == 0) {
          q4_grad(&s[3], g4);
          q4_hvp(&s[3], &d[3], h4);
          gb4 = gb[C::v4b(n)];
          ep4 = ep[C::v4b(n)];
        }
#pragma unroll
        for (int q = 0; q < NQL; ++q) {
          const int l = ang_deg(base + q);
          const float w = ang_weight(base + q), sq = s[q];
          s[q] = w * fmaf(b[l], sq, -e[l] * d[q]);
          d[q] = -w * e[l] * sq;
        }
        if constexpr (C::FB && base == 0) {
#pragma unroll
          for (int m = 0; m < 5; ++m) {
            s[3 + m] += gb4 * g4[m] - ep4 * h4[m];
            d[3 + m] -= ep4 * g4[m];
          }
        }
        if constexpr (base < NLM) {
          constexpr int m4 = (NLM - base < NQL ? NLM - base : NQL) / 4;
          float4* o = reinterpret_cast<float4*>(aL + a * R::L + n * 2 * NLM + base);
#pragma unroll
          for (int q = 0; q < m4; ++q) {
            o[q] = make_float4(s[4 * q], s[4 * q + 1], s[4 * q + 2], s[4 * q + 3]);
            o[NLM / 4 + q] = make_float4(d[4 * q], d[4 * q + 1], d[4 * q + 2], d[4 * q + 3]);
          }
        }
#pragma unroll
        for (int q = (base < NLM ? NLM - base : 0); q < NQL; ++q) {
          float* o = aH + a * R::H + (base + q - NLM) * R::HW;
          o[n] = s[q];
          o[R::HW / 2 + n] = d[q];
        }
      });
    }
    __syncwarp();
    for (int cs = p0; cs < p1; cs += 32) {
      const int p = cs + lane, np = min(32, p1 - cs);
      const int sl = pair_slot<C>(p, offl);
      const int I = __shfl_sync(0xffffffffu, typl, sl);
      if (p < p1) {
        const float4 r = rij[p], w = wij[p];
        float rr, ri;
        bond_length(r, rr, ri);
        const float ux = r.x * ri, uy = r.y * ri, uz = r.z * ri;
        const float ru = ux * w.x + uy * w.y + uz * w.z;
        float* row = rows + lane * Q::RS;
        {
          float f[Q::KG * KW], fu[Q::KG * KW];
          float fk[KA], fp[KA];
          radial_basis_d<KA>(rr, dm.rca_inv, fk, fp);
#pragma unroll
          for (int k = 0; k < Q::KG * KW; ++k) {
            f[k] = k < KA ? fk[k < KA ? k : 0] : 0.f;
            fu[k] = k < KA ? fp[k < KA ? k : 0] * ru : 0.f;
          }
#pragma unroll
          for (int j = 0; j < Q::KG; ++j)
#pragma unroll
            for (int k = 0; k < KW; k += 2) {
              const int q = j * KW + k;
              const bool two = k + 1 < KW;
              *reinterpret_cast<float4*>(row + j * Q::GW + 2 * k) =
                  make_float4(f[q], fu[q], two ? f[two ? q + 1 : q] : 0.f, two ? fu[two ? q + 1 : q] : 0.f);
            }
        }
        cls[lane] = I * NS + (int)r.w;
        float P[NQ + 1], T[NQ + 1];
        P[NQ] = T[NQ] = 0.f;
        {
          float B[NLM], D[NLM];
          harmonics_dir(ux, uy, uz, ri, w.x, w.y, w.z, B, D);
          const float4* s4 = reinterpret_cast<const float4*>(aL + sl * R::L);
#pragma unroll
          for (int m = 0; m < NQ; ++m) {
            float2 pp = make_float2(0.f, 0.f), tt = pp;
#pragma unroll
            for (int q = 0; q < NLM / 4; ++q) {
              const float4 sb = s4[m * (NLM / 2) + q], sd = s4[m * (NLM / 2) + NLM / 4 + q];
              const float2 b0 = make_float2(B[4 * q], B[4 * q + 1]), b1 = make_float2(B[4 * q + 2], B[4 * q + 3]);
              pp = fma2(lo2(sb), b0, fma2(lo2(sd), make_float2(D[4 * q], D[4 * q + 1]), pp));
              pp = fma2(hi2(sb), b1, fma2(hi2(sd), make_float2(D[4 * q + 2], D[4 * q + 3]), pp));
              tt = fma2(hi2(sd), b1, fma2(lo2(sd), b0, tt));
            }
            P[m] = pp.x + pp.y;
            T[m] = tt.x + tt.y;
          }
        }
        if constexpr (C::LMAX > 4) {
          constexpr int NP = (NQ + 1) / 2;
          float2 p2[NP], t2[NP];
#pragma unroll
          for (int m = 0; m < NP; ++m) {
            p2[m] = make_float2(P[2 * m], P[2 * m + 1]);
            t2[m] = make_float2(T[2 * m], T[2 * m + 1]);
          }
          const float* hr = aH + sl * R::H;
          solid_levels<C::LMAX>(ux, uy, uz, [&](auto lc, const auto& Rl, const auto& Ll) {
            constexpr int l = decltype(lc)::value;
            float d[2 * l + 1];
            solid_dir<l>(Ll, (w.x - ru * ux) * ri, (w.y - ru * uy) * ri, (w.z - ru * uz) * ri, d);
#pragma unroll
            for (int k = 0; k <= 2 * l; ++k) {
              const float2 b2 = dup2(solid_comp(Rl, k)), d2 = dup2(d[k]);
              float s[R::HW];
              load_row4<R::HW / 4>(hr + (l * l - 1 + k - NLM) * R::HW, s);
#pragma unroll
              for (int m = 0; m < NP; ++m) {
                const float2 sb = make_float2(s[2 * m], s[2 * m + 1]);
                const float2 sd = make_float2(s[R::HW / 2 + 2 * m], s[R::HW / 2 + 2 * m + 1]);
                p2[m] = fma2(sb, b2, fma2(sd, d2, p2[m]));
                t2[m] = fma2(sd, b2, t2[m]);
              }
            }
          });
#pragma unroll
          for (int m = 0; m < NP; ++m) {
            P[2 * m] = p2[m].x; P[2 * m + 1] = p2[m].y;
            T[2 * m] = t2[m].x; T[2 * m + 1] = t2[m].y;
          }
        }
#pragma unroll
        for (int m = 0; m + 1 < NQ; m += 2)
          *reinterpret_cast<float4*>(row + Q::PR + 2 * m) = make_float4(P[m], T[m], P[m + 1], T[m + 1]);
        if (NQ & 1) *reinterpret_cast<float2*>(row + Q::PR + 2 * (NQ - 1)) = make_float2(P[NQ - 1], T[NQ - 1]);
      }
      __syncwarp();
      if (par < Q::PARS) {
        for (int s = par; s < np; s += Q::PARS) {
          const float* row = rows + s * Q::RS;
          const float2 pr = *reinterpret_cast<const float2*>(row + Q::PR + 2 * on);
          float ff[Q::GW];
          load_row4<Q::GW / 4>(row + og * Q::GW, ff);
          const int c = cls[s];
#pragma unroll
          for (int cc = 0; cc < NS * NS; ++cc)
            if (c == cc) {
#pragma unroll
              for (int k = 0; k < KW; ++k) acc[cc][k] = fmaf(pr.x, ff[2 * k], fmaf(pr.y, ff[2 * k + 1], acc[cc][k]));
            }
        }
      }
      __syncwarp();  // the rows are read before the next chunk (or group) replaces them
    }
    offl = offn;
    typl = typn;
  }
  // fold: the lanes that share outputs, then the block's warps in order
  if constexpr (Q::PARS > 1) {
#pragma unroll
    for (int c = 0; c < NS * NS; ++c)
#pragma unroll
      for (int k = 0; k < KW; ++k) acc[c][k] += __shfl_sync(0xffffffffu, acc[c][k], (lane + Q::NOUT) & 31);
  }
  static_assert(Q::PARS <= 2, "at most two lanes share an output");
  __syncthreads();
  float* red = reinterpret_cast<float*>(smraw);  // [kAngW][c^A]
  if (par == 0) {
#pragma unroll
    for (int c = 0; c < NS * NS; ++c)
#pragma unroll
      for (int k = 0; k < KW; ++k)
        if (og * KW + k < KA) red[warp * C::NCA + (c * NQ + on) * KA + og * KW + k] = acc[c][k];
  }
  __syncthreads();
  for (int q = threadIdx.x; q < C::NCA; q += blockDim.x) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < kAngW; ++w) v += red[w * C::NCA + q];
    cpart[(size_t)blockIdx.x * (C::NCR + C::NCA) + C::NCR + q] = v;
  }
}

// Resident blocks of a warp-per-group kernel on this GPU, after its shared
// memory has been set.
template <class K>
int resident(K kern, size_t smem, int& cap) {
  int per_sm = 0;
  GNEP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  GNEP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
  GNEP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * kAngW, smem));
  if (per_sm < 1) return set_error(GNEP_ERR_CUDA, "angular sweep does not fit on an SM");
  cap = per_sm * sm_count();
  return GNEP_OK;
}
// Resident blocks per kernel (the same value on every model creation).
template <class C>
struct Caps {
  inline static int desc = 0, tangent = 0, force = 0;
};

template <class C>
int grid_for(int N, int cap) {
  const int64_t need = ((int64_t)N + Ang<C>::AW * kAngW - 1) / (Ang<C>::AW * kAngW);
  return (int)(need < cap ? need : cap);
}

}  // namespace

// ------------------------------------------------------------- launchers

int ang_block_atoms(const Shape& s) { return kAngW * (32 / (s.nqa * (s.lmax > 4 ? 2 : 1))); }

template <class C>
int ang_setup() {
  if (int rc = resident(k_ang_desc<C, false>, DescRow<C, false>::smem, Caps<C>::desc)) return rc;
  if (int rc = resident(k_ang_desc<C, true>, DescRow<C, true>::smem, Caps<C>::tangent)) return rc;
  if (int rc = resident(k_ang_force<C>, ForceRow<C>::smem, Caps<C>::force)) return rc;
  int cgrad = 0;  // its grid is cgrad_blocks
  return resident(k_ang_cgrad<C>, CgradRow<C>::smem, cgrad);
}

template <class C>
int ang_descriptors(const gnep_model* m, const gnep_nlist* nl, cudaStream_t st, float* S, float* G) {
  const int N = nl->n_atoms;
  if (N == 0) return GNEP_OK;
  (void)launch_pdl(k_ang_desc<C, false>, grid_for<C>(N, Caps<C>::desc), 32 * kAngW, DescRow<C, false>::smem, st, N,
                   m->dev(), nl->type, nl->atom_struct, nl->L[1].off, nl->L[1].j, nl->L[1].rij,
                   (const float4*)nullptr, (const float*)nullptr, (const float*)nullptr, S, G, (float4*)nullptr);
  GNEP_CHECK_LAUNCH("angular descriptor sweep");
  return GNEP_OK;
}

template <class C>
int ang_tangent(const gnep_model* m, const gnep_nlist* nl, cudaStream_t st, const float4* a, const float* Bs,
                const float* S, float* Sd, float* Gd, float4* wij) {
  const int N = nl->n_atoms;
  if (N == 0) return GNEP_OK;
  (void)launch_pdl(k_ang_desc<C, true>, grid_for<C>(N, Caps<C>::tangent), 32 * kAngW, DescRow<C, true>::smem, st, N,
                   m->dev(), nl->type, nl->atom_struct, nl->L[1].off, nl->L[1].j, nl->L[1].rij, a, Bs, S, Sd, Gd,
                   wij);
  GNEP_CHECK_LAUNCH("angular tangent sweep");
  return GNEP_OK;
}

template <class C>
int ang_force(const gnep_model* m, const gnep_nlist* nl, cudaStream_t st, const float* S, const float* Ep,
              float4* dA) {
  const int N = nl->n_atoms;
  if (N == 0 || nl->L[1].n == 0) return GNEP_OK;
  (void)launch_pdl(k_ang_force<C>, grid_for<C>(N, Caps<C>::force), 32 * kAngW, ForceRow<C>::smem, st, N, m->dev(),
                   nl->type, nl->L[1].off, nl->L[1].rij, S, Ep, dA);
  GNEP_CHECK_LAUNCH("angular force sweep");
  return GNEP_OK;
}

template <class C>
int ang_cgrad(const gnep_model* m, const gnep_nlist* nl, cudaStream_t st, int nb, const float4* wij, const float* S,
              const float* Sd, const float* Gb, const float* Ep, float* cpart) {
  (void)launch_pdl(k_ang_cgrad<C>, nb, 32 * kAngW, CgradRow<C>::smem, st, nl->n_atoms, m->dev(), nl->type,
                   nl->L[1].off, nl->L[1].rij, wij, S, Sd, Gb, Ep, cpart);
  GNEP_CHECK_LAUNCH("angular c-gradient sweep");
  return GNEP_OK;
}

// Model shapes (species, n_max+1, basis+1 radial; same angular; 4-body; l_max).
#define GNEP_ANG(...)                                                                                            \
  template int ang_setup<Sh<__VA_ARGS__>>();                                                                     \
  template int ang_descriptors<Sh<__VA_ARGS__>>(const gnep_model*, const gnep_nlist*, cudaStream_t, float*,      \
                                                float*);                                                         \
  template int ang_tangent<Sh<__VA_ARGS__>>(const gnep_model*, const gnep_nlist*, cudaStream_t, const float4*,   \
                                            const float*, const float*, float*, float*, float4*);                \
  template int ang_force<Sh<__VA_ARGS__>>(const gnep_model*, const gnep_nlist*, cudaStream_t, const float*,      \
                                          const float*, float4*);                                                \
  template int ang_cgrad<Sh<__VA_ARGS__>>(const gnep_model*, const gnep_nlist*, cudaStream_t, int,               \
                                          const float4*, const float*, const float*, const float*,               \
                                          const float*, float*);
GNEP_ANG(2, 5, 9, 5, 9, false, 4)
GNEP_ANG(2, 9, 13, 9, 13, true, 4)
GNEP_ANG(2, 9, 13, 9, 13, false, 4)
GNEP_ANG(2, 5, 9, 5, 9, false, 6)
GNEP_ANG(2, 5, 9, 5, 9, true, 8)
#undef GNEP_ANG

}  // namespace gnep
