// Device arithmetic shared by the angular sweeps: bond geometry, harmonics of
// every degree with their derivatives, packed FP32 arithmetic and the warp's
// group of atoms.
//
// Thread map of the angular sweeps (descriptor, pair force, tangent,
// coefficient gradient).  A warp owns a group of AW consecutive atoms, whose
// pairs are one contiguous range of the CSR list, and works alone: no block
// barrier, no tiles.  It alternates between two mappings through a few KB of
// its own shared memory:
//   pair lanes     one lane per pair: geometry, basis, harmonics, and whatever
//                  contracts an atom's rows with the pair (rows read by 16-byte
//                  loads that the lanes of an atom share);
//   atom lanes     lane (a, n, h) holds channel n of atom a (half h of its
//                  components above degree 4), or a tile of TN channels by eight
//                  components where it sums over the atom's pairs (in registers,
//                  in list order).
// What bounds these sweeps is shared memory: a load returns 128 bytes per cycle
// and SM whether lanes share addresses or not, i.e. one float per lane for every
// four multiply-adds the SM could do.
// All arithmetic is plain FP32 FMA, packed in pairs (fma.rn.f32x2) where two
// neighbouring components take the same operation.  An atom has about eight
// angular pairs, so per-atom tensor-core products would be padded to the
// fragment sizes (9 -> 16 channels, 13 -> 16 basis functions, masks per
// neighbour species, three products per split operand) and spend most
// instructions on splitting and masking operands.
#pragma once
#include <type_traits>

#include "device_math.cuh"
#include "gnep_internal.h"
#include "shape.cuh"

namespace gnep {

constexpr int odd4(int n) { return ((n + 3) / 4) % 2 ? (n + 3) / 4 * 4 : (n + 3) / 4 * 4 + 4; }

// Group shape of a model shape.  Shared rows are an odd number of 16-byte
// words apart, so that eight lanes' 16-byte accesses at one column, and those
// of the group's atoms, fall into different banks.
template <class C>
struct Ang {
  static constexpr int NLX = C::NLX, NQ = C::NQA, KA = C::KA, NS = C::NS;
  static constexpr int SPL = NLX > NLM ? 2 : 1;     // lanes per channel (force and c-gradient rows)
  static constexpr int NQL = NLX / SPL;             // components per channel lane
  static constexpr int LPA = NQ * SPL;              // channel lanes per atom
  static constexpr int AW = 32 / LPA;               // atoms per warp
  static constexpr int CP = AW > 4 ? 64 : 32;       // pairs per chunk (AW atoms have about 8.4 AW pairs)
  // Tile of a summing lane of the descriptor and tangent sweeps: TN channels by
  // 8 components (TN + 8 values read per 8 TN products).
  static constexpr int TN = NQ % 3 == 0 ? 3 : NQ, QG = NLX / 8, TPA = NQ / TN * QG;
  // Coefficient rows [I J]: [n][KM] with the basis functions that fill 16-byte
  // words, then the last one of every channel side by side.
  static constexpr int KM = KA / 4 * 4, CST = odd4(NQ * KM + (NQ + 3) / 4 * 4);
  static_assert(KA % 4 == 1, "one basis function beyond the 16-byte words");
  static_assert(NLX % (4 * SPL) == 0 && NLX % 8 == 0 && NQ % TN == 0 && AW >= 1 && AW * TPA <= 32, "lane maps");
};
constexpr int kAngW = 4;  // warps per block (they share the coefficients only)

// ------------------------------------------------------------- packed FP32

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(d)
      : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)),
        "l"(reinterpret_cast<unsigned long long&>(c)));
  return reinterpret_cast<float2&>(d);
}
__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float2 dup2(float v) { return make_float2(v, v); }

// r = sqrt(d2) and 1 / r from the hardware reciprocal square root, each with
// one Newton step (about half an ulp; the IEEE root and division cost three
// times the instructions).
__device__ __forceinline__ void bond_length(float4 v, float& r, float& ri) {
  const float d2 = fmaf(v.x, v.x, fmaf(v.y, v.y, v.z * v.z));
  const float y = rsqrtf(d2);
  const float s = d2 * y;
  r = fmaf(fmaf(-s, s, d2), 0.5f * y, s);
  ri = fmaf(fmaf(-r, y, 1.f), y, y);
}

// ------------------------------------------------------------- harmonics, l >= 5
//
// q_nl depends only on the addition theorem, not on the basis chosen within
// one l.  Degrees l <= 4 take the printed forms B1-B4 (device_math.cuh), which
// the 4-body term is written in; l = 5..8 take the real regular solid
// harmonics in Racah normalisation (weight C = 1 for m = 0, else 2; components
// of degree l from index l^2 - 1 on: m = 0, then (c, s) for m = 1..l), by
//   R_{l+1,l+1}^c = -sqrt((2l+1)/(2l+2)) (x R_ll^c - y R_ll^s),
//   R_{l+1,l+1}^s = -sqrt((2l+1)/(2l+2)) (y R_ll^c + x R_ll^s),
//   R_{l+1,m} = ((2l+1) z R_lm - sqrt((l+m)(l-m)) r^2 R_{l-1,m}) / sqrt((l+m+1)(l-m+1))
// on the unit vector.  r^2 is formed from its rounded components and not taken as
// 1: the homogeneous polynomial passes their error in |u| on l times, the other
// form up to l (l+1) / 2 times (near the poles; at l_max 8 forces came out 17 %
// further from their FP64 values, energies 11 %).  Their Cartesian gradients are harmonics of degree l - 1
// (with a+ = sqrt((l-m)(l-m-1))/2, a- = sqrt((l+m)(l+m-1))/2,
// az = sqrt((l-m)(l+m)), and c, s of degree l - 1):
//   d/dx R^c = a+ c_{m+1} - a- c_{m-1},  d/dy R^c =  a+ s_{m+1} + a- s_{m-1},  d/dz R^c = az c_m,
//   d/dx R^s = a+ s_{m+1} - a- s_{m-1},  d/dy R^s = -a+ c_{m+1} - a- c_{m-1},  d/dz R^s = az s_m,
// and for m = 0 d/dx R = 2 a+ c_1, d/dy R = 2 a+ s_1: the ladder relations of
// the complex solid harmonics, split into real and imaginary parts.

constexpr double csqrt_(double x) {  // Newton's method, for compile-time constants
  double r = x > 1.0 ? x : 1.0;
  for (int i = 0; i < 60; ++i) r = 0.5 * (r + x / r);
  return x > 0.0 ? r : 0.0;
}
struct Ladder {
  float ap, am, az;
};
constexpr Ladder ladder(int l, int m) {
  return {(float)(0.5 * csqrt_((double)((l - m) * (l - m - 1)))), (float)(0.5 * csqrt_((double)((l + m) * (l + m - 1)))),
          (float)csqrt_((double)((l - m) * (l + m)))};
}

// f(std::integral_constant<int, i>) for i = A..B-1: loops whose index is a
// compile-time constant, so that the factors above are too.
template <int A, int B, class F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (A < B) {
    f(std::integral_constant<int, A>{});
    static_for<A + 1, B>(static_cast<F&&>(f));
  }
}

// One degree: cosine and sine parts, m = 0..l (s[0] = 0).
template <int LMAX>
struct SolidLevel {
  float c[LMAX + 1], s[LMAX + 1];
};

// Runs the recurrence and calls f(integral l, R_l, R_{l-1}) for l = 5..LMAX.
template <int LMAX, class F>
__device__ __forceinline__ void solid_levels(float x, float y, float z, F&& f) {
  const float r2 = fmaf(x, x, fmaf(y, y, z * z));
  SolidLevel<LMAX> a, b;  // degrees l and l - 1
#pragma unroll
  for (int m = 0; m <= LMAX; ++m) a.c[m] = a.s[m] = b.c[m] = b.s[m] = 0.f;
  a.c[0] = 1.f;
  static_for<0, LMAX>([&](auto lc) {
    constexpr int l = decltype(lc)::value;
    SolidLevel<LMAX> n;
#pragma unroll
    for (int m = 0; m <= LMAX; ++m) n.c[m] = n.s[m] = 0.f;
    static_for<0, l + 1>([&](auto mc) {
      constexpr int m = decltype(mc)::value;
      constexpr double d = csqrt_((double)((l + m + 1) * (l - m + 1)));
      constexpr float p = (float)((2.0 * l + 1.0) / d), q = (float)(csqrt_((double)((l + m) * (l - m))) / d);
      const float pz = p * z, qr = q * r2;
      n.c[m] = m < l ? fmaf(pz, a.c[m], -qr * b.c[m]) : pz * a.c[m];
      if (m > 0) n.s[m] = m < l ? fmaf(pz, a.s[m], -qr * b.s[m]) : pz * a.s[m];
    });
    constexpr float e = -(float)csqrt_((2.0 * l + 1.0) / (2.0 * l + 2.0));
    const float ex = e * x, ey = e * y;
    n.c[l + 1] = l == 0 ? ex : fmaf(ex, a.c[l], -ey * a.s[l]);
    n.s[l + 1] = l == 0 ? ey : fmaf(ey, a.c[l], ex * a.s[l]);
    if constexpr (l + 1 >= 5) f(std::integral_constant<int, l + 1>{}, n, a);
    b = a;
    a = n;
  });
}

// Component k = 0..2l of a level.
template <int LMAX>
__device__ __forceinline__ float solid_comp(const SolidLevel<LMAX>& R, int k) {
  return k == 0 ? R.c[0] : (k & 1) ? R.c[(k + 1) / 2] : R.s[k / 2];
}

// w . grad of the components k = 0..2l of degree l, from the level l - 1.
template <int l, int LMAX>
__device__ __forceinline__ void solid_dir(const SolidLevel<LMAX>& L, float wx, float wy, float wz,
                                          float (&D)[2 * l + 1]) {
  float x1[l], x2[l], y1[l], y2[l];
#pragma unroll
  for (int m = 0; m < l; ++m) {
    const float a = wx * L.c[m], b = wx * L.s[m];
    x1[m] = fmaf(wy, L.s[m], a);
    x2[m] = fmaf(-wy, L.s[m], a);
    y1[m] = fmaf(-wy, L.c[m], b);
    y2[m] = fmaf(wy, L.c[m], b);
  }
  static_for<0, l + 1>([&](auto mc) {
    constexpr int m = decltype(mc)::value;
    constexpr Ladder k = ladder(l, m);
    if constexpr (m == 0) {
      D[0] = fmaf(2.f * k.ap, x1[1], k.az * wz * L.c[0]);
    } else {
      float dc = -k.am * x2[m - 1], ds = -k.am * y2[m - 1];
      if constexpr (m < l) {
        dc = fmaf(k.az * wz, L.c[m], dc);
        ds = fmaf(k.az * wz, L.s[m], ds);
      }
      if constexpr (m + 1 < l) {
        dc = fmaf(k.ap, x1[m + 1], dc);
        ds = fmaf(k.ap, y1[m + 1], ds);
      }
      D[2 * m - 1] = dc;
      D[2 * m] = ds;
    }
  });
}

// grad of component k of degree l, from the level l - 1.
template <int l, int k, int LMAX>
__device__ __forceinline__ float3 solid_grad(const SolidLevel<LMAX>& L) {
  constexpr int m = (k + 1) / 2;
  constexpr Ladder a = ladder(l, m);
  if constexpr (k == 0) {
    return make_float3(2.f * a.ap * L.c[1], 2.f * a.ap * L.s[1], a.az * L.c[0]);
  } else if constexpr (k & 1) {
    float3 g = make_float3(-a.am * L.c[m - 1], a.am * L.s[m - 1], 0.f);
    if constexpr (m < l) g.z = a.az * L.c[m];
    if constexpr (m + 1 < l) {
      g.x = fmaf(a.ap, L.c[m + 1], g.x);
      g.y = fmaf(a.ap, L.s[m + 1], g.y);
    }
    return g;
  } else {
    float3 g = make_float3(-a.am * L.s[m - 1], -a.am * L.c[m - 1], 0.f);
    if constexpr (m < l) g.z = a.az * L.s[m];
    if constexpr (m + 1 < l) {
      g.x = fmaf(a.ap, L.s[m + 1], g.x);
      g.y = fmaf(-a.ap, L.c[m + 1], g.y);
    }
    return g;
  }
}

// Weight C and degree of component q (compile-time after unrolling).
__host__ __device__ constexpr int ang_deg(int q) {
  return q < 3 ? 1 : q < 8 ? 2 : q < 15 ? 3 : q < 24 ? 4 : q < 35 ? 5 : q < 48 ? 6 : q < 63 ? 7 : 8;
}
__device__ __forceinline__ float ang_weight(int q) {
  return q < NLM ? kClm[q] : (q == ang_deg(q) * ang_deg(q) - 1 ? 1.f : 2.f);
}

__device__ __forceinline__ float ang_weight_at(int q) {  // the same at run time
  return q < NLM ? kClm[q] : (q == 24 || q == 35 || q == 48 || q == 63) ? 1.f : 2.f;
}

// ------------------------------------------------------------- the warp's group

// c^A_nk^{IJ} into shared rows (see Ang), by the whole block.
template <class C>
__device__ __forceinline__ void load_ang_coef(const DevModel& dm, float* cA) {
  using A = Ang<C>;
  for (int q = threadIdx.x; q < C::NCA; q += blockDim.x) {
    const int k = q % A::KA, r = q / A::KA, n = r % A::NQ, ij = r / A::NQ;
    cA[ij * A::CST + (k < A::KM ? n * A::KM + k : A::NQ * A::KM + n)] = dm.params[dm.off_cA + q];
  }
}

// g[n] = sum_k c_nk f_k for one coefficient row block; with TAN also ga[n] =
// sum_k c_nk fu_k from the same loads.
template <class C, bool TAN>
__device__ __forceinline__ void channel_sums(const float* cIJ, const float (&f)[C::KA], const float (&fu)[C::KA],
                                             float (&g)[C::NQA], float (&ga)[C::NQA]) {
  using A = Ang<C>;
  constexpr int KM = A::KM, NQ = A::NQ;
#pragma unroll
  for (int n = 0; n < NQ; ++n) {
    float2 s = make_float2(0.f, 0.f), u = s;
#pragma unroll
    for (int k = 0; k < KM; k += 4) {
      const float4 c = *reinterpret_cast<const float4*>(cIJ + n * KM + k);
      s = fma2(lo2(c), make_float2(f[k], f[k + 1]), s);
      s = fma2(hi2(c), make_float2(f[k + 2], f[k + 3]), s);
      if (TAN) {
        u = fma2(lo2(c), make_float2(fu[k], fu[k + 1]), u);
        u = fma2(hi2(c), make_float2(fu[k + 2], fu[k + 3]), u);
      }
    }
    g[n] = s.x + s.y;
    if (TAN) ga[n] = u.x + u.y;
  }
#pragma unroll
  for (int n = 0; n < NQ; n += 4) {
    const float4 c = *reinterpret_cast<const float4*>(cIJ + NQ * KM + n);
    const float cv[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (n + e < NQ) {
        g[n + e] = fmaf(cv[e], f[KM], g[n + e]);
        if (TAN) ga[n + e] = fmaf(cv[e], fu[KM], ga[n + e]);
      }
  }
}

// The group's offsets and species, one per lane: lane l holds off[i0 + min(l,
// AW)] (so that lanes beyond the group have empty ranges) and type[i0 + l].
template <class C>
__device__ __forceinline__ void group_fetch(int grp, int N, const int* __restrict__ off, const int* __restrict__ type,
                                            int lane, int& offl, int& typl) {
  constexpr int AW = Ang<C>::AW;
  const int i0 = grp * AW;
  offl = off[min(i0 + min(lane, AW), N)];
  typl = type[min(i0 + min(lane, AW - 1), N - 1)];
}

// Atom slot of pair p in the group, from the lanes' offsets.
template <class C>
__device__ __forceinline__ int pair_slot(int p, int offl) {
  int s = 0;
#pragma unroll
  for (int k = 1; k < Ang<C>::AW; ++k) s += p >= __shfl_sync(0xffffffffu, offl, k);
  return s;
}

__device__ __forceinline__ void load8(const float* p, float (&x)[8]) {
  const float4 u = reinterpret_cast<const float4*>(p)[0], v = reinterpret_cast<const float4*>(p)[1];
  x[0] = u.x; x[1] = u.y; x[2] = u.z; x[3] = u.w; x[4] = v.x; x[5] = v.y; x[6] = v.z; x[7] = v.w;
}
__device__ __forceinline__ void store8(float* p, const float (&x)[8]) {
  reinterpret_cast<float4*>(p)[0] = make_float4(x[0], x[1], x[2], x[3]);
  reinterpret_cast<float4*>(p)[1] = make_float4(x[4], x[5], x[6], x[7]);
}

// The five l = 2 moments (components 3..7) of the tile's rows, held by the lane
// with qg = 0, spread over the lanes qg < TN (row n0 + qg on lane qg).
template <class C>
__device__ __forceinline__ void spread_moments(const float (&x)[Ang<C>::TN][8], int lane, int qg, float (&v)[5]) {
#pragma unroll
  for (int m = 0; m < 5; ++m) {
    v[m] = x[0][3 + m];
#pragma unroll
    for (int j = 1; j < Ang<C>::TN; ++j) {
      const float t = __shfl_sync(0xffffffffu, x[j][3 + m], lane - qg);
      v[m] = qg == j ? t : v[m];
    }
  }
}
}  // namespace gnep
