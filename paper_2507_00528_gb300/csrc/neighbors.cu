// Neighbour sets of Eq. 2: N^i = { (j, n) : |r_j + n.H - r_i| < r_c, (j, n) != (i, 0) }
// over every periodic image n, for the radial (r_c^R) and angular (r_c^A)
// cut-offs, in canonical order (j ascending, then image shift lexicographic).
//
// The accept/reject decision is that of FP64 with explicitly rounded operations
// (no fused multiply-add) in the fixed order
//   s = (na a + nb b) + nc c,  d = (r_j + s) - r_i,  d2 = (dx^2 + dy^2) + dz^2,
// so the list equals that of any plain FP64 evaluation of the same expression.
// FP64 arithmetic is slow on this GPU, so candidates are first measured in
// FP32; only those whose FP32 d2 lies within a relative 2e-3 of a cut-off (far
// above the FP32 error of d2 for coordinates below 10^4 A) take the FP64 test.
// The stored r_ij is formed in float-float arithmetic (about 44 bits) and
// rounded to FP32.
#include <algorithm>
#include <cstdio>
#include <cstring>

#include "gnep_internal.h"

namespace gnep {

namespace {

// Structures with more atoms than this take the binned search, the others
// the all-pairs one (the two give identical lists).
constexpr int kCellMinAtoms = 1024;


// What the host needs to know before the lists are written (one copy back).
struct BuildResult {
  long long tot[2];  // pairs of each list
  int max;           // largest neighbour count (radial)
  int flags;         // k*Bad*, kUnwrapped, kTypesChanged
  int err;           // the model's error flag
};
enum : int { kBadEnds = 1, kBadOrder = 2, kBadType = 4, kUnwrapped = 8, kTypesChanged = 16 };
constexpr int kRefused = kBadEnds | kBadOrder | kBadType | kUnwrapped;

// The terms of a cell H (rows a, b, c) that a build needs: the inverse (FP64, for
// the wrapping check), and along each cell direction tw = rc / w with the plane
// spacing w = V / |b x c| etc., which bounds |df + n| for any pair within rc
// (rounded up by more than its FP32 error), the images needed floor(tw) + 1 and the
// bins of the binned search, floor(2 / tw) (at least 1), reduced until the
// structure has no more bins than atoms.  FP64 products only; the reciprocal of
// the determinant by Newton's iteration from FP32, roots and quotients in FP32:
// FP64 divisions and roots made this 12 us of a small build.
__device__ __forceinline__ void cell_terms(const double* H, double rc, int atoms, double (&inv)[9], int* kr, float* tw,
                                           int* nb) {
  inv[0] = H[4] * H[8] - H[5] * H[7];
  inv[1] = H[2] * H[7] - H[1] * H[8];
  inv[2] = H[1] * H[5] - H[2] * H[4];
  inv[3] = H[5] * H[6] - H[3] * H[8];
  inv[4] = H[0] * H[8] - H[2] * H[6];
  inv[5] = H[2] * H[3] - H[0] * H[5];
  inv[6] = H[3] * H[7] - H[4] * H[6];
  inv[7] = H[1] * H[6] - H[0] * H[7];
  inv[8] = H[0] * H[4] - H[1] * H[3];  // columns: b x c, c x a, a x b
  const double det = H[0] * inv[0] + H[1] * inv[3] + H[2] * inv[6];
  double id = (double)(1.f / (float)det);
  id = id * (2.0 - det * id);
  id = id * (2.0 - det * id);
  int k[3];
  for (int x = 0; x < 3; ++x) {
    const double n2 = inv[x] * inv[x] + inv[3 + x] * inv[3 + x] + inv[6 + x] * inv[6 + x];
    const float s = (float)(n2 * (rc * id) * (rc * id));  // (rc / w)^2
    const float t = sqrtf(s) * (1.f + 4e-6f);
    kr[x] = (int)fminf(floorf(t), 1e6f) + 1;
    tw[x] = t;
    k[x] = (int)fmaxf(1.f, fminf(64.f, floorf(2.f / t)));
  }
  while (k[0] * k[1] * k[2] > atoms) {  // at most 189 steps
    const int x = (k[0] >= k[1] && k[0] >= k[2]) ? 0 : (k[1] >= k[2] ? 1 : 2);
    --k[x];
  }
  for (int x = 0; x < 3; ++x) nb[x] = k[x];
#pragma unroll
  for (int q = 0; q < 9; ++q) inv[q] *= id;
}

// Bin of an atom of a structure in the binned search (from its FP32 fractional
// coordinates; any consistent assignment is valid, since the search visits
// every bin that can hold a neighbour and the lists are sorted afterwards).
__device__ __forceinline__ int atom_bin(float4 f, const int* nb) {
  const int bx = min(nb[0] - 1, max(0, (int)floorf(f.x * (float)nb[0])));
  const int by = min(nb[1] - 1, max(0, (int)floorf(f.y * (float)nb[1])));
  const int bz = min(nb[2] - 1, max(0, (int)floorf(f.z * (float)nb[2])));
  return bx + nb[0] * (by + nb[1] * bz);
}

// Device pointers of the batch being built and of the scratch of one build.
struct BuildArgs {
  int N, S, ns;
  double rc;                    // the larger cut-off
  const int *off, *type;        // the new batch
  const double *pos, *cell;
  const int* old_type;          // species of the last build (NULL: none)
  int *off_c, *type_c;          // the batch's copy, moved into the list at the end (NULL: nothing to move)
  double *pos_c, *cell_c;
  int* atom_struct;             // [N]
  int *kr, *nbin;               // [S][3]
  float *tw, *hsplit;           // [S][3], [S][18] cell as FP32 high and low parts
  float4 *frac, *phi, *plo;     // [N]
  float4* hl;                   // [N][2] the high and low parts side by side (one 32-byte gather)
  int *cnt0, *cnt1;             // [N]
  int *bcount, *bcursor;        // [N] atoms per bin (bins of structure s from its first atom index on)
  int *bstart, *batom;          // [N + S] bin starts within the structure, [N] atoms by bin
  long long* bsum;              // [blocks][2] list sums of each 1,024 atoms
  int *off0, *off1;             // [N + 1]
  BuildResult* res;
  const int* err;
};

// Last s with off[s] <= i, by a whole warp (32 pivots a step).
__device__ __forceinline__ int warp_find(const int* off, int S, int i, int lane) {
  int lo = 0, len = S;
  while (len > 1) {
    const int step = (len + 31) / 32, x = lo + lane * step;
    const unsigned m = __ballot_sync(0xffffffffu, lane * step < len && off[x] <= i);
    const int h = m ? 31 - __clz(m) : 0;
    len = min(step, len - h * step);
    lo += h * step;
  }
  return lo;
}

// The first pass over a batch, a thread per atom: the input checks (offsets,
// species, wrapping), the structure index, the fractional coordinates f = r H^-1
// (FP32; only used to bound image shifts, and checked to lie in [0, 1)), the
// position split into FP32 high and low parts (w of the high part carries the
// species) and the bin counts of structures for the binned search.  The FP64
// cell terms (FP64 is slow on this GPU) are formed once per structure and block,
// by one thread each.  A batch that fails a check leaves flags with which every
// later kernel of the build stops; nothing of the list has been touched by then.
constexpr int kPrep = 128;
__global__ void __launch_bounds__(kPrep) k_prep(BuildArgs A) {
  GNEP_PDL_START();
  __shared__ int so[kPrep + 1], sfl[2], snb[kPrep][3];
  __shared__ double sinv[kPrep][9];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int i0 = blockIdx.x * kPrep, i = i0 + tid, il = min(i0 + kPrep, A.N) - 1;
  int bad = 0;
  for (int s = i; s < A.S; s += gridDim.x * kPrep) {
    if (A.off[s + 1] <= A.off[s]) bad |= kBadOrder;
    if ((s == 0 && A.off[0] != 0) || (s == A.S - 1 && A.off[A.S] != A.N)) bad |= kBadEnds;
    if (A.off_c) {
      A.off_c[s] = A.off[s];
      if (s == A.S - 1) A.off_c[A.S] = A.off[A.S];
      for (int q = 0; q < 9; ++q) A.cell_c[9 * (size_t)s + q] = A.cell[9 * (size_t)s + q];
    }
  }
  // this atom's inputs, read beside the structures' terms
  const int ic = min(i, A.N - 1);
  const int t = A.type[ic];
  const double* p = A.pos + 3 * (size_t)ic;
  const double px = p[0], py = p[1], pz = p[2];
  const int told = A.old_type ? A.old_type[ic] : -1;
  if (warp < 2) {
    const int s = warp_find(A.off, A.S, warp ? il : i0, lane);
    if (lane == 0) sfl[warp] = s;
  }
  __syncthreads();
  const int s0 = sfl[0], ns = max(1, min(sfl[1] - s0 + 1, kPrep));  // more only with offsets that do not increase
  for (int k = tid; k <= ns; k += kPrep) so[k] = A.off[min(s0 + k, A.S)];
  __syncthreads();
  if (tid < ns) {
    const int s = s0 + tid, a0 = so[tid], a1 = so[tid + 1];
    const double* H = A.cell + 9 * (size_t)s;
    int kr[3];
    float tw[3];
    cell_terms(H, A.rc, max(1, a1 - a0), sinv[tid], kr, tw, snb[tid]);
    if (a0 >= i0) {  // the block with the structure's first atom writes its terms
      for (int x = 0; x < 3; ++x) {
        A.kr[3 * s + x] = kr[x];
        A.tw[3 * s + x] = tw[x];
        A.nbin[3 * s + x] = snb[tid][x];
      }
      for (int q = 0; q < 9; ++q) {
        const float h = (float)H[q];
        A.hsplit[18 * s + q] = h;
        A.hsplit[18 * s + 9 + q] = (float)(H[q] - (double)h);
      }
    }
  }
  __syncthreads();
  if (i < A.N) {
    if (t < 0 || t >= A.ns) bad |= kBadType;
    if (t != told) bad |= kTypesChanged;
    int lo = 0, hi = ns - 1;
    while (lo < hi) {  // last k with so[k] <= i
      const int mid = (lo + hi + 1) >> 1;
      if (so[mid] <= i) lo = mid; else hi = mid - 1;
    }
    const int s = s0 + lo, a0 = so[lo], a1 = so[lo + 1];
    if (a0 < 0 || a0 > i || a1 <= i || a1 > A.N) {
      bad |= kBadOrder;
    } else {
      if (A.off_c) {
        A.type_c[i] = t;
        A.pos_c[3 * (size_t)i] = px;
        A.pos_c[3 * (size_t)i + 1] = py;
        A.pos_c[3 * (size_t)i + 2] = pz;
      }
      const double* inv = sinv[lo];
      double f[3];
      bool wrapped = true;
      for (int x = 0; x < 3; ++x) {
        f[x] = px * inv[x] + py * inv[3 + x] + pz * inv[6 + x];
        wrapped = wrapped && f[x] > -1e-9 && f[x] < 1.0 + 1e-9;
      }
      if (!wrapped) bad |= kUnwrapped;
      A.atom_struct[i] = s;
      const float4 fr = make_float4((float)f[0], (float)f[1], (float)f[2], 0.f);
      A.frac[i] = fr;
      const float hx = (float)px, hy = (float)py, hz = (float)pz;
      const float4 h = make_float4(hx, hy, hz, (float)t);
      const float4 l = make_float4((float)(px - (double)hx), (float)(py - (double)hy), (float)(pz - (double)hz), 0.f);
      A.phi[i] = h;
      A.plo[i] = l;
      A.hl[2 * (size_t)i] = h;
      A.hl[2 * (size_t)i + 1] = l;
      if (a1 - a0 > kCellMinAtoms && wrapped) atomicAdd(&A.bcount[a0 + atom_bin(fr, snb[lo])], 1);
    }
  }
  if (bad) atomicOr(&A.res->flags, bad);
}

// Bin starts and the atoms by bin of one structure above kCellMinAtoms atoms, one
// block each (the order inside a bin is free: it only sets the order in which
// candidates are tested).
__global__ void __launch_bounds__(1024) k_bins(BuildArgs A) {
  GNEP_PDL_START();
  const int s = blockIdx.x;
  if (A.res->flags & kRefused) return;
  const int a0 = A.off[s], n = A.off[s + 1] - a0;
  if (n <= kCellMinAtoms) return;
  const int* nb = A.nbin + 3 * s;
  const int nbins = nb[0] * nb[1] * nb[2];
  __shared__ int wsum[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int* start = A.bstart + a0 + s;
  int base = 0;  // atoms in the bins of earlier rounds (every thread keeps it)
  for (int b0 = 0; b0 < nbins; b0 += 1024) {
    const int b = b0 + threadIdx.x, c = b < nbins ? A.bcount[a0 + b] : 0;
    int v = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += u;
    }
    if (lane == 31) wsum[warp] = v;
    __syncthreads();
    if (warp == 0) {
      int w = wsum[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, w, o);
        if (lane >= o) w += u;
      }
      wsum[lane] = w;
    }
    __syncthreads();
    if (b < nbins) start[b] = base + (warp ? wsum[warp - 1] : 0) + v - c;
    base += wsum[31];
    __syncthreads();  // the sums are read before the next round replaces them
  }
  if (threadIdx.x == 0) start[nbins] = n;
  for (int i = a0 + threadIdx.x; i < a0 + n; i += 1024) {
    const int b = atom_bin(A.frac[i], nb);
    A.batom[a0 + start[b] + atomicAdd(&A.bcursor[a0 + b], 1)] = i;
  }
}

// Error-free transformations for float-float arithmetic.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}
__device__ __forceinline__ void two_prod(float a, float b, float& p, float& e) {
  p = a * b;
  e = fmaf(a, b, -p);
}

// r_j + n.H - r_i in float-float (about 44 significant bits), rounded to FP32.
__device__ __forceinline__ float pair_component(float pjh, float pjl, float pih, float pil, int na, int nb, int nc,
                                                float ah, float al, float bh, float bl, float ch, float cl) {
  float h, e, t, u;
  two_sum(pjh, -pih, h, e);
  float lo = e + (pjl - pil);
  two_prod((float)na, ah, t, u);
  lo += u + (float)na * al;
  two_sum(h, t, h, e);
  lo += e;
  two_prod((float)nb, bh, t, u);
  lo += u + (float)nb * bl;
  two_sum(h, t, h, e);
  lo += e;
  two_prod((float)nc, ch, t, u);
  lo += u + (float)nc * cl;
  two_sum(h, t, h, e);
  lo += e;
  return h + lo;
}

__device__ __forceinline__ double pair_d2_exact(const double* H, const double* pi, const double* pj,
                                                int na, int nb, int nc, double d[3]) {
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    const double s = __dadd_rn(__dadd_rn(__dmul_rn((double)na, H[x]), __dmul_rn((double)nb, H[3 + x])),
                               __dmul_rn((double)nc, H[6 + x]));
    d[x] = __dsub_rn(__dadd_rn(pj[x], s), pi[x]);
  }
  return __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2]));
}

struct ListParams {
  double rc2[2];     // exact squared cut-offs (radial, angular)
  float lo2[2];      // FP32 d2 below: inside (FP32 decision)
  float hi2[2];      // FP32 d2 above: outside (FP32 decision)
  float reject2;     // max(hi2): candidates above it are outside both
};

// The list decisions for neighbour j of atom i at image n (na, nb, nc) of
// structure s: FP32 away from the cut-offs, the exact FP64 expression within
// the band.  dj = phi_j - phi_i (high parts), Hh the FP32 high parts of the
// cell.  Both searches (all pairs, binned) take their decisions here.
template <class T>
__device__ __forceinline__ void decide_pair(int i, int j, T na, T nb, T nc, const float (&dj)[3],
                                            const float (&Hh)[9], const ListParams& lp,
                                            const double* __restrict__ cell, const double* __restrict__ pos, int s,
                                            bool& in0, bool& in1) {
  in0 = in1 = false;
  if (j == i && na == T(0) && nb == T(0) && nc == T(0)) return;
  const float fx = dj[0] + ((float)na * Hh[0] + (float)nb * Hh[3] + (float)nc * Hh[6]);
  const float fy = dj[1] + ((float)na * Hh[1] + (float)nb * Hh[4] + (float)nc * Hh[7]);
  const float fz = dj[2] + ((float)na * Hh[2] + (float)nb * Hh[5] + (float)nc * Hh[8]);
  const float d2f = fx * fx + fy * fy + fz * fz;
  if (d2f > lp.reject2) return;
  in0 = d2f < lp.lo2[0];
  in1 = d2f < lp.lo2[1];
  const bool band0 = !in0 && d2f <= lp.hi2[0], band1 = !in1 && d2f <= lp.hi2[1];
  if (band0 || band1) {  // near a cut-off: the FP64 decision
    const double* Hd = cell + 9 * s;
    const double H[9] = {Hd[0], Hd[1], Hd[2], Hd[3], Hd[4], Hd[5], Hd[6], Hd[7], Hd[8]};
    const double pi[3] = {pos[3 * (size_t)i], pos[3 * (size_t)i + 1], pos[3 * (size_t)i + 2]};
    const double pj[3] = {pos[3 * (size_t)j], pos[3 * (size_t)j + 1], pos[3 * (size_t)j + 2]};
    double d[3];
    const double d2 = pair_d2_exact(H, pi, pj, (int)na, (int)nb, (int)nc, d);
    if (band0) in0 = d2 < lp.rc2[0];
    if (band1) in1 = d2 < lp.rc2[1];
  }
}

// Per-atom slots of the search: the first cap entries of atom i's radial list go
// to e[i cap + k] as (j, image and a flag: the entry is in the angular list too,
// which holds the radial entries below the smaller cut-off in the same order);
// k_compact moves them into the CSR lists once the counts are scanned.
struct Slots {
  int cap;
  int2* e;
};
__device__ __forceinline__ int2 slot_entry(int j, int na, int nb, int nc, bool ang) {
  return make_int2(j, (na & 255) | (nb & 255) << 8 | (nc & 255) << 16 | (ang ? 1 << 24 : 0));
}

// One warp per central atom i.  Lane l tests the neighbours j = a0 + l,
// a0 + l + 32, ...: in each round of 32 consecutive j every lane walks the
// images of its j in lexicographic order, and the warp places the accepted
// entries by an exclusive scan of the per-lane counts, so each list comes out
// in canonical order (j ascending, then image), written into the CSR lists at
// the offsets that the slot pass counted: the writing pass of a batch in which
// some atom has more entries than its slots hold.  It takes the slot passes'
// decisions (FP32 away from the cut-offs, FP64 within the band).  A lane
// keeps up to kBuf accepted images of its j in a packed register; a round in
// which some lane accepts more walks the images again to place them.
constexpr int kBuf = 4;

__global__ void __launch_bounds__(128) k_pairs(
    int N, const int* __restrict__ struct_off, const int* __restrict__ atom_struct,
    const double* __restrict__ pos, const double* __restrict__ cell, const int* __restrict__ krange,
    const float* __restrict__ tw, const float* __restrict__ hsplit, const float4* __restrict__ frac,
    const float4* __restrict__ phi, const float4* __restrict__ plo, ListParams lp,
    const int* __restrict__ off0, const int* __restrict__ off1, int* __restrict__ j0,
    float4* __restrict__ r0, char4* __restrict__ sh0, int* __restrict__ j1,
    int* __restrict__ own1, float4* __restrict__ r1, char4* __restrict__ sh1) {
  const int i = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= N) return;  // the whole warp
  const int s = atom_struct[i];
  const int a0 = struct_off[s], a1 = struct_off[s + 1];
  float Hh[9], Hl[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    Hh[q] = hsplit[18 * s + q];
    Hl[q] = hsplit[18 * s + 9 + q];
  }
  const float4 pih = phi[i], pil = plo[i];
  const int ka = krange[3 * s], kb = krange[3 * s + 1], kc = krange[3 * s + 2];
  const bool packable = ka <= 7 && kb <= 7 && kc <= 7;  // image indices fit 4 bits
  // |r_j + n.H - r_i| >= |df_x + n_x| w_x, so only shifts with |df_x + n_x| < rc / w_x
  // (with a margin far above FP32 rounding) can pass the test below.
  const float4 fi = frac[i];
  const float t0 = tw[3 * s] + 1e-3f, t1 = tw[3 * s + 1] + 1e-3f, t2 = tw[3 * s + 2] + 1e-3f;
  int base0 = 0, base1 = 0;
  for (int jb = a0; jb < a1; jb += 32) {
    const int j = jb + lane;
    const bool vj = j < a1;
    const float4 pjh = vj ? phi[j] : pih;
    const float4 fj = vj ? frac[j] : fi;
    const float dj[3] = {pjh.x - pih.x, pjh.y - pih.y, pjh.z - pih.z};
    const float dfa = fj.x - fi.x, dfb = fj.y - fi.y, dfc = fj.z - fi.z;
    const int alo = max(-ka, (int)ceilf(-t0 - dfa)), ahi = vj ? min(ka, (int)floorf(t0 - dfa)) : alo - 1;
    const int blo = max(-kb, (int)ceilf(-t1 - dfb)), bhi = min(kb, (int)floorf(t1 - dfb));
    const int clo = max(-kc, (int)ceilf(-t2 - dfc)), chi = min(kc, (int)floorf(t2 - dfc));
    // the list decisions for image n of this lane's j
    auto decide = [&](int na, int nb, int nc, bool& in0, bool& in1) {
      decide_pair(i, j, na, nb, nc, dj, Hh, lp, cell, pos, s, in0, in1);
    };
    // places one accepted entry at the next positions of its lists
    auto put = [&](int na, int nb, int nc, bool in0, bool in1, int& w0, int& w1) {
      const char4 sv = make_char4((signed char)na, (signed char)nb, (signed char)nc, 0);
      const float4 pjl = plo[j];
      const float rx = pair_component(pjh.x, pjl.x, pih.x, pil.x, na, nb, nc, Hh[0], Hl[0], Hh[3], Hl[3], Hh[6], Hl[6]);
      const float ry = pair_component(pjh.y, pjl.y, pih.y, pil.y, na, nb, nc, Hh[1], Hl[1], Hh[4], Hl[4], Hh[7], Hl[7]);
      const float rz = pair_component(pjh.z, pjl.z, pih.z, pil.z, na, nb, nc, Hh[2], Hl[2], Hh[5], Hl[5], Hh[8], Hl[8]);
      const float4 rv = make_float4(rx, ry, rz, pjh.w);
      if (in0) { const int d = off0[i] + w0; j0[d] = j; r0[d] = rv; sh0[d] = sv; }
      if (in1) { const int d = off1[i] + w1; j1[d] = j; own1[d] = i; r1[d] = rv; sh1[d] = sv; }
      w0 += in0;
      w1 += in1;
    };
    int n0 = 0, n1 = 0, nacc = 0;
    unsigned long long buf = 0;
    for (int na = alo; na <= ahi; ++na)
      for (int nb = blo; nb <= bhi; ++nb)
        for (int nc = clo; nc <= chi; ++nc) {
          bool in0, in1;
          decide(na, nb, nc, in0, in1);
          if (!in0 && !in1) continue;
          if (packable && nacc < kBuf)
            buf |= (unsigned long long)((na + 8) | (nb + 8) << 4 | (nc + 8) << 8 | (int)in0 << 12 | (int)in1 << 13)
                   << (16 * nacc);
          ++nacc;
          n0 += in0;
          n1 += in1;
        }
    int p0 = n0, p1 = n1;  // inclusive scan over the lanes (j order)
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u0 = __shfl_up_sync(0xffffffffu, p0, o), u1 = __shfl_up_sync(0xffffffffu, p1, o);
      if (lane >= o) {
        p0 += u0;
        p1 += u1;
      }
    }
    const int tot0 = __shfl_sync(0xffffffffu, p0, 31), tot1 = __shfl_sync(0xffffffffu, p1, 31);
    int w0 = base0 + p0 - n0, w1 = base1 + p1 - n1;
    if (!__any_sync(0xffffffffu, nacc > kBuf || (nacc > 0 && !packable))) {
      for (int e = 0; e < nacc; ++e) {
        const int v = (int)((buf >> (16 * e)) & 0xffffu);
        put((v & 15) - 8, ((v >> 4) & 15) - 8, ((v >> 8) & 15) - 8, (v >> 12) & 1, (v >> 13) & 1, w0, w1);
      }
    } else {  // walk the images again, placing each accepted one
      for (int na = alo; na <= ahi; ++na)
        for (int nb = blo; nb <= bhi; ++nb)
          for (int nc = clo; nc <= chi; ++nc) {
            bool in0, in1;
            decide(na, nb, nc, in0, in1);
            if (in0 || in1) put(na, nb, nc, in0, in1, w0, w1);
          }
    }
    base0 += tot0;
    base1 += tot1;
  }
}

// The slot pass for structures of at most kCellMinAtoms atoms, one warp per
// central atom i, with the candidates flattened: in each round of kFlatJ = 64
// consecutive j (two per lane) the lanes count the images their j may have
// within the cut-offs (the fractional bounds of k_pairs), a warp scan lays
// those (j, image) candidates out in canonical order (j ascending, then image
// lexicographic) and the lanes then take them 32 at a time, so that every lane
// tests a candidate in every step instead of walking its own j's images while
// the others wait.  The round's per-j bounds and scan sit in the warp's shared
// memory; each lane finds its candidate's j by a binary search over the scan.
// Accepted entries are placed by ballots in the same canonical order (counts
// exact; the first cap entries of each list go to the atom's slots).  Two j per
// lane fill about half of the candidate steps' lanes on cells of the
// 32-400-atom workload, where one j per lane filled under a third.
constexpr int kFlatWarps = 4, kFlatJ = 64;

struct FlatSmem {  // per warp and round: dj = phi_j - phi_i, (alo, blo, clo, j), (nb count, nc count,
                   // candidates before this j) and the inclusive candidate counts
  float4 sdj[kFlatJ];
  int4 slo[kFlatJ];
  int4 scnt[kFlatJ];
  int sincl[kFlatJ];
};

__device__ __forceinline__ void pairs_flat(const BuildArgs& A, const ListParams& lp, const Slots& sl, int i, int s,
                                           int lane, FlatSmem& sm) {
  const int a0 = A.off[s], a1 = A.off[s + 1];
  float Hh[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) Hh[q] = A.hsplit[18 * s + q];
  const float4 pih = A.phi[i];
  const int ka = A.kr[3 * s], kb = A.kr[3 * s + 1], kc = A.kr[3 * s + 2];
  const float4 fi = A.frac[i];
  const float t0 = A.tw[3 * s] + 1e-3f, t1 = A.tw[3 * s + 1] + 1e-3f, t2 = A.tw[3 * s + 2] + 1e-3f;
  const unsigned lt = (1u << lane) - 1u;
  int w0 = 0, w1 = 0;  // entries of each list so far (warp-uniform)
  for (int jb = a0; jb < a1; jb += kFlatJ) {
    int base = 0;  // candidates of the round's first half (after its scan)
#pragma unroll
    for (int h = 0; h < 2; ++h) {  // j = jb + 32 h + lane at position 32 h + lane
      const int j = jb + 32 * h + lane;
      const bool vj = j < a1;
      const float4 pjh = vj ? A.phi[j] : pih;
      const float4 fj = vj ? A.frac[j] : fi;
      const float dfa = fj.x - fi.x, dfb = fj.y - fi.y, dfc = fj.z - fi.z;
      const int alo = max(-ka, (int)ceilf(-t0 - dfa)), ahi = vj ? min(ka, (int)floorf(t0 - dfa)) : alo - 1;
      const int blo = max(-kb, (int)ceilf(-t1 - dfb)), bhi = min(kb, (int)floorf(t1 - dfb));
      const int clo = max(-kc, (int)ceilf(-t2 - dfc)), chi = min(kc, (int)floorf(t2 - dfc));
      const int nbc = max(0, bhi - blo + 1), ncc = max(0, chi - clo + 1);
      const int ncand = max(0, ahi - alo + 1) * nbc * ncc;  // this j's candidate images
      int incl = ncand;  // inclusive scan over the lanes
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
      }
      incl += base;
      const int x = 32 * h + lane;
      sm.sdj[x] = make_float4(pjh.x - pih.x, pjh.y - pih.y, pjh.z - pih.z, 0.f);
      sm.slo[x] = make_int4(alo, blo, clo, j);
      sm.scnt[x] = make_int4(nbc, ncc, incl - ncand, 0);
      sm.sincl[x] = incl;
      base = __shfl_sync(0xffffffffu, incl, 31);
    }
    __syncwarp();
    const int total = base;
    for (int cb = 0; cb < total; cb += 32) {
      const int c = cb + lane;
      const bool valid = c < total;
      int L = 0;  // the position whose j owns candidate c: incl[L - 1] <= c < incl[L] (at most 63)
#pragma unroll
      for (int st = kFlatJ / 2; st >= 1; st >>= 1)
        if (sm.sincl[L + st - 1] <= c) L += st;
      bool in0 = false, in1 = false;
      int na = 0, nb = 0, nc = 0, oj = 0;
      if (valid) {  // image m of the owner's (na, nb, nc) ranges, nc fastest (a few steps: no division)
        const float4 d4 = sm.sdj[L];
        const int4 lo = sm.slo[L], cn = sm.scnt[L];
        const float odj[3] = {d4.x, d4.y, d4.z};
        oj = lo.w;
        int r = c - cn.z;
        const int bc = cn.x * cn.y;
        na = lo.x;
        while (r >= bc) {
          r -= bc;
          ++na;
        }
        nb = lo.y;
        while (r >= cn.y) {
          r -= cn.y;
          ++nb;
        }
        nc = lo.z + r;
        decide_pair(i, oj, na, nb, nc, odj, Hh, lp, A.cell, A.pos, s, in0, in1);
      }
      const unsigned b0 = __ballot_sync(0xffffffffu, in0), b1 = __ballot_sync(0xffffffffu, in1);
      const int w = w0 + __popc(b0 & lt);
      if (in0 && w < sl.cap) sl.e[(size_t)i * sl.cap + w] = slot_entry(oj, na, nb, nc, in1);
      w0 += __popc(b0);
      w1 += __popc(b1);
    }
    __syncwarp();  // the round's shared entries are read before the next round writes them
  }
  if (lane == 0) {
    A.cnt0[i] = w0;
    A.cnt1[i] = w1;
  }
}

// Binned search, one warp per central atom i (the slot pass) of the
// structures above kCellMinAtoms atoms; the smaller ones take the all-pairs
// search (pairs_flat), which is as fast there: at cell widths below 3 r_c the
// visited bins cover about the whole cell.  The bins of structure s split its
// cell into nbin[s] parts along each cell direction; every (j, n) within r_c of
// i has f_j + n inside (f_i - t, f_i + t) along each direction (t = r_c / w_x,
// with a margin), i.e. in one of the extended bins floor((f_i - t) nbin) ..
// floor((f_i + t) nbin), so the warp visits those bins (lane per bin; extended
// bin B holds the atoms of bin B mod nbin at the image floor(B / nbin)) and
// tests their atoms with the same decision as the all-pairs search.  Accepted
// entries collect in shared memory as keys (j, image, lists); each entry's
// position in each list is its rank among the list's entries in canonical
// order (j ascending, then image lexicographic), so the slots hold exactly the
// lists of the all-pairs search.  Counts are exact even when an atom overflows
// its slots (the writing pass then takes the batch).
constexpr int kCellBuf = 160;  // accepted entries a warp ranks per atom

__device__ __forceinline__ int floor_div(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

struct CellSmem {
  unsigned long long key[kCellBuf];
  int nacc, nang;
};

__device__ __forceinline__ void pairs_cell(const BuildArgs& A, const ListParams& lp, const Slots& sl, int i, int s,
                                           int lane, CellSmem& sm) {
  const int a0 = A.off[s];
  if (lane == 0) {
    sm.nacc = sm.nang = 0;
  }
  __syncwarp();
  const int* bstart = A.bstart + a0 + s;
  const int* batom = A.batom + a0;
  float Hh[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) Hh[q] = A.hsplit[18 * s + q];
  const float4 pih = A.phi[i], fi = A.frac[i];
  const float f[3] = {fi.x, fi.y, fi.z};
  int nb[3], lo[3], cnt[3];
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    nb[x] = A.nbin[3 * s + x];
    const float t = A.tw[3 * s + x] + 2e-3f;
    lo[x] = (int)floorf((f[x] - t) * (float)nb[x]);
    cnt[x] = (int)floorf((f[x] + t) * (float)nb[x]) - lo[x] + 1;
  }
  const int NB = cnt[0] * cnt[1] * cnt[2];
  for (int e = lane; e < NB; e += 32) {
    const int B[3] = {lo[0] + e % cnt[0], lo[1] + (e / cnt[0]) % cnt[1], lo[2] + e / (cnt[0] * cnt[1])};
    int n[3], bx[3];
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      n[x] = floor_div(B[x], nb[x]);
      bx[x] = B[x] - n[x] * nb[x];
    }
    const int bin = bx[0] + nb[0] * (bx[1] + nb[1] * bx[2]);
    const int q0 = bstart[bin], q1 = bstart[bin + 1];
    for (int q = q0; q < q1; ++q) {
      const int j = batom[q];
      const float4 pjh = A.phi[j];
      const float dj[3] = {pjh.x - pih.x, pjh.y - pih.y, pjh.z - pih.z};
      bool in0, in1;
      decide_pair(i, j, n[0], n[1], n[2], dj, Hh, lp, A.cell, A.pos, s, in0, in1);
      if (!in0) continue;
      if (in1) atomicAdd(&sm.nang, 1);
      const int slot = atomicAdd(&sm.nacc, 1);
      if (slot < kCellBuf)
        sm.key[slot] = ((unsigned long long)j << 25) | ((unsigned long long)(n[0] + 128) << 17) |
                       ((unsigned long long)(n[1] + 128) << 9) | ((unsigned long long)(n[2] + 128) << 1) |
                       (unsigned long long)in1;
    }
  }
  __syncwarp();
  const int M = sm.nacc, c0 = M, c1 = sm.nang;
  if (lane == 0) {
    A.cnt0[i] = c0;
    A.cnt1[i] = c1;
  }
  if (M <= kCellBuf && c0 <= sl.cap) {  // else the writing pass takes the batch
    for (int e = lane; e < M; e += 32) {
      const unsigned long long ke = sm.key[e];
      int r = 0;
      for (int e2 = 0; e2 < M; ++e2) r += sm.key[e2] < ke;  // keys are distinct: ranks are positions
      sl.e[(size_t)i * sl.cap + r] =
          slot_entry((int)(ke >> 25), (int)((ke >> 17) & 255ull) - 128, (int)((ke >> 9) & 255ull) - 128,
                     (int)((ke >> 1) & 255ull) - 128, ke & 1ull);
    }
  }
}

// The search in cells at least 2 r_c wide along every direction (t = r_c / w < 1/2):
// a neighbour has one image that can be within r_c, n = -round(f_j - f_i), so each
// lane tests its j there, two j per lane and round, with the decision of the other
// searches.  Most structures of training batches are such cells; laying their
// (j, image) candidates out as for narrower cells took half as long again (256
// structures of 32-400 atoms: k_pairs_slots 130 us, now 93; 57 % of the issue slots,
// the rest waits on the loads of phi and frac).
__device__ __forceinline__ void pairs_min(const BuildArgs& A, const ListParams& lp, const Slots& sl, int i, int s,
                                          int lane) {
  const int a0 = A.off[s], a1 = A.off[s + 1];
  const float4* __restrict__ phi = A.phi;
  const float4* __restrict__ frac = A.frac;
  float Hh[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) Hh[q] = A.hsplit[18 * s + q];
  const float4 pih = phi[i], fi = frac[i];
  const unsigned lt = (1u << lane) - 1u;
  int2* __restrict__ out = sl.e + (size_t)i * sl.cap;
  int w0 = 0, w1 = 0;
  for (int jb = a0; jb < a1; jb += 64) {
    float4 ph[2], fr[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int j = min(jb + 32 * u + lane, a1 - 1);
      ph[u] = phi[j];
      fr[u] = frac[j];
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int j = jb + 32 * u + lane;
      const float na = -rintf(fr[u].x - fi.x), nb = -rintf(fr[u].y - fi.y), nc = -rintf(fr[u].z - fi.z);
      const float dj[3] = {ph[u].x - pih.x, ph[u].y - pih.y, ph[u].z - pih.z};
      bool in0 = false, in1 = false;
      if (j < a1 && j != i) decide_pair(i, j, na, nb, nc, dj, Hh, lp, A.cell, A.pos, s, in0, in1);
      const unsigned b0 = __ballot_sync(0xffffffffu, in0), b1 = __ballot_sync(0xffffffffu, in1);
      const int w = w0 + __popc(b0 & lt);
      if (in0 && w < sl.cap) out[w] = slot_entry(j, (int)na, (int)nb, (int)nc, in1);
      w0 += __popc(b0);
      w1 += __popc(b1);
    }
  }
  if (lane == 0) {
    A.cnt0[i] = w0;
    A.cnt1[i] = w1;
  }
}

// The search, one warp per central atom: binned in structures above kCellMinAtoms
// atoms, over all pairs in the others (at one image each in wide cells).
union PairSmem {
  FlatSmem flat;
  CellSmem cell;
};
__global__ void __launch_bounds__(32 * kFlatWarps, 8) k_pairs_slots(BuildArgs A, ListParams lp, Slots sl) {
  GNEP_PDL_START();
  __shared__ PairSmem sm[kFlatWarps];
  if (A.res->flags & kRefused) return;
  const int i = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (i >= A.N) return;  // the whole warp
  const int s = A.atom_struct[i];
  constexpr float kHalf = 0.498f;  // 1/2 less the FP32 error of tw and of the fractional coordinates
  if (A.off[s + 1] - A.off[s] > kCellMinAtoms)
    pairs_cell(A, lp, sl, i, s, lane, sm[w].cell);
  else if (A.tw[3 * s] < kHalf && A.tw[3 * s + 1] < kHalf && A.tw[3 * s + 2] < kHalf)
    pairs_min(A, lp, sl, i, s, lane);
  else
    pairs_flat(A, lp, sl, i, s, lane, sm[w].flat);
}

// The list's own arrays, written once the counts are known.
struct ListOut {
  int *struct_off, *type, *atom_struct;
  double *pos, *cell;
  int *offr, *offa;
  int *j0, *j1, *own1;
  float4 *r0, *r1;
  char4 *sh0, *sh1;
};

// The batch and the offsets into the list: atom i's entries by one warp, and
// structure i's.
__device__ __forceinline__ void commit_batch(const BuildArgs& A, const ListOut& O, int i, int lane) {
  if (lane == 0) {
    O.atom_struct[i] = A.atom_struct[i];
    if (A.off_c) O.type[i] = A.type_c[i];
  }
  if (lane < 2) {
    int* off = lane ? O.offa : O.offr;
    const int* src = lane ? A.off1 : A.off0;
    off[i] = src[i];
    if (i == A.N - 1) off[A.N] = src[A.N];
  }
  if (!A.off_c) return;
  if (lane >= 4 && lane < 7) O.pos[3 * (size_t)i + lane - 4] = A.pos_c[3 * (size_t)i + lane - 4];
  if (i < A.S && lane >= 8 && lane < 17) O.cell[9 * (size_t)i + lane - 8] = A.cell_c[9 * (size_t)i + lane - 8];
  if (i < A.S && lane == 20) {
    O.struct_off[i] = A.off_c[i];
    if (i == A.S - 1) O.struct_off[A.S] = A.off_c[A.S];
  }
}

// One 32-byte load (sm_100 and later).
__device__ __forceinline__ void load_hl(const float4* p, float4& h, float4& l) {
  asm("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
      : "=f"(h.x), "=f"(h.y), "=f"(h.z), "=f"(h.w), "=f"(l.x), "=f"(l.y), "=f"(l.z), "=f"(l.w)
      : "l"(p));
}

// Moves the per-atom slots into the CSR lists and forms r_ij, one warp per atom:
// the atom's cell, position and offsets are read once per warp, and the lanes
// take its radial entries, two each so that two rounds of gathered loads
// overlap; an entry of the angular list is written there too, at its rank among
// them.  It also moves the checked batch into the list.
__global__ void __launch_bounds__(256) k_compact(BuildArgs A, Slots sl, ListOut O) {
  const int i = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= A.N) return;  // the whole warp
  const int n0 = A.cnt0[i];  // at most the slots (the writing pass takes the batch otherwise)
  const int d0 = A.off0[i];
  int d1 = A.off1[i];
  const int2* __restrict__ slot = sl.e + (size_t)i * sl.cap;
  const float hv = A.hsplit[18 * A.atom_struct[i] + min(lane, 17)];
  float4 pih, pil;
  load_hl(A.hl + 2 * (size_t)i, pih, pil);
  float H[18];
#pragma unroll
  for (int q = 0; q < 18; ++q) H[q] = __shfl_sync(0xffffffffu, hv, q);
  const unsigned lt = (1u << lane) - 1u;
  for (int b = 0; b < n0; b += 64) {
    int2 en[2];
    float4 ph[2], pl[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) en[u] = slot[min(b + 32 * u + lane, n0 - 1)];
#pragma unroll
    for (int u = 0; u < 2; ++u) load_hl(A.hl + 2 * (size_t)en[u].x, ph[u], pl[u]);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int e = b + 32 * u + lane;
      const bool in = e < n0, ang = in && (en[u].y >> 24);
      const int na = (signed char)en[u].y, nb = (signed char)(en[u].y >> 8), nc = (signed char)(en[u].y >> 16);
      const float4 h = ph[u], l = pl[u];
      const float4 r = make_float4(
          pair_component(h.x, l.x, pih.x, pil.x, na, nb, nc, H[0], H[9], H[3], H[12], H[6], H[15]),
          pair_component(h.y, l.y, pih.y, pil.y, na, nb, nc, H[1], H[10], H[4], H[13], H[7], H[16]),
          pair_component(h.z, l.z, pih.z, pil.z, na, nb, nc, H[2], H[11], H[5], H[14], H[8], H[17]), h.w);
      const char4 sh = make_char4(na, nb, nc, 0);
      if (in) {
        O.j0[d0 + e] = en[u].x;
        O.r0[d0 + e] = r;
        O.sh0[d0 + e] = sh;
      }
      const unsigned m = __ballot_sync(0xffffffffu, ang);
      if (ang) {
        const int d = d1 + __popc(m & lt);
        O.j1[d] = en[u].x;
        O.r1[d] = r;
        O.sh1[d] = sh;
        O.own1[d] = i;
      }
      d1 += __popc(m);
    }
  }
  commit_batch(A, O, i, lane);
}

// The same moves without slots, ahead of the writing pass.
__global__ void __launch_bounds__(256) k_commit(BuildArgs A, ListOut O) {
  const int i = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (i < A.N) commit_batch(A, O, i, threadIdx.x & 31);
}

// The sums of both lists' counts over each 1,024 atoms, and the largest count.
__global__ void __launch_bounds__(1024) k_count_sums(BuildArgs A) {
  GNEP_PDL_START();
  __shared__ int ws[32][3];
  const int i = blockIdx.x * 1024 + threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c0 = i < A.N ? A.cnt0[i] : 0, c1 = i < A.N ? A.cnt1[i] : 0;
  const int t0 = __reduce_add_sync(0xffffffffu, c0), t1 = __reduce_add_sync(0xffffffffu, c1);
  const int mx = __reduce_max_sync(0xffffffffu, c0);
  if (lane == 0) {
    ws[warp][0] = t0;
    ws[warp][1] = t1;
    ws[warp][2] = mx;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    const int q = threadIdx.x;
    long long r = 0;
    for (int w = 0; w < 32; ++w) r = q < 2 ? r + ws[w][q] : max(r, (long long)ws[w][q]);
    if (q < 2)
      A.bsum[2 * blockIdx.x + q] = r;
    else
      atomicMax(&A.res->max, (int)r);
  }
}

// Offsets of both lists: each block of 1,024 atoms adds up the blocks before it
// and scans its own counts; the last one leaves the totals (64-bit, so that a
// pair count beyond 32-bit indices is seen) and the model's error flag.
__global__ void __launch_bounds__(1024) k_offsets(BuildArgs A) {
  GNEP_PDL_START();
  __shared__ long long before[2];
  __shared__ int ws[2][32];
  const int i = blockIdx.x * 1024 + threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp < 2) {  // warp q: the blocks before this one
    long long t = 0;
    for (int b = lane; b < (int)blockIdx.x; b += 32) t += A.bsum[2 * b + warp];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) before[warp] = t;
  }
  const int c0 = i < A.N ? A.cnt0[i] : 0, c1 = i < A.N ? A.cnt1[i] : 0;
  if (gridDim.x == 1) {  // a batch of one block has no k_count_sums
    const int mx = __reduce_max_sync(0xffffffffu, c0);
    if (lane == 0) atomicMax(&A.res->max, mx);
  }
  int v0 = c0, v1 = c1;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u0 = __shfl_up_sync(0xffffffffu, v0, o), u1 = __shfl_up_sync(0xffffffffu, v1, o);
    if (lane >= o) {
      v0 += u0;
      v1 += u1;
    }
  }
  if (lane == 31) {
    ws[0][warp] = v0;
    ws[1][warp] = v1;
  }
  __syncthreads();
  if (warp < 2) {
    int t = ws[warp][lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += u;
    }
    ws[warp][lane] = t;
  }
  __syncthreads();
  const long long e0 = before[0] + (warp ? ws[0][warp - 1] : 0) + v0, e1 = before[1] + (warp ? ws[1][warp - 1] : 0) + v1;
  if (i < A.N) {
    A.off0[i] = (int)(e0 - c0);
    A.off1[i] = (int)(e1 - c1);
  }
  if (i == A.N - 1) {
    A.off0[A.N] = (int)e0;
    A.off1[A.N] = (int)e1;
    A.res->tot[0] = e0;
    A.res->tot[1] = e1;
    A.res->err = *A.err;
  }
}

constexpr int kSlots = 96;  // per-atom slots of the one-pass build

// Reverse pair: the entry (i, -n) in j's list, found by binary search on the
// canonical key (j, na, nb, nc).
__global__ void k_reverse(int64_t P, const int* __restrict__ off, const int* __restrict__ jj,
                          const int* __restrict__ own, const char4* __restrict__ sh,
                          int* __restrict__ rev, int* __restrict__ err) {
  GNEP_PDL_START();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= P) return;
  const int i = own[p], j = jj[p];
  const char4 s = sh[p];
  const int key[4] = {i, -s.x, -s.y, -s.z};
  int lo = off[j], hi = off[j + 1] - 1, found = -1;
  while (lo <= hi) {
    const int mid = (lo + hi) >> 1;
    const char4 t = sh[mid];
    const int cand[4] = {jj[mid], t.x, t.y, t.z};
    int cmp = 0;
    for (int q = 0; q < 4 && cmp == 0; ++q) cmp = (cand[q] < key[q]) ? -1 : (cand[q] > key[q]) ? 1 : 0;
    if (cmp == 0) { found = mid; break; }
    if (cmp < 0) lo = mid + 1; else hi = mid - 1;
  }
  if (found < 0) { atomicOr(err, kErrRevMissing); found = (int)p; }
  rev[p] = found;
}

}  // namespace

// The lists of `nl` for the batch `b` (NULL: for the list's own positions, as a
// molecular dynamics step leaves them).  Kernels up to the host's one wait work
// in scratch alone (one stream-ordered allocation): a batch that fails its checks
// leaves the list as it was.  Launches: k_prep, k_bins (batches above
// kCellMinAtoms atoms), k_pairs_slots, k_count_sums (above 1,024 atoms),
// k_offsets, the wait, k_compact, k_reverse.  What bounds a small build is this
// chain and the wait, not work: with a launch per check, scan level, conversion
// and copy, 14 allocations, and tiles cut on the host, rebuilding and evaluating
// one structure of 139 atoms took 310 us, now 137; 256 structures 757, now 364; a
// molecular dynamics step of 4,096 atoms 316, now 146.
int build_lists(gnep_model* m, gnep_nlist* nl, const gnep_batch* b, cudaStream_t st, bool* types_changed) {
  const int N = nl->n_atoms, S = nl->n_struct;
  BuildArgs A;
  A.N = N;
  A.S = S;
  A.ns = m->shape.ns;
  A.rc = nl->rcr > nl->rca ? nl->rcr : nl->rca;
  A.err = m->err;
  const size_t n = N, s = S, nb = (n + 1023) / 1024;
  Slots sl;  // one pass into per-atom slots; atoms with more neighbours take the batch to a second, writing pass
  sl.cap = kSlots;
  // zeroed: result, bin counts and cursors; then the rest
  // host arrays, and what the kernels must not read in place, are copied over first
  const bool stage = b && !(kernel_can_use(b->struct_off, 4, nl->device) && kernel_can_use(b->type, 4, nl->device) &&
                            kernel_can_use(b->pos, 8, nl->device) && kernel_can_use(b->cell, 8, nl->device));
  struct Item { void** p; size_t bytes; };
  const Item items[] = {
      {(void**)&A.res, sizeof(BuildResult)}, {(void**)&A.bcount, 4 * n}, {(void**)&A.bcursor, 4 * n},
      {(void**)&A.atom_struct, 4 * n}, {(void**)&A.kr, 12 * s}, {(void**)&A.nbin, 12 * s}, {(void**)&A.tw, 12 * s},
      {(void**)&A.hsplit, 72 * s}, {(void**)&A.frac, 16 * n}, {(void**)&A.phi, 16 * n}, {(void**)&A.plo, 16 * n},
      {(void**)&A.cnt0, 4 * n}, {(void**)&A.cnt1, 4 * n}, {(void**)&A.bstart, 4 * (n + s)}, {(void**)&A.batom, 4 * n},
      {(void**)&A.bsum, 16 * nb}, {(void**)&A.off0, 4 * (n + 1)}, {(void**)&A.off1, 4 * (n + 1)},
      {(void**)&A.hl, 32 * n}, {(void**)&sl.e, 8 * n * kSlots},
      {(void**)&A.off_c, b ? 4 * (s + 1) : 0}, {(void**)&A.type_c, b ? 4 * n : 0},
      {(void**)&A.pos_c, b ? 24 * n : 0}, {(void**)&A.cell_c, b ? 72 * s : 0}};
  size_t total = 0;
  for (const Item& it : items) total += (it.bytes + 255) & ~size_t(255);
  char* base = nullptr;
  GNEP_CUDA(cudaMallocAsync(&base, total, st));
  struct Free {  // given back on every way out
    char* p;
    cudaStream_t st;
    ~Free() { cudaFreeAsync(p, st); }
  } give_back{base, st};
  size_t at = 0;
  for (const Item& it : items) {
    *it.p = base + at;
    at += (it.bytes + 255) & ~size_t(255);
  }
  GNEP_CUDA(cudaMemsetAsync(base, 0, (size_t)((char*)A.atom_struct - base), st));
  ListOut O;
  memset(&O, 0, sizeof(O));
  O.atom_struct = nl->atom_struct;
  if (b) {
    A.off = b->struct_off;
    A.type = b->type;
    A.pos = b->pos;
    A.cell = b->cell;
    if (stage) {
      GNEP_CUDA(cudaMemcpyAsync(A.off_c, b->struct_off, 4 * (s + 1), cudaMemcpyDefault, st));
      GNEP_CUDA(cudaMemcpyAsync(A.type_c, b->type, 4 * n, cudaMemcpyDefault, st));
      GNEP_CUDA(cudaMemcpyAsync(A.pos_c, b->pos, 24 * n, cudaMemcpyDefault, st));
      GNEP_CUDA(cudaMemcpyAsync(A.cell_c, b->cell, 72 * s, cudaMemcpyDefault, st));
      A.off = A.off_c;
      A.type = A.type_c;
      A.pos = A.pos_c;
      A.cell = A.cell_c;
    }
    A.old_type = nl->built ? nl->type : nullptr;
    O.struct_off = nl->struct_off;
    O.type = nl->type;
    O.pos = nl->pos;
    O.cell = nl->cell;
  } else {
    A.off_c = A.type_c = nullptr;
    A.pos_c = A.cell_c = nullptr;
    A.off = nl->struct_off;
    A.type = A.old_type = nl->type;
    A.pos = nl->pos;
    A.cell = nl->cell;
  }

  ListParams lp;
  lp.rc2[0] = nl->rcr * nl->rcr;
  lp.rc2[1] = nl->rca * nl->rca;
  for (int L = 0; L < 2; ++L) {
    lp.lo2[L] = (float)(lp.rc2[L] * (1.0 - 2e-3));
    lp.hi2[L] = (float)(lp.rc2[L] * (1.0 + 2e-3));
  }
  lp.reject2 = lp.hi2[0] > lp.hi2[1] ? lp.hi2[0] : lp.hi2[1];

  (void)launch_on(false, k_prep, blocks_for(N, kPrep), kPrep, 0, st, A);
  if (N > kCellMinAtoms) (void)launch_pdl(k_bins, S, 1024, 0, st, A);
  (void)launch_pdl(k_pairs_slots, blocks_for((int64_t)N * 32, 32 * kFlatWarps), 32 * kFlatWarps, 0, st, A, lp, sl);
  if (nb > 1) (void)launch_pdl(k_count_sums, (int)nb, 1024, 0, st, A);
  (void)launch_pdl(k_offsets, (int)nb, 1024, 0, st, A);
  GNEP_CHECK_LAUNCH("neighbour search");
  if (!nl->host_res) GNEP_CUDA(cudaMallocHost(&nl->host_res, sizeof(BuildResult)));
  BuildResult& r = *static_cast<BuildResult*>(nl->host_res);
  GNEP_CUDA(cudaMemcpyAsync(&r, A.res, sizeof(BuildResult), cudaMemcpyDeviceToHost, st));
  GNEP_CUDA(cudaStreamSynchronize(st));
  if (r.flags & kBadEnds) return set_error(GNEP_ERR_INVALID_ARG, "struct_off must start at 0 and end at n_atoms");
  if (r.flags & kBadOrder)
    return set_error(GNEP_ERR_INVALID_ARG, "struct_off must be strictly increasing (every structure holds an atom)");
  if (r.flags & kBadType) return set_error(GNEP_ERR_INVALID_ARG, "species index out of range");
  if (r.flags & kUnwrapped)
    return set_error(GNEP_ERR_INVALID_ARG, "positions must be wrapped into their cell (fractional coordinates in [0,1))");
  for (int L = 0; L < 2; ++L)
    if (r.tot[L] >= (1LL << 31) - 1)
      return set_error(GNEP_ERR_NEIGHBOR_OVERFLOW, "pair count exceeds 32-bit indices; split the batch");
  ++nl->gen;  // graphs captured on the list no longer launch
  // from here on the list changes: until finish_build has seen the end of it, no call takes it
  *types_changed = !nl->built || (r.flags & kTypesChanged);  // an unfinished build may have left any grouping
  nl->built = false;
  nl->last_err = r.err;

  for (int L = 0; L < 2; ++L) {
    PairList& P = nl->L[L];
    if (r.tot[L] > P.cap) {
      cudaFree(P.j); cudaFree(P.owner); cudaFree(P.rev); cudaFree(P.rij); cudaFree(P.shift);
      P.j = P.owner = P.rev = nullptr;
      P.rij = nullptr;
      P.shift = nullptr;
      P.cap = P.n = 0;
      const int64_t cap = r.tot[L] + r.tot[L] / 8 + 64;  // headroom for rebuilds (MD)
      GNEP_CUDA(cudaMalloc(&P.j, sizeof(int) * cap));
      if (L == 1) {  // the force sweep pairs angular entries
        GNEP_CUDA(cudaMalloc(&P.owner, sizeof(int) * cap));
        GNEP_CUDA(cudaMalloc(&P.rev, sizeof(int) * cap));
      }
      GNEP_CUDA(cudaMalloc(&P.rij, sizeof(float4) * cap));
      GNEP_CUDA(cudaMalloc(&P.shift, sizeof(char4) * cap));
      P.cap = cap;
    }
    if (!P.off) GNEP_CUDA(cudaMalloc(&P.off, sizeof(int) * (size_t)(N + 1)));
    P.n = r.tot[L];
    (L ? O.offa : O.offr) = P.off;
  }
  O.j0 = nl->L[0].j; O.r0 = nl->L[0].rij; O.sh0 = nl->L[0].shift;
  O.j1 = nl->L[1].j; O.own1 = nl->L[1].owner; O.r1 = nl->L[1].rij; O.sh1 = nl->L[1].shift;
  if (r.max <= sl.cap) {
    (void)launch_on(false, k_compact, blocks_for((int64_t)N * 32, 256), 256, 0, st, A, sl, O);
  } else {
    (void)launch_on(false, k_commit, blocks_for((int64_t)N * 32, 256), 256, 0, st, A, O);
    k_pairs<<<blocks_for((int64_t)N * 32, 128), 128, 0, st>>>(
        N, nl->struct_off, nl->atom_struct, nl->pos, nl->cell, A.kr, A.tw, A.hsplit, A.frac, A.phi, A.plo, lp, A.off0,
        A.off1, nl->L[0].j, nl->L[0].rij, nl->L[0].shift, nl->L[1].j, nl->L[1].owner, nl->L[1].rij,
        nl->L[1].shift);
  }
  GNEP_CHECK_LAUNCH("neighbour lists");
  // reverse entries of the angular list (the radial force terms need none)
  PairList& P = nl->L[1];
  if (P.n > 0)
    (void)launch_pdl(k_reverse, blocks_for(P.n, 256), 256, 0, st, P.n, (const int*)P.off, (const int*)P.j,
                     (const int*)P.owner, (const char4*)P.shift, P.rev, m->err);
  GNEP_CHECK_LAUNCH("k_reverse");
  return GNEP_OK;  // the reverse search sets kErrRevMissing, reported later
}

}  // namespace gnep
