// Krylov kernels: Arnoldi with classical Gram-Schmidt run twice (CGS2) over
// the tall-skinny basis, the FP64 phi-function of the small Hessenberg
// matrix, and the fused PCEXP update (Sec. 2.2 of the paper, Eq. vm-vm2,
// final; Eq. s9, s10).
//
// Basis storage: V[i] holds an unnormalised vector z_i and KState.s[i] its
// scale, v_i = s_i z_i, so normalisation costs no extra pass.  One Arnoldi
// column j runs as
//   w   = s_j J z_j = J v_j          (DG tangent-linear kernel, scale on its output)
//   P   : h_i  = s_i <z_i, w>,  ||w||                          (read V_j, w)
//   UP  : w   -= sum_i s_i^2 <z_i,w> z_i; h2_i = s_i <z_i, w>  (read V_j, w; write w)
//   UN  : z_{j+1} = w - sum_i s_i^2 <z_i,w> z_i; h_{j+1,j} = ||z_{j+1}||, s_{j+1} = 1/h_{j+1,j}
// so every stored z_i has the size of ||J|| (no growth like ||J||^i, which would
// overflow FP32 storage).  The selective form (FP32-mixed default) runs a column as
//   P, U1: z_{j+1} = w - sum_i s_i^2 <z_i,w> z_i, ||z_{j+1}||       (read V_j, w; write z_{j+1})
// and keeps that first update when ||z_{j+1}|| >= ||w|| / sqrt(2); otherwise the second
// pass follows, P2 (h2 = V_j^T z_{j+1}) and UN in place on z_{j+1}.  The second pass's
// launches leave at once in the columns that keep their first update.
// Each streaming kernel writes per-block partial sums; the last block to
// finish (atomic ticket) reduces them in a fixed order and applies the scalar
// update, so results are deterministic and no extra launch is needed.
// Partial products are accumulated in FP64 (FP64 form) or in compensated FP32
// pairs converted to FP64 once per warp (FP32-mixed form).
#include <cooperative_groups.h>
#include <atomic>
#include <cfloat>
#include <cstddef>

#include "kernels.h"

namespace pcexp {

// Elements per thread per row-loop iteration: one 16-byte load (double2 / float4).
template <class T> struct VecN {
  static constexpr int N = 16 / sizeof(T);
};

template <class T, int VN>
PCEXP_DEV void load_vec(const T* p, T (&x)[VN]) {
  if constexpr (sizeof(T) == 8) {
    double2 a = *reinterpret_cast<const double2*>(p);
    x[0] = a.x;
    x[1] = a.y;
  } else {
    float4 a = *reinterpret_cast<const float4*>(p);
    x[0] = a.x;
    x[1] = a.y;
    x[2] = a.z;
    x[3] = a.w;
  }
}
template <class T, int VN>
PCEXP_DEV void store_vec(T* p, const T (&x)[VN]) {
  if constexpr (sizeof(T) == 8) {
    *reinterpret_cast<double2*>(p) = make_double2(x[0], x[1]);
  } else {
    *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
  }
}

// Dot-product accumulator.  FP64 form: a double.  FP32-mixed form: an unevaluated
// float pair hi + lo updated with Knuth's TwoSum, so per-thread sums and the warp
// shuffle tree run on the FP32 pipe (GB300 has 1/62 the FP64 rate) while keeping
// about twice FP32 precision; each warp converts to FP64 once per column.
// Both are 8 bytes, so block partial sums are stored in the same FP64-sized slots; the
// float pair stays a pair through the block and grid reductions and is converted to
// FP64 once per column (each FP64 warp instruction costs tens of cycles here).
template <class T> struct Acc;
template <> struct Acc<double> {
  double s;
  PCEXP_DEV void zero() { s = 0.0; }
  PCEXP_DEV void add(double x) { s += x; }
  PCEXP_DEV void add_acc(const Acc& o) { s += o.s; }
  PCEXP_DEV void add_partner(int o) { s += __shfl_xor_sync(0xffffffffu, s, o); }
  PCEXP_DEV void shfl_from(const Acc& src, int o) { s = __shfl_xor_sync(0xffffffffu, src.s, o); }
  PCEXP_DEV double value() const { return s; }
};
template <> struct Acc<float> {
  float hi, lo;
  PCEXP_DEV void zero() { hi = lo = 0.f; }
  PCEXP_DEV void add(float x) {
    const float s = hi + x;
    const float bp = s - hi;
    lo += (hi - (s - bp)) + (x - bp);
    hi = s;
  }
  PCEXP_DEV void add_acc(const Acc& o) {
    add(o.hi);
    lo += o.lo;
  }
  PCEXP_DEV void add_partner(int o) {
    Acc p;
    p.shfl_from(*this, o);
    add_acc(p);
  }
  PCEXP_DEV void shfl_from(const Acc& src, int o) {
    hi = __shfl_xor_sync(0xffffffffu, src.hi, o);
    lo = __shfl_xor_sync(0xffffffffu, src.lo, o);
  }
  PCEXP_DEV double value() const { return (double)hi + (double)lo; }
};
static_assert(sizeof(Acc<float>) == 8 && sizeof(Acc<double>) == 8, "partials are 8-byte slots");

// sum_v a[v] * b[v] in T (FMA chain over one 16-byte chunk)
template <class T, int VN>
PCEXP_DEV T dot_vec(const T (&a)[VN], const T (&b)[VN]) {
  T s = 0;
#pragma unroll
  for (int v = 0; v < VN; ++v) s = fma(a[v], b[v], s);
  return s;
}

// acc += <a, b> over one chunk.  FP64: FMAs straight into the accumulator (one FP64
// instruction per element; the FP64 pipe bounds these passes).  FP32: the chunk's FMA chain,
// then one compensated addition.
template <class T, int VN>
PCEXP_DEV void acc_dot(Acc<T>& acc, const T (&a)[VN], const T (&b)[VN]) {
  if constexpr (sizeof(T) == 8) {
#pragma unroll
    for (int v = 0; v < VN; ++v) acc.s = fma(a[v], b[v], acc.s);
  } else {
    acc.add(dot_vec<T, VN>(a, b));
  }
}

// Selective re-orthogonalisation (Daniel, Gragg, Kaufman & Stewart 1976): the first pass
// is kept alone when ||w_1|| >= ||w|| / sqrt(2), i.e. when it cancelled less than that.
constexpr double DGKS_KAPPA = 0.70710678118654752440;

// Stage logic of the last block: per-column entries in parallel, scalars on thread 0.
//   PROJ      h = V^T w: column j of H (and of H1), update coefficients, ||w||
//   UPD_PROJ  h2 = V^T w_1 after the update: added to column j, new coefficients
//   PROJ2     the same for the selective form's separate second projection
//   UPD1      the selective form's first update w_1 = w - V h alone, with ||w_1||: keep it as
//             z_{j+1} (skip2) when it cancelled less than DGKS_KAPPA, else leave the column
//             to PROJ2 + UPD_NORM
//   UPD_NORM  z_{j+1} = w_1 - V h2, h_{j+1,j} = ||z_{j+1}||, breakdown test
PCEXP_DEV void cgs_finalize(int mode, int j, const double* dots, KState* ks, double eta) {
  __shared__ int bad;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  if (mode == CGS_PROJ || mode == CGS_UPD_PROJ || mode == CGS_PROJ2) {
    // w = J v_j is already normalised by s_j (applied by the J v kernel)
    for (int i = threadIdx.x; i <= j; i += blockDim.x) {
      const double si = ks->s[i];
      const double h = si * dots[i];
      if (!isfinite(h)) bad = 1;
      if (mode == CGS_PROJ) {
        ks->H[i * MMAX + j] = h;
        ks->H1[i * MMAX + j] = h;
      } else {
        ks->H[i * MMAX + j] += h;
      }
      ks->coef[i] = si * h;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      if (mode == CGS_PROJ) ks->wnorm0 = sqrt(dots[j + 1]);
      if (bad) {
        ks->err = 1;
        ks->done = 1;
      }
    }
    return;
  }
  if (threadIdx.x != 0) return;
  if (mode == CGS_NORM) {
    const double beta = sqrt(dots[0]);
    ks->beta = beta;
    ks->k = 0;
    if (!isfinite(beta)) {
      ks->err = 1;
      ks->done = 1;
    } else if (beta == 0.0) {
      ks->done = 1;
    } else {
      ks->s[0] = 1.0 / beta;
      ks->done = 0;
    }
    return;
  }
  if (mode == CGS_UPD1) {
    // a non-finite or zero norm takes the second pass, whose norm test reports it; a kept
    // first pass has ||w_1|| >= ||w|| / sqrt(2) > eta ||w||, so it needs no breakdown test
    const double n1 = sqrt(dots[0]);
    const bool keep1 = isfinite(n1) && n1 > 0.0 && n1 >= DGKS_KAPPA * ks->wnorm0;
    ks->skip2 = keep1 ? 1 : 0;
    if (keep1) {
      ks->H[(j + 1) * MMAX + j] = n1;
      ks->k = j + 1;
      ks->s[j + 1] = 1.0 / n1;
    }
    return;
  }
  // CGS_UPD_NORM
  const double hn = sqrt(dots[0]);
  ks->pass2 |= 1u << j;
  ks->H[(j + 1) * MMAX + j] = hn;
  ks->k = j + 1;
  if (!isfinite(hn)) {
    ks->err = 1;
    ks->done = 1;
  } else if (hn == 0.0 || hn <= eta * ks->wnorm0) {
    ks->done = 1;  // happy breakdown: K_{j+1} is invariant
  } else {
    ks->s[j + 1] = 1.0 / hn;
  }
}

// The passes that belong to a column's second Gram-Schmidt pass leave at once when the
// selective form kept the first pass.
PCEXP_DEV bool cgs_skipped(int fmode, const KState* ks) {
  return (fmode == CGS_PROJ2 || fmode == CGS_UPD_NORM) && ks->skip2;
}

// Warp reduction of NC accumulators at once (NC a power of two <= 32): plain
// butterfly levels until NC values remain per lane pair group, then transpose levels
// in which each lane keeps half of its columns and receives the partner's other half.
// Afterwards lane l holds the warp sum of column (l mod NC): NC - 1 + (5 - log2 NC) NC
// additions per lane instead of 5 NC.  Fixed order, so deterministic.
template <class T, int NC, int L, int O>
PCEXP_DEV void transpose_level(Acc<T> (&a)[NC], int lane) {
  if constexpr (L >= 2) {
    const bool upper = (lane & O) != 0;
#pragma unroll
    for (int i = 0; i < L / 2; ++i) {
      Acc<T> send = upper ? a[i] : a[i + L / 2];
      Acc<T> keep = upper ? a[i + L / 2] : a[i];
      Acc<T> recv;
      recv.shfl_from(send, O);
      keep.add_acc(recv);
      a[i] = keep;
    }
    transpose_level<T, NC, L / 2, O / 2>(a, lane);
  }
}

template <class T, int NC>
PCEXP_DEV Acc<T> warp_reduce_columns(Acc<T> (&a)[NC], int lane) {
  constexpr int LOGNC = NC >= 32 ? 5 : NC >= 16 ? 4 : NC >= 8 ? 3 : NC >= 4 ? 2 : NC >= 2 ? 1 : 0;
  static_assert((1 << LOGNC) == NC, "NC must be a power of two <= 32");
#pragma unroll
  for (int o = 16; o >= NC; o >>= 1) {
#pragma unroll
    for (int c = 0; c < NC; ++c) a[c].add_partner(o);
  }
  transpose_level<T, NC, NC, NC / 2>(a, lane);
  return a[0];
}

// Row Gram-Schmidt pass (NORM, PROJ, UPD_PROJ, UPD_NORM): every thread owns whole 16-byte
// chunks of rows and accumulates all columns for them; the launch bounds hold it at 128
// registers so that two blocks share an SM.
// MODE is how the pass streams; fmode (CgsMode) what its last block does with the sums.  In
// the selective form the second pass's UPD_NORM runs in place (w == out == z_{j+1}, each
// element read and then written by the same thread), so w and out are not restrict-qualified.
template <class T, int NC, int MODE>
__global__ void __launch_bounds__(256, 2) cgs_kernel(const T* __restrict__ Z, int64_t ldz, int64_t Kp, int j,
                                                  T* w, T* out, KState* ks,
                                                  double* __restrict__ partials, double eta, int fmode) {
  constexpr int VN = VecN<T>::N;
  constexpr int NACC = (MODE == CGS_PROJ) ? NC + 1 : (MODE == CGS_UPD_PROJ ? NC : 1);
  __shared__ T scoef[NC > 0 ? NC : 1];
  __shared__ Acc<T> red[8][NACC];
  __shared__ bool last;
  if (ks->done) return;  // breakdown reached earlier: uniform early exit
  if (cgs_skipped(fmode, ks)) return;
  const int nc = (MODE == CGS_NORM) ? 0 : j + 1;
  if (MODE == CGS_UPD_PROJ || MODE == CGS_UPD_NORM)
    for (int c = threadIdx.x; c < nc; c += blockDim.x) scoef[c] = (T)ks->coef[c];
  __syncthreads();
  Acc<T> acc[NACC];
#pragma unroll
  for (int c = 0; c < NACC; ++c) acc[c].zero();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x * VN;
  for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * VN; r < Kp; r += stride) {
    T x[VN];
    load_vec<T, VN>(w + r, x);
    if constexpr (MODE == CGS_NORM) {
      acc_dot<T, VN>(acc[0], x, x);
    } else if constexpr (MODE == CGS_PROJ) {
      // columns in groups of 8: a group's loads are issued together (the column index
      // clamped to the last one, so no load waits behind a branch) before its FMAs
      constexpr int G = NC < 8 ? NC : 8;
#pragma unroll
      for (int c0 = 0; c0 < NC; c0 += G) {
        if (c0 < nc) {
          T z[G][VN];
#pragma unroll
          for (int g = 0; g < G; ++g) load_vec<T, VN>(Z + (int64_t)(c0 + g < nc ? c0 + g : nc - 1) * ldz + r, z[g]);
#pragma unroll
          for (int g = 0; g < G; ++g)
            if (c0 + g < nc) acc_dot<T, VN>(acc[c0 + g], z[g], x);
        }
      }
      acc_dot<T, VN>(acc[NC], x, x);
    } else {
      // update pass in the same column groups; the projection pass of UPD_PROJ below
      // re-reads each group's chunks
      constexpr int G = NC < 8 ? NC : 8;
#pragma unroll
      for (int c0 = 0; c0 < NC; c0 += G) {
        if (c0 < nc) {
          T z[G][VN];
#pragma unroll
          for (int g = 0; g < G; ++g) load_vec<T, VN>(Z + (int64_t)(c0 + g < nc ? c0 + g : nc - 1) * ldz + r, z[g]);
#pragma unroll
          for (int g = 0; g < G; ++g)
            if (c0 + g < nc)
#pragma unroll
              for (int v = 0; v < VN; ++v) x[v] = fma(-scoef[c0 + g], z[g][v], x[v]);
        }
      }
      if constexpr (MODE == CGS_UPD_PROJ) {
        store_vec<T, VN>(w + r, x);
        // reload the chunks rather than keep all of them live across the store (255 -> 128
        // registers, two blocks per SM instead of one; the reloads hit L1/L2)
        asm volatile("" ::: "memory");
#pragma unroll
        for (int c0 = 0; c0 < NC; c0 += G) {
          if (c0 < nc) {
            T z[G][VN];
#pragma unroll
            for (int g = 0; g < G; ++g) load_vec<T, VN>(Z + (int64_t)(c0 + g < nc ? c0 + g : nc - 1) * ldz + r, z[g]);
#pragma unroll
            for (int g = 0; g < G; ++g)
              if (c0 + g < nc) acc_dot<T, VN>(acc[c0 + g], z[g], x);
          }
        }
      } else {
        store_vec<T, VN>(out + r, x);
        acc_dot<T, VN>(acc[0], x, x);
      }
    }
  }
  // block reduction in the accumulator type (fixed order): warp tree, then over warps
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if constexpr (MODE == CGS_NORM || MODE == CGS_UPD_NORM) {
    for (int o = 16; o > 0; o >>= 1) acc[0].add_partner(o);
    if (lane == 0) red[wid][0] = acc[0];
  } else {
    Acc<T> cols[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) cols[c] = acc[c];
    const Acc<T> mine = warp_reduce_columns<T, NC>(cols, lane);
    if (lane < NC) red[wid][lane] = mine;
    if constexpr (MODE == CGS_PROJ) {
      for (int o = 16; o > 0; o >>= 1) acc[NC].add_partner(o);
      if (lane == 0) red[wid][NC] = acc[NC];
    }
  }
  __syncthreads();
  const int nred = (MODE == CGS_PROJ) ? nc + 1 : (MODE == CGS_UPD_PROJ ? nc : 1);
  Acc<T>* P = reinterpret_cast<Acc<T>*>(partials);
  for (int c = threadIdx.x; c < nred; c += blockDim.x) {
    const int cc = (MODE == CGS_PROJ && c == nc) ? NC : c;
    Acc<T> a = red[0][cc];
    for (int q = 1; q < nw; ++q) a.add_acc(red[q][cc]);
    P[(int64_t)c * gridDim.x + blockIdx.x] = a;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&ks->counter, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  __shared__ double dots[MMAX + 2];
  // every lane issues all its partial loads before summing them (fixed order per lane,
  // fixed shuffle tree), so the serial tail of the last block is one L2 round trip
  constexpr int PER_LANE = (RED_BLOCKS + 31) / 32;
  for (int c = wid; c < nred; c += nw) {
    const unsigned long long* pc = reinterpret_cast<const unsigned long long*>(P + (int64_t)c * gridDim.x);
    unsigned long long pv[PER_LANE];
#pragma unroll
    for (int t = 0; t < PER_LANE; ++t) {
      const unsigned b = lane + 32u * t;
      pv[t] = b < gridDim.x ? __ldcg(pc + b) : 0ull;
    }
    Acc<T> a;
    a.zero();
#pragma unroll
    for (int t = 0; t < PER_LANE; ++t) a.add_acc(*reinterpret_cast<const Acc<T>*>(&pv[t]));
    for (int o = 16; o > 0; o >>= 1) a.add_partner(o);
    if (lane == 0) dots[c] = a.value();
  }
  __syncthreads();
  if (ks->group) {  // partitioned: the sums over all partitions are finalised afterwards
    for (int c = threadIdx.x; c < nred; c += blockDim.x) ks->gsum[c] = dots[c];
    if (threadIdx.x == 0) ks->counter = 0;
    return;
  }
  cgs_finalize(fmode, j, dots, ks, eta);
  if (threadIdx.x == 0) ks->counter = 0;
}

// Per-block sums red[0..nred) -> partials; the last block to finish (atomic ticket) reduces
// them in a fixed order and finalises the column.  Every thread of the block calls this.
template <class T>
PCEXP_DEV void cgs_grid_tail(const Acc<T>* red, int nred, int mode, int j, KState* ks, double* partials,
                             double eta) {
  __shared__ bool last;
  __shared__ double dots[MMAX + 2];
  Acc<T>* P = reinterpret_cast<Acc<T>*>(partials);
  for (int c = threadIdx.x; c < nred; c += blockDim.x) P[(int64_t)c * gridDim.x + blockIdx.x] = red[c];
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&ks->counter, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  constexpr int PER_LANE = (RED_BLOCKS + 31) / 32;
  for (int c = wid; c < nred; c += nw) {
    const unsigned long long* pc = reinterpret_cast<const unsigned long long*>(P + (int64_t)c * gridDim.x);
    unsigned long long pv[PER_LANE];
#pragma unroll
    for (int t = 0; t < PER_LANE; ++t) {
      const unsigned b = lane + 32u * t;
      pv[t] = b < gridDim.x ? __ldcg(pc + b) : 0ull;
    }
    Acc<T> a;
    a.zero();
#pragma unroll
    for (int t = 0; t < PER_LANE; ++t) a.add_acc(*reinterpret_cast<const Acc<T>*>(&pv[t]));
    for (int o = 16; o > 0; o >>= 1) a.add_partner(o);
    if (lane == 0) dots[c] = a.value();
  }
  __syncthreads();
  if (ks->group) {
    for (int c = threadIdx.x; c < nred; c += blockDim.x) ks->gsum[c] = dots[c];
    if (threadIdx.x == 0) ks->counter = 0;
    return;
  }
  cgs_finalize(mode, j, dots, ks, eta);
  if (threadIdx.x == 0) ks->counter = 0;
}

// FP32 projection pass (PROJ and PROJ2): h = V^T w and ||w||^2.  The 8 warps of a block walk the
// same tiles of rows and warp w owns the columns w, w + 8, ... (NCW of them, NCW the least that
// covers the columns), so a thread holds NCW accumulators instead of one per column.  A tile is U
// chunks of 512 bytes per column: a warp reads U consecutive chunks of each of its columns, all
// loads issued before their sums, and the grid is exactly one wave.  Bound by HBM bytes.
// Against the form with NCW = 1, 2, 4, one chunk per column and step (time per launch, 48^3 cubes
// at p = 2, K = 33.2 M; 8 / 16 / 20 / 24 / 30 columns): 188 / 340 / 520 / 537 / 622 -> 171 / 325 /
// 400 / 462 / 568 us, 6.9 to 7.2 TB/s; on 131,072 triangles at p = 3 (K = 5.2 M) 39 / 64 / 92 / 97
// / 110 -> 35 / 61 / 72 / 83 / 99 us.
constexpr int CGS_WARPS = 8;
template <int NCW, int U>
__global__ void __launch_bounds__(256) cgs_proj_kernel(const float* __restrict__ Z, int64_t ldz, int64_t Kp, int j,
                                                       const float* __restrict__ w, KState* ks,
                                                       double* __restrict__ partials, double eta, int fmode) {
  constexpr int VN = VecN<float>::N, CHUNK = 32 * VN, TR = CHUNK * U;
  __shared__ Acc<float> red[CGS_WARPS * NCW + 1];
  if (ks->done) return;  // breakdown reached earlier: uniform early exit
  if (cgs_skipped(fmode, ks)) return;
  const int nc = j + 1;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  Acc<float> acc[NCW + 1];
#pragma unroll
  for (int k = 0; k <= NCW; ++k) acc[k].zero();
  const int64_t ntile = (Kp + TR - 1) / TR;
  for (int64_t t = blockIdx.x; t < ntile; t += gridDim.x) {
    const int64_t r = t * TR + lane * VN;
    float x[U][VN], z[NCW][U][VN];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (r + u * CHUNK < Kp) {
        load_vec<float, VN>(w + r + u * CHUNK, x[u]);
      } else {
#pragma unroll
        for (int v = 0; v < VN; ++v) x[u][v] = 0.f;
      }
    }
#pragma unroll
    for (int k = 0; k < NCW; ++k) {
      const int c = wid + CGS_WARPS * k;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (c < nc && r + u * CHUNK < Kp) {
          load_vec<float, VN>(Z + (int64_t)c * ldz + r + u * CHUNK, z[k][u]);
        } else {
#pragma unroll
          for (int v = 0; v < VN; ++v) z[k][u][v] = 0.f;
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll
      for (int k = 0; k < NCW; ++k) acc_dot<float, VN>(acc[k], z[k][u], x[u]);
      if (wid == 0) acc_dot<float, VN>(acc[NCW], x[u], x[u]);
    }
  }
  // warp sums of the owned columns (fixed shuffle tree); each column has one owner warp.  Slots:
  // columns 0..nc-1, the norm at nc
#pragma unroll
  for (int k = 0; k < NCW; ++k) {
    for (int o = 16; o > 0; o >>= 1) acc[k].add_partner(o);
    if (lane == 0 && wid + CGS_WARPS * k < nc) red[wid + CGS_WARPS * k] = acc[k];
  }
  if (wid == 0) {
    for (int o = 16; o > 0; o >>= 1) acc[NCW].add_partner(o);
    if (lane == 0) red[nc] = acc[NCW];
  }
  __syncthreads();
  cgs_grid_tail<float>(red, nc + 1, fmode, j, ks, partials, eta);
}

// Column-split update-and-projection pass (FP32 with both passes on every column).  Warps and
// columns as above; each warp forms its partial sum of coef_c z_c, the partials meet in shared
// memory, warp 0 subtracts them in a fixed warp order, stores the updated tile and publishes it,
// and each warp projects it on its own columns with the chunks still in registers (two block
// barriers per tile).  Each thread copies its own chunks of the block's next tile into its own
// shared-memory slots with cp.async while it works on the current tile (two stages), so the next
// tile's loads are in flight across this tile's two block barriers without holding registers; no
// other thread reads a thread's slots, so the copies need no barrier of their own (C5: 29.5 ->
// 26.4 ms per step).
//
// 16-byte asynchronous copy global -> shared (bypassing L1), and its group fences
PCEXP_DEV void cgs_cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
PCEXP_DEV void cgs_cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
PCEXP_DEV void cgs_cp_wait_prev() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
PCEXP_DEV void cgs_cp_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <int NCW>
__global__ void __launch_bounds__(256) cgs_upd_proj_kernel(const float* __restrict__ Z, int64_t ldz, int64_t Kp, int j,
                                                           float* __restrict__ w, KState* ks,
                                                           double* __restrict__ partials, double eta, int fmode) {
  constexpr int VN = VecN<float>::N, TR = 32 * VN;
  __shared__ float scoef[CGS_WARPS * NCW];
  __shared__ float part[CGS_WARPS * TR];
  __shared__ float xs[TR];
  __shared__ Acc<float> red[CGS_WARPS * NCW];
  if (ks->done) return;  // breakdown reached earlier: uniform early exit
  if (cgs_skipped(fmode, ks)) return;
  const int nc = j + 1;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int c = threadIdx.x; c < CGS_WARPS * NCW; c += blockDim.x) scoef[c] = c < nc ? (float)ks->coef[c] : 0.f;
  __syncthreads();
  Acc<float> acc[NCW];
#pragma unroll
  for (int k = 0; k < NCW; ++k) acc[k].zero();
  const int64_t ntile = (Kp + TR - 1) / TR;
  constexpr int SLOTS = NCW + 1;  // the thread's column chunks, then its chunk of w
  __shared__ __align__(16) float stg[2 * CGS_WARPS * SLOTS * TR];
  auto slot = [&](int buf, int k) { return stg + ((buf * CGS_WARPS + wid) * SLOTS + k) * TR + lane * VN; };
  auto issue = [&](int64_t t, int buf) {
    const int64_t r = t * TR + lane * VN;
    if (r >= Kp) return;
#pragma unroll
    for (int k = 0; k < NCW; ++k)
      if (wid + CGS_WARPS * k < nc) cgs_cp16(slot(buf, k), Z + (wid + CGS_WARPS * k) * ldz + r);
    if (wid == 0) cgs_cp16(slot(buf, NCW), w + r);
  };
  if ((int64_t)blockIdx.x < ntile) issue(blockIdx.x, 0);
  cgs_cp_commit();
  int it = 0;
  for (int64_t t = blockIdx.x; t < ntile; t += gridDim.x, ++it) {
    const int64_t r = t * TR + lane * VN;
    const bool valid = r < Kp;
    if (t + gridDim.x < ntile) issue(t + gridDim.x, (it & 1) ^ 1);
    cgs_cp_commit();
    cgs_cp_wait_prev();  // this tile's copies (all but the group just committed) have landed
    float z[NCW][VN], x[VN], p[VN];
#pragma unroll
    for (int v = 0; v < VN; ++v) {
      p[v] = 0.f;
      x[v] = valid && wid == 0 ? slot(it & 1, NCW)[v] : 0.f;
    }
#pragma unroll
    for (int k = 0; k < NCW; ++k) {
      const float cf = scoef[wid + CGS_WARPS * k];
#pragma unroll
      for (int v = 0; v < VN; ++v) {
        z[k][v] = valid && wid + CGS_WARPS * k < nc ? slot(it & 1, k)[v] : 0.f;
        p[v] = fmaf(cf, z[k][v], p[v]);
      }
    }
#pragma unroll
    for (int v = 0; v < VN; ++v) part[wid * TR + lane * VN + v] = p[v];
    __syncthreads();
    // warp 0 forms the updated tile once (fixed warp order), stores it and publishes it
    if (wid == 0) {
#pragma unroll
      for (int q = 0; q < CGS_WARPS; ++q)
#pragma unroll
        for (int v = 0; v < VN; ++v) x[v] -= part[q * TR + lane * VN + v];
      if (valid) store_vec<float, VN>(w + r, x);
#pragma unroll
      for (int v = 0; v < VN; ++v) xs[lane * VN + v] = x[v];
    }
    __syncthreads();
    float xn[VN];
#pragma unroll
    for (int v = 0; v < VN; ++v) xn[v] = xs[lane * VN + v];
#pragma unroll
    for (int k = 0; k < NCW; ++k) acc_dot<float, VN>(acc[k], z[k], xn);
  }
  cgs_cp_wait_all();  // no copy outlives the block
  // warp sums of the owned columns (fixed shuffle tree); each column has one owner warp
#pragma unroll
  for (int k = 0; k < NCW; ++k) {
    for (int o = 16; o > 0; o >>= 1) acc[k].add_partner(o);
    if (lane == 0) red[wid + CGS_WARPS * k] = acc[k];
  }
  __syncthreads();
  cgs_grid_tail<float>(red, nc, fmode, j, ks, partials, eta);
}

template <class KernelT>
static unsigned wave_grid(KernelT kernel, int64_t chunks) {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 152;
  }
  int occ = 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, 256, 0);
  if (occ < 1) occ = 1;
  int64_t g = (int64_t)sms * occ;
  const int64_t need = (chunks + 255) / 256;
  if (g > need) g = need;
  if (g > RED_BLOCKS) g = RED_BLOCKS;
  return (unsigned)(g < 1 ? 1 : g);
}

template <class T, int NC, int MODE>
static void cgs_launch(const T* Z, int64_t ldz, int64_t Kp, int j, T* w, T* out, KState* ks, double* partials,
                       double eta, int fmode, cudaStream_t st) {
  static unsigned grid_cache = 0;
  static int64_t kp_cache = -1;
  if (kp_cache != Kp) {
    grid_cache = wave_grid(cgs_kernel<T, NC, MODE>, Kp / VecN<T>::N);
    kp_cache = Kp;
  }
  cgs_kernel<T, NC, MODE><<<grid_cache, 256, 0, st>>>(Z, ldz, Kp, j, w, out, ks, partials, eta, fmode);
}

// One launch of a streaming kernel on at most one wave of blocks.
template <int NCW, int U>
static void cgs_proj_launch(const float* Z, int64_t ldz, int64_t Kp, int j, const float* w, KState* ks,
                            double* partials, double eta, int fmode, cudaStream_t st) {
  static const unsigned wave = wave_grid(cgs_proj_kernel<NCW, U>, (int64_t)RED_BLOCKS * 256);
  constexpr int TR = 32 * VecN<float>::N * U;
  const int64_t tiles = (Kp + TR - 1) / TR;
  cgs_proj_kernel<NCW, U><<<(unsigned)(tiles < wave ? tiles : wave), 256, 0, st>>>(Z, ldz, Kp, j, w, ks, partials, eta, fmode);
}
template <int NCW>
static void cgs_upd_proj_launch(const float* Z, int64_t ldz, int64_t Kp, int j, float* w, KState* ks, double* partials,
                                double eta, int fmode, cudaStream_t st) {
  static const unsigned wave = wave_grid(cgs_upd_proj_kernel<NCW>, (int64_t)RED_BLOCKS * 256);
  constexpr int TR = 32 * VecN<float>::N;
  const int64_t tiles = (Kp + TR - 1) / TR;
  cgs_upd_proj_kernel<NCW><<<(unsigned)(tiles < wave ? tiles : wave), 256, 0, st>>>(Z, ldz, Kp, j, w, ks, partials, eta, fmode);
}

// Which kernel serves a precision and pass.  Measured on GB300 (192 x 64 bump and 48^3
// tetrahedra): the FP32 projections gain from the column split (fewer registers, more loads in
// flight); the FP64 passes are bound by the FP64 pipe and the update-and-norm pass keeps one
// accumulator, so the row kernel's single barrier-free sweep is faster for those.
template <class T, int MODE>
static void cgs_dispatch(int nc, const T* Z, int64_t ldz, int64_t Kp, int j, T* w, T* out, KState* ks,
                         double* partials, double eta, int fmode, cudaStream_t st) {
  if constexpr (sizeof(T) == 4 && MODE == CGS_PROJ) {
    if (nc <= CGS_WARPS) cgs_proj_launch<1, 4>(Z, ldz, Kp, j, w, ks, partials, eta, fmode, st);
    else if (nc <= 2 * CGS_WARPS) cgs_proj_launch<2, 3>(Z, ldz, Kp, j, w, ks, partials, eta, fmode, st);
    else if (nc <= 3 * CGS_WARPS) cgs_proj_launch<3, 4>(Z, ldz, Kp, j, w, ks, partials, eta, fmode, st);
    else cgs_proj_launch<4, 4>(Z, ldz, Kp, j, w, ks, partials, eta, fmode, st);
  } else if constexpr (sizeof(T) == 4 && MODE == CGS_UPD_PROJ) {
    if (nc <= CGS_WARPS) cgs_upd_proj_launch<1>(Z, ldz, Kp, j, w, ks, partials, eta, fmode, st);
    else if (nc <= 2 * CGS_WARPS) cgs_upd_proj_launch<2>(Z, ldz, Kp, j, w, ks, partials, eta, fmode, st);
    else cgs_upd_proj_launch<4>(Z, ldz, Kp, j, w, ks, partials, eta, fmode, st);
  } else {
    if (nc <= 4) cgs_launch<T, 4, MODE>(Z, ldz, Kp, j, w, out, ks, partials, eta, fmode, st);
    else if (nc <= 8) cgs_launch<T, 8, MODE>(Z, ldz, Kp, j, w, out, ks, partials, eta, fmode, st);
    else if (nc <= 16) cgs_launch<T, 16, MODE>(Z, ldz, Kp, j, w, out, ks, partials, eta, fmode, st);
    else cgs_launch<T, 32, MODE>(Z, ldz, Kp, j, w, out, ks, partials, eta, fmode, st);
  }
}

template <class T>
cudaError_t launch_cgs(int mode, const T* Z, int64_t ldz, int64_t Kp, int j, T* w, T* out, KState* ks,
                       double* partials, double eta, cudaStream_t st) {
  const int nc = j + 1;
  if (nc > MMAX) return cudaErrorInvalidValue;
  switch (mode) {
    case CGS_NORM: cgs_launch<T, 0, CGS_NORM>(Z, ldz, Kp, j, w, out, ks, partials, eta, mode, st); break;
    case CGS_PROJ:
    case CGS_PROJ2: cgs_dispatch<T, CGS_PROJ>(nc, Z, ldz, Kp, j, w, out, ks, partials, eta, mode, st); break;
    case CGS_UPD_PROJ: cgs_dispatch<T, CGS_UPD_PROJ>(nc, Z, ldz, Kp, j, w, out, ks, partials, eta, mode, st); break;
    case CGS_UPD_NORM:
    case CGS_UPD1: cgs_dispatch<T, CGS_UPD_NORM>(nc, Z, ldz, Kp, j, w, out, ks, partials, eta, mode, st); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// ------------------------------------------------ a whole Gram-Schmidt column in one launch
// One cooperative kernel does what the separate passes do for column j: project, update, and
// (CGS2, or where the selective form's first pass cancelled) project and update again.  A block
// owns a contiguous range of rows and keeps its part of w in shared memory from the load to the
// last update, so only the basis is read per sweep.
//
// Why: on vectors of up to a few MB the separate launches are bound by their tails, not by their
// sweeps.  Each of them drains, reduces its block sums in one last block and starts the next
// (8 to 30 us a pass in FP64 and 5 to 9 us in FP32 against 1 to 8 us of arithmetic), the
// selective form pays two more launches that leave at once, and a row per thread puts a
// 27,648-entry FP64 vector on 54 of the 152 SMs.  Here the rows are spread over up to all SMs and a sweep
// ends in an all-to-all exchange of the block sums through L2 instead of a launch: every block
// stores its sums and adds up all blocks' itself, in a fixed order.  A slot starts as a bit
// pattern that no arithmetic result has, so a value is its own flag and the exchange takes one
// store and one load, no counter.
// An EXP1 step with 30 columns on periodic triangles at p = 2, separate -> one launch:
//   FP64  K = 27,648 2010 -> 1274 us, 150,528 2810 -> 2230, 591,408 6641 -> 5960,
//         1,503,792 14.04 -> 13.49 ms, 1,881,792 (97 KB per block) 17.49 -> 16.98 ms
//   FP32, selective  K = 12,288 733 -> 602 us, 110,592 832 -> 708, 591,408 1176 -> 1011,
//         1,080,000 (28 KB per block) 1791 -> 1649; one block of 80 registers per SM took 2257 as
//         the separate passes on 1,503,792 (39 KB) and 3719 against 3560 on 2,764,800 (71 KB)
// hence COLUMN_MAX_BYTES: 100 KB of rows per block in FP64 (longer ones were not tried), 32 KB in
// FP32.
// The projection gives each warp its own columns (one accumulator, so one warp sum per column:
// the FP64 additions of a 32-column butterfly in every warp cost as much as the sweep of a small
// vector); the update gives each thread its own rows.
constexpr int COL_NT = 512, COL_WARPS = COL_NT / 32;
// An empty slot: a NaN, as a double and as a pair of floats alike; sums with that bit pattern are
// stored as another NaN.
constexpr unsigned long long COL_EMPTY = ~0ull;

template <class T> struct ColumnSmem {
  alignas(16) T upd[COL_NT * VecN<T>::N];  // partial updates of the column groups (16-byte accesses)
  Acc<T> lanes[(MMAX + 1) * 32];           // per column: the projection's lane sums
  Acc<T> gather[COL_WARPS][COL_SUMS];      // per warp: sums of the blocks it adds
  Acc<T> sums[COL_SUMS];                   // this block's sums
  double dots[COL_SUMS];                   // the grid's sums
  double scale[MMAX + 1];                  // s_i
  T coef[MMAX + 1];
  int bad, late;
};

PCEXP_DEV unsigned long long column_peek(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// The grid's sums of sm.sums[0..n) -> sm.dots, identical in every block.  False if a block's sums
// did not arrive within the limit of polls (ks->err = 2, *lost = 1).  Every thread of every block calls this;
// slots: [block][COL_SUMS], empty before, used by this reduction alone.
template <class T>
PCEXP_DEV bool column_grid_sum(ColumnSmem<T>& sm, int n, unsigned long long* slots, KState* ks, unsigned limit,
                               int* lost) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nblk = gridDim.x;
  __syncthreads();
  if (threadIdx.x == 0) sm.late = 0;
  for (int c = threadIdx.x; c < n; c += COL_NT) {
    unsigned long long v = *reinterpret_cast<const unsigned long long*>(&sm.sums[c]);
    if (v == COL_EMPTY) v >>= 1;  // a propagated input NaN of that payload: another NaN
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(slots + (int64_t)blockIdx.x * COL_SUMS + c), "l"(v)
                 : "memory");
  }
  bool late = false;
  if (n == 1) {  // thread = block; the warps that hold blocks add up theirs
    const int q = threadIdx.x, nw = (nblk + 31) / 32;
    if (wid < nw) {
      unsigned long long v = q < nblk ? COL_EMPTY : 0ull;
      for (unsigned polls = 0; v == COL_EMPTY && polls < limit; ++polls) v = column_peek(slots + (int64_t)q * COL_SUMS);
      late = v == COL_EMPTY;
      Acc<T> a = *reinterpret_cast<const Acc<T>*>(&v);
      for (int o = 16; o > 0; o >>= 1) a.add_partner(o);
      if (lane == 0) sm.gather[wid][0] = a;
    }
  } else {  // warp = every COL_WARPS-th block, lane = column
    constexpr int PER = COL_MAX_BLOCKS / COL_WARPS;
    for (int c = lane; c < n; c += 32) {
      unsigned long long v[PER] = {};
      bool all = false;
      for (unsigned polls = 0; !all && polls < limit; ++polls) {
        all = true;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
          const int q = wid + i * COL_WARPS;
          v[i] = q < nblk ? column_peek(slots + (int64_t)q * COL_SUMS + c) : 0ull;
          all = all && v[i] != COL_EMPTY;
        }
      }
      late = late || !all;
      Acc<T> a = *reinterpret_cast<const Acc<T>*>(&v[0]);
#pragma unroll
      for (int i = 1; i < PER; ++i) a.add_acc(*reinterpret_cast<const Acc<T>*>(&v[i]));
      sm.gather[wid][c] = a;
    }
  }
  if (late) sm.late = 1;
  __syncthreads();
  if (sm.late) {
    if (threadIdx.x == 0) {
      ks->err = 2;
      ks->done = 1;
      if (lost) *(volatile int*)lost = 1;
    }
    return false;
  }
  if (n == 1) {
    if (threadIdx.x == 0) {
      Acc<T> a = sm.gather[0][0];
      for (int q = 1; q < (nblk + 31) / 32; ++q) a.add_acc(sm.gather[q][0]);
      sm.dots[0] = a.value();
    }
  } else {  // 16 threads per column add the warps' sums (warps without columns stay out)
    static_assert(COL_WARPS == 16, "one thread per warp's sum");
    for (int c0 = 2 * wid; c0 < n; c0 += 2 * COL_WARPS) {
      const int c = c0 + lane / 16, q = lane % 16;
      Acc<T> a;
      a.zero();
      if (c < n) a = sm.gather[q][c];
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) a.add_partner(o);
      if (c < n && q == 0) sm.dots[c] = a.value();
    }
  }
  __syncthreads();
  return true;
}

// sm.sums[c] = <z_c, x> for c < nc and, with the norm, sm.sums[nc] = <x, x>, over this block's
// nch chunks x (shared memory); Zb: the first column at the block's first row
template <class T>
PCEXP_DEV void column_project(ColumnSmem<T>& sm, const T* xs, const T* __restrict__ Zb, int64_t ldz, int nc, bool norm,
                              int nch) {
  constexpr int VN = VecN<T>::N;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int ncols = nc + (norm ? 1 : 0);
  // warps: CG column groups times RS shares of the rows
  int CG = 1;
  while (CG < ncols && CG < COL_WARPS) CG *= 2;
  const int RS = COL_WARPS / CG, rs = wid / CG;
  for (int c = wid % CG; c < ncols; c += CG) {
    Acc<T> acc;
    acc.zero();
    const T* z = Zb + (int64_t)c * ldz;
    if (c < nc) {
#pragma unroll 4
      for (int ch = rs * 32 + lane; ch < nch; ch += RS * 32) {
        T a[VN], x[VN];
        load_vec<T, VN>(z + ch * VN, a);
        load_vec<T, VN>(xs + ch * VN, x);
        acc_dot<T, VN>(acc, a, x);
      }
    } else {
      for (int ch = rs * 32 + lane; ch < nch; ch += RS * 32) {
        T x[VN];
        load_vec<T, VN>(xs + ch * VN, x);
        acc_dot<T, VN>(acc, x, x);
      }
    }
    sm.lanes[(c * RS + rs) * 32 + lane] = acc;  // c RS < 16 or RS = 1: within (MMAX + 1) * 32
  }
  __syncthreads();
  int TPC = 32;  // threads per column
  while (TPC * ncols > COL_NT) TPC /= 2;
  const int c = threadIdx.x / TPC, part = threadIdx.x % TPC;
  if (wid * (32 / TPC) < ncols) {  // warp-uniform
    Acc<T> a;
    a.zero();
    if (c < ncols) {
      a = sm.lanes[c * RS * 32 + part];
      for (int i = part + TPC; i < RS * 32; i += TPC) a.add_acc(sm.lanes[c * RS * 32 + i]);
    }
    for (int o = TPC / 2; o > 0; o >>= 1) a.add_partner(o);
    if (c < ncols && part == 0) sm.sums[c] = a;
  }
}

// x -= sum_c coef_c z_c over this block's rows, in shared memory and to outb, and
// sm.sums[0] = <x, x>
template <class T>
PCEXP_DEV void column_update(ColumnSmem<T>& sm, T* xs, T* __restrict__ outb, const T* __restrict__ Zb, int64_t ldz,
                             int nc, int nch) {
  constexpr int VN = VecN<T>::N;
  constexpr int U = 8;
  Acc<T> acc;
  acc.zero();
  // few chunks: G groups of threads share the columns, so that the loads of a chunk's columns are
  // in flight together
  const int G = nch > 0 && nch * 2 <= COL_NT ? min(8, COL_NT / nch) : 1;
  if (G > 1) {
    const int g = threadIdx.x / nch, ch = threadIdx.x - g * nch;
    if (g < G) {
      T p[VN];
#pragma unroll
      for (int v = 0; v < VN; ++v) p[v] = T(0);
#pragma unroll 4
      for (int c = g; c < nc; c += G) {
        T z[VN];
        load_vec<T, VN>(Zb + (int64_t)c * ldz + ch * VN, z);
        const T cf = sm.coef[c];
#pragma unroll
        for (int v = 0; v < VN; ++v) p[v] = fma(cf, z[v], p[v]);
      }
      store_vec<T, VN>(sm.upd + threadIdx.x * VN, p);
    }
    __syncthreads();
    if ((int)threadIdx.x < nch) {
      T x[VN];
      load_vec<T, VN>(xs + threadIdx.x * VN, x);
      for (int q = 0; q < G; ++q) {
        T p[VN];
        load_vec<T, VN>(sm.upd + (q * nch + threadIdx.x) * VN, p);
#pragma unroll
        for (int v = 0; v < VN; ++v) x[v] -= p[v];
      }
      store_vec<T, VN>(xs + threadIdx.x * VN, x);
      store_vec<T, VN>(outb + threadIdx.x * VN, x);
      acc_dot<T, VN>(acc, x, x);
    }
  } else {
    for (int ch = threadIdx.x; ch < nch; ch += COL_NT) {
      T x[VN];
      load_vec<T, VN>(xs + ch * VN, x);
      for (int c0 = 0; c0 < nc; c0 += U) {
        T z[U][VN];
#pragma unroll
        for (int g = 0; g < U; ++g) load_vec<T, VN>(Zb + (int64_t)min(c0 + g, nc - 1) * ldz + ch * VN, z[g]);
#pragma unroll
        for (int g = 0; g < U; ++g)
          if (c0 + g < nc)
#pragma unroll
            for (int v = 0; v < VN; ++v) x[v] = fma(-sm.coef[c0 + g], z[g][v], x[v]);
      }
      store_vec<T, VN>(xs + ch * VN, x);
      store_vec<T, VN>(outb + ch * VN, x);
      acc_dot<T, VN>(acc, x, x);
    }
  }
  sm.lanes[threadIdx.x] = acc;
  __syncthreads();
  if (threadIdx.x < 64) {
    Acc<T> a = sm.lanes[threadIdx.x];
#pragma unroll
    for (int i = 1; i < COL_NT / 64; ++i) a.add_acc(sm.lanes[threadIdx.x + 64 * i]);
    for (int o = 16; o > 0; o >>= 1) a.add_partner(o);
    if (threadIdx.x == 32) sm.sums[1] = a;
    if (threadIdx.x == 0) sm.sums[0] = a;
  }
  __syncthreads();
  if (threadIdx.x == 0) sm.sums[0].add_acc(sm.sums[1]);
}

// coefficients of the next update from the projections sm.dots (the scalar step of cgs_finalize's
// PROJ and UPD_PROJ), in every block; block 0 records them.  False on a non-finite entry.
template <class T>
PCEXP_DEV bool column_coefficients(ColumnSmem<T>& sm, int j, bool first, KState* ks) {
  if (threadIdx.x == 0) sm.bad = 0;
  __syncthreads();
  for (int i = threadIdx.x; i <= j; i += COL_NT) {
    const double si = sm.scale[i], h = si * sm.dots[i];
    if (!isfinite(h)) sm.bad = 1;
    sm.coef[i] = (T)(si * h);
    if (blockIdx.x == 0) {
      if (first) {
        ks->H[i * MMAX + j] = h;
        ks->H1[i * MMAX + j] = h;
      } else {
        ks->H[i * MMAX + j] += h;
      }
    }
  }
  __syncthreads();
  if (sm.bad && blockIdx.x == 0 && threadIdx.x == 0) {
    ks->err = 1;
    ks->done = 1;
  }
  return !sm.bad;
}

// rows: of one block (a multiple of 64; the last block may have fewer).  slots: two sets
// of four reductions' slots; column j uses set j & 1 and empties the other for column j + 1 (set
// 0 is emptied by reset_kstate before column 0).
template <class T>
__global__ void __launch_bounds__(COL_NT, 2) cgs_column_kernel(const T* __restrict__ Z, int64_t ldz, int64_t Kp, int j,
                                                               const T* __restrict__ w, T* __restrict__ out,
                                                               KState* ks, unsigned long long* slots, double eta,
                                                               int rows, int selective, unsigned limit, int* lost) {
  constexpr int VN = VecN<T>::N;
  extern __shared__ __align__(16) unsigned char col_dyn[];
  __shared__ __align__(16) ColumnSmem<T> sm;
  static_assert(offsetof(ColumnSmem<T>, upd) % 16 == 0, "16-byte accesses");
  // uniform over the grid: done is raised only after the sums of every block have been seen below
  if (ks->done) return;
  T* xs = reinterpret_cast<T*>(col_dyn);
  const int64_t r0 = (int64_t)blockIdx.x * rows;
  const int64_t left = Kp - r0;
  const int nch = left <= 0 ? 0 : (int)((left < rows ? left : rows) / VN);
  const T* Zb = Z + r0;
  T* outb = out + r0;
  const int nc = j + 1;
  const int64_t red = (int64_t)gridDim.x * COL_SUMS;  // slots of one reduction
  unsigned long long* mine = slots + (j & 1) * 4 * red;
  {
    unsigned long long* other = slots + ((j + 1) & 1) * 4 * red + (int64_t)blockIdx.x * COL_SUMS;
    for (int i = threadIdx.x; i < 4 * COL_SUMS; i += COL_NT) other[i / COL_SUMS * red + i % COL_SUMS] = COL_EMPTY;
  }
  for (int i = threadIdx.x; i < nc; i += COL_NT) sm.scale[i] = ks->s[i];
  for (int ch = threadIdx.x; ch < nch; ch += COL_NT) {
    T x[VN];
    load_vec<T, VN>(w + r0 + ch * VN, x);
    store_vec<T, VN>(xs + ch * VN, x);
  }
  __syncthreads();
  column_project<T>(sm, xs, Zb, ldz, nc, true, nch);
  if (!column_grid_sum<T>(sm, nc + 1, mine, ks, limit, lost)) return;
  const double wnorm0 = sqrt(sm.dots[nc]);
  if (!column_coefficients<T>(sm, j, true, ks)) return;
  column_update<T>(sm, xs, outb, Zb, ldz, nc, nch);
  if (selective) {
    // keep the first pass when it cancelled less than DGKS_KAPPA (cgs_finalize's UPD1)
    if (!column_grid_sum<T>(sm, 1, mine + red, ks, limit, lost)) return;
    const double n1 = sqrt(sm.dots[0]);
    if (isfinite(n1) && n1 > 0.0 && n1 >= DGKS_KAPPA * wnorm0) {
      if (blockIdx.x == 0 && threadIdx.x == 0) {
        ks->H[(j + 1) * MMAX + j] = n1;
        ks->k = j + 1;
        ks->s[j + 1] = 1.0 / n1;
      }
      return;
    }
  }
  __syncthreads();
  column_project<T>(sm, xs, Zb, ldz, nc, false, nch);
  if (!column_grid_sum<T>(sm, nc, mine + 2 * red, ks, limit, lost)) return;
  if (!column_coefficients<T>(sm, j, false, ks)) return;
  column_update<T>(sm, xs, outb, Zb, ldz, nc, nch);
  if (!column_grid_sum<T>(sm, 1, mine + 3 * red, ks, limit, lost)) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const double hn = sqrt(sm.dots[0]);
    ks->pass2 |= 1u << j;
    ks->H[(j + 1) * MMAX + j] = hn;
    ks->k = j + 1;
    if (!isfinite(hn)) {
      ks->err = 1;
      ks->done = 1;
    } else if (hn == 0.0 || hn <= eta * wnorm0) {
      ks->done = 1;  // happy breakdown: K_{j+1} is invariant
    } else {
      ks->s[j + 1] = 1.0 / hn;
    }
  }
}

// Blocks of a column: at most one per SM, each with at least COLUMN_MIN_ROWS rows.  Every block adds up
// all blocks' sums, and contexts on several streams run side by side only while their grids fit the
// chip together (two blocks per SM: 64 registers, and up to 90 KB of rows).  Time of a PCEXP step in
// one context / of each when four threads step a context each (us), on one block per SM whatever K ->
// this rule (the separate passes):
//   FP64  K = 6,144, m = 10      778 / 1694 -> 762 / 817   (1191 / 1313)
//         K = 27,648, m = 30     2508 / 6958 -> 2544 / 5157 (4268 / 5151)
//         K = 110,592, m = 30    3850 / 12506 -> 3847 / 11684 (5871 / 11129)
//   FP32  K = 6,144, m = 10      441 / 966 -> 413 / 462    (582 / 688)
//         K = 27,648, m = 30     1278 / 3104 -> 1220 / 1393 (1950 / 2224)
//         K = 110,592, m = 30    1401 / 3573 -> 1355 / 2210 (2091 / 3020)
//         K = 442,368, m = 30    1708 / 6009 -> 1674 / 5006 (2714 / 5977)
// Fewer, longer blocks help several contexts further and cost the single one: FP64 K = 27,648 with 320
// rows 2594 / 4609, with 192 rows 2493 / 5801; FP32 K = 110,592 with 2,048 rows 1381 / 2063.
template <class T>
ColumnPlan plan_cgs_column(int64_t Kp) {
  ColumnPlan plan{0, 0, COL_POLLS, nullptr};
  int dev = 0, sms = 0, coop = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop)
    return plan;
  const int64_t most = sms < COL_MAX_BLOCKS ? sms : COL_MAX_BLOCKS, share = (Kp + most - 1) / most;
  const int64_t rows = ((share > COLUMN_MIN_ROWS<T> ? share : COLUMN_MIN_ROWS<T>) + VPAD - 1) / VPAD * VPAD;
  const int64_t bytes = rows * (int64_t)sizeof(T);
  if (bytes > COLUMN_MAX_BYTES<T>) return plan;
  // every block of the grid must be resident (they exchange sums): at most one per SM
  if (cudaFuncSetAttribute(cgs_column_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)COLUMN_MAX_BYTES<T>) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, cgs_column_kernel<T>, COL_NT, (size_t)bytes) !=
          cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    return plan;
  }
  plan.blocks = (int)((Kp + rows - 1) / rows);
  plan.rows = (int)rows;
  return plan;
}

template <class T>
cudaError_t launch_cgs_column(const ColumnPlan& plan, const T* Z, int64_t ldz, int64_t Kp, int j, const T* w, T* out,
                              KState* ks, unsigned long long* slots, double eta, bool selective, cudaStream_t st) {
  if (j + 1 > MMAX || plan.blocks < 1) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = dim3((unsigned)plan.blocks);
  cfg.blockDim = dim3(COL_NT);
  cfg.dynamicSmemBytes = (size_t)plan.rows * sizeof(T);
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, cgs_column_kernel<T>, Z, ldz, Kp, j, w, out, ks, slots, eta, plan.rows,
                            selective ? 1 : 0, plan.polls, plan.lost);
}

// ------------------------------------------------ Gram-Schmidt of a partitioned run
__global__ void __launch_bounds__(256) cgs_group_finalize_kernel(int mode, int j, KState* ks, double eta) {
  __shared__ double dots[MMAX + 2];
  if (ks->done) return;  // the pass did not run (uniform)
  if (cgs_skipped(mode, ks)) return;  // the pass did not run (uniform)
  for (int c = threadIdx.x; c < MMAX + 2; c += blockDim.x) dots[c] = ks->gtot[c];
  __syncthreads();
  cgs_finalize(mode, j, dots, ks, eta);
}
cudaError_t launch_cgs_group_finalize(int mode, int j, KState* ks, double eta, cudaStream_t st) {
  cgs_group_finalize_kernel<<<1, 256, 0, st>>>(mode, j, ks, eta);
  return cudaGetLastError();
}

__global__ void group_reduce_kernel(PartPtrs slots, int nparts, int n, double* out, int op) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    double a = reinterpret_cast<const double*>(slots.p[0])[i];
    for (int q = 1; q < nparts; ++q) {
      const double b = reinterpret_cast<const double*>(slots.p[q])[i];
      a = op == 1 ? fmin(a, b) : a + b;
    }
    out[i] = a;
  }
}
cudaError_t launch_group_reduce(PartPtrs slots, int nparts, int n, double* out, int op, cudaStream_t st) {
  group_reduce_kernel<<<1, 64, 0, st>>>(slots, nparts, n, out, op);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ phi kernel
// exp(A) by scaling and squaring of the Taylor polynomial of degree 16 at X = A / 2^s with
// ||X||_1 <= 1/2 (remainder (1/2)^17 / 17! < 3e-20, far below FP64 rounding; Paterson &
// Stockmeyer 1973 for the evaluation).
// For phi: A = [[dt H_k, e_1, 0], [0, 0, 1], [0, 0, 0]]; column k of exp(A) holds
// phi_1(dt H) e_1 and column k+1 holds phi_2(dt H) e_1.
//
// The kernels are bound by the FP64 pipe of the SMs they run on (2 FMA per clock and SM: one
// (m+2)^3 product costs one SM ~10 us) and by the chain of products.  They run as a cluster of
// PHI_CTAS CTAs: every CTA keeps a full copy of the matrices in shared memory (5 buffers),
// computes its share of the rows of each product and writes them into every CTA of the cluster
// (distributed shared memory), then the cluster barrier publishes them.  A polynomial needs no
// linear solve: a rational approximant's LU is a serial chain of m+2 pivot columns repeated in
// every CTA (two thirds of the kernel's time with the [8/8] Pade form, 157 us at k = 30 on the
// 192 x 64 bump against 36 us).  Of its six products, X^3 and X^4 share one phase, and the
// three Horner steps P X^4 + B need only the CTA's own rows of P, hence no cluster barrier.  The
// last product forms only the columns the caller reads.
constexpr int PN = MMAX + 2;      // phi: (m+2) x (m+2)
constexpr int PN2 = 2 * PN;       // phi adjoint: block-triangular 2 (m+2) x 2 (m+2)
constexpr int PHI_CTAS = 8;

namespace cg = cooperative_groups;

// sum_l a[l] B[l][0], two accumulators (the FP64 latency is longer than the issue interval of a
// CTA's few warps)
template <int LD>
PCEXP_DEV double dot_col(const double* a, const double* B, int n, double init) {
  double s0 = init, s1 = 0;
  int l = 0;
#pragma unroll 2
  for (; l + 1 < n; l += 2) {
    s0 = fma(a[l], B[l * LD], s0);
    s1 = fma(a[l + 1], B[(l + 1) * LD], s1);
  }
  if (l < n) s0 = fma(a[l], B[l * LD], s0);
  return s0 + s1;
}

// Columns [c0, c0 + nc) of this CTA's rows (i = rank, rank + PHI_CTAS, ...) of A B, written into
// the first `dst` CTAs of the cluster.  The caller synchronises.
template <int LD>
__device__ void mat_mul_rows(cg::cluster_group& cl, const double* A, const double* B, double* C, int n, int c0, int nc,
                             int dst) {
  const int rank = (int)cl.block_rank();
  const int nrow = (n - rank + PHI_CTAS - 1) / PHI_CTAS;
  for (int t = threadIdx.x; t < nrow * nc; t += blockDim.x) {
    const int i = rank + (t / nc) * PHI_CTAS, jj = c0 + t % nc;
    const double a = dot_col<LD>(A + i * LD, B + jj, n, 0.0);
    for (int r = 0; r < dst; ++r) cl.map_shared_rank(C, r)[i * LD + jj] = a;
  }
}

// 1 / j! to the last bit of a double division of exact integers (16! < 2^53)
PCEXP_DEV constexpr double inv_factorial(int j) {
  double f = 1.0;
  for (int i = 2; i <= j; ++i) f *= i;
  return 1.0 / f;
}

// exp of the n x n matrix held (identically) in buffer A of every CTA of the cluster.
// sm holds 5 LD x LD buffers; returns the buffer with the result, or nullptr if the input is
// not finite.  With nc == n the result is complete in all CTAs; with nc < n only its columns
// [c0, c0 + nc) are formed, in CTA 0.  Must be called by all threads of all CTAs.
template <int LD>
__device__ double* expm_cluster(cg::cluster_group& cl, double* sm, int n, int c0, int nc) {
  double* A = sm;
  double* X2 = A + LD * LD;
  double* X3 = X2 + LD * LD;
  double* X4 = X3 + LD * LD;
  double* Y = X4 + LD * LD;
  constexpr int LROWS = (LD + PHI_CTAS - 1) / PHI_CTAS;
  __shared__ double prow[2][LROWS * LD];  // this CTA's rows of the Horner polynomials
  __shared__ int s_sq;
  __shared__ float colsum[4][LD];
  const int rank = (int)cl.block_rank();
  // ||A||_1 from parallel column sums in FP32 (it only selects s; the same arithmetic in
  // every CTA gives the same s)
  for (int t = threadIdx.x; t < 4 * n; t += blockDim.x) {
    const int part = t / n, jj = t - part * n;
    float c = 0.f;
    for (int i = part; i < n; i += 4) c += fabsf((float)A[i * LD + jj]);
    colsum[part][jj] = c;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    float m = 0.f;
    bool finite = true;
    for (int jj = threadIdx.x; jj < n; jj += 32) {
      const float c = (colsum[0][jj] + colsum[1][jj]) + (colsum[2][jj] + colsum[3][jj]);
      finite = finite && c <= 3.0e38f;  // false for NaN too
      m = fmaxf(m, c);
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    finite = __all_sync(0xffffffffu, finite);
    if (threadIdx.x == 0) {
      int s = 0;
      if (m > 0.5f) s = (int)ceilf(log2f(m)) + 1;  // ||X||_1 <= 1/2 up to the FP32 estimate's rounding
      if (!finite || s > 1000) s = -1;             // NaN or overflow
      s_sq = s;
    }
  }
  __syncthreads();
  const int sq = s_sq;
  if (sq < 0) return nullptr;  // uniform across the cluster (same data, same arithmetic)
  const double sc = ldexp(1.0, -sq);
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) A[(t / n) * LD + t % n] *= sc;
  cl.sync();  // every CTA runs and has its scaled A before remote products land
  mat_mul_rows<LD>(cl, A, A, X2, n, 0, n, PHI_CTAS);
  cl.sync();
  mat_mul_rows<LD>(cl, X2, A, X3, n, 0, n, PHI_CTAS);
  mat_mul_rows<LD>(cl, X2, X2, X4, n, 0, n, PHI_CTAS);
  cl.sync();
  // P = c16 X4 + B_3, then P <- P X4 + B_k for k = 2, 1, 0 with
  // B_k = c_4k I + c_4k+1 X + c_4k+2 X2 + c_4k+3 X3; the last one goes to every CTA
  const int nrow = (n - rank + PHI_CTAS - 1) / PHI_CTAS;
  constexpr double c[17] = {inv_factorial(0),  inv_factorial(1),  inv_factorial(2),  inv_factorial(3),
                            inv_factorial(4),  inv_factorial(5),  inv_factorial(6),  inv_factorial(7),
                            inv_factorial(8),  inv_factorial(9),  inv_factorial(10), inv_factorial(11),
                            inv_factorial(12), inv_factorial(13), inv_factorial(14), inv_factorial(15),
                            inv_factorial(16)};
#pragma unroll
  for (int k = 3; k >= 0; --k) {
    const double* P = prow[(k & 1) ^ 1];  // of the previous step
    for (int t = threadIdx.x; t < nrow * n; t += blockDim.x) {
      const int r = t / n, i = rank + r * PHI_CTAS, jj = t - r * n, o = i * LD + jj;
      double b = fma(c[4 * k + 3], X3[o], fma(c[4 * k + 2], X2[o], c[4 * k + 1] * A[o]));
      if (i == jj) b += c[4 * k];
      if (k == 3) b = fma(c[16], X4[o], b);
      else b = dot_col<LD>(P + r * LD, X4 + jj, n, b);
      if (k > 0) {
        prow[k & 1][r * LD + jj] = b;
      } else {
        for (int q = 0; q < PHI_CTAS; ++q) cl.map_shared_rank(Y, q)[o] = b;
      }
    }
    if (k > 0) __syncthreads();
  }
  cl.sync();
  double* X = Y;
  double* Z = X2;
  for (int it = 0; it < sq; ++it) {
    const bool part = it == sq - 1 && nc < n;
    mat_mul_rows<LD>(cl, X, X, Z, n, part ? c0 : 0, part ? nc : n, part ? 1 : PHI_CTAS);
    cl.sync();
    double* t = X;
    X = Z;
    Z = t;
  }
  return X;
}

// which = 1: the update coefficients use phi_1(dt H) e_1 (Eq. s8, s9, s10); which = 2: they use
// phi_2(dt H) e_1 (the ETD2 term of Eq. s7), times dt / *dt_prev when dt_prev is given.
//
// Every evaluation also forms the relative a-posteriori error estimate of the Krylov phi_1
// product (Saad 1992, the leading term of the error of Eq. final),
//   est = dt h_{k+1,k} |e_k^T phi_2(dt H_k) e_1| / ||phi_1(dt H_k) e_1||,
// from the phi_2 column of the same exponential.  check_tol > 0 is a checkpoint of the
// adaptive dimension: only est is formed, and ks->done is raised when est <= check_tol.
// The scalars at the end run on one warp, an entry of y per lane.
__global__ void __cluster_dims__(PHI_CTAS, 1, 1) __launch_bounds__(256)
    phi_kernel(KState* ks, const double* dt_dev, double dt_host, double factor, StepState* ss, int stage, int which,
               const double* dt_prev, double check_tol) {
  extern __shared__ double sm[];
  static_assert(MMAX <= 32, "one lane per Krylov column");
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank();
  const int k = ks->k;
  const double dt = dt_dev ? *dt_dev : dt_host;
  if (check_tol > 0.0 && (k == 0 || ks->err || ks->done)) return;  // uniform across the cluster
  if (k == 0 || ks->err) {  // uniform across the cluster: no shared-memory traffic happens
    if (rank == 0 && threadIdx.x == 0) {
      for (int i = 0; i <= MMAX; ++i) ks->acoef[i] = 0.0;
      if (ss) {
        ss->k[stage] = 0;
        ss->beta[stage] = ks->beta;
        ss->pass2[stage] = ks->pass2;
        if (ks->err) ss->err = ks->err;
      }
    }
    return;
  }
  const int n = k + 2;
  double* A = sm;
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
    const int i = t / n, jj = t - i * n;
    double a = 0.0;
    if (i < k && jj < k) a = dt * ks->H[i * MMAX + jj];
    else if ((i == 0 && jj == k) || (i == k && jj == k + 1)) a = 1.0;
    A[i * PN + jj] = a;
  }
  __syncthreads();
  const double* X = expm_cluster<PN>(cl, sm, n, k, 2);
  if (rank != 0 || threadIdx.x >= 32) return;
  const int i = threadIdx.x;
  if (!X) {
    if (i == 0) {
      ks->err = 1;
      if (ss) ss->err = 1;
    }
    return;
  }
  const double y1 = i < k ? X[i * PN + k] : 0.0, y2 = i < k ? X[i * PN + k + 1] : 0.0;
  double n1 = y1 * y1;
  for (int o = 16; o > 0; o >>= 1) n1 += __shfl_xor_sync(0xffffffffu, n1, o);
  const double est = dt * fabs(ks->H[k * MMAX + k - 1]) * fabs(__shfl_sync(0xffffffffu, y2, k - 1)) / sqrt(n1);
  if (i == 0) ks->err_est = est;
  if (check_tol > 0.0) {
    if (i == 0 && est <= check_tol) ks->done = 1;  // the estimate may be NaN: then the process goes on
    return;
  }
  const double beta = ks->beta;
  const double f = dt_prev ? factor * dt / *dt_prev : factor;
  const double ac = i < k ? f * dt * beta * (which == 2 ? y2 : y1) * ks->s[i] : 0.0;
  const bool ok = __all_sync(0xffffffffu, isfinite(ac));
  if (i < k) {
    ks->y[i] = y1;
    ks->y2[i] = y2;
  }
  ks->acoef[i] = ac;
  if (i != 0) return;
  for (int q = 32; q <= MMAX; ++q) ks->acoef[q] = 0.0;
  if (!ok) ks->err = 1;
  if (ss) {
    ss->k[stage] = k;
    ss->beta[stage] = beta;
    ss->kerr[stage] = est;
    ss->pass2[stage] = ks->pass2;
    if (!ok) ss->err = 1;
  }
}

// Adjoint of y = phi_1(dt H) e_1 (the first k entries of column k of exp(A)):
//   Hbar = dt [L_exp(A^T, Xbar)]_{0:k,0:k},  Xbar = ybar in rows 0..k-1 of column k,
// where L_exp(M, E), the Frechet derivative of exp, is the top-right block of
// exp([[M, E], [0, M]]) (block-triangular identity; Najfeld & Havel 1995).
__global__ void __cluster_dims__(PHI_CTAS, 1, 1) __launch_bounds__(256)
    phi_adjoint_kernel(const double* __restrict__ H, int k, int ldh, double dt, const double* __restrict__ ybar,
                       double* __restrict__ Hbar, int* __restrict__ err) {
  extern __shared__ double sm[];
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank();
  const int n0 = k + 2, n = 2 * n0;
  double* M = sm;
  for (int t = threadIdx.x; t < PN2 * PN2; t += blockDim.x) M[t] = 0.0;
  __syncthreads();
  // M = [[A^T, Xbar], [0, A^T]] with A = [[dt H, e_1, 0], [0, 0, 1], [0, 0, 0]]
  for (int t = threadIdx.x; t < k * k; t += blockDim.x) {
    const int i = t / k, jj = t - i * k;
    const double a = dt * H[jj * ldh + i];  // (A^T)_{ij} = A_{ji}
    M[i * PN2 + jj] = a;
    M[(n0 + i) * PN2 + n0 + jj] = a;
  }
  for (int t = threadIdx.x; t < k; t += blockDim.x) M[t * PN2 + n0 + k] = ybar[t];
  if (threadIdx.x == 0) {
    M[k * PN2 + 0] = 1.0;  // (A^T)_{k,0} = A_{0,k} = 1
    M[(k + 1) * PN2 + k] = 1.0;
    M[(n0 + k) * PN2 + n0 + 0] = 1.0;
    M[(n0 + k + 1) * PN2 + n0 + k] = 1.0;
  }
  __syncthreads();
  const double* X = expm_cluster<PN2>(cl, sm, n, 0, n);
  if (rank == 0) {
    if (!X) {
      if (threadIdx.x == 0) *err = 1;
      return;
    }
    for (int t = threadIdx.x; t < k * k; t += blockDim.x) {
      const int i = t / k, jj = t - i * k;
      Hbar[i * ldh + jj] = dt * X[i * PN2 + n0 + jj];
    }
  }
}

// Raises a kernel's dynamic shared-memory limit on the current device, once per device (bits of
// done): the limit belongs to the device's context.
static cudaError_t allow_shared(const void* kernel, size_t bytes, std::atomic<unsigned long long>& done) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
  if (done.load() & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) done.fetch_or(bit);
  return e;
}
static cudaError_t phi_smem_attr(size_t smem) {
  static std::atomic<unsigned long long> done{0};
  return allow_shared((const void*)phi_kernel, smem, done);
}

cudaError_t launch_phi(KState* ks, const double* dt_dev, double dt, double factor, StepState* ss, int stage,
                       cudaStream_t st, int which, const double* dt_prev) {
  const size_t smem = 5 * PN * PN * sizeof(double);
  cudaError_t e = phi_smem_attr(smem);
  if (e != cudaSuccess) return e;
  phi_kernel<<<PHI_CTAS, 256, smem, st>>>(ks, dt_dev, dt, factor, ss, stage, which, dt_prev, 0.0);
  return cudaGetLastError();
}

cudaError_t launch_phi_check(KState* ks, const double* dt_dev, double tol, cudaStream_t st) {
  const size_t smem = 5 * PN * PN * sizeof(double);
  cudaError_t e = phi_smem_attr(smem);
  if (e != cudaSuccess) return e;
  phi_kernel<<<PHI_CTAS, 256, smem, st>>>(ks, dt_dev, 1.0, 1.0, nullptr, 0, 1, nullptr, tol);
  return cudaGetLastError();
}

cudaError_t launch_phi_adjoint(const double* H, int k, int ldh, double dt, const double* ybar, double* Hbar, int* err,
                               cudaStream_t st) {
  if (k < 1 || k > MMAX) return cudaErrorInvalidValue;
  const size_t smem = 5 * PN2 * PN2 * sizeof(double);
  static std::atomic<unsigned long long> done{0};
  const cudaError_t e = allow_shared((const void*)phi_adjoint_kernel, smem, done);
  if (e != cudaSuccess) return e;
  phi_adjoint_kernel<<<PHI_CTAS, 256, smem, st>>>(H, k, ldh, dt, ybar, Hbar, err);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ axpy
template <class T>
__global__ void __launch_bounds__(256) krylov_axpy_kernel(const double* __restrict__ base64, double* __restrict__ out64,
                                                          T* __restrict__ shadow, T* __restrict__ delta,
                                                          const T* __restrict__ Z, int64_t ldz, int64_t Kp,
                                                          const KState* ks) {
  __shared__ T sc[MMAX];
  const int k = ks->k;
  for (int i = threadIdx.x; i < MMAX; i += blockDim.x) sc[i] = (T)ks->acoef[i];
  __syncthreads();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < Kp; r += stride) {
    T a = 0;
    for (int i = 0; i < k; ++i) a = fma(sc[i], Z[i * ldz + r], a);
    const double o = base64[r] + (double)a;
    out64[r] = o;
    if (delta) delta[r] = a;
    if (shadow && (void*)shadow != (void*)out64) shadow[r] = (T)o;
  }
}

template <class T>
cudaError_t launch_krylov_axpy(const double* base64, double* out64, T* shadow, T* delta, const T* Z, int64_t ldz,
                               int64_t Kp, const KState* ks, cudaStream_t st) {
  int64_t g = (Kp + 255) / 256;
  if (g > 152 * 8) g = 152 * 8;
  krylov_axpy_kernel<T><<<(unsigned)(g < 1 ? 1 : g), 256, 0, st>>>(base64, out64, shadow, delta, Z, ldz, Kp, ks);
  return cudaGetLastError();
}

template <class T>
__global__ void combine_kernel(T* __restrict__ a, const T* __restrict__ b, const T* __restrict__ c, int64_t n) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x)
    a[r] = b[r] - a[r] - c[r];
}
template <class T>
cudaError_t launch_combine_corrector(T* a, const T* b, const T* c, int64_t Kp, cudaStream_t st) {
  int64_t g = (Kp + 255) / 256;
  if (g > 152 * 8) g = 152 * 8;
  combine_kernel<T><<<(unsigned)(g < 1 ? 1 : g), 256, 0, st>>>(a, b, c, Kp);
  return cudaGetLastError();
}

// out = x - y - z (z nullable)
template <class T>
__global__ void lincomb3_kernel(T* __restrict__ out, const T* __restrict__ x, const T* __restrict__ y,
                                const T* __restrict__ z, int64_t n) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x)
    out[r] = z ? x[r] - y[r] - z[r] : x[r] - y[r];
}
template <class T>
cudaError_t launch_lincomb3(T* out, const T* x, const T* y, const T* z, int64_t Kp, cudaStream_t st) {
  int64_t g = (Kp + 255) / 256;
  if (g > 152 * 8) g = 152 * 8;
  lincomb3_kernel<T><<<(unsigned)(g < 1 ? 1 : g), 256, 0, st>>>(out, x, y, z, Kp);
  return cudaGetLastError();
}

template <class Tin, class Tout>
__global__ void cast_kernel(const Tin* __restrict__ x, Tout* __restrict__ y, int64_t n) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x)
    y[r] = (Tout)x[r];
}
template <class Tin, class Tout>
cudaError_t launch_cast(const Tin* x, Tout* y, int64_t n, cudaStream_t st) {
  int64_t g = (n + 255) / 256;
  if (g > 152 * 8) g = 152 * 8;
  cast_kernel<Tin, Tout><<<(unsigned)(g < 1 ? 1 : g), 256, 0, st>>>(x, y, n);
  return cudaGetLastError();
}

__global__ void reset_kstate_kernel(KState* ks, unsigned long long* slots, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) slots[i] = COL_EMPTY;
  if (blockIdx.x != 0) return;
  if (threadIdx.x == 0) {
    ks->k = 0;
    ks->done = 0;
    ks->err = 0;
    ks->counter = 0;
    ks->beta = 0;
    ks->err_est = 0;
    ks->skip2 = 0;
    ks->pass2 = 0u;
  }
  for (int i = threadIdx.x; i < (MMAX + 1) * MMAX; i += blockDim.x) ks->H[i] = 0.0;
}
cudaError_t launch_reset_kstate(KState* ks, cudaStream_t st, unsigned long long* slots, const ColumnPlan* plan) {
  const int n = slots ? 4 * COL_SUMS * plan->blocks : 0;  // the first of the two sets
  reset_kstate_kernel<<<n > 0 ? 32 : 1, 256, 0, st>>>(ks, slots, n);
  return cudaGetLastError();
}

__global__ void set_dt_kernel(StepState* ss, double dt) { ss->dt = dt; }
__global__ void set_cfl_kernel(StepState* ss, double cfl) { ss->cfl = cfl; }
cudaError_t launch_set_cfl(StepState* ss, double cfl, cudaStream_t st) {
  set_cfl_kernel<<<1, 1, 0, st>>>(ss, cfl);
  return cudaGetLastError();
}
__global__ void keep_dt_kernel(StepState* ss) { ss->dt_prev = ss->dt; }
__global__ void cap_cfl_kernel(StepState* ss, double cap) { ss->cfl = fmin(ss->cfl, cap); }
cudaError_t launch_cap_cfl(StepState* ss, double cap, cudaStream_t st) {
  cap_cfl_kernel<<<1, 1, 0, st>>>(ss, cap);
  return cudaGetLastError();
}
cudaError_t launch_keep_dt(StepState* ss, cudaStream_t st) {
  keep_dt_kernel<<<1, 1, 0, st>>>(ss);
  return cudaGetLastError();
}
__global__ void set_param_kernel(double* p, double v) { *p = v; }
__global__ void copy_dt_kernel(StepState* ss, const double* p) { ss->dt = *p; }
cudaError_t launch_set_param(double* param, double v, cudaStream_t st) {
  set_param_kernel<<<1, 1, 0, st>>>(param, v);
  return cudaGetLastError();
}
cudaError_t launch_copy_dt(StepState* ss, const double* param, cudaStream_t st) {
  copy_dt_kernel<<<1, 1, 0, st>>>(ss, param);
  return cudaGetLastError();
}
cudaError_t launch_set_dt(StepState* ss, double dt, cudaStream_t st) {
  set_dt_kernel<<<1, 1, 0, st>>>(ss, dt);
  return cudaGetLastError();
}

template cudaError_t launch_cgs<double>(int, const double*, int64_t, int64_t, int, double*, double*, KState*, double*,
                                        double, cudaStream_t);
template cudaError_t launch_cgs<float>(int, const float*, int64_t, int64_t, int, float*, float*, KState*, double*,
                                       double, cudaStream_t);
template ColumnPlan plan_cgs_column<double>(int64_t);
template ColumnPlan plan_cgs_column<float>(int64_t);
template cudaError_t launch_cgs_column<double>(const ColumnPlan&, const double*, int64_t, int64_t, int, const double*,
                                               double*, KState*, unsigned long long*, double, bool, cudaStream_t);
template cudaError_t launch_cgs_column<float>(const ColumnPlan&, const float*, int64_t, int64_t, int, const float*,
                                              float*, KState*, unsigned long long*, double, bool, cudaStream_t);
template cudaError_t launch_krylov_axpy<double>(const double*, double*, double*, double*, const double*, int64_t,
                                                int64_t, const KState*, cudaStream_t);
template cudaError_t launch_krylov_axpy<float>(const double*, double*, float*, float*, const float*, int64_t,
                                               int64_t, const KState*, cudaStream_t);
template cudaError_t launch_lincomb3<double>(double*, const double*, const double*, const double*, int64_t,
                                             cudaStream_t);
template cudaError_t launch_lincomb3<float>(float*, const float*, const float*, const float*, int64_t, cudaStream_t);
template cudaError_t launch_combine_corrector<double>(double*, const double*, const double*, int64_t, cudaStream_t);
template cudaError_t launch_combine_corrector<float>(float*, const float*, const float*, int64_t, cudaStream_t);
template cudaError_t launch_cast<double, float>(const double*, float*, int64_t, cudaStream_t);
template cudaError_t launch_cast<float, double>(const float*, double*, int64_t, cudaStream_t);
template cudaError_t launch_cast<double, double>(const double*, double*, int64_t, cudaStream_t);

}  // namespace pcexp
