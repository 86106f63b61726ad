// Dimension-free kernels of the DG path: basis conversion at the interface,
// per-element scaling and the density-residual norm of Eq. cfl with the CFL ramp.
#include <cfloat>

#include "kernels.h"

namespace pcexp {

// ------------------------------------------------------------ basis conversion
// Both bases are orthonormal and graded by total degree (each spans P^0, P^1, ... in turn), so
// Q_e couples functions of equal degree only: one block per degree, of 1, 2, 3, 4 (triangles) or
// 1, 3, 6 (tetrahedra) functions, and the degree-0 block is 1.  The blocks of degrees 1..p are
// stored packed, row-major, [E][QN] (pack_basis_change).
//
// A conversion is bound by the FP64 pipe (the FP64 rate is 1/62 of FP32's): the blocks take 45
// instead of 100 FMAs per variable on tetrahedra at p = 2.  One thread per (element, variable)
// row forms the whole row, so a warp runs the same block sizes; rows and blocks are staged in
// shared memory for coalesced global access.  Tetrahedra at p = 2, 33^3 cubes (K = 10.8 M): the
// three conversions of an FP32-mixed J v call (two in, one out) take 357 us together, against 852
// us with a thread per output and the full matrix.
template <int D, int P> struct QBlocks {
  static constexpr int NV = D + 2, NB = D == 2 ? (P + 1) * (P + 2) / 2 : (P + 1) * (P + 2) * (P + 3) / 6;
  __host__ __device__ static constexpr int size(int deg) { return D == 2 ? deg + 1 : (deg + 1) * (deg + 2) / 2; }
  __host__ __device__ static constexpr int first(int deg) { return deg == 0 ? 0 : first(deg - 1) + size(deg - 1); }
  __host__ __device__ static constexpr int offset(int deg) { return deg <= 1 ? 0 : offset(deg - 1) + size(deg - 1) * size(deg - 1); }
  static constexpr int QN = offset(P + 1);
  static constexpr int ET = D == 2 ? 64 : 48, NT = ET * NV;  // elements and threads per block
  static constexpr int ROW = NB | 1;                          // padded shared-memory row
};

// x[block of degree DEG, ...] = Q (or Q^T) in, for degrees DEG..P
template <int D, int P, bool TRANS, int DEG>
PCEXP_DEV void apply_blocks(const double* q, const double (&in)[QBlocks<D, P>::NB], double* x) {
  using B = QBlocks<D, P>;
  if constexpr (DEG <= P) {
    constexpr int n = B::size(DEG), f = B::first(DEG), o = B::offset(DEG);
#pragma unroll
    for (int i = 0; i < n; ++i) {
      double a = 0;
#pragma unroll
      for (int j = 0; j < n; ++j) a = fma(TRANS ? q[o + j * n + i] : q[o + i * n + j], in[f + j], a);
      x[f + i] = a;
    }
    apply_blocks<D, P, TRANS, DEG + 1>(q, in, x);
  }
}

// TRANS: dst = Q^T src (paper -> internal), else dst = Q src.  dst2 (nullable): a second, FP32 copy.
template <class Tin, class Tout, int D, int P, bool TRANS>
__global__ void __launch_bounds__(QBlocks<D, P>::NT) change_basis_kernel(const Tin* __restrict__ src,
                                                                        Tout* __restrict__ dst,
                                                                        float* __restrict__ dst2,
                                                                        const double* __restrict__ Q, int64_t E) {
  using B = QBlocks<D, P>;
  constexpr int NB = B::NB, NV = B::NV, QN = B::QN, ROW = B::ROW;
  __shared__ double sq[B::ET * QN + 1];
  __shared__ double sx[B::NT * ROW];
  const int64_t e0 = (int64_t)blockIdx.x * B::ET;
  const int ne = (int)((E - e0) < B::ET ? (E - e0) : B::ET);
  for (int i = threadIdx.x; i < ne * QN; i += B::NT) sq[i] = Q[e0 * QN + i];
  for (int i = threadIdx.x; i < ne * NV * NB; i += B::NT) sx[i / NB * ROW + i % NB] = (double)src[e0 * NV * NB + i];
  __syncthreads();
  if (threadIdx.x < ne * NV) {
    double* x = sx + threadIdx.x * ROW;
    const double* q = sq + threadIdx.x / NV * QN;
    double in[NB];
#pragma unroll
    for (int j = 0; j < NB; ++j) in[j] = x[j];
    apply_blocks<D, P, TRANS, 1>(q, in, x);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < ne * NV * NB; i += B::NT) {
    const double a = sx[i / NB * ROW + i % NB];
    dst[e0 * NV * NB + i] = (Tout)a;
    if (dst2) dst2[e0 * NV * NB + i] = (float)a;
  }
}

// The same with a thread per entry (src and dst distinct): a chain of at most 6 FMAs instead of the 46
// of a row (p = 2 on tetrahedra), at 30% more FP64 instructions.  162 tetrahedra: 6.4 -> 2.2 us a
// launch; residual calls (two conversions) on 6,000 tetrahedra at p = 2 in FP32-mixed 75 -> 64 us,
// where the row form on 2,058 was slower than a thread per output of the full matrix (64 against 60
// us, now 57).  At 256 rows per SM both forms are bound by the FP64 pipe.
template <class Tin, class Tout, int D, int P, bool TRANS>
__global__ void __launch_bounds__(256) change_basis_entry_kernel(const Tin* __restrict__ src, Tout* __restrict__ dst,
                                                                 float* __restrict__ dst2,
                                                                 const double* __restrict__ Q, int64_t E) {
  using B = QBlocks<D, P>;
  constexpr int NB = B::NB, NV = B::NV, QN = B::QN, MAXN = D == 2 ? P + 1 : (P + 1) * (P + 2) / 2;
  const int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (idx >= E * NV * NB) return;
  const int64_t row = idx / NB;
  const int i = (int)(idx - row * NB);
  int f = 0, o = 0, n = 1;  // first entry, offset in Q and size of this entry's degree
#pragma unroll
  for (int deg = 1; deg <= P; ++deg) {
    if (i >= f + n) {
      f += n;
      if (deg > 1) o += n * n;
      n = D == 2 ? deg + 1 : (deg + 1) * (deg + 2) / 2;
    }
  }
  double a = 0;
  if (i == 0) {
    a = (double)src[idx];
  } else {
    const double* q = Q + row / NV * QN + o;
#pragma unroll
    for (int j = 0; j < MAXN; ++j)
      if (j < n) a = fma(q[TRANS ? j * n + i - f : (i - f) * n + j], (double)src[row * NB + f + j], a);
  }
  dst[idx] = (Tout)a;
  if (dst2) dst2[idx] = (float)a;
}

// Rows per SM up to which the entry form is the faster one (measured above).
constexpr int64_t ENTRY_ROWS = 256;

template <class Tin, class Tout, int D, int P, bool TRANS>
static cudaError_t change_basis_p(const Tin* src, Tout* dst, float* dst2, const double* Q, int64_t E, cudaStream_t st) {
  using B = QBlocks<D, P>;
  if (E * B::NV <= ENTRY_ROWS * sm_count() && (const void*)src != (const void*)dst && (const void*)src != (const void*)dst2) {
    change_basis_entry_kernel<Tin, Tout, D, P, TRANS>
        <<<(unsigned)((E * B::NV * B::NB + 255) / 256), 256, 0, st>>>(src, dst, dst2, Q, E);
    return cudaGetLastError();
  }
  change_basis_kernel<Tin, Tout, D, P, TRANS>
      <<<(unsigned)((E + B::ET - 1) / B::ET), B::NT, 0, st>>>(src, dst, dst2, Q, E);
  return cudaGetLastError();
}
template <class Tin, class Tout, bool TRANS>
static cudaError_t change_basis(const Tin* src, Tout* dst, float* dst2, const double* Q, int64_t E, int nb, int nv,
                                cudaStream_t st) {
  switch (nv * 16 + nb) {
    case 4 * 16 + 1: return change_basis_p<Tin, Tout, 2, 0, TRANS>(src, dst, dst2, Q, E, st);
    case 4 * 16 + 3: return change_basis_p<Tin, Tout, 2, 1, TRANS>(src, dst, dst2, Q, E, st);
    case 4 * 16 + 6: return change_basis_p<Tin, Tout, 2, 2, TRANS>(src, dst, dst2, Q, E, st);
    case 4 * 16 + 10: return change_basis_p<Tin, Tout, 2, 3, TRANS>(src, dst, dst2, Q, E, st);
    case 5 * 16 + 1: return change_basis_p<Tin, Tout, 3, 0, TRANS>(src, dst, dst2, Q, E, st);
    case 5 * 16 + 4: return change_basis_p<Tin, Tout, 3, 1, TRANS>(src, dst, dst2, Q, E, st);
    case 5 * 16 + 10: return change_basis_p<Tin, Tout, 3, 2, TRANS>(src, dst, dst2, Q, E, st);
  }
  return cudaErrorInvalidValue;
}

std::vector<double> pack_basis_change(const std::vector<double>& Q, int64_t E, int nb, int dim) {
  std::vector<double> out;
  out.reserve(Q.size());
  for (int64_t e = 0; e < E; ++e)
    for (int deg = 1, f = 1; f < nb; ++deg) {
      const int n = dim == 2 ? deg + 1 : (deg + 1) * (deg + 2) / 2;
      for (int i = 0; i < n; ++i)
        for (int j = 0; j < n; ++j) out.push_back(Q[((size_t)e * nb + f + i) * nb + f + j]);
      f += n;
    }
  return out;
}

static unsigned grid_for(int64_t n) {
  int64_t b = (n + 255) / 256;
  if (b > 152 * 16) b = 152 * 16;
  return (unsigned)(b < 1 ? 1 : b);
}

template <class T>
cudaError_t launch_paper_to_internal(const double* src, T* dst, const double* Q, int64_t E, int nb, int nv,
                                     cudaStream_t st, float* dst32) {
  return change_basis<double, T, true>(src, dst, dst32, Q, E, nb, nv, st);
}
template <class T>
cudaError_t launch_internal_to_paper(const T* src, double* dst, const double* Q, int64_t E, int nb, int nv, cudaStream_t st) {
  return change_basis<T, double, false>(src, dst, nullptr, Q, E, nb, nv, st);
}

template <class T>
__global__ void scale_elements_kernel(T* __restrict__ x, const T* __restrict__ s, int64_t E, int nvb) {
  const int64_t n = E * nvb;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += (int64_t)gridDim.x * blockDim.x)
    x[idx] *= s[idx / nvb];
}
template <class T>
cudaError_t launch_scale_elements(T* x, const T* s, int64_t E, int nvb, cudaStream_t st) {
  scale_elements_kernel<T><<<grid_for(E * nvb), 256, 0, st>>>(x, s, E, nvb);
  return cudaGetLastError();
}

// Density residual norm of Eq. cfl with the orthonormal basis:
// (1/|Omega|) sqrt(sum_e sum_i (R[e][0][i] / s_e)^2); then CFL(n) of Eq. cfl.
template <class T>
__global__ void __launch_bounds__(256) density_norm_kernel(const T* __restrict__ R, const T* __restrict__ s,
                                                           int64_t E, int nb, int nv, double volume,
                                                           StepState* ss, double* __restrict__ partials,
                                                           int ramp_n, int p, double cfl_max) {
  __shared__ double red[8];
  __shared__ bool last;
  double acc = 0;
  const int64_t n = E * nb;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = idx / nb;
    const int i = (int)(idx - e * nb);
    double r = (double)R[e * nv * nb + i];
    if (s) r /= (double)s[e];
    acc += r * r;
  }
  if (grid_reduce<SumOf>(acc, red, last, partials, &ss->counter)) {
    const double rn = sqrt(acc) / volume;
    ss->res_norm = rn;
    if (!isfinite(rn)) ss->err = 1;
    if (ramp_n > 0) {
      const double a = rn > 0 ? 1.0 / (rn * rn * rn) : DBL_MAX;
      const double b2 = 1.0 + (double)(ramp_n - 1) / (2 * p + 1);
      ss->cfl = fmin(cfl_max, fmax(a, b2));
    }
  }
}

template <class T>
cudaError_t launch_density_norm(const T* R, const T* s, int64_t E, int nb, int nv, double volume, StepState* ss,
                                double* partials, int ramp_n, int p, double cfl_max, cudaStream_t st) {
  int64_t b = (E * nb + 255) / 256;
  if (b > RED_BLOCKS) b = RED_BLOCKS;
  density_norm_kernel<T><<<(unsigned)(b < 1 ? 1 : b), 256, 0, st>>>(R, s, E, nb, nv, volume, ss, partials, ramp_n, p, cfl_max);
  return cudaGetLastError();
}

// Entropy error of Eq. entropy_error (Sec. 5.1) on the FP64 master state, before the
// final square root: sum_e sum_q w^_q |det A_e| (s / s0)^2 with s = p / rho^gamma at the
// volume points, U(x_q) = |det A_e|^-1/2 sum_j phi^_j(xi_q) u_j.  sd[e] = sqrt|det A_e| in
// FP64; Bv [nq][nb] and Wv [nq] the FP64 reference tables.  Fixed-order last-block sum.
__global__ void __launch_bounds__(256) entropy_sum_kernel(const double* __restrict__ u, const double* __restrict__ Bv,
                                                          const double* __restrict__ Wv, const double* __restrict__ sd,
                                                          int64_t E, int nb, int nq, int nv, double gamma,
                                                          double s0, double* __restrict__ value,
                                                          double* __restrict__ partials, unsigned* counter) {
  __shared__ double red[8];
  __shared__ bool last;
  double acc = 0;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < E; e += (int64_t)gridDim.x * blockDim.x) {
    const double s = sd[e], is = 1.0 / s;
    const double* ue = u + e * nv * nb;
    for (int q = 0; q < nq; ++q) {
      double U[5];
      for (int v = 0; v < nv; ++v) {
        double a = 0;
        for (int j = 0; j < nb; ++j) a += Bv[q * nb + j] * ue[v * nb + j];
        U[v] = a * is;
      }
      double m2 = 0;
      for (int k = 1; k < nv - 1; ++k) m2 += U[k] * U[k];
      const double p = (gamma - 1.0) * (U[nv - 1] - 0.5 * m2 / U[0]);
      const double r = p / pow(U[0], gamma) / s0;
      acc += Wv[q] * s * s * r * r;
    }
  }
  if (grid_reduce<SumOf>(acc, red, last, partials, counter)) *value = acc;
}

cudaError_t launch_entropy_sum(const double* u, const double* Bv, const double* Wv, const double* sd, int64_t E, int nb,
                               int nq, int nv, double gamma, double s0, double* value, double* partials,
                               unsigned* counter, cudaStream_t st) {
  int64_t b = (E + 255) / 256;
  if (b > RED_BLOCKS) b = RED_BLOCKS;
  entropy_sum_kernel<<<(unsigned)(b < 1 ? 1 : b), 256, 0, st>>>(u, Bv, Wv, sd, E, nb, nq, nv, gamma, s0, value,
                                                                partials, counter);
  return cudaGetLastError();
}

__global__ void scale_by_inverse_kernel(double* __restrict__ x, const double* __restrict__ s, int64_t n) {
  const double f = 1.0 / *s;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    x[i] *= f;
}
cudaError_t launch_scale_by_inverse(double* x, const double* s, int64_t n, cudaStream_t st) {
  scale_by_inverse_kernel<<<grid_for(n), 256, 0, st>>>(x, s, n);
  return cudaGetLastError();
}

// FP64 FMA throughput of this GPU: NCH independent DFMA chains per thread on every SM, no
// memory traffic.  The result depends on the inputs only through the final store, which a
// comparison that never holds keeps alive.
constexpr int FMA_CHAINS = 8;
template <class T>
__global__ void __launch_bounds__(256) fma_chain_kernel(T* out, int iters, T a, T b) {
  T x[FMA_CHAINS];
#pragma unroll
  for (int k = 0; k < FMA_CHAINS; ++k) x[k] = T(1e-3) * (T)(threadIdx.x + k);
  for (int i = 0; i < iters; ++i)
#pragma unroll
    for (int k = 0; k < FMA_CHAINS; ++k) x[k] = fma(x[k], a, b);
  T s = 0;
#pragma unroll
  for (int k = 0; k < FMA_CHAINS; ++k) s += x[k];
  if (s == T(-1)) out[blockIdx.x] = s;
}

// FMA rate (TFLOP/s, an FMA counts 2) of the current device in FP64 or FP32: independent
// chains on 8 blocks of 256 threads per SM, best of three timed launches after a warm-up.
template <class T>
cudaError_t measure_fma_rate(double* tflops) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  cudaStream_t st = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  T* out = nullptr;
  if ((e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking)) != cudaSuccess) return e;
  e = cudaEventCreate(&e0);
  if (e == cudaSuccess) e = cudaEventCreate(&e1);
  if (e == cudaSuccess) e = cudaMalloc(&out, sizeof(T) * sms * 8);
  // FP32 FMAs issue far faster than FP64 ones: more iterations keep the launch near 10 ms
  const int iters = sizeof(T) == 8 ? 1 << 14 : 1 << 17, blocks = sms * 8, threads = 256;
  float best = 1e30f;
  for (int rep = 0; e == cudaSuccess && rep < 4; ++rep) {
    cudaEventRecord(e0, st);
    fma_chain_kernel<T><<<blocks, threads, 0, st>>>(out, iters, T(0.9999999), T(1e-7));
    cudaEventRecord(e1, st);
    e = cudaEventSynchronize(e1);
    float ms = 0;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    if (e == cudaSuccess && rep > 0 && ms < best) best = ms;  // the first launch is a warm-up
  }
  if (e == cudaSuccess) *tflops = 2.0 * FMA_CHAINS * (double)iters * blocks * threads / (best * 1e-3) / 1e12;
  if (out) cudaFree(out);
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  cudaStreamDestroy(st);
  return e;
}
cudaError_t measure_fp64_fma_rate(double* tflops) { return measure_fma_rate<double>(tflops); }
cudaError_t measure_fp32_fma_rate(double* tflops) { return measure_fma_rate<float>(tflops); }

// ---- partitioned runs: ghost element rows from the owning partitions
template <class T>
__global__ void gather_ghosts_kernel(T* __restrict__ x, PartPtrs srcs, const int32_t* __restrict__ src_part,
                                     const int32_t* __restrict__ src_elem, int64_t n_local, int64_t n_ghost, int nvb) {
  const int64_t n = n_ghost * nvb;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t g = i / nvb;
    const int k = (int)(i - g * nvb);
    const T* src = reinterpret_cast<const T*>(srcs.p[src_part[g]]);
    x[(n_local + g) * nvb + k] = src[(int64_t)src_elem[g] * nvb + k];
  }
}
template <class T>
cudaError_t launch_gather_ghosts(T* x, PartPtrs srcs, const int32_t* src_part, const int32_t* src_elem, int64_t n_local,
                                 int64_t n_ghost, int nvb, cudaStream_t st) {
  if (n_ghost <= 0) return cudaSuccess;
  gather_ghosts_kernel<T><<<grid_for(n_ghost * nvb), 256, 0, st>>>(x, srcs, src_part, src_elem, n_local, n_ghost, nvb);
  return cudaGetLastError();
}
template <class T>
__global__ void zero_range_kernel(T* __restrict__ x, int64_t from, int64_t to) {
  for (int64_t i = from + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < to; i += (int64_t)gridDim.x * blockDim.x)
    x[i] = T(0);
}
template <class T>
cudaError_t launch_zero_range(T* x, int64_t from, int64_t to, cudaStream_t st) {
  if (to <= from) return cudaSuccess;
  zero_range_kernel<T><<<grid_for(to - from), 256, 0, st>>>(x, from, to);
  return cudaGetLastError();
}

#define PCEXP_INST(T)                                                                                         \
  template cudaError_t launch_paper_to_internal<T>(const double*, T*, const double*, int64_t, int, int,        \
                                                   cudaStream_t, float*);                                      \
  template cudaError_t launch_internal_to_paper<T>(const T*, double*, const double*, int64_t, int, int,        \
                                                   cudaStream_t);                                              \
  template cudaError_t launch_scale_elements<T>(T*, const T*, int64_t, int, cudaStream_t);                     \
  template cudaError_t launch_gather_ghosts<T>(T*, PartPtrs, const int32_t*, const int32_t*, int64_t, int64_t,  \
                                               int, cudaStream_t);                                              \
  template cudaError_t launch_zero_range<T>(T*, int64_t, int64_t, cudaStream_t);                                \
  template cudaError_t launch_density_norm<T>(const T*, const T*, int64_t, int, int, double, StepState*,       \
                                              double*, int, int, double, cudaStream_t);
PCEXP_INST(double)
PCEXP_INST(float)

}  // namespace pcexp
