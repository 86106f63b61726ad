// DG operator kernels on triangles (D = 2) and tetrahedra (D = 3): the residual
// R(u) of Eq. euler3 (Sec. 4.2), its tangent-linear J(u) v (the exact Jacobian of
// Eq. jac1 / jac2, applied matrix-free), the transpose and second-order adjoints,
// the output functionals and the element time-step rule of Eq. x3d.  Each
// dimension is instantiated in its own translation unit (dg2d.cu, dg3d.cu).
//
// Basis: a reference-simplex orthonormal basis phi^_j mapped affinely and scaled
// by |det A_e|^-1/2, so it is orthonormal on every element (the mass matrix is the
// identity, as with the paper's basis).  With x = v0 + A xi:
//   U(x_q)        = |det A|^-1/2 sum_j phi^_j(xi_q) u_j
//   volume term   = |det A|^1/2 sum_q w_q sum_d' d phi^_i/d xi_d'(xi_q) Fhat_d'
//                   with Fhat_d' = sum_d (A^-1)_{d' d} F_d(U(x_q))
//   face term     = -|det A|^-1/2 sum_q w_q |f| phi^_i(x_q) F~_n(x_q)
// Two launches per operator: a face kernel (one thread per face point) writes
// |f| w_q F~_n into the face-flux buffer G; an element kernel (a tile of 32 elements
// per block) adds the volume term and lifts the face fluxes of its D+1 faces.  Every face flux is computed once and every output is
// written once, in a fixed order (deterministic).
//
// Face points are those of the face's L element (its local face-vertex order).
// The trace tables Bf[face][perm][q][j] hold phi^_j at face point q of local face
// `face` when the element's face vertices are the L element's permuted by `perm`
// (perm 0 = identity; in 2D perm 1 reverses the edge).  An element's face slot
// ef = (face index << 4) | (side << 3) | perm.
#pragma once
#include <cfloat>
#include <type_traits>

#include "kernels.h"

namespace pcexp {

template <int D, int P> struct Ord {
  static constexpr int NV = D + 2;
  static constexpr int NB = D == 2 ? (P + 1) * (P + 2) / 2 : (P + 1) * (P + 2) * (P + 3) / 6;
  // volume and face points: collapsed rules with p + 1 points per direction, except
  // tetrahedra at p = 2 (the symmetric 14-point volume and 7-point face rules)
  static constexpr int NQ = D == 2 ? (P + 1) * (P + 1) : P == 2 ? 14 : (P + 1) * (P + 1) * (P + 1);
  static constexpr int NFQ = D == 2 ? P + 1 : P == 2 ? 7 : (P + 1) * (P + 1);
  static constexpr int NF = D + 1;                  // faces per element
  static constexpr int NPERM = D == 2 ? 2 : 6;      // vertex permutations of a face
  static constexpr int GEO = D == 2 ? 8 : 12;       // geometry record: A^-1 (D x D), sqrt|det|, h, 1/sqrt|det|
  static constexpr int SD = D * D;       // sqrt|det A|
  static constexpr int HE = D * D + 1;   // h
  static constexpr int ISD = D * D + 2;  // 1 / sqrt|det A| (multiplications instead of FP64 divisions)
  static constexpr int NVB = NV * NB;
  // elements per block (tetrahedra: at most 16, which keeps the FP64 tile within 48 KB)
  static constexpr int ET0 = (256 / NQ) > 128 ? 128 : (256 / NQ);
  static constexpr int ET = (D == 3 && ET0 > 16) ? 16 : ET0;
  static constexpr int NJF = 2 * NV * NV;           // face point-Jacobian entries
  static constexpr int NBF = NF * NPERM * NFQ * NB;  // trace-table entries
  static constexpr bool SMEM_BF = D == 2;            // stage the trace tables in shared memory
};

template <class S> struct PartOf;
template <> struct PartOf<double> { PCEXP_DEV static double get(double x) { return x; } };
template <> struct PartOf<float> { PCEXP_DEV static float get(float x) { return x; } };
template <class T> struct PartOf<Tangent<T>> { PCEXP_DEV static T get(Tangent<T> x) { return x.d; } };

// table read: shared memory, or global memory through the read-only cache
template <bool SMEM, class T> PCEXP_DEV T tab(const T* p) {
  if constexpr (SMEM) return *p;
  else return __ldg(p);
}

// slip wall or symmetry plane: both take the slip-wall ghost state
PCEXP_DEV bool mirror_bc(int eR) { return -eR == PCEXP_BC_SLIP_WALL || -eR == PCEXP_BC_SYMMETRY; }

// Source term of a rotating frame on the orthonormal basis: S = -omega x m is linear in U, so
// int_E phi_i S(U_h) dx = -(omega x m_i) coefficient-wise (m_i the momentum coefficients of
// test function i).  Returns component k (0..D-1) given the D momentum coefficients m.
template <class T, int D>
PCEXP_DEV T rot_source(const T* om, const T (&m)[D], int k) {
  const T mx = m[0], my = m[1], mz = D == 3 ? m[D - 1] : T(0);
  const T c = k == 0 ? om[1] * mz - om[2] * my : (k == 1 ? om[2] * mx - om[0] * mz : om[0] * my - om[1] * mx);
  return -c;
}

template <class O> PCEXP_DEV int slot_face(int fs) { return fs >> 4; }
PCEXP_DEV int slot_side(int fs) { return (fs >> 3) & 1; }
PCEXP_DEV int slot_perm(int fs) { return fs & 7; }

// FP32 on tetrahedra stores a record per interior face point (RoeRecord, 16 values in 16-byte chunks
// [4][interior points][4]) and an nv x nv block per boundary point after them; the other forms
// blocks for all points (bface_at).
template <class T, int D> constexpr bool FACE_RECORDS = std::is_same<T, float>::value && D == 3;

// Table rows and face-flux records are padded to whole 16-byte vectors where they are read with
// 16-byte loads.
template <class T> constexpr int VECW = 16 / (int)sizeof(T);
template <class T, int N> constexpr int PADV = (N + VECW<T> - 1) / VECW<T> * VECW<T>;

// r[0..N) = p[0..N) from a 16-byte-aligned row (shared memory, or global through the
// read-only cache), N a multiple of VECW<T>
template <class T, int N, bool GLOBAL = false>
PCEXP_DEV void load_row(const T* p, T (&r)[N]) {
  if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int k = 0; k < N / 4; ++k) {
      const float4 a = GLOBAL ? __ldg(reinterpret_cast<const float4*>(p) + k) : reinterpret_cast<const float4*>(p)[k];
      r[4 * k] = a.x;
      r[4 * k + 1] = a.y;
      r[4 * k + 2] = a.z;
      r[4 * k + 3] = a.w;
    }
  } else {
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
      const double2 a = GLOBAL ? __ldg(reinterpret_cast<const double2*>(p) + k) : reinterpret_cast<const double2*>(p)[k];
      r[2 * k] = a.x;
      r[2 * k + 1] = a.y;
    }
  }
}

// c[0..N) = p[0..N), coefficients of one variable of an element (read-only in the kernel):
// 8-byte loads of FP32 pairs when N is even (rows then start on 8-byte boundaries)
template <class T, int N>
PCEXP_DEV void load_coeffs(const T* __restrict__ p, T (&c)[N]) {
  if constexpr (sizeof(T) == 4 && N % 2 == 0) {
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
      const float2 a = __ldg(reinterpret_cast<const float2*>(p) + k);
      c[2 * k] = a.x;
      c[2 * k + 1] = a.y;
    }
  } else {
#pragma unroll
    for (int k = 0; k < N; ++k) c[k] = __ldg(p + k);
  }
}

// Face fluxes G: [F][nv][GS] with GS = nfq rounded up to whole 16-byte vectors, or [F][nv][nfq]
// (PADG false: the fixed scratch of the no-allocation entry point).
template <class T, int D, int P, bool PADG = true> constexpr int GSTRIDE = PADG ? PADV<T, Ord<D, P>::NFQ> : Ord<D, P>::NFQ;

// One face point's fluxes into G.  The last point also writes the records' padding: a sector that is
// never completely written costs a read when it leaves the L2 (face J v on 48^3 cubes: 392 -> 470
// us without this).
template <class T, int D, int P, bool PADG>
PCEXP_DEV void store_face_flux(T* __restrict__ G, int64_t f, int q, const T (&x)[D + 2]) {
  constexpr int NFQ = Ord<D, P>::NFQ, NV = D + 2, GS = GSTRIDE<T, D, P, PADG>;
  T* g = G + f * NV * GS + q;
#pragma unroll
  for (int v = 0; v < NV; ++v) g[v * GS] = x[v];
  if constexpr (GS > NFQ) {
    if (q == NFQ - 1) {
#pragma unroll
      for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int k = 1; k <= GS - NFQ; ++k) g[v * GS + k] = T(0);
    }
  }
}

// ------------------------------------------------------------------ face kernel
template <class T, int D, int P, bool TAN, bool PADG>
__global__ void __launch_bounds__(256) face_kernel(DGData<T> d, const T* __restrict__ u,
                                                   const T* __restrict__ du, T* __restrict__ G,
                                                   const int* __restrict__ skip) {
  using O = Ord<D, P>;
  constexpr int NB = O::NB, NFQ = O::NFQ, NV = O::NV, NPERM = O::NPERM, GEO = O::GEO;
  constexpr bool SM = O::SMEM_BF;
  using S = typename std::conditional<TAN, Tangent<T>, T>::type;
  __shared__ T sBf[SM ? O::NBF : 1];
  __shared__ T sWf[NFQ];
  if (skip && *skip) return;
  if constexpr (SM)
    for (int i = threadIdx.x; i < O::NBF; i += blockDim.x) sBf[i] = d.Bf[i];
  for (int i = threadIdx.x; i < NFQ; i += blockDim.x) sWf[i] = d.Wf[i];
  __syncthreads();
  const T* Bf = SM ? sBf : d.Bf;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= d.F * NFQ) return;
  const int64_t f = idx / NFQ;
  const int q = (int)(idx - f * NFQ);
  const int eL = d.fel[2 * f], eR = d.fel[2 * f + 1];
  const int loc = d.floc[f];
  const int fL = loc & 0xff, fR = (loc >> 8) & 0xff, pR = loc >> 16;
  T n[D];
#pragma unroll
  for (int k = 0; k < D; ++k) n[k] = d.fgeo[4 * f + k];
  const T meas = d.fgeo[4 * f + D];
  S UL[NV], UR[NV];
  {
    const T isd = d.geo[GEO * (int64_t)eL + O::ISD];
    const T* ue = u + (int64_t)eL * NV * NB;
    const T* be = Bf + ((fL * NPERM) * NFQ + q) * NB;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      T a = 0, b = 0;
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        const T bj = tab<SM>(be + j);
        a += bj * ue[v * NB + j];
        if constexpr (TAN) b += bj * du[(int64_t)eL * NV * NB + v * NB + j];
      }
      if constexpr (TAN) UL[v] = S{a * isd, b * isd};
      else UL[v] = a * isd;
    }
  }
  if (eR >= 0) {
    const T isd = d.geo[GEO * (int64_t)eR + O::ISD];
    const T* ue = u + (int64_t)eR * NV * NB;
    const T* be = Bf + ((fR * NPERM + pR) * NFQ + q) * NB;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      T a = 0, b = 0;
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        const T bj = tab<SM>(be + j);
        a += bj * ue[v * NB + j];
        if constexpr (TAN) b += bj * du[(int64_t)eR * NV * NB + v * NB + j];
      }
      if constexpr (TAN) UR[v] = S{a * isd, b * isd};
      else UR[v] = a * isd;
    }
  } else if (mirror_bc(eR)) {
    ghost_slip_wall<D, S, T>(UL, n, UR, d.rot ? d.vrn[idx] : T(0));
  } else {
    ghost_farfield<D, S, T>(UL, n, d.fs, UR);
  }
  S Fn[NV];
  roe_flux<D, S, T>(UL, UR, n, d.fs.gamma, Fn, d.rot ? d.vrn[idx] : T(0));
  const T wl = meas * sWf[q];
  T fx[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) fx[v] = wl * PartOf<S>::get(Fn[v]);
  store_face_flux<T, D, P, PADG>(G, f, q, fx);
}

// --------------------------------------------------------------- element kernel
// The reference tables of one (D, p) in constant memory, read at warp-uniform addresses as operands
// of the FMAs (outside the load/store pipe).  They depend on the reference simplex alone, so
// every context of that order uploads the same bytes (upload_tables).
//   Bv [nq][nb]        phi_j at the volume points
//   Wm [nq][nb1]       w_q phi_k at the volume points, k < nb1 (the basis of order p - 1)
//   Cm [D][nb][nb1]    <d phi_i / d xi_d, phi_k>: the gradients of the basis in the basis of order p - 1
//   Bf [nf][nfq][nb]   phi_j at the face points, the element's own face-vertex order
//   Ch, Cl [D][nb]     int d phi_i / d xi_d (the test of a constant) and what its rounding lost
template <int D, int P> struct TabLayout {
  using O = Ord<D, P>;
  static constexpr int NB1 = P == 0 ? 0 : Ord<D, P == 0 ? 0 : P - 1>::NB;
  static constexpr int BV = 0, WM = BV + O::NQ * O::NB, CM = WM + O::NQ * NB1, BF = CM + D * O::NB * NB1;
  static constexpr int CH = BF + O::NF * O::NFQ * O::NB, CL = CH + D * O::NB;
  static constexpr int N = CL + D * O::NB;
};
template <class T, int D, int P> __constant__ T c_tab[TabLayout<D, P>::N];

// Degree of basis function i (the basis is graded)
template <int D> __host__ __device__ constexpr int degree_of(int i) {
  int deg = 0, n = 1;
  while (i >= n) {
    ++deg;
    n += D == 2 ? deg + 1 : (deg + 1) * (deg + 2) / 2;
  }
  return deg;
}
template <int D> __host__ __device__ constexpr int basis_size(int p) {
  return p < 0 ? 0 : D == 2 ? (p + 1) * (p + 2) / 2 : (p + 1) * (p + 2) * (p + 3) / 6;
}

// What the volume term is the flux of: the state u (residual), or the flux's derivative along du at
// u, from the traces of u (TANGENT) or from the point values stored by the linearisation (STORED).
enum ElemMode { ELEM_FLUX = 0, ELEM_TANGENT = 1, ELEM_STORED = 2 };

// The NFQ fluxes of one face and variable in the order of the element's own face points: the L
// element's as stored; on the R side the points of a symmetric rule are permuted with the face
// vertices (2D: reversed; the 7-point rule: the centroid, then two orbits of three points whose
// distinguished vertices are 0, 2, 1).
template <class T, int D, int P, int GS>
PCEXP_DEV void face_fluxes(const T (&r)[GS], int fs, T (&x)[Ord<D, P>::NFQ]) {
  constexpr int NFQ = Ord<D, P>::NFQ;
  const int side = slot_side(fs);
  if constexpr (D == 2) {
#pragma unroll
    for (int q = 0; q < NFQ; ++q) x[q] = side ? r[NFQ - 1 - q] : r[q];
  } else if constexpr (NFQ == 7) {
    // entry s' of an orbit comes from the L vertex s with perm(s) = s'
    constexpr unsigned long long INV = 36ull | 24ull << 6 | 33ull << 12 | 18ull << 18 | 9ull << 24 | 6ull << 30;
    const int code = (int)(INV >> (6 * slot_perm(fs))) & 63;
    constexpr int AT[3] = {0, 2, 1};  // position in the orbit of the point distinguished by vertex s
    x[0] = r[0];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      const int from = (code >> (2 * s)) & 3;
#pragma unroll
      for (int o = 1; o <= 4; o += 3) x[o + AT[s]] = from == 0 ? r[o + AT[0]] : from == 1 ? r[o + AT[1]] : r[o + AT[2]];
    }
  } else {
#pragma unroll
    for (int q = 0; q < NFQ; ++q) x[q] = r[q];
  }
#pragma unroll
  for (int q = 0; q < NFQ; ++q) x[q] = side ? x[q] : -x[q];
}

// acc[i] += sum_k C[i][k] m[k] for i >= I: the gradient of a function of degree g lies in degrees < g
template <class T, int D, int P, int I, int N>
PCEXP_DEV void combine_modes(const T* C, const T (&m)[N], T (&acc)[Ord<D, P>::NB]) {
  if constexpr (I < Ord<D, P>::NB) {
    constexpr int n = basis_size<D>(degree_of<D>(I) - 1);
#pragma unroll
    for (int k = 0; k < n; ++k) acc[I] = fma(C[I * TabLayout<D, P>::NB1 + k], m[k], acc[I]);
    combine_modes<T, D, P, I + 1>(C, m, acc);
  }
}

// cp.async copies (global -> shared, no register staging)
PCEXP_DEV void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
PCEXP_DEV void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
PCEXP_DEV void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Four values from a 16-byte boundary, issued where it stands (volatile: not sunk past a barrier
// to the first use)
PCEXP_DEV void load_early(const float* p, float (&x)[4]) {
  asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3])
               : "l"(p));
}
PCEXP_DEV void load_early(const double* p, double (&x)[4]) {
  asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(x[0]), "=d"(x[1]) : "l"(p));
  asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(x[2]), "=d"(x[3]) : "l"(p + 2));
}

template <class T, int D, int P, int MODE, int SL = 1> struct ElemTile {
  using O = Ord<D, P>;
  static constexpr int ET = 32 / SL, NT = 32 * O::NV;
  static constexpr int RS = O::NVB | 1;  // odd row stride: lanes (elements) hit distinct banks
  static constexpr int ROWS = ET * RS * (MODE == ELEM_TANGENT ? 2 : 1);
  static constexpr int FLUX = P == 0 ? 0 : O::NQ * D * O::NV * ET;
  // FP32: the threads' own face-flux records, copied in while the volume part is computed
  static constexpr bool AHEAD = sizeof(T) == 4 && SL == 1;
  static constexpr int GV = GSTRIDE<T, D, P> / VECW<T>;  // 16-byte vectors of a record
  static constexpr int ROWS4 = (ROWS + 3) / 4 * 4;       // the records start on a 16-byte boundary
  static constexpr int RECS = AHEAD ? O::NF * GV * NT * VECW<T> : 0;
  static constexpr size_t BYTES = sizeof(T) * (size_t)(ROWS4 + RECS + FLUX);
  // blocks per SM the registers are bounded for (the shared memory allows as many or more, but for
  // FP32 TANGENT on tetrahedra at p = 2: 60 KB, three blocks; its 80 registers spill nothing)
  static constexpr int MINB = sizeof(T) == 4 ? (D == 3 ? 4 : MODE == ELEM_STORED ? 7 : 5) : (D == 3 ? 2 : 3);
};

// A block owns 32 elements and has a warp per variable.
//   Phase 1: lane = element, the warps share the volume points.  Each lane reads its element's rows
//   from shared memory once for all its warp's points, forms the traces, the flux (or its
//   derivative) in the element's reference directions (contravariant form: q_d = A^-1_d . v, no
//   Cartesian flux is formed and mapped) and stores it as [point][direction][variable][element].
//   Phase 2: lane = element, warp = variable.  Each thread tests its variable's flux against the
//   gradients and lifts its face fluxes, nb accumulators in registers.  The gradients of P^p lie
//   in P^(p-1): the fluxes are first projected on that basis (Wm), then combined (Cm), e.g. 249
//   instead of 420 FMAs per variable on tetrahedra at p = 2.
// Every table index is warp-uniform, every shared-memory access conflict-free, and no partial
// sums cross warps; both forms (FP32 and FP64) run the same code.  FP32 is bound by instruction
// issue and, on meshes whose face fluxes leave the L2, by the latency of their gather: each thread
// copies its records into shared memory by cp.async before the volume part (48^3 cubes at p = 2:
// 509 us without that).  FP64 is bound by its pipe.
// Measured against the kernels this one replaces, per launch of the Krylov J v: FP32 48^3 cubes at
// p = 2 449 -> 277 us (a persistent kernel whose six warps each kept 50 partial sums and recomputed
// the flux derivative from u), FP32 131,072 triangles at p = 3 111 -> 34 us (lanes sharing an
// element's test functions), FP64 20^3 cubes at p = 2 485 -> 427 us (stored D nv x nv Jacobians);
// the residual's: FP64 24^3 cubes at p = 2 1117 -> 717 us.
//
// FP32 sums: one chain of FMAs per entry through all faces, points and directions adds the rounding
// of up to 50 terms, and R is the small difference of its volume and face terms.  So every face and
// every direction has a sum of its own and the sums are added (PARTS); the projection of the
// derivatives runs in two chains (HALVES); and the projection of R's fluxes takes their differences
// from the first point's, the test of that constant coming from a table rounded to twice FP32
// (SHIFT: a smooth flux loses only the rounding of its variation; on the derivatives along rough
// Krylov vectors it would add 5 to 8%).  Error against 64 bits, one chain -> this (two to four lanes
// sharing the sums, as the kernels before this one did): a step on 48^3 cubes at p = 2 1.85e-7 ->
// 1.31e-7 (1.47e-7), on 131,072 triangles at p = 3 2.14e-7 -> 1.48e-7 (1.69e-7); R on 24^3 cubes at
// p = 2 8.5e-5 -> 7.2e-5 (7.6e-5).  It costs 0.2 of 277 us per J v on the cubes, 1.5 of 37.5 us on
// the triangles (the second chain's registers; seven blocks per SM instead of five keep it there: 41
// us with five) and 14 of 266 us per R on the cubes.  FP64 keeps one chain: its pipe is the bound.
//
// SL > 1: a block owns 32 / SL elements and SL lanes share one.  They split the points of phase 1 and
// of the projection (its sums meet by shuffles) and the rows (test functions) of the lift and the
// combination, so a tile takes about a third of the time at SL = 4 and four times the SMs work on a
// small mesh; the tables are then read at SL addresses per warp and the splits leave lanes idle,
// so the total work grows.  Per launch of the FP64 Krylov J v at p = 2: 14.5 -> 7.9 us on 1,152
// triangles, but 24.0 -> 28.4 us on 6,144; residual calls on 4,608 triangles 77 -> 70 us and on
// 10,082 105 -> 112 us.  FP32: 6.3 -> 5.8 us on 162 tetrahedra, 71 -> 76 us a J v call on 20,402
// triangles.  Hence the limit of 32 elements per SM (one tile of 32 per SM).
template <class T, int D, int P, int MODE, bool PADG, int SL>
__global__ void __launch_bounds__(ElemTile<T, D, P, MODE, SL>::NT, ElemTile<T, D, P, MODE, SL>::MINB)
    elem_op_kernel(DGData<T> d, const T* __restrict__ u, const T* __restrict__ du, const T* __restrict__ pts,
                   const T* __restrict__ G, T* __restrict__ out, const T* __restrict__ escale,
                   const int* __restrict__ skip, const double* __restrict__ oscale) {
  using O = Ord<D, P>;
  using L = ElemTile<T, D, P, MODE, SL>;
  using X = TabLayout<D, P>;
  constexpr int NB = O::NB, NQ = O::NQ, NFQ = O::NFQ, NV = O::NV, NVB = O::NVB, GEO = O::GEO, NF = O::NF;
  constexpr int NPERM = O::NPERM, ET = L::ET, RS = L::RS, NB1 = X::NB1;
  constexpr int GS = GSTRIDE<T, D, P, PADG>;
  extern __shared__ __align__(16) unsigned char elem_dyn[];
  T* rows = reinterpret_cast<T*>(elem_dyn);
  T* sG = rows + L::ROWS4;  // [face][vector][thread][16 bytes]
  T* sF = sG + L::RECS;
  if (skip && *skip) return;
  const T* tab = c_tab<T, D, P>;
  const int64_t e0 = (int64_t)blockIdx.x * ET;
  const int ne = (int)((d.E - e0) < ET ? (d.E - e0) : ET);
  // the warp's index through a shuffle, so that it is known to be uniform (table loads by it)
  const int lane = threadIdx.x & 31, w = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
  const int tl = SL == 1 ? lane : lane % ET, sub = SL == 1 ? 0 : lane / ET;
  const int64_t e = e0 + (tl < ne ? tl : 0);  // lanes past the last element repeat element e0; discarded
  int slots[NF];
  if constexpr (NF == 4) {
    const int4 s4 = __ldg(reinterpret_cast<const int4*>(d.ef) + e);
    slots[0] = s4.x;
    slots[1] = s4.y;
    slots[2] = s4.z;
    slots[NF - 1] = s4.w;
  } else {
#pragma unroll
    for (int k = 0; k < NF; ++k) slots[k] = __ldg(d.ef + NF * e + k);
  }
  // the tile's rows: ET * NVB = NT * NB / SL values, all loads issued before the first store
  {
    const T* src = (MODE == ELEM_FLUX ? u : du) + e0 * NVB;
    constexpr int KR = (NB + SL - 1) / SL;
    T x[KR], y[MODE == ELEM_TANGENT ? KR : 1];
#pragma unroll
    for (int k = 0; k < KR; ++k) {
      const int i = threadIdx.x + k * L::NT;
      x[k] = i < ne * NVB ? src[i] : T(0);
      if constexpr (MODE == ELEM_TANGENT) y[k] = i < ne * NVB ? u[e0 * NVB + i] : T(0);
    }
    if constexpr (L::AHEAD) {
#pragma unroll
      for (int k = 0; k < NF; ++k) {
        const T* g = G + ((int64_t)slot_face<O>(slots[k]) * NV + w) * GS;
#pragma unroll
        for (int h = 0; h < L::GV; ++h)
          cp_async16(sG + ((k * L::GV + h) * L::NT + threadIdx.x) * VECW<T>, g + h * VECW<T>);
      }
      cp_async_commit();
    }
#pragma unroll
    for (int k = 0; k < KR; ++k) {
      const int i = threadIdx.x + k * L::NT, r = i / NVB * RS + i % NVB;
      if (i < ne * NVB) {
        rows[r] = x[k];
        if constexpr (MODE == ELEM_TANGENT) rows[ET * RS + r] = y[k];
      }
    }
  }
  T ge[GEO];
  load_row<T, GEO, true>(d.geo + GEO * e, ge);
  const T isd = ge[O::ISD];
  constexpr int WS = NV * SL, PP = P == 0 ? 1 : (NQ + WS - 1) / WS;  // shares of the points, points per share
  const int q0 = w * SL + sub, qc = WS <= NQ || q0 < NQ ? q0 : 0;      // this lane's first point (in range: qc)
  T pv[MODE == ELEM_STORED ? PP : 1][4];
  if constexpr (MODE == ELEM_STORED && P > 0) {
#pragma unroll
    for (int i = 0; i < PP; ++i) load_early(pts + ((int64_t)(q0 + i * WS < NQ ? q0 + i * WS : qc) * d.E + e) * 4, pv[i]);
  }
  __syncthreads();
  const int el = tl < ne ? tl : 0;
  if constexpr (P > 0) {
    const T gm = d.fs.gamma - T(1);
    T Ai[D][D];
#pragma unroll
    for (int k = 0; k < D * D; ++k) Ai[k / D][k % D] = ge[k];
    // traces of this lane's element at its points q0, q0 + WS, ... (the last may be past NQ: it repeats
    // the first point and is not stored)
    T t[PP][NV], s[MODE == ELEM_TANGENT ? PP : 1][NV];
    const T* ra = rows + el * RS;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
#pragma unroll
      for (int i = 0; i < PP; ++i) {
        t[i][v] = T(0);
        if constexpr (MODE == ELEM_TANGENT) s[i][v] = T(0);
      }
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        const T c = ra[v * NB + j];
        T c2 = T(0);
        if constexpr (MODE == ELEM_TANGENT) c2 = ra[ET * RS + v * NB + j];
#pragma unroll
        for (int i = 0; i < PP; ++i) {
          const int q = q0 + i * WS < NQ ? q0 + i * WS : qc;
          const T b = tab[X::BV + q * NB + j];
          t[i][v] = fma(b, c, t[i][v]);
          if constexpr (MODE == ELEM_TANGENT) s[i][v] = fma(b, c2, s[i][v]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < PP; ++i) {
      const int q = q0 + i * WS;
      if (q >= NQ) break;
      T vel[D], H, k2 = T(0);
      T F[D][NV];
      if constexpr (MODE == ELEM_STORED) {
#pragma unroll
        for (int k = 0; k < D; ++k) vel[k] = pv[MODE == ELEM_STORED ? i : 0][k];
        H = pv[MODE == ELEM_STORED ? i : 0][D];
#pragma unroll
        for (int k = 0; k < D; ++k) k2 = fma(T(0.5) * vel[k], vel[k], k2);
      } else {
        T U[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) U[v] = (MODE == ELEM_TANGENT ? s[MODE == ELEM_TANGENT ? i : 0][v] : t[i][v]) * isd;
        const T ir = T(1) / U[0];
#pragma unroll
        for (int k = 0; k < D; ++k) {
          vel[k] = U[1 + k] * ir;
          k2 = fma(T(0.5) * vel[k], vel[k], k2);
        }
        const T p = gm * (U[NV - 1] - k2 * U[0]);
        if constexpr (MODE == ELEM_FLUX) {
#pragma unroll
          for (int dd = 0; dd < D; ++dd) {
            T qd = Ai[dd][0] * vel[0];
#pragma unroll
            for (int k = 1; k < D; ++k) qd = fma(Ai[dd][k], vel[k], qd);
            F[dd][0] = U[0] * qd;
#pragma unroll
            for (int k = 0; k < D; ++k) F[dd][1 + k] = fma(U[1 + k], qd, Ai[dd][k] * p);
            F[dd][NV - 1] = (U[NV - 1] + p) * qd;
          }
          if (d.rot) {
#pragma unroll
            for (int v = 0; v < NV; ++v) t[i][v] = U[v];
          }
        }
        H = (U[NV - 1] + p) * ir;
      }
      if constexpr (MODE != ELEM_FLUX) {
        // derivative along the trace t: with w_d = rho dq_d = A^-1_d . dm - q_d drho,
        // dF_d = (A^-1_d . dm, v w_d + q_d dm + A^-1_d dp, H w_d + q_d (dE + dp))
        T dp = fma(k2, t[i][0], t[i][NV - 1]);
#pragma unroll
        for (int k = 0; k < D; ++k) dp = fma(-vel[k], t[i][1 + k], dp);
        dp *= gm;
        const T de = t[i][NV - 1] + dp;
#pragma unroll
        for (int dd = 0; dd < D; ++dd) {
          T qd = Ai[dd][0] * vel[0], f0 = Ai[dd][0] * t[i][1];
#pragma unroll
          for (int k = 1; k < D; ++k) {
            qd = fma(Ai[dd][k], vel[k], qd);
            f0 = fma(Ai[dd][k], t[i][1 + k], f0);
          }
          const T wd = fma(-qd, t[i][0], f0);
          F[dd][0] = f0;
#pragma unroll
          for (int k = 0; k < D; ++k) F[dd][1 + k] = fma(vel[k], wd, fma(qd, t[i][1 + k], Ai[dd][k] * dp));
          F[dd][NV - 1] = fma(H, wd, qd * de);
        }
      }
      if (d.rot) {  // rotating frame: the flux is F - U v_r^T
        const T* vr = d.vrq + (e * NQ + q) * D;
#pragma unroll
        for (int dd = 0; dd < D; ++dd) {
          T vd = Ai[dd][0] * vr[0];
#pragma unroll
          for (int k = 1; k < D; ++k) vd = fma(Ai[dd][k], vr[k], vd);
#pragma unroll
          for (int v = 0; v < NV; ++v) F[dd][v] = fma(-vd, t[i][v], F[dd][v]);
        }
      }
#pragma unroll
      for (int dd = 0; dd < D; ++dd)
#pragma unroll
        for (int v = 0; v < NV; ++v) sF[((q * D + dd) * NV + v) * ET + tl] = F[dd][v];
    }
    __syncthreads();
  }
  // phase 2: variable w of this lane's element
  if constexpr (L::AHEAD) cp_async_wait_all();  // a thread reads its own copies only
  constexpr int NR = (NB + SL - 1) / SL;  // rows sub, sub + SL, ... of this lane (past NB: repeated, not stored)
  // the order of the FP32 sums (see above)
  constexpr bool PARTS = sizeof(T) == 4, SHIFT = PARTS && MODE == ELEM_FLUX, HALVES = PARTS && MODE != ELEM_FLUX;
  auto row = [&](int i) { return SL == 1 ? i : (i * SL + sub < NB ? i * SL + sub : NB - 1); };
  T acc[NR];
#pragma unroll
  for (int i = 0; i < NR; ++i) acc[i] = T(0);
#pragma unroll
  for (int k = 0; k < NF; ++k) {
    const int fs = slots[k];
    T r[GS], x[NFQ];
    if constexpr (L::AHEAD) {
#pragma unroll
      for (int h = 0; h < L::GV; ++h) {
        T y[VECW<T>];
        load_row<T, VECW<T>>(sG + ((k * L::GV + h) * L::NT + threadIdx.x) * VECW<T>, y);
#pragma unroll
        for (int i = 0; i < VECW<T>; ++i) r[h * VECW<T> + i] = y[i];
      }
    } else {
      const T* g = G + ((int64_t)slot_face<O>(fs) * NV + w) * GS;
      if constexpr (PADG) {
        load_row<T, GS, true>(g, r);
      } else {
#pragma unroll
        for (int q = 0; q < NFQ; ++q) r[q] = __ldg(g + q);
      }
    }
    face_fluxes<T, D, P, GS>(r, fs, x);
    T face[NR];
#pragma unroll
    for (int i = 0; i < NR; ++i) face[i] = PARTS ? T(0) : acc[i];
    if constexpr (D == 3 && P == 1) {
      // the collapsed face rule is not symmetric: the table of the side's vertex permutation
      const T* tb = d.BfP + ((k * NPERM + slot_perm(fs)) * NFQ) * PADV<T, NB>;
#pragma unroll
      for (int q = 0; q < NFQ; ++q) {
        if constexpr (SL == 1) {
          T tr[PADV<T, NB>];
          load_row<T, PADV<T, NB>, true>(tb + q * PADV<T, NB>, tr);
#pragma unroll
          for (int i = 0; i < NR; ++i) face[i] = fma(tr[i], x[q], face[i]);
        } else {
#pragma unroll
          for (int i = 0; i < NR; ++i) face[i] = fma(__ldg(tb + q * PADV<T, NB> + row(i)), x[q], face[i]);
        }
      }
    } else {
#pragma unroll
      for (int q = 0; q < NFQ; ++q)
#pragma unroll
        for (int i = 0; i < NR; ++i) face[i] = fma(tab[X::BF + (k * NFQ + q) * NB + row(i)], x[q], face[i]);
    }
#pragma unroll
    for (int i = 0; i < NR; ++i) acc[i] = PARTS ? acc[i] + face[i] : face[i];
  }
  // the lift carries 1/sqrt|det|; the volume term sqrt|det| (flux) or nothing (the factors of the
  // trace and the test cancel in the derivative)
  const T ls = MODE == ELEM_FLUX ? isd * isd : isd;
#pragma unroll
  for (int i = 0; i < NR; ++i) acc[i] *= ls;
  if constexpr (P > 0) {
#pragma unroll
    for (int dd = 0; dd < D; ++dd) {
      T m[NB1 > 0 ? NB1 : 1], m2[NB1 > 0 ? NB1 : 1], vol[NR];
#pragma unroll
      for (int k = 0; k < NB1; ++k) m[k] = m2[k] = T(0);
      const T f0 = SHIFT ? sF[(dd * NV + w) * ET + tl] : T(0);
#pragma unroll
      for (int i = 0; i < (NQ + SL - 1) / SL; ++i) {
        const bool in = NQ % SL == 0 || i * SL + sub < NQ;
        const int q = in ? i * SL + sub : 0;
        T f = in ? sF[((q * D + dd) * NV + w) * ET + tl] : T(0);
        if constexpr (SHIFT) f = in ? f - f0 : T(0);
#pragma unroll
        for (int k = 0; k < NB1; ++k) {
          if (HALVES && (i & 1)) m2[k] = fma(tab[X::WM + q * NB1 + k], f, m2[k]);
          else m[k] = fma(tab[X::WM + q * NB1 + k], f, m[k]);
        }
      }
      if constexpr (HALVES) {
#pragma unroll
        for (int k = 0; k < NB1; ++k) m[k] += m2[k];
      }
#pragma unroll
      for (int i = 0; i < NR; ++i) vol[i] = PARTS ? T(0) : acc[i];
      if constexpr (SL == 1) {
        combine_modes<T, D, P, 1>(tab + X::CM + dd * NB * NB1, m, vol);
      } else {
#pragma unroll
        for (int k = 0; k < NB1; ++k)
#pragma unroll
          for (int o = ET; o < 32; o *= 2) m[k] += __shfl_xor_sync(0xffffffffu, m[k], o);
#pragma unroll
        for (int i = 0; i < NR; ++i)
#pragma unroll
          for (int k = 0; k < NB1; ++k) vol[i] = fma(tab[X::CM + (dd * NB + row(i)) * NB1 + k], m[k], vol[i]);
      }
      if constexpr (SHIFT) {
#pragma unroll
        for (int i = 0; i < NR; ++i)
          vol[i] = fma(tab[X::CH + dd * NB + row(i)], f0, fma(tab[X::CL + dd * NB + row(i)], f0, vol[i]));
      }
#pragma unroll
      for (int i = 0; i < NR; ++i) acc[i] = PARTS ? acc[i] + vol[i] : vol[i];
    }
  }
  T sc = oscale ? (T)*oscale : T(1);
  if (escale) sc *= escale[e];
  if (d.rot && w >= 1 && w <= D) {  // the frame's source, on the coefficients of u (R) or du (J v)
    const T so = MODE == ELEM_FLUX ? isd : T(1);
    const T* ra = rows + el * RS;
#pragma unroll
    for (int i = 0; i < NR; ++i) {
      T m[D];
#pragma unroll
      for (int k = 0; k < D; ++k) m[k] = ra[(1 + k) * NB + row(i)];
      acc[i] += rot_source<T, D>(d.om, m, w - 1) * so;
    }
  }
  if (d.rot) __syncthreads();  // the rows have been read before they are overwritten
  if constexpr (MODE == ELEM_FLUX) sc *= ge[O::SD];
#pragma unroll
  for (int i = 0; i < NR; ++i)
    if (SL == 1 || i * SL + sub < NB) rows[tl * RS + w * NB + row(i)] = acc[i] * sc;
  __syncthreads();
  for (int i = threadIdx.x; i < ne * NVB; i += L::NT) out[e0 * NVB + i] = rows[i / NVB * RS + i % NVB];
}

// Elements per SM up to which four lanes share an element (measured, see elem_op_kernel).
constexpr int FEW_ELEMENTS = 32;
template <class T, int D, int P, int MODE, bool PADG>
static void elem_op_launch(const DGData<T>& d, const T* u, const T* du, const T* pts, const T* G, T* out,
                           const T* escale, const int* skip, const double* oscale, cudaStream_t st) {
  auto run = [&](auto lanes) {
    constexpr int SL = decltype(lanes)::value;
    using L = ElemTile<T, D, P, MODE, SL>;
    elem_op_kernel<T, D, P, MODE, PADG, SL><<<(unsigned)((d.E + L::ET - 1) / L::ET), L::NT, L::BYTES, st>>>(
        d, u, du, pts, G, out, escale, skip, oscale);
  };
  if constexpr (P > 0) {
    if (d.E <= FEW_ELEMENTS * (int64_t)sm_count()) return run(std::integral_constant<int, 4>());
  }
  run(std::integral_constant<int, 1>());
}

template <class T, int D, int P>
cudaError_t dg_op_p(const DGData<T>& d, const T* u, const T* du, T* out, T* G, const T* escale, const int* skip,
                    const double* oscale, cudaStream_t st, const cudaEvent_t* ev, bool tight) {
  using O = Ord<D, P>;
  const int64_t nfp = d.F * O::NFQ;
  const unsigned nb = (unsigned)((nfp + 255) / 256);
  if (tight) {
    if constexpr (std::is_same<T, double>::value) {
      if (du) return cudaErrorInvalidValue;
      if (nfp > 0) face_kernel<T, D, P, false, false><<<nb, 256, 0, st>>>(d, u, du, G, skip);
      elem_op_launch<T, D, P, ELEM_FLUX, false>(d, u, nullptr, nullptr, G, out, escale, skip, oscale, st);
      return cudaGetLastError();
    }
    return cudaErrorInvalidValue;
  }
  if (ev) cudaEventRecord(ev[0], st);
  if (nfp > 0) {
    if (du) face_kernel<T, D, P, true, true><<<nb, 256, 0, st>>>(d, u, du, G, skip);
    else face_kernel<T, D, P, false, true><<<nb, 256, 0, st>>>(d, u, du, G, skip);
  }
  if (ev) cudaEventRecord(ev[1], st);
  if (du) elem_op_launch<T, D, P, ELEM_TANGENT, true>(d, u, du, nullptr, G, out, escale, skip, oscale, st);
  else elem_op_launch<T, D, P, ELEM_FLUX, true>(d, u, nullptr, nullptr, G, out, escale, skip, oscale, st);
  if (ev) cudaEventRecord(ev[2], st);
  return cudaGetLastError();
}

// Uploads c_tab and raises the shared-memory limits of the element kernels (current device).
template <class T, int D, int P>
cudaError_t upload_tables_p(const double* Bv, const double* Dv, const double* Wv, const double* Bf, cudaStream_t st) {
  using O = Ord<D, P>;
  using X = TabLayout<D, P>;
  constexpr int NB = O::NB, NQ = O::NQ, NB1 = X::NB1;
  T tab[X::N];
  for (int i = 0; i < NQ * NB; ++i) tab[X::BV + i] = (T)Bv[i];
  for (int q = 0; q < NQ; ++q)
    for (int k = 0; k < NB1; ++k) tab[X::WM + q * NB1 + k] = (T)(Wv[q] * Bv[q * NB + k]);
  for (int dd = 0; dd < D; ++dd)
    for (int i = 0; i < NB; ++i)
      for (int k = 0; k < NB1; ++k) {
        double a = 0;  // sum_q w_q d phi_i / d xi_d phi_k (Dv carries w_q)
        for (int q = 0; q < NQ; ++q) a += Dv[(dd * NQ + q) * NB + i] * Bv[q * NB + k];
        tab[X::CM + (dd * NB + i) * NB1 + k] = (T)a;
      }
  for (int dd = 0; dd < D; ++dd)
    for (int i = 0; i < NB; ++i) {
      double a = 0;
      for (int q = 0; q < NQ; ++q) a += Dv[(dd * NQ + q) * NB + i];
      tab[X::CH + dd * NB + i] = (T)a;
      tab[X::CL + dd * NB + i] = (T)(a - (double)(T)a);
    }
  for (int f = 0; f < O::NF; ++f)
    for (int i = 0; i < O::NFQ * NB; ++i) tab[X::BF + f * O::NFQ * NB + i] = (T)Bf[(f * O::NPERM) * O::NFQ * NB + i];
  cudaError_t e = cudaMemcpyToSymbolAsync(c_tab<T, D, P>, tab, sizeof(tab), 0, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  auto allow = [&](auto kernel, size_t bytes) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  };
  allow(elem_op_kernel<T, D, P, ELEM_FLUX, true, 1>, ElemTile<T, D, P, ELEM_FLUX>::BYTES);
  allow(elem_op_kernel<T, D, P, ELEM_TANGENT, true, 1>, ElemTile<T, D, P, ELEM_TANGENT>::BYTES);
  allow(elem_op_kernel<T, D, P, ELEM_STORED, true, 1>, ElemTile<T, D, P, ELEM_STORED>::BYTES);
  if constexpr (std::is_same<T, double>::value)
    allow(elem_op_kernel<T, D, P, ELEM_FLUX, false, 1>, ElemTile<T, D, P, ELEM_FLUX>::BYTES);
  return e;
}

// U[v] = isd sum_j b[j] ue[v][j]: the trace of an element's coefficients at a point, table row b
// in global memory
template <class T, int D, int P>
PCEXP_DEV void point_trace(const T* b, const T* __restrict__ ue, T isd, T (&U)[D + 2]) {
  constexpr int NB = Ord<D, P>::NB, NV = D + 2;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    T a = 0;
#pragma unroll
    for (int j = 0; j < NB; ++j) a += __ldg(b + j) * ue[v * NB + j];
    U[v] = a * isd;
  }
}

// Reverse sweep of a face's Riemann flux: Lb, Rb += its adjoints; on boundary faces (eR < 0, R the
// ghost state of L) the ghost's adjoint is folded into Lb.
template <class T, int D>
PCEXP_DEV void face_flux_vjp(const DGData<T>& d, int eR, const T (&L)[D + 2], const T (&R)[D + 2], const T (&n)[D],
                             T vrn, const T (&gb)[D + 2], T (&Lb)[D + 2], T (&Rb)[D + 2]) {
  roe_flux_vjp<D, T, T>(L, R, n, d.fs.gamma, gb, Lb, Rb, vrn);
  if (eR >= 0) return;
  if (mirror_bc(eR)) {
    ghost_slip_wall_vjp<D, T, T>(n, Rb, Lb, vrn);
  } else {
    T vib[D];
#pragma unroll
    for (int k = 0; k < D; ++k) vib[k] = T(0);
    ghost_farfield_vjp<D, T, T>(L, n, d.fs, Rb, Lb, vib);
  }
}

// ------------------------------------------------------- linearisation
// The exact Jacobian of the scheme (Eq. jac1, jac2) point by point.  Faces: the Riemann-flux
// Jacobians dF~/dU_L, dF~/dU_R, evaluated exactly by reverse sweeps (the paper obtains them by AD as
// well).  Volume: the velocity and the total enthalpy, from which the derivative of the Euler flux
// along any direction costs fewer operations than a product with its stored D nv x nv Jacobian
// (51 against 75 FMAs per point on tetrahedra), and 4 values per point instead of D nv^2.
// Every J v of a PCEXP step is taken at u_n, so both are built once per step.
//   pts [nq][E][4]: velocity (D), H = (E + p) / rho; in 2D the fourth entry is unused
template <class T, int D, int P>
__global__ void __launch_bounds__(256) linearize_vol_kernel(DGData<T> d, const T* __restrict__ u,
                                                            T* __restrict__ pts) {
  using O = Ord<D, P>;
  constexpr int NB = O::NB, NQ = O::NQ, NV = O::NV, GEO = O::GEO;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;  // points of an element together
  if (idx >= d.E * NQ) return;
  const int64_t e = idx / NQ;
  const int q = (int)(idx - e * NQ);
  T U[NV];
  point_trace<T, D, P>(d.Bv + q * NB, u + e * NV * NB, d.geo[GEO * e + O::ISD], U);
  const T ir = T(1) / U[0];
  T x[4] = {T(0), T(0), T(0), T(0)}, k2 = T(0);
#pragma unroll
  for (int k = 0; k < D; ++k) {
    x[k] = U[1 + k] * ir;
    k2 = fma(T(0.5) * x[k], x[k], k2);
  }
  x[D] = (U[NV - 1] + (d.fs.gamma - T(1)) * (U[NV - 1] - k2 * U[0])) * ir;
  T* o = pts + ((int64_t)q * d.E + e) * 4;
#pragma unroll
  for (int k = 0; k < 4; ++k) o[k] = x[k];
}

// The face blocks come row by row from reverse sweeps of the Roe flux: with the adjoint e_v one
// sweep gives row v of both dF~/dU_L and dF~/dU_R (the flux's own intermediates are hoisted out of
// the loop), where a forward sweep per side carries D + 2 directions through every operation.
// FP64 at p = 2, 20^3 Kuhn cubes (96,000 faces): 3.5 -> 1.6 ms; bound by the FP64 pipe.
template <class T, int D, int P>
__global__ void __launch_bounds__(128) linearize_face_kernel(DGData<T> d, const T* __restrict__ u,
                                                             T* __restrict__ Bface) {
  using O = Ord<D, P>;
  constexpr int NB = O::NB, NFQ = O::NFQ, NV = O::NV, NPERM = O::NPERM, GEO = O::GEO, NN = NV * NV;
  const int64_t n = d.F * NFQ;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n) return;
  const int64_t f = idx / NFQ;
  const int q = (int)(idx - f * NFQ);
  const int eL = d.fel[2 * f], eR = d.fel[2 * f + 1];
  const int loc = d.floc[f];
  const int fL = loc & 0xff, fR = (loc >> 8) & 0xff, pR = loc >> 16;
  T nr[D];
#pragma unroll
  for (int k = 0; k < D; ++k) nr[k] = d.fgeo[4 * f + k];
  const T wq = d.fgeo[4 * f + D] * d.Wf[q];
  const T vrn = d.rot ? d.vrn[idx] : T(0);
  T L[NV], R[NV];
  const T isdL = d.geo[GEO * (int64_t)eL + O::ISD];
  T isdR = T(0);
  point_trace<T, D, P>(d.Bf + ((fL * NPERM) * NFQ + q) * NB, u + (int64_t)eL * NV * NB, isdL, L);
  if (eR >= 0) {
    isdR = d.geo[GEO * (int64_t)eR + O::ISD];
    point_trace<T, D, P>(d.Bf + ((fR * NPERM + pR) * NFQ + q) * NB, u + (int64_t)eR * NV * NB, isdR, R);
  } else if (mirror_bc(eR)) {
    ghost_slip_wall<D, T, T>(L, nr, R, vrn);
  } else {
    ghost_farfield<D, T, T>(L, nr, d.fs, R);
  }
  if constexpr (FACE_RECORDS<T, D>) {
    if (eR >= 0) {
      const RoeRecord<T, D> r = roe_record<D, T>(L, R, d.fs.gamma);
      const int64_t ni = d.F_int * NFQ;
      float4* o = reinterpret_cast<float4*>(Bface) + idx;
      o[0] = make_float4(r.vL[0], r.vL[1], r.vL[2], r.HL);
      o[ni] = make_float4(r.vR[0], r.vR[1], r.vR[2], r.HR);
      o[2 * ni] = make_float4(r.rL, r.irL, r.rR, r.irR);
      o[3 * ni] = make_float4(r.w, r.c, r.i2c, r.dp);
      return;
    }
  }
#pragma unroll 1
  for (int v = 0; v < NV; ++v) {
    T gb[NV], Lb[NV], Rb[NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) {
      gb[c] = c == v ? T(1) : T(0);
      Lb[c] = Rb[c] = T(0);
    }
    face_flux_vjp<T, D>(d, eR, L, R, nr, vrn, gb, Lb, Rb);
#pragma unroll
    for (int c = 0; c < NV; ++c) {
      if constexpr (FACE_RECORDS<T, D>) {
        const int64_t ni = d.F_int * NFQ;  // boundary blocks [nv nv][boundary points] after the records
        Bface[16 * ni + (v * NV + c) * (n - ni) + idx - ni] = wq * isdL * Lb[c];
      } else {
        Bface[bface_at<T, 2 * NN>(v * NV + c, idx, n)] = wq * isdL * Lb[c];
        Bface[bface_at<T, 2 * NN>(NN + v * NV + c, idx, n)] = eR >= 0 ? wq * isdR * Rb[c] : T(0);
      }
    }
  }
}

template <class T, int D, int P>
__global__ void __launch_bounds__(256) face_apply_kernel(DGData<T> d, const T* __restrict__ Bface,
                                                         const T* __restrict__ dv, T* __restrict__ G,
                                                         const int* __restrict__ skip) {
  using O = Ord<D, P>;
  constexpr int NB = O::NB, NFQ = O::NFQ, NV = O::NV, NPERM = O::NPERM, NN = NV * NV;
  constexpr bool SM = O::SMEM_BF;
  __shared__ T sBf[SM ? O::NBF : 1];
  if (skip && *skip) return;
  if constexpr (SM)
    for (int i = threadIdx.x; i < O::NBF; i += blockDim.x) sBf[i] = d.Bf[i];
  __syncthreads();
  const T* Bf = SM ? sBf : d.Bf;
  const int64_t n = d.F * NFQ;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n) return;
  const int64_t f = idx / NFQ;
  const int q = (int)(idx - f * NFQ);
  const int eL = d.fel[2 * f], eR = d.fel[2 * f + 1];
  const int loc = d.floc[f];
  const int fL = loc & 0xff, fR = (loc >> 8) & 0xff, pR = loc >> 16;
  // the point's block in 16-byte vectors (bface_at); chunks wholly on the R side are not
  // loaded on boundary faces (the linearisation stores zeros there)
  T B[O::NJF];
  {
    constexpr int VEC = 16 / (int)sizeof(T), NCH = O::NJF / VEC, R = O::NJF % VEC;
    const bool two = eR >= 0;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      if (c * VEC < NN || two) {
        T x[VEC];
        load_row<T, VEC, true>(Bface + ((int64_t)c * n + idx) * VEC, x);
#pragma unroll
        for (int i = 0; i < VEC; ++i) B[c * VEC + i] = x[i];
      } else {
#pragma unroll
        for (int i = 0; i < VEC; ++i) B[c * VEC + i] = T(0);
      }
    }
    if constexpr (R > 0) {
      static_assert(R == 2 && sizeof(T) == 4, "the remainder of a point's block is one float pair");
      const float2 x = two ? __ldg(reinterpret_cast<const float2*>(Bface + (int64_t)NCH * VEC * n + idx * R))
                           : make_float2(0.f, 0.f);
      B[NCH * VEC] = x.x;
      B[NCH * VEC + 1] = x.y;
    }
  }
  // traces of dv at the point from each side: the table row (shared memory in 2D; in 3D the
  // padded copy, 16-byte loads) and the element's rows of dv (8-byte loads when nb is even:
  // the kernel is bound by its load instructions as much as by its bytes)
  constexpr int NBP = PADV<T, NB>;
  auto trace = [&](int64_t e, int fl, int pm, T(&t)[NV]) {
    T b[NBP];
    if constexpr (SM) {
      const T* be = Bf + ((fl * NPERM + pm) * NFQ + q) * NB;
#pragma unroll
      for (int j = 0; j < NB; ++j) b[j] = be[j];
    } else {
      load_row<T, NBP, true>(d.BfP + ((fl * NPERM + pm) * NFQ + q) * NBP, b);
    }
    const T* ve = dv + e * NV * NB;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      T c[NB];
      load_coeffs<T, NB>(ve + v * NB, c);
      T a = 0;
#pragma unroll
      for (int j = 0; j < NB; ++j) a += b[j] * c[j];
      t[v] = a;
    }
  };
  T tL[NV], tR[NV];
  trace(eL, fL, 0, tL);
  if (eR >= 0) trace(eR, fR, pR, tR);
  T g[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    T a = 0;
#pragma unroll
    for (int c = 0; c < NV; ++c) a += B[v * NV + c] * tL[c];
    if (eR >= 0) {
#pragma unroll
      for (int c = 0; c < NV; ++c) a += B[NN + v * NV + c] * tR[c];
    }
    g[v] = a;
  }
  store_face_flux<T, D, P, true>(G, f, q, g);
}

// Face part of the FP32 J v on tetrahedra.  With stored Jacobians (50 values per point) it was bound
// by their bytes, 85% of its traffic; it now recomputes the Roe flux's derivative from 16 stored
// values of the linearisation (about 210 FMAs, next to 100 of the two traces): FP32 arithmetic is
// cheap here, bytes are not.  Per launch 392 -> 279 us on 48^3 cubes at p = 2, 18.5 -> 12.5 us on
// 21^3 cubes at p = 1.  What bounds it now is the latency of the gather face -> elements -> rows
// against the warps in flight: with 70 registers (three blocks per SM) it took 340 us, with two
// points per thread 366.  Boundary points, whose ghost state's derivative may hold powers, keep
// their nv x nv block.  FP64 keeps blocks: there the arithmetic is the bound and a block product
// (50 FMAs) is the cheaper form.  On triangles a block has 32 values and the gather of dv's rows
// through L1 is the bound: 28.6 us with blocks, 28.8 with records (131,072 triangles at p = 3), so
// blocks stay.
template <int D, int P>
__global__ void __launch_bounds__(256, 4) face_record_kernel(DGData<float> d, const float* __restrict__ rec,
                                                          const float* __restrict__ dv, float* __restrict__ G,
                                                          const int* __restrict__ skip) {
  using O = Ord<D, P>;
  constexpr int NB = O::NB, NFQ = O::NFQ, NV = O::NV, NPERM = O::NPERM, GEO = O::GEO, NBP = PADV<float, NB>;
  if (skip && *skip) return;
  const int64_t n = d.F * NFQ, ni = d.F_int * NFQ;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n) return;
  const int64_t f = idx / NFQ;
  const int q = (int)(idx - f * NFQ);
  const int2 el = __ldg(reinterpret_cast<const int2*>(d.fel) + f);
  const int loc = __ldg(d.floc + f);
  // traces of dv from each side: a padded table row and the element's rows of dv
  auto trace = [&](int64_t e, int row, float isd, float(&t)[NV]) {
    float b[NBP];
    load_row<float, NBP, true>(d.BfP + (int64_t)row * NBP, b);
    const float* ve = dv + e * NV * NB;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      float c[NB];
      load_coeffs<float, NB>(ve + v * NB, c);
      float a = 0.f;
#pragma unroll
      for (int j = 0; j < NB; ++j) a = fmaf(b[j], c[j], a);
      t[v] = a * isd;
    }
  };
  float tL[NV], g[NV];
  if (idx >= ni) {
    trace(el.x, ((loc & 0xff) * NPERM) * NFQ + q, 1.f, tL);
    const float* B = rec + 16 * ni + (idx - ni);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      g[v] = 0.f;
#pragma unroll
      for (int c = 0; c < NV; ++c) g[v] = fmaf(__ldg(B + (v * NV + c) * (n - ni)), tL[c], g[v]);
    }
    store_face_flux<float, D, P, true>(G, f, q, g);
    return;
  }
  const float4* x = reinterpret_cast<const float4*>(rec) + idx;
  const float4 xL = __ldg(x), xR = __ldg(x + ni), rho = __ldg(x + 2 * ni), m = __ldg(x + 3 * ni);
  const float4 geo = __ldg(reinterpret_cast<const float4*>(d.fgeo) + f);
  const float nr[D] = {geo.x, geo.y, geo.z};
  float tR[NV], dF[NV];
  trace(el.x, ((loc & 0xff) * NPERM) * NFQ + q, __ldg(d.geo + GEO * (int64_t)el.x + O::ISD), tL);
  trace(el.y, (((loc >> 8) & 0xff) * NPERM + (loc >> 16)) * NFQ + q, __ldg(d.geo + GEO * (int64_t)el.y + O::ISD), tR);
  RoeRecord<float, D> r;
  r.vL[0] = xL.x, r.vL[1] = xL.y, r.vL[2] = xL.z, r.HL = xL.w;
  r.vR[0] = xR.x, r.vR[1] = xR.y, r.vR[2] = xR.z, r.HR = xR.w;
  r.rL = rho.x, r.irL = rho.y, r.rR = rho.z, r.irR = rho.w;
  r.w = m.x, r.c = m.y, r.i2c = m.z, r.dp = m.w;
  roe_derivative<D, float>(r, nr, d.fs.gamma, d.rot ? d.vrn[idx] : 0.f, tL, tR, dF);
  const float wl = geo.w * __ldg(d.Wf + q);
#pragma unroll
  for (int v = 0; v < NV; ++v) g[v] = wl * dF[v];
  store_face_flux<float, D, P, true>(G, f, q, g);
}

template <class T, int D, int P>
cudaError_t linearize_p(const DGData<T>& d, const T* u, LinData<T> lin, cudaStream_t st) {
  using O = Ord<D, P>;
  const int64_t nv = d.E * O::NQ, nf = d.F * O::NFQ;
  linearize_vol_kernel<T, D, P><<<(unsigned)((nv + 255) / 256), 256, 0, st>>>(d, u, lin.pts);
  if (nf > 0) linearize_face_kernel<T, D, P><<<(unsigned)((nf + 127) / 128), 128, 0, st>>>(d, u, lin.Bface);
  return cudaGetLastError();
}

// J v from the face point Jacobians and the stored volume points.
template <class T, int D, int P>
cudaError_t jac_apply_p(const DGData<T>& d, LinData<T> lin, const T* dv, T* out, T* G, const T* escale,
                        const int* skip, const double* oscale, cudaStream_t st, const cudaEvent_t* ev) {
  using O = Ord<D, P>;
  const int64_t nf = d.F * O::NFQ;
  if (ev) cudaEventRecord(ev[0], st);
  if (nf > 0) {
    const unsigned nb = (unsigned)((nf + 255) / 256);
    if constexpr (FACE_RECORDS<T, D>) face_record_kernel<D, P><<<nb, 256, 0, st>>>(d, lin.Bface, dv, G, skip);
    else face_apply_kernel<T, D, P><<<nb, 256, 0, st>>>(d, lin.Bface, dv, G, skip);
  }
  if (ev) cudaEventRecord(ev[1], st);
  elem_op_launch<T, D, P, ELEM_STORED, true>(d, nullptr, dv, lin.pts, G, out, escale, skip, oscale, st);
  if (ev) cudaEventRecord(ev[2], st);
  return cudaGetLastError();
}

// ------------------------------------------------------------- adjoint J^T w
// Transpose of the point-Jacobian J v (same linearisation state).  With the output
// factors of J v folded into w (w~ = osc * escale_e * w), the face kernel forms the
// adjoint of the lifted face flux at every face point,
//   Gbar = -(1/sd_L) sum_i Bf_L[i] w~_L[i] + (1/sd_R) sum_i Bf_R[i] w~_R[i],
// and stores B_L^T Gbar and B_R^T Gbar; the element kernel applies the transposed
// flux derivatives to the transposed test of w~ and gathers the transposed traces
// of its faces.  Deterministic (no atomics).
template <class T, int D, int P>
__global__ void __launch_bounds__(256) face_adjoint_kernel(DGData<T> d, const T* __restrict__ Bface,
                                                           const T* __restrict__ w, T* __restrict__ GT,
                                                           const T* __restrict__ escale, T osc) {
  using O = Ord<D, P>;
  constexpr int NB = O::NB, NFQ = O::NFQ, NV = O::NV, NPERM = O::NPERM, GEO = O::GEO, NN = NV * NV;
  constexpr bool SM = O::SMEM_BF;
  static_assert(!FACE_RECORDS<T, D>, "this kernel reads a block per face point, not a record");
  __shared__ T sBf[SM ? O::NBF : 1];
  if constexpr (SM)
    for (int i = threadIdx.x; i < O::NBF; i += blockDim.x) sBf[i] = d.Bf[i];
  __syncthreads();
  const T* Bf = SM ? sBf : d.Bf;
  const int64_t n = d.F * NFQ;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n) return;
  const int64_t f = idx / NFQ;
  const int q = (int)(idx - f * NFQ);
  const int eL = d.fel[2 * f], eR = d.fel[2 * f + 1];
  const int loc = d.floc[f];
  const int fL = loc & 0xff, fR = (loc >> 8) & 0xff, pR = loc >> 16;
  T gb[NV];
  {
    const T sc = -osc * (escale ? escale[eL] : T(1)) * d.geo[GEO * (int64_t)eL + O::ISD];
    const T* be = Bf + ((fL * NPERM) * NFQ + q) * NB;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      T a = 0;
#pragma unroll
      for (int i = 0; i < NB; ++i) a += tab<SM>(be + i) * w[(int64_t)eL * NV * NB + v * NB + i];
      gb[v] = sc * a;
    }
  }
  if (eR >= 0) {
    const T sc = osc * (escale ? escale[eR] : T(1)) * d.geo[GEO * (int64_t)eR + O::ISD];
    const T* be = Bf + ((fR * NPERM + pR) * NFQ + q) * NB;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      T a = 0;
#pragma unroll
      for (int i = 0; i < NB; ++i) a += tab<SM>(be + i) * w[(int64_t)eR * NV * NB + v * NB + i];
      gb[v] += sc * a;
    }
  }
  T* o = GT + idx * 2 * NV;
#pragma unroll
  for (int side = 0; side < 2; ++side)
#pragma unroll
    for (int c = 0; c < NV; ++c) {
      T a = 0;
      if (side == 0 || eR >= 0) {
#pragma unroll
        for (int v = 0; v < NV; ++v) a += Bface[bface_at<T, 2 * NN>(side * NN + v * NV + c, idx, n)] * gb[v];
      }
      o[side * NV + c] = a;
    }
}

// transposed face traces of the D+1 faces for coefficient j of variable c of element e
template <class T, int D, int P, bool SM>
PCEXP_DEV T gather_faces_T(const DGData<T>& d, const T* Bf, const T* __restrict__ GT, int64_t e, int c, int j) {
  using O = Ord<D, P>;
  constexpr int NB = O::NB, NFQ = O::NFQ, NV = O::NV, NPERM = O::NPERM, NF = O::NF;
  T acc = 0;
#pragma unroll
  for (int k = 0; k < NF; ++k) {
    const int fs = d.ef[NF * e + k];
    const T* gt = GT + (int64_t)slot_face<O>(fs) * NFQ * 2 * NV + slot_side(fs) * NV + c;
    const T* tb = Bf + ((k * NPERM + slot_perm(fs)) * NFQ) * NB + j;
#pragma unroll
    for (int q = 0; q < NFQ; ++q) acc += tab<SM>(tb + q * NB) * gt[q * 2 * NV];
  }
  return acc;
}

template <class T, int D, int P>
__global__ void __launch_bounds__(256) elem_adjoint_kernel(DGData<T> d, const T* __restrict__ pts,
                                                           const T* __restrict__ w, const T* __restrict__ GT,
                                                           T* __restrict__ out, const T* __restrict__ escale,
                                                           T osc) {
  using O = Ord<D, P>;
  constexpr int NB = O::NB, NQ = O::NQ, ET = O::ET, NVB = O::NVB, NV = O::NV;
  constexpr bool SM = O::SMEM_BF;
  __shared__ T sBv[NQ * NB];
  __shared__ T sDv[D * NQ * NB];
  __shared__ T sBf[SM ? O::NBF : 1];
  __shared__ T sw[ET * NVB];
  __shared__ T sU[ET * NQ * NV];
  static_assert(ET * NQ <= 256, "one volume point per thread");
  const int64_t e0 = (int64_t)blockIdx.x * ET;
  const int ne = (int)((d.E - e0) < ET ? (d.E - e0) : ET);
  for (int i = threadIdx.x; i < NQ * NB; i += blockDim.x) sBv[i] = d.Bv[i];
  for (int i = threadIdx.x; i < D * NQ * NB; i += blockDim.x) sDv[i] = d.Dv[i];
  if constexpr (SM)
    for (int i = threadIdx.x; i < O::NBF; i += blockDim.x) sBf[i] = d.Bf[i];
  for (int i = threadIdx.x; i < ne * NVB; i += blockDim.x)
    sw[i] = w[e0 * NVB + i] * osc * (escale ? escale[e0 + i / NVB] : T(1));
  __syncthreads();
  // phase 1: transposed test, then the transposed flux derivative, at this thread's point
  const int el1 = threadIdx.x / NQ, q1 = threadIdx.x - (threadIdx.x / NQ) * NQ;
  if (threadIdx.x < ne * NQ) {
    const int64_t e = e0 + el1;
    T fb[D][NV];
#pragma unroll
    for (int dd = 0; dd < D; ++dd)
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        T a = 0;
#pragma unroll
        for (int i = 0; i < NB; ++i) a += sDv[(dd * NQ + q1) * NB + i] * sw[el1 * NVB + v * NB + i];
        fb[dd][v] = a;
      }
    T pv[4], Ub[NV], k2 = T(0), dpb = T(0);
    load_row<T, 4, true>(pts + ((int64_t)q1 * d.E + e) * 4, pv);
    const T gm = d.fs.gamma - T(1);
#pragma unroll
    for (int c = 0; c < NV; ++c) Ub[c] = T(0);
#pragma unroll
    for (int k = 0; k < D; ++k) k2 = fma(T(0.5) * pv[k], pv[k], k2);
    // transpose of the derivative of elem_op_kernel: w_d = A_d . dm - q_d drho,
    // dF_d = (A_d . dm, v w_d + q_d dm + A_d dp, H w_d + q_d (dE + dp))
#pragma unroll
    for (int dd = 0; dd < D; ++dd) {
      const T* A = d.geo + O::GEO * e + dd * D;
      T qd = A[0] * pv[0], wb = fb[dd][NV - 1] * pv[D], pb = T(0);
#pragma unroll
      for (int k = 1; k < D; ++k) qd = fma(A[k], pv[k], qd);
#pragma unroll
      for (int k = 0; k < D; ++k) {
        wb = fma(fb[dd][1 + k], pv[k], wb);
        pb = fma(fb[dd][1 + k], A[k], pb);
      }
      const T f0b = fb[dd][0] + wb, eb = fb[dd][NV - 1] * qd;
      dpb += pb + eb;
      Ub[NV - 1] += eb;
      Ub[0] = fma(-qd, wb, Ub[0]);
#pragma unroll
      for (int k = 0; k < D; ++k) Ub[1 + k] = fma(A[k], f0b, fma(fb[dd][1 + k], qd, Ub[1 + k]));
      if (d.rot) {  // rotating frame: the flux is F - U v_r^T
        const T* vr = d.vrq + (e * NQ + q1) * D;
        T vd = A[0] * vr[0];
#pragma unroll
        for (int k = 1; k < D; ++k) vd = fma(A[k], vr[k], vd);
#pragma unroll
        for (int c = 0; c < NV; ++c) Ub[c] = fma(-vd, fb[dd][c], Ub[c]);
      }
    }
    dpb *= gm;
    Ub[0] = fma(k2, dpb, Ub[0]);
    Ub[NV - 1] += dpb;
#pragma unroll
    for (int k = 0; k < D; ++k) Ub[1 + k] = fma(-pv[k], dpb, Ub[1 + k]);
#pragma unroll
    for (int c = 0; c < NV; ++c) sU[(el1 * NQ + q1) * NV + c] = Ub[c];
  }
  __syncthreads();
  const T* Bf = SM ? sBf : d.Bf;
  // phase 2: transposed volume traces plus the transposed face traces
  for (int it = threadIdx.x; it < ne * NVB; it += blockDim.x) {
    const int el = it / NVB, r = it - el * NVB;
    const int c = r / NB, j = r - c * NB;
    T acc = 0;
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc += sBv[q * NB + j] * sU[(el * NQ + q) * NV + c];
    acc += gather_faces_T<T, D, P, SM>(d, Bf, GT, e0 + el, c, j);
    if (d.rot && c >= 1 && c <= D) {  // transpose of the source -omega x: +omega x w~ (antisymmetric)
      T m[D];
#pragma unroll
      for (int k = 0; k < D; ++k) m[k] = sw[el * NVB + (1 + k) * NB + j];
      acc -= rot_source<T, D>(d.om, m, c - 1);
    }
    out[e0 * NVB + it] = acc;
  }
}

template <class T, int D, int P>
cudaError_t jac_adjoint_p(const DGData<T>& d, LinData<T> lin, const T* w, T* out, T* GT, const T* escale, T osc,
                          cudaStream_t st) {
  using O = Ord<D, P>;
  const int64_t nf = d.F * O::NFQ;
  if (nf > 0) face_adjoint_kernel<T, D, P><<<(unsigned)((nf + 255) / 256), 256, 0, st>>>(d, lin.Bface, w, GT, escale, osc);
  const int64_t eb = (d.E + O::ET - 1) / O::ET;
  elem_adjoint_kernel<T, D, P><<<(unsigned)eb, 256, 0, st>>>(d, lin.pts, w, GT, out, escale, osc);
  return cudaGetLastError();
}

// ------------------------------------------- second-order adjoint (d(J(u) v)/du)^T w
// S(u) = w~^T J(u) v is differentiated with respect to the linearisation state u: at every
// point the transposed test (volume) or transposed lift (faces) of w~ is the adjoint of the flux,
// the reverse sweep of the flux (roe_flux_vjp, euler_flux_vjp, the ghost states') runs on
// Tangent numbers carrying the traces of v, and the derivative parts of its results are
// d/du [w~^T F'(u) v], mapped back through the transposed traces.  Same output factors and
// scratch layout as the adjoint kernels.
//
// Bound by the FP64 pipe (2 FMA per clock and SM).  One sweep serves both sides of a face; on
// hyper-dual numbers every operation carried 2 (D + 2) + 2 components and each side took a pass
// of its own.  Bump channel, 6,144 triangles at p = 2, m = 30: the reverse step 48.2 -> 27.0 ms,
// 61 launches of each kernel (faces 311, elements 67 and the separate free-stream pass 78 us per
// launch before).
//
// theta (nullable): per boundary-face point (faces f0..F) two sums that grow by
// osc * (*osc_dev) * d/dtheta_k [gbar^T (dF~/dU_L) t_L], theta = (Mach number, flow angle), from the
// far-field ghost state's adjoint of the free-stream velocity; dvel = {dvel/dMach (x, y),
// dvel/dalpha (x, y)}.  Each entry belongs to one thread; theta_sum_kernel adds them up.
template <class T, int D, int P>
__global__ void __launch_bounds__(128) face_hess_kernel(DGData<T> d, const T* __restrict__ u,
                                                        const T* __restrict__ v, const T* __restrict__ w,
                                                        T* __restrict__ GT, const T* __restrict__ escale, T osc,
                                                        ThetaSums<T> th) {
  using O = Ord<D, P>;
  constexpr int NB = O::NB, NFQ = O::NFQ, NV = O::NV, NPERM = O::NPERM, GEO = O::GEO;
  using S = Tangent<T>;
  const int64_t n = d.F * NFQ;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n) return;
  const int64_t f = idx / NFQ;
  const int q = (int)(idx - f * NFQ);
  const int eL = d.fel[2 * f], eR = d.fel[2 * f + 1];
  const int loc = d.floc[f];
  const int fL = loc & 0xff, fR = (loc >> 8) & 0xff, pR = loc >> 16;
  T nr[D];
#pragma unroll
  for (int k = 0; k < D; ++k) nr[k] = d.fgeo[4 * f + k];
  const T wq = d.fgeo[4 * f + D] * d.Wf[q];
  const T isdL = d.geo[GEO * (int64_t)eL + O::ISD];
  const T isdR = eR >= 0 ? d.geo[GEO * (int64_t)eR + O::ISD] : T(0);
  const T* bL = d.Bf + ((fL * NPERM) * NFQ + q) * NB;
  const T* bR = d.Bf + ((fR * NPERM + (eR >= 0 ? pR : 0)) * NFQ + q) * NB;
  S L[NV], R[NV];
  T gb[NV];
  const T scL = -osc * (escale ? escale[eL] : T(1)) * isdL;
#pragma unroll
  for (int c = 0; c < NV; ++c) {
    T a = 0, b = 0, g = 0;
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      const int64_t o = (int64_t)eL * NV * NB + c * NB + j;
      const T bj = __ldg(bL + j);
      a += bj * u[o];
      b += bj * v[o];
      g += bj * w[o];
    }
    L[c] = S{a * isdL, b * isdL};
    gb[c] = scL * g;
  }
  if (eR >= 0) {
    const T scR = osc * (escale ? escale[eR] : T(1)) * isdR;
#pragma unroll
    for (int c = 0; c < NV; ++c) {
      T a = 0, b = 0, g = 0;
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        const int64_t o = (int64_t)eR * NV * NB + c * NB + j;
        const T bj = __ldg(bR + j);
        a += bj * u[o];
        b += bj * v[o];
        g += bj * w[o];
      }
      R[c] = S{a * isdR, b * isdR};
      gb[c] += scR * g;
    }
  } else if (mirror_bc(eR)) {
    ghost_slip_wall<D, S, T>(L, nr, R);
  } else {
    ghost_farfield<D, S, T>(L, nr, d.fs, R);
  }
  S Lb[NV], Rb[NV];
#pragma unroll
  for (int c = 0; c < NV; ++c) Lb[c] = Rb[c] = S{T(0), T(0)};
  roe_flux_vjp<D, S, T>(L, R, nr, d.fs.gamma, gb, Lb, Rb);
  if (eR < 0) {
    if (mirror_bc(eR)) {
      ghost_slip_wall_vjp<D, S, T>(nr, Rb, Lb);
    } else {
      S vib[D];
#pragma unroll
      for (int k = 0; k < D; ++k) vib[k] = S{T(0), T(0)};
      ghost_farfield_vjp<D, S, T>(L, nr, d.fs, Rb, Lb, vib);
      if (th.sums && eL < d.E_loc) {  // a halo element's faces count in their own partition
        const T sc = th.osc * (th.osc_dev ? *th.osc_dev : T(1)) * wq;
        T* o = th.sums + ((f - th.f0) * NFQ + q) * 2;
        o[0] += sc * (th.dvel[0] * vib[0].d + th.dvel[1] * vib[1].d);
        o[1] += sc * (th.dvel[2] * vib[0].d + th.dvel[3] * vib[1].d);
      }
    }
  }
  T* o = GT + idx * 2 * NV;
#pragma unroll
  for (int c = 0; c < NV; ++c) {
    o[c] = wq * isdL * Lb[c].d;
    o[NV + c] = eR >= 0 ? wq * isdR * Rb[c].d : T(0);
  }
}

// Element part of the second-order adjoint (HESS) or of J(u)^T w without stored Jacobians.
template <class T, int D, int P, bool HESS>
__global__ void __launch_bounds__(256) elem_hess_kernel(DGData<T> d, const T* __restrict__ u, const T* __restrict__ v,
                                                        const T* __restrict__ w, const T* __restrict__ GT,
                                                        T* __restrict__ out, const T* __restrict__ escale, T osc) {
  using O = Ord<D, P>;
  constexpr int NB = O::NB, NQ = O::NQ, ET = O::ET, NVB = O::NVB, NV = O::NV, GEO = O::GEO;
  constexpr bool SM = O::SMEM_BF;
  using S = typename std::conditional<HESS, Tangent<T>, T>::type;
  __shared__ T sBv[NQ * NB];
  __shared__ T sDv[D * NQ * NB];
  __shared__ T sBf[SM ? O::NBF : 1];
  __shared__ T su[ET * NVB];
  __shared__ T sv[HESS ? ET * NVB : 1];
  __shared__ T sw[ET * NVB];
  __shared__ T sU[ET * NQ * NV];
  __shared__ T sgeo[ET * GEO];
  static_assert(ET * NQ <= 256, "one volume point per thread");
  const int64_t e0 = (int64_t)blockIdx.x * ET;
  const int ne = (int)((d.E - e0) < ET ? (d.E - e0) : ET);
  for (int i = threadIdx.x; i < NQ * NB; i += blockDim.x) sBv[i] = d.Bv[i];
  for (int i = threadIdx.x; i < D * NQ * NB; i += blockDim.x) sDv[i] = d.Dv[i];
  if constexpr (SM)
    for (int i = threadIdx.x; i < O::NBF; i += blockDim.x) sBf[i] = d.Bf[i];
  for (int i = threadIdx.x; i < ne * NVB; i += blockDim.x) {
    su[i] = u[e0 * NVB + i];
    if constexpr (HESS) sv[i] = v[e0 * NVB + i];
    sw[i] = w[e0 * NVB + i] * osc * (escale ? escale[e0 + i / NVB] : T(1));
  }
  for (int i = threadIdx.x; i < ne * GEO; i += blockDim.x) sgeo[i] = d.geo[e0 * GEO + i];
  __syncthreads();
  const int el1 = threadIdx.x / NQ, q1 = threadIdx.x - (threadIdx.x / NQ) * NQ;
  if (threadIdx.x < ne * NQ) {
    const T* ge = sgeo + el1 * GEO;
    const T isd = ge[O::ISD];
    S U[NV], Ub[NV];
    T fb[D][NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) {
      T a = 0, b = 0;
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        a += sBv[q1 * NB + j] * su[el1 * NVB + c * NB + j];
        if constexpr (HESS) b += sBv[q1 * NB + j] * sv[el1 * NVB + c * NB + j];
      }
      if constexpr (HESS) U[c] = S{a * isd, b};  // the sqrt(det) factors of trace and test cancel
      else U[c] = a * isd;
      Ub[c] = Lift<S, T>::of(T(0));
      // adjoint of the flux along the Cartesian axes: the transposed test, mapped by A^-1
      T t[D];
#pragma unroll
      for (int dd = 0; dd < D; ++dd) {
        T h = 0;
#pragma unroll
        for (int i = 0; i < NB; ++i) h += sDv[(dd * NQ + q1) * NB + i] * sw[el1 * NVB + c * NB + i];
        t[dd] = h;
      }
#pragma unroll
      for (int k = 0; k < D; ++k) {
        T h = ge[k] * t[0];
#pragma unroll
        for (int dd = 1; dd < D; ++dd) h += ge[dd * D + k] * t[dd];
        fb[k][c] = h;
      }
    }
    euler_flux_vjp<D, S, T>(U, d.fs.gamma, fb, Ub);
#pragma unroll
    for (int c = 0; c < NV; ++c) {
      T o;
      if constexpr (HESS) {
        o = Ub[c].d * isd;
      } else {
        o = Ub[c];
        if (d.rot) {  // rotating frame: the flux is F - U v_r^T
          const T* vr = d.vrq + ((e0 + el1) * NQ + q1) * D;
#pragma unroll
          for (int k = 0; k < D; ++k) o -= fb[k][c] * vr[k];
        }
      }
      sU[(el1 * NQ + q1) * NV + c] = o;
    }
  }
  __syncthreads();
  const T* Bf = SM ? sBf : d.Bf;
  for (int it = threadIdx.x; it < ne * NVB; it += blockDim.x) {
    const int el = it / NVB, r = it - el * NVB;
    const int c = r / NB, j = r - c * NB;
    T acc = 0;
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc += sBv[q * NB + j] * sU[(el * NQ + q) * NV + c];
    acc += gather_faces_T<T, D, P, SM>(d, Bf, GT, e0 + el, c, j);
    if constexpr (!HESS) {
      if (d.rot && c >= 1 && c <= D) {  // transpose of the source -omega x: +omega x w~ (antisymmetric)
        T m[D];
#pragma unroll
        for (int k = 0; k < D; ++k) m[k] = sw[el * NVB + (1 + k) * NB + j];
        acc -= rot_source<T, D>(d.om, m, c - 1);
      }
    }
    out[e0 * NVB + it] = acc;
  }
}

template <class T, int D, int P>
cudaError_t jvp_state_adjoint_p(const DGData<T>& d, const T* u, const T* v, const T* w, T* out, T* GT,
                                const T* escale, T osc, cudaStream_t st, const ThetaSums<T>& th) {
  using O = Ord<D, P>;
  const int64_t nf = d.F * O::NFQ;
  if (nf > 0) face_hess_kernel<T, D, P><<<(unsigned)((nf + 127) / 128), 128, 0, st>>>(d, u, v, w, GT, escale, osc, th);
  const int64_t eb = (d.E + O::ET - 1) / O::ET;
  elem_hess_kernel<T, D, P, true><<<(unsigned)eb, 256, 0, st>>>(d, u, v, w, GT, out, escale, osc);
  return cudaGetLastError();
}

// ------------------------------------------- J(u)^T w for a single product
// Reverse sweeps of the fluxes at u with the transposed lift and test of w as adjoints: no point
// Jacobians are formed (building them for one product took 72% of pcexp_vjp).  Scratch layout of
// the adjoint kernels.  Vortex, 20,402 triangles at p = 3, FP64: a call takes 334 us against 842
// with the Jacobians (503 + 117 us of building them).
template <class T, int D, int P>
__global__ void __launch_bounds__(128) face_vjp_kernel(DGData<T> d, const T* __restrict__ u, const T* __restrict__ w,
                                                       T* __restrict__ GT) {
  using O = Ord<D, P>;
  constexpr int NB = O::NB, NFQ = O::NFQ, NV = O::NV, NPERM = O::NPERM, GEO = O::GEO;
  const int64_t n = d.F * NFQ;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n) return;
  const int64_t f = idx / NFQ;
  const int q = (int)(idx - f * NFQ);
  const int eL = d.fel[2 * f], eR = d.fel[2 * f + 1];
  const int loc = d.floc[f];
  const int fL = loc & 0xff, fR = (loc >> 8) & 0xff, pR = loc >> 16;
  T nr[D];
#pragma unroll
  for (int k = 0; k < D; ++k) nr[k] = d.fgeo[4 * f + k];
  const T wq = d.fgeo[4 * f + D] * d.Wf[q];
  const T vrn = d.rot ? d.vrn[idx] : T(0);
  const T isdL = d.geo[GEO * (int64_t)eL + O::ISD];
  T isdR = T(0), L[NV], R[NV], gb[NV];
  const T* bL = d.Bf + ((fL * NPERM) * NFQ + q) * NB;
  point_trace<T, D, P>(bL, u + (int64_t)eL * NV * NB, isdL, L);
  point_trace<T, D, P>(bL, w + (int64_t)eL * NV * NB, -isdL, gb);
  if (eR >= 0) {
    isdR = d.geo[GEO * (int64_t)eR + O::ISD];
    const T* bR = d.Bf + ((fR * NPERM + pR) * NFQ + q) * NB;
    T g[NV];
    point_trace<T, D, P>(bR, u + (int64_t)eR * NV * NB, isdR, R);
    point_trace<T, D, P>(bR, w + (int64_t)eR * NV * NB, isdR, g);
#pragma unroll
    for (int c = 0; c < NV; ++c) gb[c] += g[c];
  } else if (mirror_bc(eR)) {
    ghost_slip_wall<D, T, T>(L, nr, R, vrn);
  } else {
    ghost_farfield<D, T, T>(L, nr, d.fs, R);
  }
  T Lb[NV], Rb[NV];
#pragma unroll
  for (int c = 0; c < NV; ++c) Lb[c] = Rb[c] = T(0);
  face_flux_vjp<T, D>(d, eR, L, R, nr, vrn, gb, Lb, Rb);
  T* o = GT + idx * 2 * NV;
#pragma unroll
  for (int c = 0; c < NV; ++c) {
    o[c] = wq * isdL * Lb[c];
    o[NV + c] = eR >= 0 ? wq * isdR * Rb[c] : T(0);
  }
}

template <class T, int D, int P>
cudaError_t vjp_p(const DGData<T>& d, const T* u, const T* w, T* out, T* GT, cudaStream_t st) {
  using O = Ord<D, P>;
  const int64_t nf = d.F * O::NFQ;
  if (nf > 0) face_vjp_kernel<T, D, P><<<(unsigned)((nf + 127) / 128), 128, 0, st>>>(d, u, w, GT);
  const int64_t eb = (d.E + O::ET - 1) / O::ET;
  elem_hess_kernel<T, D, P, false><<<(unsigned)eb, 256, 0, st>>>(d, u, nullptr, w, GT, out, nullptr, T(1));
  return cudaGetLastError();
}

// ------------------------------------------- adjoint with respect to the free stream
// theta = (Mach number, flow angle in degrees) enters the operator only through the
// free-stream velocity of the far-field ghost state.  For the far-field faces (indices >= f0)
// this kernel adds to acc[0..1]
//   osc sum_q sum_v gbar_q[v] dF~_v/dtheta_k                       (osc (dR/dtheta)^T w)
// with gbar_q[v] = -|f| w_q / sqrt|det A_L| sum_i phi_i(x_q) w[e_L][v][i] (the transposed lift
// of w, the face term of R at the L element).  Jet numbers seeded on the velocity give the
// derivatives.  dvel = {dvel/dMach (D), dvel/dalpha (D)}.  Fixed-order sum: per-block partials,
// the last block adds them to acc.
template <class T, int D, int P>
__global__ void __launch_bounds__(128) param_adjoint_kernel(DGData<T> d, int64_t f0, const T* __restrict__ u,
                                                            const T* __restrict__ w, double osc, double dvm0,
                                                            double dvm1, double dva0, double dva1,
                                                            double* __restrict__ acc, double* __restrict__ partials,
                                                            unsigned* counter) {
  using O = Ord<D, P>;
  constexpr int NB = O::NB, NFQ = O::NFQ, NV = O::NV, NPERM = O::NPERM, GEO = O::GEO;
  __shared__ double red[2][4];
  __shared__ bool last;
  double a0 = 0.0, a1 = 0.0;
  const int64_t n = (d.F - f0) * NFQ;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t f = f0 + idx / NFQ;
    const int q = (int)(idx % NFQ);
    if (-d.fel[2 * f + 1] != PCEXP_BC_FARFIELD) continue;
    const int eL = d.fel[2 * f];
    const int fL = d.floc[f] & 0xff;
    T nr[D];
#pragma unroll
    for (int k = 0; k < D; ++k) nr[k] = d.fgeo[4 * f + k];
    const T isd = d.geo[GEO * (int64_t)eL + O::ISD];
    const T* be = d.Bf + ((fL * NPERM) * NFQ + q) * NB;
    const T wl = d.fgeo[4 * f + D] * d.Wf[q];
    T uL[NV], gb[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      T a = 0, c = 0;
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        const T bj = __ldg(be + j);
        const int64_t o = (int64_t)eL * NV * NB + v * NB + j;
        a += bj * u[o];
        c += bj * w[o];
      }
      uL[v] = a * isd;
      gb[v] = (T)(-osc) * wl * isd * c;
    }
    const double dm[3] = {dvm0, dvm1, 0.0}, da[3] = {dva0, dva1, 0.0};
    using J = Jet<T, 2>;
    J L[NV], R[NV], F[NV], vi[3];
#pragma unroll
    for (int v = 0; v < NV; ++v) L[v] = Lift<J, T>::of(uL[v]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      vi[k].v = d.fs.vel[k];
      vi[k].d[0] = (T)dm[k];
      vi[k].d[1] = (T)da[k];
    }
    ghost_farfield_v<D, J, T>(L, nr, d.fs.gamma, d.fs.rho, d.fs.p, vi, R);
    roe_flux<D, J, T>(L, R, nr, d.fs.gamma, F);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      a0 += (double)gb[v] * (double)F[v].d[0];
      a1 += (double)gb[v] * (double)F[v].d[1];
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    a0 += __shfl_xor_sync(0xffffffffu, a0, o);
    a1 += __shfl_xor_sync(0xffffffffu, a1, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = a0;
    red[1][threadIdx.x >> 5] = a1;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double b0 = 0, b1 = 0;
    for (int ww = 0; ww < (int)(blockDim.x >> 5); ++ww) {
      b0 += red[0][ww];
      b1 += red[1][ww];
    }
    partials[2 * blockIdx.x] = b0;
    partials[2 * blockIdx.x + 1] = b1;
    __threadfence();
    last = atomicAdd(counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (last && threadIdx.x == 0) {
    double b0 = 0, b1 = 0;
    for (unsigned i = 0; i < gridDim.x; ++i) {
      b0 += __ldcg(partials + 2 * i);
      b1 += __ldcg(partials + 2 * i + 1);
    }
    acc[0] += b0;
    acc[1] += b1;
    *counter = 0;
  }
}

template <class T, int D, int P>
cudaError_t param_adjoint_p(const DGData<T>& d, int64_t f0, const T* u, const T* w, double osc, const double* dvel,
                            double* acc, double* partials, unsigned* counter, cudaStream_t st) {
  const int64_t n = (d.F - f0) * Ord<D, P>::NFQ;
  if (n <= 0) return cudaSuccess;
  int64_t g = (n + 127) / 128;
  if (g > RED_BLOCKS) g = RED_BLOCKS;
  param_adjoint_kernel<T, D, P><<<(unsigned)g, 128, 0, st>>>(d, f0, u, w, osc, dvel[0], dvel[1], dvel[2], dvel[3], acc,
                                                             partials, counter);
  return cudaGetLastError();
}

// ------------------------------------------------------------ output functionals
// fixed-order sum of one double per thread into *value (last-block reduction)
PCEXP_DEV void block_sum_last(double acc, double* value, double* partials, unsigned* counter, bool sqrt_out) {
  __shared__ double red[8];
  __shared__ bool last;
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double b = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) b += red[w];
    partials[blockIdx.x] = b;
    __threadfence();
    last = atomicAdd(counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (last && threadIdx.x == 0) {
    double b = 0;
    for (unsigned i = 0; i < gridDim.x; ++i) b += __ldcg(partials + i);
    *value = sqrt_out ? sqrt(b) : b;
    *counter = 0;
  }
}

// Pressure force on the slip walls along the unit direction a:
//   J = sum_{wall faces} sum_q |f| w_q p(U_L(x_q)) (n . a),  p = (gamma-1)(E - |m|^2 / (2 rho)),
// with its gradient dJ/du (trace transpose of dp/dU); value by a fixed-order reduction.
template <class T, int D, int P>
__global__ void __launch_bounds__(256) wall_force_kernel(DGData<T> d, int64_t f0, const T* __restrict__ u, double ax,
                                                         double ay, double az, double* __restrict__ grad,
                                                         double* __restrict__ value, double* __restrict__ partials,
                                                         unsigned* counter) {
  using O = Ord<D, P>;
  constexpr int NB = O::NB, NFQ = O::NFQ, NV = O::NV, NPERM = O::NPERM, GEO = O::GEO;
  const double a3[3] = {ax, ay, az};
  double acc = 0;
  const T gm = d.fs.gamma - T(1);
  for (int64_t f = f0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; f < d.F; f += (int64_t)gridDim.x * blockDim.x) {
    if (-d.fel[2 * f + 1] != PCEXP_BC_SLIP_WALL) continue;
    const int e = d.fel[2 * f];
    const int fl = d.floc[f] & 0xff;
    double na = 0;
    for (int k = 0; k < D; ++k) na += (double)d.fgeo[4 * f + k] * a3[k];
    const double meas = (double)d.fgeo[4 * f + D];
    const double isd = (double)d.geo[GEO * (int64_t)e + O::ISD];
    double g[NV * NB];
    for (int k = 0; k < NV * NB; ++k) g[k] = 0.0;
    for (int q = 0; q < NFQ; ++q) {
      const T* b = d.Bf + ((fl * NPERM) * NFQ + q) * NB;
      double U[NV];
      for (int c = 0; c < NV; ++c) {
        double a = 0;
        for (int j = 0; j < NB; ++j) a += (double)b[j] * (double)u[(int64_t)e * NV * NB + c * NB + j];
        U[c] = a * isd;
      }
      double vel[D], v2 = 0;
      for (int k = 0; k < D; ++k) {
        vel[k] = U[1 + k] / U[0];
        v2 += vel[k] * vel[k];
      }
      const double p = (double)gm * (U[NV - 1] - 0.5 * U[0] * v2);
      const double wq = meas * (double)d.Wf[q] * na;
      acc += wq * p;
      double dp[NV];
      dp[0] = (double)gm * 0.5 * v2;
      for (int k = 0; k < D; ++k) dp[1 + k] = -(double)gm * vel[k];
      dp[NV - 1] = (double)gm;
      for (int c = 0; c < NV; ++c)
        for (int j = 0; j < NB; ++j) g[c * NB + j] += wq * dp[c] * (double)b[j] * isd;
    }
    // on the 2D walls at most two wall faces meet in one element, and a + b is the same
    // in either order; elements with three or more wall faces sum in arrival order
    if (grad)
      for (int k = 0; k < NV * NB; ++k) atomicAdd(grad + (int64_t)e * NV * NB + k, g[k]);
  }
  block_sum_last(acc, value, partials, counter, false);
}

// Vortex-error functional J = ||U_h - U_exact||_L2 (all conservative variables) with the
// exact state of the translated isentropic vortex at the volume points, and the
// unnormalised gradient sum_q w_q (U_h - U_ex)_v dU_h/du_{e,v,j} (scaled by 1/J afterwards).
// prm: eps, x_c, y_c, period (<= 0: none), t.  The field lies in the x-y plane.
template <class T, int D, int P>
__global__ void __launch_bounds__(256) vortex_error_kernel(DGData<T> d, const T* __restrict__ u,
                                                           const double* __restrict__ xq, double eps, double xc,
                                                           double yc, double period, double t,
                                                           double* __restrict__ grad, double* __restrict__ value,
                                                           double* __restrict__ partials, unsigned* counter) {
  using O = Ord<D, P>;
  constexpr int NB = O::NB, NQ = O::NQ, NV = O::NV, GEO = O::GEO;
  double acc = 0;
  const double g = (double)d.fs.gamma, rinf = (double)d.fs.rho, pinf = (double)d.fs.p;
  const double u0 = (double)d.fs.vel[0], v0 = (double)d.fs.vel[1];
  const double Tinf = pinf / rinf, pi = 3.141592653589793238462643383279502884;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < d.E; e += (int64_t)gridDim.x * blockDim.x) {
    const double sd = (double)d.geo[GEO * e + O::SD];
    double ge[NV * NB];
    for (int k = 0; k < NV * NB; ++k) ge[k] = 0.0;
    for (int q = 0; q < NQ; ++q) {
      double dx = xq[(e * NQ + q) * D] - (xc + u0 * t), dy = xq[(e * NQ + q) * D + 1] - (yc + v0 * t);
      if (period > 0) {
        dx -= period * nearbyint(dx / period);
        dy -= period * nearbyint(dy / period);
      }
      const double r2 = dx * dx + dy * dy;
      const double fe = eps / (2 * pi) * exp(0.5 * (1 - r2));
      const double uu = u0 - fe * dy, vv = v0 + fe * dx;
      const double Tv = Tinf - (g - 1) * eps * eps / (8 * g * pi * pi) * exp(1 - r2);
      const double rho = rinf * pow(Tv / Tinf, 1.0 / (g - 1));
      const double p = rho * Tv;
      double Ue[NV];
      Ue[0] = rho;
      Ue[1] = rho * uu;
      Ue[2] = rho * vv;
      if (D == 3) Ue[3] = 0.0;
      Ue[NV - 1] = p / (g - 1) + 0.5 * rho * (uu * uu + vv * vv);
      const double wq = (double)d.Wv[q] * sd * sd;  // |det A| w^_q
      for (int c = 0; c < NV; ++c) {
        double a = 0;
        for (int j = 0; j < NB; ++j) a += (double)d.Bv[q * NB + j] * (double)u[e * NV * NB + c * NB + j];
        const double diff = a / sd - Ue[c];
        acc += wq * diff * diff;
        for (int j = 0; j < NB; ++j) ge[c * NB + j] += wq * diff * (double)d.Bv[q * NB + j] / sd;
      }
    }
    if (grad)
      for (int k = 0; k < NV * NB; ++k) grad[e * NV * NB + k] = ge[k];
  }
  block_sum_last(acc, value, partials, counter, true);
}

// Partials of the vortex-error functional with respect to theta = (Mach, alpha in degrees,
// eps) at a fixed state: out[0] = sum w_q |U_h - U_ex|^2 (= J^2), out[1 + k] = sum w_q
// (U_h - U_ex) . dU_ex/dtheta_k, so dJ/dtheta_k = -out[1 + k] / J.  The exact state is
// evaluated on Jet numbers seeded with the free-stream velocity derivatives (dvel: d/dMach
// x, y, then d/dalpha x, y) and with eps.  Fixed-order last-block sums.
template <class T, int D, int P>
__global__ void __launch_bounds__(256) vortex_param_grad_kernel(DGData<T> d, const T* __restrict__ u,
                                                                const double* __restrict__ xq, double eps, double xc,
                                                                double yc, double period, double t, double dvm0,
                                                                double dvm1, double dva0, double dva1,
                                                                double* __restrict__ out, double* __restrict__ partials,
                                                                unsigned* counter) {
  using O = Ord<D, P>;
  constexpr int NB = O::NB, NQ = O::NQ, NV = O::NV, GEO = O::GEO;
  using J = Jet<double, 3>;
  __shared__ double red[4][8];
  __shared__ bool last;
  double acc[4] = {0, 0, 0, 0};
  const double g = (double)d.fs.gamma, rinf = (double)d.fs.rho, pinf = (double)d.fs.p;
  const double Tinf = pinf / rinf, pi = 3.141592653589793238462643383279502884;
  J u0, v0, ep;
  u0.v = (double)d.fs.vel[0];
  u0.d[0] = dvm0;
  u0.d[1] = dva0;
  u0.d[2] = 0.0;
  v0.v = (double)d.fs.vel[1];
  v0.d[0] = dvm1;
  v0.d[1] = dva1;
  v0.d[2] = 0.0;
  ep.v = eps;
  ep.d[0] = ep.d[1] = 0.0;
  ep.d[2] = 1.0;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < d.E; e += (int64_t)gridDim.x * blockDim.x) {
    const double sd = (double)d.geo[GEO * e + O::SD];
    for (int q = 0; q < NQ; ++q) {
      J dx = (xq[(e * NQ + q) * D] - xc) - u0 * t;
      J dy = (xq[(e * NQ + q) * D + 1] - yc) - v0 * t;
      if (period > 0) {
        dx = dx - period * nearbyint(dx.v / period);
        dy = dy - period * nearbyint(dy.v / period);
      }
      const J r2 = dx * dx + dy * dy;
      const J fe = ep * (1.0 / (2 * pi)) * exp_s(0.5 * (1.0 - r2));
      const J uu = u0 - fe * dy, vv = v0 + fe * dx;
      const J Tv = Tinf - ((g - 1) / (8 * g * pi * pi)) * (ep * ep) * exp_s(1.0 - r2);
      const J rho = rinf * pow_s(Tv * (1.0 / Tinf), 1.0 / (g - 1));
      const J p = rho * Tv;
      J Ue[NV];
      Ue[0] = rho;
      Ue[1] = rho * uu;
      Ue[2] = rho * vv;
      if (D == 3) Ue[3] = Lift<J, double>::of(0.0);
      Ue[NV - 1] = p * (1.0 / (g - 1)) + 0.5 * rho * (uu * uu + vv * vv);
      const double wq = (double)d.Wv[q] * sd * sd;
      for (int c = 0; c < NV; ++c) {
        double a = 0;
        for (int j = 0; j < NB; ++j) a += (double)d.Bv[q * NB + j] * (double)u[e * NV * NB + c * NB + j];
        const double diff = a / sd - Ue[c].v;
        acc[0] += wq * diff * diff;
        for (int k = 0; k < 3; ++k) acc[1 + k] += wq * diff * Ue[c].d[k];
      }
    }
  }
  for (int k = 0; k < 4; ++k) {
    for (int o = 16; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
    if ((threadIdx.x & 31) == 0) red[k][threadIdx.x >> 5] = acc[k];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 0; k < 4; ++k) {
      double b = 0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) b += red[k][w];
      partials[4 * blockIdx.x + k] = b;
    }
    __threadfence();
    last = atomicAdd(counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (last && threadIdx.x == 0) {
    for (int k = 0; k < 4; ++k) {
      double b = 0;
      for (unsigned i = 0; i < gridDim.x; ++i) b += __ldcg(partials + 4 * i + k);
      out[k] = b;
    }
    *counter = 0;
  }
}

template <class T, int D, int P>
cudaError_t vortex_param_grad_p(const DGData<T>& d, const T* u, const double* xq, const double* prm, const double* dvel,
                                double* out, double* partials, unsigned* counter, cudaStream_t st) {
  int64_t nb = (d.E + 255) / 256;
  if (nb > RED_BLOCKS / 2) nb = RED_BLOCKS / 2;
  vortex_param_grad_kernel<T, D, P><<<(unsigned)(nb < 1 ? 1 : nb), 256, 0, st>>>(
      d, u, xq, prm[0], prm[1], prm[2], prm[3], prm[4], dvel[0], dvel[1], dvel[2], dvel[3], out, partials, counter);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ time step
// dt_e = CFL h_e / ((2p+1)(|v| + c)) with v, c at the element centroid (Eq. x3d).
template <class T, int D, int P>
__global__ void __launch_bounds__(256) local_dt_kernel(DGData<T> d, const T* __restrict__ u,
                                                       const double* cfl_dev, double cfl_host,
                                                       T* __restrict__ dte, double* __restrict__ dtmin,
                                                       double* __restrict__ partials,
                                                       unsigned* __restrict__ counter) {
  using O = Ord<D, P>;
  constexpr int NB = O::NB, NV = O::NV, GEO = O::GEO;
  __shared__ double red[8];
  __shared__ bool last;
  const double cfl = cfl_dev ? *cfl_dev : cfl_host;
  double mn = DBL_MAX;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < d.E_loc; e += (int64_t)gridDim.x * blockDim.x) {
    const T isd = d.geo[GEO * e + O::ISD];
    double U[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      T a = 0, c[NB];
      load_coeffs<T, NB>(u + (e * NV + v) * NB, c);
#pragma unroll
      for (int j = 0; j < NB; ++j) a += d.Bc[j] * c[j];
      U[v] = (double)(a * isd);
    }
    const double gam = (double)d.fs.gamma;
    double v2 = 0;
    for (int k = 0; k < D; ++k) v2 += (U[1 + k] / U[0]) * (U[1 + k] / U[0]);
    const double p = (gam - 1.0) * (U[NV - 1] - 0.5 * U[0] * v2);
    const double c = sqrt(gam * p / U[0]);
    if (d.rot) {  // the velocity relative to the rotating frame carries the waves
      v2 = 0;
      for (int k = 0; k < D; ++k) {
        const double vk = U[1 + k] / U[0] - (double)d.vrc[e * D + k];
        v2 += vk * vk;
      }
    }
    const double h = (double)d.geo[GEO * e + O::HE];
    const double dt = cfl * h / ((2 * d.p + 1) * (sqrt(v2) + c));
    if (dte) dte[e] = (T)dt;
    mn = fmin(mn, dt);
  }
  if (grid_reduce<MinOf>(mn, red, last, partials, counter)) *dtmin = mn;
}

// ------------------------------------------------------------------ launchers
// The launchers below dispatch on p for one dimension D; orders above PMAX<D> are
// rejected when a context is created.
template <int D> constexpr int PMAX = D == 2 ? 3 : 2;

#define PCEXP_PSWITCH(D, CALL)                       \
  switch (d.p) {                                     \
    case 0: { constexpr int P_ = 0; return CALL; }   \
    case 1: { constexpr int P_ = 1; return CALL; }   \
    case 2: { constexpr int P_ = 2; return CALL; }   \
    case 3: {                                        \
      if constexpr (PMAX<D> >= 3) {                  \
        constexpr int P_ = PMAX<D> >= 3 ? 3 : 0;     \
        return CALL;                                 \
      }                                              \
      break;                                         \
    }                                                \
  }                                                  \
  return cudaErrorInvalidValue;

template <class T, int D>
cudaError_t launch_dg_operator_d(const DGData<T>& d, const T* u, const T* du, T* out, T* G, const T* escale,
                                 const int* skip, cudaStream_t st, const cudaEvent_t* ev, const double* oscale,
                                 bool tight) {
  PCEXP_PSWITCH(D, (dg_op_p<T, D, P_>(d, u, du, out, G, escale, skip, oscale, st, ev, tight)))
}
template <class T, int D>
cudaError_t launch_linearize_d(const DGData<T>& d, const T* u, LinData<T> lin, cudaStream_t st) {
  PCEXP_PSWITCH(D, (linearize_p<T, D, P_>(d, u, lin, st)))
}
template <class T, int D>
cudaError_t launch_jac_apply_d(const DGData<T>& d, LinData<T> lin, const T* dv, T* out, T* G, const T* escale,
                               const int* skip, const double* oscale, cudaStream_t st, const cudaEvent_t* ev) {
  PCEXP_PSWITCH(D, (jac_apply_p<T, D, P_>(d, lin, dv, out, G, escale, skip, oscale, st, ev)))
}
template <class T, int D>
cudaError_t upload_tables_d(const DGData<T>& d, const double* Bv, const double* Dv, const double* Wv, const double* Bf,
                            cudaStream_t st) {
  PCEXP_PSWITCH(D, (upload_tables_p<T, D, P_>(Bv, Dv, Wv, Bf, st)))
}
template <class T, int D>
int64_t face_flux_size_d(const DGData<T>& d) {
  const int nv = D + 2;
  switch (d.p) {
    case 0: return d.F * nv * GSTRIDE<T, D, 0>;
    case 1: return d.F * nv * GSTRIDE<T, D, 1>;
    case 2: return d.F * nv * GSTRIDE<T, D, 2>;
    default: return d.F * nv * GSTRIDE<T, D, (PMAX<D> >= 3 ? 3 : 2)>;
  }
}
template <class T, int D>
cudaError_t launch_jac_adjoint_d(const DGData<T>& d, LinData<T> lin, const T* w, T* out, T* GT, const T* escale,
                                 T osc, cudaStream_t st) {
  PCEXP_PSWITCH(D, (jac_adjoint_p<T, D, P_>(d, lin, w, out, GT, escale, osc, st)))
}
template <class T, int D>
cudaError_t launch_jvp_state_adjoint_d(const DGData<T>& d, const T* u, const T* v, const T* w, T* out, T* GT,
                                       const T* escale, T osc, cudaStream_t st, const ThetaSums<T>& th) {
  PCEXP_PSWITCH(D, (jvp_state_adjoint_p<T, D, P_>(d, u, v, w, out, GT, escale, osc, st, th)))
}

template <class T, int D>
cudaError_t launch_vjp_d(const DGData<T>& d, const T* u, const T* w, T* out, T* GT, cudaStream_t st) {
  PCEXP_PSWITCH(D, (vjp_p<T, D, P_>(d, u, w, out, GT, st)))
}

template <class T, int D>
cudaError_t launch_param_adjoint_d(const DGData<T>& d, int64_t f0, const T* u, const T* w, double osc,
                                   const double* dvel, double* acc, double* partials, unsigned* counter,
                                   cudaStream_t st) {
  PCEXP_PSWITCH(D, (param_adjoint_p<T, D, P_>(d, f0, u, w, osc, dvel, acc, partials, counter, st)))
}

template <class T, int D, int P>
cudaError_t wall_force_p(const DGData<T>& d, int64_t f0, const T* u, double ax, double ay, double az, double* grad,
                         double* value, double* partials, unsigned* counter, cudaStream_t st) {
  const int64_t nb = d.F - f0;
  unsigned g = (unsigned)((nb + 255) / 256);
  if (g < 1) g = 1;
  if (g > RED_BLOCKS) g = RED_BLOCKS;
  wall_force_kernel<T, D, P><<<g, 256, 0, st>>>(d, f0, u, ax, ay, az, grad, value, partials, counter);
  return cudaGetLastError();
}
template <class T, int D>
cudaError_t launch_wall_force_d(const DGData<T>& d, int64_t f0, const T* u, double ax, double ay, double az,
                                double* grad, double* value, double* partials, unsigned* counter, cudaStream_t st) {
  PCEXP_PSWITCH(D, (wall_force_p<T, D, P_>(d, f0, u, ax, ay, az, grad, value, partials, counter, st)))
}

template <class T, int D, int P>
cudaError_t vortex_error_p(const DGData<T>& d, const T* u, const double* xq, const double* prm, double* grad,
                           double* value, double* partials, unsigned* counter, cudaStream_t st) {
  int64_t nb = (d.E + 255) / 256;
  if (nb > RED_BLOCKS) nb = RED_BLOCKS;
  vortex_error_kernel<T, D, P><<<(unsigned)(nb < 1 ? 1 : nb), 256, 0, st>>>(
      d, u, xq, prm[0], prm[1], prm[2], prm[3], prm[4], grad, value, partials, counter);
  return cudaGetLastError();
}
template <class T, int D>
cudaError_t launch_vortex_error_d(const DGData<T>& d, const T* u, const double* xq, const double* prm, double* grad,
                                  double* value, double* partials, unsigned* counter, cudaStream_t st) {
  PCEXP_PSWITCH(D, (vortex_error_p<T, D, P_>(d, u, xq, prm, grad, value, partials, counter, st)))
}

template <class T, int D>
cudaError_t launch_vortex_param_grad_d(const DGData<T>& d, const T* u, const double* xq, const double* prm,
                                       const double* dvel, double* out, double* partials, unsigned* counter,
                                       cudaStream_t st) {
  PCEXP_PSWITCH(D, (vortex_param_grad_p<T, D, P_>(d, u, xq, prm, dvel, out, partials, counter, st)))
}

template <class T, int D, int P>
cudaError_t local_dt_p(const DGData<T>& d, const T* u, const double* cfl_dev, double cfl, T* dte, double* dtmin,
                       double* partials, unsigned* counter, cudaStream_t st) {
  int64_t nb = (d.E + 255) / 256;
  if (nb > RED_BLOCKS) nb = RED_BLOCKS;
  local_dt_kernel<T, D, P><<<(unsigned)nb, 256, 0, st>>>(d, u, cfl_dev, cfl, dte, dtmin, partials, counter);
  return cudaGetLastError();
}
template <class T, int D>
cudaError_t launch_local_dt_d(const DGData<T>& d, const T* u, const double* cfl_dev, double cfl, T* dte,
                              double* dtmin, double* partials, unsigned* counter, cudaStream_t st) {
  PCEXP_PSWITCH(D, (local_dt_p<T, D, P_>(d, u, cfl_dev, cfl, dte, dtmin, partials, counter, st)))
}

#undef PCEXP_PSWITCH

#define PCEXP_INST_D(T, D)                                                                                         \
  template cudaError_t launch_dg_operator_d<T, D>(const DGData<T>&, const T*, const T*, T*, T*, const T*,           \
                                                  const int*, cudaStream_t, const cudaEvent_t*, const double*,     \
                                                  bool);                                                           \
  template cudaError_t launch_linearize_d<T, D>(const DGData<T>&, const T*, LinData<T>, cudaStream_t);             \
  template cudaError_t launch_jac_apply_d<T, D>(const DGData<T>&, LinData<T>, const T*, T*, T*, const T*,          \
                                                const int*, const double*, cudaStream_t, const cudaEvent_t*);      \
  template cudaError_t upload_tables_d<T, D>(const DGData<T>&, const double*, const double*, const double*,        \
                                             const double*, cudaStream_t);                                         \
  template int64_t face_flux_size_d<T, D>(const DGData<T>&);                                                       \
  template cudaError_t launch_jvp_state_adjoint_d<T, D>(const DGData<T>&, const T*, const T*, const T*, T*, T*,    \
                                                        const T*, T, cudaStream_t, const ThetaSums<T>&);           \
  template cudaError_t launch_vjp_d<T, D>(const DGData<T>&, const T*, const T*, T*, T*, cudaStream_t);             \
  template cudaError_t launch_wall_force_d<T, D>(const DGData<T>&, int64_t, const T*, double, double, double,      \
                                                 double*, double*, double*, unsigned*, cudaStream_t);              \
  template cudaError_t launch_vortex_error_d<T, D>(const DGData<T>&, const T*, const double*, const double*,       \
                                                   double*, double*, double*, unsigned*, cudaStream_t);            \
  template cudaError_t launch_local_dt_d<T, D>(const DGData<T>&, const T*, const double*, double, T*, double*,     \
                                               double*, unsigned*, cudaStream_t);                                  \
  template cudaError_t launch_vortex_param_grad_d<T, D>(const DGData<T>&, const T*, const double*, const double*,   \
                                                        const double*, double*, double*, unsigned*, cudaStream_t); \
  template cudaError_t launch_param_adjoint_d<T, D>(const DGData<T>&, int64_t, const T*, const T*, double,         \
                                                    const double*, double*, double*, unsigned*, cudaStream_t);

// (the stored-block forms of double precision alone)
#define PCEXP_INST_FP64(D)                                                                                         \
  template cudaError_t launch_jac_adjoint_d<double, D>(const DGData<double>&, LinData<double>, const double*,      \
                                                       double*, double*, const double*, double, cudaStream_t);

}  // namespace pcexp
