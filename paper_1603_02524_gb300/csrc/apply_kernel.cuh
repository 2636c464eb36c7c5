// Sum-factorised DG operator apply (shared by the FP64 / fp32 library
// kernels and the double-float outer apply).
//
// Paper: Stiller, arXiv 1603.02524, Sec. 2.4 (1-D blocks of Eq. L:generic) and
// the tensor form of the discrete problem (Sec. 2.2, reading C1 in 3-D).
#pragma once

#include <type_traits>

#include "pmg_internal.h"

namespace pmg {

// table / vector loads through the read-only path (dfloat: one 8-byte load)
template <typename T>
__device__ __forceinline__ T ldg(const T* p) { return __ldg(p); }

// c + a * b, fused (dfloat: the accumulate form of dfloat.cuh)
__device__ __forceinline__ double madd(double a, double b, double c) { return ::fma(a, b, c); }
__device__ __forceinline__ float madd(float a, float b, float c) { return fmaf(a, b, c); }

// 16-byte vector of T read through the read-only path (dfloat: two values per vector)
template <typename T> struct AVec;
template <> struct AVec<float> {
  using V = float4;
  static constexpr int W = 4;
  __device__ static float get(const float4& v, int k) { return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w; }
};
template <> struct AVec<double> {
  using V = double2;
  static constexpr int W = 2;
  __device__ static double get(const double2& v, int k) { return k == 0 ? v.x : v.y; }
};
template <> struct AVec<dfloat> {
  using V = float4;
  static constexpr int W = 2;
  __device__ static dfloat get(const float4& v, int k) { return k == 0 ? dfloat(v.x, v.y) : dfloat(v.z, v.w); }
};
template <typename T>
__host__ __device__ constexpr int apad(int n) { return (n + AVec<T>::W - 1) / AVec<T>::W * AVec<T>::W; }

// acc[0..N) += row[0..N) * x, row a 16-byte aligned, padded row of a global table
template <typename T, int N>
__device__ __forceinline__ void apply_axpy(T (&acc)[N], const T* row, T x) {
  using A = AVec<T>;
  const typename A::V* r = reinterpret_cast<const typename A::V*>(row);
#pragma unroll
  for (int c = 0; c < apad<T>(N) / A::W; ++c) {
    const typename A::V w = __ldg(r + c);
#pragma unroll
    for (int k = 0; k < A::W; ++k)
      if (c * A::W + k < N) acc[c * A::W + k] = madd(A::get(w, k), x, acc[c * A::W + k]);
  }
}

// ---------------------------------------------------------------------------
// Transfers between orders (Sec. 3.2): J (NF x NC, J[a][o] = coarse basis function
// o at fine GLL node a) is centro-symmetric, J[NF-1-a][NC-1-o] = J[a][o], because
// both node sets are symmetric about the element centre.  Along one axis the
// restriction y = J^T x and the prolongation y = J x then split into an even part
// on the sums x[i] + x[n-1-i] and an odd part on the differences (the middle node,
// where there is one, enters the even part alone):
//   e[a][o] = (J[a][o] + J[a][NC-1-o]) / 2   (a <= middle, o <= middle)
//   d[a][o] = (J[a][o] - J[a][NC-1-o]) / 2   (a, o below the middle)
// about half the multiply-adds of the dense contraction.  The folded coefficients
// are kernel parameters: the contractions below index them with compile-time
// indices only, so they are read as constant operands, with no load instruction.
// ---------------------------------------------------------------------------
template <typename T, int NF, int NC>
struct FoldedJ {
  static constexpr int HF = NF / 2, HC = NC / 2, EF = NF - HF, EC = NC - HC;
  T e[EF * EC];
  T d[(HF * HC) > 0 ? HF * HC : 1];
};
template <typename T, int NF>
struct FoldedJ<T, NF, 0> {};

// host: the folded coefficients of J (row-major NF x NC, FP64), rounded to T
template <typename T, int NF, int NC>
FoldedJ<T, NF, NC> fold_interpolation(const double* J) {
  using F = FoldedJ<T, NF, NC>;
  F f{};
  for (int a = 0; a < F::EF; ++a)
    for (int o = 0; o < F::EC; ++o) f.e[a * F::EC + o] = T(0.5 * (J[a * NC + o] + J[a * NC + (NC - 1 - o)]));
  for (int a = 0; a < F::HF; ++a)
    for (int o = 0; o < F::HC; ++o) f.d[a * F::HC + o] = T(0.5 * (J[a * NC + o] - J[a * NC + (NC - 1 - o)]));
  return f;
}

// y[0..NC) = J^T x[0..NF) along one axis; each output is handed to put(index, value)
// as soon as it is formed (an output pair at a time), so no output array is held
template <typename T, int NF, int NC, typename Put>
__device__ __forceinline__ void fold_restrict(const FoldedJ<T, NF, NC>& J, const T (&x)[NF], Put&& put) {
  using F = FoldedJ<T, NF, NC>;
  T sp[F::EF], sm[F::HF > 0 ? F::HF : 1];
#pragma unroll
  for (int a = 0; a < F::HF; ++a) {
    sp[a] = x[a] + x[NF - 1 - a];
    sm[a] = x[a] - x[NF - 1 - a];
  }
  if constexpr (F::EF > F::HF) sp[F::HF] = x[F::HF];
#pragma unroll
  for (int o = 0; o < F::EC; ++o) {
    T ev = T(0);
#pragma unroll
    for (int a = 0; a < F::EF; ++a) ev = madd(J.e[a * F::EC + o], sp[a], ev);
    if (o < F::HC) {
      T od = T(0);
#pragma unroll
      for (int a = 0; a < F::HF; ++a) od = madd(J.d[a * F::HC + o], sm[a], od);
      put(o, ev + od);
      put(NC - 1 - o, ev - od);
    } else {
      put(o, ev);
    }
  }
}

// y[0..NF) = J x[0..NC) along one axis, outputs handed to put(index, value)
template <typename T, int NF, int NC, typename Put>
__device__ __forceinline__ void fold_prolong(const FoldedJ<T, NF, NC>& J, const T (&x)[NC], Put&& put) {
  using F = FoldedJ<T, NF, NC>;
  T sp[F::EC], sm[F::HC > 0 ? F::HC : 1];
#pragma unroll
  for (int o = 0; o < F::HC; ++o) {
    sp[o] = x[o] + x[NC - 1 - o];
    sm[o] = x[o] - x[NC - 1 - o];
  }
  if constexpr (F::EC > F::HC) sp[F::HC] = x[F::HC];
#pragma unroll
  for (int a = 0; a < F::EF; ++a) {
    T ev = T(0);
#pragma unroll
    for (int o = 0; o < F::EC; ++o) ev = madd(J.e[a * F::EC + o], sp[o], ev);
    if (a < F::HF) {
      T od = T(0);
#pragma unroll
      for (int o = 0; o < F::HC; ++o) od = madd(J.d[a * F::HC + o], sm[o], od);
      put(a, ev + od);
      put(NF - 1 - a, ev - od);
    } else {
      put(a, ev);
    }
  }
}

// Allow `bytes` of dynamic shared memory for kernel `fn` (once per kernel).
template <typename K>
static bool set_smem(K fn, size_t bytes) {
  if (bytes <= 48 * 1024) return true;
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) ==
         cudaSuccess;
}

// ---------------------------------------------------------------------------
// Operator apply: v = A u or v = f - A u  (Eq. discrete problem, 3-D tensor form)
//
// One thread owns one nodal line of one element per axis pass.  The element is
// staged in shared memory; the line is contracted with the element's dense
// 1-D block L^0 (Eq. L:generic); the neighbour blocks L^-/L^+ have rank <= 3
// and need only the neighbour line's end value and end derivative
// (sum_k D_{P,k} u_k^{m-1}, sum_k D_{0,k} u_k^{m+1}).  The axes accumulate in
// shared memory; the last one multiplies by the masses and writes v from registers.
//
// What bounds it (fp32, 3-D): the load unit (72 % busy at P = 8) and the latency of the
// neighbour reads, which used to precede each axis pass (long-scoreboard stalls 13.6 of 21
// cycles per instruction, load unit 53 %).  Now the ends of all axes are read at the start,
// the x neighbours through shared memory (apply_staged), and the last pass needs no sweep of
// its own.  fp32 residuals: P = 8 at 8192 elements 76 -> 54 us, P = 16 at 4096 elements
// 240 -> 200, its fused restriction 257 -> 213, P = 2 at 8192 12.2 -> 9.3; FP64 2-D solves
// 16 x 16 P = 8 2.62 -> 2.47 ms.
// ---------------------------------------------------------------------------
// The tables of axis d, selected with compile-time indices (a runtime index into
// the kernel-parameter arrays would copy them to local memory).
template <typename T>
struct ApplyAxis {
  const T* L0;
  const int* sym;
  const T* cpl;
  int m;              // element index along the axis
  int ned;            // elements along the axis
  long long estride;  // element stride of the axis
};
template <typename T>
__device__ __forceinline__ ApplyAxis<T> apply_axis(const LevelDims& dm, const ApplyTables<T>& at,
                                                   const int (&me)[3], int d) {
  ApplyAxis<T> a;
  a.L0 = d == 0 ? at.L0[0] : (d == 1 ? at.L0[1] : at.L0[2]);
  a.sym = d == 0 ? at.sym[0] : (d == 1 ? at.sym[1] : at.sym[2]);
  a.cpl = d == 0 ? at.cpl[0] : (d == 1 ? at.cpl[1] : at.cpl[2]);
  a.m = d == 0 ? me[0] : (d == 1 ? me[1] : me[2]);
  a.ned = d == 0 ? dm.ne[0] : (d == 1 ? dm.ne[1] : dm.ne[2]);
  a.estride = (d == 0) ? 1 : (d == 1 ? (long long)dm.ne[0] : (long long)dm.ne[0] * dm.ne[1]);
  return a;
}

// What a line of axis d takes from its neighbours: the end value and end derivative of the
// line before (uP, dP) and behind (u0, d0); zero where there is none.
template <typename T>
struct LineEnds {
  T uP = T(0), dP = T(0), u0 = T(0), d0 = T(0);
  bool hasL = false, hasR = false;
};

// End value and end derivative (row Drow of the differentiation matrix) of the neighbour line
// un (nodes `stride` apart).  Double-float apply of an FP64 vector: the dot product runs in
// FP64 and only its result and the end value are split into two fp32 words (splitting all NP
// values and accumulating in double-float took about half of that kernel's issue slots; the
// FP64 pipe is otherwise idle there).
template <typename T, int NP, typename TIO, typename Load>
__device__ __forceinline__ void end_terms(const T* Drow, const double* Drow_d, int iend, Load&& load, T& uend, T& dend) {
  if constexpr (std::is_same<T, dfloat>::value && std::is_same<TIO, double>::value) {
    double s = 0.0, v = 0.0;
#pragma unroll
    for (int a = 0; a < NP; ++a) {
      const double val = load(a);
      s = ::fma(__ldg(Drow_d + a), val, s);
      if (a == iend) v = val;
    }
    uend = T(v);
    dend = T(s);
  } else {
    using A = AVec<T>;                           // the row is padded to whole vectors
    T s = T(0), v = T(0);
#pragma unroll
    for (int c = 0; c < NP; c += A::W) {
      const typename A::V w = __ldg(reinterpret_cast<const typename A::V*>(Drow + c));
#pragma unroll
      for (int k = 0; k < A::W; ++k)
        if (c + k < NP) {
          const T val = T(load(c + k));
          s = madd(A::get(w, k), val, s);
          if (c + k == iend) v = val;
        }
    }
    uend = v;
    dend = s;
  }
}

template <typename T, int NP>
__device__ __forceinline__ const T* coupling_rows(const ApplyAxis<T>& ax) {
  return ax.cpl + (size_t)ax.m * (2 * apad<T>(NP) + 8);
}
template <typename T>
__device__ __forceinline__ long long left_neighbour(const ApplyAxis<T>& ax, long long e) {
  return ax.m > 0 ? e - ax.estride : e + (long long)(ax.ned - 1) * ax.estride;
}
template <typename T>
__device__ __forceinline__ long long right_neighbour(const ApplyAxis<T>& ax, long long e) {
  return ax.m < ax.ned - 1 ? e + ax.estride : e - (long long)(ax.ned - 1) * ax.estride;
}
// the ends of the adjacent lines, read from global u
template <typename T, int NP, int NODES, typename TIO>
__device__ __forceinline__ LineEnds<T> line_ends(const ApplyTables<T>& at, const ApplyAxis<T>& ax,
                                                 const TIO* __restrict__ u, long long e, int off, int stride) {
  constexpr int PNP = apad<T>(NP);
  const T* c = coupling_rows<T, NP>(ax);
  LineEnds<T> le;
  le.hasL = ldg(c + 2 * PNP + 2) != T(0);
  le.hasR = ldg(c + 2 * PNP + 5) != T(0);
  if (le.hasL) {                                 // neighbour m-1
    const TIO* un = u + left_neighbour(ax, e) * NODES + off;
    end_terms<T, NP, TIO>(at.DP, at.DPd, NP - 1, [&](int a) { return __ldg(un + a * stride); }, le.uP, le.dP);
  }
  if (le.hasR) {                                 // neighbour m+1
    const TIO* un = u + right_neighbour(ax, e) * NODES + off;
    end_terms<T, NP, TIO>(at.D0, at.D0d, 0, [&](int a) { return __ldg(un + a * stride); }, le.u0, le.d0);
  }
  return le;
}

// y = M_d^-1 L_d u on one line of an element along axis d (values x): the element's own block
// L^0 (even-odd form when the block is centro-symmetric), plus the neighbour blocks L^-, L^+
// (rank <= 3, already scaled by M_d^-1) from the ends of the adjacent lines.  Mirrored
// coupling rows are folded into the even-odd accumulation (the tables flag them; 8-byte types).
template <typename T, int NP>
__device__ __forceinline__ void apply_line(const ApplyAxis<T>& ax, const LineEnds<T>& le, const T (&x)[NP], T (&y)[NP]) {
  constexpr int P = NP - 1;
  constexpr int H = NP / 2, NE = NP - H, NO = H;
  constexpr int PNP = apad<T>(NP);
  const T* L0 = ax.L0 + (size_t)ax.m * NP * PNP;
  const T* c = coupling_rows<T, NP>(ax);
  // c_R[P - i] = c_L[i]: c_L u_P + c_R u_0 = even part x (u_P + u_0) + odd part x (u_P - u_0)
  const bool csym = ldg(c + 2 * PNP + 6) != T(0);
  if (__ldg(ax.sym + ax.m)) {
    // even-odd split of the centro-symmetric block (folded, transposed rows)
    constexpr int PE = apad<T>(NE), PO = apad<T>(NO > 0 ? NO : 1);
    T xp[NE], xm[NO > 0 ? NO : 1];
#pragma unroll
    for (int a = 0; a < H; ++a) {
      xp[a] = x[a] + x[P - a];
      xm[a] = x[a] - x[P - a];
    }
    if (NE > H) xp[NE - 1] = x[H];
    T ae[NE], ao[NO > 0 ? NO : 1];
#pragma unroll
    for (int i = 0; i < NE; ++i) ae[i] = T(0);
#pragma unroll
    for (int i = 0; i < NO; ++i) ao[i] = T(0);
#pragma unroll
    for (int a = 0; a < NE; ++a) apply_axpy<T, NE>(ae, L0 + a * PE, xp[a]);
    if constexpr (NO > 0) {
#pragma unroll
      for (int a = 0; a < NO; ++a)
        apply_axpy<T, NO>(reinterpret_cast<T(&)[NO]>(ao), L0 + NE * PE + a * PO, xm[a]);
    }
    if (csym) {
      apply_axpy<T, NE>(ae, c, le.uP + le.u0);
      if constexpr (NO > 0) apply_axpy<T, NO>(reinterpret_cast<T(&)[NO]>(ao), c + PNP, le.uP - le.u0);
    }
#pragma unroll
    for (int i = 0; i < H; ++i) {
      y[i] = ae[i] + ao[i];
      y[P - i] = ae[i] - ao[i];
    }
    if (NE > H) y[H] = ae[H];
  } else {
#pragma unroll
    for (int i = 0; i < NP; ++i) y[i] = T(0);
#pragma unroll
    for (int a = 0; a < NP; ++a) apply_axpy<T, NP>(y, L0 + a * PNP, x[a]);
  }
  if (!csym) {
    if (le.hasL) apply_axpy<T, NP>(y, c, le.uP);
    if (le.hasR) apply_axpy<T, NP>(y, c + PNP, le.u0);
  }
  if (le.hasL) y[0] += ldg(c + 2 * PNP + 0) * le.dP - ldg(c + 2 * PNP + 1) * le.uP;
  if (le.hasR) y[P] = y[P] - (ldg(c + 2 * PNP + 3) * le.d0 + ldg(c + 2 * PNP + 4) * le.u0);
}

// SMALL: about one warp per CTA, for grids whose full CTAs would leave SMs idle
template <int DIM, int NP, bool SMALL = false>
struct ApplyShape {
  static constexpr int LINES = (DIM == 3) ? NP * NP : NP;
  static constexpr int NODES = (DIM == 3) ? NP * NP * NP : NP * NP;
  static constexpr int EPB = ((SMALL ? 32 : 128) / LINES) > 0 ? ((SMALL ? 32 : 128) / LINES) : 1;
  static constexpr int THREADS = ((EPB * LINES + 31) / 32) * 32;
  // CTAs per SM the register budget must allow (8-byte types): two for the 3-D
  // P = 16 kernel (320 threads), whose double-float form would otherwise take 114
  // registers and run one CTA per SM
  static constexpr int MINB8 = (DIM == 3 && NP == 17) ? 2 : 0;
  // fp32, staged: three CTAs per SM at P = 16 (64 registers; their shared memory), ten at P = 8
  static constexpr int MINB4 = (DIM == 3 && NP == 17) ? 3 : (DIM == 3 && NP == 9) ? 10 : 0;
};

// Whether the neighbours along x are staged in shared memory for their end derivatives: read
// line by line from global memory, a warp's load of one column touches a cache line per node
// line (17 wavefronts of the load unit at P = 16, 9 at P = 8, for 1 when staged).
template <typename T, int DIM, int NP>
constexpr bool apply_staged() {
  return sizeof(T) == 4 && DIM == 3 && (NP == 9 || NP == 17);
}
template <typename T, int DIM, int NP, bool SMALL = false>
constexpr size_t apply_smem_bytes() {
  using S = ApplyShape<DIM, NP, SMALL>;
  return sizeof(T) * ((size_t)2 * S::EPB * S::NODES + (apply_staged<T, DIM, NP>() ? S::NODES : 0));
}
template <typename T>
__device__ __forceinline__ void copy_async(T* smem, const T* global) {
  static_assert(sizeof(T) == 4, "one word");
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(global)
               : "memory");
}

// T: arithmetic and table type; TIO: type of u, f, v in global memory.
// NPC > 0 (with RESIDUAL): the residual is not stored but restricted at once,
// fc = (J (x) J (x) J)^T (f - A u) element by element (Sec. 3.2; J folded as in
// FoldedJ), in the operation order of the separate restriction kernel.
template <typename T, int DIM, int NP, bool RESIDUAL, typename TIO = T, int NPC = 0, bool SMALL = false>
__global__ void __launch_bounds__(ApplyShape<DIM, NP, SMALL>::THREADS,
                                  sizeof(T) == 8 ? ApplyShape<DIM, NP>::MINB8 : ApplyShape<DIM, NP>::MINB4)
apply_kernel(LevelDims dm, ApplyTables<T> at, const TIO* __restrict__ u, const TIO* __restrict__ f,
             TIO* __restrict__ v, FoldedJ<T, NP, NPC> J = FoldedJ<T, NP, NPC>{}, TIO* __restrict__ fc = nullptr,
             const int* __restrict__ unz = nullptr) {
  static_assert(!apply_staged<T, DIM, NP>() || std::is_same<T, TIO>::value, "staged raw");
  static_assert(NPC == 0 || (RESIDUAL && NPC < NP), "fused restriction: residual, coarser order");
  using S = ApplyShape<DIM, NP, SMALL>;
  constexpr bool STAGED = apply_staged<T, DIM, NP>();
  // axes unrolled (line offsets and strides become compile-time constants) and the ends of all
  // axes read at the start for the fp32 and FP64 kernels, except FP64 at P = 16, whose register
  // cap would then spill; the double-float kernel was measured faster with neither (instruction
  // cache, registers: P = 8 0.34 ms against 0.45 at 31 x 23 x 17 elements)
  constexpr bool EARLY = !std::is_same<T, dfloat>::value && !(sizeof(T) == 8 && NP == 17);
  constexpr int UNR = EARLY ? DIM : 1;
  extern __shared__ __align__(16) unsigned char apply_smem[];
  T* su = reinterpret_cast<T*>(apply_smem);
  T* acc = su + S::EPB * S::NODES;
  const int tid = threadIdx.x;
  const long long e0 = (long long)blockIdx.x * S::EPB;
  const int nodes_blk = (int)(dm.nelem - e0 < S::EPB ? dm.nelem - e0 : S::EPB) * S::NODES;
  const TIO* ub = u + e0 * S::NODES;
  if constexpr (NPC == 0) {
    // u identically zero (flag from any_nonzero_kernel): A u = 0, so v = f (or 0)
    if (unz && __ldg(unz) == 0) {
      for (int t = tid; t < nodes_blk; t += blockDim.x)
        v[e0 * S::NODES + t] = RESIDUAL ? f[e0 * S::NODES + t] : TIO(0);
      return;
    }
  }
  const int el = tid / S::LINES;
  const int line = tid % S::LINES;
  const bool active = el < S::EPB && e0 + el < dm.nelem;
  const long long e = active ? e0 + el : e0;
  const unsigned ne0 = (unsigned)dm.ne[0], ne1 = (unsigned)dm.ne[1], row = (unsigned)e / ne0;
  const int me[3] = {(int)((unsigned)e - row * ne0), DIM == 3 ? (int)(row % ne1) : (int)row, DIM == 3 ? (int)(row / ne1) : 0};
  auto line_off = [&](int d) { return d == 0 ? line * NP : DIM == 3 && d == 1 ? (line / NP) * NP * NP + line % NP : line; };
  auto line_stride = [](int d) { return d == 0 ? 1 : d == 1 ? NP : NP * NP; };
  // staged: the neighbours along x, the left one where pass x will accumulate (a thread reads
  // there the very entries that it then writes), the right one behind it
  TIO* xl = reinterpret_cast<TIO*>(acc);
  TIO* xr = reinterpret_cast<TIO*>(acc + S::NODES);
  LineEnds<T> ends[EARLY ? DIM : 1];
  if constexpr (STAGED) {
    const ApplyAxis<T> ax = apply_axis(dm, at, me, 0);
    const T* c = coupling_rows<T, NP>(ax);
    ends[0].hasL = ldg(c + 2 * apad<T>(NP) + 2) != T(0);
    ends[0].hasR = ldg(c + 2 * apad<T>(NP) + 5) != T(0);
    const TIO* ul = u + left_neighbour(ax, e) * S::NODES;
    const TIO* ur = u + right_neighbour(ax, e) * S::NODES;
    for (int t = tid; t < S::NODES; t += blockDim.x) {
      copy_async(su + t, ub + t);
      if (ends[0].hasL) copy_async(xl + t, ul + t);
      if (ends[0].hasR) copy_async(xr + t, ur + t);
    }
  }
  if constexpr (!STAGED)
    for (int t = tid; t < nodes_blk; t += blockDim.x) su[t] = T(ub[t]);
  if (EARLY && active) {
#pragma unroll
    for (int d = STAGED ? 1 : 0; d < DIM; ++d)
      ends[d] = line_ends<T, NP, S::NODES, TIO>(at, apply_axis(dm, at, me, d), u, e, line_off(d), line_stride(d));
  }
  if constexpr (STAGED) asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  if constexpr (STAGED) {
    if (active) {
      LineEnds<T>& le = ends[0];
      if (le.hasL) end_terms<T, NP, TIO>(at.DP, at.DPd, NP - 1, [&](int a) { return xl[line * NP + a]; }, le.uP, le.dP);
      if (le.hasR) end_terms<T, NP, TIO>(at.D0, at.D0d, 0, [&](int a) { return xr[line * NP + a]; }, le.u0, le.d0);
    }
  }
  T* sel = su + el * S::NODES;
  T* ael = acc + el * S::NODES;
#pragma unroll UNR
  for (int d = 0; d < DIM; ++d) {
    if (active) {
      const int off = line_off(d), stride = line_stride(d);
      T x[NP], y[NP];
#pragma unroll
      for (int a = 0; a < NP; ++a) x[a] = sel[off + a * stride];
      const ApplyAxis<T> ax = apply_axis(dm, at, me, d);
      LineEnds<T> le;
      if constexpr (EARLY) le = ends[d];
      else le = line_ends<T, NP, S::NODES, TIO>(at, ax, u, e, off, stride);
      apply_line<T, NP>(ax, le, x, y);
      if (d < DIM - 1) {
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          if (d == 0) ael[off + i * stride] = y[i];
          else ael[off + i * stride] += y[i];
        }
      } else {
        // v = (M_z (x) M_y (x) M_x) * (sum over axes of M_d^-1 L_d u), straight from the last
        // axis's lines (stride LINES: neighbouring threads hold neighbouring nodes)
        const T mx = ldg(at.M[0] + (size_t)me[0] * NP + line % NP);
        const T mxy = DIM == 3 ? mx * ldg(at.M[1] + (size_t)me[1] * NP + line / NP) : mx;
        const T* Ml = at.M[DIM - 1] + (size_t)me[DIM - 1] * NP;
        const long long g0 = e * S::NODES + line;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          const int k = i * S::LINES;
          const T val = mxy * ldg(Ml + i) * (ael[line + k] + y[i]);
          if constexpr (NPC > 0) ael[line + k] = T(f[g0 + k]) - val;
          else v[g0 + k] = RESIDUAL ? TIO(T(f[g0 + k]) - val) : TIO(val);
        }
      }
    }
    if (NPC > 0 || d < DIM - 1) __syncthreads();
  }
  if constexpr (NPC > 0) {
    // restriction of the element residuals (in acc): x, y and z passes with J^T,
    // one thread per line of a pass (even-odd folded, coefficients in parameters)
    constexpr int NZF = (DIM == 3) ? NP : 1;
    constexpr int B1 = NPC * NP * NZF, B2 = NPC * NPC * NZF;
    T* b1 = su;                                  // staged u is no longer needed
    #pragma unroll 1
    for (int t = tid; t < S::EPB * NP * NZF; t += blockDim.x) {      // x: lines (y, z)
      const int le = t / (NP * NZF), rest = t - le * (NP * NZF);
      const T* rr = acc + le * S::NODES + rest * NP;
      T x[NP];
#pragma unroll
      for (int a = 0; a < NP; ++a) x[a] = rr[a];
      T* dst = b1 + le * B1 + rest * NPC;
      fold_restrict<T, NP, NPC>(J, x, [&](int o, T v) { dst[o] = v; });
    }
    __syncthreads();
    T* b2 = acc;
    #pragma unroll 1
    for (int t = tid; t < S::EPB * NPC * NZF; t += blockDim.x) {     // y: lines (x', z)
      const int le = t / (NPC * NZF), tt = t - le * (NPC * NZF);
      const int i = tt % NPC, c = tt / NPC;
      T x[NP];
#pragma unroll
      for (int a = 0; a < NP; ++a) x[a] = b1[le * B1 + (c * NP + a) * NPC + i];
      if (DIM == 2) {
        if (e0 + le < dm.nelem) {
          TIO* dst = fc + (e0 + le) * B2 + i;
          fold_restrict<T, NP, NPC>(J, x, [&](int o, T v) { dst[o * NPC] = TIO(v); });
        }
      } else {
        T* dst = b2 + le * B2 + c * NPC * NPC + i;
        fold_restrict<T, NP, NPC>(J, x, [&](int o, T v) { dst[o * NPC] = v; });
      }
    }
    if (DIM == 3) {
      __syncthreads();
      constexpr int NC3 = NPC * NPC * NPC;
      #pragma unroll 1
      for (int t = tid; t < S::EPB * NPC * NPC; t += blockDim.x) {   // z: lines (x', y')
        const int le = t / (NPC * NPC), ij = t - le * (NPC * NPC);
        T x[NP];
#pragma unroll
        for (int a = 0; a < NP; ++a) x[a] = b2[le * B2 + a * NPC * NPC + ij];
        if (e0 + le < dm.nelem) {
          TIO* dst = fc + (e0 + le) * NC3 + ij;
          fold_restrict<T, NP, NPC>(J, x, [&](int o, T v) { dst[o * NPC * NPC] = TIO(v); });
        }
      }
    }
  }
}

// 3-D elements too large to stage in shared memory (P = 32: 33^3 nodes): one
// launch per axis d and one thread per (element, line).  The partial sums over
// the axes are kept in v between the launches (the same additions, in the same
// order, as the staged kernel's accumulator); the launch of the last axis applies
// the masses and forms v = A u or f - A u.
template <typename T, int NP, bool RESIDUAL, typename TIO>
// CTAs per SM: fp32 5 (96 registers), 8-byte types 3 (the double-float line needs 214 registers uncapped)
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 5 : 3)
apply_axis_kernel(LevelDims dm, ApplyTables<T> at, const TIO* __restrict__ u,
                  const TIO* __restrict__ f, TIO* __restrict__ v, int d, const int* __restrict__ unz) {
  constexpr int LINES = NP * NP, NODES = NP * NP * NP;
  const long long gid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (gid >= dm.nelem * LINES) return;
  const long long e = gid / LINES;
  const int line = (int)(gid - e * LINES);
  if (unz && __ldg(unz) == 0) {
    // u identically zero: v = f (or 0), written by the last axis's launch, line by line
    if (d == 2) {
#pragma unroll 1
      for (int i = 0; i < NP; ++i) {
        const long long g = e * NODES + line + (long long)i * NP * NP;
        v[g] = RESIDUAL ? f[g] : TIO(0);
      }
    }
    return;
  }
  const int me[3] = {(int)(e % dm.ne[0]), (int)((e / dm.ne[0]) % dm.ne[1]),
                     (int)(e / ((long long)dm.ne[0] * dm.ne[1]))};
  int off, stride;
  if (d == 0) { off = line * NP; stride = 1; }
  else if (d == 1) { off = (line / NP) * NP * NP + line % NP; stride = NP; }
  else { off = line; stride = NP * NP; }
  const TIO* ue = u + e * NODES;
  TIO* ve = v + e * NODES;
  T x[NP], y[NP];
#pragma unroll
  for (int a = 0; a < NP; ++a) x[a] = T(ue[off + a * stride]);
  const ApplyAxis<T> ax = apply_axis(dm, at, me, d);
  apply_line<T, NP>(ax, line_ends<T, NP, NODES, TIO>(at, ax, u, e, off, stride), x, y);
  if (d == 0) {
#pragma unroll
    for (int i = 0; i < NP; ++i) ve[off + i * stride] = TIO(y[i]);
  } else if (d == 1) {
#pragma unroll
    for (int i = 0; i < NP; ++i) ve[off + i * stride] = TIO(T(ve[off + i * stride]) + y[i]);
  } else {
#pragma unroll 1
    for (int i = 0; i < NP; ++i) {
      const int nd = off + i * stride;
      const int ii = nd % NP, jj = (nd / NP) % NP, kk = nd / (NP * NP);
      T m = ldg(at.M[0] + (size_t)me[0] * NP + ii) * ldg(at.M[1] + (size_t)me[1] * NP + jj);
      m = m * ldg(at.M[2] + (size_t)me[2] * NP + kk);
      const T val = m * (T(ve[nd]) + y[i]);
      ve[nd] = RESIDUAL ? TIO(T(f[e * NODES + nd]) - val) : TIO(val);
    }
  }
}

template <typename T, int NP, typename TIO>
static int apply_dispatch_axes(const LevelDims& dm, const ApplyTables<T>& at, const TIO* u, const TIO* f,
                               TIO* v, cudaStream_t s, const int* unz = nullptr) {
  const long long threads = dm.nelem * NP * NP;
  const long long blocks = (threads + 127) / 128;
  for (int d = 0; d < 3; ++d) {
    count_launch();
    if (f) apply_axis_kernel<T, NP, true, TIO><<<(unsigned)blocks, 128, 0, s>>>(dm, at, u, f, v, d, unz);
    else apply_axis_kernel<T, NP, false, TIO><<<(unsigned)blocks, 128, 0, s>>>(dm, at, u, f, v, d, unz);
  }
  return cudaGetLastError() == cudaSuccess ? PMG_OK : PMG_ECUDA;
}

// Whether the grid should take one-warp CTAs: full ones (4 warps of elements) would not fill
// two per SM.  2-D 16 x 16 elements, P = 8: 19 CTAs of 14 elements -> 86 of 3.
template <int DIM, int NP>
static bool small_grid(long long nelem) {
  using S = ApplyShape<DIM, NP>;
  return S::EPB > 1 && nelem < 2 * 152 * (long long)S::EPB;
}

template <typename T, int DIM, int NP, bool SMALL, typename TIO = T>
static int apply_dispatch_size(const LevelDims& dm, const ApplyTables<T>& at, const TIO* u, const TIO* f,
                               TIO* v, cudaStream_t s, const int* unz) {
  using S = ApplyShape<DIM, NP, SMALL>;
  long long blocks = (dm.nelem + S::EPB - 1) / S::EPB;
  const size_t smem = apply_smem_bytes<T, DIM, NP, SMALL>();
  auto fn = f ? apply_kernel<T, DIM, NP, true, TIO, 0, SMALL> : apply_kernel<T, DIM, NP, false, TIO, 0, SMALL>;
  if (!set_smem(fn, smem)) return PMG_ECUDA;
  count_launch();
  fn<<<(unsigned)blocks, S::THREADS, smem, s>>>(dm, at, u, f, v, FoldedJ<T, NP, 0>{}, nullptr, unz);
  return cudaGetLastError() == cudaSuccess ? PMG_OK : PMG_ECUDA;
}

template <typename T, int DIM, int NP, typename TIO = T>
static int apply_dispatch(const LevelDims& dm, const ApplyTables<T>& at, const TIO* u, const TIO* f,
                          TIO* v, cudaStream_t s, const int* unz = nullptr) {
  if constexpr (ApplyShape<DIM, NP>::EPB > 1)
    if (small_grid<DIM, NP>(dm.nelem)) return apply_dispatch_size<T, DIM, NP, true, TIO>(dm, at, u, f, v, s, unz);
  return apply_dispatch_size<T, DIM, NP, false, TIO>(dm, at, u, f, v, s, unz);
}

// v-less residual + restriction: fc = I^T (f - A u) for the staged kernel's shapes;
// PMG_EINVAL where no fused kernel exists (the caller then runs the two kernels).
template <typename T, int DIM, int NP, int NPC, bool SMALL>
static int residual_restrict_size(const LevelDims& dm, const ApplyTables<T>& at, const T* u, const T* f,
                                  const double* Jh, T* fc, cudaStream_t s) {
  const FoldedJ<T, NP, NPC> J = fold_interpolation<T, NP, NPC>(Jh);
  using S = ApplyShape<DIM, NP, SMALL>;
  long long blocks = (dm.nelem + S::EPB - 1) / S::EPB;
  const size_t smem = apply_smem_bytes<T, DIM, NP, SMALL>();
  auto fn = apply_kernel<T, DIM, NP, true, T, NPC, SMALL>;
  if (!set_smem(fn, smem)) return PMG_ECUDA;
  count_launch();
  fn<<<(unsigned)blocks, S::THREADS, smem, s>>>(dm, at, u, f, nullptr, J, fc, nullptr);
  return cudaGetLastError() == cudaSuccess ? PMG_OK : PMG_ECUDA;
}
template <typename T, int DIM, int NP, int NPC>
static int residual_restrict_dispatch(const LevelDims& dm, const ApplyTables<T>& at, const T* u, const T* f,
                                      const double* Jh, T* fc, cudaStream_t s) {
  if constexpr (ApplyShape<DIM, NP>::EPB > 1)
    if (small_grid<DIM, NP>(dm.nelem)) return residual_restrict_size<T, DIM, NP, NPC, true>(dm, at, u, f, Jh, fc, s);
  return residual_restrict_size<T, DIM, NP, NPC, false>(dm, at, u, f, Jh, fc, s);
}

}  // namespace pmg
