// CUDA kernels of the p-multigrid DG Poisson solver (sm_103a): operator apply,
// mass, restriction / prolongation, exact coarse solve, CG vector kernels.
// The Schwarz patch kernel lives in fdm_kernel.cuh.
//
// Paper: Stiller, arXiv 1603.02524 (Sec. 2.4 operator, Sec. 3.2 transfers,
// Algorithm 2 vector steps).
#include <cstdint>
#include <cstdio>
#include <type_traits>

#include "apply_kernel.cuh"

namespace pmg {

template <typename T>
int launch_apply(const LevelDims& dm, const ApplyTables<T>& at, const T* u, const T* f, T* v,
                 cudaStream_t s, const int* unz) {
  if (dm.nelem == 0) return PMG_OK;
  if constexpr (sizeof(T) == 8) {
    const int st = launch_apply_split(dm, at, u, f, v, s, unz);
    if (st != PMG_EINVAL) return st;
  }
#define PMG_APPLY_CASE(DIMV, NPV) \
  if (dm.dim == DIMV && dm.NP == NPV) return apply_dispatch<T, DIMV, NPV>(dm, at, u, f, v, s, unz);
  PMG_APPLY_CASE(3, 2) PMG_APPLY_CASE(3, 3) PMG_APPLY_CASE(3, 5) PMG_APPLY_CASE(3, 9)
  PMG_APPLY_CASE(3, 17)
  if (dm.dim == 3 && dm.NP == 33) return apply_dispatch_axes<T, 33, T>(dm, at, u, f, v, s, unz);
  PMG_APPLY_CASE(2, 2) PMG_APPLY_CASE(2, 3) PMG_APPLY_CASE(2, 5) PMG_APPLY_CASE(2, 9)
  PMG_APPLY_CASE(2, 17) PMG_APPLY_CASE(2, 33)
#undef PMG_APPLY_CASE
  return PMG_EINVAL;
}
// fc = I^T (f - A u) in one kernel (the residual is not stored); PMG_EINVAL for
// shapes without the fused kernel (3-D P = 32), where the caller runs the two.
template <typename T>
int launch_residual_restrict(const LevelDims& dm, const ApplyTables<T>& at, const T* u, const T* f,
                             const T* /*J*/, const double* Jh, T* fc, cudaStream_t s) {
  if (dm.nelem == 0) return PMG_OK;
  if constexpr (sizeof(T) == 8) {
    const int st = launch_residual_restrict_split(dm, at, u, f, fc, s);
    if (st != PMG_EINVAL) return st;
  }
  if (!Jh) return PMG_EINVAL;
#define PMG_RR_CASE(DIMV, NPV, NPCV) \
  if (dm.dim == DIMV && dm.NP == NPV) return residual_restrict_dispatch<T, DIMV, NPV, NPCV>(dm, at, u, f, Jh, fc, s);
  PMG_RR_CASE(3, 3, 2) PMG_RR_CASE(3, 5, 3) PMG_RR_CASE(3, 9, 5) PMG_RR_CASE(3, 17, 9)
  PMG_RR_CASE(2, 3, 2) PMG_RR_CASE(2, 5, 3) PMG_RR_CASE(2, 9, 5) PMG_RR_CASE(2, 17, 9) PMG_RR_CASE(2, 33, 17)
#undef PMG_RR_CASE
  return PMG_EINVAL;
}
template int launch_residual_restrict<double>(const LevelDims&, const ApplyTables<double>&, const double*,
                                              const double*, const double*, const double*, double*,
                                              cudaStream_t);
template int launch_residual_restrict<float>(const LevelDims&, const ApplyTables<float>&, const float*,
                                             const float*, const float*, const double*, float*, cudaStream_t);

template int launch_apply<double>(const LevelDims&, const ApplyTables<double>&, const double*,
                                  const double*, double*, cudaStream_t, const int*);
template int launch_apply<float>(const LevelDims&, const ApplyTables<float>&, const float*,
                                 const float*, float*, cudaStream_t, const int*);

// *flag = 1 if some x[i] != 0 (a NaN counts as nonzero); the caller zeroes the flag
__global__ void __launch_bounds__(256) any_nonzero_kernel(const double* __restrict__ x, long long n, int* flag) {
  bool nz = false;
  for (long long i = blockIdx.x * 256LL + threadIdx.x; i < n; i += (long long)gridDim.x * 256) nz |= !(x[i] == 0.0);
  if (__syncthreads_or(nz) && threadIdx.x == 0) *flag = 1;
}
void launch_any_nonzero(const double* x, long long n, int* flag, cudaStream_t s) {
  if (n <= 0) return;
  long long blocks = (n + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  count_launch();
  any_nonzero_kernel<<<(unsigned)blocks, 256, 0, s>>>(x, n, flag);
}

// ---------------------------------------------------------------------------
// g = M f: diagonal GLL mass (Sec. 2.4 right-hand side)
// ---------------------------------------------------------------------------
__global__ void mass_kernel(LevelDims dm, ApplyTables<double> at, const double* __restrict__ f,
                            double* __restrict__ g) {
  const int NP = dm.NP;
  const long long nodes = (dm.dim == 3) ? (long long)NP * NP * NP : (long long)NP * NP;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < dm.ndof;
       t += (long long)gridDim.x * blockDim.x) {
    long long e = t / nodes;
    int n = (int)(t % nodes);
    int i = n % NP, j = (n / NP) % NP, k = n / (NP * NP);
    int mx = (int)(e % dm.ne[0]), my = (int)((e / dm.ne[0]) % dm.ne[1]);
    int mz = (int)(e / ((long long)dm.ne[0] * dm.ne[1]));
    double s = at.M[0][(size_t)mx * NP + i] * at.M[1][(size_t)my * NP + j];
    if (dm.dim == 3) s *= at.M[2][(size_t)mz * NP + k];
    g[t] = s * f[t];
  }
}

void launch_mass(const LevelDims& dm, const ApplyTables<double>& at, const double* f, double* g,
                 cudaStream_t s) {
  long long blocks = (dm.ndof + 255) / 256;
  if (blocks > 65535 * 8) blocks = 65535 * 8;
  count_launch(); mass_kernel<<<(unsigned)blocks, 256, 0, s>>>(dm, at, f, g);
}

// ---------------------------------------------------------------------------
// Transfers (Sec. 3.2): prolongation u_f += (J (x) J (x) J) u_c, restriction
// f_c = (J (x) J (x) J)^T r_f, element by element, with J even-odd folded (FoldedJ
// in apply_kernel.cuh).  One CTA per element; three passes through shared memory,
// one thread per line of a pass.
// ---------------------------------------------------------------------------
template <typename T, int DIM, int NPF, int NPC, bool PROLONG>
__global__ void __launch_bounds__(256)
transfer_kernel(long long nelem, FoldedJ<T, NPF, NPC> J, const T* __restrict__ in, T* __restrict__ out) {
  constexpr int NIN = PROLONG ? NPC : NPF;      // per-axis size of the input
  constexpr int NOUT = PROLONG ? NPF : NPC;
  constexpr int NZI = (DIM == 3) ? NIN : 1;
  constexpr int NZO = (DIM == 3) ? NOUT : 1;
  extern __shared__ __align__(16) unsigned char tr_smem[];
  T* b0 = reinterpret_cast<T*>(tr_smem);
  T* b1 = b0 + NIN * NIN * NZI;
  T* b2 = b1 + NOUT * NIN * NZI;
  const long long e = blockIdx.x;
  // FP64: the coefficients from a shared-memory copy (as constant operands the
  // compiler keeps all of them in registers, 130 per thread, one CTA per SM)
  __shared__ FoldedJ<T, NPF, NPC> sJ;
  if constexpr (sizeof(T) == 8) {
    if (threadIdx.x == 0) sJ = J;
  }
  for (int t = threadIdx.x; t < NIN * NIN * NZI; t += blockDim.x)
    b0[t] = in[e * (NIN * NIN * NZI) + t];
  __syncthreads();
  // one axis line: NIN inputs `sstride` apart -> NOUT outputs (even-odd folded J),
  // each handed to put(index, value)
  auto line = [&](const T* src, int sstride, auto&& put) {
    T x[NIN];
#pragma unroll
    for (int a = 0; a < NIN; ++a) x[a] = src[a * sstride];
    const FoldedJ<T, NPF, NPC>* jp = &J;
    if constexpr (sizeof(T) == 8) {
      jp = &sJ;
      asm volatile("" : "+l"(jp));             // opaque per line: loaded as used, not hoisted
    }
    if constexpr (PROLONG) fold_prolong<T, NPF, NPC>(*jp, x, put);
    else fold_restrict<T, NPF, NPC>(*jp, x, put);
  };
#pragma unroll 1
  for (int r = threadIdx.x; r < NIN * NZI; r += blockDim.x) {          // x: lines (y, z)
    T* dst = b1 + r * NOUT;
    line(b0 + r * NIN, 1, [&](int o, T v) { dst[o] = v; });
  }
  __syncthreads();
#pragma unroll 1
  for (int t = threadIdx.x; t < NOUT * NZI; t += blockDim.x) {         // y: lines (x', z)
    const int i = t % NOUT, c = t / NOUT;
    if (DIM == 2) {
      T* dst = out + e * (NOUT * NOUT) + i;
      line(b1 + c * NIN * NOUT + i, NOUT, [&](int o, T v) {
        if (PROLONG) dst[o * NOUT] += v;
        else dst[o * NOUT] = v;
      });
    } else {
      T* dst = b2 + c * NOUT * NOUT + i;
      line(b1 + c * NIN * NOUT + i, NOUT, [&](int o, T v) { dst[o * NOUT] = v; });
    }
  }
  if (DIM == 2) return;
  __syncthreads();
#pragma unroll 1
  for (int ij = threadIdx.x; ij < NOUT * NOUT; ij += blockDim.x) {     // z: lines (x', y')
    T* dst = out + e * (NOUT * NOUT * NZO) + ij;
    line(b2 + ij, NOUT * NOUT, [&](int o, T v) {
      if (PROLONG) dst[o * NOUT * NOUT] += v;
      else dst[o * NOUT * NOUT] = v;
    });
  }
}

// 3-D transfers between P = 32 and P = 16 (33 and 17 nodes per axis): the
// three element-sized buffers of transfer_kernel do not fit shared memory, so the
// passes share one buffer of 17 x 33 x 33 entries: the first pass reads global
// memory, the middle pass works in place line by line (a thread holds its whole
// line in registers before it writes it), the last pass writes global memory.
template <typename T, bool PROLONG>
__global__ void __launch_bounds__(256)
transfer_big_kernel(long long nelem, const T* __restrict__ J, const T* __restrict__ in,
                    T* __restrict__ out) {
  constexpr int F = 33, C = 17;
  extern __shared__ __align__(16) unsigned char trb_smem[];
  T* sJ = reinterpret_cast<T*>(trb_smem);          // J[f][c]
  T* b = sJ + F * C;                                // [C][F][F]
  const long long e = blockIdx.x;
  for (int t = threadIdx.x; t < F * C; t += blockDim.x) sJ[t] = J[t];
  __syncthreads();
  if (!PROLONG) {
    const T* ie = in + e * (F * F * F);
    for (int t = threadIdx.x; t < C * F * F; t += blockDim.x) {   // z: F -> C
      const int oz = t / (F * F), rem = t - oz * F * F;
      T s = T(0);
#pragma unroll 1
      for (int k = 0; k < F; ++k) s = fma(sJ[k * C + oz], ie[k * F * F + rem], s);
      b[t] = s;
    }
    __syncthreads();
    for (int l = threadIdx.x; l < C * F; l += blockDim.x) {       // y: F -> C, in place
      const int oz = l / F, i = l - oz * F;
      T v[F];
#pragma unroll
      for (int j = 0; j < F; ++j) v[j] = b[(oz * F + j) * F + i];
#pragma unroll
      for (int oj = 0; oj < C; ++oj) {
        T s = T(0);
#pragma unroll
        for (int j = 0; j < F; ++j) s = fma(sJ[j * C + oj], v[j], s);
        b[(oz * F + oj) * F + i] = s;
      }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < C * C * C; t += blockDim.x) {   // x: F -> C, to global
      const int ox = t % C, oj = (t / C) % C, oz = t / (C * C);
      const T* row = b + (oz * F + oj) * F;
      T s = T(0);
#pragma unroll
      for (int i = 0; i < F; ++i) s = fma(sJ[i * C + ox], row[i], s);
      out[e * (C * C * C) + t] = s;
    }
  } else {
    const T* ie = in + e * (C * C * C);
    for (int t = threadIdx.x; t < C * C * F; t += blockDim.x) {   // x: C -> F
      const int xo = t % F, jc = (t / F) % C, kc = t / (F * C);
      const T* row = ie + (kc * C + jc) * C;
      T s = T(0);
#pragma unroll
      for (int ic = 0; ic < C; ++ic) s = fma(sJ[xo * C + ic], row[ic], s);
      b[(kc * F + jc) * F + xo] = s;
    }
    __syncthreads();
    for (int l = threadIdx.x; l < C * F; l += blockDim.x) {       // y: C -> F, in place
      const int kc = l / F, xo = l - kc * F;
      T v[C];
#pragma unroll
      for (int jc = 0; jc < C; ++jc) v[jc] = b[(kc * F + jc) * F + xo];
#pragma unroll
      for (int yo = 0; yo < F; ++yo) {
        T s = T(0);
#pragma unroll
        for (int jc = 0; jc < C; ++jc) s = fma(sJ[yo * C + jc], v[jc], s);
        b[(kc * F + yo) * F + xo] = s;
      }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < F * F * F; t += blockDim.x) {   // z: C -> F, add to global
      const int xy = t % (F * F), zo = t / (F * F);
      T s = T(0);
#pragma unroll
      for (int kc = 0; kc < C; ++kc) s = fma(sJ[zo * C + kc], b[kc * F * F + xy], s);
      out[e * (F * F * F) + t] += s;
    }
  }
}

template <typename T, bool PROLONG>
static int transfer_launch(const LevelDims& fine, const LevelDims& coarse, const T* J, const double* Jh,
                           const T* in, T* out, cudaStream_t s) {
  if (fine.nelem == 0) return PMG_OK;
  unsigned blocks = (unsigned)fine.nelem;
#define PMG_TR_CASE(DIMV, NPF, NPC) \
  if (fine.dim == DIMV && fine.NP == NPF && coarse.NP == NPC) { \
    if (!Jh) return PMG_EINVAL; \
    constexpr int NIN = PROLONG ? NPC : NPF, NOUT = PROLONG ? NPF : NPC; \
    constexpr int NZI = DIMV == 3 ? NIN : 1; \
    const size_t smem = sizeof(T) * (NIN * NIN * NZI + NOUT * NIN * NZI + NOUT * NOUT * NZI); \
    if (!set_smem(transfer_kernel<T, DIMV, NPF, NPC, PROLONG>, smem)) return PMG_ECUDA; \
    count_launch(); \
    transfer_kernel<T, DIMV, NPF, NPC, PROLONG><<<blocks, 256, smem, s>>>( \
        fine.nelem, fold_interpolation<T, NPF, NPC>(Jh), in, out); \
    return cudaGetLastError() == cudaSuccess ? PMG_OK : PMG_ECUDA; }
  PMG_TR_CASE(3, 3, 2) PMG_TR_CASE(3, 5, 3) PMG_TR_CASE(3, 9, 5) PMG_TR_CASE(3, 17, 9)
  PMG_TR_CASE(2, 3, 2) PMG_TR_CASE(2, 5, 3) PMG_TR_CASE(2, 9, 5) PMG_TR_CASE(2, 17, 9)
  PMG_TR_CASE(2, 33, 17)
#undef PMG_TR_CASE
  if (fine.dim == 3 && fine.NP == 33 && coarse.NP == 17) {
    const size_t smem = sizeof(T) * (33 * 17 + 17 * 33 * 33);
    if (!set_smem(transfer_big_kernel<T, PROLONG>, smem)) return PMG_ECUDA;
    count_launch(); transfer_big_kernel<T, PROLONG><<<blocks, 256, smem, s>>>(fine.nelem, J, in, out);
    return cudaGetLastError() == cudaSuccess ? PMG_OK : PMG_ECUDA;
  }
  return PMG_EINVAL;
}

template <typename T>
int launch_restrict(const LevelDims& fine, const LevelDims& coarse, const T* J, const double* Jh,
                    const T* rf, T* fc, cudaStream_t s) {
  return transfer_launch<T, false>(fine, coarse, J, Jh, rf, fc, s);
}
template <typename T>
int launch_prolong(const LevelDims& fine, const LevelDims& coarse, const T* J, const double* Jh,
                   const T* uc, T* uf, cudaStream_t s) {
  return transfer_launch<T, true>(fine, coarse, J, Jh, uc, uf, s);
}
template int launch_restrict<double>(const LevelDims&, const LevelDims&, const double*, const double*,
                                     const double*, double*, cudaStream_t);
template int launch_restrict<float>(const LevelDims&, const LevelDims&, const float*, const double*,
                                    const float*, float*, cudaStream_t);
template int launch_prolong<double>(const LevelDims&, const LevelDims&, const double*, const double*,
                                    const double*, double*, cudaStream_t);
template int launch_prolong<float>(const LevelDims&, const LevelDims&, const float*, const double*,
                                   const float*, float*, cudaStream_t);

// ---------------------------------------------------------------------------
// Exact coarse solve at P = 1 (A_0^+ f_0): the coarse operator is
// M3(x)M2(x)L1 + M3(x)L2(x)M1 + L3(x)M2(x)M1 with global 1-D factors, so
// A_0^{-1} = (S3(x)S2(x)S1) (sum Lambda)^{-1} (S3(x)S2(x)S1)^T  -- the fast
// diagonalisation of Sec. 3.1 applied to the whole coarse grid.  The zero mode
// of a periodic grid (all three lambda = 0) is dropped (pseudo-inverse).
// ---------------------------------------------------------------------------
__device__ __forceinline__ long long coarse_off(const LevelDims& dm, int X, int Y, int Z) {
  int ex = X >> 1, i = X & 1, ey = Y >> 1, j = Y & 1;
  if (dm.dim == 2) return ((long long)ey * dm.ne[0] + ex) * 4 + j * 2 + i;
  int ez = Z >> 1, k = Z & 1;
  return (((long long)ez * dm.ne[1] + ey) * dm.ne[0] + ex) * 8 + (k * 2 + j) * 2 + i;
}

// Eigenvalue sum of a coarse mode: its inverse, or 0 for the zero mode of a periodic grid.
__device__ __forceinline__ double coarse_scale(const LevelDims& dm, const CoarseFdm& c, int X, int Y, int Z, double v,
                                               double tol) {
  const double l = c.lam[0][X] + c.lam[1][Y] + (dm.dim == 3 ? c.lam[2][Z] : 0.0);
  return l > tol ? v / l : 0.0;
}

// One pass over all lines of an axis, nl lines per CTA staged in shared memory: forward
// transform (MODE 0), backward (1), or on the last axis forward, scaling by the inverse
// eigenvalue sums and backward at once (2).  The S tables are read with consecutive outputs
// in consecutive lanes (forward S, backward its transpose ST).  Five launches in 3-D, three in
// 2-D, on the vectors of the V-cycle's own precision; one more for a last axis beyond kCoarseLine.
template <int MODE, typename TI, typename TO>
__global__ void __launch_bounds__(128)
coarse_lines_kernel(LevelDims dm, CoarseFdm c, int axis, int nl, const TI* __restrict__ in, TO* __restrict__ out,
                    double tol) {
  extern __shared__ __align__(16) unsigned char cl_smem[];
  const int NX = dm.ne[0] * 2, NY = dm.ne[1] * 2, NZ = (dm.dim == 3) ? dm.ne[2] * 2 : 1;
  const int N = axis == 0 ? NX : axis == 1 ? NY : NZ, n1 = axis == 0 ? NY : NX;
  const long long lines = (long long)NX * NY * NZ / N;
  const double* S = axis == 0 ? c.S[0] : axis == 1 ? c.S[1] : c.S[2];
  const double* ST = axis == 0 ? c.ST[0] : axis == 1 ? c.ST[1] : c.ST[2];
  double* a = reinterpret_cast<double*>(cl_smem);           // [nl][N]
  double* b = a + (size_t)nl * N;                            // MODE 2 only
  const long long l0 = (long long)blockIdx.x * nl;
  const int nlb = (int)min((long long)nl, lines - l0);
  // coordinates of entry o of line l (x slowest-varying choice per axis)
  auto where = [&](int l, int o, int& X, int& Y, int& Z) {
    const int u = (int)((l0 + l) % n1), w = (int)((l0 + l) / n1);
    X = axis == 0 ? o : u;
    Y = axis == 0 ? u : axis == 1 ? o : w;
    Z = axis == 2 ? o : w;
  };
  for (int t = threadIdx.x; t < nlb * N; t += blockDim.x) {
    int X, Y, Z;
    where(t / N, t % N, X, Y, Z);
    a[t] = (double)in[coarse_off(dm, X, Y, Z)];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < nlb * N; t += blockDim.x) {
    const int l = t / N, o = t - l * N;
    const double* M = MODE == 1 ? ST : S;
    double s = 0.0;
#pragma unroll 8
    for (int k = 0; k < N; ++k) s = fma(__ldg(M + (size_t)k * N + o), a[l * N + k], s);
    int X, Y, Z;
    where(l, o, X, Y, Z);
    if constexpr (MODE == 2) b[t] = coarse_scale(dm, c, X, Y, Z, s, tol);
    else out[coarse_off(dm, X, Y, Z)] = (TO)s;
  }
  if constexpr (MODE == 2) {
    __syncthreads();
    for (int t = threadIdx.x; t < nlb * N; t += blockDim.x) {
      const int l = t / N, o = t - l * N;
      double s = 0.0;
#pragma unroll 8
      for (int k = 0; k < N; ++k) s = fma(__ldg(ST + (size_t)k * N + o), b[l * N + k], s);
      int X, Y, Z;
      where(l, o, X, Y, Z);
      out[coarse_off(dm, X, Y, Z)] = (TO)s;
    }
  }
}

// One pass over the lines of a long axis: a CTA forms 128 outputs of a line, whose inputs are
// staged a chunk at a time, so the length has no limit.  MODE 0, 1 as above; 3: forward and scaling.
constexpr int kCoarseLine = 2048;         // longest line of coarse_lines_kernel
template <int MODE, typename TI, typename TO>
__global__ void __launch_bounds__(128)
coarse_long_kernel(LevelDims dm, CoarseFdm c, int axis, const TI* __restrict__ in, TO* __restrict__ out, double tol) {
  constexpr int CHUNK = 1024;
  __shared__ double a[CHUNK];
  const int NX = dm.ne[0] * 2, NY = dm.ne[1] * 2, NZ = (dm.dim == 3) ? dm.ne[2] * 2 : 1;
  const int N = axis == 0 ? NX : axis == 1 ? NY : NZ, n1 = axis == 0 ? NY : NX;
  const int u = (int)(blockIdx.x % n1), w = (int)(blockIdx.x / n1), o = blockIdx.y * 128 + threadIdx.x;
  const double* M = MODE == 1 ? (axis == 0 ? c.ST[0] : axis == 1 ? c.ST[1] : c.ST[2])
                              : (axis == 0 ? c.S[0] : axis == 1 ? c.S[1] : c.S[2]);
  auto X = [&](int q) { return axis == 0 ? q : u; };
  auto Y = [&](int q) { return axis == 0 ? u : axis == 1 ? q : w; };
  auto Z = [&](int q) { return axis == 2 ? q : w; };
  double s = 0.0;
  for (int k0 = 0; k0 < N; k0 += CHUNK) {
    const int nk = min(CHUNK, N - k0);
    __syncthreads();
    for (int k = threadIdx.x; k < nk; k += 128) a[k] = (double)in[coarse_off(dm, X(k0 + k), Y(k0 + k), Z(k0 + k))];
    __syncthreads();
    if (o < N) {
#pragma unroll 8
      for (int k = 0; k < nk; ++k) s = fma(__ldg(M + (size_t)(k0 + k) * N + o), a[k], s);
    }
  }
  if (o < N) out[coarse_off(dm, X(o), Y(o), Z(o))] = (TO)(MODE == 3 ? coarse_scale(dm, c, X(o), Y(o), Z(o), s, tol) : s);
}

// The whole solve in one CTA, for coarse grids whose passes are shorter than a launch.
template <typename TI, typename TO>
__global__ void __launch_bounds__(512)
coarse_small_kernel(LevelDims dm, CoarseFdm c, const TI* __restrict__ in, TO* __restrict__ out, double tol) {
  extern __shared__ __align__(16) unsigned char cl_smem[];
  const int NX = dm.ne[0] * 2, NY = dm.ne[1] * 2, NZ = (dm.dim == 3) ? dm.ne[2] * 2 : 1;
  const int total = NX * NY * NZ;
  double* a = reinterpret_cast<double*>(cl_smem);
  double* b = a + total;
  for (int t = threadIdx.x; t < total; t += blockDim.x)
    a[t] = (double)in[coarse_off(dm, t % NX, t / NX % NY, t / (NX * NY))];
  for (int q = 0; q < 2 * dm.dim; ++q) {
    const int d = q < dm.dim ? q : 2 * dm.dim - 1 - q;
    const int N = d == 0 ? NX : d == 1 ? NY : NZ, st = d == 0 ? 1 : d == 1 ? NX : NX * NY;
    const double* M = q < dm.dim ? (d == 0 ? c.S[0] : d == 1 ? c.S[1] : c.S[2])
                                 : (d == 0 ? c.ST[0] : d == 1 ? c.ST[1] : c.ST[2]);
    __syncthreads();
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
      const int o = t / st % N;
      const double* line = a + t - o * st;
      double s = 0.0;
#pragma unroll 8
      for (int k = 0; k < N; ++k) s = fma(__ldg(M + (size_t)k * N + o), line[k * st], s);
      if (q == dm.dim - 1) s = coarse_scale(dm, c, t % NX, t / NX % NY, t / (NX * NY), s, tol);
      b[t] = s;
    }
    double* w = a;
    a = b;
    b = w;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < total; t += blockDim.x)
    out[coarse_off(dm, t % NX, t / NX % NY, t / (NX * NY))] = (TO)a[t];
}

template <typename TIO>
int launch_coarse_fdm(const LevelDims& dm, const CoarseFdm& c, const TIO* f, TIO* u, cudaStream_t s) {
  const double tol = 1e-13 * c.lam_max;
  const long long total = (long long)c.N[0] * c.N[1] * (dm.dim == 3 ? c.N[2] : 1);
  const int nsum = c.N[0] + c.N[1] + (dm.dim == 3 ? c.N[2] : 0);
  // one CTA up to 12 k multiply-adds per direction (its SM's FP64 pipe: at most 7 us each way)
  if (total <= 2048 && total * nsum <= 12288) {
    count_launch();
    const int threads = total <= 64 ? 64 : total <= 256 ? 256 : 512;
    coarse_small_kernel<TIO, TIO><<<1, threads, 2 * sizeof(double) * total, s>>>(dm, c, f, u, tol);
    return cudaGetLastError() == cudaSuccess ? PMG_OK : PMG_ECUDA;
  }
  const int last = dm.dim - 1;
  int rc = PMG_OK;
  // mode 0: forward, 1: backward, 2: forward, scaled and backward, 3: forward and scaled
  auto pass = [&](int axis, auto mode, auto in, auto out) {
    using TI = std::remove_cv_t<std::remove_pointer_t<decltype(in)>>;
    using TO = std::remove_pointer_t<decltype(out)>;
    constexpr int MODE = decltype(mode)::value;
    if (rc != PMG_OK) return;
    const int N = c.N[axis];
    const long long lines = total / N;
    count_launch();
    if constexpr (MODE != 2) {
      if (N > kCoarseLine)
        coarse_long_kernel<MODE, TI, TO><<<dim3((unsigned)lines, (N + 127) / 128), 128, 0, s>>>(dm, c, axis, in, out, tol);
    }
    if constexpr (MODE != 3) {
      if (N <= kCoarseLine) {
        const int nl = N < 128 ? 128 / N : 1;
        const size_t smem = sizeof(double) * (size_t)nl * N * (MODE == 2 ? 2 : 1);
        coarse_lines_kernel<MODE, TI, TO><<<(unsigned)((lines + nl - 1) / nl), 128, smem, s>>>(dm, c, axis, nl, in, out, tol);
      }
    }
    if (cudaGetLastError() != cudaSuccess) rc = PMG_ECUDA;
  };
  double* t[2] = {c.tmp[0], c.tmp[1]};
  int k = 0;
  pass(0, std::integral_constant<int, 0>{}, f, t[0]);
  auto next = [&](int axis, auto mode) {
    pass(axis, mode, (const double*)t[k], t[k ^ 1]);
    k ^= 1;
  };
  if (last == 2) next(1, std::integral_constant<int, 0>{});
  if (c.N[last] > kCoarseLine) {
    next(last, std::integral_constant<int, 3>{});
    next(last, std::integral_constant<int, 1>{});
  } else {
    next(last, std::integral_constant<int, 2>{});
  }
  if (last == 2) next(1, std::integral_constant<int, 1>{});
  pass(0, std::integral_constant<int, 1>{}, (const double*)t[k], u);
  return rc;
}
template int launch_coarse_fdm<double>(const LevelDims&, const CoarseFdm&, const double*, double*, cudaStream_t);
template int launch_coarse_fdm<float>(const LevelDims&, const CoarseFdm&, const float*, float*, cudaStream_t);

// ---------------------------------------------------------------------------
// Vector kernels of Algorithm 2.  Reductions are deterministic: fixed grid,
// per-block partial sums in a fixed order, final sum by the last block to
// finish (threadfence + counter), also in a fixed order.
// ---------------------------------------------------------------------------
template <typename Ta, typename Tb>
__global__ void convert_kernel(const Ta* __restrict__ in, Tb* __restrict__ out, long long n) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    out[t] = (Tb)in[t];
}
template <typename Ta, typename Tb>
void launch_convert(const Ta* in, Tb* out, long long n, cudaStream_t s) {
  long long blocks = (n + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  if (blocks < 1) blocks = 1;
  count_launch(); convert_kernel<Ta, Tb><<<(unsigned)blocks, 256, 0, s>>>(in, out, n);
}
template void launch_convert<double, float>(const double*, float*, long long, cudaStream_t);
template void launch_convert<float, double>(const float*, double*, long long, cudaStream_t);

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Block-level sum of two values in fixed order; result valid in thread 0.
__device__ __forceinline__ void block_sum2(double& a, double& b) {
  __shared__ double sa[32], sb[32];
  a = warp_sum(a);
  b = warp_sum(b);
  int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) { sa[w] = a; sb[w] = b; }
  __syncthreads();
  if (w == 0) {
    int nw = blockDim.x >> 5;
    a = l < nw ? sa[l] : 0.0;
    b = l < nw ? sb[l] : 0.0;
    a = warp_sum(a);
    b = warp_sum(b);
  }
}

// Final reduction of the per-block partials by the last block; out[0..1].  True in that block.
__device__ bool finish_reduce(double a, double b, double* partial, unsigned* counter, double* out,
                              int* status, int check) {
  if (gridDim.x == 1) {                    // one block: its sums are final
    if (threadIdx.x == 0) {
      out[0] = a;
      out[1] = b;
      if (check && status && *status == 0 && !(a == a && a < 1e300)) *status = PMG_ENAN;
    }
    return true;
  }
  __shared__ bool last;
  if (threadIdx.x == 0) {
    partial[2 * blockIdx.x] = a;
    partial[2 * blockIdx.x + 1] = b;
    __threadfence();
    unsigned prev = atomicAdd(counter, 1u);
    last = (prev == gridDim.x - 1);
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double sa = 0.0, sb = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) {
    sa += ((volatile double*)partial)[2 * i];
    sb += ((volatile double*)partial)[2 * i + 1];
  }
  block_sum2(sa, sb);
  if (threadIdx.x == 0) {
    out[0] = sa;
    out[1] = sb;
    if (check && status && *status == 0 && !(sa == sa && sa < 1e300)) *status = PMG_ENAN;
    *counter = 0u;
  }
  return true;
}

// fp32 <-> FP64 without the FP64 pipe (a conversion takes a multiply-add's slot there, and the
// kernels below are bound by that pipe: dot of an fp32 z with two vectors at 161 M values 0.88
// -> 0.64 ms); subnormal and overflowing values take the conversion.
__device__ __forceinline__ double to_double(double x) { return x; }
__device__ __forceinline__ double to_double(float x) {
  const unsigned u = __float_as_uint(x);
  return (u & 0x7f800000u) == 0u && (u << 1) != 0u ? (double)x : widen(x);
}
template <typename T>
__device__ __forceinline__ T from_double(double x) {
  if constexpr (sizeof(T) == 8) {
    return x;
  } else {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)(b >> 52) & 0x7ff;
    if (e < 897 || e > 1150) return (float)x;
    // rebias, then round to nearest even at bit 29 (a carry runs into the exponent)
    const unsigned long long r = (b & 0x7fffffffffffffffull) - (896ull << 52);
    const unsigned v = (unsigned)((r + 0x0fffffffull + ((r >> 29) & 1ull)) >> 29);
    return __uint_as_float(v | ((unsigned)(b >> 32) & 0x80000000u));
  }
}

// V consecutive values as one load or store (V = 2: 16 bytes of doubles, 8 of floats), as doubles.
template <int V, typename T>
__device__ __forceinline__ void load_v(const T* p, long long t, double (&x)[V]) {
  if constexpr (V == 1) {
    x[0] = to_double(p[t]);
  } else {
    using P = std::conditional_t<sizeof(T) == 8, double2, float2>;
    const P v = reinterpret_cast<const P*>(p)[t];
    x[0] = to_double(v.x);
    x[1] = to_double(v.y);
  }
}
template <int V, typename T>
__device__ __forceinline__ void store_v(T* p, long long t, const double (&x)[V]) {
  if constexpr (V == 1) {
    p[t] = from_double<T>(x[0]);
  } else {
    using P = std::conditional_t<sizeof(T) == 8, double2, float2>;
    P v;
    v.x = from_double<T>(x[0]);
    v.y = from_double<T>(x[1]);
    reinterpret_cast<P*>(p)[t] = v;
  }
}
// pairs need segments of even length (each then starts on 16 bytes) and aligned vectors;
// the caller's u may start anywhere on 8 bytes
static bool pairs_ok(long long n, const void* u = nullptr) {
  return n % 2 == 0 && (reinterpret_cast<uintptr_t>(u) & 15) == 0;
}

// The CG vector kernels below run on `k` segments at once (one per right-hand side of
// the hierarchy; vectors hold the segments back to back, n entries each): grid.y = k,
// segment s = blockIdx.y with its own scalars (scal + s S_NUM), reduction partials
// (partial + s kPartialStride, counter + s) and control words (ctrl + kCtrlSeg + 4 s).
// A segment whose solve has finished (its active word is 0) is left untouched.
__device__ __forceinline__ int* seg_ctrl(int* ctrl, int s) { return ctrl + kCtrlSeg + 4 * s; }
__device__ __forceinline__ bool seg_active(const int* ctrl, int s) {
  return ctrl == nullptr || ctrl[kCtrlSeg + 4 * s + C_ACTIVE] != 0;
}

// out[0] = x.y ; out[1] = x.y2 (y2 may be null -> 0), per segment (out + s S_NUM)
template <typename TX, int V>
__global__ void __launch_bounds__(256) dot_kernel(const TX* __restrict__ x, const double* __restrict__ y,
                           const double* __restrict__ y2, long long n, double* partial,
                           unsigned* counter, double* out) {
  const long long o = (long long)blockIdx.y * n / V;
  double a = 0.0, b = 0.0;
  auto add = [&](auto two) {
#pragma unroll 4
    for (long long t = blockIdx.x * 256ll + threadIdx.x; t < n / V; t += (long long)gridDim.x * 256) {
      double xv[V], yv[V], wv[V];
      load_v<V>(x, o + t, xv);
      load_v<V>(y, o + t, yv);
      if constexpr (two()) load_v<V>(y2, o + t, wv);
#pragma unroll
      for (int k = 0; k < V; ++k) {
        a = fma(xv[k], yv[k], a);
        if constexpr (two()) b = fma(xv[k], wv[k], b);
      }
    }
  };
  if (y2) add(std::true_type{});
  else add(std::false_type{});
  block_sum2(a, b);
  finish_reduce(a, b, partial + blockIdx.y * kPartialStride, counter + blockIdx.y, out + blockIdx.y * S_NUM,
                nullptr, 0);
}

template <typename TX>
void launch_dot(const TX* x, const double* y, const double* y2, long long n, int k, double* partial,
                unsigned* counter, double* out, int nblocks, cudaStream_t s) {
  count_launch();
  auto fn = pairs_ok(n) ? dot_kernel<TX, 2> : dot_kernel<TX, 1>;
  fn<<<dim3(nblocks, k), 256, 0, s>>>(x, y, y2, n, partial, counter, out);
}
template void launch_dot<double>(const double*, const double*, const double*, long long, int, double*, unsigned*,
                                 double*, int, cudaStream_t);
template void launch_dot<float>(const float*, const double*, const double*, long long, int, double*, unsigned*,
                                double*, int, cudaStream_t);

// p = z + beta p.  beta = z.(r - r_old) / delta_old (reading C8); since r = r_old - alpha q with
// alpha = delta_old / p.q, that is -(z.q) / (p.q) with the q and p.q of the last iteration, so
// no copy of r_old is kept.  Iteration 1 sets the first direction p = z; in iteration 2
// Algorithm 2 still has r_old = 0: beta = z.r / delta_old (Fletcher-Reeves).
template <typename TZ, int V>
__global__ void __launch_bounds__(256) p_update_kernel(double* __restrict__ p, const TZ* __restrict__ z,
                                const double* __restrict__ scal_all, long long n, const int* ctrl) {
  const int sg = blockIdx.y;
  if (!seg_active(ctrl, sg)) return;
  const double* scal = scal_all + sg * S_NUM;
  const int it = ctrl[C_ITER];
  const double beta = it == 2 ? scal[S_ZR] / scal[S_DELTA] : -scal[S_ZQ] / scal[S_PQ];
  const long long o = (long long)sg * n / V;
  auto run = [&](auto first) {
#pragma unroll 4
    for (long long t = blockIdx.x * 256ll + threadIdx.x; t < n / V; t += (long long)gridDim.x * 256) {
      double zv[V], pv[V];
      load_v<V>(z, o + t, zv);
      if constexpr (!first()) {
        load_v<V>(p, o + t, pv);
#pragma unroll
        for (int k = 0; k < V; ++k) zv[k] = fma(beta, pv[k], zv[k]);
      }
      store_v<V>(p, o + t, zv);
    }
  };
  if (it == 1) run(std::true_type{});
  else run(std::false_type{});
}

template <typename TZ>
void launch_p_update(double* p, const TZ* z, const double* scal, long long n, int k, cudaStream_t s,
                     const int* ctrl) {
  long long blocks = (n + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  count_launch();
  auto fn = pairs_ok(n) ? p_update_kernel<TZ, 2> : p_update_kernel<TZ, 1>;
  fn<<<dim3((unsigned)blocks, k), 256, 0, s>>>(p, z, scal, n, ctrl);
}
template void launch_p_update<double>(double*, const double*, const double*, long long, int, cudaStream_t, const int*);
template void launch_p_update<float>(double*, const float*, const double*, long long, int, cudaStream_t, const int*);

// MGCG control (Algorithm 2 with the convergence tests on the device), for k segments:
// ctrl[C_ITER] = current iteration, ctrl[C_ACTIVE] = segments still iterating; per
// segment its status word, iterations, result and active flag.  Host-driven solves
// read the control words after each iteration; a captured solve's loop is a graph
// `while` node whose condition these kernels set (GRAPH).
template <bool GRAPH>
__global__ void solve_begin_kernel(double* scal_all, int* ctrl, double* hist, int hstride, int k,
                                   cudaGraphConditionalHandle cond) {
  if (threadIdx.x != 0) return;
  int active = 0;
  for (int sg = 0; sg < k; ++sg) {
    double* scal = scal_all + sg * S_NUM;
    int* c = seg_ctrl(ctrl, sg);
    const double rr0 = scal[S_RR0];
    const double r0 = sqrt(rr0);
    hist[sg * hstride] = r0;
    scal[S_RR] = rr0;
    const bool go = (r0 == r0) && r0 != 0.0;
    c[C_ACTIVE] = go ? 1 : 0;
    c[C_ITER] = 0;
    c[C_RES] = (r0 == r0) ? (go ? PMG_ENOCONV : PMG_OK) : PMG_ENAN;
    active += go;
  }
  ctrl[C_ITER] = active ? 1 : 0;
  ctrl[C_ACTIVE] = active;
  if constexpr (GRAPH) cudaGraphSetConditional(cond, active ? 1u : 0u);
}

// After iteration ctrl[C_ITER]: record every active segment's ||r||; a segment stops on
// the global status word (a failure of a kernel shared by all segments), on its own
// status word, on ||r|| <= rtol ||r_0|| or at max_iter; the loop goes on while any
// segment is active.  One thread; the segments' words come from other SMs (volatile).
template <bool GRAPH>
__device__ void solve_control(const double* scal_all, int* ctrl_all, double* hist, int hstride, int k, double rtol,
                              int max_iter, cudaGraphConditionalHandle cond) {
  volatile int* ctrl = ctrl_all;
  const int it = ctrl[C_ITER];
  int active = 0;
  for (int sg = 0; sg < k; ++sg) {
    volatile int* c = ctrl + kCtrlSeg + 4 * sg;
    if (!c[C_ACTIVE]) continue;
    const volatile double* scal = scal_all + sg * S_NUM;
    const double rn = sqrt(scal[S_RR]);
    const double r0 = sqrt(scal[S_RR0]);
    hist[sg * hstride + it] = rn;
    c[C_ITER] = it;
    int res = 1;
    if (ctrl[C_STATUS] != 0) res = ctrl[C_STATUS];
    else if (c[C_STATUS] != 0) res = c[C_STATUS];
    else if (rn <= rtol * r0) res = PMG_OK;
    else if (it >= max_iter) res = PMG_ENOCONV;
    if (res != 1) {
      c[C_RES] = res;
      c[C_ACTIVE] = 0;
    } else {
      ++active;
    }
  }
  ctrl[C_ACTIVE] = active;
  if (active) ctrl[C_ITER] = it + 1;
  if constexpr (GRAPH) cudaGraphSetConditional(cond, active ? 1u : 0u);
}

// alpha = z.r / (p.q); u += alpha p; r -= alpha q (also rounded into r32, the next V-cycle's
// right-hand side, where the V-cycle is fp32); S_RR = r.r, S_DELTA = z.r.  The block that
// finishes last over all segments then runs the stopping tests (solve_control): one launch
// for what took four (set delta, update, conversion, control).
template <bool GRAPH, int V>
__global__ void __launch_bounds__(256)
cg_update_kernel(double* __restrict__ u, double* __restrict__ r, float* __restrict__ r32,
                 const double* __restrict__ p, const double* __restrict__ q, double* scal_all, long long n, int k,
                 double* partial, unsigned* counter, int* ctrl, double* hist, int hstride, double rtol, int max_iter,
                 cudaGraphConditionalHandle cond) {
  const int sg = blockIdx.y;
  unsigned* done = counter + k;                      // segments finished in this launch
  auto finish = [&] {                                // thread 0 of a segment's last block
    if (k > 1) {
      __threadfence();
      if (atomicAdd(done, 1u) != (unsigned)k - 1u) return;
      *done = 0u;
      __threadfence();
    }
    solve_control<GRAPH>(scal_all, ctrl, hist, hstride, k, rtol, max_iter, cond);
  };
  if (!seg_active(ctrl, sg)) {                      // uniform over the segment's blocks
    if (blockIdx.x == 0 && threadIdx.x == 0) finish();
    return;
  }
  double* scal = scal_all + sg * S_NUM;
  int* status = seg_ctrl(ctrl, sg) + C_STATUS;
  const double pq = scal[S_PQ], zr = scal[S_ZR];
  const double alpha = zr / pq;
  if (blockIdx.x == 0 && threadIdx.x == 0 && *status == 0) {             // the first status stays
    if (!(zr > 0.0)) *status = (zr == zr) ? PMG_EBREAKDOWN : PMG_ENAN;
    else if (!(pq > 0.0)) *status = (pq == pq) ? PMG_EBREAKDOWN : PMG_ENAN;
  }
  const long long o = (long long)sg * n / V;
  double a = 0.0, b = 0.0;
#pragma unroll 2
  for (long long t = blockIdx.x * 256ll + threadIdx.x; t < n / V; t += (long long)gridDim.x * 256) {
    double uv[V], pv[V], qv[V], rv[V];
    load_v<V>(u, o + t, uv);
    load_v<V>(p, o + t, pv);
    load_v<V>(q, o + t, qv);
    load_v<V>(r, o + t, rv);
#pragma unroll
    for (int k = 0; k < V; ++k) {
      uv[k] = fma(alpha, pv[k], uv[k]);
      rv[k] = fma(-alpha, qv[k], rv[k]);
      a = fma(rv[k], rv[k], a);
    }
    store_v<V>(u, o + t, uv);
    store_v<V>(r, o + t, rv);
    if (r32) store_v<V>(r32, o + t, rv);
  }
  block_sum2(a, b);
  if (finish_reduce(a, b, partial + sg * kPartialStride, counter + sg, scal + S_RR, status, 1) && threadIdx.x == 0) {
    scal[S_DELTA] = zr;
    finish();
  }
}

void launch_cg_update(double* u, double* r, float* r32, const double* p, const double* q, double* scal, long long n,
                      int k, double* partial, unsigned* counter, int* ctrl, int nblocks, double* hist, int hstride,
                      double rtol, int max_iter, const cudaGraphConditionalHandle* cond, cudaStream_t s) {
  count_launch();
  const bool v2 = pairs_ok(n, u);
  auto fn = cond ? (v2 ? cg_update_kernel<true, 2> : cg_update_kernel<true, 1>)
                 : (v2 ? cg_update_kernel<false, 2> : cg_update_kernel<false, 1>);
  fn<<<dim3(nblocks, k), 256, 0, s>>>(u, r, r32, p, q, scal, n, k, partial, counter, ctrl, hist, hstride, rtol,
                                      max_iter, cond ? *cond : cudaGraphConditionalHandle{});
}

__global__ void solve_result_kernel(const double* scal_all, const int* ctrl, SolveResult* out, int k) {
  for (int sg = threadIdx.x; sg < k; sg += blockDim.x) {
    const double* scal = scal_all + sg * S_NUM;
    const int* c = ctrl + kCtrlSeg + 4 * sg;
    out[sg].r0 = sqrt(scal[S_RR0]);
    out[sg].rn = sqrt(scal[S_RR]);
    out[sg].iterations = c[C_ITER];
    out[sg].status = c[C_RES];
  }
}

void launch_solve_result(const double* scal, const int* ctrl, SolveResult* out, int k, cudaStream_t s) {
  count_launch(); solve_result_kernel<<<1, 32, 0, s>>>(scal, ctrl, out, k);
}

void launch_solve_begin(double* scal, int* ctrl, double* hist, int hstride, int k, const cudaGraphConditionalHandle* cond,
                        cudaStream_t s) {
  count_launch();
  if (cond) solve_begin_kernel<true><<<1, 1, 0, s>>>(scal, ctrl, hist, hstride, k, *cond);
  else solve_begin_kernel<false><<<1, 1, 0, s>>>(scal, ctrl, hist, hstride, k, cudaGraphConditionalHandle{});
}
// x -= mean(x)   (projection onto range(A) for periodic grids)
__global__ void sum_kernel(const double* __restrict__ x, long long n, double* partial,
                           unsigned* counter, double* out) {
  double a = 0.0, b = 0.0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    a += x[t];
  block_sum2(a, b);
  finish_reduce(a, b, partial, counter, out, nullptr, 0);
}
__global__ void sub_kernel(double* __restrict__ x, long long n, const double* __restrict__ sum) {
  const double m = sum[0] / (double)n;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    x[t] -= m;
}
void launch_sub_mean(double* x, long long n, double* partial, unsigned* counter, double* scal,
                     int nblocks, cudaStream_t s) {
  count_launch(); sum_kernel<<<nblocks, 256, 0, s>>>(x, n, partial, counter, scal + S_MEAN);
  long long blocks = (n + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  count_launch(); sub_kernel<<<(unsigned)blocks, 256, 0, s>>>(x, n, scal + S_MEAN);
}

}  // namespace pmg
