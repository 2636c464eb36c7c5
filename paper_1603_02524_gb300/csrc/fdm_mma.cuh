// Schwarz patch solve (Sec. 3.1) in fp32 with the six line passes on the tensor cores.
//
// Every fp32 operand is cut exactly into three bf16 terms of eight bits (x = x0 + x1 + x2,
// two truncations and two exact subtractions); the products x_i t_j with i + j <= 2 are six
// bf16 MMAs with fp32 accumulation, which keeps fp32 accuracy (the terms left out are below
// 2^-24 of a product).  Against the SIMT passes this removes the table reads: a thread of
// those reads every row of the table from shared memory for each of its lines, 16 bytes for
// four multiply-adds, and that traffic was their bound.  Here the table fragments stay in
// registers for all the tiles of a pass.
//
// Precision: the tensor core rounds its sums toward zero; the tables carry the mean of that
// (bf16_fragments), and each output is rounded once at full scale (inputs beyond 16 go to a
// second accumulator).  A sweep's error against FP64 is 7-9e-8 of its norm, the SIMT passes'
// 1.3-1.5e-7.
//
// What bounds it: instruction issue (73 % at 13^3; tensor pipe 26 %).  Sweeps, SIMT -> here: EA
// at 16^3 elements P = 16 548 -> 428 us, P = 8 87 -> 75; FA 16 x 13 x 13 at 64 x 16 x 8 elements
// 230 -> 150 us; 2-D 40 x 40 P = 16 56 -> 18 us, 64 x 48 P = 8 27 -> 11 us.
//
// One CTA per patch, the patch in shared memory; every pass works in place on tiles of eight
// lines per warp (as in fdm_split.cuh: a lane loads four inputs of one line and holds two
// outputs of two lines).
#pragma once

#include "fdm_kernel.cuh"
#include "split.cuh"

namespace pmg {

template <int NA, int NB, int NC>
struct MmaShape {
  static constexpr int NN = NA * NB * NC;
  static constexpr int NOFF = NA + NB + NC;
  static constexpr size_t ROW = 8 * (size_t)NOFF;                            // after off[NOFF]
  static constexpr size_t LAM = ROW + 8 * (size_t)(NB * NC);
  static constexpr size_t BUF = LAM + 4 * (size_t)NOFF;
  static constexpr size_t BYTES = BUF + 4 * (size_t)NN;
  static constexpr int THREADS = patch_threads(NA, NB, NC);
  static constexpr int MINB = (NA > 16 || NB > 16 ? 768 : 1024) / THREADS;   // 80 or 64 registers per thread
};

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// the three bf16 terms of two values, packed
__device__ __forceinline__ void bf16_terms(float x, float y, uint32_t (&b)[3]) {
  b[0] = __byte_perm(__float_as_uint(x), __float_as_uint(y), 0x7632);
  const float x1 = x - __uint_as_float(__float_as_uint(x) & 0xffff0000u);
  const float y1 = y - __uint_as_float(__float_as_uint(y) & 0xffff0000u);
  b[1] = __byte_perm(__float_as_uint(x1), __float_as_uint(y1), 0x7632);
  const float x2 = x1 - __uint_as_float(__float_as_uint(x1) & 0xffff0000u);
  const float y2 = y1 - __uint_as_float(__float_as_uint(y1) & 0xffff0000u);
  b[2] = __byte_perm(__float_as_uint(x2), __float_as_uint(y2), 0x7632);
}

// acc += table x line, smallest terms first
__device__ __forceinline__ void bf16_mma(float (&acc)[4], const uint4 (&A)[3], const uint32_t (&b0)[3],
                                         const uint32_t (&b1)[3]) {
#pragma unroll
  for (int w = 2; w >= 0; --w)
#pragma unroll
    for (int i = w; i >= 0; --i) mma_bf16(acc, A[w - i], b0[i], b1[i]);
}

__device__ __forceinline__ void load_terms(uint4 (&A)[3], const uint4* __restrict__ frag) {
#pragma unroll
  for (int j = 0; j < 3; ++j) A[j] = __ldg(frag + j * 32);
}

// One in-place pass along an axis of N nodes, line l at base(l), nodes `stride` apart; scale(l)
// gives the functor applied to (output, value) of line l.
template <int N, bool FORWARD, typename Base, typename Scale>
__device__ __forceinline__ void mma_pass(bool fold, const uint4* __restrict__ frag, float* buf, int nlines, int stride,
                                         Base&& base, Scale&& scale) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int ntiles = (nlines + 7) >> 3;
  frag += lane;
  if constexpr (N <= 16) {
    uint4 A[3];
    load_terms(A, frag);
#pragma unroll 1
    for (int tile = warp; tile < ntiles; tile += nwarps) {
      const int o = base(min(tile * 8 + g, nlines - 1)) + t * stride;
      const int l0 = tile * 8 + 2 * t;
      auto val = [&](int s) { return t + 4 * s < N ? buf[o + 4 * s * stride] : 0.0f; };
      uint32_t b0[3], b1[3] = {};
      bf16_terms(val(0), N > 4 ? val(1) : 0.0f, b0);
      if constexpr (N > 8) bf16_terms(val(2), N > 12 ? val(3) : 0.0f, b1);
      float acc[4] = {};
      bf16_mma(acc, A, b0, b1);
      __syncwarp();
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const bool on = l0 + c < nlines;
        float* p = buf + base(l0 + c) + g * stride;
        auto f = scale(l0 + c);
        if (on && (N >= 8 || g < N)) p[0] = f(g, acc[c]);
        if (N > 8 && on && g + 8 < N) p[8 * stride] = f(g + 8, acc[2 + c]);
      }
      __syncwarp();
    }
  } else if (fold) {
    constexpr int H = N / 2, NE = N - H, NO = H;
    uint4 Ae[3], Ao[3];
    load_terms(Ae, frag);
    load_terms(Ao, frag + 3 * 32);
#pragma unroll 1
    for (int tile = warp; tile < ntiles; tile += nwarps) {
      const int o = base(min(tile * 8 + g, nlines - 1));
      const int l0 = tile * 8 + 2 * t;
      float Xe[4], Xo[4];
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const int a = t + 4 * s;
        if constexpr (FORWARD) {
          const float v = a < NE ? buf[o + a * stride] : 0.0f;
          const float w = a < H ? buf[o + (N - 1 - a) * stride] : 0.0f;
          Xe[s] = v + w;
          Xo[s] = a < H ? v - w : 0.0f;
        } else {
          Xe[s] = a < NE ? buf[o + a * stride] : 0.0f;
          Xo[s] = a < NO ? buf[o + (NE + a) * stride] : 0.0f;
        }
      }
      // up to 12 rows per block: the third rows of both blocks share a register (the
      // antisymmetric table has its third rows in the fourth slots)
      uint32_t be[3], bo[3], b2[3], b3[3];
      bf16_terms(Xe[0], Xe[1], be);
      bf16_terms(Xo[0], Xo[1], bo);
      if constexpr (NE <= 12) {
        bf16_terms(Xe[2], Xo[2], b2);
      } else {
        bf16_terms(Xe[2], Xe[3], b2);
        bf16_terms(Xo[2], Xo[3], b3);
      }
      float e[4] = {}, d[4] = {};
      bf16_mma(e, Ae, be, b2);
      bf16_mma(d, Ao, bo, NE <= 12 ? b2 : b3);
      __syncwarp();
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const bool on = l0 + c < nlines;
        const int oo = base(l0 + c);
        auto f = scale(l0 + c);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int out = g + 8 * r;
          const float x = e[2 * r + c], y = d[2 * r + c];
          const bool in = on && (8 * r + 7 < NO || out < NO);             // both blocks
          const bool mid = on && NE > H && (8 * r <= H && H < 8 * r + 8) && out == H;
          if constexpr (FORWARD) {
            if (in || mid) buf[oo + out * stride] = f(out, x);
            if (in) buf[oo + (NE + out) * stride] = f(NE + out, y);
          } else {
            if (in || mid) buf[oo + out * stride] = f(out, mid ? x : x + y);
            if (in) buf[oo + (N - 1 - out) * stride] = f(N - 1 - out, x - y);
          }
        }
      }
      __syncwarp();
    }
  } else {
#pragma unroll 1
    for (int tile = warp; tile < ntiles; tile += nwarps) {
      const int o = base(min(tile * 8 + g, nlines - 1)) + t * stride;
      const int l0 = tile * 8 + 2 * t;
      auto val = [&](int s) { return t + 4 * s < N ? buf[o + 4 * s * stride] : 0.0f; };
      uint32_t b[4][3] = {};
      bf16_terms(val(0), val(1), b[0]);
      bf16_terms(val(2), val(3), b[1]);
      bf16_terms(val(4), val(5), b[2]);
      if constexpr (N > 24) bf16_terms(val(6), val(7), b[3]);
      __syncwarp();
#pragma unroll
      for (int mt = 0; mt < 2; ++mt) {
        // the two halves of the inputs apart: the tensor core rounds toward zero once each
        float x[4] = {}, y[4] = {};
        uint4 A[3];
        load_terms(A, frag + mt * 2 * 3 * 32);
        bf16_mma(x, A, b[0], b[1]);
        load_terms(A, frag + (mt * 2 + 1) * 3 * 32);
        bf16_mma(y, A, b[2], b[3]);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const bool on = l0 + c < nlines;
          auto f = scale(l0 + c);
          const int out = mt * 16 + g;
          float* p = buf + base(l0 + c) + out * stride;
          if (on && out < N) p[0] = f(out, x[c] + y[c]);
          if (on && out + 8 < N) p[8 * stride] = f(out + 8, x[2 + c] + y[2 + c]);
        }
      }
      __syncwarp();
    }
  }
}

template <int NA, int NB, int NC>
__global__ void __launch_bounds__(MmaShape<NA, NB, NC>::THREADS, MmaShape<NA, NB, NC>::MINB)
fdm_kernel_mma(FdmFamily<float> fam, const float* __restrict__ r, float* __restrict__ u) {
  using MS = MmaShape<NA, NB, NC>;
  constexpr int NN = MS::NN;
  extern __shared__ __align__(16) unsigned char mm_smem[];
  long long* off = reinterpret_cast<long long*>(mm_smem);
  long long* rowoff = reinterpret_cast<long long*>(mm_smem + MS::ROW);
  float* la = reinterpret_cast<float*>(mm_smem + MS::LAM);
  float* lb = la + NA;
  float* lc = lb + NB;
  float* buf = reinterpret_cast<float*>(mm_smem + MS::BUF);
  const int tid = threadIdx.x, nt = blockDim.x;
  const int pidx[3] = {(int)blockIdx.x, (int)blockIdx.y, (int)blockIdx.z};
  const int nq[3] = {NA, NB, NC};
  bool fold[3] = {};
  const uint4 *Ff[3] = {}, *Fb[3] = {};
  float* lq[3] = {la, lb, lc};
  long long* offq[3] = {off, off + NA, off + NA + NB};
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const FdmAxis<float>& ax = fam.ax[q];
    const int n = nq[q];
    const size_t p = pidx[q];
    if (q < 2 || NC > 1) {
      const int tab = __ldg(ax.fid + p);
      fold[q] = n > 16 && __ldg(ax.sym + p) != 0;
      const size_t len = (size_t)split_blocks(n) * 3 * 32;
      Ff[q] = ax.SF + tab * len;
      Fb[q] = ax.WF + tab * len;
    }
    for (int a = tid; a < n; a += nt) {
      lq[q][a] = ax.lam[p * n + a];
      offq[q][a] = __ldg(ax.goff + p * n + a);
    }
  }
  __syncthreads();
  for (int rr = tid; rr < NB * NC; rr += nt) rowoff[rr] = off[NA + rr % NB] + off[NA + NB + rr / NB];
  __syncthreads();
  const PatchRows<NA> rows(off);
  rows.template gather<NB * NC, 8>(r, rowoff, [&](int t, float v) { buf[t] = v; });
  __syncthreads();
  auto base_a = [](int l) { return l * NA; };
  auto base_b = [](int l) { return l % NA + (l / NA) * (NA * NB); };
  [[maybe_unused]] auto base_c = [](int l) { return l; };
  auto plain = [](int) { return [](int, float v) { return v; }; };
  // the last forward pass multiplies by 1 / (lambda_a + lambda_b + lambda_c)
  mma_pass<NA, true>(fold[0], Ff[0], buf, NB * NC, 1, base_a, plain);
  __syncthreads();
  if constexpr (NC > 1) {
    mma_pass<NB, true>(fold[1], Ff[1], buf, NA * NC, NA, base_b, plain);
    __syncthreads();
    mma_pass<NC, true>(fold[2], Ff[2], buf, NA * NB, NA * NB, base_c, [&](int l) {
      const float s = la[l % NA] + lb[l / NA];
      return [s, lc](int o, float v) { return v * recip(s + lc[o]); };
    });
    __syncthreads();
    mma_pass<NC, false>(fold[2], Fb[2], buf, NA * NB, NA * NB, base_c, plain);
  } else {
    mma_pass<NB, true>(fold[1], Ff[1], buf, NA, NA, base_b, [&](int l) {
      const float s = la[l] + lc[0];
      return [s, lb](int o, float v) { return v * recip(s + lb[o]); };
    });
  }
  __syncthreads();
  mma_pass<NB, false>(fold[1], Fb[1], buf, NA * NC, NA, base_b, plain);
  __syncthreads();
  mma_pass<NA, false>(fold[0], Fb[0], buf, NB * NC, 1, base_a, plain);
  __syncthreads();
  rows.template scatter<NB * NC>(u, rowoff, [&](int t, int) { return buf[t]; });
}

template <int NA, int NB, int NC>
int fdm_launch_mma(const FdmFamily<float>& fam, const float* r, float* u, cudaStream_t s) {
  using MS = MmaShape<NA, NB, NC>;
  static_assert(MS::BYTES <= 227 * 1024, "patch does not fit in shared memory");
  if (MS::BYTES > 48 * 1024 &&
      cudaFuncSetAttribute(fdm_kernel_mma<NA, NB, NC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)MS::BYTES) != cudaSuccess)
    return PMG_ECUDA;
  if (fam.count_total <= 0) return PMG_OK;
  // any whole number of warps up to the default works (the tuner times them)
  int threads = (fam.threads >= 32 && fam.threads % 32 == 0) ? fam.threads : MS::THREADS;
  if (threads > MS::THREADS) threads = MS::THREADS;
  count_launch();
  fdm_kernel_mma<NA, NB, NC><<<patch_grid(fam), threads, MS::BYTES, s>>>(fam, r, u);
  return cudaGetLastError() == cudaSuccess ? PMG_OK : PMG_ECUDA;
}

// ---------------------------------------------------------------------------
// P = 32 patches (33 to 64 nodes per axis, up to 473 KB) in slabs of c-planes, three kernels per
// group of patches: the forward a and b passes of a slab run in shared memory and leave its
// planes in a scratch buffer; the c-lines, both passes, in registers; the backward b and a
// passes of a slab and the scatter.  One CTA per slab (not per patch) fills the chip where a
// level has as many patches as SMs; the groups keep their scratch planes in L2.
//
// c-lines: sixteen lines are the first operand of an MMA, whose sums (lines x modes), scaled by
// the inverse eigenvalue sums and cut again, are the first operand of the backward product.
//
// The table fragments (up to 24 KB) do not fit the registers; a warp applies each to two tiles
// of eight lines (or one of sixteen), 12 wavefronts of the load unit for 12 MMAs.
//
// What bounds it: the fragments' loads and the MMAs' issue at 16 warps of 128 registers.  The
// SIMT kernel it replaces (one persistent CTA per patch) was bound by latency, issue 22 %: a
// 64 x 43 x 43 sweep of 160 patches 840 -> 306 us (109 forward, 70 c-lines, 127 backward), the
// error against FP64 2.2e-7 -> 1.0e-7 of the norm.  The same passes with one CTA per patch
// took 644 us: eight warps on most SMs, the second patch of the others behind them.
// ---------------------------------------------------------------------------
template <int NA, int NB, int NC>
struct SlabMmaShape {
  static constexpr int THREADS = 256, MINB = 2;              // 128 registers per thread
  static constexpr int CS = 5;                               // planes per slab
  static constexpr int SLABS = (NC + CS - 1) / CS;
  static constexpr int NAP = (NA + 3) / 8 * 8 + 4;           // rows 4 banks (mod 8) apart: a-lines without conflicts
  static constexpr int PL = NB * NAP;                        // a padded plane
  static constexpr int PS = (NA * NB + 7) / 8 * 8;           // a plane of the scratch buffer
  static constexpr int TILES = (NA * NB + 15) / 16;          // of c-lines
  static constexpr size_t ROW = 8 * (size_t)(NA + NB + CS);  // after off[NA + NB + CS]
  static constexpr size_t BUF = ROW + 8 * (size_t)(CS * NB);
  static constexpr size_t BYTES = BUF + 4 * (size_t)CS * PL;
  static_assert(NAP >= NA && NA <= 64 && NB <= 64 && NC <= 48, "slab shape");
};

// One in-place pass over lines of N > 32 nodes in shared memory, sixteen lines per warp.
template <int N, typename Base>
__device__ __forceinline__ void mma_pass_long(const uint4* __restrict__ frag, float* buf, int nlines, int stride,
                                              Base&& base) {
  constexpr int KT = (N + 15) / 16;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  frag += lane;
#pragma unroll 1
  for (int tile = warp; tile < (nlines + 15) >> 4; tile += nwarps) {
    uint32_t b[2][KT][2][3];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float* p = buf + base(min(tile * 16 + h * 8 + g, nlines - 1)) + t * stride;
#pragma unroll
      for (int kt = 0; kt < KT; ++kt) {
        auto val = [&](int s) { return t + 4 * s + 16 * kt < N ? p[(4 * s + 16 * kt) * stride] : 0.0f; };
        bf16_terms(val(0), val(1), b[h][kt][0]);
        bf16_terms(val(2), val(3), b[h][kt][1]);
      }
    }
    __syncwarp();
#pragma unroll 1
    for (int mt = 0; mt < KT; ++mt) {
      float sum[2][4] = {};
#pragma unroll
      for (int kt = 0; kt < KT; ++kt) {
        // every 16 inputs apart: the tensor core rounds toward zero once each
        uint4 A[3];
        load_terms(A, frag + (mt * KT + kt) * 3 * 32);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float acc[4] = {};
          bf16_mma(acc, A, b[h][kt][0], b[h][kt][1]);
#pragma unroll
          for (int r = 0; r < 4; ++r) sum[h][r] += acc[r];
        }
      }
      const int out = mt * 16 + g;
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int l = tile * 16 + h * 8 + 2 * t + c;
          if (l < nlines) {
            float* p = buf + base(l) + out * stride;
            if (out < N) p[0] = sum[h][c];
            if (out + 8 < N) p[8 * stride] = sum[h][2 + c];
          }
        }
    }
    __syncwarp();
  }
}

// x (sixteen lines x inputs, as bf16 terms) times a table with B-form fragments
template <int KT>
__device__ __forceinline__ void mma_lines(float (&y)[2 * KT][4], const uint4 (&x)[KT][3], const uint4* __restrict__ frag) {
#pragma unroll
  for (int ot = 0; ot < KT; ++ot) {
#pragma unroll
    for (int kt = 0; kt < KT; ++kt) {
      uint4 B[3];
      load_terms(B, frag + (kt * KT + ot) * 3 * 32);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float acc[4] = {};
#pragma unroll
        for (int w = 2; w >= 0; --w)
#pragma unroll
          for (int i = w; i >= 0; --i)
            mma_bf16(acc, x[kt][i], h ? B[w - i].z : B[w - i].x, h ? B[w - i].w : B[w - i].y);
#pragma unroll
        for (int r = 0; r < 4; ++r) y[2 * ot + h][r] = kt ? y[2 * ot + h][r] + acc[r] : acc[r];
      }
    }
  }
}
// the terms of sixteen inputs of lines g and g + 8 in the first operand's layout
__device__ __forceinline__ void line_terms(uint4 (&x)[3], const float (&lo)[4], const float (&hi)[4]) {
  uint32_t b[4][3];
  bf16_terms(lo[0], lo[1], b[0]);
  bf16_terms(lo[2], lo[3], b[1]);
  bf16_terms(hi[0], hi[1], b[2]);
  bf16_terms(hi[2], hi[3], b[3]);
#pragma unroll
  for (int j = 0; j < 3; ++j) x[j] = make_uint4(b[0][j], b[1][j], b[2][j], b[3][j]);
}

struct SlabPatch {
  int p[3];
};
__device__ __forceinline__ SlabPatch slab_patch(const FdmFamily<float>& fam, int pid) {
  const int ca = fam.ax[0].count, cb = fam.ax[1].count;
  return SlabPatch{{pid % ca, (pid / ca) % cb, pid / (ca * cb)}};
}
// fragments of position p of an axis with n nodes
__device__ __forceinline__ size_t slab_table(const FdmAxis<float>& ax, int p, int n) {
  return (size_t)__ldg(ax.fid + p) * split_blocks(n) * 3 * 32;
}

// The a and b passes of slab blockIdx.x of patch first + blockIdx.y: FORWARD gathers r and
// leaves the planes in scratch, backward takes them from there and adds them to u.
template <int NA, int NB, int NC, bool FORWARD>
__global__ void __launch_bounds__(SlabMmaShape<NA, NB, NC>::THREADS, SlabMmaShape<NA, NB, NC>::MINB)
fdm_kernel_slab_mma(FdmFamily<float> fam, int first, const float* __restrict__ r, float* __restrict__ u) {
  using MS = SlabMmaShape<NA, NB, NC>;
  constexpr int NAP = MS::NAP, CS = MS::CS;
  extern __shared__ __align__(16) unsigned char mm_smem[];
  long long* off = reinterpret_cast<long long*>(mm_smem);
  long long* rowoff = reinterpret_cast<long long*>(mm_smem + MS::ROW);
  float* sb = reinterpret_cast<float*>(mm_smem + MS::BUF);              // CS padded planes [k][b][a]
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarps = nt >> 5;
  const SlabPatch sp = slab_patch(fam, first + (int)blockIdx.y);
  const int c0 = (int)blockIdx.x * CS, cs = min(NC - c0, CS), rows = cs * NB;
  float* buf = fam.scratch + (long long)blockIdx.y * fam.scratch_stride + (long long)c0 * MS::PS;
  for (int a = tid; a < NA + NB + cs; a += nt)
    off[a] = a < NA        ? __ldg(fam.ax[0].goff + (size_t)sp.p[0] * NA + a)
             : a < NA + NB ? __ldg(fam.ax[1].goff + (size_t)sp.p[1] * NB + a - NA)
                           : __ldg(fam.ax[2].goff + (size_t)sp.p[2] * NC + c0 + a - NA - NB);
  __syncthreads();
  for (int rr = tid; rr < rows; rr += nt) rowoff[rr] = off[NA + rr % NB] + off[NA + NB + rr / NB];
  __syncthreads();
  auto base_a = [](int l) { return l * NAP; };
  auto base_b = [](int l) { return l % NA + (l / NA) * MS::PL; };
  // a warp takes rows, a lane two columns of them
  const bool on[2] = {lane < NA, lane + 32 < NA};
  const long long oa[2] = {on[0] ? off[lane] : kInvalidOffset, on[1] ? off[lane + 32] : kInvalidOffset};
  auto scratch_row = [&](int row) { return buf + (long long)(row / NB) * MS::PS + row % NB * NA + lane; };
  constexpr int U = 8;
  for (int r0 = warp; r0 < rows; r0 += U * nwarps) {
    float v[U][2];
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int row = min(r0 + j * nwarps, rows - 1);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        if constexpr (FORWARD) {
          const long long o = oa[k] + rowoff[row];
          v[j][k] = o >= 0 ? __ldg(r + o) : 0.0f;
        } else {
          v[j][k] = on[k] ? scratch_row(row)[32 * k] : 0.0f;
        }
      }
    }
#pragma unroll
    for (int j = 0; j < U; ++j)
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (on[k] && r0 + j * nwarps < rows) sb[(r0 + j * nwarps) * NAP + lane + 32 * k] = v[j][k];
  }
  __syncthreads();
  const FdmAxis<float>&ax = fam.ax[0], &bx = fam.ax[1];
  if constexpr (FORWARD) {
    mma_pass_long<NA>(ax.SF + slab_table(ax, sp.p[0], NA), sb, rows, 1, base_a);
    __syncthreads();
    mma_pass_long<NB>(bx.SF + slab_table(bx, sp.p[1], NB), sb, NA * cs, NAP, base_b);
  } else {
    mma_pass_long<NB>(bx.WF + slab_table(bx, sp.p[1], NB), sb, NA * cs, NAP, base_b);
    __syncthreads();
    mma_pass_long<NA>(ax.WF + slab_table(ax, sp.p[0], NA), sb, rows, 1, base_a);
  }
  __syncthreads();
#pragma unroll 4
  for (int row = warp; row < rows; row += nwarps)
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float x = on[k] ? sb[row * NAP + lane + 32 * k] : 0.0f;
      if constexpr (FORWARD) {
        if (on[k]) scratch_row(row)[32 * k] = x;
      } else {
        const long long o = oa[k] + rowoff[row];
        if (o >= 0) atomicAdd(u + o, x);
      }
    }
}

// The c-lines of patch first + blockIdx.y, one tile of sixteen per warp: forward, times
// 1 / (lambda_a + lambda_b + lambda_c), backward.
template <int NA, int NB, int NC>
__global__ void __launch_bounds__(256, 2) fdm_kernel_clines_mma(FdmFamily<float> fam, int first) {
  using MS = SlabMmaShape<NA, NB, NC>;
  constexpr int PS = MS::PS, KT = (NC + 15) / 16;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int tile = (int)blockIdx.x * 8 + (int)(threadIdx.x >> 5);
  if (tile >= MS::TILES) return;
  const SlabPatch sp = slab_patch(fam, first + (int)blockIdx.y);
  float* buf = fam.scratch + (long long)blockIdx.y * fam.scratch_stride;
  const int l0 = tile * 16 + g, l1 = l0 + 8;                 // the lane's lines
  const int m0 = min(l0, NA * NB - 1), m1 = min(l1, NA * NB - 1);
  uint4 x[KT][3];
#pragma unroll
  for (int kt = 0; kt < KT; ++kt) {
    float lo[4], hi[4];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int i = kt * 16 + 2 * t + k, j = i + 8;
      lo[k] = i < NC ? buf[i * PS + m0] : 0.0f;
      lo[2 + k] = i < NC ? buf[i * PS + m1] : 0.0f;
      hi[k] = j < NC ? buf[j * PS + m0] : 0.0f;
      hi[2 + k] = j < NC ? buf[j * PS + m1] : 0.0f;
    }
    line_terms(x[kt], lo, hi);
  }
  const FdmAxis<float>& cx = fam.ax[2];
  const size_t tab = slab_table(cx, sp.p[2], NC) + lane;
  float y[2 * KT][4];
  mma_lines<KT>(y, x, cx.SF + tab);
  const float* la = fam.ax[0].lam + (size_t)sp.p[0] * NA;
  const float* lb = fam.ax[1].lam + (size_t)sp.p[1] * NB;
  const float* lc = cx.lam + (size_t)sp.p[2] * NC;
  const float s0 = __ldg(la + m0 % NA) + __ldg(lb + m0 / NA), s1 = __ldg(la + m1 % NA) + __ldg(lb + m1 / NA);
#pragma unroll
  for (int j = 0; j < 2 * KT; ++j)
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float lk = __ldg(lc + min(j * 8 + 2 * t + k, NC - 1));
      y[j][k] *= recip(s0 + lk);
      y[j][2 + k] *= recip(s1 + lk);
    }
#pragma unroll
  for (int kt = 0; kt < KT; ++kt) line_terms(x[kt], y[2 * kt], y[2 * kt + 1]);
  mma_lines<KT>(y, x, cx.WF + tab);
#pragma unroll
  for (int j = 0; j < 2 * KT; ++j)
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int o = j * 8 + 2 * t + k;
      if (o < NC && l0 < NA * NB) buf[o * PS + l0] = y[j][k];
      if (o < NC && l1 < NA * NB) buf[o * PS + l1] = y[j][2 + k];
    }
}

template <int NA, int NB, int NC>
int fdm_launch_slab_mma(const FdmFamily<float>& fam, const float* r, float* u, cudaStream_t s) {
  using MS = SlabMmaShape<NA, NB, NC>;
  static_assert(MS::BYTES <= 113 * 1024, "two CTAs per SM");
  if (!fam.scratch || fam.scratch_ctas <= 0 || fam.scratch_stride < (long long)MS::PS * NC) return PMG_EINVAL;
  auto fwd = fdm_kernel_slab_mma<NA, NB, NC, true>;
  auto bwd = fdm_kernel_slab_mma<NA, NB, NC, false>;
  for (auto fn : {fwd, bwd})
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MS::BYTES) != cudaSuccess)
      return PMG_ECUDA;
  if (fam.count_total <= 0) return PMG_OK;
  // equal groups of at most scratch_ctas patches (96 MB of planes)
  const int groups = (fam.count_total + fam.scratch_ctas - 1) / fam.scratch_ctas;
  const int per = (fam.count_total + groups - 1) / groups;
  for (int first = 0; first < fam.count_total; first += per) {
    const unsigned n = (unsigned)(fam.count_total - first < per ? fam.count_total - first : per);
    for (int k = 0; k < 3; ++k) count_launch();
    fwd<<<dim3(MS::SLABS, n), MS::THREADS, MS::BYTES, s>>>(fam, first, r, u);
    fdm_kernel_clines_mma<NA, NB, NC><<<dim3((MS::TILES + 7) / 8, n), 256, 0, s>>>(fam, first);
    bwd<<<dim3(MS::SLABS, n), MS::THREADS, MS::BYTES, s>>>(fam, first, r, u);
  }
  return cudaGetLastError() == cudaSuccess ? PMG_OK : PMG_ECUDA;
}

}  // namespace pmg
