// FP64 line contractions on the tensor cores by exact digit splitting (the scheme of
// Ozaki, Ogita, Oishi and Rump, 2012, "Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication"): GB300's FP64 pipes
// issue 1.7 multiply-adds per SM and clock (measured), its fp16 tensor path 960.
//
// A table entry and a line value are fixed-point integers cut into six balanced
// base-1024 digits, which fp16 holds exactly.  The products of digits i and j with
// i + j = w are summed by fp16 MMAs into one fp32 accumulator per weight w = 0..6.
// The sums w <= 3 are integers below 2^24 (split_fragments checks the bound for each
// table), so these accumulators are exact, and the rounding of the others does not count;
// added as 64-bit integers they give the product to about 2^-60 of (largest value) x
// (largest entry).  Without the weight 6 the error of P = 16 sweeps against 64 bits was a third above
// that of the plain FP64 kernel (EA 1.02e-14 against 7.9e-15); the terms w >= 7 are below 2^-60.
//
// Scaling: B = M 2^(59 + t - e), where sum_k |M_k| <= 2^e for every output of the table (one e
// per table; a backward even-odd table counts both blocks of a node); t = 0, or 2 in the
// operator's tables (kApplyBits); X = x 2^-ex with |X| < 2^60.  B = sum_j b_j 2^(50 - 10 j),
// X = sum_i x_i 2^(52 - 10 i), hence sum M x = T 2^(e + 2 - g - t + ex) with
// T = sum_w acc_w 2^(41 + g - 10 w), |T| <= 2^(58 + g + t).
#pragma once

#include <cstdint>
#include <cuda_fp16.h>

#include "pmg_internal.h"

namespace pmg {

constexpr int kSplitDigits = 6;
constexpr int kSplitWeights = 7;

// blocks of 16 x 16 table entries per table: one up to 16 nodes; above, those of a general
// table (up to 32 nodes an even-odd folded one takes the first two)
__host__ __device__ constexpr int split_blocks(int n) { return ((n + 15) / 16) * ((n + 15) / 16); }
// uint4 (four packed fp16 pairs of a lane's A fragment) per table
__host__ __device__ constexpr int split_frag_len(int n) { return split_blocks(n) * kSplitDigits * 32; }

// Host form of a table: 16 x 16 blocks [input][output].
struct SplitBlocks {
  int nblk;
  bool chain = false;      // blocks 2 i and 2 i + 1 (two input halves) share their accumulators
  bool join_out = false;   // outputs of the blocks are added (even-odd recombination)
  bool swap1 = false;      // block 1 has its inputs 8..11 in the fourth slots (they share
                           // registers with those of block 0)
  std::vector<double> v;
  explicit SplitBlocks(int n) : nblk(n), v((size_t)n * 256, 0.0) {}
  double& at(int b, int k, int o) { return v[((size_t)b * 16 + k) * 16 + o]; }
  double at(int b, int k, int o) const { return v[((size_t)b * 16 + k) * 16 + o]; }
};
constexpr int kApplyBits = 2;
void split_fragments(const SplitBlocks& B, int& expo, bool& ok, uint32_t* frag, int more_bits = 0);
// the same blocks as bf16 terms (fdm_mma.cuh), each entry the sum of three
constexpr int kBf16Terms = 3;
void bf16_fragments(const SplitBlocks& B, uint32_t* frag);
// the same fragments for the table as the second MMA operand (n > 32, the slab kernel's c-lines)
void bf16_fragments_b(const SplitBlocks& B, uint32_t* frag);
SplitBlocks patch_blocks(const double* M, int n, bool folded, bool backward);
// scales every output of a backward patch table to entries that sum to about 1; rexp[n]: the
// exponents taken out
void scale_patch_outputs(SplitBlocks& B, int n, bool folded, int* rexp);
// 1-D operator of element m of an axis with its neighbour terms as further inputs (see
// setup.cpp); kd: the derivative inputs come times 2^-kd.  folded: even-odd form.  rexp[NP]:
// exponent of each output.
SplitBlocks apply_blocks(const Axis1DHost& a, int m, int kd, bool& folded, int* rexp);
int apply_deriv_shift(const Axis1DHost& a);
// centro-symmetric table M[k][out] (nin x nout): even-odd folded above 16 entries
SplitBlocks sym_blocks(const double* M, int nin, int nout);

#ifdef __CUDACC__

__device__ __forceinline__ void mma_f16(float (&d)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void mma_f16_zero(float (&d)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1), "f"(0.0f));
}

// Digit i of two values as one fp16 pair, from the biased words (value + kSplitBias) in
// w0, w1 (the high words for i < 3, the low words for i >= 3): digits at bits 20, 10, 0 of
// the high word and 22, 12, 2 of the low one.  1024 + digit is formed by the exponent trick,
// then 1024 + 512 is subtracted.  Byte permutes move whole halves where a digit lies within
// 16 bits; the shifts to the left become multiplies (the logic pipe is this code's bound).
__device__ __forceinline__ uint32_t digit_pair(uint32_t w0, uint32_t w1, int i) {
  uint32_t h;
  if (i == 0) h = __byte_perm(w0, w1, 0x7632) >> 4;
  else if (i == 2) h = __byte_perm(w0, w1, 0x5410);
  else if (i == 3) h = __byte_perm(w0, w1, 0x7632) >> 6;
  else if (i == 5) h = __byte_perm(w0, w1, 0x5410) >> 2;
  else if (i == 1) h = ((w0 >> 10) & 0x3ffu) | ((w1 << 6) & 0x3ff0000u);
  else h = ((w0 >> 12) & 0x3ffu) | ((w1 << 4) & 0x3ff0000u);
  h = (h & 0x3ff03ffu) | 0x64006400u;
  uint32_t r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(h), "r"(0x66006600u));
  return r;
}

// half a unit of the last digit (rounding) and 512 at every digit (balancing)
constexpr unsigned long long kSplitBias =
    (1ull << 61) | (1ull << 51) | (1ull << 41) | (1ull << 31) | (1ull << 21) | (1ull << 11) | 2ull;

// X 2^s + kSplitBias, 0 <= s < 32, as multiplies by mul = 2^s
__device__ __forceinline__ unsigned long long split_word(long long X, unsigned mul) {
  const unsigned long long lo = (unsigned long long)(unsigned)X * mul + kSplitBias;
  return lo + ((unsigned long long)((unsigned)((unsigned long long)X >> 32) * mul) << 32);
}

// acc[w] = sum_{i + j = w} (table digit j) x (line digit i), or += with ADD; NW weights
template <bool ADD = false, int NW>
__device__ __forceinline__ void split_mma(float (&acc)[NW][4], const uint4 (&A)[kSplitDigits],
                                          const uint32_t (&b0)[kSplitDigits], const uint32_t (&b1)[kSplitDigits]) {
#pragma unroll
  for (int i = 0; i < kSplitDigits; ++i)
#pragma unroll
    for (int j = 0; i + j < NW && j < kSplitDigits; ++j) {
      if (!ADD && (i == 0 || (i == 1 && j == kSplitDigits - 1))) mma_f16_zero(acc[i + j], A[j], b0[i], b1[i]);
      else mma_f16(acc[i + j], A[j], b0[i], b1[i]);
    }
}

// T = sum_w acc_w 2^(42 - 10 w), the last three accumulators merged in fp32; |acc_0| < 2^20
// and |acc_1| < 2^23 by the row-sum scaling, so the first two merge in 32 bits.  |T| <= 2^59 (2^61
// with kApplyBits), so the normalisation of the next pass of a patch never shifts to the right.
__device__ __forceinline__ long long split_join(const float (&acc)[kSplitWeights][4], int r) {
  const int i0 = __float2int_rn(acc[0][r]), i1 = __float2int_rn(acc[1][r]), i2 = __float2int_rn(acc[2][r]),
            i3 = __float2int_rn(acc[3][r]),
            i4 = __float2int_rn(__fmaf_rn(acc[4][r], 4.0f, __fmaf_rn(acc[6][r], 0x1p-18f, acc[5][r] * 0x1p-8f)));
  long long T = (long long)i3 * 4096 + i4;
  T += (long long)i2 * 4194304;
  return T + (long long)((unsigned long long)(unsigned)(i0 * 1024 + i1) << 32);
}

// T = sum_w acc_w 2^(41 - 10 w) of six weights
__device__ __forceinline__ long long split_join(const float (&acc)[kSplitDigits][4], int r) {
  const int i0 = __float2int_rn(acc[0][r]), i1 = __float2int_rn(acc[1][r] + acc[1][r]),
            i2 = __float2int_rn(acc[2][r]), i3 = __float2int_rn(acc[3][r]),
            i4 = __float2int_rn(__fmaf_rn(acc[4][r], 2.0f, acc[5][r] * 0x1p-9f));
  long long T = (long long)i3 * 2048 + i4;
  T += (long long)i2 * 2097152;
  return T + (long long)(i0 * 2048 + i1) * 1073741824;
}

// x 2^(1075 + UP - E) rounded down, for the bits of a finite double below 2^(E - 1022), E >= 1
// the biased exponent of the largest: |result| <= 2^(53 + UP).  Down for both signs (~v, also
// for -0): split_word's rounding of the two last bits then has no bias; truncated negative values got one.
template <int UP = 6>
__device__ __forceinline__ long long double_fixed(long long bits, int E) {
  const int hi = (int)(bits >> 32);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned mh = e ? ((unsigned)hi & 0xfffffu) | 0x100000u : 0u;   // subnormals count as zero
  const unsigned long long m = ((unsigned long long)mh << 32 | (unsigned)bits) << UP;
  const int sh = min(E - e, 63);
  const long long v = (long long)(m >> sh);
  return hi < 0 ? ~v : v;
}

// (-1)^neg a 2^k rounded to nearest, by integer operations; a result in the normal range.
// The leading bit of m >> 11 adds one to the exponent field, and a rounding carry does too.
__device__ __forceinline__ double scaled_double(unsigned long long a, bool neg, int k) {
  const int lz = __clzll((long long)a);
  const unsigned long long m = a << (lz & 63);
  const unsigned long long v = ((unsigned long long)(unsigned)(1085 + k - lz) << 52) + (m >> 11) + ((m >> 10) & 1ull);
  return __longlong_as_double((long long)(a ? v | ((unsigned long long)neg << 63) : 0ull));
}

// T 2^k rounded to nearest, by integer operations (a conversion takes a slot of the FP64
// pipe, about 75 times one of these); the result must lie in the normal range
__device__ __forceinline__ double fixed_double(long long T, int k) {
  return scaled_double((unsigned long long)(T < 0 ? -T : T), T < 0, k);
}
// the same for any k
static __device__ __noinline__ double any_double(long long T, int k) { return scalbn((double)T, k); }
__device__ __forceinline__ double fixed_double_any(long long T, int k) {
  return (unsigned)(k + 1000) < 1900u ? fixed_double(T, k) : any_double(T, k);
}

#endif  // __CUDACC__

}  // namespace pmg
