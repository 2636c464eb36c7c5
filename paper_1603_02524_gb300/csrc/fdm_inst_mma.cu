// Instantiations of the fp32 patch kernel with bf16-term MMA passes (fdm_mma.cuh): 3-D and
// 2-D patch shapes (EA: n^d; FA: 2P x n_t^(d-1), and with the first two swapped) of at most 32
// nodes per axis and of the sizes that attach_split gives it (kMmaMinNodes, kMmaMinNodesFa,
// kSplitMinNodes2), and the 3-D shapes of P = 32 in slabs.
#include "fdm_mma.cuh"

namespace pmg {

int fdm_dispatch_mma(const FdmFamily<float>& fam, const float* r, float* u, cudaStream_t s) {
  const int na = fam.ax[0].n, nb = fam.ax[1].n, nc = fam.ax[2].n;
#define C(A, B, CC) \
  if (na == A && nb == B && nc == CC) return fdm_launch_mma<A, B, CC>(fam, r, u, s);
  C(13, 13, 13) C(17, 17, 17) C(23, 23, 23) C(8, 9, 9) C(16, 9, 9) C(16, 13, 13)
  C(9, 8, 9) C(9, 16, 9) C(13, 16, 13)
  C(32, 17, 17) C(32, 23, 23)
  C(17, 32, 17) C(23, 32, 23)
  C(5, 5, 1) C(7, 7, 1) C(9, 9, 1) C(13, 13, 1) C(17, 17, 1) C(23, 23, 1)
  C(4, 5, 1) C(8, 5, 1) C(8, 7, 1) C(8, 9, 1) C(16, 9, 1) C(16, 13, 1)
  C(32, 17, 1) C(32, 23, 1)
#undef C
#define C(A, B, CC) \
  if (na == A && nb == B && nc == CC) return fdm_launch_slab_mma<A, B, CC>(fam, r, u, s);
  C(43, 43, 43) C(64, 33, 33) C(64, 43, 43) C(33, 64, 33) C(43, 64, 43)    // P = 32
#undef C
  return PMG_EINVAL;
}

}  // namespace pmg
