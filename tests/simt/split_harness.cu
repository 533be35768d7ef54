// TEST INFRASTRUCTURE: runs pieces of a split's decomposition in the CPU
// emulation (see block_harness.cu): the register-resident binary32 Jacobi,
// the binary64-accurate finish of a binary32 result and the
// orthonormalisation of its V (hm_refine.cuh), the integer conversions and the
// truncation rule by one warp.  Built only by test_split_emulated.py.
#include <vector>

#include "hm_block.cuh"
#include "hm_refine.cuh"

namespace {

namespace blk = hm::blk;
namespace refine = hm::refine;

__global__ void convert_probe(const double* d, float* f, const float* g, double* e, int n) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    f[i] = blk::narrow(d[i]);
    e[i] = blk::widen(g[i]);
  }
}

__global__ void trunc_probe(const double* s, int n, int chi_max, double cutoff, double* out) {
  double kept, tail;
  const int k = blk::warp_trunc_rank(s, n, chi_max, cutoff, &kept, &tail);
  if (threadIdx.x == 0) {
    out[0] = k;
    out[1] = kept;
    out[2] = tail;
  }
}

// W, V: binary32 with ld4 leading dimensions; the sweeps, then the polish.
__global__ void svd_probe(float* W, int q, int p, float* V, float* terms, float* KT, double* W64, double* V64,
                          int* out) {
  __shared__ blk::GroupSh gs;
  const int lw = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int ldw = blk::ld4(q), ldv = blk::ld4(p);
  float *ah = terms, *al = ah + p, *dl = al + p;
  const int sweeps = blk::jacobi_group<float>(W, q, ldw, p, V, ldv, ah, lw, nw, 1, 0, gs, 1e-3f, 60);
  __syncthreads();
  refine::column_terms(W, q, ldw, V, p, ldv, ah, al, dl, KT, lw, nw);
  __syncthreads();
  refine::pair_terms<false>(W, q, ldw, p, ah, al, KT, lw, nw);
  __syncthreads();
  int x = 0;
  refine::add_product<false>(W, q, ldw, p, KT, W64, q, lw, nw, x);
  refine::add_product<false>(V, p, ldv, p, KT, V64, p, lw, nw, x);
  __syncthreads();
  int found = 0;
  if (lw == 0) found = refine::rotate_near(W64, q, V64, p, ah, 2 * p);
  __syncthreads();
  refine::unit_columns(W64, q, V64, p, lw, nw);
  if (threadIdx.x == 0) {
    out[0] = sweeps;
    out[1] = found;
  }
}

// V (binary32, ld4) to binary64 with orthonormal columns.
__global__ void ortho_probe(float* V, int p, float* ah, float* KT, double* V64) {
  const int lw = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int ldv = blk::ld4(p);
  refine::unit_terms(V, p, ldv, ah, KT, lw, nw);
  __syncthreads();
  refine::pair_terms<true>(V, p, ldv, p, ah, ah, KT, lw, nw);
  __syncthreads();
  int x = 0;
  refine::add_product<false>(V, p, ldv, p, KT, V64, p, lw, nw, x);
  __syncthreads();
  refine::ortho_terms64(V64, p, p, KT, lw, nw);
  __syncthreads();
  x = 0;
  refine::add_product<true>(V, p, ldv, p, KT, V64, p, lw, nw, x);
}

}  // namespace

extern "C" void hm_probe_convert(const double* d, float* f, const float* g, double* e, int n) {
  convert_probe<<<1, 32, 0, nullptr>>>(d, f, g, e, n);
}

extern "C" void hm_probe_warp_trunc(const double* s, int n, int chi_max, double cutoff, double* out) {
  trunc_probe<<<1, 32, 0, nullptr>>>(s, n, chi_max, cutoff, out);
}

extern "C" void hm_probe_svd(float* W, int q, int p, float* V, double* W64, double* V64, int* out) {
  alignas(16) static float KT[260 * 260];
  std::vector<float> terms(3 * p);
  svd_probe<<<1, 128, 0, nullptr>>>(W, q, p, V, terms.data(), KT, W64, V64, out);
}

extern "C" void hm_probe_ortho(float* V, int p, double* V64) {
  alignas(16) static float KT[260 * 260];
  std::vector<float> ah(p);
  ortho_probe<<<1, 128, 0, nullptr>>>(V, p, ah.data(), KT, V64);
}
