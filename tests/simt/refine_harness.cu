// TEST INFRASTRUCTURE: the mixed kernel's own path of one block in the CPU
// emulation: binary32 sweeps, then refine_block (hm_mixed.cu) with its flags and
// fallbacks.  The kernel source is built once more under another namespace.  Built
// only by test_refine_emulated.py.
#define hm hm_probe_ns
#define HM_MIXED_NT 256
#define HM_MIXED_CTAS_PER_SM 2
#include "hm_mixed.cu"
#undef hm

namespace {

namespace p_ = hm_probe_ns;

// buf: W (p x ld4(q)), V (p x ld4(p)), the finish's terms.
__global__ void refine_probe(float* buf, int q, int p, float* K, p_::ChainDev* c, int polish, int* out) {
  __shared__ p_::blk::GroupSh gs;
  const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  float* V = buf + (size_t)p * p_::blk::ld4(q);
  p_::blk::BlockRec r = {};
  r.q = (int16_t)q;
  r.p = (int16_t)p;
  const int sw = p_::blk::jacobi_group<float>(buf, q, p_::blk::ld4(q), p, V, p_::blk::ld4(p),
                                              V + (size_t)p * p_::blk::ld4(p), warp, nw, 1, 0, gs,
                                              p_::kStop32Polished, p_::kMaxSweeps);
  const int s64 = p_::refine_block(c, r, buf, V, K, polish, warp, nw, 1, 0, gs);
  __syncthreads();
  if (threadIdx.x == 0) {
    out[0] = sw;
    out[1] = s64;
    out[2] = gs.flag[0];
    out[3] = (int)gs.rbits[0];
  }
}

}  // namespace

// out: binary32 sweeps, refine_block's return value, its last flag, the bits of the
// largest overlap (a binary64 sweep to its stop leaves 0 there).
extern "C" void hm_probe_refine(float* buf, int q, int p, int polish, double* W64, double* V64, double* sig, int* out) {
  alignas(16) static float K[260 * 260];
  p_::ChainDev c = {};
  c.W = W64;
  c.V = V64;
  c.sig = sig;
  refine_probe<<<1, 128, 0, nullptr>>>(buf, q, p, K, &c, polish, out);
}

namespace {

// A dense block (every charge 0) of a pair with bonds chil and chir.
__global__ void staged_probe(const float* theta, int chil, int chir, p_::ChainDev* c, int polish, int* out) {
  float* smem = (float*)simt::dynamic_smem();
  __shared__ p_::Scal sc;
  __shared__ p_::blk::SplitSh ss;
  __shared__ p_::blk::GroupSh gs;
  p_::blk::BlockRec r = {};
  r.mq = (int16_t)(3 * chil);
  r.nq = (int16_t)(3 * chir);
  r.trans = chir > chil;
  r.q = (int16_t)(3 * max(chil, chir));
  r.p = (int16_t)(3 * min(chil, chir));
  for (int t = 0; t < 3; ++t) {
    r.roff[t] = (int16_t)(t * chil);
    r.coff[t] = (int16_t)(t * chir);
  }
  if (threadIdx.x == 0)
    for (int o = 0; o < 9; ++o) {
      ss.nt[o] = 1;
      ss.tt[o][0] = (int16_t)o;
      ss.gh[o][0] = 1.0f;
      ss.gl[o][0] = 0.0f;
    }
  __syncthreads();
  const int code = p_::decompose_staged(c, 0, ss, r, theta, 4, polish, smem, sc, gs);
  if (threadIdx.x == 0) *out = code;
}

}  // namespace

// theta: 3 chil x 3 chir.  X: binary32 scratch, or null.  Returns binary32 sweeps + 1000 x binary64 ones.
extern "C" int hm_probe_staged(const float* theta, int chil, int chir, float* X, int polish, double* W64, double* V64,
                               double* sig) {
  int out = 0;
  int32_t chi[3] = {chil, 0, chir};
  p_::ChainDev c = {};
  c.W = W64;
  c.V = V64;
  c.sig = sig;
  c.X = X;
  c.chi = chi;
  staged_probe<<<1, p_::NT, p_::kBlockSmem, nullptr>>>(theta, chil, chir, &c, polish, &out);
  return out;
}

// Whether a block's wave layout, and its layout without padding, fit the kernel's buffer.
extern "C" int hm_probe_layouts(int q, int p, int64_t bytes) {
  const int64_t n = bytes / 4;
  return (p_::block_floats(q, p) <= n ? 1 : 0) + (p_::tight_floats(q, p) <= n ? 2 : 0);
}

// Cluster size for n chains when 75, 37 and 18 clusters of 2, 4 and 8 CTAs fit.
extern "C" int hm_probe_team(int n, int chi_cap) {
  const int most[4] = {0, 75, 37, 18};
  return p_::pick_team(most, n, chi_cap);
}
