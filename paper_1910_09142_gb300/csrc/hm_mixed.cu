// Mixed-precision evolve (step 2 of Sec. I.C.1) for GB300.
//
// GB300 runs binary32 FMA about 58x faster than binary64 (measured 69.9 vs
// 1.2 TFLOP/s on 152 SMs), so this path forms the two-site tensor and applies
// the 9x9 gate in binary32 and runs the one-sided Jacobi sweeps of every
// charge block (Sec. II.C, hm_block.cuh) in binary32.  HM_MIXED then finishes
// each block as a binary64 sweep would (hm_refine.cuh: one first-order sweep as a
// product, binary64 rotations where that does not hold; what it leaves is stated
// there); HM_MIXED32 stops at the binary32 sweeps.  The truncation weights (Sec. II), the renormalisation
// of the kept singular values and the stored site tensors stay binary64.
// Measurement and collapse (steps 3-4) are the binary64 kernels of hm_fp64.cu.
//
// A chain has one CTA of 512 threads on an SM of its own, a cluster of such CTAs
// in small batches (hm_team.h), or (hm_mixed_pair.cu) half an SM, 256
// threads, in batches wider than the GPU.  The blocks of a split that fit in
// shared memory together form a wave and are decomposed at once by warp
// groups; a block too large for shared memory keeps W and V in global memory
// and works on pairs of column blocks staged in shared memory (intra-block
// pairs once per sweep, then every cross pair of two staged blocks).
#include <cuda_runtime.h>

#include <cfloat>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "hm_block.cuh"
#include "hm_internal.h"
#include "hm_refine.cuh"
#include "hm_team.h"

namespace hm {

namespace {

// This file builds the kernel twice: one CTA of 512 threads per SM (218 KB
// of shared memory), and, from hm_mixed_pair.cu, two CTAs of 256 threads per
// SM (109 KB each) for batches with more chains than SMs.
#ifndef HM_MIXED_NT
#define HM_MIXED_NT 512
#define HM_MIXED_CTAS_PER_SM 1
#endif
constexpr int NT = HM_MIXED_NT;
constexpr int kCtasPerSm = HM_MIXED_CTAS_PER_SM;
constexpr int kMaxSweeps = 60;
constexpr int GM = kMixedGM, GN = kMixedGN, GK = kMixedGK;   // binary32 GEMM tile (2x4 or 4x4 outputs a thread)

struct Scal {
  int32_t ival[4];
};

__device__ __forceinline__ float warp_sumf(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Rotate the column pair (x, y) of length q (W) and (vx, vy) of length p (V)
// so that x . y = 0 (Hestenes).  Warp-cooperative; returns 1 if rotated.
__device__ __forceinline__ int rotate_pair(float* x, float* y, int q, float* vx, float* vy, int p, float tol,
                                           int lane, float* rmax) {
  float al = 0.f, be = 0.f, ga = 0.f;
  for (int i = lane; i < q; i += 32) {
    const float a = x[i], b = y[i];
    al = fmaf(a, a, al);
    be = fmaf(b, b, be);
    ga = fmaf(a, b, ga);
  }
  al = warp_sumf(al);
  be = warp_sumf(be);
  ga = warp_sumf(ga);
  if (!(ga != 0.f && al > 0.f && be > 0.f && fabsf(ga) > tol * sqrtf(al) * sqrtf(be))) return 0;
  *rmax = fmaxf(*rmax, fabsf(ga) / (sqrtf(al) * sqrtf(be)));
  const float zeta = (be - al) / (2.f * ga);
  float t;
  if (fabsf(zeta) > 1e18f) t = 0.5f / zeta;
  else t = copysignf(1.f, zeta) / (fabsf(zeta) + sqrtf(1.f + zeta * zeta));
  const float cs = rsqrtf(1.f + t * t), sn = cs * t;
  for (int i = lane; i < q; i += 32) {
    const float a = x[i], b = y[i];
    x[i] = cs * a - sn * b;
    y[i] = sn * a + cs * b;
  }
  for (int i = lane; i < p; i += 32) {
    const float a = vx[i], b = vy[i];
    vx[i] = cs * a - sn * b;
    vy[i] = sn * a + cs * b;
  }
  return 1;
}

// Stage columns [c0, c0 + nc) of W (stride q) and V (stride p) into smem.
__device__ void stage(const float* W, const float* V, int q, int p, int c0, int nc, float* sw, float* sv) {
  for (int e = threadIdx.x; e < nc * q; e += NT) sw[e] = W[(size_t)c0 * q + e];
  for (int e = threadIdx.x; e < nc * p; e += NT) sv[e] = V[(size_t)c0 * p + e];
}

__device__ void unstage(float* W, float* V, int q, int p, int c0, int nc, const float* sw, const float* sv) {
  for (int e = threadIdx.x; e < nc * q; e += NT) W[(size_t)c0 * q + e] = sw[e];
  for (int e = threadIdx.x; e < nc * p; e += NT) V[(size_t)c0 * p + e] = sv[e];
}

// Cross pairs of the block Jacobi with the I column in registers: in every
// round t warp w pairs column I_w with J_{(w+t) mod b}, so warp w keeps I_w
// (and its V column) in registers for all later blocks J and only the J
// column crosses shared memory (one load and one store per element of W and
// of V).  Column norms are cached in `norm` (recomputed here first), so each
// rotation needs one dot product.  q <= 32 QL.
template <int QL>
__device__ void cross_phase_reg(float* W, float* V, int q, int p, int b, int nb, float* swJ, float* svJ,
                                float* norm, float tol, int& rot, float& rmax) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int nwarps = NT / 32;
  for (int j = warp; j < p; j += nwarps) {
    const float* cj = W + (size_t)j * q;
    float s2 = 0.f;
    for (int i = lane; i < q; i += 32) s2 = fmaf(cj[i], cj[i], s2);
    s2 = warp_sumf(s2);
    if (lane == 0) norm[j] = s2;
  }
  __syncthreads();
  for (int I = 0; I + 1 < nb; ++I) {
    const int cI = I * b, nI = min(b, p - cI);
    const bool own = warp < nI;
    const int col = cI + warp;
    float xr[QL], vr[QL];
    float nx = 0.f;
#pragma unroll
    for (int k = 0; k < QL; ++k) {
      xr[k] = 0.f;
      vr[k] = 0.f;
    }
    if (own) {
      const float* xw = W + (size_t)col * q;
      const float* vw = V + (size_t)col * p;
#pragma unroll
      for (int k = 0; k < QL; ++k) {
        if (32 * k >= q) break;               // warp-uniform: only live chunks
        const int i = lane + 32 * k;
        xr[k] = i < q ? xw[i] : 0.f;
        vr[k] = i < p ? vw[i] : 0.f;
      }
      nx = norm[col];
    }
    for (int J = I + 1; J < nb; ++J) {
      const int cJ = J * b, nJ = min(b, p - cJ);
      for (int e = tid; e < nJ * q; e += NT) swJ[e] = W[(size_t)cJ * q + e];
      for (int e = tid; e < nJ * p; e += NT) svJ[e] = V[(size_t)cJ * p + e];
      __syncthreads();
      for (int t = 0; t < b; ++t) {
        const int j = (warp + t) % b;
        if (own && j < nJ) {
          float* y = swJ + (size_t)j * q;
          float* vy = svJ + (size_t)j * p;
          float yr[QL];
          float ga = 0.f;
#pragma unroll
          for (int k = 0; k < QL; ++k) {
            if (32 * k >= q) break;
            const int i = lane + 32 * k;
            yr[k] = i < q ? y[i] : 0.f;
            ga = fmaf(xr[k], yr[k], ga);
          }
          ga = warp_sumf(ga);
          const float be = norm[cJ + j];
          if (ga != 0.f && nx > 0.f && be > 0.f && fabsf(ga) > tol * sqrtf(nx) * sqrtf(be)) {
            rmax = fmaxf(rmax, fabsf(ga) / (sqrtf(nx) * sqrtf(be)));
            const float zeta = (be - nx) / (2.f * ga);
            float tt;
            if (fabsf(zeta) > 1e18f) tt = 0.5f / zeta;
            else tt = copysignf(1.f, zeta) / (fabsf(zeta) + sqrtf(1.f + zeta * zeta));
            const float cs = rsqrtf(1.f + tt * tt), sn = cs * tt;
#pragma unroll
            for (int k = 0; k < QL; ++k) {
              if (32 * k >= q) break;
              const int i = lane + 32 * k;
              const float a = xr[k], bb = yr[k];
              xr[k] = cs * a - sn * bb;
              if (i < q) y[i] = sn * a + cs * bb;
            }
#pragma unroll
            for (int k = 0; k < QL; ++k) {
              if (32 * k >= p) break;
              const int i = lane + 32 * k;
              if (i < p) {
                const float a = vr[k], bb = vy[i];
                vr[k] = cs * a - sn * bb;
                vy[i] = sn * a + cs * bb;
              }
            }
            nx -= tt * ga;
            __syncwarp();
            if (lane == 0) norm[cJ + j] = be + tt * ga;
            rot = 1;
          }
        }
        __syncthreads();
      }
      for (int e = tid; e < nJ * q; e += NT) W[(size_t)cJ * q + e] = swJ[e];
      for (int e = tid; e < nJ * p; e += NT) V[(size_t)cJ * p + e] = svJ[e];
      __syncthreads();
    }
    if (own) {
      float* xw = W + (size_t)col * q;
      float* vw = V + (size_t)col * p;
#pragma unroll
      for (int k = 0; k < QL; ++k) {
        if (32 * k >= q) break;
        const int i = lane + 32 * k;
        if (i < q) xw[i] = xr[k];
        if (i < p) vw[i] = vr[k];
      }
      if (lane == 0) norm[col] = nx;
    }
    __syncthreads();
  }
}

// Block one-sided Jacobi on W (q x p column-major, q >= p) with V (p x p).
// smem holds two blocks of b columns of W and of V.  Returns sweeps or -1.
__device__ int cta_jacobi_f32(float* W, int q, int p, float* V, int b, float* smem, Scal& sc) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int nwarps = NT / 32;
  for (int e = tid; e < p * p; e += NT) V[e] = (e % (p + 1) == 0) ? 1.f : 0.f;
  __syncthreads();
  float* swI = smem;
  float* swJ = swI + (size_t)b * q;
  float* svI = swJ + (size_t)b * q;
  float* svJ = svI + (size_t)b * p;
  const float tol = sqrtf((float)q) * FLT_EPSILON;
  const int nb = (p + b - 1) / b;
  int done = 0;
  bool converged = false;
  while (done < kMaxSweeps) {
    if (tid == 0) {
      sc.ival[0] = 0;
      sc.ival[2] = 0;                   // largest rotation ratio of the sweep (float bits)
    }
    __syncthreads();
    int rot = 0;
    float rmax = 0.f;
    // intra-block pairs: round-robin tournament inside each block
    for (int I = 0; I < nb; ++I) {
      const int c0 = I * b, nc = min(b, p - c0);
      stage(W, V, q, p, c0, nc, swI, svI);
      __syncthreads();
      const int n2 = nc + (nc & 1);
      for (int r = 0; r < n2 - 1; ++r) {
        for (int pi = warp; pi < n2 / 2; pi += nwarps) {
          int a, bb;
          if (pi == 0) { a = r; bb = n2 - 1; } else { a = (r + pi) % (n2 - 1); bb = (r - pi + n2 - 1) % (n2 - 1); }
          if (a >= nc || bb >= nc) continue;
          rot |= rotate_pair(swI + (size_t)a * q, swI + (size_t)bb * q, q, svI + (size_t)a * p, svI + (size_t)bb * p,
                             p, tol, lane, &rmax);
        }
        __syncthreads();
      }
      unstage(W, V, q, p, c0, nc, swI, svI);
      __syncthreads();
    }
    // cross pairs of two different blocks: round t pairs column i of I with
    // column (i + t) mod b of J, b disjoint pairs per round
    if (q > 128 && q <= 32 * 24 && b <= nwarps) {
      cross_phase_reg<24>(W, V, q, p, b, nb, swJ, svJ, svJ + (size_t)b * p, tol, rot, rmax);
    } else
    for (int I = 0; I < nb; ++I) {
      const int cI = I * b, nI = min(b, p - cI);
      stage(W, V, q, p, cI, nI, swI, svI);
      for (int J = I + 1; J < nb; ++J) {
        const int cJ = J * b, nJ = min(b, p - cJ);
        stage(W, V, q, p, cJ, nJ, swJ, svJ);
        __syncthreads();
        for (int t = 0; t < b; ++t) {
          for (int i = warp; i < nI; i += nwarps) {
            const int j = (i + t) % b;
            if (j >= nJ) continue;
            rot |= rotate_pair(swI + (size_t)i * q, swJ + (size_t)j * q, q, svI + (size_t)i * p, svJ + (size_t)j * p,
                               p, tol, lane, &rmax);
          }
          __syncthreads();
        }
        unstage(W, V, q, p, cJ, nJ, swJ, svJ);
        __syncthreads();
      }
      unstage(W, V, q, p, cI, nI, swI, svI);
      __syncthreads();
    }
    if (rot && lane == 0) sc.ival[0] = 1;
    if (lane == 0) atomicMax(&sc.ival[2], __float_as_int(rmax));
    __syncthreads();
    const int any = sc.ival[0];
    const float rm = __int_as_float(sc.ival[2]);
    __syncthreads();
    ++done;
    // no rotation: converged; all rotations tiny: quadratic convergence puts
    // the next sweep's off-diagonals (O(rm^2)) below the tolerance
    if (!any || rm < 2e-4f) {
      converged = true;
      break;
    }
  }
  return converged ? done : -1;
}

__device__ void set_error(const ChainDev* c, int code, int where, int32_t* ctx_err) {
  if (threadIdx.x == 0) {
    if (atomicCAS(c->status, 0, code) == 0) *c->err_where = where;
    if (ctx_err) atomicCAS(ctx_err, 0, code);
  }
}

// Column scales 1 / |v_j| of V (binary32, leading dimension ldv) into scale.
// A binary32 Givens rotation with a small angle t has cs = 1 exactly once
// 1 + t^2 rounds to 1, so it stretches both columns by sqrt(1 + t^2): a bias
// that never cancels, and after the ~10^3 rotations a column sees it leaves
// V's columns longer than 1 by ~1e-5.  Left in, each kept singular vector
// would be weighted by its column's stretch, a systematic energy error of
// ~2e-5 in every sample (measured on GB300).  The rotations stay conformal,
// and W = theta V holds column by column, so scaling a column of W and of V
// by the same factor removes the stretch.  One warp per column.
__device__ void column_scales(const float* V32, int ldv, int p, double* scale) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int j = warp; j < p; j += NT / 32) {
    const float* v = V32 + (size_t)j * ldv;
    double s2 = 0.0;
    for (int i = lane; i < p; i += 32) s2 = fma((double)v[i], (double)v[i], s2);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    if (lane == 0) scale[j] = s2 > 0.0 ? 1.0 / sqrt(s2) : 1.0;
  }
  __syncthreads();
}

// After the binary32 sweeps: W64 = W32 with unit-column scales, V32 scaled
// in place to unit columns (a binary32 product: V32 holds binary32 values
// anyway, and the binary64 pipe is GB300's scarce one).  scale: p doubles.
__device__ void promote_w(const float* W32, int ldw, float* V32, int ldv, int q, int p, double* W64, double* scale) {
  column_scales(V32, ldv, p, scale);
  for (int e = threadIdx.x; e < q * p; e += NT) W64[e] = (double)W32[(size_t)(e / q) * ldw + e % q] * scale[e / q];
  for (int e = threadIdx.x; e < p * p; e += NT) V32[(size_t)(e / p) * ldv + e % p] *= (float)scale[e / p];
}

// After the polish: V64 = V32 with unit columns, W64 scaled alike (the
// binary64 sweep's rotations are binary32 in V).  Without a polish V32 has
// unit columns from promote_w already and is only widened.
__device__ void promote_v(const float* V32, int ldv, int q, int p, double* W64, double* V64, double* scale,
                          int rescale) {
  if (!rescale) {
    for (int e = threadIdx.x; e < p * p; e += NT) V64[e] = (double)V32[(size_t)(e / p) * ldv + e % p];
    return;
  }
  column_scales(V32, ldv, p, scale);
  for (int e = threadIdx.x; e < q * p; e += NT) W64[e] *= scale[e / q];
  for (int e = threadIdx.x; e < p * p; e += NT) V64[e] = (double)V32[(size_t)(e / p) * ldv + e % p] * scale[e / p];
}

// Shared memory of the binary32 block Jacobi; the kernel's dynamic shared
// memory is at least this (and at least the staged fallback's plan, made for
// kStagedBudget).  One CTA may opt into 227 KB with its 4 KB of static shared
// memory; two CTAs share the SM's 228 KB, 1 KB of it reserved for each.
constexpr size_t kBlockSmem = kCtasPerSm == 1 ? 218 * 1024 : kPairBlockSmem;
constexpr size_t kStagedBudget = kCtasPerSm == 1 ? 210 * 1024 : 108 * 1024;
// Of it, what the blocks of a wave may take.
#ifndef HM_WAVE_SMEM
#define HM_WAVE_SMEM kBlockSmem
#endif
constexpr size_t kWaveSmem = HM_WAVE_SMEM;
constexpr int64_t kWaveFloats = (int64_t)(kWaveSmem / sizeof(float));
constexpr int kTileDoubles = NT / 32 * 8 * 33;   // finish()'s transposition tiles
static_assert(sizeof(blk::PrepTab) <= kBlockSmem, "prepare's tables");

// Stopping rule of the binary64 polish: a sweep whose largest rotation ratio
// is below this leaves off-diagonals of order its square for the next sweep.
// After the binary32 sweeps that ratio is ~1e-6, so one binary64 sweep ends
// the polish with off-diagonals of order 1e-12.
constexpr double kPolishStop = 1e-5;

// Stopping ratio of the binary32 sweeps (warp-group path): 2e-4 when they
// are the whole SVD (HM_MIXED32; the next sweep's off-diagonals would be
// ~4e-8, below binary32 resolution), 1e-3 when a binary64 sweep follows
// (HM_MIXED): the off-diagonals it inherits are then ~1e-6, below
// kPolishStop, so one binary64 sweep still ends the polish.
constexpr float kStop32 = 2e-4f, kStop32Polished = 1e-3f;

// The binary64 sweeps of a block the first-order step does not settle.  Rare:
// kept out of line, away from the hot code.
__device__ HM_COLD int sweep64(double* W, int q, int p, double* V, double* nrm, int lw, int nw, int bar, int g,
                                    blk::GroupSh& gs) {
  return blk::jacobi_group<double, double, 2>(W, q, q, p, V, p, nrm, lw, nw, bar, g, gs, kPolishStop, kMaxSweeps);
}

// From a block's binary32 result (W32, V32 in shared memory, followed by
// refine::extra floats) to its binary64 W and V (global memory), by the nw
// warps of its group.  polish: the binary64 finish of hm_refine.cuh
// (2: on a state whose norm is not known to be 1, see check_range); otherwise only
// the unit-column scales.  K: scratch for the block's K.  Returns
// the polish passes (1, or the binary64 sweeps it fell back on), -1 when
// those did not converge.
__device__ int refine_block(ChainDev* c, const blk::BlockRec& r, float* W32, float* V32, float* K,
                            int polish, int lw, int nw, int bar, int g, blk::GroupSh& gs) {
  const int q = r.q, p = r.p, ldw = blk::ld4(q), ldv = blk::ld4(p);
  float* ah = V32 + (size_t)p * ldv;
  float* al = ah + p;
  float* dl = al + p;
  double* W64 = c->W + r.woff;
  double* V64 = c->V + r.voff;
  const int nthr = 32 * nw;
  if (q > 128) {                              // the sweeps went through jacobi_blocks: pad the columns
    refine::pad_rows(W32, q, ldw, p, lw, nw);
    refine::pad_rows(V32, p, ldv, p, lw, nw);
  }
  blk::group_sync(bar, nthr);                 // the sweeps' last reads of the norms
  const bool out =
      refine::column_terms(W32, q, ldw, V32, p, ldv, ah, al, dl, polish ? K : nullptr, lw, nw, polish == 2);
  if (lw == 0 && (threadIdx.x & 31) == 0) {
    gs.flag[g] = 0;
    gs.rbits[g] = 0u;
  }
  blk::group_sync(bar, nthr);
  bool plain = polish == 0;                   // only the unit-column scales
  if (polish) {
    float e = refine::pair_terms<false>(W32, q, ldw, p, ah, al, K, lw, nw);
    if (out) e = refine::kOutOfRange;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e = fmaxf(e, __shfl_xor_sync(0xffffffffu, e, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&gs.rbits[g], __float_as_uint(e));
    blk::group_sync(bar, nthr);               // K and its largest entry are complete
    plain = __uint_as_float(gs.rbits[g]) >= refine::kOutOfRange;
  }
  int x = 0;
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    const int n = side ? p : q;
    if (plain) refine::scale_columns(side ? V32 : W32, n, side ? ldv : ldw, p, dl, side ? V64 : W64, lw, nw);
    else refine::add_product<false>(side ? V32 : W32, n, side ? ldv : ldw, p, K, side ? V64 : W64, n, lw, nw, x);
  }
  if (!polish) return 0;
  blk::group_sync(bar, nthr);
  if (lw == 0) {
    const int found = plain ? 0 : refine::rotate_near(W64, q, V64, p, ah, 2 * p);
    if ((threadIdx.x & 31) == 0)
      gs.flag[g] = found > 2 * p || __uint_as_float(gs.rbits[g]) >= (float)kPolishStop ? 2 : (found > 0 ? 1 : 0);
  }
  blk::group_sync(bar, nthr);
  const int more = gs.flag[g];
  if (more == 0) return 1;
  blk::group_sync(bar, nthr);                 // every warp has read the flag
  int s64 = 1;
  if (more == 2) {
    s64 = sweep64(W64, q, p, V64, c->sig + r.svoff, lw, nw, bar, g, gs);
    blk::group_sync(bar, nthr);
  }
  refine::unit_columns(W64, q, V64, p, lw, nw);
  return s64;
}

// Shared-memory floats of one block: W, V and the finish's terms.
__device__ __forceinline__ int64_t block_floats(int q, int p) {
  return (int64_t)p * blk::ld4(q) + (int64_t)p * blk::ld4(p) + blk::ld4(refine::extra(p));
}

// The same with no padding but odd leading dimensions: W, V and the norms.
__device__ __forceinline__ int64_t tight_floats(int q, int p) {
  return (int64_t)p * (q | 1) + (int64_t)p * (p | 1) + p;
}

// One block by the whole CTA whose wave layout (block_floats) does not fit in
// shared memory: binary32 sweeps, then a binary64 sweep.  Columns without padding
// (tight_floats) take a few per cent less, and where they fit the sweeps run on
// them in shared memory; otherwise on column blocks staged from global memory.
// GB300, one split in a buffer of 210 KB: 168 x 159 13.6 ms against 17.0 ms staged,
// 165 x 162 15.1 against 20.3 (both fit the wave layout in 218 KB).
// Returns the binary32 sweeps + 1000 x the binary64 ones, or -1.  Out of line: it is
// rare, and its code would crowd the usual path's.
__device__ HM_COLD int decompose_staged(ChainDev* c, int k, const blk::SplitSh& ss, const blk::BlockRec& r,
                                             const float* theta, int bcols, int polish, float* smem, Scal& sc,
                                             blk::GroupSh& gs) {
  const int warp = threadIdx.x >> 5, q = r.q, p = r.p;
  const bool fits = tight_floats(q, p) <= kWaveFloats;
  const int ldw = fits ? q | 1 : q, ldv = fits ? p | 1 : p;
  float* W32 = fits ? smem : c->X;
  float* V32 = W32 + (size_t)p * ldw;
  int c0 = 0;
  blk::gather_block<NT, float, float>(c, k, ss, r, theta, W32, ldw, V32, ldv, c0);
  __syncthreads();
  const int sw = fits ? blk::jacobi_group<float>(W32, q, ldw, p, V32, ldv, V32 + (size_t)p * ldv, warp, NT / 32, 1, 0,
                                                 gs, polish ? kStop32Polished : kStop32, kMaxSweeps)
                      : cta_jacobi_f32(W32, q, p, V32, bcols, smem, sc);
  if (sw < 0) return -1;
  double* W64 = c->W + r.woff;
  double* V64 = c->V + r.voff;
  promote_w(W32, ldw, V32, ldv, q, p, W64, c->sig);
  __syncthreads();
  const int s64 = polish ? blk::jacobi_group<double, float, 2>(W64, q, q, p, V32, ldv, c->sig, warp, NT / 32, 1, 0, gs,
                                                               kPolishStop, kMaxSweeps)
                         : 0;
  __syncthreads();
  promote_v(V32, ldv, q, p, W64, V64, c->sig, polish);
  return s64 < 0 ? -1 : sw + 1000 * s64;
}

// One two-site op (step 2 of Sec. I.C.1) in charge blocks (Sec. II.C):
// theta and the gate in binary32 (operands rounded from the binary64 site
// tensors, binary32 accumulation, gate coefficients as binary32 pairs); the
// blocks of a split in waves that fit in shared memory, each block of a wave
// decomposed by its own warp group at the same time: a binary32 one-sided
// Jacobi, then (HM_MIXED) refine_block.  A block too large for
// shared memory runs alone, its binary32 sweeps on column blocks staged from
// global memory, then a binary64 sweep.  Then the truncation rule (Sec. II), renormalisation and
// absorb in binary64.
__device__ void two_site_op_mixed(ChainDev* c, const OpDev op, int t, int bcols, int polish, float* smem, Scal& sc,
                                  blk::SplitSh& ss, blk::WaveSh& wv, blk::GroupSh& gs, const blk::Team& tm,
                                  int32_t* ctx_err) {
  const int tid = threadIdx.x, warp = tid >> 5;
  blk::PrepTab& tab = *reinterpret_cast<blk::PrepTab*>(smem);
  if (!blk::prepare<NT>(c, op, ss, tab, tm)) blk::prepare<NT>(c, op, ss, tab, tm);
  float* theta = reinterpret_cast<float*>(c->theta);
  blk::theta_blocks<NT, GM, GN, GK>(c, op.k, ss, theta, smem, tm);
  int sw32 = 0, sw64 = 0;
  int64_t cost = -1;
  constexpr int64_t cap = kWaveFloats;
  if (tid == 0) blk::own_blocks(ss, tm, wv, [&](int q, int p) { return block_floats(q, p) <= cap; });
  __syncthreads();
  const int nown = wv.nown;
  bool failed = false;
  for (int b0 = 0; b0 < nown && !failed;) {
    if (tid == 0) {
      // as many of the CTA's blocks as fit in shared memory (at most 15 and
      // one warp each); a block that does not fit alone takes the global path
      int64_t used = 0;
      int n = 0, p[15], cost[15];
      while (b0 + n < nown && n < 15 && n < NT / 32) {
        const blk::BlockRec& r = ss.b[blk::own_block(wv, b0 + n)];
        const int64_t need = block_floats(r.q, r.p);
        if (used + need > cap) break;
        wv.off[n] = (int32_t)used;
        p[n] = r.p;
        cost[n] = blk::block_cost(r.q, r.p);
        used += need;
        ++n;
      }
      wv.b0 = b0;
      wv.n = n;
      wv.ng = n > 0 ? blk::assign_warps(p, cost, n, NT / 32, wv.grp, wv.w0, wv.nw) : 0;
    }
    __syncthreads();
    const int n = wv.n;
    if (n == 0) {
      const blk::BlockRec& r = ss.b[blk::own_block(wv, b0)];
      const int code = decompose_staged(c, op.k, ss, r, theta, bcols, polish, smem, sc, gs);
      if (code < 0) {
        set_error(c, HM_ERR_NUMERIC, t, ctx_err);
        failed = true;
        break;
      }
      const int64_t cb = (int64_t)r.q * r.p * r.p;
      if (cb > cost) cost = cb, sw32 = code % 1000, sw64 = code / 1000;
      b0 += 1;
      continue;
    }
    int c0 = 0;
    for (int i = 0; i < n; ++i) {
      const blk::BlockRec& r = ss.b[blk::own_block(wv, b0 + i)];
      float* W32 = smem + wv.off[i];
      float* V32 = W32 + (size_t)r.p * blk::ld4(r.q);
      blk::gather_block<NT, float, float>(c, op.k, ss, r, theta, W32, blk::ld4(r.q), V32, blk::ld4(r.p), c0);
    }
    __syncthreads();
    const int g = blk::my_group(wv, warp);
    for (int i = 0; g >= 0 && i < n; ++i) {
      if (wv.grp[i] != g) continue;
      const int ib = blk::own_block(wv, b0 + i);
      const blk::BlockRec& r = ss.b[ib];
      float* W32 = smem + wv.off[i];
      float* V32 = W32 + (size_t)r.p * blk::ld4(r.q);
      const int lw = warp - wv.w0[g], nw = wv.nw[g];
      const int sw = blk::jacobi_group<float>(W32, r.q, blk::ld4(r.q), r.p, V32, blk::ld4(r.p),
                                              V32 + (size_t)r.p * blk::ld4(r.p), lw, nw, g + 1, g, gs,
                                              polish ? kStop32Polished : kStop32, kMaxSweeps);
      const int s64 =
          sw < 0 ? 0 : refine_block(c, r, W32, V32, c->X + refine::k_offset(ss, ib), polish, lw, nw, g + 1, g, gs);
      if (lw == 0 && (tid & 31) == 0) wv.sw[i] = sw < 0 || s64 < 0 ? -1 : sw + 1000 * s64;
      blk::group_sync(g + 1, 32 * nw);          // the group's flags are free for its next block
    }
    __syncthreads();
    for (int i = 0; i < n; ++i) {
      const int code = wv.sw[i];
      if (code < 0) {
        set_error(c, HM_ERR_NUMERIC, t, ctx_err);
        failed = true;
        break;
      }
      const blk::BlockRec& r = ss.b[blk::own_block(wv, b0 + i)];
      const int64_t cb = (int64_t)r.q * r.p * r.p;
      if (cb > cost) cost = cb, sw32 = code % 1000, sw64 = code / 1000;
    }
    b0 += n;
    __syncthreads();
  }
  // a failed decomposition ends in finish(), behind the team's barrier
  __syncthreads();
  double* tiles = reinterpret_cast<double*>(smem);
  char* scratch = reinterpret_cast<char*>(tiles + kTileDoubles);
  const size_t need = blk::finish_bytes(ss.P);
  if (kTileDoubles * sizeof(double) + need > kBlockSmem) scratch = reinterpret_cast<char*>(c->theta) + tm.rank * need;
  blk::finish<NT>(c, op, t, ss, wv, tm, scratch, tiles, ctx_err, sw32, sw64);
}

// Whether the state's norm may be far from 1, so that a column's length does not
// say what it weighs: a state from outside (dense until its next collapse), or explicit ops now or since
// the last reset.  The planned schedules start at norm 1 and keep it.
__device__ __forceinline__ bool check_range(const BatchArg& b, const ChainDev* c) {
  return b.ops_override || c->counters[3] || c->counters[5];
}

// team: CTAs of a cluster that share one chain (1: no cluster).
__global__ void __launch_bounds__(NT, kCtasPerSm) evolve_mixed_kernel(BatchArg b, OutArg o, int bcols, int polish,
                                                                      int team) {
  extern __shared__ float4 dsm[];                            // 16-byte aligned: 128-bit loads of the columns
  float* smem = reinterpret_cast<float*>(dsm);
  __shared__ Scal sc;
  __shared__ blk::SplitSh ss;
  __shared__ blk::WaveSh wv;
  __shared__ blk::GroupSh gs;
  const blk::Team tm = {(int)blockIdx.x % team, team};
  ChainDev* c = b.c[blockIdx.x / team];
  const OpDev* ops = b.ops_override ? b.ops_override : c->ops;
  const int n_ops = b.ops_override ? b.n_override : c->n_ops;
  const int t0 = b.budget > 0 ? c->counters[4] : b.t0;
  const int t1 = b.budget > 0 ? min(t0 + b.budget, n_ops) : (b.t1 < n_ops ? b.t1 : n_ops);
  if (polish && check_range(b, c)) polish = 2;
  blk::team_sync(tm);                                        // every thread has read the cursor and the marks
  if (b.budget > 0 && threadIdx.x == 0 && tm.rank == 0) c->counters[4] = t1;
  if (b.ops_override && threadIdx.x == 0 && tm.rank == 0) c->counters[5] = 1;
  for (int t = t0; t < t1; ++t) {
    // the team agrees: a CTA sets the status only behind a barrier of the op
    if (*(volatile int32_t*)c->status != 0) return;
    __syncthreads();
    two_site_op_mixed(c, ops[t], t, bcols, polish, smem, sc, ss, wv, gs, tm, o.ctx_err);
    blk::team_sync(tm);
  }
}

// Dynamic shared memory the staged path may plan for: what one CTA may opt into
// less the kernel's static shared memory.
#ifndef HM_STAGED_SMEM
#define HM_STAGED_SMEM (kMaxSharedOptIn - 8 * 1024)
#endif
constexpr size_t kStagedSmem = HM_STAGED_SMEM;

// Opt-in to the kernel's dynamic shared memory (per device, cached, under a
// lock: serving workers may launch from several host threads), then launch.
int launch_kernel(const BatchArg& b, const OutArg& o, int chi_cap, int polish, void* stream) {
  int bcols = 16;
  size_t plan = mixed_smem_bytes(chi_cap, &bcols, kStagedBudget);
  if (plan > kStagedSmem) {
    // caps near the admission limit: one column a staged block, so that the
    // plan fits beside the kernel's static shared memory
    bcols = 1;
    plan = (2 * 6 + 3) * (size_t)chi_cap * sizeof(float);
  }
  const size_t smem = plan > kBlockSmem ? plan : kBlockSmem;
  static std::mutex mu;
  static size_t configured[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return HM_ERR_CUDA;
  {
    std::lock_guard<std::mutex> lock(mu);
    if (dev < 0 || dev >= 64 || smem > configured[dev]) {
      if (cudaFuncSetAttribute(evolve_mixed_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
          cudaSuccess)
        return HM_ERR_CUDA;
      if (dev >= 0 && dev < 64) configured[dev] = smem;
    }
  }
#if HM_MIXED_CTAS_PER_SM == 1 && !defined(HM_HOST_EMULATION)
  const int team = team_size((const void*)evolve_mixed_kernel, NT, smem, b.n, chi_cap);
  if (team > 1) return launch_team(evolve_mixed_kernel, b, o, team, NT, smem, stream, bcols, polish, team);
#endif
  evolve_mixed_kernel<<<b.n, NT, smem, (cudaStream_t)stream>>>(b, o, bcols, polish, 1);
  return cudaGetLastError() == cudaSuccess ? HM_OK : HM_ERR_CUDA;
}

}  // namespace

#if HM_MIXED_CTAS_PER_SM == 1
int device_sm_count() {
  static std::mutex mu;
  static int count[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  std::lock_guard<std::mutex> lock(mu);
  if (count[dev] == 0 && cudaDeviceGetAttribute(&count[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    count[dev] = 0;
  return count[dev];
}
#endif

#if HM_MIXED_CTAS_PER_SM == 1
// A batch with more chains than SMs whose charge blocks fit half an SM's
// shared memory runs two chains per SM (hm_mixed_pair.cu): all of them are
// resident at once, and each SM interleaves two independent CTAs.
int launch_evolve_mixed(const BatchArg& b, const OutArg& o, int chi_cap, int polish, void* stream) {
  if (b.n <= 0) return HM_OK;
  const int sms = device_sm_count();
  if (chi_cap <= kPairChiCap && sms > 0 && b.n > sms) return launch_evolve_mixed_pair(b, o, chi_cap, polish, stream);
  return launch_kernel(b, o, chi_cap, polish, stream);
}
#else
int launch_evolve_mixed_pair(const BatchArg& b, const OutArg& o, int chi_cap, int polish, void* stream) {
  if (b.n <= 0) return HM_OK;
  return launch_kernel(b, o, chi_cap, polish, stream);
}
#endif

}  // namespace hm
