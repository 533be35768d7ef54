// FP64 path of the hybrid purification-METTS sampler (arXiv:1910.09142).
//
// One CTA (in small batches of an evolution a cluster, hm_team.h) owns one
// Markov chain for the whole call: every two-site op of the Trotter schedule,
// the cluster measurement and the environment collapse run as a device-side
// loop over that chain's data.  On GB300 the binary64 pipe (about 2 DFMA per
// clock per SM) is the scarce unit of every step here.
//
// Steps (Sec. I.C.1): evolve (step 2) = theta GEMM + 9x9 gate + one-sided
// Jacobi SVD (found in binary32, finished in binary64) + truncation (Sec. II) +
// absorb, all in S^z charge blocks (Sec. II.C, hm_block.cuh); measure (step 3) = transfer matrices with S^z /
// S^+ / S^- insertions (Eq. H), contracted by charge block; collapse + reset
// (step 4, Eq. detailbalance1, Bell pairs of Sec. I.C), the reset writing the
// next initial state with its charges.  An S^x-basis sample is stored with
// every leg rotated by R (rows: the S^x eigenvectors), which exchanges S^x
// and S^z and leaves the gates and the Bell pairs unchanged, so it is blocked
// too; counters[2] records that frame for the measurement and the collapse.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <mutex>

#include "hm_block.cuh"
#include "hm_internal.h"
#include "hm_refine.cuh"
#include "hm_team.h"
#include "hm_transfer.cuh"

namespace hm {

namespace {

constexpr int NT = 256;          // threads per CTA
constexpr int kMaxSweeps = 60;   // one-sided Jacobi sweep budget
constexpr int TM = 64, TN = 64, TK = 16;

struct GemmSmem {
  double a[TK][TM + 1];
  double b[TK][TN + 1];
};

// Shared memory of the measurement, susceptibility and collapse kernels.
struct TransferSh {
  tr::Tabs tab;
  double red[NT / 32 * 3];
  double scal[2];
  int32_t ival;
};

// Dynamic shared memory of the evolve kernel: one CTA of 512 threads per SM,
// or two of 256 (a batch with more chains than SMs).  In turn the charge-run
// tables of a split, the decompositions of a wave of blocks, and finish()'s
// transposition tiles and value lists.
constexpr int kWideNT = 512;
constexpr size_t kWideSmem = 204 * 1024, kPairSmem = 104 * 1024;
static_assert(sizeof(blk::PrepTab) <= kPairSmem, "prepare's tables");
struct EvolveSh {
  blk::SplitSh split;
  blk::WaveSh wave;
  blk::GroupSh gs;
};

struct Shared {
  GemmSmem g;
  double red[NT / 32][4];
  double scal[8];
  int32_t ival[8];
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// C[M x N] = alpha op(A) op(B) (+ beta C), row-major.  TA: A stored K x M.
// TB: B stored N x K.  Whole CTA cooperates; ends with a barrier.
template <bool TA, bool TB>
__device__ void cta_gemm(int M, int N, int K, double alpha, const double* __restrict__ A, int lda,
                         const double* __restrict__ B, int ldb, double beta, double* __restrict__ C,
                         int ldc, GemmSmem& sm) {
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  for (int i0 = 0; i0 < M; i0 += TM) {
    for (int j0 = 0; j0 < N; j0 += TN) {
      double acc[4][4];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = 0.0;
      for (int k0 = 0; k0 < K; k0 += TK) {
        for (int e = tid; e < TM * TK; e += NT) {
          int ii, kk;
          if (TA) { ii = e % TM; kk = e / TM; } else { kk = e % TK; ii = e / TK; }
          const int gi = i0 + ii, gk = k0 + kk;
          double v = 0.0;
          if (gi < M && gk < K) v = TA ? A[(size_t)gk * lda + gi] : A[(size_t)gi * lda + gk];
          sm.a[kk][ii] = v;
        }
        for (int e = tid; e < TN * TK; e += NT) {
          int jj, kk;
          if (TB) { kk = e % TK; jj = e / TK; } else { jj = e % TN; kk = e / TN; }
          const int gj = j0 + jj, gk = k0 + kk;
          double v = 0.0;
          if (gj < N && gk < K) v = TB ? B[(size_t)gj * ldb + gk] : B[(size_t)gk * ldb + gj];
          sm.b[kk][jj] = v;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < TK; ++kk) {
          double a[4], b[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) a[r] = sm.a[kk][ty + 16 * r];
#pragma unroll
          for (int c = 0; c < 4; ++c) b[c] = sm.b[kk][tx + 16 * c];
#pragma unroll
          for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[r][c] = fma(a[r], b[c], acc[r][c]);
        }
        __syncthreads();
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int i = i0 + ty + 16 * r;
        if (i >= M) continue;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int j = j0 + tx + 16 * c;
          if (j >= N) continue;
          double v = alpha * acc[r][c];
          if (beta != 0.0) v += beta * C[(size_t)i * ldc + j];
          C[(size_t)i * ldc + j] = v;
        }
      }
    }
  }
  __syncthreads();
}

__device__ void set_error(const ChainDev* c, int code, int where, int32_t* ctx_err) {
  if (threadIdx.x == 0) {
    if (atomicCAS(c->status, 0, code) == 0) *c->err_where = where;
    if (ctx_err) atomicCAS(ctx_err, 0, code);
  }
}

// ---------------------------------------------------------------------------
// Step 2: one two-site op (Sec. I.A gates, Sec. II truncated SVD).
// ---------------------------------------------------------------------------

// One-sided (Hestenes) Jacobi on the q x p column-major matrix W (q >= p),
// accumulating the rotations in V (p x p).  Columns are paired by the
// round-robin tournament so that each round's pairs are disjoint; each warp
// rotates one pair at a time.  Returns sweeps used, or -1 if not converged.
__device__ int cta_jacobi(double* __restrict__ W, int q, int p, double* __restrict__ V, Shared& sh) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nwarps = NT / 32;
  for (int e = tid; e < p * p; e += NT) V[e] = (e % (p + 1) == 0) ? 1.0 : 0.0;
  const double tol = sqrt((double)q) * 2.220446049250313e-16;
  const int p2 = p + (p & 1);
  int done = 0;
  bool converged = false;
  double rmax = 0.0;
  while (done < kMaxSweeps) {
    if (tid == 0) {
      sh.ival[0] = 0;
      sh.scal[5] = 0.0;                 // largest rotation ratio of the sweep
    }
    __syncthreads();
    rmax = 0.0;
    for (int r = 0; r < p2 - 1; ++r) {
      for (int pi = warp; pi < p2 / 2; pi += nwarps) {
        int a, b;
        if (pi == 0) {
          a = r;
          b = p2 - 1;
        } else {
          a = (r + pi) % (p2 - 1);
          b = (r - pi + (p2 - 1)) % (p2 - 1);
        }
        if (a >= p || b >= p) continue;
        double* ca = W + (size_t)a * q;
        double* cb = W + (size_t)b * q;
        double al = 0.0, be = 0.0, ga = 0.0;
        for (int i = lane; i < q; i += 32) {
          const double x = ca[i], y = cb[i];
          al = fma(x, x, al);
          be = fma(y, y, be);
          ga = fma(x, y, ga);
        }
        al = warp_sum(al);
        be = warp_sum(be);
        ga = warp_sum(ga);
        if (ga != 0.0 && al > 0.0 && be > 0.0 && fabs(ga) > tol * sqrt(al) * sqrt(be)) {
          rmax = fmax(rmax, fabs(ga) / (sqrt(al) * sqrt(be)));
          const double zeta = (be - al) / (2.0 * ga);
          double t;
          if (fabs(zeta) > 1e150) t = 0.5 / zeta;
          else t = copysign(1.0, zeta) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
          const double cs = 1.0 / sqrt(1.0 + t * t), sn = cs * t;
          for (int i = lane; i < q; i += 32) {
            const double x = ca[i], y = cb[i];
            ca[i] = cs * x - sn * y;
            cb[i] = sn * x + cs * y;
          }
          double* va = V + (size_t)a * p;
          double* vb = V + (size_t)b * p;
          for (int i = lane; i < p; i += 32) {
            const double x = va[i], y = vb[i];
            va[i] = cs * x - sn * y;
            vb[i] = sn * x + cs * y;
          }
          if (lane == 0) sh.ival[0] = 1;
        }
      }
      __syncthreads();
    }
    if (lane == 0) atomicMax(reinterpret_cast<unsigned long long*>(&sh.scal[5]),
                             (unsigned long long)__double_as_longlong(rmax));
    __syncthreads();
    const int rotated = sh.ival[0];
    const double rm = sh.scal[5];
    __syncthreads();
    ++done;
    // no rotation: converged; all rotations tiny: quadratic convergence puts
    // the next sweep's off-diagonals (O(rm^2)) far below the tolerance
    if (!rotated || rm < 1e-9) {
      converged = true;
      break;
    }
  }
  return converged ? done : -1;
}

__device__ void two_site_op(ChainDev* c, const OpDev op, int t, Shared& sh, int32_t* ctx_err) {
  const int tid = threadIdx.x;
  const int k = op.k;
  const int chil = c->chi[k], chim = c->chi[k + 1], chir = c->chi[k + 2];
  const int m = 3 * chil, n = 3 * chir;
  double* Ak = c->site[k];
  double* Ak1 = c->site[k + 1];
  double* theta = c->theta;
  double* W = c->W;
  double* V = c->V;

  // theta[(l s1), (s2 r)] = sum_m A_k[(l s1), m] A_{k+1}[m, (s2 r)]
  cta_gemm<false, false>(m, n, chim, 1.0, Ak, chim, Ak1, n, 0.0, theta, n, sh.g);

  // Gate on the physical legs, written column-oriented for the Jacobi:
  // trans = 0: W (m x n col-major) = X;  trans = 1: W (n x m col-major) = X^T.
  const bool trans = n > m;
  const int q = trans ? n : m, p = trans ? m : n;
  const double* G = c->gates + (size_t)op.gate * 81;
  for (int e = tid; e < chil * chir; e += NT) {
    const int l = e / chir, r = e % chir;
    double th[9];
#pragma unroll
    for (int s1 = 0; s1 < 3; ++s1)
#pragma unroll
      for (int s2 = 0; s2 < 3; ++s2) th[3 * s1 + s2] = theta[(size_t)(3 * l + s1) * n + s2 * chir + r];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        double x = 0.0;
#pragma unroll
        for (int u = 0; u < 9; ++u) x = fma(G[(3 * a + b) * 9 + u], th[u], x);
        const int row = 3 * l + a, col = b * chir + r;
        if (!trans) W[(size_t)col * q + row] = x;
        else W[(size_t)row * q + col] = x;
      }
  }
  __syncthreads();

  const int sweeps = cta_jacobi(W, q, p, V, sh);
  if (sweeps < 0) {
    set_error(c, HM_ERR_NUMERIC, t, ctx_err);
    return;
  }

  // column norms (singular values), then rank-sort descending
  double* sig_raw = theta;               // theta is free now
  double* tail = theta + p;              // p + 1 doubles
  const int lane = tid & 31, warp = tid >> 5;
  for (int j = warp; j < p; j += NT / 32) {
    const double* cj = W + (size_t)j * q;
    double s2 = 0.0;
    for (int i = lane; i < q; i += 32) s2 = fma(cj[i], cj[i], s2);
    s2 = warp_sum(s2);
    if (lane == 0) sig_raw[j] = sqrt(s2);
  }
  __syncthreads();
  for (int j = tid; j < p; j += NT) {
    const double sj = sig_raw[j];
    int rank = 0;
    for (int i = 0; i < p; ++i) {
      const double si = sig_raw[i];
      rank += (si > sj) || (si == sj && i < j);
    }
    c->sig[rank] = sj;
    c->perm[rank] = j;
  }
  __syncthreads();
  if (tid == 0) {
    const double* s = c->sig;
    double total;
    int kk;
    double nrm = 1.0;
    if (!op.exact) {
      kk = blk::trunc_rank(s, p, c->chi_max, c->cutoff, tail, &total);
      if (!(total > 0.0) || !isfinite(total)) kk = -1;
      else {
        double kept = 0.0;
        for (int i = 0; i < kk; ++i) kept += s[i] * s[i];
        nrm = 1.0 / sqrt(kept);
        c->stats[ST_DISC] += tail[kk] / total;
      }
    } else {
      kk = 0;
      while (kk < p && kk < chim && s[kk] > 0.0) ++kk;
      if (kk == 0) kk = -1;
    }
    sh.ival[1] = kk;
    sh.scal[0] = nrm;
    if (kk > 0) {
      const double mm = (double)(m > n ? m : n), nn = (double)(m > n ? n : m);
      c->stats[ST_K1] += 2.0 * chil * 3.0 * chim * 3.0 * chir;
      c->stats[ST_K2] += 2.0 * 81.0 * chil * chir;
      c->stats[ST_SVD] += 4.0 * mm * mm * nn + 8.0 * mm * nn * nn + 9.0 * nn * nn * nn;
      c->stats[ST_SWEEPS] += sweeps;
      c->stats[ST_SPLITS] += 1.0;
      if (kk > c->stats[ST_MAXCHI]) c->stats[ST_MAXCHI] = kk;
    }
  }
  __syncthreads();
  const int kk = sh.ival[1];
  const double nrm = sh.scal[0];
  if (kk <= 0) {
    set_error(c, HM_ERR_NUMERIC, t, ctx_err);
    return;
  }
  const bool absorb_left = op.absorb == 0;
  // A_k[(l s), i] and A_{k+1}[i, (s r)] from the sorted singular triplets
  for (int e = tid; e < m * kk; e += NT) {
    const int row = e / kk, i = e % kk;
    const int j = c->perm[i];
    const double sg = c->sig[i];
    double v;
    if (!trans) {
      const double w = W[(size_t)j * q + row];   // = U sigma
      v = absorb_left ? w * nrm : w / sg;
    } else {
      const double u = V[(size_t)j * p + row];   // left vector
      v = absorb_left ? u * sg * nrm : u;
    }
    Ak[e] = v;
  }
  for (int e = tid; e < kk * n; e += NT) {
    const int i = e / n, col = e % n;
    const int j = c->perm[i];
    const double sg = c->sig[i];
    double v;
    if (!trans) {
      const double u = V[(size_t)j * p + col];   // right vector
      v = absorb_left ? u : u * sg * nrm;
    } else {
      const double w = W[(size_t)j * q + col];   // = V sigma
      v = absorb_left ? w / sg : w * nrm;
    }
    Ak1[e] = v;
  }
  __syncthreads();
  if (tid == 0) c->chi[k + 1] = kk;
  __syncthreads();
}

// Blocks of fewer columns go straight to the binary64 sweeps.  GB300, ms a
// Markov step with the line at 6, 12, 20 and 32 columns: one METTS chain of Lx = 4
// 17.6, 19.6, 22.3, 22.4; 4 chains of Lx = 4, 2W = 4 (chi = 64) 99, 98, 120, 132;
// 152 chains of Lx = 6, 2W = 4 (chi = 96) 254, 264, 312, 415.
constexpr int kPrecond = 6;
// Stopping ratios: of the binary64 sweeps (the next sweep's off-diagonals
// would be of order its square), and of the binary32 sweeps before them (what
// they leave, ~1e-6, is binary32 resolution).
constexpr double kStop64 = 1e-9;
constexpr float kStopPre = 1e-3f;

// Shared memory of a block, in doubles: W's part (W, leading dimension q | 1,
// or the binary32 stage before it: W, V and their norms), V (leading dimension
// p | 1), the column norms.
__device__ __forceinline__ int w_doubles(int q, int p) {
  return p * max(q | 1, (blk::ld4(q) + blk::ld4(p) + 2) / 2);
}
__device__ __forceinline__ int block_doubles(int q, int p) { return (w_doubles(q, p) + p * (p | 1) + p + 1) & ~1; }

// Decomposition of one block by the nw warps of a group: A (q x p, global) to W
// = A V with orthogonal columns and orthonormal V, both in shared memory.
//
// What bounds it is the binary64 pipe: a Jacobi sweep costs 4.5 q p^2 of its
// instructions, and from scratch it takes 7 to 10 sweeps.  The first ones only
// look for the vectors, and binary32 does that 64 x faster: binary32 sweeps on
// the rounded block give V to ~1e-6, two orthonormalisation steps V <- V - V (V^T V -
// 1) / 2 make it orthonormal to binary64 (the first on split binary32 sums, the
// second with p^3 / 2 binary64 products; both corrections are small enough to
// be multiplied in binary32), W = A V is formed in binary64 (q p^2), and the
// binary64 sweeps run from there under their own stopping rule, 2 or 3 of
// them, the last mostly tests.  So nothing of the binary32 stage reaches the
// result but the starting point.  KT: scratch, p ldk_of(p) floats (global).
// Returns the binary64 sweeps, or -1.
__device__ int decompose_block(const double* A, int q, int p, double* base, float* KT, int lw, int nw, int bar, int g,
                               blk::GroupSh& gs) {
  const int lane = threadIdx.x & 31, nthr = 32 * nw;
  const int ldw = q | 1, ldv = p | 1;
  double* W = base;
  double* V = base + w_doubles(q, p);
  double* nrm = V + (size_t)p * ldv;
  int pre = 0;
  if (p >= kPrecond) {
    const int lw4 = blk::ld4(q), lv4 = blk::ld4(p);
    float* W32 = reinterpret_cast<float*>(base);
    float* V32 = W32 + (size_t)p * lw4;
    float* n32 = V32 + (size_t)p * lv4;
    for (int j = lw; j < p; j += nw) {
      for (int i = lane; i < q; i += 32) W32[(size_t)j * lw4 + i] = blk::narrow(A[(size_t)j * q + i]);
      for (int i = lane; i < lv4; i += 32) V32[(size_t)j * lv4 + i] = i == j ? 1.0f : 0.0f;
    }
    blk::group_sync(bar, nthr);
    pre = blk::jacobi_group<float>(W32, q, lw4, p, V32, lv4, n32, lw, nw, bar, g, gs, kStopPre, kMaxSweeps);
    blk::group_sync(bar, nthr);
    if (pre > 0) {
      // V -> binary64, orthonormal
      refine::unit_terms(V32, p, lv4, n32, KT, lw, nw);
      blk::group_sync(bar, nthr);
      refine::pair_terms<true>(V32, p, lv4, p, n32, n32, KT, lw, nw);
      blk::group_sync(bar, nthr);
      int x = 0;
      refine::add_product<false>(V32, p, lv4, p, KT, V, ldv, lw, nw, x);
      blk::group_sync(bar, nthr);
      refine::ortho_terms64(V, p, ldv, KT, lw, nw);
      blk::group_sync(bar, nthr);
      x = 0;
      refine::add_product<true>(V32, p, lv4, p, KT, V, ldv, lw, nw, x);
      blk::group_sync(bar, nthr);
      refine::product64(A, q, p, V, ldv, W, ldw, lw, nw);
    }
  }
  if (pre <= 0) {
    // a small block, or binary32 did not converge: from A and V = 1
    for (int j = lw; j < p; j += nw) {
      for (int i = lane; i < q; i += 32) W[(size_t)j * ldw + i] = A[(size_t)j * q + i];
      for (int i = lane; i < p; i += 32) V[(size_t)j * ldv + i] = i == j ? 1.0 : 0.0;
    }
  }
  blk::group_sync(bar, nthr);
  return blk::jacobi_group<double, double, 2>(W, q, ldw, p, V, ldv, nrm, lw, nw, bar, g, gs, kStop64, kMaxSweeps);
}

// The sweeps of a block too large for shared memory, in global memory by the
// whole CTA.  Rare: kept out of line, away from the hot code.
__device__ HM_COLD int sweep_global(double* W, int q, int p, double* V, double* nrm, int warp, int nw,
                                         blk::GroupSh& gs) {
  return blk::jacobi_group<double, double, 2>(W, q, q, p, V, p, nrm, warp, nw, 1, 0, gs, kStop64, kMaxSweeps);
}

// One two-site op of a chain, block by block in the S^z charge of the new
// middle bond (Sec. II.C): theta by block GEMMs, the gate within its
// conserved sectors, the blocks' decompositions, then one truncation over the
// union of the blocks' singular values (Sec. II).  The blocks of a split that
// fit in shared memory together form a wave and are decomposed at once, each
// by its own warp group; a block too large for shared memory takes the whole
// CTA and works on global memory.
template <int NTE>
__device__ void two_site_op_blocked(ChainDev* c, const OpDev op, int t, double* buf, size_t buf_bytes, EvolveSh& sh,
                                    const blk::Team& tm, int32_t* ctx_err) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  blk::SplitSh& ss = sh.split;
  blk::WaveSh& wv = sh.wave;
  blk::PrepTab& tab = *reinterpret_cast<blk::PrepTab*>(buf);
  if (!blk::prepare<NTE>(c, op, ss, tab, tm)) blk::prepare<NTE>(c, op, ss, tab, tm);
  blk::theta_direct<NTE, double>(c, op.k, ss, c->theta, tm);
  const int64_t cap = (int64_t)(buf_bytes / sizeof(double));
  if (tid == 0) blk::own_blocks(ss, tm, wv, [&](int q, int p) { return block_doubles(q, p) <= cap; });
  __syncthreads();
  const int nown = wv.nown;
  {
    int c0 = 0;
    for (int i = 0; i < nown; ++i) {
      const blk::BlockRec& r = ss.b[blk::own_block(wv, i)];
      blk::gather_block<NTE, double, double>(c, op.k, ss, r, c->theta, c->W + r.woff, r.q, c->V + r.voff, r.p, c0);
    }
  }
  __syncthreads();
  int sweeps = 0;
  int64_t cost = -1;
  bool failed = false;
  for (int b0 = 0; b0 < nown && !failed;) {
    if (tid == 0) {
      int64_t used = 0;
      int n = 0, p[15], cost[15];
      while (b0 + n < nown && n < 15 && n < NTE / 32) {
        const blk::BlockRec& r = ss.b[blk::own_block(wv, b0 + n)];
        const int64_t need = block_doubles(r.q, r.p);
        if (used + need > cap) break;
        wv.off[n] = (int32_t)used;
        p[n] = r.p;
        cost[n] = blk::block_cost(r.q, r.p);
        used += need;
        ++n;
      }
      wv.b0 = b0;
      wv.n = n;
      wv.ng = n > 0 ? blk::assign_warps(p, cost, n, NTE / 32, wv.grp, wv.w0, wv.nw) : 0;
    }
    __syncthreads();
    const int n = wv.n;
    if (n == 0) {
      const blk::BlockRec& r = ss.b[blk::own_block(wv, b0)];
      const int sw = sweep_global(c->W + r.woff, r.q, r.p, c->V + r.voff, c->sig, warp, NTE / 32, sh.gs);
      if (sw < 0) {
        set_error(c, HM_ERR_NUMERIC, t, ctx_err);
        failed = true;
        break;
      }
      const int64_t cb = (int64_t)r.q * r.p * r.p;   // sweeps of the costliest block
      if (cb > cost) cost = cb, sweeps = sw;
      b0 += 1;
      __syncthreads();
      continue;
    }
    const int g = blk::my_group(wv, warp);
    for (int i = 0; g >= 0 && i < n; ++i) {
      if (wv.grp[i] != g) continue;
      const int ib = blk::own_block(wv, b0 + i);
      const blk::BlockRec& r = ss.b[ib];
      const int lw = warp - wv.w0[g], nw = wv.nw[g], q = r.q, p = r.p;
      double* W = buf + wv.off[i];
      // the transfer workspace is free during an evolution: it holds the K's
      const int sw = decompose_block(c->W + r.woff, q, p, W,
                                     reinterpret_cast<float*>(c->env_ws) + refine::k_offset(ss, ib), lw, nw, g + 1, g,
                                     sh.gs);
      if (lw == 0 && lane == 0) wv.sw[i] = sw;
      blk::group_sync(g + 1, 32 * nw);          // every warp's last rotations; the flags are free again
      const double* V = W + w_doubles(q, p);
      for (int j = lw; j < p; j += nw) {
        for (int e = lane; e < q; e += 32) c->W[r.woff + (size_t)j * q + e] = W[(size_t)j * (q | 1) + e];
        for (int e = lane; e < p; e += 32) c->V[r.voff + (size_t)j * p + e] = V[(size_t)j * (p | 1) + e];
      }
    }
    __syncthreads();
    for (int i = 0; i < n; ++i) {
      if (wv.sw[i] < 0) {
        set_error(c, HM_ERR_NUMERIC, t, ctx_err);
        failed = true;
        break;
      }
      const blk::BlockRec& r = ss.b[blk::own_block(wv, b0 + i)];
      const int64_t cb = (int64_t)r.q * r.p * r.p;
      if (cb > cost) cost = cb, sweeps = wv.sw[i];
    }
    b0 += n;
    __syncthreads();
  }
  // a failed decomposition ends in finish(), behind the team's barrier
  __syncthreads();
  constexpr int tiles = NTE / 32 * 8 * 33;
  char* scratch = reinterpret_cast<char*>(buf + tiles);
  const size_t need = blk::finish_bytes(ss.P);
  if (tiles * sizeof(double) + need > buf_bytes) scratch = reinterpret_cast<char*>(c->theta) + tm.rank * need;
  blk::finish<NTE>(c, op, t, ss, wv, tm, scratch, buf, ctx_err, sweeps, 0);
}

// team: CTAs of a cluster that share one chain (1: no cluster).
template <int NTE>
__device__ void evolve_chain(const BatchArg& b, const OutArg& o, double* buf, size_t buf_bytes, EvolveSh& sh, int team) {
  const blk::Team tm = {(int)blockIdx.x % team, team};
  ChainDev* c = b.c[blockIdx.x / team];
  const OpDev* ops = b.ops_override ? b.ops_override : c->ops;
  const int n_ops = b.ops_override ? b.n_override : c->n_ops;
  const int t0 = b.budget > 0 ? c->counters[4] : b.t0;
  const int t1 = b.budget > 0 ? min(t0 + b.budget, n_ops) : (b.t1 < n_ops ? b.t1 : n_ops);
  blk::team_sync(tm);                                        // every thread has read the cursor
  if (b.budget > 0 && threadIdx.x == 0 && tm.rank == 0) c->counters[4] = t1;
  for (int t = t0; t < t1; ++t) {
    // the team agrees: a CTA sets the status only behind a barrier of the op
    if (*(volatile int32_t*)c->status != 0) return;
    __syncthreads();
    two_site_op_blocked<NTE>(c, ops[t], t, buf, buf_bytes, sh, tm, o.ctx_err);
    blk::team_sync(tm);
  }
}

__global__ void __launch_bounds__(kWideNT, 1) evolve_fp64_wide_kernel(BatchArg b, OutArg o, int team) {
  extern __shared__ double2 dsm[];                           // 16-byte aligned: 128-bit loads of the columns
  __shared__ EvolveSh sh;
  evolve_chain<kWideNT>(b, o, reinterpret_cast<double*>(dsm), kWideSmem, sh, team);
}

__global__ void __launch_bounds__(NT, 2) evolve_fp64_pair_kernel(BatchArg b, OutArg o) {
  extern __shared__ double2 dsm[];
  __shared__ EvolveSh sh;
  evolve_chain<NT>(b, o, reinterpret_cast<double*>(dsm), kPairSmem, sh, 1);
}

// Step 3 (Sec. I.C.1): <S_i.S_j> and <Sz_i Sz_j> on every measured bond.
// Right environments are built explicitly from the last site (no reliance on
// the canonical form), so <psi|psi> is the full contraction and every value
// is divided by it.
__global__ void __launch_bounds__(NT) measure_fp64_kernel(BatchArg b, OutArg o) {
  __shared__ TransferSh sh;
  ChainDev* c = b.c[blockIdx.x];
  const int tid = threadIdx.x;
  double* out = o.obs + (size_t)blockIdx.x * o.n_obs;
  if (*(volatile int32_t*)c->status != 0) {
    for (int e = tid; e < o.n_obs; e += NT) out[e] = NAN;
    return;
  }
  const int64_t cc = (int64_t)c->chi_cap * c->chi_cap;
  double* Lp[2] = {c->env_ws, c->env_ws + cc};
  double* Ep[2] = {c->env_ws + 2 * cc, c->env_ws + 3 * cc};
  double* Z = c->env_ws + 4 * cc;          // 3 cc
  double* Et = c->env_ws + 7 * cc;         // cc
  double* Rp[2] = {c->env_ws + 8 * cc, c->env_ws + 9 * cc};
  double* Rend = c->env_ws + 10 * cc;      // one cc slot per distinct measured end site
  long long fma_n = 0;
  if (tid == 0) Rp[0][0] = 1.0;
  __syncthreads();
  // right sweep: R(pos) = environment of sites >= pos; keep R(b + 1) per end b
  int rc = 0;
  for (int pos = c->n_sites - 1; pos >= 0; --pos) {
    for (int q = 0; q < c->n_meas; ++q) {
      if (c->meas_j[q] == pos) {            // R(pos + 1) is current
        const int slot = c->meas_slot[q];
        const int n2 = c->chi[pos + 1] * c->chi[pos + 1];
        for (int e = tid; e < n2; e += NT) Rend[(size_t)slot * cc + e] = Rp[rc][e];
      }
    }
    __syncthreads();
    tr::right_transfer<NT>(c, pos, Rp[rc], 0, tr::op_id(), Rp[rc ^ 1], Z, false, false, sh.tab, fma_n);
    rc ^= 1;
  }
  const double nrm = Rp[rc][0];            // <psi|psi>
  if (tid == 0) Lp[0][0] = 1.0;
  __syncthreads();
  int pos = 0, cur = 0;
  double E_est = 0.0;
  // A chain in frame 1 stores R^N |psi> (R exchanges S^x and S^z, R S^z R =
  // S^x): there <Sz_i Sz_j> of |psi> is <Sx_i Sx_j> of the stored state,
  // which for a state of definite total S^z is (<S+_i S-_j> + <S-_i S+_j>)/4;
  // S_i.S_j is invariant.  Passes: (Sz Sz) and (S+ S-); the tensors are real,
  // so <S-_i S+_j>, the adjoint of <S+_i S-_j>, is the same number.
  const int frame = c->counters[2];
  const tr::Op1 ops1[2] = {tr::op_sz(), tr::op_sp()};
  const tr::Op1 ops2[2] = {tr::op_sz(), tr::op_sm()};
  int bi = 0;
  while (bi < c->n_meas) {
    const int a = c->meas_i[bi];
    int bend = bi;
    while (bend < c->n_meas && c->meas_i[bend] == a) ++bend;
    const int blast = c->meas_j[bend - 1];
    while (pos < a) {
      tr::left_transfer<NT>(c, pos, Lp[cur], 0, tr::op_id(), Lp[cur ^ 1], Z, false, false, sh.tab, fma_n);
      cur ^= 1;
      ++pos;
    }
    double vals[2][8];   // up to 8 bonds per start site
    for (int o1 = 0; o1 < 2; ++o1) {
      int ec = 0;
      int D = tr::left_transfer<NT>(c, a, Lp[cur], 0, ops1[o1], Ep[ec], Z, false, false, sh.tab, fma_n);
      for (int kk = a + 1; kk <= blast; ++kk) {
        for (int q = bi; q < bend; ++q) {
          if (c->meas_j[q] == kk) {
            const int D2 = tr::left_transfer<NT>(c, kk, Ep[ec], D, ops2[o1], Et, Z, false, false, sh.tab, fma_n);
            // the right environment has shift 0: another shift closes to 0
            vals[o1][q - bi] = D2 != 0 ? 0.0
                                       : tr::block_dot<NT>(sh.tab, 0, Et, Rend + (size_t)c->meas_slot[q] * cc,
                                                           c->chi[kk + 1], sh.red);
          }
        }
        if (kk < blast) {
          D = tr::left_transfer<NT>(c, kk, Ep[ec], D, tr::op_id(), Ep[ec ^ 1], Z, false, false, sh.tab, fma_n);
          ec ^= 1;
        }
      }
    }
    if (tid == 0) {
      for (int q = bi; q < bend; ++q) {
        const double pm = 2.0 * vals[1][q - bi] / nrm;
        const double ss = vals[0][q - bi] / nrm + 0.5 * pm;
        const double zz = frame ? 0.25 * pm : vals[0][q - bi] / nrm;
        out[1 + 2 * q] = ss;
        out[2 + 2 * q] = zz;
        E_est += c->meas_J[q] * ss;
      }
    }
    bi = bend;
  }
  if (tid == 0) {
    out[0] = E_est;
    c->stats[ST_TRANSFER] += 2.0 * (double)fma_n;
  }
}

// Uniform susceptibility (Eq. sus, Sec. II.A): the double sum
// sum_{a in M} sum_{b physical} <S_a . S_b> / <psi|psi>, written to o.obs[chain].
// A right sweep carries the plain right environment R and the running sums
// R_z, R_- of right environments with S^z, S^- inserted on every physical site
// to the right, and keeps all three at each region site a (R(a+1)); a left
// sweep carries the mirrored sums L, L_z, L_+ and closes, at each region site
// a, O_a on L against the right sums (b > a) and the left sums with O_a against R
// (b < a).  The tensors are real, so <S-_a S+_b>, the adjoint of <S+_a S-_b>, is
// the same number and takes no sums of its own.  Linear in the chain length.
// Charge blocks throughout: S^z leaves an environment's shift at 0, S^+ and
// S^- move it by the sign of the physical legs.  A chain whose physical
// positions hold legs of different signs (explicit op lists can leave it so)
// mixes shifts in one sum and is contracted densely.
__global__ void __launch_bounds__(NT) susceptibility_fp64_kernel(BatchArg b, OutArg o) {
  __shared__ TransferSh sh;
  ChainDev* c = b.c[blockIdx.x];
  const int tid = threadIdx.x;
  double* out = o.obs + blockIdx.x;
  if (*(volatile int32_t*)c->status != 0) {
    if (tid == 0) *out = NAN;
    return;
  }
  const int64_t cc = (int64_t)c->chi_cap * c->chi_cap;
  constexpr int NE = 3;                    // plain, S^z, S^- (right) or S^+ (left)
  double* Rc[NE];
  double* Rn[NE];
  double* Lc[NE];
  double* Ln[NE];
  for (int qq = 0; qq < NE; ++qq) {
    Rc[qq] = c->env_ws + qq * cc;
    Rn[qq] = c->env_ws + (4 + qq) * cc;
    Lc[qq] = c->env_ws + (8 + qq) * cc;
    Ln[qq] = c->env_ws + (12 + qq) * cc;
  }
  double* Z = c->env_ws + 16 * cc;         // 3 cc
  double* Et = c->env_ws + 19 * cc;
  double* store = c->env_ws + 20 * cc;     // 4 cc per region site
  const tr::Op1 ropk[NE] = {tr::op_id(), tr::op_sz(), tr::op_sm()};
  const tr::Op1 lopk[NE] = {tr::op_id(), tr::op_sz(), tr::op_sp()};
  // the one sign of the physical legs; dense when there is none
  int leg = 0;
  bool dense = false;
  for (int pos = 0; pos < c->n_sites; ++pos) {
    if (c->site_kind[pos] == SITE_ANC) continue;
    if (leg == 0) leg = c->sgn[pos];
    if (c->sgn[pos] != leg || leg == 0) dense = true;
  }
  if (dense) {
    leg = 0;
    blk::clear_forbidden<NT>(c);
  }
  // shifts of the right sums (bra minus ket charge) and of the left ones
  const int rD[NE] = {0, 0, leg};
  const int lD[NE] = {0, 0, leg};
  long long fma_n = 0;
  if (tid == 0) {
    Rc[0][0] = 1.0;
    Rc[1][0] = Rc[2][0] = 0.0;
    Lc[0][0] = 1.0;
    Lc[1][0] = Lc[2][0] = 0.0;
  }
  __syncthreads();
  const int n = c->n_sites;
  int amax = -1;
  for (int s2 = 0; s2 < c->n_region; ++s2) amax = max(amax, c->region[s2]);
  for (int pos = n - 1; pos >= 0; --pos) {
    const int cr = c->chi[pos + 1];
    int slot = -1;
    for (int s2 = 0; s2 < c->n_region; ++s2)
      if (c->region[s2] == pos) slot = s2;
    if (slot >= 0) {
      for (int qq = 0; qq < NE; ++qq)
        for (int e = tid; e < cr * cr; e += NT) store[(size_t)(4 * slot + qq) * cc + e] = Rc[qq][e];
      __syncthreads();
    }
    const bool phys = c->site_kind[pos] != SITE_ANC;
    for (int qq = 0; qq < NE; ++qq) {
      tr::right_transfer<NT>(c, pos, Rc[qq], rD[qq], tr::op_id(), Rn[qq], Z, false, dense, sh.tab, fma_n);
      if (qq > 0 && phys) tr::right_transfer<NT>(c, pos, Rc[0], 0, ropk[qq], Rn[qq], Z, true, dense, sh.tab, fma_n);
    }
    for (int qq = 0; qq < NE; ++qq) {
      double* t = Rc[qq];
      Rc[qq] = Rn[qq];
      Rn[qq] = t;
    }
  }
  const double nrm = Rc[0][0];             // <psi|psi>
  double total = 0.0;
  for (int pos = 0; pos <= amax; ++pos) {
    const int cr = c->chi[pos + 1];
    int slot = -1;
    for (int s2 = 0; s2 < c->n_region; ++s2)
      if (c->region[s2] == pos) slot = s2;
    if (slot >= 0) {
      const double* R0 = store + (size_t)(4 * slot) * cc;
      const double* Rz = R0 + cc;
      const double* Rm = R0 + 2 * cc;
      // b > a: O_a on L, closed against the right sums; b < a: the left sums
      // with O_a, closed against R
      const tr::Op1 oa[4] = {tr::op_sz(), tr::op_sp(), tr::op_sz(), tr::op_sm()};
      const double* right[4] = {Rz, Rm, R0, R0};
      for (int u = 0; u < 4; ++u) {
        const int from = u < 2 ? 0 : u - 1;
        const int D = tr::left_transfer<NT>(c, pos, Lc[from], lD[from], oa[u], Et, Z, false, dense, sh.tab, fma_n);
        total += tr::block_dot<NT>(sh.tab, D, Et, right[u], cr, sh.red);
      }
      total += 2.0 * nrm;                  // b = a: S.S = s(s+1) = 2
    }
    if (pos == amax) break;
    const bool phys = c->site_kind[pos] != SITE_ANC;
    for (int qq = 0; qq < NE; ++qq) {
      tr::left_transfer<NT>(c, pos, Lc[qq], lD[qq], tr::op_id(), Ln[qq], Z, false, dense, sh.tab, fma_n);
      if (qq > 0 && phys) tr::left_transfer<NT>(c, pos, Lc[0], 0, lopk[qq], Ln[qq], Z, true, dense, sh.tab, fma_n);
    }
    for (int qq = 0; qq < NE; ++qq) {
      double* t = Lc[qq];
      Lc[qq] = Ln[qq];
      Ln[qq] = t;
    }
  }
  if (tid == 0) {
    *out = total / nrm;
    c->stats[ST_TRANSFER] += 2.0 * (double)fma_n;
  }
}

// ---------------------------------------------------------------------------
// Step 4: collapse and reset.
// ---------------------------------------------------------------------------

__device__ __forceinline__ void philox_round(uint32_t& c0, uint32_t& c1, uint32_t& c2, uint32_t& c3,
                                             uint32_t k0, uint32_t k1) {
  const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
  const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
  const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
  c0 = n0;
  c1 = lo1;
  c2 = n2;
  c3 = lo0;
}

// Philox4x32-10 (Salmon et al., SC'11): counter (n, ordinal, seed_hi, 0),
// key (seed_lo, chain_id); u = ((x0 >> 5) 2^26 + (x1 >> 6)) 2^-53.
__device__ double philox_uniform(uint32_t n, uint32_t ordinal, uint32_t seed_hi, uint32_t seed_lo,
                                 uint32_t chain) {
  uint32_t c0 = n, c1 = ordinal, c2 = seed_hi, c3 = 0u;
  uint32_t k0 = seed_lo, k1 = chain;
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    philox_round(c0, c1, c2, c3, k0, k1);
  }
  return ((double)(c0 >> 5) * 67108864.0 + (double)(c1 >> 6)) * (1.0 / 9007199254740992.0);
}

// First b with u < cumulative p_b, else the last b with p_b > 0.
__device__ int choose3(const double p[3], double u) {
  double acc = 0.0;
  for (int b = 0; b < 3; ++b) {
    acc += p[b];
    if (u < acc) return b;
  }
  for (int b = 2; b >= 0; --b)
    if (p[b] > 0.0) return b;
  return -1;
}

__device__ void basis_rows(const ChainDev* c, int basis, double B[9]) {
  for (int i = 0; i < 9; ++i) B[i] = basis ? c->xbasis[i] : ((i % 4 == 0) ? 1.0 : 0.0);
}

// Sequential projective measurement of the environment, left to right, in the
// basis of sample n (Sec. I.C.1 step 4); cluster sites are traced out, which
// turns the boundary vector into a density matrix (Eq. detailbalance1).
__global__ void __launch_bounds__(NT) collapse_fp64_kernel(BatchArg b, OutArg o) {
  __shared__ TransferSh sh;
  ChainDev* c = b.c[blockIdx.x];
  const int tid = threadIdx.x;
  if (*(volatile int32_t*)c->status != 0) return;
  const int n_sample = c->counters[0];
  const int basis = (c->basis_zx && (n_sample & 1)) ? 1 : 0;
  // the measured basis as seen by the stored state: R maps the S^z basis to
  // the S^x basis and back (R e_b = v_b, R v_b = e_b), so a frame-1 state is
  // measured in the other basis; the outcome order is the same
  double B[9];
  basis_rows(c, basis ^ c->counters[2], B);
  const int64_t cc = (int64_t)c->chi_cap * c->chi_cap;
  double* R[2] = {c->env_ws, c->env_ws + cc};
  double* X = c->env_ws + 2 * cc;      // cl x 3cr
  double* Y = c->env_ws + 6 * cc;      // cl x cr
  long long fma_n = 0;
  int cur = 0;
  bool vec_mode = true;
  if (tid == 0) R[0][0] = 1.0;           // v = [1]
  __syncthreads();
  int e_ord = 0;
  double logp = 0.0;
  for (int k = 0; k < c->n_sites; ++k) {
    const double* A = c->site[k];
    const int cl = c->chi[k], cr = c->chi[k + 1];
    const int sg = c->sgn[k];
    const int16_t* qL = c->qn + (size_t)k * c->chi_cap;
    const int16_t* qR = qL + c->chi_cap;
    tr::build_tabs<NT>(c, k, false, sh.tab);
    if (c->site_kind[k] == SITE_ENV) {
      double q[3] = {0.0, 0.0, 0.0};
      // X[i, s, r] = sum_l rho[i, l] A[l, s, r]; a vector boundary is one row
      tr::row_times_site<NT>(c, k, sh.tab, R[cur], vec_mode ? 1 : cl, X);
      if (vec_mode) {
        for (int r = tid; r < cr; r += NT) {
          const double x0 = X[r], x1 = X[cr + r], x2 = X[2 * cr + r];
          for (int bb = 0; bb < 3; ++bb) {
            const double w = B[3 * bb] * x0 + B[3 * bb + 1] * x1 + B[3 * bb + 2] * x2;
            q[bb] = fma(w, w, q[bb]);
          }
        }
      } else {
        // q_b = sum_{s,t} B[b][s] B[b][t] G[s][t], G[s][t] = sum_{i,r} A[i,s,r] X[i,t,r]:
        // an (i, r) whose charges allow no s is skipped, and the others cost one
        // product per t instead of both basis rotations
        double G[9] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        for (int e = tid; e < cl * cr; e += NT) {
          const int i = e / cr, r = e % cr;
          const int m = (qR[r] - qL[i]) * sg;            // m(s) of the one allowed s (sg = 0: all)
          if (sg != 0 && (m < -1 || m > 1)) continue;
          const double* a = A + (size_t)i * 3 * cr + r;
          const double* x = X + (size_t)i * 3 * cr + r;
          const double x0 = x[0], x1 = x[cr], x2 = x[2 * cr];
#pragma unroll
          for (int s = 0; s < 3; ++s) {
            if (sg != 0 && m != blk::mval(s)) continue;
            const double as = a[s * cr];
            G[3 * s] = fma(as, x0, G[3 * s]);
            G[3 * s + 1] = fma(as, x1, G[3 * s + 1]);
            G[3 * s + 2] = fma(as, x2, G[3 * s + 2]);
          }
        }
#pragma unroll
        for (int bb = 0; bb < 3; ++bb)
#pragma unroll
          for (int s = 0; s < 3; ++s)
            q[bb] = fma(B[3 * bb + s], B[3 * bb] * G[3 * s] + B[3 * bb + 1] * G[3 * s + 1] + B[3 * bb + 2] * G[3 * s + 2],
                        q[bb]);
      }
      tr::block_sums<NT, 3>(q, sh.red);
      if (tid == 0) {
        const double tot = q[0] + q[1] + q[2];
        int pick = -1;
        double pb = 0.0;
        if (tot > 0.0 && isfinite(tot)) {
          const double p[3] = {q[0] / tot, q[1] / tot, q[2] / tot};
          if (o.cond)
            for (int bb = 0; bb < 3; ++bb) o.cond[((size_t)blockIdx.x * o.n_env + e_ord) * 3 + bb] = p[bb];
          const double u = philox_uniform((uint32_t)n_sample, (uint32_t)e_ord, c->seed_hi, c->seed_lo,
                                          c->chain_id);
          pick = choose3(p, u);
          if (pick >= 0) pb = p[pick];
        }
        sh.ival = pick;
        sh.scal[1] = pick >= 0 ? q[pick] : 0.0;
        if (pick >= 0) logp += log(pb);
      }
      __syncthreads();
      const int pick = sh.ival;
      const double qb = sh.scal[1];
      if (pick < 0) {
        set_error(c, HM_ERR_NUMERIC, 100000 + k, o.ctx_err);
        return;
      }
      if (tid == 0) {
        c->env_out[e_ord] = pick;
        if (o.env) o.env[(size_t)blockIdx.x * o.n_env + e_ord] = (int8_t)pick;
      }
      const double b0 = B[3 * pick], b1 = B[3 * pick + 1], b2 = B[3 * pick + 2];
      if (vec_mode) {
        const double sc = 1.0 / sqrt(qb);
        for (int r = tid; r < cr; r += NT)
          R[cur ^ 1][r] = (b0 * X[r] + b1 * X[cr + r] + b2 * X[2 * cr + r]) * sc;
        __syncthreads();
      } else {
        for (int e = tid; e < cl * cr; e += NT) {
          const int i = e / cr, r = e % cr;
          const double* x = X + (size_t)i * 3 * cr + r;
          Y[e] = b0 * x[0] + b1 * x[cr] + b2 * x[2 * cr];
        }
        __syncthreads();
        const double bv[3] = {b0, b1, b2};
        tr::site_times_rows<NT>(c, k, sh.tab, bv, 1.0 / qb, Y, 0, cr, R[cur ^ 1]);
        if (tid == 0) fma_n += (cl + cr) * tr::site_entries(sh.tab, sg);
      }
      cur ^= 1;
      ++e_ord;
    } else {
      if (vec_mode) {
        // rho = v v^T
        for (int e = tid; e < cl * cl; e += NT) R[cur ^ 1][e] = R[cur][e / cl] * R[cur][e % cl];
        __syncthreads();
        cur ^= 1;
        vec_mode = false;
      }
      const double one[3] = {1.0, 1.0, 1.0};
      tr::row_times_site<NT>(c, k, sh.tab, R[cur], cl, X);
      tr::site_times_rows<NT>(c, k, sh.tab, one, 1.0, X, cr, 3 * cr, R[cur ^ 1]);
      if (tid == 0) fma_n += (cl + cr) * tr::site_entries(sh.tab, sg);
      cur ^= 1;
    }
  }
  if (tid == 0) {
    if (o.logp) o.logp[blockIdx.x] = logp;
    c->counters[0] = n_sample + 1;
    c->counters[1] = basis;
    c->stats[ST_TRANSFER] += 2.0 * (double)fma_n;
  }
}

// Writes the initial state |i>_E |B>_C from env_out and counters[1]
// (Sec. I.C.1 step 1): environment sites (1,3,1) basis vectors, cluster
// physical sites delta(s, 2 - a)/sqrt(3) of shape (1,3,3), ancillas
// delta(2 - a, s) of shape (3,3,1) (the Bell bond ordered by ascending
// S^z charge).  An environment drawn in the S^x basis is stored in frame 1:
// every leg rotated by R (rows: the S^x eigenvectors), which maps the S^x
// eigenvector v_b to e_b and leaves the Bell pairs and the Heisenberg gates
// unchanged (R is real orthogonal and the gates commute with R (x) R), so
// every initial state is a product of S^z eigenstates and Bell pairs with
// definite total S^z, and every sample evolves in charge blocks (Sec. II.C).
// With draw_initial, first draws the environment in the Sz basis with
// p = 1/3 each and sample index n = -1.
__global__ void __launch_bounds__(NT) reset_kernel(BatchArg b, OutArg o, int draw_initial) {
  ChainDev* c = b.c[blockIdx.x];
  const int tid = threadIdx.x;
  if (*(volatile int32_t*)c->status != 0) return;
  if (draw_initial) {
    const double third = 1.0 / 3.0;
    const double p[3] = {third, third, third};
    for (int e = tid; e < c->n_env; e += NT) {
      const double u = philox_uniform(0xFFFFFFFFu, (uint32_t)e, c->seed_hi, c->seed_lo, c->chain_id);
      c->env_out[e] = choose3(p, u);
    }
    if (tid == 0) {
      c->counters[0] = 0;
      c->counters[1] = 0;
    }
    __syncthreads();
  }
  const double r3 = 1.0 / sqrt(3.0);
  // env ordinal of site k = number of env sites before k
  for (int k = tid; k < c->n_sites; k += NT) {
    double* A = c->site[k];
    const int kind = c->site_kind[k];
    if (kind == SITE_ENV) {
      int ord = 0;
      for (int s = 0; s < k; ++s) ord += c->site_kind[s] == SITE_ENV;
      const int pick = c->env_out[ord];
      for (int s = 0; s < 3; ++s) A[s] = s == pick ? 1.0 : 0.0;
      c->sgn[k] = 1;
    } else if (kind == SITE_CPHYS) {
      for (int e = 0; e < 9; ++e) A[e] = (e / 3 == 2 - e % 3) ? r3 : 0.0;     // A[0, s, a]
      c->sgn[k] = 1;
    } else {
      for (int e = 0; e < 9; ++e) A[e] = (e / 3 == 2 - e % 3) ? 1.0 : 0.0;    // A[a, s, 0]
      c->sgn[k] = -1;
    }
  }
  for (int i = tid; i <= c->n_sites; i += NT)
    c->chi[i] = (i > 0 && i < c->n_sites && c->site_kind[i - 1] == SITE_CPHYS) ? 3 : 1;
  if (tid == 0) {
    // bond charges: q_0 = 0, q_{k+1} = q_k + m(pick) after an environment
    // site; the Bell bond carries q_k + (-1, 0, +1); back to q_k after the ancilla
    const int cap = c->chi_cap;
    int q = 0, ord = 0;
    c->qn[0] = 0;
    for (int k = 0; k < c->n_sites; ++k) {
      const int kind = c->site_kind[k];
      int16_t* next = c->qn + (size_t)(k + 1) * cap;
      if (kind == SITE_ENV) {
        q += 1 - c->env_out[ord++];
        next[0] = (int16_t)q;
      } else if (kind == SITE_CPHYS) {
        next[0] = (int16_t)(q - 1);
        next[1] = (int16_t)q;
        next[2] = (int16_t)(q + 1);
      } else {
        next[0] = (int16_t)q;
      }
    }
    c->counters[2] = c->counters[1];
    c->counters[3] = 0;
    c->counters[4] = 0;
    c->counters[5] = 0;
  }
}

}  // namespace

static int check_launch() {
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? HM_OK : HM_ERR_CUDA;
}

int launch_evolve_fp64(const BatchArg& b, const OutArg& o, void* stream) {
  if (b.n <= 0) return HM_OK;
  // opt in to the dynamic shared memory once per device (a lock: serving
  // workers may launch from several host threads)
  static std::mutex mu;
  static bool ready[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return HM_ERR_CUDA;
  {
    std::lock_guard<std::mutex> lock(mu);
    if (dev < 0 || dev >= 64 || !ready[dev]) {
      if (cudaFuncSetAttribute(evolve_fp64_wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWideSmem) !=
              cudaSuccess ||
          cudaFuncSetAttribute(evolve_fp64_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPairSmem) !=
              cudaSuccess)
        return HM_ERR_CUDA;
      if (dev >= 0 && dev < 64) ready[dev] = true;
    }
  }
  const int sms = device_sm_count();
  if (sms > 0 && b.n > sms) {
    evolve_fp64_pair_kernel<<<b.n, NT, kPairSmem, (cudaStream_t)stream>>>(b, o);
  } else {
#if !defined(HM_HOST_EMULATION)
    const int team = team_size((const void*)evolve_fp64_wide_kernel, kWideNT, kWideSmem, b.n, b.chi_cap);
    if (team > 1) return launch_team(evolve_fp64_wide_kernel, b, o, team, kWideNT, kWideSmem, stream, team);
#endif
    evolve_fp64_wide_kernel<<<b.n, kWideNT, kWideSmem, (cudaStream_t)stream>>>(b, o, 1);
  }
  return check_launch();
}

int launch_measure_fp64(const BatchArg& b, const OutArg& o, void* stream) {
  if (b.n <= 0) return HM_OK;
  measure_fp64_kernel<<<b.n, NT, 0, (cudaStream_t)stream>>>(b, o);
  return check_launch();
}

int launch_susceptibility_fp64(const BatchArg& b, const OutArg& o, void* stream) {
  if (b.n <= 0) return HM_OK;
  susceptibility_fp64_kernel<<<b.n, NT, 0, (cudaStream_t)stream>>>(b, o);
  return check_launch();
}

int launch_collapse_fp64(const BatchArg& b, const OutArg& o, void* stream) {
  if (b.n <= 0) return HM_OK;
  collapse_fp64_kernel<<<b.n, NT, 0, (cudaStream_t)stream>>>(b, o);
  const int rc = check_launch();
  if (rc != HM_OK) return rc;
  reset_kernel<<<b.n, NT, 0, (cudaStream_t)stream>>>(b, o, 0);
  return check_launch();
}

int launch_reset(const BatchArg& b, const OutArg& o, int draw_initial, void* stream) {
  if (b.n <= 0) return HM_OK;
  reset_kernel<<<b.n, NT, 0, (cudaStream_t)stream>>>(b, o, draw_initial);
  return check_launch();
}

}  // namespace hm

// ---------------------------------------------------------------------------
// Allocation-free two-site update (hm_two_site_update_static).
//
// For callers that cannot allocate device memory: code running inside
// another library's memory pool, in a process whose allocator is owned by
// someone else, or on a path that must not allocate while it runs.  The scratch of the
// update (chain descriptor, site slots, theta, Jacobi matrices, singular
// values) lives in one file-scope device array of fixed size; every GPU that
// loads this library holds it until the process exits.  All calls share the
// array, so two calls whose kernels overlap on the GPU race on it.
// ---------------------------------------------------------------------------

namespace hm {
namespace {

constexpr int kStaticChi = 128;                                       // largest chi_l, chi_m, chi_r
constexpr int64_t kStaticSlot = (int64_t)kStaticChi * 3 * kStaticChi;  // one site tensor
constexpr int64_t kStaticWs = (int64_t)(3 * kStaticChi) * (3 * kStaticChi);
constexpr int kStaticSv = 3 * kStaticChi;
constexpr int64_t kStaticDoubles = 64 + 2 * kStaticSlot + 3 * kStaticWs + 2 * kStaticSv;

static __device__ __align__(256) double g_static_scratch[kStaticDoubles];
static_assert(sizeof(ChainDev) + 2 * sizeof(double*) + 6 * sizeof(int32_t) <= 48 * sizeof(double),
              "descriptor and meta data must fit below the statistics slots");

__global__ void __launch_bounds__(NT)
two_site_static_kernel(double* scratch, const double* A, const double* B, int chi_l, int chi_m, int chi_r,
                       const double* gate, int chi_max, double cutoff, int absorb, double* A_out,
                       double* B_out, int32_t* k_out) {
  __shared__ Shared sh;
  ChainDev* c = reinterpret_cast<ChainDev*>(scratch);
  char* meta = reinterpret_cast<char*>(scratch) + sizeof(ChainDev);   // 64 doubles hold struct + meta
  double** sites = reinterpret_cast<double**>(meta);
  int32_t* chi = reinterpret_cast<int32_t*>(meta + 2 * sizeof(double*));
  int32_t* status = chi + 4;
  double* stats = scratch + 48;
  double* slotA = scratch + 64;
  double* slotB = slotA + kStaticSlot;
  double* ws = slotB + kStaticSlot;
  if (threadIdx.x == 0) {
    // everything that must start at zero is cleared here, every call
    ChainDev d = {};
    d.n_sites = 2;
    d.n_gates = 1;
    d.chi_max = chi_max;
    d.cutoff = cutoff;
    d.gates = gate;
    d.site = sites;
    d.chi = chi;
    d.stats = stats;
    d.status = status;
    d.err_where = status + 1;
    d.theta = ws;
    d.W = ws + kStaticWs;
    d.V = ws + 2 * kStaticWs;
    d.sig = ws + 3 * kStaticWs;
    d.perm = reinterpret_cast<int32_t*>(ws + 3 * kStaticWs + kStaticSv);
    d.ws_cap = kStaticWs;
    d.sv_cap = kStaticSv;
    d.chi_cap = kStaticChi;
    *c = d;
    sites[0] = slotA;
    sites[1] = slotB;
    chi[0] = chi_l;
    chi[1] = chi_m;
    chi[2] = chi_r;
    status[0] = status[1] = 0;
    for (int i = 0; i < ST_N; ++i) stats[i] = 0.0;
  }
  for (int e = threadIdx.x; e < chi_l * 3 * chi_m; e += NT) slotA[e] = A[e];
  for (int e = threadIdx.x; e < chi_m * 3 * chi_r; e += NT) slotB[e] = B[e];
  __syncthreads();
  const OpDev op = {0, 0, absorb, 0};
  two_site_op(c, op, 0, sh, nullptr);
  __syncthreads();
  const int code = *(volatile int32_t*)status;
  const int kk = chi[1];
  if (code != 0) {
    if (threadIdx.x == 0) *k_out = code;
    return;
  }
  for (int e = threadIdx.x; e < chi_l * 3 * kk; e += NT) A_out[e] = slotA[e];
  for (int e = threadIdx.x; e < kk * 3 * chi_r; e += NT) B_out[e] = slotB[e];
  if (threadIdx.x == 0) *k_out = kk;
}

}  // namespace

}  // namespace hm

namespace {

std::mutex g_static_mu;
double* g_static_ptr[64] = {};   // device address of g_static_scratch, per device

}  // namespace

extern "C" int hm_two_site_update_static(const double* A_dev, const double* B_dev, int32_t chi_l, int32_t chi_m,
                                         int32_t chi_r, const double* gate_dev, int32_t chi_max, double cutoff,
                                         int32_t absorb, double* A_out_dev, double* B_out_dev,
                                         int32_t* k_out_dev, void* cuda_stream) {
  using namespace hm;
  if (!A_dev || !B_dev || !gate_dev || !A_out_dev || !B_out_dev || !k_out_dev) {
    set_global_error("hm_two_site_update_static: null pointer argument");
    return HM_ERR_ARG;
  }
  if (chi_l < 1 || chi_m < 1 || chi_r < 1 || chi_max < 1 || chi_l > kStaticChi || chi_m > kStaticChi ||
      chi_r > kStaticChi || chi_max > kStaticChi) {
    set_global_error("hm_two_site_update_static: chi_l, chi_m, chi_r and chi_max must lie in [1, 128] "
                     "(the size of its fixed scratch array)");
    return HM_ERR_ARG;
  }
  if ((absorb != 0 && absorb != 1) || !(cutoff >= 0.0) || !(cutoff < 1.0)) {
    set_global_error("hm_two_site_update_static: absorb must be 0 or 1 and cutoff in [0, 1)");
    return HM_ERR_ARG;
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    set_global_error("hm_two_site_update_static: no current CUDA device");
    return HM_ERR_CUDA;
  }
  double* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_static_mu);
    if (!g_static_ptr[dev]) {
      // one-time set-up on this device (the device is current here): the
      // host-side symbol is only a stand-in, the kernel needs the device address
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) {
        set_global_error("hm_two_site_update_static: cudaGetSymbolAddress of the scratch array failed");
        return HM_ERR_CUDA;
      }
      g_static_ptr[dev] = static_cast<double*>(p);
    }
    scratch = g_static_ptr[dev];
  }
  two_site_static_kernel<<<1, NT, 0, (cudaStream_t)cuda_stream>>>(scratch, A_dev, B_dev, chi_l, chi_m, chi_r,
                                                                  gate_dev, chi_max, cutoff, absorb, A_out_dev,
                                                                  B_out_dev, k_out_dev);
  if (cudaGetLastError() != cudaSuccess) {
    set_global_error("hm_two_site_update_static: kernel launch failed");
    return HM_ERR_CUDA;
  }
  return HM_OK;
}
