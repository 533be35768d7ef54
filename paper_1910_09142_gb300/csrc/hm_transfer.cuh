// Transfer matrices of the measurement, the collapse and the susceptibility
// (steps 3 and 4 of Sec. I.C.1), contracted by S^z charge (Sec. II.C).
//
// What bounds them: GB300 issues about 2 binary64 FMA per clock and SM, so a
// warp's binary64 instruction takes 16 clocks whatever its idle lanes, and
// everything else (loads, index arithmetic) is nearly free beside it.  The
// charge blocks of a transfer are small (10 to 60 on a side) and there are 20
// to 40 of them.  So a transfer is two passes over the union of its blocks,
// with one output element a thread and the elements of a block dense over the
// lanes: no padding to a tile, no shared-memory staging, and two barriers a
// transfer instead of two per K tile and block.  The operands are read
// straight through L1 (a block is a few KB; one of the two loads is a
// broadcast, the other is contiguous over the lanes).
#pragma once

#include <cstdint>

#include "hm_block.cuh"
#include "hm_internal.h"

namespace hm {
namespace tr {

// One-site operator with at most one entry a row: <s|O|t[s]> = w[s] (0: an
// empty row), all with m(s) - m(t) = d.
struct Op1 {
  int t[3];
  double w[3];
  int d;
};

constexpr double kR2 = 1.4142135623730951;
__device__ __forceinline__ Op1 op_id() { return {{0, 1, 2}, {1.0, 1.0, 1.0}, 0}; }
__device__ __forceinline__ Op1 op_sz() { return {{0, 1, 2}, {1.0, 0.0, -1.0}, 0}; }
// S+ = sqrt(2) (|+1><0| + |0><-1|); S- its transpose (basis m = +1, 0, -1)
__device__ __forceinline__ Op1 op_sp() { return {{1, 2, 0}, {kR2, kR2, 0.0}, 1}; }
__device__ __forceinline__ Op1 op_sm() { return {{0, 0, 1}, {0.0, kR2, kR2}, -1}; }

// Charge runs of the two bonds of a site (shared memory): charge q0 + x owns
// the bond indices [st, en).  A dense view is one run with charge 0.
struct Tabs {
  int32_t q0[2], nq[2];
  int32_t st[2][blk::kWin], en[2][blk::kWin];
};

__device__ __forceinline__ blk::Seg run_of(const Tabs& t, int b, int Q) {
  const int x = Q - t.q0[b];
  if (x < 0 || x >= t.nq[b]) return {0, 0};
  return {t.st[b][x], t.en[b][x] - t.st[b][x]};
}

// Runs of the bonds left and right of site pos.  Bond indices are grouped by
// charge, ascending, and a bond's charges span less than kWin (the evolution
// switches a chain to dense mode otherwise: every charge 0).
template <int NT>
__device__ void build_tabs(const ChainDev* c, int pos, bool dense, Tabs& t) {
  __syncthreads();                          // the previous site's tables are no longer read
  for (int b = 0; b < 2; ++b) {
    const int n = c->chi[pos + b];
    const int16_t* q = c->qn + (size_t)(pos + b) * c->chi_cap;
    const int q0 = dense ? 0 : q[0];
    const int nq = dense ? 1 : min(q[n - 1] - q0 + 1, blk::kWin);
    if (threadIdx.x == 0) {
      t.q0[b] = q0;
      t.nq[b] = nq;
    }
    for (int x = threadIdx.x; x < nq; x += NT) t.st[b][x] = t.en[b][x] = 0;
  }
  __syncthreads();
  for (int b = 0; b < 2; ++b) {
    const int n = c->chi[pos + b];
    const int16_t* q = c->qn + (size_t)(pos + b) * c->chi_cap;
    for (int e = threadIdx.x; e < n; e += NT) {
      const int Q = dense ? 0 : q[e];
      if (e == 0 || (!dense && q[e - 1] != Q)) t.st[b][Q - t.q0[b]] = e;
      if (e == n - 1 || (!dense && q[e + 1] != Q)) t.en[b][Q - t.q0[b]] = e + 1;
    }
  }
  __syncthreads();
}

using blk::share;

// Sum over k < n of x[k sx] y[k sy].
__device__ __forceinline__ double dot_strided(const double* __restrict__ x, size_t sx, const double* __restrict__ y,
                                              size_t sy, int n, double acc) {
#pragma unroll 4
  for (int k = 0; k < n; ++k) acc = fma(x[k * sx], y[k * sy], acc);
  return acc;
}

// Left environment through site pos with operator o:
// Eout[i', j'] (+)= sum_{s,t} O[s][t] sum_{i,j} A[i,s,i'] Ein[i,j] A[j,t,j'].
// Ein[i, j] (bra i, ket j) is nonzero only where q_i - q_j = D; the result
// has shift D + sigma d (returned), and only its blocks are written.
// Z: scratch of 3 cl cr doubles.  fma_n: multiply-adds so far (an integer: a
// binary64 counter would itself cost the binary64 pipe).
template <int NT>
__device__ int left_transfer(const ChainDev* c, int pos, const double* Ein, int D, const Op1& o, double* Eout,
                             double* Z, bool acc, bool dense, Tabs& tb, long long& fma_n) {
  build_tabs<NT>(c, pos, dense, tb);
  const int cl = c->chi[pos], cr = c->chi[pos + 1];
  const double* __restrict__ A = c->site[pos];
  const int sg = dense ? 0 : c->sgn[pos];
  const int D2 = D + sg * o.d;
  for (int pass = 0; pass < 2; ++pass) {
    int c0 = 0;
    size_t zo = 0;
    for (int x = 0; x < tb.nq[1]; ++x) {
      const int Qb = tb.q0[1] + x, Qk = Qb - D2;
      const blk::Seg b = run_of(tb, 1, Qb), k = run_of(tb, 1, Qk);   // bra and ket run
      if (b.len == 0 || k.len == 0) continue;
      int is[3], il[3];
      size_t z[3];
      for (int s = 0; s < 3; ++s) {
        const blk::Seg i = run_of(tb, 0, Qb - sg * blk::mval(s));
        const blk::Seg j = run_of(tb, 0, Qk - sg * blk::mval(o.t[s]));
        is[s] = i.start;
        il[s] = o.w[s] != 0.0 && j.len > 0 ? i.len : 0;
        z[s] = zo;
        zo += (size_t)il[s] * k.len;
        if (il[s] == 0) continue;
        if (pass == 0) {
          // Z (il x kl) = w Ein[i-run, j-run] A[j-run, t, k-run]
          double* zz = Z + z[s];
          const double* y0 = A + ((size_t)3 * j.start + o.t[s]) * cr + k.start;
          const double* x0 = Ein + (size_t)i.start * cl + j.start;
          const double w = o.w[s];
          const int kl = k.len, jl = j.len;
          share<NT>(i.len * kl, c0, [&](int e) {
            const int r = e / kl, q = e - r * kl;
            zz[e] = w * dot_strided(x0 + (size_t)r * cl, 1, y0 + q, (size_t)3 * cr, jl, 0.0);
          });
          fma_n += (long long)i.len * jl * kl;
        } else {
          fma_n += (long long)i.len * b.len * k.len;
        }
      }
      if (pass == 1) {
        // Eout[b-run, k-run] (+)= sum_s A[i-run, s, b-run]^T Z_s
        double* out = Eout + (size_t)b.start * cr + k.start;
        const int kl = k.len;
        share<NT>(b.len * kl, c0, [&](int e) {
          const int r = e / kl, q = e - r * kl;
          double* dst = out + (size_t)r * cr + q;
          double v = acc ? *dst : 0.0;
#pragma unroll
          for (int s = 0; s < 3; ++s)
            v = dot_strided(A + ((size_t)3 * is[s] + s) * cr + b.start + r, (size_t)3 * cr, Z + z[s] + q, kl, il[s], v);
          *dst = v;
        });
      }
    }
    __syncthreads();
  }
  return D2;
}

// Right environment through site pos with operator o:
// Rout[i, j] (+)= sum_{s,t} O[s][t] sum_{a,b} A[i,s,a] Rin[a,b] A[j,t,b].
// Rin has shift D (q_a - q_b = D); the result has shift D - sigma d
// (returned).  Y: scratch of 3 cl cr doubles; the intermediate is kept
// transposed, so that both passes read one operand contiguously over the lanes.
template <int NT>
__device__ int right_transfer(const ChainDev* c, int pos, const double* Rin, int D, const Op1& o, double* Rout,
                              double* Y, bool acc, bool dense, Tabs& tb, long long& fma_n) {
  build_tabs<NT>(c, pos, dense, tb);
  const int cl = c->chi[pos], cr = c->chi[pos + 1];
  const double* __restrict__ A = c->site[pos];
  const int sg = dense ? 0 : c->sgn[pos];
  const int D2 = D - sg * o.d;
  for (int pass = 0; pass < 2; ++pass) {
    int c0 = 0;
    size_t yo = 0;
    for (int x = 0; x < tb.nq[0]; ++x) {
      const int Qi = tb.q0[0] + x, Qj = Qi - D2;
      const blk::Seg i = run_of(tb, 0, Qi), j = run_of(tb, 0, Qj);
      if (i.len == 0 || j.len == 0) continue;
      int bs[3], bl[3];
      size_t y[3];
      for (int s = 0; s < 3; ++s) {
        const blk::Seg a = run_of(tb, 1, Qi + sg * blk::mval(s));
        const blk::Seg b = run_of(tb, 1, Qj + sg * blk::mval(o.t[s]));
        bs[s] = b.start;
        bl[s] = o.w[s] != 0.0 && a.len > 0 ? b.len : 0;
        y[s] = yo;
        yo += (size_t)bl[s] * i.len;
        if (bl[s] == 0) continue;
        if (pass == 0) {
          // Y^T (bl x il) = w (A[i-run, s, a-run] Rin[a-run, b-run])^T
          double* yy = Y + y[s];
          const double* x0 = A + ((size_t)3 * i.start + s) * cr + a.start;
          const double* r0 = Rin + (size_t)a.start * cr + b.start;
          const double w = o.w[s];
          const int n = b.len, al = a.len, il = i.len;
          share<NT>(il * n, c0, [&](int e) {
            const int r = e / n, q = e - r * n;
            yy[(size_t)q * il + r] = w * dot_strided(x0 + (size_t)r * 3 * cr, 1, r0 + q, cr, al, 0.0);
          });
          fma_n += (long long)il * al * n;
        } else {
          fma_n += (long long)i.len * j.len * bl[s];
        }
      }
      if (pass == 1) {
        // Rout[i-run, j-run] (+)= sum_s Y_s A[j-run, t, b-run]^T
        double* out = Rout + (size_t)i.start * cl + j.start;
        const int il = i.len;
        share<NT>(j.len * il, c0, [&](int e) {
          const int r = e / il, q = e - r * il;              // column r of the block, row q
          double* dst = out + (size_t)q * cl + r;
          double v = acc ? *dst : 0.0;
#pragma unroll
          for (int s = 0; s < 3; ++s)
            v = dot_strided(A + ((size_t)3 * (j.start + r) + o.t[s]) * cr + bs[s], 1, Y + y[s] + q, il, bl[s], v);
          *dst = v;
        });
      }
    }
    __syncthreads();
  }
  return D2;
}

// Block-wide sums of N values, the result in every thread.  red: NT / 32 x N
// doubles of shared memory.
template <int NT, int N>
__device__ void block_sums(double (&v)[N], double* red) {
  constexpr int NW = NT / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < N; ++q) v[q] = blk::warp_sum64(v[q]);
  __syncthreads();
  if (lane == 0)
    for (int q = 0; q < N; ++q) red[warp * N + q] = v[q];
  __syncthreads();
#pragma unroll
  for (int q = 0; q < N; ++q) {
    double a = red[(lane % NW) * N + q];
#pragma unroll
    for (int w = NW / 2; w > 0; w >>= 1) a += __shfl_xor_sync(0xffffffffu, a, w);
    v[q] = a;
  }
}

// sum X[k, l] Y[k, l] over the blocks q_k - q_l = D of bond pos + 1 (the
// right bond of the tables built last); X and Y have leading dimension n.
template <int NT>
__device__ double block_dot(const Tabs& tb, int D, const double* __restrict__ X, const double* __restrict__ Y, int n,
                            double* red) {
  double v[1] = {0.0};
  int c0 = 0;
  for (int x = 0; x < tb.nq[1]; ++x) {
    const int Q = tb.q0[1] + x;
    const blk::Seg k = run_of(tb, 1, Q), l = run_of(tb, 1, Q - D);
    if (k.len == 0 || l.len == 0) continue;
    const size_t o = (size_t)k.start * n + l.start;
    share<NT>(k.len * l.len, c0, [&](int e) {
      const int r = e / l.len, q = e - r * l.len;
      v[0] = fma(X[o + (size_t)r * n + q], Y[o + (size_t)r * n + q], v[0]);
    });
  }
  block_sums<NT, 1>(v, red);
  return v[0];
}

// Entries of the site's tensor that its charges allow.
__device__ __forceinline__ long long site_entries(const Tabs& tb, int sg) {
  long long n = 0;
  for (int x = 0; x < tb.nq[1]; ++x)
    for (int s = 0; s < 3; ++s)
      n += (long long)(tb.en[1][x] - tb.st[1][x]) * run_of(tb, 0, tb.q0[1] + x - sg * blk::mval(s)).len;
  return n;
}

// X[i, s, r] = sum_j rho[i, j] A[j, s, r] for a rho without charge structure
// (the collapse measures in the basis conjugate to the stored one); A's
// structure leaves one run of j per (s, r).  rho: rows x cl; X: rows x 3 cr.
// Tables of site pos.
template <int NT>
__device__ void row_times_site(const ChainDev* c, int pos, const Tabs& tb, const double* rho, int rows, double* X) {
  const int cl = c->chi[pos], cr = c->chi[pos + 1];
  const double* __restrict__ A = c->site[pos];
  const int16_t* qR = c->qn + (size_t)(pos + 1) * c->chi_cap;
  const int sg = c->sgn[pos];
  const int n = rows * 3 * cr;
  for (int e = threadIdx.x; e < n; e += NT) {
    const int i = e / (3 * cr), col = e - i * 3 * cr;
    const int s = col / cr;
    const blk::Seg j = run_of(tb, 0, qR[col - s * cr] - sg * blk::mval(s));
    X[e] = dot_strided(rho + (size_t)i * cl + j.start, 1, A + (size_t)3 * j.start * cr + col, (size_t)3 * cr, j.len, 0.0);
  }
  __syncthreads();
}

// Eout[a, r] = scale sum_s b_s sum_i A[i, s, a] Y_s[i, r], i over the one run
// A's structure leaves per (s, a); Y_s = Y + s soff, leading dimension ldy.
// A row with b_s = 0 is skipped.  Tables of site pos.
template <int NT>
__device__ void site_times_rows(const ChainDev* c, int pos, const Tabs& tb, const double (&b)[3], double scale,
                                const double* Y, int soff, int ldy, double* Eout) {
  const int cr = c->chi[pos + 1];
  const double* __restrict__ A = c->site[pos];
  const int16_t* qR = c->qn + (size_t)(pos + 1) * c->chi_cap;
  const int sg = c->sgn[pos];
  for (int e = threadIdx.x; e < cr * cr; e += NT) {
    const int a = e / cr, r = e - a * cr;
    double v = 0.0;
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      if (b[s] == 0.0) continue;
      const blk::Seg i = run_of(tb, 0, qR[a] - sg * blk::mval(s));
      const double d = dot_strided(A + ((size_t)3 * i.start + s) * cr + a, (size_t)3 * cr,
                                   Y + (size_t)i.start * ldy + s * soff + r, ldy, i.len, 0.0);
      v = fma(b[s], d, v);
    }
    Eout[e] = scale * v;
  }
  __syncthreads();
}

}  // namespace tr
}  // namespace hm
