// Binary64 finish of a block that the binary32 Jacobi sweeps have
// diagonalised (HM_MIXED), without a binary64 sweep.
//
// After the sweeps W (q x p, binary32, shared memory) has columns that are
// orthogonal to E ~ 1e-6 relative, and V its rotations.  A binary64 Jacobi
// sweep on W takes 2.5 q p^2 instructions of the binary64 pipe (2 a clock and
// SM): 1.2 M clocks at q = p = 100.  Its rotations
// are tiny, so to first order they commute and the whole sweep is one product
//   W' = W (I + K),  V' = V (I + K),  K_ij = -K_ji = tan of pair (i, j),
// with K ~ 1e-6: a binary32 product K-wise gives W' to 1e-13 and leaves
// off-diagonals of order E^2, as the sweep does.  What needs more than
// binary32 is E itself.  W holds binary32 numbers, so a product of two of its
// entries splits exactly into two binary32 numbers, and a sum against a
// constant larger than every partial sum splits exactly too: dot2 below spends
// seven binary32 instructions a term (64 x the rate of the binary64 pipe) and
// returns the Gram entry to about 2^-45 of the columns' norms.  Measured on Lx =
// 16, 2W = 8, chi = 256 (256 chains, beta = 0.3) when it was made: the evolution
// 1043 -> 800 ms, sweep, promotion to binary64 and the scales together 37 -> about
// 15 % of it (the whole step is 392 ms with the steps after it).
//
// Two columns of nearly the same norm have a large angle whatever their
// overlap; their pairs (|b - a| < kNear max(a, b)) are left out of K and
// rotated one after another in binary64 afterwards.  When too many pairs are near (an
// exactly degenerate spectrum), or E is not small, the binary64 sweeps of
// jacobi_group run on W' and V' as well; they run on W and V themselves when a
// state of unknown norm has columns outside binary32's range (column_terms).
//
// What is left, on the CPU emulation of this code (blocks of 11 to 73 columns):
// relative overlaps of W's columns of 1e-13 to 1e-10, as after a binary64 sweep on
// the same blocks (at 147 to 162 columns, measured, 6e-10 to 2e-9 against the
// sweep's 1e-10 to 5e-10), but up to E where three or more values lie close together
// (2e-7 to 3e-7 on triple and six-fold values; 2e-7 to 4e-7 after the sweep).
// Rotating such clusters down to 1e-9 took 1 to 4 % of a step.  V's columns have
// length 1 to 1e-12 and overlap by the binary32 sweeps' ~1e-6, and W - theta V is
// 1e-6 of the largest entry, with either finish: the binary32 rotations are what
// HM_MIXED resolves.
//
// The columns of V come out of the sweeps up to ~1e-5 longer than 1 (a
// binary32 rotation with a small angle has cosine exactly 1, so it stretches
// both columns by sqrt(1 + t^2), always the same way).  Left in, that weights
// each kept vector: a systematic energy error of ~2e-5 (measured).  The
// rotations stay conformal and W = theta V holds column by column, so column
// j of both factors is scaled by 1 / |v_j| = 1 + delta_j; delta is K's diagonal.
#pragma once

#include <cstdint>

#include "hm_block.cuh"
#include "hm_internal.h"

namespace hm {
namespace refine {

// Relative gap of two squared column norms below which a pair is rotated
// explicitly.  Outside it |t| < E / 0.02 ~ 1e-4, and the terms the first
// order leaves out are below 1e-4 E.
constexpr float kNear = 0.02f;

// Squared norm above which a sum of binary32 products may overflow (Dot2's
// constant is up to 24 times the norm).
constexpr float kHuge32 = 1e36f;

// What a block's largest |E| becomes when a column lies outside [kTiny32, kHuge32].
constexpr float kOutOfRange = 4.0f;

// A value as an unevaluated binary32 sum.
struct F2 {
  float h, l;
};

// Sum of two F2 (Knuth's exact two-sum on the leading parts).
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  const float s = a.h + b.h, bb = s - a.h;
  const float e = (a.h - (s - bb)) + (b.h - bb);
  return {s, e + a.l + b.l};
}

__device__ __forceinline__ F2 normal2(F2 a) {
  const float s = a.h + a.l;
  return {s, a.l - (s - a.h)};
}

// Two running dot products (of the even and the odd rows): t = big + the
// products rounded to big's last bit, l = everything below.  big > 2 |every
// partial sum|, so t + p, (t + p) - t and p - ((t + p) - t) are exact splits
// (Dekker's fast two-sum).  Seven packed instructions for two terms.
struct Dot2 {
  float2 t, l;
  __device__ __forceinline__ void start(float big) {
    t = {big, big};
    l = {0.0f, 0.0f};
  }
  // ny = -y
  __device__ __forceinline__ void add(float2 x, float2 y, float2 ny) {
    const float2 p = blk::mul2(x, y);
    const float2 e = blk::fma2(x, ny, p);                  // -(the product's low part)
    const float2 s = blk::add2p(t, p);
    l = blk::add2p(l, blk::sub2p(p, blk::sub2p(s, t)));
    l = blk::sub2p(l, e);
    t = s;
  }
  __device__ __forceinline__ F2 get(float big) const { return add2({t.x - big, l.x}, {t.y - big, l.y}); }
};

// Power of two above 4 x (x > 0, normal).
__device__ __forceinline__ float above(float x) {
  return __uint_as_float((__float_as_uint(x) & 0x7f800000u) + (3u << 23));
}

// Shared-memory floats a block needs besides W and V: squared norms (high and
// low part), delta.
__device__ __forceinline__ int extra(int p) { return 3 * p; }

// Leading dimension of K's transpose (four entries are loaded at once).
__device__ __forceinline__ int ldk_of(int p) { return (p + 3) & ~3; }

// Offset (floats, a multiple of 4) of block b's K in the chain's scratch.
__device__ __forceinline__ int k_offset(const blk::SplitSh& s, int b) {
  int k = 0;
  for (int i = 0; i < b; ++i) k += s.b[i].p * ldk_of(s.b[i].p);
  return k;
}

__device__ __forceinline__ bool near_pair(float a, float b) { return fabsf(b - a) < kNear * fmaxf(a, b); }

// Squared norm of a column (zero rows up to a multiple of four) by its eight
// lanes; top: about its size, not below half of it.
__device__ __forceinline__ F2 norm2(const float* x, int n, float top) {
  const int sl = threadIdx.x & 7;
  const float big = above(fmaxf(top, 1e-36f));
  Dot2 d;
  d.start(big);
  for (int r = 4 * sl; r < n; r += 32) {
    const float4 v = *reinterpret_cast<const float4*>(x + r);
    d.add({v.x, v.y}, {v.x, v.y}, {-v.x, -v.y});
    d.add({v.z, v.w}, {v.z, v.w}, {-v.z, -v.w});
  }
  F2 s = d.get(big);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1)
    s = add2(s, {__shfl_xor_sync(0xffffffffu, s.h, o), __shfl_xor_sync(0xffffffffu, s.l, o)});
  return normal2(s);
}

// x' = x + (x delta + products with K): one column entry, binary64.
__device__ __forceinline__ double corrected(float x, float corr) { return blk::widen(x) + blk::widen(corr); }

// delta_j and the squared norms of the columns (ah holds the sweeps' running
// ones); KT: zeroed padding and the diagonal.  W and V: zero rows up to a
// multiple of four (jacobi_regs leaves them so; padded here for the other
// orderings by pad_rows).  Eight lanes a column.  check: returns whether this lane saw
// a nonzero column that the binary32 sweeps have left alone (blk::kTiny32) or
// cannot sum (kHuge32).  In a state of norm 1 a column shorter than 1e-15 lies
// below the resolution of theta itself, and swept in binary64 it only shrinks
// on (a null column loses 16 digits a sweep: 3 % of a step at Lx = 6, chi = 96, 304 chains).
__device__ inline bool column_terms(const float* W, int q, int ldw, const float* V, int p, int ldv, float* ah, float* al,
                                    float* dl, float* KT, int lw, int nw, bool check = false) {
  const int sub = (threadIdx.x & 31) >> 3, sl = threadIdx.x & 7;
  const int ldk = ldk_of(p);
  bool out = false;
  for (int j0 = 4 * lw; j0 < p; j0 += 4 * nw) {
    const int j = j0 + sub, jj = j < p ? j : p - 1;
    const F2 a = norm2(W + (size_t)jj * ldw, q, 1.5f * ah[jj]);
    const F2 v = norm2(V + (size_t)jj * ldv, p, 1.5f);
    __syncwarp();                             // every lane has read its column's running norm
    if (j >= p) continue;
    if (check && !(a.h > blk::kTiny32 && a.h < kHuge32))
      for (int r = sl; r < q; r += 8) out |= W[(size_t)j * ldw + r] != 0.0f;
    if (sl == 0) {
      ah[j] = a.h;
      al[j] = a.l;
      // 1 / sqrt(1 + u) - 1 (u ~ 1e-5; a null column keeps its scale)
      const float u = (v.h - 1.0f) + v.l;
      const float d = v.h > 0.5f ? u * (-0.5f + u * (0.375f - 0.3125f * u)) : 0.0f;
      dl[j] = d;
      if (KT) KT[(size_t)j * ldk + j] = d;
    }
    if (KT && p + sl < ldk) KT[(size_t)j * ldk + p + sl] = 0.0f;
  }
  return out;
}

// Zero rows n .. up to a multiple of four of p columns.
__device__ inline void pad_rows(float* X, int n, int ldx, int p, int lw, int nw) {
  const int lane = threadIdx.x & 31;
  for (int j = lw; j < p; j += nw)
    if (n + lane < ((n + 3) & ~3)) X[(size_t)j * ldx + n + lane] = 0.0f;
}

// The diagonal of the orthonormalisation step, -1/2 of |v_j|^2 - 1, and the
// squared norms (ah); KT: zeroed padding.  V: zero rows up to a multiple of four.
__device__ inline void unit_terms(const float* V, int p, int ldv, float* ah, float* KT, int lw, int nw) {
  const int sub = (threadIdx.x & 31) >> 3, sl = threadIdx.x & 7;
  const int ldk = ldk_of(p);
  for (int j0 = 4 * lw; j0 < p; j0 += 4 * nw) {
    const int j = j0 + sub, jj = j < p ? j : p - 1;
    const F2 v = norm2(V + (size_t)jj * ldv, p, 1.5f);
    if (j >= p) continue;
    if (sl == 0) {
      ah[j] = v.h;
      KT[(size_t)j * ldk + j] = -0.5f * ((v.h - 1.0f) + v.l);
    }
    if (p + sl < ldk) KT[(size_t)j * ldk + p + sl] = 0.0f;
  }
}

// K's off-diagonal entries: a warp takes four columns i against 32 columns j
// (a lane each).  ORTHO = false: the rotations of W's columns.  ORTHO = true (al
// unused): -1/2 of the overlaps of V's columns, the step that makes them
// orthonormal.  Returns this lane's largest |E|.
template <bool ORTHO>
__device__ inline float pair_terms(const float* W, int q, int ldw, int p, const float* ah, const float* al, float* KT, int lw,
                            int nw) {
  constexpr int R = 4;
  const int lane = threadIdx.x & 31;
  const int ldk = ldk_of(p);
  const int gi = (p + R - 1) / R;
  float emax = 0.0f;
  int x = 0;
  for (int g = 0; g < gi; ++g) {
    for (int j0 = (g * R) & ~31; j0 < p; j0 += 32, ++x) {
      if (x % nw != lw) continue;
      const int j = j0 + lane, jj = j < p ? j : p - 1;
      const float b = ah[jj];
      Dot2 d[R];
      float big[R];
      const float* xi[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = min(g * R + r, p - 1);
        xi[r] = W + (size_t)i * ldw;
        const float a = ah[i];
        // |every partial sum| <= sqrt(a b)
        big[r] = above(fmaxf(sqrtf(a) * sqrtf(b), 1e-36f));
        d[r].start(big[r]);
      }
      const float* y = W + (size_t)jj * ldw;
      // rows in fours (128-bit loads; the rows from q on are zeros)
      for (int k = 0; k < q; k += 4) {
        const float4 yv = *reinterpret_cast<const float4*>(y + k);
        const float2 y0 = {yv.x, yv.y}, y1 = {yv.z, yv.w}, n0 = {-yv.x, -yv.y}, n1 = {-yv.z, -yv.w};
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const float4 xv = *reinterpret_cast<const float4*>(xi[r] + k);
          d[r].add({xv.x, xv.y}, y0, n0);
          d[r].add({xv.z, xv.w}, y1, n1);
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = g * R + r;
        if (i >= p || j >= p || j <= i) continue;
        const float a = ah[i];
        const F2 s = normal2(d[r].get(big[r]));
        float t = 0.0f;
        if (ORTHO) {
          KT[(size_t)i * ldk + j] = KT[(size_t)j * ldk + i] = -0.5f * (s.h + s.l);
          continue;
        }
        if (a > blk::kTiny32 && b > blk::kTiny32) {
          emax = fmaxf(emax, fabsf(s.h) * (rsqrtf(a) * rsqrtf(b)));
          // b - a exactly to binary32, then the rotation's tangent
          if (s.h != 0.0f && !near_pair(a, b)) t = blk::jacobi_tangent32((b - a) + (al[j] - al[i]), s.h);
        }
        KT[(size_t)i * ldk + j] = -t;         // w_i' = w_i - t w_j
        KT[(size_t)j * ldk + i] = t;          // w_j' = w_j + t w_i
      }
    }
  }
  return emax;
}

// out[:, j] = base[:, j] + X K[:, j], X n x p (shared, leading dimension ldx); base
// = X, or out itself (ADD).  out: binary64 column-major, leading dimension
// ldo.  A warp takes 64 rows x 4 columns.  Its four columns of K are loaded
// 32 entries at a time, an entry a lane, and handed round by shuffles: K lies in
// global memory, and a load per step of the product would wait for each.
// x: running task count (the tasks go round the warps).
template <bool ADD>
__device__ inline void add_product(const float* X, int n, int ldx, int p, const float* KT, double* out, int ldo,
                                   int lw, int nw, int& x) {
  const int lane = threadIdx.x & 31;
  const int ldk = ldk_of(p);
  for (int r0 = 0; r0 < n; r0 += 64) {
    const bool in0 = r0 + lane < n, in1 = r0 + 32 + lane < n;
    for (int j0 = 0; j0 < p; j0 += 4, ++x) {
      if (x % nw != lw) continue;
      float acc[2][4];
#pragma unroll
      for (int y = 0; y < 4; ++y) acc[0][y] = acc[1][y] = 0.0f;
      for (int i0 = 0; i0 < p; i0 += 32) {
        float k[4];
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          const float* col = KT + (size_t)min(j0 + y, p - 1) * ldk;
          k[y] = i0 + lane < p ? col[i0 + lane] : 0.0f;
        }
        const int ni = min(32, p - i0);
        const float* row = X + (size_t)i0 * ldx + r0 + lane;
#pragma unroll 4
        for (int i = 0; i < ni; ++i) {
          const float w0 = in0 ? row[0] : 0.0f, w1 = in1 ? row[32] : 0.0f;
          row += ldx;
#pragma unroll
          for (int y = 0; y < 4; ++y) {
            const float kz = blk::lane_value(k[y], i);
            acc[0][y] = fmaf(w0, kz, acc[0][y]);
            acc[1][y] = fmaf(w1, kz, acc[1][y]);
          }
        }
      }
#pragma unroll 1
      for (int u = 0; u < 2; ++u) {
        const int r = r0 + 32 * u + lane;
        if (r >= n) break;
#pragma unroll
        for (int y = 0; y < 4; ++y)
          if (j0 + y < p) {
            double* o = out + (size_t)(j0 + y) * ldo + r;
            const float c = u ? acc[1][y] : acc[0][y];
            *o = ADD ? *o + blk::widen(c) : corrected(X[(size_t)(j0 + y) * ldx + r], c);
          }
      }
    }
  }
}

// out[:, j] = (1 + delta_j) X[:, j].
__device__ inline void scale_columns(const float* X, int n, int ldx, int p, const float* dl, double* out, int lw, int nw) {
  const int lane = threadIdx.x & 31;
  for (int j = lw; j < p; j += nw) {
    const float d = dl[j];
    for (int r = lane; r < n; r += 32) {
      const float v = X[(size_t)j * ldx + r];
      out[(size_t)j * n + r] = corrected(v, v * d);
    }
  }
}

// KT for the columns of a binary64 V that are orthonormal to binary32: -1/2 of
// the overlaps minus 1, binary64 sums.  Same task split as pair_terms.
__device__ inline void ortho_terms64(const double* V, int p, int ldv, float* KT, int lw, int nw) {
  constexpr int R = 4;
  const int lane = threadIdx.x & 31;
  const int ldk = ldk_of(p);
  int x = 0;
  for (int g = 0; g < (p + R - 1) / R; ++g) {
    for (int j0 = (g * R) & ~31; j0 < p; j0 += 32, ++x) {
      if (x % nw != lw) continue;
      const int j = j0 + lane, jj = j < p ? j : p - 1;
      const double* y = V + (size_t)jj * ldv;
      const double* xi[R];
      double d[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        xi[r] = V + (size_t)min(g * R + r, p - 1) * ldv;
        d[r] = 0.0;
      }
#pragma unroll 2
      for (int k = 0; k < p; ++k) {
        const double yk = y[k];
#pragma unroll
        for (int r = 0; r < R; ++r) d[r] = fma(xi[r][k], yk, d[r]);
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = g * R + r;
        if (i >= p || j >= p || j < i) continue;
        const float v = blk::narrow(-0.5 * (i == j ? d[r] - 1.0 : d[r]));
        KT[(size_t)i * ldk + j] = v;
        if (i != j) KT[(size_t)j * ldk + i] = v;
      }
    }
  }
}

// out = A V: A q x p binary64 column-major (leading dimension q, global), V p x
// p (shared, leading dimension ldv), out leading dimension ldo.  32 rows x 4
// columns a warp.
__device__ inline void product64(const double* A, int q, int p, const double* V, int ldv, double* out,
                                 int ldo, int lw, int nw) {
  const int lane = threadIdx.x & 31;
  int x = 0;
  for (int r0 = 0; r0 < q; r0 += 32) {
    const int r = r0 + lane, rr = r < q ? r : q - 1;
    for (int j0 = 0; j0 < p; j0 += 4, ++x) {
      if (x % nw != lw) continue;
      double acc[4] = {0.0, 0.0, 0.0, 0.0};
      const double* a = A + rr;
      const double* v[4];
#pragma unroll
      for (int y = 0; y < 4; ++y) v[y] = V + (size_t)min(j0 + y, p - 1) * ldv;
      const int nj = min(4, p - j0);
#pragma unroll 4
      for (int i = 0; i < p; ++i) {
        const double ai = a[(size_t)i * q];
#pragma unroll
        for (int y = 0; y < 4; ++y)
          if (y < nj) acc[y] = fma(ai, v[y][i], acc[y]);
      }
      if (r < q)
#pragma unroll
        for (int y = 0; y < 4; ++y)
          if (y < nj) out[(size_t)(j0 + y) * ldo + r] = acc[y];
    }
  }
}

// One binary64 rotation of columns i, j of W (q x p) and V (p x p) by a warp.
__device__ inline void rotate64(double* W, int q, double* V, int p, int i, int j) {
  const int lane = threadIdx.x & 31;
  double* x = W + (size_t)i * q;
  double* y = W + (size_t)j * q;
  double a = 0.0, b = 0.0, g = 0.0;
  for (int r = lane; r < q; r += 32) {
    const double xr = x[r], yr = y[r];
    a = fma(xr, xr, a);
    b = fma(yr, yr, b);
    g = fma(xr, yr, g);
  }
  a = blk::warp_sum64(a);
  b = blk::warp_sum64(b);
  g = blk::warp_sum64(g);
  if (g == 0.0 || !(a > 0.0) || !(b > 0.0)) return;
  const double t = blk::jacobi_tangent64(b - a, g);
  const double cs = rsqrt(1.0 + t * t), sn = cs * t;
  for (int r = lane; r < q; r += 32) {
    const double xr = x[r], yr = y[r];
    x[r] = cs * xr - sn * yr;
    y[r] = sn * xr + cs * yr;
  }
  for (int r = lane; r < p; r += 32) {
    const double xr = V[(size_t)i * p + r], yr = V[(size_t)j * p + r];
    V[(size_t)i * p + r] = cs * xr - sn * yr;
    V[(size_t)j * p + r] = sn * xr + cs * yr;
  }
  __syncwarp();
}

// Scales the columns of V to length 1 and those of W alike.  The explicit
// rotations need it: V's columns overlap by the binary32 sweeps' ~1e-6, so a
// large angle moves their lengths by as much (the first-order step's do not).
__device__ inline void unit_columns(double* W, int q, double* V, int p, int lw, int nw) {
  const int lane = threadIdx.x & 31;
  for (int j = lw; j < p; j += nw) {
    double s = 0.0;
    for (int r = lane; r < p; r += 32) s = fma(V[(size_t)j * p + r], V[(size_t)j * p + r], s);
    s = blk::warp_sum64(s);
    if (fabs(s - 1.0) < 1e-13 || !(s > 0.5)) continue;
    const double f = rsqrt(s);
    for (int r = lane; r < p; r += 32) V[(size_t)j * p + r] *= f;
    for (int r = lane; r < q; r += 32) W[(size_t)j * q + r] *= f;
  }
}

// Rotates the near pairs in the order of their columns, one warp.  Columns
// below binary32 resolution against the largest carry the rounding of theta
// itself and are left as they are.  Returns the number found; stops (and the
// caller sweeps) beyond `most`.
__device__ inline int rotate_near(double* W, int q, double* V, int p, const float* ah, int most) {
  const int lane = threadIdx.x & 31;
  float top = 0.0f;
  for (int j = lane; j < p; j += 32) top = fmaxf(top, ah[j]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
  const float floor = fmaxf(blk::kTiny32, top * 1.4e-14f);
  int found = 0;
  for (int i = 0; i + 1 < p; ++i) {
    const float a = ah[i];
    if (!(a > floor)) continue;
    for (int j0 = i + 1; j0 < p; j0 += 32) {
      const int j = j0 + lane;
      const bool hit = j < p && ah[j] > floor && near_pair(a, ah[j]);
      if (!__any_sync(0xffffffffu, hit)) continue;
      for (int l = 0; l < 32; ++l) {
        if (!blk::lane_value(hit ? 1 : 0, l)) continue;
        if (++found > most) return found;
        rotate64(W, q, V, p, i, j0 + l);
      }
    }
  }
  return found;
}

}  // namespace refine
}  // namespace hm
