// Charge blocks of the two-site update, shared by the binary64 evolve
// (hm_fp64.cu) and the mixed-precision evolve (hm_mixed.cu).
//
// Sec. II.C ("Exploiting Conserved Quantum Numbers"): the gates exp(-tau J
// S_i.S_j) conserve S^z_i + S^z_j, and an initial state |i>_E |B>_C whose
// environment is a product of S^z eigenstates has a definite total S^z.  So
// every bond index carries a charge q, every position's leg a sign sigma
// (+1 for a spin, -1 for an ancilla: its Bell partner carries the opposite
// S^z, which makes each Bell pair neutral), and A[l, s, r] = 0 unless
// q(l) + sigma m(s) = q(r), with m = +1, 0, -1 for s = 0, 1, 2.  A SWAP
// moves a site's content, and with it its sign, to the other position.
//
// After the gate, the two-site tensor theta[(l a), (b r)] is block diagonal
// in the charge Q of the new middle bond: rows with q(l) + sigma_k m(a) = Q
// against columns with q(r) - sigma_{k+1} m(b) = Q.  Each block is decomposed
// on its own.  The singular values of theta are the union of the blocks'
// values, so the truncation rule (Sec. II) runs on that union and keeps the
// set a dense SVD keeps; each kept value's block labels its new bond index.
//
// Bond indices stay grouped by charge in ascending order, so one charge is
// one contiguous run of a bond, and a block's rows (and columns) are three
// runs, one per local state.  A chain in dense mode (every charge and sign 0)
// has a single block: the unblocked split.
//
// Entries outside the blocks are never computed, written or read: the block
// GEMMs write only entries whose row and column charges agree, the gate is
// applied only within its conserved sectors, and the absorb writes the blocks
// alone (clear_forbidden).  So the structure holds exactly, in any precision.
#pragma once

#include <cstdint>
#include <cstring>

#include "hm_internal.h"

namespace hm {
namespace blk {

constexpr int kWin = 512;                 // charges one split may span (window)
constexpr int kMaxBlocks = kWin;

// m(s) of the local basis s = 0, 1, 2 (m = +1, 0, -1).
__device__ __forceinline__ int mval(int s) { return 1 - s; }

// One theta block of a split (a middle charge with rows and columns): per
// local state the first index and the offset in the block's row and column
// lists, and the charge's run of the middle bond.
struct InRec {
  int16_t rst[3], roff[4], cst[3], coff[4];
  int16_t mst, mlen;
};

// One output block of a split.  Lengths and offsets are below 3 x 4096.
struct BlockRec {
  int16_t Q, mq, nq, trans;               // charge, rows (l a), columns (b r), W holds the transpose
  int16_t q, p;                           // W is q x p column-major, q >= p
  int16_t rst[3], rlen[3], roff[3];       // per a: first l, count, offset in the row list
  int16_t cst[3], clen[3], coff[3];       // per b: first r, count, offset in the column list
  int32_t svoff;                          // first slot in the value list
  int64_t woff, voff;                     // offsets (elements) of the block's W and V
};

// Split metadata in the chain's meta workspace (splits of more than kShBlk blocks).
struct Meta {
  InRec in[kWin];
  BlockRec b[kMaxBlocks];
};

static_assert(sizeof(Meta) <= kMetaBytes, "meta workspace of a chain");

// Charge-run tables of the three bonds while a split is prepared: (start,
// end) of each charge of the window.  12 KB of the CTA's scratch memory.
struct PrepTab {
  int32_t t[3][kWin][2];
};

// Records of the usual split (at most 11 blocks measured on the benchmark
// ladder) stay in shared memory; a split with more keeps all of its records
// in the meta workspace.
#ifndef HM_SH_BLK
#define HM_SH_BLK 14
#endif
constexpr int kShBlk = HM_SH_BLK;

// Shared scalars of a split (CTA shared memory).
struct SplitSh {
  int32_t sk, sk1, osk, osk1;             // input and output leg signs of sites k, k+1
  int32_t qbase, qtop, nin, nblk, ok, P;  // P: singular values over all blocks
  int32_t nt[9];                          // per output (a b): terms of its conserved sector
  int16_t tt[9][9];                       // term: input 3 s1 + s2
  double G[9][9];                         // term: coefficient
  float gh[9][9], gl[9][9];               // the coefficient as a binary32 pair hi + lo
  int32_t kk;
  double nrm;
  const InRec* in;
  const BlockRec* b;
  double k1;                              // multiply-adds of the theta blocks
  InRec in_sh[kShBlk];
  BlockRec b_sh[kShBlk];
};

struct Seg {
  int32_t start, len;
};

// The CTAs that work on one chain together (a thread-block cluster), or one.
struct Team {
  int rank, size;
};

// Barrier of the team's threads; orders their accesses to global memory.
__device__ __forceinline__ void team_sync(const Team& tm) {
#if defined(__CUDA_ARCH__)
  if (tm.size > 1) {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    return;
  }
#elif defined(HM_TEAM_EMULATION)
  if (tm.size > 1) {
    simt::team_sync();
    return;
  }
#endif
  __syncthreads();
}

__device__ __forceinline__ Seg seg_of(const PrepTab& T, int bond, int qbase, int q) {
  const int i = q - qbase;
  if (i < 0 || i >= kWin) return {0, 0};   // callers stay within [qbase, qtop + 3]
  return {T.t[bond][i][0], T.t[bond][i][1] - T.t[bond][i][0]};
}

// The value of another lane of the warp.
template <typename T>
__device__ __forceinline__ T lane_value(T v, int src) {
  return __shfl_xor_sync(0xffffffffu, v, (threadIdx.x & 31) ^ src);
}

// Exclusive sum over the lanes of a warp; *total gets the warp's sum.
__device__ __forceinline__ int lane_prefix(int v, int* total) {
  const int lane = threadIdx.x & 31;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = lane_value(x, lane >= o ? lane - o : lane);
    if (lane >= o) x += y;
  }
  *total = lane_value(x, 31);
  return x - v;
}

// binary32 <-> binary64 by integer instructions: GB300 converts to and from
// 64-bit types on its binary64 pipe (2 a clock and SM).  Both equal the
// conversion instruction for every input (zero and normal binary32 values
// take the integer form, the rest the instruction).
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f), e = (u >> 23) & 0xffu;
  if ((u << 1) == 0u || (e != 0u && e != 255u)) {
    const unsigned hi = (u << 1) == 0u ? u : (u & 0x80000000u) | ((e + 896u) << 20) | ((u >> 3) & 0xfffffu);
    const unsigned long long b = ((unsigned long long)hi << 32) | (unsigned)(u << 29);
    double d;
    memcpy(&d, &b, 8);
    return d;
  }
  return (double)f;
}

__device__ __forceinline__ float narrow(double d) {
  unsigned long long b;
  memcpy(&b, &d, 8);
  const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
  const unsigned e = (hi >> 20) & 0x7ffu;
  if (e > 896u && e < 1151u) {
    unsigned u = ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
    const unsigned rest = lo << 3;                       // the bits below, round half to even
    u += (rest > 0x80000000u || (rest == 0x80000000u && (u & 1u))) ? 1u : 0u;
    return __uint_as_float((hi & 0x80000000u) | u);
  }
  if ((b << 1) == 0ull) return __uint_as_float(hi);
  return (float)d;
}

template <typename T>
__device__ __forceinline__ T from64(double d);
template <>
__device__ __forceinline__ double from64<double>(double d) {
  return d;
}
template <>
__device__ __forceinline__ float from64<float>(double d) {
  return narrow(d);
}

// Zeros in the entries of every site tensor that its charges forbid.  A split
// writes only the allowed entries (finish) and every kernel reads only those,
// so the others hold whatever an earlier, differently shaped tensor left in the
// slot; whoever wants the full tensors clears them first.
template <int NT>
__device__ void clear_forbidden(ChainDev* c) {
  for (int k = 0; k < c->n_sites; ++k) {
    const int cl = c->chi[k], cr = c->chi[k + 1], sg = c->sgn[k];
    const int16_t* qL = c->qn + (size_t)k * c->chi_cap;
    const int16_t* qR = qL + c->chi_cap;
    double* A = c->site[k];
    for (int e = threadIdx.x; e < cl * 3 * cr; e += NT) {
      const int row = e / cr, r = e - row * cr, l = row / 3;
      if (qL[l] + sg * mval(row - 3 * l) != qR[r]) A[e] = 0.0;
    }
  }
  __syncthreads();
}

// Marks a chain as having no usable charge structure from here on: every
// charge and sign 0 (one block per split).  Sec. II.C's blocking is an
// optimisation; the dense split computes the same decomposition.
template <int NT>
__device__ void go_dense(ChainDev* c) {
  clear_forbidden<NT>(c);
  const int nb = (c->n_sites + 1) * c->chi_cap;
  for (int e = threadIdx.x; e < nb; e += NT) c->qn[e] = 0;
  for (int e = threadIdx.x; e < c->n_sites; e += NT) c->sgn[e] = 0;
  if (threadIdx.x == 0) c->counters[3] = 1;
  __syncthreads();
}

// Phase A: signs, charge-run tables of the three bonds, the middle charges
// of the theta blocks and the output blocks with their workspace offsets.
// Returns false if the chain had to switch to dense mode first (then call again).
// One thread a candidate charge: a serial loop over them, each step a chain of
// dependent loads, took as long as the blocks' arithmetic on small bonds.
template <int NT>
__device__ bool prepare(ChainDev* c, const OpDev& op, SplitSh& s, PrepTab& T, const Team& tm) {
  const int tid = threadIdx.x;
  const int k = op.k;
  const int chil = c->chi[k], chim = c->chi[k + 1], chir = c->chi[k + 2];
  const int16_t* qL = c->qn + (size_t)k * c->chi_cap;
  const int16_t* qM = qL + c->chi_cap;
  const int16_t* qR = qM + c->chi_cap;
  Meta* M = reinterpret_cast<Meta*>(c->meta);
  const int info = c->gate_info[op.gate];
  __shared__ int lo_sh, hi_sh, bad_sh;
  if (tid == 0) {
    lo_sh = 1 << 30;
    hi_sh = -(1 << 30);
    bad_sh = 0;
    const int a = c->sgn[k], b = c->sgn[k + 1];
    s.ok = 1;
    // a gate that is not a permutation conserves m1 + m2 only: on legs of
    // unequal sign (a spin next to an ancilla) it breaks the charge rule
    if ((info & 2) && a != b) s.ok = 0;
    s.sk = a;
    s.sk1 = b;
    s.osk = (info & 1) ? b : a;
    s.osk1 = (info & 1) ? a : b;
  }
  __syncthreads();
  {
    // charge range of the three bonds; each charge must be one run, ascending
    int lo = 1 << 30, hi = -(1 << 30), bad = 0;
    const int nall = chil + chim + chir;
    for (int e = tid; e < nall; e += NT) {
      int i;
      const int16_t* q;
      if (e < chil) i = e, q = qL;
      else if (e < chil + chim) i = e - chil, q = qM;
      else i = e - chil - chim, q = qR;
      lo = min(lo, (int)q[i]);
      hi = max(hi, (int)q[i]);
      if (i > 0 && q[i] < q[i - 1]) bad = 1;
    }
    if (lo <= hi) {
      atomicMin(&lo_sh, lo);
      atomicMax(&hi_sh, hi);
    }
    if (bad) atomicMax(&bad_sh, 1);
  }
  __syncthreads();
  if (tid == 0) {
    s.qbase = lo_sh - 3;
    s.qtop = hi_sh;
    if (hi_sh - lo_sh + 7 > kWin || bad_sh) s.ok = 0;
  }
  __syncthreads();
  if (!s.ok) {
    // every CTA of the team reads the same labels and comes here, or none does
    team_sync(tm);
    if (c->counters[3]) return true;      // already dense: every charge is 0, cannot fail again
    team_sync(tm);                        // every CTA has read the mark
    if (tm.rank == 0) go_dense<NT>(c);
    team_sync(tm);
    return false;
  }
  const int qb = s.qbase;
  const int span = s.qtop - qb + 4;        // window entries any lookup of this split reaches
  for (int e = tid; e < 3 * span; e += NT) {
    T.t[e / span][e % span][0] = 0;
    T.t[e / span][e % span][1] = 0;
  }
  __syncthreads();
  const int nall = chil + chim + chir;
  for (int e = tid; e < nall; e += NT) {
    int bond, i, n;
    const int16_t* q;
    if (e < chil) bond = 0, i = e, n = chil, q = qL;
    else if (e < chil + chim) bond = 1, i = e - chil, n = chim, q = qM;
    else bond = 2, i = e - chil - chim, n = chir, q = qR;
    const int Q = q[i];
    if (i == 0 || q[i - 1] != Q) T.t[bond][Q - qb][0] = i;
    if (i == n - 1 || q[i + 1] != Q) T.t[bond][Q - qb][1] = i + 1;
  }
  __syncthreads();
  if (tid >= 32 && tid < 41) {
    // conserved sector of the outputs (a b) of the gate, its coefficients also as binary32 pairs
    const int o = tid - 32, a = o / 3, b = o % 3;
    const double* g = c->gates + (size_t)op.gate * 81 + o * 9;
    int n = 0;
    for (int u = 0; u < 9; ++u) {
      const double x = g[u];
      if (s.sk * mval(u / 3) + s.sk1 * mval(u % 3) == s.osk * mval(a) + s.osk1 * mval(b) && x != 0.0) {
        s.tt[o][n] = (int16_t)u;
        s.G[o][n] = x;
        s.gh[o][n] = (float)x;
        s.gl[o][n] = (float)(x - (double)(float)x);
        ++n;
      }
    }
    s.nt[o] = n;
  }
  if (tid < 32) {
    // candidate charges [lowest - 2, highest + 2] of the three bonds, 32 at a time:
    // records in ascending charge, offsets by sums over the lanes
    const int cand = s.qtop - qb + 2;
    int nin = 0, nblk = 0, svoff = 0;
    int64_t woff = 0, voff = 0;
    double k1 = 0.0;
    bool shared = true;
    for (int pass = 0; pass < 2; ++pass) {
      // pass 0 counts, so that the records of one split are all in one place
      nin = nblk = svoff = 0;
      woff = voff = 0;
      for (int i0 = 1; i0 <= cand; i0 += 32) {
        const int i = i0 + tid, Q = qb + i;
        InRec in;
        BlockRec r;
        int rows = 0, cols = 0, mq = 0, nq = 0;
        for (int t = 0; t < 3; ++t) {
          const Seg a = seg_of(T, 0, qb, Q - s.sk * mval(t)), b = seg_of(T, 2, qb, Q + s.sk1 * mval(t));
          in.rst[t] = (int16_t)a.start, in.roff[t] = (int16_t)rows;
          in.cst[t] = (int16_t)b.start, in.coff[t] = (int16_t)cols;
          rows += a.len;
          cols += b.len;
          const Seg x = seg_of(T, 0, qb, Q - s.osk * mval(t)), y = seg_of(T, 2, qb, Q + s.osk1 * mval(t));
          r.rst[t] = (int16_t)x.start, r.rlen[t] = (int16_t)x.len, r.roff[t] = (int16_t)mq;
          r.cst[t] = (int16_t)y.start, r.clen[t] = (int16_t)y.len, r.coff[t] = (int16_t)nq;
          mq += x.len;
          nq += y.len;
        }
        const bool is_in = i <= cand && rows > 0 && cols > 0, is_out = i <= cand && mq > 0 && nq > 0;
        const Seg mid = seg_of(T, 1, qb, Q);
        in.roff[3] = (int16_t)rows, in.coff[3] = (int16_t)cols;
        in.mst = (int16_t)mid.start, in.mlen = (int16_t)mid.len;
        int n_in, n_out, n_sv;
        const int at_in = lane_prefix(is_in ? 1 : 0, &n_in), at_out = lane_prefix(is_out ? 1 : 0, &n_out);
        if (pass == 1) {
          // a team's CTAs write the same records
          InRec* ri = shared ? s.in_sh : M->in;
          BlockRec* ro = shared ? s.b_sh : M->b;
          const int p = mq < nq ? mq : nq, q = mq < nq ? nq : mq;
          const int at_sv = lane_prefix(is_out ? p : 0, &n_sv);
          // W and V offsets, in elements: sums of up to 32 x 12288^2 in two halves
          int lo_t, hi_t, vlo_t, vhi_t;
          const int64_t w = is_out ? (int64_t)q * p : 0, v = is_out ? (int64_t)p * p : 0;
          const int wl = lane_prefix((int)(w & 0xfffff), &lo_t), wh = lane_prefix((int)(w >> 20), &hi_t);
          const int vl = lane_prefix((int)(v & 0xfffff), &vlo_t), vh = lane_prefix((int)(v >> 20), &vhi_t);
          if (is_in) ri[nin + at_in] = in;
          if (is_out) {
            r.Q = (int16_t)Q;
            r.mq = (int16_t)mq;
            r.nq = (int16_t)nq;
            r.trans = nq > mq;
            r.q = (int16_t)q;
            r.p = (int16_t)p;
            r.svoff = svoff + at_sv;
            r.woff = woff + wl + ((int64_t)wh << 20);
            r.voff = voff + vl + ((int64_t)vh << 20);
            ro[nblk + at_out] = r;
          }
          svoff += n_sv;
          woff += lo_t + ((int64_t)hi_t << 20);
          voff += vlo_t + ((int64_t)vhi_t << 20);
        }
        nin += n_in;
        nblk += n_out;
      }
      shared = nin <= kShBlk && nblk <= kShBlk;
    }
    __syncwarp();
    if (tid == 0) {
      s.nin = nin;
      s.nblk = nblk;
      s.P = svoff;
      s.in = shared ? s.in_sh : M->in;
      s.b = shared ? s.b_sh : M->b;
      for (int i = 0; i < nin; ++i) k1 += (double)s.in[i].roff[3] * s.in[i].mlen * s.in[i].coff[3];
      s.k1 = k1;
    }
  }
  __syncthreads();
  return true;
}

// Calls f(e) for this lane's share of the n elements of one block: the
// CTA's warps take chunks of 32 elements in turn over all blocks of a phase
// (c0 counts the chunks so far), so that a phase over many small blocks keeps
// every warp busy without a barrier or an idle warp between blocks.
template <int NT, typename F>
__device__ __forceinline__ void share(int n, int& c0, F&& f) {
  constexpr int NW = NT / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nch = (n + 31) >> 5;
  for (int ch = (unsigned)(warp - c0) % NW; ch < nch; ch += NW) {
    const int e = ch * 32 + lane;
    if (e < n) f(e);
  }
  c0 += nch;
}

// The same over all CTAs of a team.
template <int NT, typename F>
__device__ __forceinline__ void share(const Team& tm, int n, int& c0, F&& f) {
  const int lane = threadIdx.x & 31;
  const unsigned nw = NT / 32 * tm.size;           // a power of two
  const int warp = (threadIdx.x >> 5) + NT / 32 * tm.rank;
  const int nch = (n + 31) >> 5;
  for (int ch = (unsigned)(warp - c0) & (nw - 1); ch < nch; ch += nw) {
    const int e = ch * 32 + lane;
    if (e < n) f(e);
  }
  c0 += nch;
}

// Phase B: theta[(l s1), (s2 r)] = sum_m A_k[(l s1), m] A_{k+1}[m, (s2 r)] for
// every entry whose row charge q(l) + sigma_k m(s1) and column charge
// q(r) - sigma_{k+1} m(s2) agree (Sec. I.A two-site tensor), one GEMM per
// middle charge over that charge's run of the middle bond.  Entries of a
// charge absent from the middle bond are written as 0.  A, B are binary64
// site tensors; T is the accumulation and storage type of theta.
//
// Two forms.  Direct: a warp takes R rows x 32 columns of a block and reads both
// operands through L1, all blocks at once, no barrier.  Binary64 always takes
// it: its pipe (16 clocks a warp instruction) hides the loads, and a padded
// tile would be charged in full.  Binary32 takes it while the split has at most
// kThetaDirect products; there a conversion costs as much as several products,
// so A's entries are loaded and converted 32 at a time, one a lane, and handed
// round by shuffles.  Above, the CTA goes through the blocks in TM x TN x TK
// tiles in shared memory, which load and convert each operand once per tile.
// The line is not critical: at 0 (tiles only), 65,536, 262,144 and 1,048,576
// products ladders of Lx = 4 to 16 and chi = 256 take the same time to 2 % (Lx = 16,
// 256 chains: 394, 386, 390, 390 ms a step); it bounds what the direct form reads
// through L1 more than once.
#ifndef HM_THETA_DIRECT
#define HM_THETA_DIRECT 262144.0
#endif
constexpr double kThetaDirect = HM_THETA_DIRECT;

template <int NT, typename T>
__device__ void theta_direct(const ChainDev* c, int k, const SplitSh& s, T* __restrict__ theta, const Team& tm) {
  constexpr bool F32 = sizeof(T) < sizeof(double);
  constexpr int R = F32 ? 8 : 4;
  const int lane = threadIdx.x & 31;
  const unsigned nw = NT / 32 * tm.size;           // a power of two
  const int warp = (threadIdx.x >> 5) + NT / 32 * tm.rank;
  const int chim = c->chi[k + 1], chir = c->chi[k + 2];
  const int n = 3 * chir;
  const double* A = c->site[k];
  const double* B = c->site[k + 1];
  int c0 = 0;
  for (int bi = 0; bi < s.nin; ++bi) {
    const InRec& r = s.in[bi];
    const int Mv = r.roff[3], Nv = r.coff[3], K = r.mlen, mst = r.mst;
    const int nu = (Nv + 31) >> 5, tasks = ((Mv + R - 1) / R) * nu;
    for (int x = (unsigned)(warp - c0) & (nw - 1); x < tasks; x += nw) {
      const int g = x / nu, u = (x - g * nu) * 32 + lane;
      const int uu = min(u, Nv - 1);
      const int t2 = uu >= r.coff[2] ? 2 : (uu >= r.coff[1] ? 1 : 0);
      const int col = t2 * chir + r.cst[t2] + uu - r.coff[t2];
      const double* b = B + (size_t)mst * n + col;
      const int nr = min(R, Mv - g * R);
      int row[R];
      T acc[R];
#pragma unroll
      for (int y = 0; y < R; ++y) {
        const int v = min(g * R + y, Mv - 1);
        const int t = v >= r.roff[2] ? 2 : (v >= r.roff[1] ? 1 : 0);
        row[y] = 3 * (r.rst[t] + v - r.roff[t]) + t;
        acc[y] = T(0);
      }
      if constexpr (F32) {
        for (int k0 = 0; k0 < K; k0 += 32) {
          const int kn = min(32, K - k0);
          T av[R];
#pragma unroll
          for (int y = 0; y < R; ++y)
            av[y] = lane < kn ? from64<T>(A[(size_t)row[y] * chim + mst + k0 + lane]) : T(0);
#pragma unroll 2
          for (int kk = 0; kk < kn; ++kk) {
            const T bv = from64<T>(b[(size_t)(k0 + kk) * n]);
#pragma unroll
            for (int y = 0; y < R; ++y) acc[y] = fma(lane_value(av[y], kk), bv, acc[y]);
          }
        }
      } else {
#pragma unroll 4
        for (int kk = 0; kk < K; ++kk) {
          const double bv = b[(size_t)kk * n];
#pragma unroll
          for (int y = 0; y < R; ++y)
            if (y < nr) acc[y] = fma(A[(size_t)row[y] * chim + mst + kk], bv, acc[y]);
        }
      }
      if (u < Nv)
#pragma unroll
        for (int y = 0; y < R; ++y)
          if (y < nr) theta[(size_t)row[y] * n + col] = acc[y];
    }
    c0 += tasks;
  }
  team_sync(tm);
}

template <int NT, int TM, int TN, int TK>
__device__ void theta_blocks(const ChainDev* c, int k, const SplitSh& s, float* __restrict__ theta, float* smem,
                             const Team& tm) {
  using T = float;
  if (s.k1 <= kThetaDirect) return theta_direct<NT, T>(c, k, s, theta, tm);
  const int tid = threadIdx.x;
  const int chim = c->chi[k + 1], chir = c->chi[k + 2];
  const int n = 3 * chir;
  const double* A = c->site[k];
  const double* B = c->site[k + 1];
  // thread tile: rows ty + TY a (a < RA), columns tx + TX b (b < 4)
  constexpr int RB = 4, TX = TN / RB, TY = NT / TX, RA = TM / TY;
  static_assert(TN % RB == 0 && NT % TX == 0 && TM % TY == 0, "tile must split evenly over the CTA");
  const int tx = tid % TX, ty = tid / TX;
  T* sa = smem;                            // [TK][TM + 1]
  T* sb = smem + TK * (TM + 1);            // [TK][TN + 1]
  int tile = 0;
  for (int bi = 0; bi < s.nin; ++bi) {
    const InRec& r = s.in[bi];
    const int Mv = r.roff[3], Nv = r.coff[3], K = r.mlen, mst = r.mst;
    for (int i0 = 0; i0 < Mv; i0 += TM) {
      for (int j0 = 0; j0 < Nv; j0 += TN) {
        if (tile++ % tm.size != tm.rank) continue;        // tiles go round the team
        T acc[RA][RB];
#pragma unroll
        for (int a = 0; a < RA; ++a)
#pragma unroll
          for (int b = 0; b < RB; ++b) acc[a][b] = T(0);
        for (int k0 = 0; k0 < K; k0 += TK) {
          for (int e = tid; e < TM * TK; e += NT) {
            const int ii = e / TK, kk = e % TK;
            const int v = i0 + ii, g = k0 + kk;
            T x = T(0);
            if (v < Mv && g < K) {
              const int t = v >= r.roff[2] ? 2 : (v >= r.roff[1] ? 1 : 0);
              const int l = r.rst[t] + v - r.roff[t];
              x = from64<T>(A[(size_t)(3 * l + t) * chim + mst + g]);
            }
            sa[kk * (TM + 1) + ii] = x;
          }
          for (int e = tid; e < TN * TK; e += NT) {
            const int jj = e % TN, kk = e / TN;
            const int u = j0 + jj, g = k0 + kk;
            T x = T(0);
            if (u < Nv && g < K) {
              const int t = u >= r.coff[2] ? 2 : (u >= r.coff[1] ? 1 : 0);
              x = from64<T>(B[(size_t)(mst + g) * n + t * chir + r.cst[t] + u - r.coff[t]]);
            }
            sb[kk * (TN + 1) + jj] = x;
          }
          __syncthreads();
          const int kn = min(TK, K - k0);
#pragma unroll 4
          for (int kk = 0; kk < kn; ++kk) {
            T bv[RB];
#pragma unroll
            for (int b = 0; b < RB; ++b) bv[b] = sb[kk * (TN + 1) + tx + TX * b];
#pragma unroll
            for (int a = 0; a < RA; ++a) {
              const T av = sa[kk * (TM + 1) + ty + TY * a];
#pragma unroll
              for (int b = 0; b < RB; ++b) acc[a][b] = fma(av, bv[b], acc[a][b]);
            }
          }
          __syncthreads();
        }
#pragma unroll
        for (int a = 0; a < RA; ++a) {
          const int v = i0 + ty + TY * a;
          if (v >= Mv) continue;
          const int t = v >= r.roff[2] ? 2 : (v >= r.roff[1] ? 1 : 0);
          const int row = 3 * (r.rst[t] + v - r.roff[t]) + t;
#pragma unroll
          for (int b = 0; b < RB; ++b) {
            const int u = j0 + tx + TX * b;
            if (u >= Nv) continue;
            const int tt = u >= r.coff[2] ? 2 : (u >= r.coff[1] ? 1 : 0);
            theta[(size_t)row * n + tt * chir + r.cst[tt] + u - r.coff[tt]] = acc[a][b];
          }
        }
      }
    }
  }
  team_sync(tm);
}

// Phase C input: block r of theta after the gate (Sec. I.A: the gate acts on
// the physical legs only), written column-major into W (q x p, leading
// dimension ldw; the transpose when the block is wider than tall).  V = I.
// c0: see share().  A binary32 theta takes each coefficient as a binary32 pair
// (hi + lo): rounding the gate itself would repeat the same relative error at
// every application of that gate and add up coherently over the evolution,
// while the rounding of the products does not.  The pairs are split once per
// split (prepare): split at every use they put four binary64 instructions
// on each of the up to three terms of an entry.
template <int NT, typename TT, typename TW>
__device__ void gather_block(const ChainDev* c, int k, const SplitSh& s, const BlockRec& r,
                             const TT* theta, TW* W, int ldw, TW* V, int ldv, int& c0) {
  const int chir = c->chi[k + 2];
  const int n = 3 * chir;
  const int nq = r.nq;
  share<NT>(r.mq * nq, c0, [&](int e) {
    const int v = e / nq, u = e - v * nq;              // u fastest: r runs contiguously in theta
    const int a = v >= r.roff[2] ? 2 : (v >= r.roff[1] ? 1 : 0);
    const int b = u >= r.coff[2] ? 2 : (u >= r.coff[1] ? 1 : 0);
    const int o = 3 * a + b;
    const TT* th = theta + (size_t)(3 * (r.rst[a] + v - r.roff[a])) * n + r.cst[b] + u - r.coff[b];
    const int nt = s.nt[o];
    TT x = TT(0), y = TT(0);
    for (int t = 0; t < nt; ++t) {
      const int in = s.tt[o][t];
      const TT h = th[(size_t)(in / 3) * n + (in % 3) * chir];
      if constexpr (sizeof(TT) < sizeof(double)) {
        x = fma(s.gh[o][t], h, x);
        y = fma(s.gl[o][t], h, y);
      } else {
        x = fma(s.G[o][t], h, x);
      }
    }
    if constexpr (sizeof(TT) < sizeof(double)) x += y;
    if (r.trans) W[(size_t)v * ldw + u] = (TW)x;
    else W[(size_t)u * ldw + v] = (TW)x;
  });
  const int p = r.p;
  share<NT>(p * p, c0, [&](int e) {
    const int j = e / p, i = e - j * p;
    V[(size_t)j * ldv + i] = (i == j) ? TW(1) : TW(0);
  });
}

// Barrier of the nthreads threads (a multiple of 32) of a warp group; ids
// 1..15 (0 is __syncthreads).  HM_HOST_EMULATION: the kernels compiled as
// host C++ by the CPU emulation of the tests.
__device__ __forceinline__ void group_sync(int id, int nthreads) {
#if defined(__CUDA_ARCH__)
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
#elif defined(HM_HOST_EMULATION)
  simt::named_sync(id, nthreads);
#endif
}

template <typename T>
__device__ __forceinline__ T warp_sum_t(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Tangent t of the Jacobi rotation that makes columns with Gram entries
// (a, g; g, b) orthogonal: t = sign(z) / (|z| + sqrt(1 + z^2)),
// z = (b - a) / (2 g) = d / (2 g).  It sits on the critical path of every
// pass, so it takes the short-latency binary32 forms (approximate divide and
// reciprocal square root, a few ulp): a rotation is exactly conformal
// whatever its angle, the stretch c^2 + s^2 - 1 is removed with the column
// scales when W and V are promoted, and an angle that is off by 1e-7
// relative leaves an off-diagonal 1e-7 times the one it removed, which the
// next sweep takes.  The binary64 kernels need it cheaply too:
// GB300 has few binary64 units, and a binary64 square root or divide is a
// sequence of them.  The rotation (c, s) = (1, t) / sqrt(1 + t^2) is
// orthogonal to binary64 rounding whatever t is, so t only has to be close:
// z is formed in binary32 from d and g scaled by the same power of two (z
// does not change; bits_to_float, integer instructions only), which leaves
// an off-diagonal of relative size ~1e-7 times the one it removes, for the
// next sweep.  Operands too far apart for binary32 take the binary64 formula.
// Squared column norm below which the binary32 sweeps leave a column alone:
// a normal number whose square root (1e-15) is far below binary32
// resolution against columns of order one.  With both norms above it, a
// rotated pair's |g| > tol sqrt(a b) > 1e-37 is normal too.
constexpr float kTiny32 = 1e-30f;

__device__ __forceinline__ float jacobi_tangent32(float d, float g) {
  const float z = __fdividef(d, 2.0f * g);
  if (fabsf(z) > 1e18f) return __fdividef(0.5f, z);
  const float w = 1.0f + z * z;
  return copysignf(__fdividef(1.0f, fabsf(z) + w * rsqrtf(w)), z);
}

// Biased binary64 exponent of x (0 for zero and subnormals).
__device__ __forceinline__ int bexp64(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// x * 2^(1023 - e) as a binary32 number, built from the bits of x by integer
// instructions (no binary64 or conversion instruction): the top 23 bits of
// the mantissa, truncated (relative error < 2^-23).  0 when x is zero,
// subnormal, or 2^126 or more below 2^(e - 1023).  e >= the exponent of x.
__device__ __forceinline__ float bits_to_float(double x, int e) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int ex = (int)((hi >> 20) & 0x7ffu);
  const int ef = ex - e + 127;
  if (ex == 0 || ef <= 0) return 0.0f;
  return __uint_as_float((hi & 0x80000000u) | ((unsigned)ef << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
}

__device__ __forceinline__ double jacobi_tangent64(double d, double g) {
  const int e = max(bexp64(d), bexp64(g));
  const float gf = bits_to_float(g, e);
  if (fabsf(gf) >= 1e-30f) return (double)jacobi_tangent32(bits_to_float(d, e), gf);
  const double z = d / (2.0 * g);
  return fabs(z) > 1e150 ? 0.5 / z : copysign(1.0, z) / (fabs(z) + sqrt(1.0 + z * z));
}

// Per-group convergence words of a grouped Jacobi (shared memory).
struct GroupSh {
  int32_t flag[16];
  uint32_t rbits[16];                     // largest rotation ratio of the sweep, binary32 bits
};

// One pass: the L lanes of this lane's pair (a, b) (a < 0: no pair) take the
// dot product of the two columns, the rotation angle and the rotation of W
// and V, then the pair's first lane stores the two new norms.  Every lane of
// the warp takes part (the reductions are warp shuffles).  A lane moves its
// rows in batches of B, every load of a batch issued before the first store
// (a store to one column could alias the next load of the other, so the
// compiler keeps them in program order), and its first batch stays in
// registers from the dot product to the rotation: a pass waits on one memory
// latency per batch, not one per row.  Binary64 (T = double): the rotation
// tests and the tangent take binary32 values built from the operands' bits,
// so that a pass spends its binary64 instructions on the rotation itself
// (GB300 runs binary64 at about 1/64 of the binary32 rate).  rmax: largest
// ratio |g| / sqrt(a b) seen (binary64: 1 once some ratio reached `stop`);
// rot: set when a rotation was applied.
template <typename T, typename TV, int L, int B>
__device__ __forceinline__ void jacobi_pass(T* __restrict__ W, int q, int ldw, int p, TV* __restrict__ V, int ldv,
                                            T* __restrict__ nrm, int a, int b, int sl, T tol, T stop, T& rmax,
                                            int& rot) {
  constexpr bool SC = sizeof(T) == sizeof(double);   // binary64 form of the angle
          T* x = W + (size_t)(a < 0 ? 0 : a) * ldw;
          T* y = W + (size_t)(b < 0 ? 0 : b) * ldw;
          // rows sl + u L (u < B) of both columns stay in registers from the
          // dot product to the rotation; further rows go in batches of B whose
          // loads are all issued before any use (one memory latency a batch)
          T x0[B], y0[B], gacc[B];
  #pragma unroll
          for (int u = 0; u < B; ++u) {
            const int i = sl + u * L;
            const bool in = a >= 0 && i < q;
            x0[u] = in ? x[i] : T(0);
            y0[u] = in ? y[i] : T(0);
          }
  #pragma unroll
          for (int u = 0; u < B; ++u) gacc[u] = x0[u] * y0[u];
          if (a >= 0) {
            for (int i0 = sl + B * L; i0 < q; i0 += B * L) {
              T xr[B], yr[B];
  #pragma unroll
              for (int u = 0; u < B; ++u) {
                const int i = i0 + u * L;
                xr[u] = i < q ? x[i] : T(0);
                yr[u] = i < q ? y[i] : T(0);
              }
  #pragma unroll
              for (int u = 0; u < B; ++u) gacc[u] = fma(xr[u], yr[u], gacc[u]);
            }
          }
          T ga = gacc[0];
  #pragma unroll
          for (int u = 1; u < B; ++u) ga += gacc[u];
  #pragma unroll
          for (int o = L / 2; o > 0; o >>= 1) ga += __shfl_xor_sync(0xffffffffu, ga, o);
          bool done = false;
          T na = T(0), nb = T(0);
          if (a >= 0) {
            const T al = nrm[a], be = nrm[b];
            bool go;
            T ratio = T(0);
            float rf = 0.0f;
            if constexpr (SC) {
              // |g| / sqrt(a b) in binary32 from the operands' bits (integer
              // pipe), each scaled by its own power of two: a, b in [1, 2), g
              // by the mean exponent, so the ratio holds over the whole
              // binary64 range and no pair is skipped for its columns' sizes
              const int ea = bexp64(al), eb = bexp64(be);
              const float af = bits_to_float(al, ea), bf = bits_to_float(be, eb);
              rf = fabsf(bits_to_float(ga, (ea + eb) >> 1)) * rsqrtf(fmax(af * bf, 1.0f));
              if ((ea + eb) & 1) rf *= 0.70710678f;
              go = ga != T(0) && af > 0.0f && bf > 0.0f && rf > (float)tol;
            } else {
              // columns below kTiny32 are noise at binary32 resolution, and
              // the fast reciprocal square root flushes subnormal inputs to 0
              ratio = fabs(ga) * (rsqrtf(fmax(al, kTiny32)) * rsqrtf(fmax(be, kTiny32)));
              go = ga != T(0) && al > kTiny32 && be > kTiny32 && ratio > tol;
            }
            if (go) {
              T t, cs;
              if constexpr (SC) {
                // binary64 pipe: b - a, 1 + t^2, one rsqrt, s = c t
                if (rf >= (float)stop) rmax = T(1);
                t = jacobi_tangent64(be - al, ga);
                cs = rsqrt(T(1) + t * t);
              } else {
                rmax = fmax(rmax, ratio);
                t = jacobi_tangent32(be - al, ga);
                cs = rsqrtf(T(1) + t * t);
              }
              const T sn = cs * t;
  #pragma unroll
              for (int u = 0; u < B; ++u) {
                const int i = sl + u * L;
                if (i < q) {
                  x[i] = cs * x0[u] - sn * y0[u];
                  y[i] = sn * x0[u] + cs * y0[u];
                }
              }
              for (int i0 = sl + B * L; i0 < q; i0 += B * L) {
                T xr[B], yr[B];
  #pragma unroll
                for (int u = 0; u < B; ++u) {
                  const int i = i0 + u * L;
                  xr[u] = i < q ? x[i] : T(0);
                  yr[u] = i < q ? y[i] : T(0);
                }
  #pragma unroll
                for (int u = 0; u < B; ++u) {
                  const int i = i0 + u * L;
                  if (i < q) {
                    x[i] = cs * xr[u] - sn * yr[u];
                    y[i] = sn * xr[u] + cs * yr[u];
                  }
                }
              }
              TV* vx = V + (size_t)a * ldv;
              TV* vy = V + (size_t)b * ldv;
              const TV cv = (TV)cs, sv = (TV)sn;
              for (int i0 = sl; i0 < p; i0 += B * L) {
                TV xr[B], yr[B];
  #pragma unroll
                for (int u = 0; u < B; ++u) {
                  const int i = i0 + u * L;
                  xr[u] = i < p ? vx[i] : TV(0);
                  yr[u] = i < p ? vy[i] : TV(0);
                }
  #pragma unroll
                for (int u = 0; u < B; ++u) {
                  const int i = i0 + u * L;
                  if (i < p) {
                    vx[i] = cv * xr[u] - sv * yr[u];
                    vy[i] = sv * xr[u] + cv * yr[u];
                  }
                }
              }
              na = al - t * ga;
              nb = be + t * ga;
              done = true;
              rot = 1;
            }
          }
          __syncwarp();              // every lane of the pair has read the old norms
          if (done && sl == 0) {
            nrm[a] = na;
            nrm[b] = nb;
          }
}

// One-sided (Hestenes) Jacobi run by a group of nw warps (warp lw of the
// group, barrier id bar): W (q x p column-major, q >= p, leading dimension
// ldw), rotations accumulated into V (p x p, leading dimension ldv, holds the
// starting basis), column norms cached in nrm and recomputed at every sweep
// start.  Round-robin pairing: every round's pairs are disjoint.  L lanes
// work on one pair, so a warp rotates 32 / L pairs at once (more pairs in
// flight, shorter reductions; the rotations are latency-bound, not
// arithmetic-bound); each pair's work is one jacobi_pass.  Stops after a
// sweep with no rotation or whose largest ratio |g| / sqrt(a b) is below
// `stop` (the next sweep's off-diagonals are then of order stop^2).  Returns
// the sweeps, or -1 when max_sweeps ran out.
template <typename T, typename TV, int L, int B>
__device__ int jacobi_lanes(T* __restrict__ W, int q, int ldw, int p, TV* __restrict__ V, int ldv,
                            T* __restrict__ nrm, int lw, int nw, int bar, int g, GroupSh& gs, T stop, int max_sweeps) {
  constexpr int PPW = 32 / L;              // pairs per warp at once
  const int lane = threadIdx.x & 31;
  const int sub = lane / L, sl = lane % L;
  const int nthr = 32 * nw;
  const T eps = sizeof(T) == sizeof(double) ? T(2.220446049250313e-16) : T(1.1920928955078125e-07);
  const T tol = sqrt((T)q) * eps;
  const int p2 = p + (p & 1);
  const int npair = p2 / 2;
  for (int sweep = 1; sweep <= max_sweeps; ++sweep) {
    for (int j = lw; j < p; j += nw) {
      const T* cj = W + (size_t)j * ldw;
      T s2 = T(0);
      for (int i = lane; i < q; i += 32) s2 = fma(cj[i], cj[i], s2);
      s2 = warp_sum_t(s2);
      if (lane == 0) nrm[j] = s2;
    }
    if (lw == 0 && lane == 0) {
      gs.flag[g] = 0;
      gs.rbits[g] = 0u;
    }
    group_sync(bar, nthr);
    T rmax = T(0);
    int rot = 0;
    for (int rd = 0; rd < p2 - 1; ++rd) {
      for (int base = lw * PPW; base < npair; base += nw * PPW) {   // warp-uniform
        const int pi = base + sub;
        int a = -1, b = -1;
        if (pi < npair) {
          const int m = p2 - 1;          // (rd +- pi) mod m, 0 <= rd < m, 0 < pi < m
          if (pi == 0) {
            a = rd;
            b = m;
          } else {
            a = rd + pi;
            if (a >= m) a -= m;
            b = rd - pi;
            if (b < 0) b += m;
          }
          if (a >= p || b >= p) a = b = -1;
        }
        jacobi_pass<T, TV, L, B>(W, q, ldw, p, V, ldv, nrm, a, b, sl, tol, stop, rmax, rot);
      }
      group_sync(bar, nthr);
    }
    // warp max of the ratios, then one atomic per warp
    float rm32 = (float)rmax;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rm32 = fmaxf(rm32, __shfl_xor_sync(0xffffffffu, rm32, o));
    const int anyrot = __any_sync(0xffffffffu, rot);
    if (lane == 0) {
      if (anyrot) atomicMax(&gs.flag[g], 1);
      atomicMax(&gs.rbits[g], __float_as_uint(rm32));
    }
    group_sync(bar, nthr);
    const int any = gs.flag[g];
    const T rm = (T)__uint_as_float(gs.rbits[g]);
    group_sync(bar, nthr);
    if (!any || rm < stop) return sweep;
  }
  return -1;
}

// Block-ordered one-sided Jacobi for the binary32 sweeps.  The columns form
// super-columns of C = 4, and the round-robin tournament pairs the
// super-columns (ns2 - 1 super-rounds, ns2 = super-columns rounded up to
// even).  A warp owns the eight columns of its super-pair for a whole
// super-round.  It rotates every column of one super-column against every
// column of the other: four sub-rounds of four disjoint pairs, one pair per
// 8 lanes.  In the first super-round it also rotates the pairs inside both
// super-columns (three sub-rounds).  Only __syncwarp separates its
// sub-rounds.  A sweep still visits every pair once, as in jacobi_lanes,
// with the same passes per warp, but waits at ns2 - 1 group barriers
// instead of p - 1: the barrier, not the arithmetic, was what the sweeps
// waited on.  Same arguments, stopping rule and result as jacobi_lanes.
template <typename T, typename TV, int B>
__device__ int jacobi_blocks(T* __restrict__ W, int q, int ldw, int p, TV* __restrict__ V, int ldv,
                             T* __restrict__ nrm, int lw, int nw, int bar, int g, GroupSh& gs, T stop, int max_sweeps) {
  constexpr int L = 8, C = 4;              // 32 / L = C pairs per pass
  const int lane = threadIdx.x & 31;
  const int sub = lane / L, sl = lane % L;
  const int nthr = 32 * nw;
  const T eps = sizeof(T) == sizeof(double) ? T(2.220446049250313e-16) : T(1.1920928955078125e-07);
  const T tol = sqrt((T)q) * eps;
  const int ns = (p + C - 1) / C, ns2 = ns + (ns & 1), nsp = ns2 / 2;
  for (int sweep = 1; sweep <= max_sweeps; ++sweep) {
    for (int j = lw; j < p; j += nw) {
      const T* cj = W + (size_t)j * ldw;
      T s2 = T(0);
      for (int i = lane; i < q; i += 32) s2 = fma(cj[i], cj[i], s2);
      s2 = warp_sum_t(s2);
      if (lane == 0) nrm[j] = s2;
    }
    if (lw == 0 && lane == 0) {
      gs.flag[g] = 0;
      gs.rbits[g] = 0u;
    }
    group_sync(bar, nthr);
    T rmax = T(0);
    int rot = 0;
    for (int sr = 0; sr < ns2 - 1; ++sr) {
      for (int sp = lw; sp < nsp; sp += nw) {                       // warp-uniform
        const int m = ns2 - 1;             // (sr +- sp) mod m, as for the columns
        int A, Bc;
        if (sp == 0) {
          A = sr;
          Bc = m;
        } else {
          A = sr + sp;
          if (A >= m) A -= m;
          Bc = sr - sp;
          if (Bc < 0) Bc += m;
        }
        const bool okA = A < ns, okB = Bc < ns;                     // ns2 > ns: one padding super-column
        if (sr == 0) {
          // pairs inside A (lanes 0-15) and inside B (lanes 16-31): the
          // round robin of four columns, (k, 3) and ((k + 1) % 3, (k + 2) % 3)
          const int base = (sub < 2 ? A : Bc) * C;
          const bool ok = sub < 2 ? okA : okB;
          for (int k = 0; k < C - 1; ++k) {
            int a = base + ((sub & 1) == 0 ? k : (k + 1) % (C - 1));
            int b = base + ((sub & 1) == 0 ? C - 1 : (k + 2) % (C - 1));
            if (!ok || a >= p || b >= p) a = b = -1;
            jacobi_pass<T, TV, L, B>(W, q, ldw, p, V, ldv, nrm, a, b, sl, tol, stop, rmax, rot);
            __syncwarp();                  // the norms stored by the pass are read by other lanes next
          }
        }
        if (okA && okB) {
          for (int k = 0; k < C; ++k) {
            int a = A * C + sub, b = Bc * C + ((sub + k) & (C - 1));
            if (a >= p || b >= p) a = b = -1;
            jacobi_pass<T, TV, L, B>(W, q, ldw, p, V, ldv, nrm, a, b, sl, tol, stop, rmax, rot);
            __syncwarp();
          }
        }
      }
      group_sync(bar, nthr);
    }
    float rm32 = (float)rmax;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rm32 = fmaxf(rm32, __shfl_xor_sync(0xffffffffu, rm32, o));
    const int anyrot = __any_sync(0xffffffffu, rot);
    if (lane == 0) {
      if (anyrot) atomicMax(&gs.flag[g], 1);
      atomicMax(&gs.rbits[g], __float_as_uint(rm32));
    }
    group_sync(bar, nthr);
    const int any = gs.flag[g];
    const T rm = (T)__uint_as_float(gs.rbits[g]);
    group_sync(bar, nthr);
    if (!any || rm < stop) return sweep;
  }
  return -1;
}

// Two binary32 operations in one instruction (sm_100 and later).
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
#if defined(__CUDA_ARCH__)
  unsigned long long x, y, z, r;
  memcpy(&x, &a, 8);
  memcpy(&y, &b, 8);
  memcpy(&z, &c, 8);
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(x), "l"(y), "l"(z));
  float2 d;
  memcpy(&d, &r, 8);
  return d;
#else
  return {fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y)};
#endif
}

__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
#if defined(__CUDA_ARCH__)
  unsigned long long x, y, r;
  memcpy(&x, &a, 8);
  memcpy(&y, &b, 8);
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
  float2 d;
  memcpy(&d, &r, 8);
  return d;
#else
  return {a.x * b.x, a.y * b.y};
#endif
}

__device__ __forceinline__ float2 add2p(float2 a, float2 b) {
#if defined(__CUDA_ARCH__)
  unsigned long long x, y, r;
  memcpy(&x, &a, 8);
  memcpy(&y, &b, 8);
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
  float2 d;
  memcpy(&d, &r, 8);
  return d;
#else
  return {a.x + b.x, a.y + b.y};
#endif
}

// a - b as one multiply-add (exact product with -1).
__device__ __forceinline__ float2 sub2p(float2 a, float2 b) { return fma2(b, {-1.0f, -1.0f}, a); }

// Leading dimension of a binary32 column for jacobi_regs: a multiple of four
// (128-bit loads), an odd one (lanes that read the same rows of eight columns
// hit different banks).
__host__ __device__ __forceinline__ int ld4(int n) { return (((n + 3) >> 2) | 1) * 4; }

// Register rows of jacobi_regs: lane sl of a column's eight holds rows 4 (sl + 8
// u) .. + 3, u < U, as two pairs; n rows (zeros beyond, and up to a multiple of 4
// in memory).
template <int U>
__device__ __forceinline__ void load_rows(const float* col, int n, int sl, bool ok, float2 (&x)[2 * U]) {
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int r = 4 * (sl + 8 * u);
    float4 v = {0.0f, 0.0f, 0.0f, 0.0f};
    if (ok && r < n) v = *reinterpret_cast<const float4*>(col + r);
    x[2 * u] = {v.x, v.y};
    x[2 * u + 1] = {v.z, v.w};
  }
}

template <int U>
__device__ __forceinline__ void store_rows(float* col, int n, int sl, bool ok, const float2 (&x)[2 * U]) {
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int r = 4 * (sl + 8 * u);
    if (ok && r < n)
      *reinterpret_cast<float4*>(col + r) = {x[2 * u].x, x[2 * u].y, x[2 * u + 1].x, x[2 * u + 1].y};
  }
}

// (x, y) <- (c x - s y, s x + c y).  Conformal whatever the rounding of c and s:
// three shears by tan(angle / 2) and sin(angle) would take three operations
// instead of four, but those two are rounded apart, and V's overlaps then
// grew to 2e-6 (measured).
template <int U>
__device__ __forceinline__ void rotate_rows(float2 (&x)[2 * U], float2 (&y)[2 * U], float c, float s) {
  const float2 cc = {c, c}, ss = {s, s}, ms = {-s, -s};
#pragma unroll
  for (int v = 0; v < 2 * U; ++v) {
    const float2 a = x[v], b = y[v];
    x[v] = fma2(cc, a, mul2(ms, b));
    y[v] = fma2(cc, b, mul2(ss, a));
  }
}

template <int U>
__device__ __forceinline__ void move_rows(float2 (&x)[2 * U], int src) {
#pragma unroll
  for (int v = 0; v < 2 * U; ++v) {
    x[v].x = lane_value(x[v].x, src);
    x[v].y = lane_value(x[v].y, src);
  }
}

template <int U>
__device__ __forceinline__ float dot_rows(const float2 (&x)[2 * U], const float2 (&y)[2 * U]) {
  float2 a = {0.0f, 0.0f}, b = {0.0f, 0.0f};
#pragma unroll
  for (int u = 0; u < U; ++u) {
    a = fma2(x[2 * u], y[2 * u], a);
    b = fma2(x[2 * u + 1], y[2 * u + 1], b);
  }
  return (a.x + b.x) + (a.y + b.y);
}

// Rotation (c, s) and tangent t of a pair with squared norms na, nb and dot
// product ga, by half-angle forms: with d = nb - na and h = sqrt(d^2 + 4 ga^2), c^2
// = (1 + |d| / h) / 2 and s = sign(d) ga / (h c).  Two dependent reciprocal
// square roots instead of two divides and two reciprocal square roots: the
// angle is the longest link of a sub-round's chain.  d and ga are scaled by 1 /
// sqrt(na nb), known before the dot product is.  (c, s) is conformal whatever
// its rounding.  Returns the ratio |ga| / sqrt(na nb), or 0 (and c = 1, s = t =
// 0) when the pair is not rotated: below tol, a column below kTiny32 (noise
// at binary32 resolution; the fast reciprocal square root flushes subnormal
// inputs to 0), or |d|, the ratio of the two lengths, above 1e18: its square
// would overflow from 1.8e19 on, and the angle is far below binary32 resolution.  (An
// exact form for those, one more reciprocal and a select on the chain, took
// 2 to 3 % of a step; the binary64 finish rotates such a pair.)
__device__ __forceinline__ float jacobi_angle32(float na, float nb, float ga, float tol, float& c, float& s, float& t) {
  const float inv = rsqrtf(fmaxf(na, kTiny32)) * rsqrtf(fmaxf(nb, kTiny32));
  const float d = (nb - na) * inv, g = ga * inv;
  const float ratio = fabsf(g);
  const bool go = ratio > tol && na > kTiny32 && nb > kTiny32 && fabsf(d) < 1e18f;
  const float ih = rsqrtf(fmaf(d, d, 4.0f * (g * g)));
  const float c2 = fmaf(0.5f, fabsf(d) * ih, 0.5f);
  const float rc = rsqrtf(c2);
  const float sg = d < 0.0f ? -g : g;
  c = go ? c2 * rc : 1.0f;
  s = go ? sg * ih * rc : 0.0f;
  t = go ? s * rc : 0.0f;
  return go ? ratio : 0.0f;
}

// The three rounds of pairs inside a super-column of four, its column a lane
// group's x (W) and v (V) with squared norm nx (0: no column): groups exchange
// copies with the group m away, m = 1, 2, 3, and each rotates its own column.
template <int U>
__device__ __forceinline__ void intra_rows(float2 (&x)[2 * U], float2 (&v)[2 * U], float& nx, float tol, float& rmax) {
  const int lane = threadIdx.x & 31, sub = lane >> 3;
#pragma unroll 1
  for (int m = 1; m < 4; ++m) {
    const int src = lane ^ (8 * m);
    const bool first = sub < (sub ^ m);
    float2 y[2 * U];
#pragma unroll
    for (int u = 0; u < 2 * U; ++u) y[u] = x[u];
    move_rows<U>(y, src);
    const float ny = lane_value(nx, src);
    float ga = dot_rows<U>(x, y);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) ga += __shfl_xor_sync(0xffffffffu, ga, o);
    float c, s, t;
    const float ratio = jacobi_angle32(first ? nx : ny, first ? ny : nx, ga, tol, c, s, t);
    rmax = fmaxf(rmax, ratio);
    nx += first ? -t * ga : t * ga;
    const float ps = first ? -s : s;
    const float2 cc = {c, c}, ss = {ps, ps};
#pragma unroll
    for (int u = 0; u < 2 * U; ++u) {
      x[u] = fma2(cc, x[u], mul2(ss, y[u]));
      const float2 o = {lane_value(v[u].x, src), lane_value(v[u].y, src)};
      v[u] = fma2(cc, v[u], mul2(ss, o));
    }
  }
}

// Block-ordered one-sided Jacobi as in jacobi_blocks, with a super-pair's eight
// columns of W and V in registers for all of its sub-rounds (q <= 32 U; W
// and V 16-byte aligned, leading dimensions multiples of 4).
//
// jacobi_blocks loads and stores every column of W and V once per rotation: 8 n
// shared-memory words a pair against 9 n multiply-adds, and shared memory moves
// 32 words a clock where the SM does 128 multiply-adds, so its traffic bounded
// the sweeps of large blocks (82k clocks a sweep of a split against 107k at full
// traffic, Lx = 16, chi = 200).  Here a column is loaded and stored once per
// super-pair (128-bit accesses); lane group `sub` keeps column A + sub, and the
// columns of the other super-column move on to the next group by shuffles.
// What is left is the chain of a sub-round (dot product, reduction, angle,
// rotation: ~300 clocks).  Super-columns of eight (4 lanes a pair) measured 3 %
// faster on blocks of up to 32 rows and 10 % slower above.
// Lx = 9, 2W = 8, chi = 256, binary32, 152 chains: 269 ms a Markov step with
// jacobi_blocks, 208 ms with this (170 ms with the steps after it).
//
// Two copies, U = 2 and 4, for every size.  The groups of a CTA work on blocks of
// different sizes at once, and four copies (and the shared-memory pass for the pairs
// inside a super-column) overflowed the instruction cache: 8.6 of 21.9
// clocks an instruction went to waiting for instructions (Lx = 6, chi = 96, two
// chains per SM).  One copy that skips unused rows by branches was faster
// there (ladder of Lx = 16, 256 chains: 761 -> 651 ms a step) but its branches sit
// on the chain of every sub-round (Lx = 9, one chain per SM: 196 -> 256 ms).
template <int U>
__device__ int jacobi_regs(float* __restrict__ W, int q, int ldw, int p, float* __restrict__ V, int ldv,
                                  float* __restrict__ nrm, int lw, int nw, int bar, int g, GroupSh& gs, float stop,
                                  int max_sweeps) {
  constexpr int L = 8, C = 4;
  const int lane = threadIdx.x & 31;
  const int sub = lane / L, sl = lane % L;
  const int nthr = 32 * nw;
  const float tol = sqrtf((float)q) * 1.1920928955078125e-07f;
  const int ns = (p + C - 1) / C, ns2 = ns + (ns & 1), nsp = ns2 / 2;
  const int next = ((sub + 1) & (C - 1)) * L + sl;   // the lane whose column this one takes next
  for (int j = lw; j < p; j += nw) {                 // padding rows
    if (q + lane < ((q + 3) & ~3)) W[(size_t)j * ldw + q + lane] = 0.0f;
    if (p + lane < ((p + 3) & ~3)) V[(size_t)j * ldv + p + lane] = 0.0f;
  }
  for (int sweep = 1; sweep <= max_sweeps; ++sweep) {
    for (int j = lw; j < p; j += nw) {
      const float* cj = W + (size_t)j * ldw;
      float s2 = 0.0f;
      for (int i = lane; i < q; i += 32) s2 = fmaf(cj[i], cj[i], s2);
      s2 = warp_sum_t(s2);
      if (lane == 0) nrm[j] = s2;
    }
    if (lw == 0 && lane == 0) gs.rbits[g] = 0u;
    group_sync(bar, nthr);
    float rmax = 0.0f;                     // > 0: some pair was rotated
    for (int sr = 0; sr < ns2 - 1; ++sr) {
      for (int sp = lw; sp < nsp; sp += nw) {                       // warp-uniform
        const int m = ns2 - 1;             // (sr +- sp) mod m, as for the columns
        int A, Bc;
        if (sp == 0) {
          A = sr;
          Bc = m;
        } else {
          A = sr + sp;
          if (A >= m) A -= m;
          Bc = sr - sp;
          if (Bc < 0) Bc += m;
        }
        const bool both = A < ns && Bc < ns;         // ns2 > ns: one padding super-column
        if (!both && sr > 0) continue;
        const int a = A * C + sub;
        int b = Bc * C + sub;
        float2 xa[2 * U], xb[2 * U], va[2 * U], vb[2 * U];
        load_rows<U>(W + (size_t)a * ldw, q, sl, a < p, xa);
        load_rows<U>(W + (size_t)b * ldw, q, sl, b < p, xb);
        load_rows<U>(V + (size_t)a * ldv, p, sl, a < p, va);
        load_rows<U>(V + (size_t)b * ldv, p, sl, b < p, vb);
        float na = a < p ? nrm[a] : 0.0f, nb = b < p ? nrm[b] : 0.0f;   // 0: no pair
        float rs = 0.0f;                             // largest ratio rotated here
        if (sr == 0) {
          intra_rows<U>(xa, va, na, tol, rs);
          intra_rows<U>(xb, vb, nb, tol, rs);
        }
        if (both) {
          float ga = dot_rows<U>(xa, xb);
#pragma unroll
          for (int o = L / 2; o > 0; o >>= 1) ga += __shfl_xor_sync(0xffffffffu, ga, o);
#pragma unroll 1
          for (int k = 0; k < C; ++k) {
            float cs, sn, t;
            rs = fmaxf(rs, jacobi_angle32(na, nb, ga, tol, cs, sn, t));
            na -= t * ga;
            nb += t * ga;
            rotate_rows<U>(xa, xb, cs, sn);
            // the next pair's dot product first: V's rotation and move fill the
            // latency of its reduction (the last move brings the columns home)
            move_rows<U>(xb, next);
            nb = lane_value(nb, next);
            ga = dot_rows<U>(xa, xb);
            ga += __shfl_xor_sync(0xffffffffu, ga, 4);
            rotate_rows<U>(va, vb, cs, sn);
            ga += __shfl_xor_sync(0xffffffffu, ga, 2);
            move_rows<U>(vb, next);
            ga += __shfl_xor_sync(0xffffffffu, ga, 1);
          }
        }
        if (__any_sync(0xffffffffu, rs > 0.0f)) {
          rmax = fmaxf(rmax, rs);
          store_rows<U>(W + (size_t)a * ldw, q, sl, a < p, xa);
          store_rows<U>(W + (size_t)b * ldw, q, sl, b < p, xb);
          store_rows<U>(V + (size_t)a * ldv, p, sl, a < p, va);
          store_rows<U>(V + (size_t)b * ldv, p, sl, b < p, vb);
          if (sl == 0) {
            if (a < p) nrm[a] = na;
            if (b < p) nrm[b] = nb;
          }
        }
        __syncwarp();
      }
      group_sync(bar, nthr);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rmax = fmaxf(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
    if (lane == 0) atomicMax(&gs.rbits[g], __float_as_uint(rmax));
    group_sync(bar, nthr);
    const float rm = __uint_as_float(gs.rbits[g]);
    group_sync(bar, nthr);
    if (rm < stop) return sweep;             // 0: no rotation
  }
  return -1;
}

// One-sided Jacobi of one block by a warp group: jacobi_regs for binary32
// blocks of up to 128 rows; above, the block ordering in shared memory for 16
// columns or more; otherwise (binary64) the round-robin ordering with 8 lanes a
// pair.  None of them depends on the number of warps, nor does anything else a
// block goes through that fits the kernel's buffer.  So a chain's results are the
// same bits in every batch and team while all its blocks fit half an SM (104 KB in
// binary64: 79 x 79; 109 KB in the mixed kernel: 116 x 116).  A wider block takes a path of
// its own in the build for two chains per SM, and its bits depend on the build.
// TV: element type of V.  A binary64 polish of a binary32 result may keep V
// in binary32: V carries binary32 accuracy from the preconditioning sweeps
// anyway, and the polish's rotations are tiny (angles ~1e-6).
// B: rows per lane and batch (register budget: 4 B values of T in flight).
// A lane's rows are rounded up to a multiple of B, and on the binary64 pipe
// every issued instruction costs the same whatever the lanes' predicates, so
// the binary64 kernels take B = 2.
template <typename T, typename TV = T, int B = 4>
__device__ int jacobi_group(T* __restrict__ W, int q, int ldw, int p, TV* __restrict__ V, int ldv,
                            T* __restrict__ nrm, int lw, int nw, int bar, int g, GroupSh& gs, T stop, int max_sweeps) {
  if constexpr (sizeof(T) == sizeof(float)) {
    const bool vec = ((ldw | ldv) & 3) == 0 && ((reinterpret_cast<uintptr_t>(W) | reinterpret_cast<uintptr_t>(V)) & 15) == 0;
    if (vec && q <= 64) return jacobi_regs<2>(W, q, ldw, p, V, ldv, nrm, lw, nw, bar, g, gs, stop, max_sweeps);
    if (vec && q <= 128) return jacobi_regs<4>(W, q, ldw, p, V, ldv, nrm, lw, nw, bar, g, gs, stop, max_sweeps);
    if (p >= 16) return jacobi_blocks<T, TV, B>(W, q, ldw, p, V, ldv, nrm, lw, nw, bar, g, gs, stop, max_sweeps);
  }
  return jacobi_lanes<T, TV, 8, B>(W, q, ldw, p, V, ldv, nrm, lw, nw, bar, g, gs, stop, max_sweeps);
}

// Work of one block's sweeps, in units that only matter relative to each
// other: p^2 / 2 pairs, each a fixed part (reduction, angle) and its rows.
__device__ __forceinline__ int block_cost(int q, int p) { return p * p * (q + 48) / 8 + 256 * p; }

// Warp groups for one wave of nblk <= 15 blocks (costs `cost`, columns p).
// With warps for all super-pairs of all blocks (a sub-round handles eight
// columns), every block has a group of its own.  Otherwise a block that is
// worth a warp or more does, and smaller ones are put together, one after
// another, until they are worth one: with one warp at least for every block,
// a split of eight blocks on eight warps took 2.6 times as long as its work
// (Lx = 16, chi = 256, 256 chains: 808 -> 750 ms a step when it was made, 392 ms with
// the steps after it; but 16 chains of Lx = 5, where the warps are plenty, 77 -> 84 ms, hence
// the first case).  Then the
// warps go one at a time to the group that takes longest, at most p / 2 to
// one.  Writes every block's group and every group's first warp and warp
// count; returns the groups.  One thread.
__device__ inline int assign_warps(const int* p, const int* cost, int nblk, int nwarps, int32_t* grp, int32_t* w0,
                                   int32_t* nw) {
  int total = 0, pairs = 0;
  for (int b = 0; b < nblk; ++b) total += cost[b] >> 4, pairs += (p[b] + 7) / 8;
  const bool plenty = pairs <= nwarps;
  const int share = total / nwarps + 1;
  int load[15], cap[15], ng = 0, open = -1;
  for (int b = 0; b < nblk; ++b) {
    const bool own = plenty || ((cost[b] >> 4) >= share && ng < nwarps);
    int g = own ? -1 : open;
    if (g < 0) {
      // at most nwarps groups: past that, blocks join the lightest one
      if (ng < nwarps) {
        g = ng++;
        load[g] = 0;
        cap[g] = 1;
        nw[g] = 1;
      } else {
        g = 0;
        for (int i = 1; i < ng; ++i)
          if (load[i] < load[g]) g = i;
      }
    }
    grp[b] = g;
    load[g] += cost[b] >> 4;
    cap[g] = max(cap[g], (p[b] + 1) / 2);
    if (!own) open = load[g] >= share ? -1 : g;
  }
  for (int used = ng; used < nwarps; ++used) {
    int best = -1, bt = -1;
    for (int g = 0; g < ng; ++g)
      if (nw[g] < cap[g] && load[g] / nw[g] > bt) bt = load[g] / nw[g], best = g;
    if (best < 0) break;
    ++nw[best];
  }
  for (int g = 0, w = 0; g < ng; ++g) w0[g] = w, w += nw[g];
  return ng;
}

// Blocks a team shares out one by one; a split with more stays with rank 0.
constexpr int kTeamBlk = 64;

// One wave of the blocks a CTA owns: its blocks [b0, b0 + n) decomposed at
// once, group g (barrier id g + 1) taking those with grp[i] = g in turn on its
// warps [w0[g], w0[g] + nw[g]).
struct WaveSh {
  int32_t nown;                           // blocks of this CTA
  int32_t all;                            // it has them all (own unused)
  int16_t own[kTeamBlk];
  int32_t b0, n, ng;
  int32_t grp[15], w0[15], nw[15], sw[15];
  int32_t off[15];                        // shared-memory offset (elements) of block i
};

__device__ __forceinline__ int own_block(const WaveSh& wv, int i) { return wv.all ? i : wv.own[i]; }

// Shares the blocks of a split out over the team: the costliest block still
// unassigned goes to the CTA with the least work (q p^2).  Every CTA computes
// the same assignment.  One thread.  fits(q, p): the block can be decomposed
// in shared memory; a split with one that cannot stays with rank 0, whose
// scratch is then the whole buffer.
template <typename F>
__device__ inline void own_blocks(const SplitSh& s, const Team& tm, WaveSh& wv, F&& fits) {
  bool alone = tm.size == 1 || s.nblk > kTeamBlk;
  for (int b = 0; b < s.nblk && !alone; ++b) alone = !fits(s.b[b].q, s.b[b].p);
  wv.all = alone;
  wv.nown = alone && tm.rank == 0 ? s.nblk : 0;
  if (alone) return;
  int load[16];
  for (int r = 0; r < tm.size; ++r) load[r] = 0;
  unsigned long long done = 0;
  for (int t = 0; t < s.nblk; ++t) {
    int best = -1, bc = -1;
    for (int b = 0; b < s.nblk; ++b) {
      const int cost = block_cost(s.b[b].q, s.b[b].p);
      if (!((done >> b) & 1ull) && cost > bc) bc = cost, best = b;
    }
    done |= 1ull << best;
    int to = 0;
    for (int r = 1; r < tm.size; ++r)
      if (load[r] < load[to]) to = r;
    load[to] += bc;
    if (to == tm.rank) wv.own[wv.nown++] = (int16_t)best;
  }
}

// Index of this warp's group in the wave, or -1 (an idle warp).
__device__ __forceinline__ int my_group(const WaveSh& wv, int warp) {
  for (int i = 0; i < wv.ng; ++i)
    if (warp >= wv.w0[i] && warp < wv.w0[i] + wv.nw[i]) return i;
  return -1;
}

__device__ __forceinline__ double warp_sum64(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Truncation rule (Sec. II): smallest k >= 1 whose discarded weight
// sum_{q>=k} s_q^2 / sum s^2 <= cutoff, then min(k, chi_max), then lowered to
// the nearest gap s_k < s_{k-1} (1 - 1e-8).  s sorted descending; one thread (the
// allocation-free update; the evolve kernels take warp_trunc_rank).
__device__ inline int trunc_rank(const double* s, int n, int chi_max, double cutoff, double* tail, double* total_out) {
  tail[n] = 0.0;
  for (int q = n - 1; q >= 0; --q) tail[q] = tail[q + 1] + s[q] * s[q];
  const double total = tail[0];
  *total_out = total;
  int k = n;
  for (int kk = 1; kk <= n; ++kk) {
    if (tail[kk] <= cutoff * total) {
      k = kk;
      break;
    }
  }
  if (k > chi_max) k = chi_max;
  while (k > 1 && k < n && s[k] >= s[k - 1] * (1.0 - 1e-8)) --k;
  return k;
}

// Dense-SVD flop count 4 M^2 N + 8 M N^2 + 9 N^3 of an m x n matrix (M >= N).
__device__ __forceinline__ double svd_count(double m, double n) {
  const double M = m > n ? m : n, N = m > n ? n : m;
  return 4.0 * M * M * N + 8.0 * M * N * N + 9.0 * N * N * N;
}

// Order-preserving integer key of a value >= 0 (compares on the integer
// pipe; a binary64 compare is a binary64 instruction).
__device__ __forceinline__ unsigned long long sort_key(double x) {
  unsigned long long b;
  memcpy(&b, &x, 8);
  return b;
}

// Bytes of finish()'s scratch for P values.
__device__ __forceinline__ size_t finish_bytes(int P) { return (size_t)P * (4 * sizeof(double) + 4 * sizeof(int32_t)); }

// The truncation rule of trunc_rank on n sorted values by one warp: every
// lane owns a run of values and sums it from its smallest value up, the
// runs are joined by a suffix sum over the lanes.  Returns the kept count;
// *kept and *tail get the kept and the discarded weight.
// Rolled loops: one warp runs it once an op while the others wait, and on small
// splits it is bound by fetching its instructions (one rung, METTS: 32.2 us an op
// unrolled, 31.5 rolled, HM_MIXED32; 24.4 and 23.3, HM_FP64).
__device__ inline int warp_trunc_rank(const double* s, int n, int chi_max, double cutoff, double* kept, double* tail) {
  const int lane = threadIdx.x & 31;
  const int per = (n + 31) / 32;
  const int i0 = min(lane * per, n), i1 = min(i0 + per, n);
  double own = 0.0;
  for (int i = i1 - 1; i >= i0; --i) own = fma(s[i], s[i], own);
  double suf = own;                        // sum over this lane and the later ones
#pragma unroll 1
  for (int o = 1; o < 32; o <<= 1) {
    const double y = lane_value(suf, lane + o < 32 ? lane + o : lane);
    if (lane + o < 32) suf += y;
  }
  const double total = lane_value(suf, 0);
  double run = lane_value(suf, lane < 31 ? lane + 1 : 31);
  if (lane == 31) run = 0.0;
  // smallest kk >= 1 with sum_{q >= kk} s_q^2 <= cutoff total
  int k = n;
  const double bar = cutoff * total;
  for (int i = i1 - 1; i >= i0; --i) {
    // run = tail of kept count i + 1
    if (run <= bar) k = min(k, i + 1);
    run = fma(s[i], s[i], run);
  }
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) k = min(k, __shfl_xor_sync(0xffffffffu, k, o));
  if (k > chi_max) k = chi_max;
  while (k > 1 && k < n && s[k] >= s[k - 1] * (1.0 - 1e-8)) --k;
  double a = 0.0, b = 0.0;
  for (int i = lane; i < n; i += 32) {
    if (i < k) a = fma(s[i], s[i], a);
    else b = fma(s[i], s[i], b);
  }
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  *kept = a;
  *tail = b;
  return k;
}

// Phase D: singular values of every block (column norms of its converged W,
// binary64), one descending order over all blocks, the truncation rule,
// renormalisation, then the new bond grouped by charge (ascending; by value
// within a charge), the absorb into A_k and A_{k+1} (the blocks only) and the
// new middle charges.  W and V hold every block's binary64
// result.  scratch: finish_bytes(P) bytes; tiles: per warp 8 x 33 doubles of
// shared memory (the transposition of the left factor).
//
// The binary64 pipe and dependent loads bound this phase, not its traffic: the
// order compares integer keys, the truncation sums run over a warp, a kept
// value's scales cost one divide each (not one per element), the absorb goes
// block by block instead of looking up each element's block, and it writes the
// blocks only: zeros around them were four fifths of its writes (two tensors
// of 3 chi^2 doubles a split).
template <int NT>
__device__ void finish(ChainDev* c, const OpDev& op, int t, SplitSh& s, const WaveSh& wv, const Team& tm,
                       char* __restrict__ scratch, double* tiles, int32_t* ctx_err, int sweeps32, int sweeps64) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = NT / 32;
  const int k = op.k;
  const int chil = c->chi[k], chim = c->chi[k + 1], chir = c->chi[k + 2];
  const int m = 3 * chil, n = 3 * chir;
  const int nb = s.nblk, P = s.P;
  double* sraw = reinterpret_cast<double*>(scratch);  // P: value of slot
  double* sig = sraw + P;                             // P: sorted values
  double* lsc = sig + P;                              // scales of the kept values in the left factor
  double* rsc = lsc + P;                              // and in the right one
  int32_t* sblk = reinterpret_cast<int32_t*>(rsc + P);   // block of slot
  int32_t* perm = sblk + P;                           // slot of sorted value
  int32_t* key = perm + P;                            // kept value: block, rank
  int32_t* newslot = key + P;                         // slot of new index
  // column norms of this CTA's blocks -> raw values, slot = svoff + column
  {
    int c0 = 0;
    for (int i = 0; i < wv.nown; ++i) {
      const BlockRec& r = s.b[own_block(wv, i)];
      const double* Wb = c->W + r.woff;
      // four columns a warp, eight lanes each
      const int nj = (r.p + 3) >> 2;
      for (int x = (unsigned)(warp - c0) % NW; x < nj; x += NW) {
        const int j = 4 * x + (lane >> 3);
        const double* cj = Wb + (size_t)min(j, r.p - 1) * r.q;
        double s2 = 0.0;
#pragma unroll 4
        for (int e = lane & 7; e < r.q; e += 8) s2 = fma(cj[e], cj[e], s2);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        if ((lane & 7) == 0 && j < r.p) c->sig[r.svoff + j] = sqrt(s2);
      }
      c0 += nj;
    }
  }
  team_sync(tm);                          // every block's W, V and values are there
  // A decomposition failed: nothing to absorb.  One thread reads the status for
  // its CTA: rank 0 may set it below while another CTA of the team is still
  // here, and threads of one CTA that saw different values would part at the next
  // barrier.  (A CTA that sees that later value returns, as it would below.)
  if (tid == 0) s.ok = *(volatile int32_t*)c->status == 0;
  for (int j = tid; j < P; j += NT) sraw[j] = c->sig[j];
  for (int b = warp; b < nb; b += NW)
    for (int j = lane; j < s.b[b].p; j += 32) sblk[s.b[b].svoff + j] = b;
  __syncthreads();
  if (!s.ok) return;
  // descending rank (ties by slot): sig[rank] = value, perm[rank] = slot
  for (int j = tid; j < P; j += NT) {
    const double sj = sraw[j];
    const unsigned long long kj = sort_key(sj);
    int rank = 0;
#pragma unroll 8
    for (int i = 0; i < j; ++i) rank += sort_key(sraw[i]) >= kj;
#pragma unroll 8
    for (int i = j + 1; i < P; ++i) rank += sort_key(sraw[i]) > kj;
    sig[rank] = sj;
    perm[rank] = j;
  }
  __syncthreads();
  if (warp == 0) {
    double kept = 1.0, tail = 0.0, nrm = 1.0;
    int kk;
    if (!op.exact) {
      kk = warp_trunc_rank(sig, P, c->chi_max, c->cutoff, &kept, &tail);
      const double total = kept + tail;
      if (!(total > 0.0) || !isfinite(total)) kk = -1;
      else {
        nrm = 1.0 / sqrt(kept);
        tail /= total;
      }
    } else {
      int pos = 0, nan = 0;                  // nonzero values; any that is no number
      for (int i = lane; i < P; i += 32) {
        const unsigned long long v = sort_key(sig[i]);
        pos += v != 0ull;
        nan |= v > 0x7ff0000000000000ull;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) pos += __shfl_xor_sync(0xffffffffu, pos, o);
      kk = min(pos, chim);
      if (kk == 0 || __any_sync(0xffffffffu, nan)) kk = -1;
    }
    if (lane == 0) {
      s.kk = kk;
      s.nrm = nrm;
      if (kk > 0 && tm.rank == 0) {
        double svd = 0.0;
        for (int b = 0; b < nb; ++b) svd += svd_count(s.b[b].mq, s.b[b].nq);
        c->stats[ST_K1] += 2.0 * s.k1;
        c->stats[ST_K2] += 2.0 * 81.0 * chil * chir;
        c->stats[ST_SVD] += svd;
        c->stats[ST_SVD_DENSE] += svd_count(m, n);
        c->stats[ST_DISC] += tail;
        c->stats[ST_SWEEPS] += sweeps32;
        c->stats[ST_SWEEPS64] += sweeps64;
        c->stats[ST_SPLITS] += 1.0;
        c->stats[ST_BLOCKS] += nb;
        if (kk > c->stats[ST_MAXCHI]) c->stats[ST_MAXCHI] = kk;
      }
    }
  }
  __syncthreads();
  const int kk = s.kk;
  const double nrm = s.nrm;
  if (kk <= 0) {
    if (tid == 0 && tm.rank == 0) {
      if (atomicCAS(c->status, 0, HM_ERR_NUMERIC) == 0) *c->err_where = t;
      if (ctx_err) atomicCAS(ctx_err, 0, HM_ERR_NUMERIC);
    }
    return;
  }
  double* __restrict__ Ak = c->site[k];
  double* __restrict__ Ak1 = c->site[k + 1];
  // new position of kept rank i: kept values of lower-charge blocks first,
  // then by rank within the block
  for (int i = tid; i < kk; i += NT) key[i] = sblk[perm[i]] * 16384 + i;
  __syncthreads();
  const bool absorb_left = op.absorb == 0;
  int16_t* qM = c->qn + (size_t)(k + 1) * c->chi_cap;
  for (int i = tid; i < kk; i += NT) {
    const int ki = key[i];
    int pos = 0;
#pragma unroll 8
    for (int j = 0; j < kk; ++j) pos += key[j] < ki;
    const int slot = perm[i], b = sblk[slot];
    newslot[pos] = slot;
    if (tm.rank == 0) qM[pos] = s.b[b].Q;
    const double sg = sraw[slot];
    // W column = U sigma (left) or V sigma (right, transposed block); V column a unit vector
    const bool w_left = !s.b[b].trans;
    const double unit = absorb_left ? (w_left ? 1.0 : sg * nrm) : (w_left ? sg * nrm : 1.0);   // V's side
    const double wsc = absorb_left == w_left ? nrm : 1.0 / sg;
    lsc[pos] = w_left ? wsc : unit;
    rsc[pos] = w_left ? unit : wsc;
  }
  __syncthreads();
  double* tile = tiles + warp * (8 * 33);
  int c0 = 0, pos0 = 0;
  for (int b = 0; b < nb; ++b) {
    const BlockRec& r = s.b[b];
    // kept values of this block: new indices [pos0, pos0 + kb)
    int kb = 0;
    while (pos0 + kb < kk && sblk[newslot[pos0 + kb]] == b) ++kb;
    if (kb == 0) continue;
    const double* L = r.trans ? c->V + r.voff : c->W + r.woff;
    const double* Rf = r.trans ? c->W + r.woff : c->V + r.voff;
    const int ldl = r.trans ? r.p : r.q, ldr = r.trans ? r.q : r.p;
    const int mq = r.mq, nq = r.nq, sv = r.svoff;
    // left factor A_k[(l a), i]: 32 rows x 8 kept values a warp, transposed in shared memory
    const int tv = (mq + 31) >> 5, ti = (kb + 7) >> 3;
    for (int x = (unsigned)(warp + NW * tm.rank - c0) & (NW * tm.size - 1); x < tv * ti; x += NW * tm.size) {
      const int v0 = (x % tv) * 32, j0 = (x / tv) * 8;
      const int nv = min(32, mq - v0), nj = min(8, kb - j0);
      __syncwarp();
      if (lane < nv)
#pragma unroll
        for (int y = 0; y < 8; ++y)
          if (y < nj) {
            const int i = pos0 + j0 + y;
            tile[y * 33 + lane] = L[(size_t)(newslot[i] - sv) * ldl + v0 + lane] * lsc[i];
          }
      __syncwarp();
#pragma unroll
      for (int y = 0; y < 8; ++y) {
        const int vv = y * 4 + (lane >> 3), jj = lane & 7;
        if (vv < nv && jj < nj) {
          const int v = v0 + vv;
          const int a = v >= r.roff[2] ? 2 : (v >= r.roff[1] ? 1 : 0);
          Ak[(size_t)(3 * (r.rst[a] + v - r.roff[a]) + a) * kk + pos0 + j0 + jj] = tile[jj * 33 + vv];
        }
      }
    }
    c0 += tv * ti;
    // right factor A_{k+1}[i, (b r)]
    share<NT>(tm, kb * nq, c0, [&](int e) {
      const int i = pos0 + e / nq, u = e % nq;
      const int bb = u >= r.coff[2] ? 2 : (u >= r.coff[1] ? 1 : 0);
      Ak1[(size_t)i * n + bb * chir + r.cst[bb] + u - r.coff[bb]] =
          Rf[(size_t)(newslot[i] - sv) * ldr + u] * rsc[i];
    });
    pos0 += kb;
  }
  // chi, the signs and qM are read by the split's records only: the barrier
  // at the op's end orders them before the next op
  if (tid == 0 && tm.rank == 0) {
    c->chi[k + 1] = kk;
    c->sgn[k] = s.osk;
    c->sgn[k + 1] = s.osk1;
  }
  __syncthreads();
}

}  // namespace blk
}  // namespace hm
