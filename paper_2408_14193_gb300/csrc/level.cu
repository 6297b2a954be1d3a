// One level of the spaLU factorization (Sec. 4.3, Alg. 2, l = L..1) and its solve.
//
// Data model: the Schur complement A^(l) is the sum over the depth-l boxes of dense
// "frontal" blocks over each box's boundary unknowns (its four sides and corners); a side
// shared by two boxes is one segment.  Per level:
//   sparsify_kernel   one CTA per segment: hybrid sketch Y = [B_N; G B_F / sqrt(h)] of
//                     B = [A_{n,i}; A_{i,n}^T] (Eqs. (Phi), (ID [A_ni; A_in])), column-pivoted
//                     QR and T = R_1^{-1} R_2 (Eqs. (RRQR 1), (RRQR 2)), the transform of the
//                     segment's own block by U_t, L_t (Eq. (UtALt)), LU of the remainder and
//                     its Schur update onto the skeleton (Eq. (L^-1 * A * U^-1)).
//   merge_*_kernels   one parent (depth l-1 box) at a time: extend-add of its two children
//                     restricted to skeletons (the permutation E_(l)), LU of the level-l
//                     separator's skeleton block and the Schur update onto the parent's
//                     boundary, which is the parent's frontal for level l-1.
// The neighbour couplings of a remainder are dropped (they are O(eps) after the
// transform), and the couplings between skeletons are unchanged by the transforms, so only
// the segment's own diagonal block is transformed.
//
// Every kernel is templated on the working precision T (double; float in mixed mode).
// Column norms, pivots and the truncation test of the column-pivoted QR stay in FP64.
// GB300 runs FP64 at 2 FMA per clock per SM, so per-column scalars (Householder coefficients,
// norm downdates) are computed once for 32 columns at a time (one lane per column) and
// divisions are replaced by stored reciprocals.
#include <algorithm>
#include <cfloat>
#include <cmath>

#include <cooperative_groups.h>

#include "pred_infer.cuh"
#include "spalu_internal.h"
#include "work.cuh"

namespace spalu {
namespace {

constexpr int NEAR_MAX = 16;      // near unknowns per segment (the geometry gives <= 10)
constexpr int RUN_MAX = 16;
constexpr int SK_CHUNK = 16;      // far unknowns per chunk of the sketch product (at least)
constexpr int SK_CHUNK_MAX = 64;  // ... and at most, where the shared-memory budget has room
constexpr int NW = 8;             // warps per CTA of the sparsify kernel (segments with e > 32)
constexpr int NW_SMALL = 2;       // ... and for levels whose segments have at most 16 unknowns
constexpr double TIE_RTOL = 1e-12;
constexpr int RSTAGE = 96;        // triangular blocks up to this order are staged in shared memory

// ------------------------------------------------------------ Philox4x32-10 (SC'11)
__device__ __forceinline__ void philox4x32_10(uint32_t c[4], uint32_t k0, uint32_t k1) {
  const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u, W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) { k0 += W0; k1 += W1; }
    uint32_t hi0 = __umulhi(M0, c[0]), lo0 = M0 * c[0];
    uint32_t hi1 = __umulhi(M1, c[2]), lo1 = M1 * c[2];
    uint32_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
  }
}

// Entries of the sampling matrix G for sketch rows 4 g .. 4 g + 3 of one far row: counter
// (g, node, 2l+t, sid), key = seed; the four output words give u1..u4 (odd multiples of
// 2^-24), and float32 Box-Muller turns each pair into two normals:
// z = {R1 cos(2 pi u2), R1 sin(2 pi u2), R2 cos(2 pi u4), R2 sin(2 pi u4)}, R = sqrt(-2 log u).
__device__ __forceinline__ void sketch_gauss4(unsigned long long seed, int l, int sid, int g, int node, int t,
                                              float (&z)[4]) {
  uint32_t c[4] = {(uint32_t)g, (uint32_t)node, (uint32_t)(2 * l + t), (uint32_t)sid};
  philox4x32_10(c, (uint32_t)(seed & 0xffffffffull), (uint32_t)(seed >> 32));
  float u[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) u[i] = (float)(((c[i] >> 9) << 1) | 1u) * 0x1p-24f;
  const float r1 = sqrtf(-2.0f * logf(u[0])), r2 = sqrtf(-2.0f * logf(u[2]));
  const float a1 = 6.283185307179586f * u[1], a2 = 6.283185307179586f * u[3];
  z[0] = r1 * cosf(a1);
  z[1] = r1 * sinf(a1);
  z[2] = r2 * cosf(a2);
  z[3] = r2 * sinf(a2);
}

// ------------------------------------------------------------ neighbour runs of a segment
struct Run {
  int p1, p2, len, ref;   // positions in box 1 / box 2 (-1: absent), count, seg id or -2-node
};

struct SegCtx {
  int sid, e, b1, b2, s1, s2;   // boxes (b1 = lower/left owner) and position of the segment
  int horiz, line, lo, hi;      // geometric extent
  int nrun, nb;
  Run run[RUN_MAX];
};

__device__ void seg_context(const LevelDev& d, int sid, SegCtx& S) {
  const Geo g = d.g;
  int I1, J1, I2, J2;
  S.sid = sid;
  S.e = d.cnt[sid];
  if (sid < g.nh()) {
    int I = sid % g.bx, J = sid / g.bx + 1;
    I1 = I; J1 = J - 1; I2 = I; J2 = J;
    S.s1 = g.side_pos(SIDE_TOP);
    S.s2 = g.side_pos(SIDE_BOTTOM);
    S.horiz = 1;
    S.line = J * (g.h + 1) - 1;
    S.lo = I * (g.w + 1);
    S.hi = S.lo + g.w - 1;
  } else {
    int t = sid - g.nh();
    int I = t % (g.bx - 1) + 1, J = t / (g.bx - 1);
    I1 = I - 1; J1 = J; I2 = I; J2 = J;
    S.s1 = g.side_pos(SIDE_RIGHT);
    S.s2 = g.side_pos(SIDE_LEFT);
    S.horiz = 0;
    S.line = I * (g.w + 1) - 1;
    S.lo = J * (g.h + 1);
    S.hi = S.lo + g.h - 1;
  }
  S.b1 = I1 + g.bx * J1;
  S.b2 = I2 + g.bx * J2;
  const int skip1 = S.horiz ? SIDE_TOP : SIDE_RIGHT;
  const int skip2 = S.horiz ? SIDE_BOTTOM : SIDE_LEFT;
  int n = 0, nb = 0;
  for (int side = 0; side < 4; ++side) {
    if (side == skip1) continue;
    int sg = g.box_side(I1, J1, side);
    if (sg >= 0) { S.run[n] = {g.side_pos(side), -1, d.cnt[sg], sg}; nb += S.run[n].len; ++n; }
  }
  for (int side = 0; side < 4; ++side) {
    if (side == skip2) continue;
    int sg = g.box_side(I2, J2, side);
    if (sg >= 0) { S.run[n] = {-1, g.side_pos(side), d.cnt[sg], sg}; nb += S.run[n].len; ++n; }
  }
  // shared corners: horizontal (b1 below b2): b1.TL = b2.BL, b1.TR = b2.BR;
  //                 vertical (b1 left of b2):  b1.BR = b2.BL, b1.TR = b2.TL
  for (int c = 0; c < 4; ++c) {
    int cid = g.box_corner(I1, J1, c);
    if (cid < 0) continue;
    int c2 = -1;
    if (S.horiz) { if (c == C_TL) c2 = C_BL; else if (c == C_TR) c2 = C_BR; }
    else { if (c == C_BR) c2 = C_BL; else if (c == C_TR) c2 = C_TL; }
    S.run[n] = {g.corner_pos(c), c2 >= 0 ? g.corner_pos(c2) : -1, 1, -2 - g.junction_node(cid, d.nx)};
    ++nb; ++n;
  }
  for (int c = 0; c < 4; ++c) {
    int cid = g.box_corner(I2, J2, c);
    if (cid < 0) continue;
    bool shared = S.horiz ? (c == C_BL || c == C_BR) : (c == C_BL || c == C_TL);
    if (shared) continue;
    S.run[n] = {-1, g.corner_pos(c), 1, -2 - g.junction_node(cid, d.nx)};
    ++nb; ++n;
  }
  S.nrun = n;
  S.nb = nb;
}

__device__ __forceinline__ void locate(const SegCtx& S, int f, int& r, int& i) {
  r = 0;
  while (f >= S.run[r].len) { f -= S.run[r].len; ++r; }
  i = f;
}

__device__ __forceinline__ int run_node(const LevelDev& d, const Run& R, int i) {
  return R.ref >= 0 ? d.nodes[(size_t)R.ref * d.capS + i] : (-2 - R.ref);
}

__device__ __forceinline__ int cheb(const SegCtx& S, int node, int nx) {
  int x = node % nx, y = node / nx;
  int a = S.horiz ? y : x, b = S.horiz ? x : y;
  int da = abs(a - S.line);
  int db = max(0, max(S.lo - b, b - S.hi));
  return max(da, db);
}

// B entry for neighbour (run R, element i), half t (0: A[v, s_c], 1: A[s_c, v]), column c
template <typename T>
__device__ __forceinline__ T bval(const LevelDev& d, const SegCtx& S, const T* F1, const T* F2,
                                  const Run& R, int i, int t, int c) {
  const size_t ld = d.ldF;
  T v = T(0);
  if (R.p1 >= 0) {
    int p = R.p1 + i;
    v += t == 0 ? F1[p + ld * (S.s1 + c)] : F1[(S.s1 + c) + ld * p];
  }
  if (R.p2 >= 0) {
    int p = R.p2 + i;
    v += t == 0 ? F2[p + ld * (S.s2 + c)] : F2[(S.s2 + c) + ld * p];
  }
  return v;
}

// Neighbour table of a segment (shared memory, built once per segment when it has at most
// NB_MAX neighbours): grid node, positions in the frontal blocks of box 1 / box 2 (-1 when
// absent) and the near flag of neighbour f.  Without the table the same values come from the
// runs.
constexpr int NB_MAX = 512;
struct NbrTab {
  const int* node;
  const short* p1;
  const short* p2;
  const unsigned char* nearf;
  bool on;
};
struct Nbr {
  int node, p1, p2;
  bool nearf;
};

__device__ __forceinline__ Nbr nbr_get(const LevelDev& d, const SegCtx& S, const NbrTab& tb, int f) {
  Nbr q;
  if (tb.on) {
    q.node = tb.node[f];
    q.p1 = tb.p1[f];
    q.p2 = tb.p2[f];
    q.nearf = tb.nearf[f] != 0;
  } else {
    int r, i;
    locate(S, f, r, i);
    const Run& R = S.run[r];
    q.node = run_node(d, R, i);
    q.p1 = R.p1 >= 0 ? R.p1 + i : -1;
    q.p2 = R.p2 >= 0 ? R.p2 + i : -1;
    q.nearf = cheb(S, q.node, d.nx) <= d.near_radius;
  }
  return q;
}

// B entry of neighbour q, half t, column c (as bval)
template <typename T>
__device__ __forceinline__ T bval_q(const LevelDev& d, const SegCtx& S, const T* F1, const T* F2, const Nbr& q,
                                    int t, int c) {
  const size_t ld = d.ldF;
  T v = T(0);
  if (q.p1 >= 0) v += t == 0 ? F1[q.p1 + ld * (S.s1 + c)] : F1[(S.s1 + c) + ld * q.p1];
  if (q.p2 >= 0) v += t == 0 ? F2[q.p2 + ld * (S.s2 + c)] : F2[(S.s2 + c) + ld * q.p2];
  return v;
}

// non-negative doubles order like their bit patterns
__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }
// ... one that is not a number above them all once its sign is gone: squared norms are kept without
// it, such a column becomes the pivot, and what is not a number reaches R, T and the solution instead
// of passing for a zero column
__device__ __forceinline__ double unsign(double x) { return __longlong_as_double(dbits(x) & 0x7fffffffffffffffll); }
// the smallest pattern that ties with the largest squared norm mx (a pattern)
__device__ __forceinline__ long long tie_bits(long long mx) {
  const double tie = (1.0 - TIE_RTOL) * (1.0 - TIE_RTOL);   // on squared norms
  return mx > 0x7ff0000000000000ll ? mx : dbits(__longlong_as_double(mx) * tie);
}

// ------------------------------------------------------------ column-pivoted QR
// Businger-Golub Householder QR with column pivoting of Y (m x e, ld ldy, precision T),
// stopped at the first step i with |R_ii| <= eps |R_00|.  Squared column norms are tracked
// and downdated in FP64 — s <- s - R_ij^2, recomputed when s <= sqrt(eps_64) s_ref (the
// Drmac-Bujanovic guard written for squared norms: no division or square root per column and
// step) — and the pivot is chosen from them; the Householder products and their column sums
// run in T.  perm receives the column order; on exit the first k rows of Y hold [R_1 R_2] in
// the permuted order.  Returns k.  The factorization also stops after kstop steps (returning
// kstop): a caller that only needs to know whether k exceeds kstop - 1 skips the rest.
// sh: >= NWT*32 + 3*64 doubles of shared scratch; flags: >= e.  NWT = warps of the CTA.
template <typename T, int NWT>
__device__ int block_cpqr(T* Y, int ldy, int m, int e, double eps, int* perm, double* vn1,
                          double* vn2, double* sh, int* flags, int* shi, int kstop) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T* part = reinterpret_cast<T*>(sh);                   // [NWT][32] partial dots
  T* coef = reinterpret_cast<T*>(sh + NWT * 32);         // [64]
  double* scal = sh + NWT * 32 + 64;                     // alpha, v0, c2, normx
  for (int j = threadIdx.x; j < e; j += blockDim.x) perm[j] = j;
  if (m == 0 || e == 0) { __syncthreads(); return 0; }
  // initial column norms (one warp per column)
  for (int j = warp; j < e; j += NWT) {
    T s = T(0);
    for (int r = lane; r < m; r += 32) { T v = Y[r + (size_t)ldy * j]; s += v * v; }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      vn1[j] = unsign((double)s);
      vn2[j] = (double)s;
    }
  }
  __syncthreads();
  const double tol3z = sqrt(DBL_EPSILON);
  const int kmax = min(min(m, e), kstop);
  double ref = 0.0;
  int k = kmax;
  for (int i = 0; i < kmax; ++i) {
    // the per-step scalar tasks rotate over the warps (and CTAs), so that the FP64 work of
    // co-resident CTAs does not pile up on one SM sub-partition
    const int wp = (i + blockIdx.x) % NWT, wh = (i + 1 + blockIdx.x) % NWT;
    const int wr = (i + 2 + blockIdx.x) % NWT, wd = (i + 3 + blockIdx.x) % NWT;
    if (warp == wp) {         // pivot: largest norm, near-ties -> lowest index
      long long mx = -1;
      for (int j = i + lane; j < e; j += 32) mx = max(mx, dbits(vn1[j]));
      for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const long long thr = tie_bits(mx);
      int best = e;
      for (int j = i + lane; j < e; j += 32)
        if (dbits(vn1[j]) >= thr && j < best) best = j;
      for (int o = 16; o > 0; o >>= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, o));
      if (lane == 0) shi[0] = best < e ? best : i;
    }
    __syncthreads();
    const int p = shi[0];
    if (p != i) {
      for (int r = threadIdx.x; r < m; r += blockDim.x) {
        T a = Y[r + (size_t)ldy * i];
        Y[r + (size_t)ldy * i] = Y[r + (size_t)ldy * p];
        Y[r + (size_t)ldy * p] = a;
      }
      if (threadIdx.x == 0) {
        int t = perm[i]; perm[i] = perm[p]; perm[p] = t;
        double a = vn1[i]; vn1[i] = vn1[p]; vn1[p] = a;
        a = vn2[i]; vn2[i] = vn2[p]; vn2[p] = a;
      }
      __syncthreads();
    }
    // Householder vector of column i (scalars by one thread)
    if (warp == wh) {
      T s = T(0);
      for (int r = i + lane; r < m; r += 32) { T v = Y[r + (size_t)ldy * i]; s += v * v; }
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) {
        const T normx = sqrt(s);
        const T x0 = Y[i + (size_t)ldy * i];
        const T alpha = x0 >= T(0) ? -normx : normx;
        const T v0 = x0 - alpha;
        const T vv = v0 * v0 + (s - x0 * x0);
        scal[0] = (double)alpha;
        scal[1] = (double)v0;
        scal[2] = vv > T(0) ? (double)(T(2) / vv) : 0.0;
        scal[3] = (double)normx;
      }
    }
    __syncthreads();
    const double normx = scal[3];
    if (i == 0) ref = normx;
    if (ref == 0.0) { k = 0; break; }
    if (normx <= eps * ref || normx == 0.0) { k = i; break; }
    const T v0 = (T)scal[1];
    const T c2 = (T)scal[2];
    const int ncol = e - i - 1;
    // dots of v with the trailing columns (lanes over columns, warps over rows), then update
    for (int cg = 0; cg < ncol; cg += 32) {
      const int j = i + 1 + cg + lane;
      T acc = T(0);
      if (j < e) {
        const T* yj = Y + (size_t)ldy * j;
        const T* yi = Y + (size_t)ldy * i;
        if (warp == 0) acc = v0 * yj[i];
        for (int r = i + 1 + warp; r < m; r += NWT) acc += yi[r] * yj[r];
      }
      part[warp * 32 + lane] = acc;
      __syncthreads();
      if (warp == wr && j < e) {
        T s = T(0);
        for (int w = 0; w < NWT; ++w) s += part[w * 32 + lane];
        coef[lane] = s * c2;
      }
      __syncthreads();
      if (j < e) {
        const T cj = coef[lane];
        T* yj = Y + (size_t)ldy * j;
        const T* yi = Y + (size_t)ldy * i;
        if (warp == 0) yj[i] -= cj * v0;
        for (int r = i + 1 + warp; r < m; r += NWT) yj[r] -= cj * yi[r];
      }
      __syncthreads();
    }
    // FP64 downdates of the squared norms, one lane per column; guarded recomputations after
    if (warp == wd) {
      for (int j = i + 1 + lane; j < e; j += 32) {
        const double sq = vn1[j];
        int fl = 0;
        if (sq != 0.0) {
          const double rij = (double)Y[i + (size_t)ldy * j];
          const double sn = fmax(sq - rij * rij, 0.0);
          if (sn <= tol3z * vn2[j]) fl = 1;
          else vn1[j] = sn;
        }
        flags[j] = fl;
      }
    }
    __syncthreads();
    for (int j = i + 1 + warp; j < e; j += NWT) {
      if (!flags[j]) continue;
      double s = 0.0;
      for (int r = i + 1 + lane; r < m; r += 32) { double v = (double)Y[r + (size_t)ldy * j]; s += v * v; }
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) {
        vn1[j] = unsign(s);
        vn2[j] = s;
      }
    }
    if (threadIdx.x == 0) Y[i + (size_t)ldy * i] = (T)scal[0];
    __syncthreads();
  }
  __syncthreads();
  return k;
}

// T (k x (e-k), ld ldt) = R_1^{-1} R_2 from the R held in Y (ld ldy); rinv: >= k scratch
template <typename T>
__device__ void block_interp(const T* Y, int ldy, int k, int e, T* Tm, int ldt, T* rinv) {
  for (int a = threadIdx.x; a < k; a += blockDim.x) rinv[a] = T(1) / Y[a + (size_t)ldy * a];
  __syncthreads();
  for (int j = threadIdx.x; j < e - k; j += blockDim.x) {
    for (int a = k - 1; a >= 0; --a) {
      T s = Y[a + (size_t)ldy * (k + j)];
      for (int b = a + 1; b < k; ++b) s -= Y[a + (size_t)ldy * b] * Tm[b + (size_t)ldt * j];
      Tm[a + (size_t)ldt * j] = s * rinv[a];
    }
  }
  __syncthreads();
}

// LU with partial pivoting of the n x n block of A at (r0, r0) (ld lda), with the row
// operations carried over columns [0, ncol) outside the factored block; multipliers are
// stored below the diagonal and (unless `all`) not interchanged afterwards (the solve interleaves
// interchanges and eliminations).  inv receives the reciprocal pivots.  Returns false on an
// exactly zero pivot.
template <typename T>
__device__ bool block_gepp(T* A, int lda, int r0, int n, int ncol, int* piv, T* inv, int* shi, bool all) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  bool ok = true;
  for (int j = 0; j < n; ++j) {
    const int cj = r0 + j;
    if (warp == 0) {
      double best = -1.0;
      int bi = n;
      for (int r = j + lane; r < n; r += 32) {
        double v = fabs((double)A[(r0 + r) + (size_t)lda * cj]);
        if (v > best || (v == best && r < bi)) { best = v; bi = r; }
      }
      for (int o = 16; o > 0; o >>= 1) {
        double ob = __shfl_xor_sync(0xffffffffu, best, o);
        int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
      }
      if (bi >= n) bi = j;     // only where no entry of the column is a number
      if (lane == 0) { shi[0] = bi; shi[1] = best == 0.0; piv[j] = bi; }
    }
    __syncthreads();
    const int p = shi[0];
    if (shi[1]) { ok = false; if (threadIdx.x == 0) inv[j] = T(0); __syncthreads(); continue; }
    if (p != j) {
      for (int c = threadIdx.x; c < ncol; c += blockDim.x) {
        if (!all && c >= r0 && c < cj) continue;
        T a = A[(r0 + j) + (size_t)lda * c];
        A[(r0 + j) + (size_t)lda * c] = A[(r0 + p) + (size_t)lda * c];
        A[(r0 + p) + (size_t)lda * c] = a;
      }
      __syncthreads();
    }
    const T ipv = T(1) / A[(r0 + j) + (size_t)lda * cj];
    if (threadIdx.x == 0) inv[j] = ipv;
    for (int r = j + 1 + threadIdx.x; r < n; r += blockDim.x) A[(r0 + r) + (size_t)lda * cj] *= ipv;
    __syncthreads();
    const int nr = n - j - 1;
    const int nc = ncol - 1;   // every column but cj
    for (int e = threadIdx.x; e < nr * nc; e += blockDim.x) {
      int r = j + 1 + e % nr;
      int c = e / nr;
      if (c >= cj) ++c;
      if (c >= r0 && c < cj) continue;   // multipliers of earlier steps
      A[(r0 + r) + (size_t)lda * c] -= A[(r0 + r) + (size_t)lda * cj] * A[(r0 + j) + (size_t)lda * c];
    }
    __syncthreads();
  }
  return ok;
}


// ------------------------------------------------------------ block reductions (FP64)
__device__ __forceinline__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double s = 0.0;
  for (int w = 0; w < nw; ++w) s += red[w];
  __syncthreads();
  return s;
}

// ------------------------------------------------------------ tensor-core helpers (TF32)
// mma.sync m16n8k8 with TF32 operands and FP32 accumulation.  TF32 keeps 10 mantissa bits, so
// each operand is split into a high part tf32(x) and a low part tf32(x - hi) and three products
// are accumulated (the two cross terms first, then hi*hi): the result matches an FP32 product
// to about FP32 rounding (the lo*lo term, below 2^-22 relative, is dropped).
// Fragment layouts of m16n8k8 (PTX ISA, tf32): g = lane / 4, q = lane % 4;
//   A (16 x 8, row major): a0 (g, q), a1 (g + 8, q), a2 (g, q + 4), a3 (g + 8, q + 4);
//   B (8 x 8, column major): b0 (q, g), b1 (q + 4, g);
//   C (16 x 8): c0 (g, 2q), c1 (g, 2q + 1), c2 (g + 8, 2q), c3 (g + 8, 2q + 1).
__device__ __forceinline__ uint32_t to_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;\n" : "=r"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ void split_tf32(float x, uint32_t& hi, uint32_t& lo) {
  hi = to_tf32(x);
  lo = to_tf32(x - __uint_as_float(hi));
}
__device__ __forceinline__ void mma_tf32(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}


// ------------------------------------------------------------ far-row sketch
// Yr[rr, c] = sum over far neighbour rows f of G[rr, f] B_F[f, c] for r0 <= rr < hh (unscaled),
// neighbours taken in chunks of ch (near ones get zero weight).  Yr has leading dimension ldy.
// Rows below r0 are left alone (the one-pass sketch takes them from the probe, whose rows are
// the same rows of G).
template <typename T, class BGet>
__device__ void sketch_far(const LevelDev& d, const SegCtx& S, const NbrTab& tb, BGet bget,
                           int sid, int halves, int e, int r0, int hh, T* Yr, int ldy, T* Bc, T* Gc,
                           int ch) {
  const int nr = hh - r0;
  for (int x = threadIdx.x; x < nr * e; x += blockDim.x) Yr[(r0 + x % nr) + (size_t)ldy * (x / nr)] = T(0);
  __syncthreads();
  for (int f0 = 0; f0 < S.nb; f0 += ch) {
    const int nc = min(ch, S.nb - f0);
    const int rows = halves * nc;
    for (int x = threadIdx.x; x < rows * e; x += blockDim.x) {
      int row = x % rows, c = x / rows;
      int t = row / nc, jj = row % nc;
      Bc[row + (size_t)rows * c] = bget(t, f0 + jj, c);
    }
    // one Philox counter per group of four sketch rows (r0 is a multiple of 4)
    const int g0 = r0 >> 2, ng = ((hh + 3) >> 2) - g0;
    for (int x = threadIdx.x; x < ng * rows; x += blockDim.x) {
      const int gi = x % ng, row = x / ng;
      const int t = row / nc, jj = row % nc;
      const Nbr q = nbr_get(d, S, tb, f0 + jj);
      float z[4] = {0.f, 0.f, 0.f, 0.f};
      if (!q.nearf) sketch_gauss4(d.seed, d.l, sid, g0 + gi, q.node, t, z);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int rr = 4 * (g0 + gi) + i - r0;
        if (rr < nr) Gc[rr + (size_t)nr * row] = (T)z[i];
      }
    }
    __syncthreads();
    if constexpr (sizeof(T) == 4) {
      if (d.sketch_tc) {
        // Y_chunk (nr x e) += G_chunk (nr x rows) B_chunk (rows x e) on the tensor cores: the
        // warps take 16 x 8 output tiles in turn, k in steps of 8 rows (zero past the end)
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
        const int g = lane >> 2, q = lane & 3;
        const int mt = (nr + 15) >> 4, nt = (e + 7) >> 3;
        auto Ga = [&](int r, int k) { return (r < nr && k < rows) ? (float)Gc[r + (size_t)nr * k] : 0.f; };
        auto Bb = [&](int k, int c) { return (k < rows && c < e) ? (float)Bc[k + (size_t)rows * c] : 0.f; };
        for (int t = warp; t < mt * nt; t += nw) {
          const int m0 = 16 * (t % mt), n0 = 8 * (t / mt);
          float acc[4] = {0.f, 0.f, 0.f, 0.f};
          for (int k0 = 0; k0 < rows; k0 += 8) {
            uint32_t ah[4], al[4], bh[2], bl[2];
            split_tf32(Ga(m0 + g, k0 + q), ah[0], al[0]);
            split_tf32(Ga(m0 + g + 8, k0 + q), ah[1], al[1]);
            split_tf32(Ga(m0 + g, k0 + q + 4), ah[2], al[2]);
            split_tf32(Ga(m0 + g + 8, k0 + q + 4), ah[3], al[3]);
            split_tf32(Bb(k0 + q, n0 + g), bh[0], bl[0]);
            split_tf32(Bb(k0 + q + 4, n0 + g), bh[1], bl[1]);
            mma_tf32(acc, al, bh);
            mma_tf32(acc, ah, bl);
            mma_tf32(acc, ah, bh);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int rr = m0 + g + 8 * (u >> 1), c = n0 + 2 * q + (u & 1);
            if (rr < nr && c < e) Yr[(r0 + rr) + (size_t)ldy * c] += (T)acc[u];
          }
        }
        __syncthreads();
        continue;
      }
    }
    // sums over blocks of SK_CHUNK far unknowns (both halves of a block, then the next block):
    // the same order of operations for every chunk size, so that the sketch does not depend on
    // the shared-memory budget the level runs with
    for (int x = threadIdx.x; x < nr * e; x += blockDim.x) {
      const int rr = x % nr, c = x / nr;
      const T* g = Gc + rr;
      const T* bc = Bc + (size_t)rows * c;
      T y = Yr[(r0 + rr) + (size_t)ldy * c];
      for (int b0 = 0; b0 < nc; b0 += SK_CHUNK) {
        const int b1 = min(nc, b0 + SK_CHUNK);
        T acc = T(0);
#pragma unroll 4
        for (int row = b0; row < b1; ++row) acc += g[(size_t)nr * row] * bc[row];
        if (halves == 2) {
#pragma unroll 4
          for (int row = nc + b0; row < nc + b1; ++row) acc += g[(size_t)nr * row] * bc[row];
        }
        y += acc;
      }
      Yr[(r0 + rr) + (size_t)ldy * c] = y;
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------ learned rank predictor
// (no counterpart in the paper; the definitions are those of the oracle's predictor module)
// Probe sketch Y8[r + PRED_PROBE c] = sum over the far rows of G[r, row] B[row, c], r < 8: the
// first PRED_PROBE rows of the sketch matrix of this segment, unscaled.  Warps take rows in
// turn; lanes hold columns lane + 32 q of a 64-column chunk in registers; the warps' sums meet
// in Y8 (zeroed by the caller) through shared-memory atomics.
template <typename T, class BGet>
__device__ void probe_sketch(const LevelDev& d, const SegCtx& S, const NbrTab& tb, BGet bget,
                             int sid, int halves, int e, T* Y8) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int nrows = halves * S.nb;
  const int ro = lane >> 3, r8 = lane & 7;                 // lane: row ro of a group of 4, probe row r8
  for (int c0 = 0; c0 < e; c0 += 64) {
    T acc[2][PRED_PROBE];
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int r = 0; r < PRED_PROBE; ++r) acc[q][r] = T(0);
    for (int g0 = 4 * warp; g0 < nrows; g0 += 4 * nw) {
      const int row = g0 + ro;
      Nbr q{0, -1, -1, true};
      int t = 0;
      if (row < nrows) {
        t = row / S.nb;
        q = nbr_get(d, S, tb, row % S.nb);
      }
      // lanes r8 = 0 and 4 of each node row draw the two counters (rows 0-3, 4-7); the
      // others take their component by shuffle
      float z[4] = {0.f, 0.f, 0.f, 0.f};
      if (!q.nearf && (r8 & 3) == 0) sketch_gauss4(d.seed, d.l, sid, r8 >> 2, q.node, t, z);
      const int srcl = lane & ~3;
      float zc = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float v = __shfl_sync(0xffffffffu, z[i], srcl);
        if ((r8 & 3) == i) zc = v;
      }
      const T g = q.nearf ? T(0) : (T)zc;
#pragma unroll
      for (int rr = 0; rr < 4; ++rr) {
        const int src = 8 * rr;
        if (__shfl_sync(0xffffffffu, (int)q.nearf, src)) continue;   // near or past the end
        const int rowr = g0 + rr, tr = rowr / S.nb, fr = rowr % S.nb;
        T b[2];
#pragma unroll
        for (int qc = 0; qc < 2; ++qc) {
          const int c = c0 + 32 * qc + lane;
          b[qc] = c < e ? bget(tr, fr, c) : T(0);
        }
#pragma unroll
        for (int r = 0; r < PRED_PROBE; ++r) {
          const T gr = __shfl_sync(0xffffffffu, g, src + r);
#pragma unroll
          for (int qc = 0; qc < 2; ++qc) acc[qc][r] += gr * b[qc];
        }
      }
    }
    // the warps add their partial sums in warp order (a fixed summation order: the probe, and
    // through it the predicted sketch size, is the same in every factorization)
    for (int w = 0; w < nw; ++w) {
      if (warp == w) {
#pragma unroll
        for (int qc = 0; qc < 2; ++qc) {
          const int c = c0 + 32 * qc + lane;
          if (c < e)
#pragma unroll
            for (int r = 0; r < PRED_PROBE; ++r) Y8[r + PRED_PROBE * c] += acc[qc][r];
        }
      }
      __syncthreads();
    }
  }
}

// Features of segment sid into xf[16] (shared), needs >= 2 warps; every thread calls it.
// Arithmetic in the factor's precision T (features are inputs of a BF16 network).
// Warp 0: column-pivoted QR of the probe Y8 (PRED_PROBE x e, pitch PRED_PROBE, overwritten)
// by Gram-Schmidt with exactly recomputed column norms, lane c owning columns c + 32 q; the
// pivot is the largest norm, near-ties (relative 1e-12) to the lowest column.  Warp 1: the
// coefficient statistics of the segment's nodes from the per-node table.
template <typename T>
__device__ void probe_features(const LevelDev& d, int sid, int e, int nnear, int nfar, int nb,
                               T* Y8, float* xf) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp == 0) {
    const int nd = min(PRED_PROBE, e);
    T rd[PRED_PROBE];
#pragma unroll
    for (int i = 0; i < PRED_PROBE; ++i) rd[i] = T(0);
    unsigned used = 0;                                       // bit q: column lane + 32 q pivoted
    T sq[4];
    for (int i = 0; i < nd; ++i) {
      T mx = T(0);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int c = lane + 32 * q;
        sq[q] = T(-1);
        if (c < e && !(used >> q & 1)) {
          T a = T(0);
#pragma unroll
          for (int r = 0; r < PRED_PROBE; ++r) a += Y8[r + PRED_PROBE * c] * Y8[r + PRED_PROBE * c];
          sq[q] = a;
          mx = a > mx ? a : mx;
        }
      }
      for (int o = 16; o > 0; o >>= 1) { const T w = __shfl_xor_sync(0xffffffffu, mx, o); mx = w > mx ? w : mx; }
      if (!(mx > T(0))) break;
      const T thr = mx * (T)((1.0 - TIE_RTOL) * (1.0 - TIE_RTOL));
      int best = 1 << 30;
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (sq[q] >= thr) best = min(best, lane + 32 * q);
      for (int o = 16; o > 0; o >>= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, o));
      T v[PRED_PROBE];
      T pn = T(0);
#pragma unroll
      for (int r = 0; r < PRED_PROBE; ++r) {
        v[r] = Y8[r + PRED_PROBE * best];
        pn += v[r] * v[r];
      }
      pn = sqrt(pn);
      rd[i] = pn;
      const T inv = T(1) / pn;
#pragma unroll
      for (int r = 0; r < PRED_PROBE; ++r) v[r] *= inv;
      if ((best & 31) == lane) used |= 1u << (best >> 5);
      __syncwarp();
      for (int q = 0, c = lane; c < e; ++q, c += 32) {
        if (used >> q & 1) continue;
        T* col = Y8 + PRED_PROBE * c;
        T dot = T(0);
#pragma unroll
        for (int r = 0; r < PRED_PROBE; ++r) dot += v[r] * col[r];
#pragma unroll
        for (int r = 0; r < PRED_PROBE; ++r) col[r] -= dot * v[r];
      }
      __syncwarp();
    }
    if (lane < 5) {                                          // one decay ratio per lane
      const int js[5] = {1, 2, 3, 5, 7};
      const int j = js[lane];
      const T le = (T)d.log10eps;
      T val;
      if (j >= nd || rd[0] == T(0)) val = T(-16) - le;
      else {
        T rj = rd[0];
#pragma unroll
        for (int q = 1; q < PRED_PROBE; ++q) if (q == j) rj = rd[q];
        const T ratio = rj / rd[0];
        val = log10(ratio > T(1e-16) ? ratio : T(1e-16)) - le;
      }
      xf[11 + lane] = (float)val;
    }
  } else if (warp == 1) {
    const int* nodes = d.nodes + (size_t)sid * d.capS;
    float lmin = 3.0e38f, lmax = -3.0e38f, lsum = 0.f, dsum = 0.f, ssum = 0.f, asum = 0.f;
    for (int t = lane; t < e; t += 32) {
      const float4 st = d.nstat[nodes[t]];
      lmin = fminf(lmin, st.x);
      lmax = fmaxf(lmax, st.x);
      lsum += st.x;
      dsum += st.y;
      ssum += st.z;
      asum += st.w;
    }
    for (int o = 16; o > 0; o >>= 1) {
      lmin = fminf(lmin, __shfl_xor_sync(0xffffffffu, lmin, o));
      lmax = fmaxf(lmax, __shfl_xor_sync(0xffffffffu, lmax, o));
      lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
      dsum += __shfl_xor_sync(0xffffffffu, dsum, o);
      ssum += __shfl_xor_sync(0xffffffffu, ssum, o);
      asum += __shfl_xor_sync(0xffffffffu, asum, o);
    }
    const float mean = lsum / e;
    float vsum = 0.f;
    for (int t = lane; t < e; t += 32) {
      const float dv = d.nstat[nodes[t]].x - mean;
      vsum += dv * dv;
    }
    for (int o = 16; o > 0; o >>= 1) vsum += __shfl_xor_sync(0xffffffffu, vsum, o);
    if (lane == 0) {
      xf[0] = (float)(d.L - d.l);
      xf[1] = log2f((float)e);
      xf[2] = log2f(1.0f + nb);
      xf[3] = (float)nnear;
      xf[4] = log2f(1.0f + nfar);
      xf[5] = lmin - mean;
      xf[6] = lmax - mean;
      xf[7] = sqrtf(vsum / e);
      xf[8] = dsum / e;
      xf[9] = ssum / e;
      xf[10] = asum / e;
    }
  }
  __syncthreads();
}

// Measured ID error test ||B_r - B_s T||_F <= 10 eps ||B||_F on the exact B (all neighbour
// rows, both halves of a non-symmetric B): one thread per row of B, entries read directly.
template <typename T, class BGet>
__device__ bool id_error_ok(const SegCtx& S, BGet bget, int halves, int e, int k, const int* perm,
                            const T* Tw, int ldt, double eps, double* red) {
  const int r = e - k;
  T num = T(0), den = T(0);                 // per-thread sums in T, the block sum in FP64
  for (int row = threadIdx.x; row < halves * S.nb; row += blockDim.x) {
    const int f = row % S.nb, t = row / S.nb;
    for (int c = 0; c < e; ++c) {
      const T v = bget(t, f, c);
      den += v * v;
    }
    for (int j = 0; j < r; ++j) {
      T s = bget(t, f, perm[k + j]);
      for (int a = 0; a < k; ++a) s -= bget(t, f, perm[a]) * Tw[a + (size_t)ldt * j];
      num += s * s;
    }
  }
  const double nsum = block_sum((double)num, red);
  const double dsum = block_sum((double)den, red);
  return sqrt(nsum) <= 10.0 * eps * sqrt(dsum);
}

// ------------------------------------------------------------ sparsify: one CTA per segment
// Barrier of the first QW warps of a CTA of NWT (all of them: the CTA's barrier).
template <int QW, int NWT>
__device__ __forceinline__ void qr_bar() {
  if constexpr (QW == NWT) __syncthreads();
  else asm volatile("bar.sync 1, %0;" ::"n"(QW * 32) : "memory");
}

__device__ __forceinline__ unsigned bits_hi(double x) { return (unsigned)((unsigned long long)dbits(x) >> 32); }
__device__ __forceinline__ unsigned bits_lo(double x) { return (unsigned)(unsigned long long)dbits(x); }
__device__ __forceinline__ unsigned abs_hi(double x) { return bits_hi(x) & 0x7fffffffu; }
__device__ __forceinline__ unsigned abs_hi(float x) { return __float_as_uint(x) & 0x7fffffffu; }
__device__ __forceinline__ unsigned abs_lo(double x) { return bits_lo(x); }
__device__ __forceinline__ unsigned abs_lo(float) { return 0u; }

// normx = sqrt(s) of a sum of squares: in FP64 from the reciprocal square root (a division or square
// root costs 6 to 10 dependent FP64 instructions of 67 cycles each).  Only a sum of exactly 0 gives
// 0, the mark of a column without entries; one that is not finite gives NaN.
__device__ __forceinline__ float qr_norm(float s) { return sqrtf(s); }
__device__ __forceinline__ double qr_norm(double s) { return dbits(s) == 0 ? 0.0 : s * rsqrt(s); }

// The pivot of a step, chosen by one warp: among its columns at positions >= i, the largest
// squared norm, near-ties (TIE_RTOL) to the lowest position.  Norms are compared as bit patterns
// (an FP64 comparison is an instruction of the FP64 pipe).  Returns the position; *col the column.
template <int CS>
__device__ __forceinline__ int qr_pivot(const double (&n1)[CS], const int (&pos)[CS], int i, int e, int* col) {
  unsigned hi = 0, lo = 0, best = 0xffffffffu;
#pragma unroll
  for (int t = 0; t < CS; ++t)
    if (pos[t] >= i && pos[t] < e) hi = max(hi, bits_hi(n1[t]));
  hi = __reduce_max_sync(0xffffffffu, hi);
#pragma unroll
  for (int t = 0; t < CS; ++t)
    if (pos[t] >= i && pos[t] < e && bits_hi(n1[t]) == hi) lo = max(lo, bits_lo(n1[t]));
  lo = __reduce_max_sync(0xffffffffu, lo);
  const long long thr = tie_bits(((long long)hi << 32) | lo);
#pragma unroll
  for (int t = 0; t < CS; ++t)
    if (pos[t] >= i && pos[t] < e && dbits(n1[t]) >= thr) best = min(best, (unsigned)pos[t]);
  best = __reduce_min_sync(0xffffffffu, best);
  if (best >= (unsigned)e) best = (unsigned)i;
  *col = 0;
#pragma unroll
  for (int t = 0; t < CS; ++t) {
    const unsigned b = __ballot_sync(0xffffffffu, pos[t] == (int)best);
    if (b) *col = 32 * t + __ffs(b) - 1;
  }
  return (int)best;
}

// Column-pivoted Householder QR for e <= 32 CS, on Y in place by the first QW warps (all threads
// call it): pivot rule, truncation and kstop as in block_cpqr; norm downdates in FP64 with the
// same guard, but where one column falls below it all norms are recomputed (they decay together, so
// this happens two or three times per factorization instead of once or more per column).  Lanes
// own columns (lane l: slots l, l + 32), warps own rows (r mod QW).  Columns are not interchanged:
// a column's position in the pivot order is a register.  perm receives the columns by position,
// slot their places: R(a, b) is Y[a + ldy slot[b]] on return (rows < k).  Once at most 32 columns
// are left, those in slots 32 .. move to slots whose columns are done, and one set of lanes goes on.
// What bounds it: the latency of a step, k steps in a row, and in FP64 the instructions of the
// FP64 pipe (64 cycles each).  So a step has two barriers and one reduction: every warp applies the
// previous reflection to its rows and, in the same pass, forms its partial products of the next
// pivot column x with all columns (x itself among them); one warp sums them, d_j = x^T y_j, and
// has the whole step from them: ||x||^2 = d_x, v^T y_j = d_j - alpha y_ij with v = x - alpha e_i, the
// new row i of R, the norm downdates and the next pivot.  That warp differs between the CTAs of an
// SM (rw), so that their FP64 chains do not meet on one sub-partition.
// Measured per segment (1023^2, clock64, all passes) against the form with three phases, three
// barriers and a norm recomputed per column: mixed 63 -> 30 us at level 11 (e ~ 21, four CTAs per
// SM), 72 -> 36 us at level 7; FP64 (also with its working set in shared memory now)
// 514 -> 101 us at level 11, 255 -> 162 us at level 6 (e ~ 37, one CTA per SM).
// shr: 64 doubles (coef), then QW * 32 CS doubles (part); shi: >= 6.
template <typename T, int NWT, int QW, int CS>
__device__ int fast_cpqr(T* Y, int ldy, int m, int e, double eps, int* perm, int* slot, double* shr, int* shi,
                         int kstop) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int EC = 32 * CS;
  if (m == 0 || e == 0) {
    for (int j = threadIdx.x; j < e; j += blockDim.x) { perm[j] = j; slot[j] = j; }
    __syncthreads();
    return 0;
  }
  T* coef = reinterpret_cast<T*>(shr);
  T* part = reinterpret_cast<T*>(shr + 64);
  double* part2 = shr + 64;                // the same place: norms, when they are recomputed
  const int kmax = min(min(m, e), kstop);
  const int rw = (int)(blockIdx.x + blockIdx.x / 152u) & (QW - 1);
  if (warp < QW) {
    int pos[CS], id[CS];                   // position and original column of the lane's slots
    T acc[CS];
    T* yc[CS];                             // the slots (clamped: every address is valid)
    double n1[CS], g2[CS];                 // warp rw: squared norm; sqrt(eps_64) times its reference
    const double tol3z = sqrt(DBL_EPSILON);
    int cs = CS;                           // sets of lanes with columns left
#pragma unroll
    for (int t = 0; t < CS; ++t) {
      const int j = lane + 32 * t;
      pos[t] = id[t] = j;
      acc[t] = T(0);
      yc[t] = Y + ldy * min(j, e - 1);
      n1[t] = g2[t] = 0.0;
      if (j < e)
        for (int r = warp; r < m; r += QW) { const T v = yc[t][r]; acc[t] += v * v; }
      part[warp * EC + j] = acc[t];
    }
    qr_bar<QW, NWT>();
    if (warp == rw) {
#pragma unroll
      for (int t = 0; t < CS; ++t) {
        T s = T(0);
        for (int w = 0; w < QW; ++w) s += part[w * EC + lane + 32 * t];
        n1[t] = lane + 32 * t < e ? unsign((double)s) : 0.0;
        g2[t] = tol3z * n1[t];
      }
      int pc;
      const int pp = qr_pivot<CS>(n1, pos, 0, e, &pc);
      if (lane == 0) { shi[0] = pc; shi[1] = pp; }
    }
    qr_bar<QW, NWT>();
    int p = shi[0], pp = shi[1];           // pivot slot of the step and its position so far
    T ref_eps = T(0);                      // warp rw: the truncation threshold eps |R_00|
    bool dots = true;                      // the products of step i with column p are still to form
    for (int i = 0;; ++i) {
#pragma unroll
      for (int t = 0; t < CS; ++t) {
        const int j = lane + 32 * t;
        if (j == p) pos[t] = i;
        else if (pos[t] == i) pos[t] = pp;
      }
      if (dots) {
        const T* yp = Y + ldy * p;
#pragma unroll
        for (int t = 0; t < CS; ++t) {
          acc[t] = T(0);
          if (t < cs && pos[t] >= i && pos[t] < e)
#pragma unroll 2
            for (int r = i + ((warp - i) & (QW - 1)); r < m; r += QW) acc[t] += yp[r] * yc[t][r];
        }
      }
#pragma unroll
      for (int t = 0; t < CS; ++t) part[warp * EC + lane + 32 * t] = acc[t];
      qr_bar<QW, NWT>();
      if (warp == rw) {
        T d[CS], yi[CS];
#pragma unroll
        for (int t = 0; t < CS; ++t) {
          const int j = lane + 32 * t;
          d[t] = yi[t] = T(0);
          if (t < cs) {
            T q[QW];
#pragma unroll
            for (int w = 0; w < QW; ++w) q[w] = part[w * EC + j];
#pragma unroll
            for (int o = QW / 2; o > 0; o >>= 1)
#pragma unroll
              for (int w = 0; w < o; ++w) q[w] += q[w + o];
            d[t] = q[0];
            yi[t] = yc[t][i];
          }
        }
        T dp = d[0], yp = yi[0];
        if constexpr (CS == 2) { if (p >> 5) { dp = d[1]; yp = yi[1]; } }
        const T s = __shfl_sync(0xffffffffu, dp, p & 31), x0 = __shfl_sync(0xffffffffu, yp, p & 31);
        const T normx = qr_norm(s);
        int stop = 0;
        if (i == 0) {
          if constexpr (sizeof(T) == 4) ref_eps = __double2float_rd(eps * (double)normx);   // exact test in T
          else ref_eps = eps * normx;
          if (normx == T(0)) stop = 2;
        }
        if (!stop && (normx <= ref_eps || normx == T(0))) stop = 1;
        bool low = false;                  // some norm fell below the guard
        int pn = 0, ppn = 0;
        if (!stop) {
          const T alpha = x0 >= T(0) ? -normx : normx;
          const T v0 = x0 - alpha;
          const T den = s + (x0 >= T(0) ? x0 : -x0) * normx;      // v^T v / 2
          const T c2 = den > T(0) ? T(1) / den : T(0);
#pragma unroll
          for (int t = 0; t < CS; ++t) {
            if (t < cs) {
              const int j = lane + 32 * t;
              const bool act = pos[t] > i && pos[t] < e;
              const T cj = act ? c2 * (d[t] - alpha * yi[t]) : T(0);
              const T rij = yi[t] - cj * v0;
              coef[j] = cj;
              if (act) {
                yc[t][i] = rij;
                if (dbits(n1[t]) != 0) {
                  const double rd = (double)rij, sn = n1[t] - rd * rd;
                  const long long sb = dbits(sn) < 0 ? 0 : dbits(sn);
                  if (sb <= dbits(g2[t])) low = true;
                  else n1[t] = __longlong_as_double(sb);
                }
              } else if (j == p) {
                yc[t][i] = alpha;                                 // R_ii
              }
            }
          }
          low = __any_sync(0xffffffffu, low);
          if (!low && i + 1 < kmax) ppn = qr_pivot<CS>(n1, pos, i + 1, e, &pn);
        }
        if (lane == 0) { shi[0] = pn; shi[1] = ppn; shi[2] = stop; shi[3] = low; }
      }
      qr_bar<QW, NWT>();
      const int stop = shi[2], low = shi[3];
      if (stop || i + 1 >= kmax) {
        if (threadIdx.x == 0) shi[5] = stop == 2 ? 0 : stop == 1 ? i : kmax;
        break;
      }
      const T* v = Y + ldy * p;            // the reflection's column (rows > i)
      const int r0 = i + 1 + ((warp - i - 1) & (QW - 1));
      T cj[CS];
      bool act[CS];
#pragma unroll
      for (int t = 0; t < CS; ++t) {
        act[t] = t < cs && pos[t] > i && pos[t] < e;
        cj[t] = coef[lane + 32 * t];
        acc[t] = T(0);
      }
      const bool shrink = CS == 2 && cs == 2 && e - i - 1 <= 32;
      if (!low && !shrink) {
        p = shi[0];
        pp = shi[1];
        const bool inset1 = p >= 32;
#pragma unroll 4
        for (int r = r0; r < m; r += QW) {
          const T vr = v[r];
          T y[CS];
#pragma unroll
          for (int t = 0; t < CS; ++t) {
            y[t] = T(0);
            if (act[t]) {
              y[t] = yc[t][r] - cj[t] * vr;
              yc[t][r] = y[t];
            }
          }
          T yq = y[0];
          if constexpr (CS == 2) { if (inset1) yq = y[1]; }
          const T xr = __shfl_sync(0xffffffffu, yq, p & 31);
#pragma unroll
          for (int t = 0; t < CS; ++t)
            if (act[t]) acc[t] += xr * y[t];
        }
        dots = false;
        continue;
      }
      // the update alone (and the norms in FP64), then what precedes the next pivot's products
      double a2[CS];
#pragma unroll
      for (int t = 0; t < CS; ++t) {
        a2[t] = 0.0;
        if (act[t])
#pragma unroll 2
          for (int r = r0; r < m; r += QW) {
            const T y = yc[t][r] - cj[t] * v[r];
            yc[t][r] = y;
            if (low) a2[t] += (double)y * (double)y;
          }
      }
      p = shi[0];
      pp = shi[1];
      if (low) {
#pragma unroll
        for (int t = 0; t < CS; ++t) part2[warp * EC + lane + 32 * t] = a2[t];
        qr_bar<QW, NWT>();
        if (warp == rw) {
#pragma unroll
          for (int t = 0; t < CS; ++t) {
            if (t < cs) {
              double q = part2[lane + 32 * t];
              for (int w = 1; w < QW; ++w) q += part2[w * EC + lane + 32 * t];
              if (act[t]) { n1[t] = unsign(q); g2[t] = tol3z * q; }
            }
          }
          int pn;
          const int ppn = qr_pivot<CS>(n1, pos, i + 1, e, &pn);
          if (lane == 0) { shi[0] = pn; shi[1] = ppn; }
        }
        qr_bar<QW, NWT>();
        p = shi[0];
        pp = shi[1];
      }
      if constexpr (CS == 2) {
        if (shrink) {
          // at most 32 columns left: the x-th of those in slots 32 .. changes places with the x-th
          // done column of slots 0 .. 31 (there are at least as many)
          const unsigned mv = __ballot_sync(0xffffffffu, act[1]);
          const unsigned fr = __ballot_sync(0xffffffffu, !act[0]);   // done (every slot < 32 exists)
          qr_bar<QW, NWT>();                                         // all rows updated
          const int src = act[1] ? __popc(mv & ((1u << lane) - 1u)) : -1;
          int to = -1, from = -1;                                    // set 1 lane -> slot, set 0 slot <- lane
          unsigned f = fr, g = mv;
          for (int x = 0; g; ++x) {
            const int a = __ffs(f) - 1, b = __ffs(g) - 1;
            f &= f - 1;
            g &= g - 1;
            if (x % QW == warp) {
              T* ya = Y + ldy * a;
              T* yb = Y + ldy * (b + 32);
              for (int r = lane; r < m; r += 32) { const T q = ya[r]; ya[r] = yb[r]; yb[r] = q; }
            }
            if (src == x) to = a;
            if (lane == a) from = b;
            if (p == b + 32) p = a;
          }
          // exchange the registers of the two sets (a lane gives its set 1 to the lane `to` and
          // takes that lane's set 0)
          const int pf = __shfl_sync(0xffffffffu, pos[1], from < 0 ? lane : from);
          const int jf = __shfl_sync(0xffffffffu, id[1], from < 0 ? lane : from);
          const double nf = __shfl_sync(0xffffffffu, n1[1], from < 0 ? lane : from);
          const double gf = __shfl_sync(0xffffffffu, g2[1], from < 0 ? lane : from);
          const int pt = __shfl_sync(0xffffffffu, pos[0], to < 0 ? lane : to);
          const int jt = __shfl_sync(0xffffffffu, id[0], to < 0 ? lane : to);
          if (to >= 0) { pos[1] = pt; id[1] = jt; }
          if (from >= 0) { pos[0] = pf; id[0] = jf; n1[0] = nf; g2[0] = gf; }
          cs = 1;
          qr_bar<QW, NWT>();
        }
      }
      dots = true;
    }
    if (warp == rw) {
#pragma unroll
      for (int t = 0; t < CS; ++t)
        if (lane + 32 * t < e) {
          perm[pos[t]] = id[t];
          slot[pos[t]] = lane + 32 * t;
        }
    }
  }
  __syncthreads();
  return shi[5];
}

// T (k x (e-k), ld ldt) = R_1^{-1} R_2 with R(a, b) = Y[a + ldy slot[b]] (k <= 64): four columns per
// warp, lanes over the rows; the column of R_1 is scaled by its reciprocal pivot once for the four.
// rinv: >= k scratch.
template <typename T, int NWT>
__device__ void fast_interp(const T* Y, int ldy, int k, int e, const int* slot, T* Tm, int ldt, T* rinv) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int CJ = 4;
  for (int a = threadIdx.x; a < k; a += blockDim.x) rinv[a] = T(1) / Y[a + ldy * slot[a]];
  __syncthreads();
  for (int j0 = CJ * warp; j0 < e - k; j0 += CJ * NWT) {
    T s[2][CJ];
#pragma unroll
    for (int q = 0; q < CJ; ++q) {
      const int col = slot[min(k + j0 + q, e - 1)];
#pragma unroll
      for (int t = 0; t < 2; ++t) s[t][q] = lane + 32 * t < k ? Y[min(lane + 32 * t, k - 1) + ldy * col] : T(0);
    }
    for (int a = k - 1; a >= 0; --a) {
      const T* ra = Y + ldy * slot[a];
      const T iv = rinv[a];
      T x[CJ];
#pragma unroll
      for (int q = 0; q < CJ; ++q) x[q] = __shfl_sync(0xffffffffu, a < 32 ? s[0][q] : s[1][q], a & 31);
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        if (lane + 32 * t < a) {
          const T g = ra[lane + 32 * t] * iv;
#pragma unroll
          for (int q = 0; q < CJ; ++q) s[t][q] -= g * x[q];
        }
      }
    }
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int a = lane + 32 * t;
      if (a < k) {
#pragma unroll
        for (int q = 0; q < CJ; ++q)
          if (j0 + q < e - k) Tm[a + (size_t)ldt * (j0 + q)] = s[t][q] * rinv[a];
      }
    }
  }
  __syncthreads();
}

// Elimination of the last n = e - k rows and columns of the e x e block A (e <= 32 RS) with partial
// pivoting among those rows: L, U and the multipliers in place (interchanged with their rows),
// W = L^{-1} P A_rk, Z = A_kr U^{-1} and A_kk - Z W, one pass per pivot: lanes own rows (lane l:
// rows l, l + 32), warps own columns.  One barrier per pivot: the warp that holds the next pivot
// column updates it first, finds its pivot, scales it (and the Z entries) and publishes both while
// the others update the remaining columns.  q receives the permutation ((P b)_i = b_{q_i}), inv
// the reciprocal pivots: n each; shi: >= 4.  False on a zero pivot.
// What bounds it: that chain (update, pivot search on bit patterns, one reciprocal, barrier); it
// replaces five barriers per pivot and two serial sweeps for Z and the Schur update (1023^2, per
// segment: FP64 33 -> 13 us at level 6, level 1 with e = 44 106 -> 41 us; mixed 18 -> 9, 54 -> 22 us).
template <typename T, int NWT, int RS>
__device__ bool fast_elim(T* A, int lda, int k, int e, int* q, T* inv, int* shi, int* okf) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = e - k;
  // column cj = k + j of the block: pivot among rows >= cj, swap, scale rows below and rows < k
  auto prepare = [&](int j) {
    const int cj = k + j;
    T* col = A + lda * cj;
    T x[RS];
    unsigned hi = 0, lo = 0, best = 0xffffffffu;
#pragma unroll
    for (int t = 0; t < RS; ++t) {
      const int r = lane + 32 * t;
      x[t] = r < e ? col[min(r, e - 1)] : T(0);
      if (r >= cj && r < e) hi = max(hi, abs_hi(x[t]));
    }
    hi = __reduce_max_sync(0xffffffffu, hi);
    if constexpr (sizeof(T) == 8) {
#pragma unroll
      for (int t = 0; t < RS; ++t) {
        const int r = lane + 32 * t;
        if (r >= cj && r < e && abs_hi(x[t]) == hi) lo = max(lo, abs_lo(x[t]));
      }
      lo = __reduce_max_sync(0xffffffffu, lo);
    }
#pragma unroll
    for (int t = 0; t < RS; ++t) {
      const int r = lane + 32 * t;
      if (r >= cj && r < e && abs_hi(x[t]) == hi && abs_lo(x[t]) == lo) best = min(best, (unsigned)r);
    }
    best = __reduce_min_sync(0xffffffffu, best);
    const int p = (int)min(best, (unsigned)(e - 1));
    const bool zero = (hi | lo) == 0u;
    const T pv = __shfl_sync(0xffffffffu, p < 32 ? x[0] : x[RS - 1], p & 31);
    const T old = __shfl_sync(0xffffffffu, cj < 32 ? x[0] : x[RS - 1], cj & 31);
    const T iv = zero ? T(0) : T(1) / pv;
#pragma unroll
    for (int t = 0; t < RS; ++t) {
      const int r = lane + 32 * t;
      if (r < e) {
        if (r == cj) col[r] = pv;
        else if (r > cj) col[r] = (r == p ? old : x[t]) * iv;
        else if (r < k) col[r] = x[t] * iv;
      }
    }
    if (lane == 0) {
      shi[j & 1] = p;
      const int a = q[j], b = q[p - k];
      q[j] = b;
      q[p - k] = a;
      inv[j] = iv;
      if (zero) *okf = 0;
    }
  };
  if (threadIdx.x == 0) *okf = 1;
  for (int j = threadIdx.x; j < n; j += blockDim.x) q[j] = j;
  __syncthreads();
  if (warp == 0) prepare(0);
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    const int cj = k + j, p = shi[j & 1];
    T l[RS];
    bool act[RS];
#pragma unroll
    for (int t = 0; t < RS; ++t) {
      const int r = lane + 32 * t;
      act[t] = r < e && (r < k || r > cj);
      l[t] = act[t] ? A[min(r, e - 1) + lda * cj] : T(0);
    }
    // one column of the update: row cj takes row p's entry, row p the old row cj's
    auto column = [&](int c) {
      T* col = A + lda * c;
      const T u = col[p], oc = col[cj];
      T x[RS];
#pragma unroll
      for (int t = 0; t < RS; ++t) {
        const int r = lane + 32 * t;
        x[t] = act[t] ? (r == p ? oc : col[min(r, e - 1)]) - l[t] * u : u;
      }
      __syncwarp();
#pragma unroll
      for (int t = 0; t < RS; ++t) {
        const int r = lane + 32 * t;
        if (act[t] || r == cj) col[min(r, e - 1)] = x[t];
      }
      __syncwarp();
    };
    // the multipliers of earlier steps follow their rows
    if (p != cj)
      for (int c = k + threadIdx.x; c < cj; c += blockDim.x) {
        const T a = A[cj + lda * c];
        A[cj + lda * c] = A[p + lda * c];
        A[p + lda * c] = a;
      }
    // columns 0 .. k-1 and cj+1 .. e-1; the next pivot column by warp (j + 1) mod NWT alone, the
    // others by the other warps in turn
    const int wn = (j + 1) % NWT;
    const int nc = k + (n - j - 2 > 0 ? n - j - 2 : 0);
    if (warp == wn && j + 1 < n) {
      column(cj + 1);
      prepare(j + 1);
    } else {
      const int nw = j + 1 < n ? NWT - 1 : NWT;
      int w = warp;
      if (j + 1 < n) w = (warp - wn - 1 + NWT) % NWT;      // 0 .. NWT-2
      for (int x = w; x < nc; x += nw) column(x < k ? x : cj + 2 + (x - k));
    }
    __syncthreads();
  }
  return *okf != 0;
}

// X (n x n, ld n) = [L^{-1} \ U^{-1}] of the factored n x n block A (ld lda, n <= 32 RS; unit lower
// L below the diagonal, reciprocal pivots rinv): the solve applies the two as products.  Four
// columns per warp, lanes over the rows, one step per row of the block; U is scaled by the
// reciprocal pivot of the step once for the four columns.
template <typename T, int NWT, int RS>
__device__ void fast_invert(const T* A, int lda, int n, const T* rinv, T* X) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int CJ = 4;
  for (int j0 = CJ * warp; j0 < n; j0 += CJ * NWT) {
    T s[RS][CJ];
#pragma unroll
    for (int t = 0; t < RS; ++t)
#pragma unroll
      for (int q = 0; q < CJ; ++q) {
        const int i = lane + 32 * t, j = j0 + q;
        const T v = A[min(i, n - 1) + lda * min(j, n - 1)];
        s[t][q] = (i > j && i < n) ? v : T(0);
      }
    for (int m = j0 + 1; m < n; ++m) {             // L x = e_j: x_i = -(L_ij + sum_m L_im x_m)
      T x[CJ];
#pragma unroll
      for (int q = 0; q < CJ; ++q) x[q] = __shfl_sync(0xffffffffu, m < 32 ? s[0][q] : s[RS - 1][q], m & 31);
#pragma unroll
      for (int t = 0; t < RS; ++t) {
        const int i = lane + 32 * t;
        if (i > m && i < n) {
          const T l = A[i + lda * m];
#pragma unroll
          for (int q = 0; q < CJ; ++q) s[t][q] -= l * x[q];
        }
      }
    }
#pragma unroll
    for (int t = 0; t < RS; ++t)
#pragma unroll
      for (int q = 0; q < CJ; ++q) {
        const int i = lane + 32 * t, j = j0 + q;
        if (i > j && i < n) X[i + n * j] = -s[t][q];
        s[t][q] = T(0);
      }
    for (int m = min(j0 + CJ, n) - 1; m >= 0; --m) {   // U x = e_j: x_i = -rinv_i sum_{m > i} U_im x_m
      T x[CJ];
#pragma unroll
      for (int q = 0; q < CJ; ++q) {
        x[q] = __shfl_sync(0xffffffffu, m < 32 ? s[0][q] : s[RS - 1][q], m & 31);
        if (m == j0 + q) x[q] = T(-1);
      }
      const T iv = rinv[m];
#pragma unroll
      for (int t = 0; t < RS; ++t) {
        const int i = lane + 32 * t;
        if (i < m) {
          const T g = A[i + lda * m] * iv;
#pragma unroll
          for (int q = 0; q < CJ; ++q) s[t][q] -= g * x[q];
        }
      }
    }
#pragma unroll
    for (int t = 0; t < RS; ++t)
#pragma unroll
      for (int q = 0; q < CJ; ++q) {
        const int i = lane + 32 * t, j = j0 + q;
        if (i <= j && j < n) X[i + n * j] = i == j ? rinv[i] : -s[t][q] * rinv[i];
      }
  }
  __syncthreads();
}

// Largest-first work list of a level (scheduling, not in the paper): a counting sort of the
// segment ids by decreasing unknown count, so that the sparsify CTAs, which the hardware
// starts roughly in index order, begin with the longest segments and the last wave holds the
// shortest.  Ids of equal count land in any order: every CTA writes only its own segment's
// outputs and keys its sketch by the segment id, so the order changes no result.
constexpr int ORD_B = 256;
__global__ void __launch_bounds__(1024) seg_order_kernel(const int* cnt, int nseg, int* order) {
  __shared__ int start[ORD_B];
  auto key = [](int e) { return ORD_B - 1 - min(max(e, 0), ORD_B - 1); };
  for (int i = threadIdx.x; i < ORD_B; i += blockDim.x) start[i] = 0;
  __syncthreads();
  for (int s = threadIdx.x; s < nseg; s += blockDim.x) atomicAdd(&start[key(cnt[s])], 1);
  __syncthreads();
  if (threadIdx.x < 32) {            // exclusive scan of the 256 bucket sizes by one warp
    constexpr int PER = ORD_B / 32;
    const int lane = threadIdx.x;
    int v[PER], t = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) { v[j] = start[lane * PER + j]; t += v[j]; }
    int incl = t;
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    int run = incl - t;
#pragma unroll
    for (int j = 0; j < PER; ++j) { start[lane * PER + j] = run; run += v[j]; }
  }
  __syncthreads();
  for (int s = threadIdx.x; s < nseg; s += blockDim.x) order[atomicAdd(&start[key(cnt[s])], 1)] = s;
}

constexpr int WIDE_EMAX = 512;    // rows that wide_interp keeps in registers; shared memory ends before
                                  // (sparsify_wide_plan)
// Segments of at most 32 unknowns go to a cluster from this many entries of B; larger ones always do.
// Measured per level, one CTA / cluster: e 31 with 4000 entries 291 / 322 us, e 31 with 9000 312 / 291,
// e 46 with 4500 457 / 406, e 267 without neighbours (the last separator) 12.9 ms / 0.74 ms.
constexpr int WIDE_MIN = 5000;
__device__ __forceinline__ bool wide_takes(const LevelDev& d, const SegCtx& S, int tb);   // below

// Shared memory of a segment besides its blocks (norms, permutations, pivots, reciprocals), and the
// values of its interpolation matrix (k (e - k) <= e^2 / 4, and room for the 8 probe rows)
__host__ __device__ inline size_t sparsify_smem_small(int e, int tbytes) {
  return 2 * (size_t)e * 8 + (3 * (size_t)e + 4) * 4 + (size_t)e * tbytes + 64;
}
__host__ __device__ inline int sparsify_t_values(int e) { return e * e / 4 > 8 * e ? e * e / 4 : 8 * e; }

// Segment of this CTA: ID, elimination of the remainder, outputs (every thread calls it).
template <typename T, int NWT>
__device__ __forceinline__ void sparsify_segment(const LevelDev& d, int smem_bytes) {
  extern __shared__ double sm[];
  __shared__ SegCtx S;
  __shared__ double shr[NWT * 64 + 3 * 64];
  __shared__ int shi[8];
  __shared__ int nearlist[NEAR_MAX];
  __shared__ int nnear_sh, nfar_sh;

  const int sid = d.use_order ? d.order[blockIdx.x] : blockIdx.x;
  if (threadIdx.x == 0) seg_context(d, sid, S);
  __syncthreads();
  const int e = S.e;
  const int capS = d.capS;
  if (wide_takes(d, S, sizeof(T))) return;             // sparsify_wide_kernel's
  int* perm_out = d.perm + (size_t)sid * capS;
  if (threadIdx.x == 0) atomicMax(d.lstat + LS_EMAX, e);
  if (e == 0) {
    if (threadIdx.x == 0) { d.kk[sid] = 0; d.hs[sid] = 0; }
    return;
  }
  const size_t ld = d.ldF;
  const T* F1 = static_cast<const T*>(d.F) + (size_t)S.b1 * ld * ld;
  const T* F2 = static_cast<const T*>(d.F) + (size_t)S.b2 * ld * ld;
  T* Dg = static_cast<T*>(d.Dm) + (size_t)sid * capS * capS;
  T* Tg = static_cast<T*>(d.T) + (size_t)sid * capS * capS;
  T* Ig = static_cast<T*>(d.Dinv) + (size_t)sid * capS;
  const int halves = d.symmetric ? 1 : 2;

  // eps == 0: no sparsification, the whole segment is skeleton
  if (d.eps == 0.0) {
    for (int x = threadIdx.x; x < e * e; x += blockDim.x) {
      int a = x % e, b = x / e;
      Dg[a + (size_t)capS * b] = F1[(S.s1 + a) + ld * (S.s1 + b)] + F2[(S.s2 + a) + ld * (S.s2 + b)];
    }
    for (int j = threadIdx.x; j < e; j += blockDim.x) {
      perm_out[j] = j;
      d.snodes[(size_t)sid * capS + j] = d.nodes[(size_t)sid * capS + j];
    }
    if (threadIdx.x == 0) {
      d.kk[sid] = e;
      d.hs[sid] = 0;
      atomicAdd(d.flops + 2, (unsigned long long)(e * e * sizeof(T) + 2 * e * sizeof(int)));
    }
    return;
  }

  // near / far split of the neighbours (ordered scan, warp 0)
  if (threadIdx.x < 32) {
    int lane = threadIdx.x, nn = 0;
    for (int base = 0; base < S.nb; base += 32) {
      int f = base + lane;
      bool isnear = false;
      if (f < S.nb) {
        int r, i;
        locate(S, f, r, i);
        isnear = cheb(S, run_node(d, S.run[r], i), d.nx) <= d.near_radius;
      }
      unsigned msk = __ballot_sync(0xffffffffu, isnear);
      int pos = nn + __popc(msk & ((1u << lane) - 1u));
      if (isnear && pos < NEAR_MAX) nearlist[pos] = f;
      nn += __popc(msk);
    }
    if (lane == 0) {
      if (nn > NEAR_MAX) atomicOr(d.err, ERR_CAPACITY);
      nnear_sh = min(nn, NEAR_MAX);
      nfar_sh = S.nb - nn;
    }
  }
  // neighbour table (all threads)
  __shared__ int tb_node[NB_MAX];
  __shared__ short tb_p1[NB_MAX], tb_p2[NB_MAX];
  __shared__ unsigned char tb_nf[NB_MAX];
  const NbrTab tb{tb_node, tb_p1, tb_p2, tb_nf, S.nb <= NB_MAX};
  if (tb.on) {
    const NbrTab none{nullptr, nullptr, nullptr, nullptr, false};
    for (int f = threadIdx.x; f < S.nb; f += blockDim.x) {
      const Nbr q = nbr_get(d, S, none, f);
      tb_node[f] = q.node;
      tb_p1[f] = (short)q.p1;
      tb_p2[f] = (short)q.p2;
      tb_nf[f] = q.nearf ? 1 : 0;
    }
  }
  __syncthreads();
  const int nnear = nnear_sh;
  const int nN = halves * nnear;
  const int nF = halves * nfar_sh;
  const int hcap = max(d.h0, 2 * (e + d.p_over));
  const int hmax = min(nF, hcap);

  // rank bound (k <= e): a segment with e + p <= 2 h0 is sketched once with
  // h = min(2 h0, hmax) >= min(|F|, e + p), the size the adaptive schedule reaches at its
  // second pass, and that pass always stands; the predictor serves the larger segments.
  // Every h stays <= hbuf, the rows the sketch buffer was sized for.
  const bool small = e + d.p_over <= 2 * d.h0;
  const int hbuf = small ? min(hmax, 2 * d.h0) : hmax;
  const int mmax = nN + hbuf;

  // working storage: vectors and sketch chunks in shared memory; Y, D, T too when they
  // fit, else the global scratch of this segment.  The sketch chunks and D share their place (D
  // is formed when the last sketch is done), T holds k (e - k) values (or the 8 probe rows)
  const size_t TD = sizeof(T);
  const size_t small_b = sparsify_smem_small(e, (int)TD);
  const size_t per_ch_b = (size_t)halves * (e + hbuf) * TD;
  const size_t y_b = (size_t)max(mmax + 1, e) * e * TD, t_b = (size_t)sparsify_t_values(e) * TD;
  const size_t d_b = (size_t)e * e * TD;
  auto fit_b = [&](int c) { return small_b + y_b + t_b + max(c * per_ch_b, d_b); };
  // chunk of the sketch product: the largest of 64, 32 and 16 far unknowns whose working set
  // fits the budget together with the staged B block (or without it, where B never fits):
  // fewer chunks, fewer barriers on the coarse levels' long far fields
  int ch = SK_CHUNK;
  {
    const size_t bsz = (size_t)halves * S.nb * e * TD + 48;
    const bool keep_b = fit_b(SK_CHUNK) + bsz <= (size_t)smem_bytes;
    for (int c = SK_CHUNK_MAX; c > SK_CHUNK; c >>= 1)
      if (fit_b(c) + (keep_b ? bsz : 0) <= (size_t)smem_bytes) { ch = c; break; }
  }
  bool in_smem = fit_b(ch) <= (size_t)smem_bytes;
  if (!in_smem) {
    size_t room = (size_t)smem_bytes > small_b ? (size_t)smem_bytes - small_b : 0;
    ch = (int)min((size_t)SK_CHUNK, room / (per_ch_b > 0 ? per_ch_b : 1));
    if (ch < 1) { ch = 1; if (threadIdx.x == 0) atomicOr(d.err, ERR_CAPACITY); }
  }
  T *Y, *Dw, *Tw, *Bc, *Gc, *rinv, *Bs;
  bool bstage;
  double *vn1, *vn2;
  int *perm, *piv, *flags;
  int ldy, ldd;
  {
    char* q = reinterpret_cast<char*>(sm);
    vn1 = reinterpret_cast<double*>(q); q += (size_t)e * 8;
    vn2 = reinterpret_cast<double*>(q); q += (size_t)e * 8;
    perm = reinterpret_cast<int*>(q); q += (size_t)e * 4;
    piv = reinterpret_cast<int*>(q); q += (size_t)e * 4;
    flags = reinterpret_cast<int*>(q); q += ((size_t)e + 4) * 4;
    q = reinterpret_cast<char*>(((uintptr_t)q + 15) & ~(uintptr_t)15);
    rinv = reinterpret_cast<T*>(q); q += (size_t)e * TD;
    q = reinterpret_cast<char*>(((uintptr_t)q + 15) & ~(uintptr_t)15);
    Bc = reinterpret_cast<T*>(q);
    Gc = Bc + (size_t)halves * ch * e;
    if (in_smem) {
      Dw = Bc; ldd = e;
      q += max(ch * per_ch_b, d_b);
      Y = reinterpret_cast<T*>(q); q += y_b; ldy = mmax | 1;   // odd pitch
      Tw = reinterpret_cast<T*>(q); q += t_b;
    } else {
      q += ch * per_ch_b;
      Y = static_cast<T*>(d.Yg) + (size_t)sid * d.Ycap * capS; ldy = d.Ycap;
      Dw = Dg; ldd = capS;
      Tw = Tg;
    }
    // the segment's B block (every neighbour row, e columns) in what is left, when it fits
    q = reinterpret_cast<char*>(((uintptr_t)q + 15) & ~(uintptr_t)15);
    Bs = reinterpret_cast<T*>(q);
    bstage = (size_t)(q - reinterpret_cast<char*>(sm)) + (size_t)halves * S.nb * e * TD <= (size_t)smem_bytes;
  }
  if (!in_smem && (mmax > d.Ycap || d.Yg == nullptr)) {   // no room: report, touch nothing
    if (threadIdx.x == 0) { atomicOr(d.err, ERR_CAPACITY); d.kk[sid] = 0; d.hs[sid] = 0; }
    return;
  }
  if (!in_smem && threadIdx.x == 0) atomicAdd(d.lstat + LS_SCRATCH, 1);
  // B staged once (all loads in flight) for the near rows, every sketch pass, the probe and
  // the error test; otherwise each reads the frontal blocks through the neighbour table
  if (bstage) {
    for (int x = threadIdx.x; x < halves * S.nb * e; x += blockDim.x) {
      const int row = x / e, c = x % e;
      Bs[x] = bval_q<T>(d, S, F1, F2, nbr_get(d, S, tb, row % S.nb), row / S.nb, c);
    }
    __syncthreads();
  }
  auto bget = [&](int t, int f, int c) -> T {
    return bstage ? Bs[((size_t)t * S.nb + f) * e + c] : bval_q<T>(d, S, F1, F2, nbr_get(d, S, tb, f), t, c);
  };

  // ---- learned rank predictor (not in the paper): features from an 8-row probe of the
  //      far rows, then the network's one-pass sketch size (PRED_PREDICT) or a training
  //      record of the features and the adaptive rank (PRED_RECORD)
  __shared__ float xf[PRED_NFEAT], zs[PRED_NFEAT], hid[PRED_NHID], pout[PRED_NOUT];
  const bool use_pred = d.pred_mode != PRED_OFF && nF > max(d.h0, PRED_PROBE) && e <= PRED_EMAX && !small;
  int h = (nF <= d.h0) ? nF : small ? min(hmax, 2 * d.h0) : min(hmax, d.h0);
  bool predicted = false;
  if (use_pred) {
    for (int x = threadIdx.x; x < PRED_PROBE * e; x += blockDim.x) Y[x] = T(0);   // Y8, pitch 8
    __syncthreads();
    probe_sketch<T>(d, S, tb, bget, sid, halves, e, Y);
    __syncthreads();
    if (d.pred_mode == PRED_PREDICT && e >= PRED_PROBE) {
      // keep the probe (the first PRED_PROBE rows of this segment's G times B_F, unscaled) for
      // the one-pass sketch: the features' QR overwrites it, and T is free until the ID
      for (int x = threadIdx.x; x < PRED_PROBE * e; x += blockDim.x) Tw[x] = Y[x];
      __syncthreads();
    }
    probe_features<T>(d, sid, e, nnear, nfar_sh, S.nb, Y, xf);
    if (d.pred_mode == PRED_RECORD) {
      if (threadIdx.x < PRED_NFEAT) d.feat[(size_t)sid * PRED_NFEAT + threadIdx.x] = xf[threadIdx.x];
    } else {
      mlp_infer_block(*d.pred, xf, zs, hid, pout);
      h = pred_sketch_size(pout, nF, e, d.p_over, d.h0, d.pred_margin);
      predicted = true;
    }
  }

  h = min(h, hbuf);          // the sketch buffer holds nN + hbuf rows
  // ---- adaptive sketch + ID (Sec. 4.2.3; h = k + p with k unknown: double h until k <= h - p)
  int k = 0;
  int passes = 0;
  int ldt = capS;            // in shared memory: k
  bool fellback = false, have_t = false;
  const bool fast = NWT != NW || e <= 64;   // the register-and-lane forms of the QR and what follows
  // A pass that may have to be repeated with a larger h leaves its unscaled sketch rows in the
  // segment's global scratch: the larger sketch has the same first rows (same counters, same
  // sums), so only the new ones are formed
  T* Ykeep = (in_smem && d.Yg) ? static_cast<T*>(d.Yg) + (size_t)sid * d.Ycap * capS : nullptr;
  int have = 0;
  const bool was_predicted = predicted;
  unsigned long long work_done = 0;       // algorithmic FLOPs of this segment (thread 0)
  while (true) {
    const bool full = (h >= nF);
    const int hh = full ? nF : h;
    const int m = nN + hh;
    if (threadIdx.x == 0 && !full) work_done += work::sketch(hh, nF, e);
    // near rows
    for (int x = threadIdx.x; x < nN * e; x += blockDim.x) {
      int row = x % nN, c = x / nN;
      int t = row / nnear, a = row % nnear;
      Y[row + (size_t)ldy * c] = bget(t, nearlist[a], c);
    }
    if (full) {
      // Phi = I on the far block: far rows in the enumeration order of the neighbours;
      // position of far neighbour f = f minus the near ones before it
      for (int f = threadIdx.x; f < S.nb; f += blockDim.x) {
        int before = 0;
        bool isnear = false;
        for (int a = 0; a < nnear; ++a) {
          if (nearlist[a] < f) ++before;
          if (nearlist[a] == f) isnear = true;
        }
        if (isnear) continue;
        int j = f - before;
        for (int t = 0; t < halves; ++t)
          for (int c = 0; c < e; ++c)
            Y[(nN + t * nfar_sh + j) + (size_t)ldy * c] = bget(t, f, c);
      }
    } else {
      // Y_F = G B_F, chunks of neighbours (near ones get zero weight); the one-pass sketch of
      // a predicted segment takes its first PRED_PROBE rows from the probe
      const bool probe = predicted && e >= PRED_PROBE;
      const int r0 = probe ? min(PRED_PROBE, hh) : have;
      if (r0 < hh) sketch_far<T>(d, S, tb, bget, sid, halves, e, r0, hh, Y + nN, ldy, Bc, Gc, ch);
      const T sc = (T)(1.0 / sqrt((double)hh));
      const bool keep = Ykeep && (predicted || e > hh - d.p_over);
      for (int x = threadIdx.x; x < hh * e; x += blockDim.x) {
        const int rr = x % hh, c = x / hh;
        T* yv = Y + (nN + rr) + (size_t)ldy * c;
        const T v = rr >= r0 ? *yv : probe ? Tw[rr + PRED_PROBE * c] : Ykeep[rr + (size_t)d.Ycap * c];
        if (keep && rr >= have) Ykeep[rr + (size_t)d.Ycap * c] = v;
        *yv = v * sc;
      }
      if (keep) have = hh & ~3;              // whole counters of four rows
    }
    __syncthreads();
    // a pass that can still double h only needs to know whether k > h - p: its QR stops at
    // step h - p + 1 (the same decision, the remaining steps skipped)
    const int kstop = (!full && h < nF) ? max(1, hh - d.p_over + 1) : e;
    {
      constexpr int QW = NWT != NW ? NWT : sizeof(T) == 8 ? 4 : 8;
      if (!fast) k = block_cpqr<T, NWT>(Y, ldy, m, e, d.eps, perm, vn1, vn2, shr, flags, shi, kstop);
      else if (NWT != NW || e <= 32) k = fast_cpqr<T, NWT, QW, 1>(Y, ldy, m, e, d.eps, perm, flags, shr, shi, kstop);
      else if constexpr (NWT == NW) k = fast_cpqr<T, NWT, QW, 2>(Y, ldy, m, e, d.eps, perm, flags, shr, shi, kstop);
    }
    ++passes;
    if (threadIdx.x == 0) work_done += work::qr(m, e, k);
    if (in_smem) ldt = max(k, 1);
    if (predicted) {          // the one-pass ID stands if it passes the measured-error test
      predicted = false;
      if (full) break;
      bool ok = k <= h - d.p_over;
      if (ok) {
        if (fast) fast_interp<T, NWT>(Y, ldy, k, e, flags, Tw, ldt, rinv);
        else block_interp<T>(Y, ldy, k, e, Tw, ldt, rinv);
        have_t = true;
        ok = id_error_ok<T>(S, bget, halves, e, k, perm, Tw, ldt, d.eps, shr);
      }
      if (ok) break;
      fellback = true;
      have_t = false;
      h = min(2 * h, hmax);     // hmax = min(|F|, max(h0, 2(e+p))): k <= e < hmax - p
      __syncthreads();
      continue;
    }
    if (!full && k > h - d.p_over && h < nF) {
      h = min(2 * h, hmax);     // never binds without a prediction (h < 2(k+p))
      __syncthreads();
      continue;
    }
    break;
  }
  if (threadIdx.x == 0) {
    atomicAdd(d.lstat + LS_PASSES, passes);
    if (fellback) atomicAdd(d.lstat + LS_FALLBACK, 1);
    if (was_predicted) atomicAdd(d.lstat + LS_PREDICTED, 1);
    if (use_pred && d.pred_mode == PRED_RECORD) {
      int* tg = d.tgt + (size_t)sid * 4;
      tg[0] = k; tg[1] = nF; tg[2] = 1; tg[3] = passes;
    }
  }
  const int r = e - k;
  if (!have_t) {
    if (fast) fast_interp<T, NWT>(Y, ldy, k, e, flags, Tw, ldt, rinv);
    else block_interp<T>(Y, ldy, k, e, Tw, ldt, rinv);
  }

  // ---- transformed diagonal block in [skeleton | remainder] order (Eq. (UtALt))
  for (int x = threadIdx.x; x < e * e; x += blockDim.x) {
    int a = x % e, b = x / e;
    int pa = perm[a], pb = perm[b];
    Dw[a + (size_t)ldd * b] = F1[(S.s1 + pa) + ld * (S.s1 + pb)] + F2[(S.s2 + pa) + ld * (S.s2 + pb)];
  }
  __syncthreads();
  if (k > 0 && r > 0) {
    // column operation: D[:, k:] -= D[:, :k] T
    for (int x = threadIdx.x; x < e * r; x += blockDim.x) {
      int a = x % e, b = x / e;
      T s = T(0);
      for (int c = 0; c < k; ++c) s += Dw[a + (size_t)ldd * c] * Tw[c + (size_t)ldt * b];
      Dw[a + (size_t)ldd * (k + b)] -= s;
    }
    __syncthreads();
    // row operation: D[k:, :] -= T^T D[:k, :]
    for (int x = threadIdx.x; x < r * e; x += blockDim.x) {
      int a = x % r, b = x / r;
      T s = T(0);
      for (int c = 0; c < k; ++c) s += Tw[c + (size_t)ldt * a] * Dw[c + (size_t)ldd * b];
      Dw[(k + a) + (size_t)ldd * b] -= s;
    }
    __syncthreads();
  }
  // ---- eliminate the remainder: LU(A_rr) with W = L^{-1} P A_rk, Z = A_kr U^{-1},
  //      A_kk -= Z W  (Eq. (L^-1 * A * U^-1) for the segments of level l)
  if (r > 0 && fast) {
    bool ok;
    if (NWT != NW || e <= 32) ok = fast_elim<T, NWT, 1>(Dw, ldd, k, e, piv, rinv, shi, shi + 6);
    else ok = fast_elim<T, NWT, 2>(Dw, ldd, k, e, piv, rinv, shi, shi + 6);
    if (!ok && threadIdx.x == 0) atomicOr(d.err, ERR_SINGULAR);
  } else if (r > 0) {
    bool ok = block_gepp<T>(Dw, ldd, k, r, e, piv, rinv, shi, r <= INV_MAX);
    if (!ok && threadIdx.x == 0) atomicOr(d.err, ERR_SINGULAR);
    if (k > 0) {
      for (int a = threadIdx.x; a < k; a += blockDim.x) {     // Z = A_kr U^{-1}, row by row
        for (int j = 0; j < r; ++j) {
          T s = Dw[a + (size_t)ldd * (k + j)];
          for (int i2 = 0; i2 < j; ++i2) s -= Dw[a + (size_t)ldd * (k + i2)] * Dw[(k + i2) + (size_t)ldd * (k + j)];
          Dw[a + (size_t)ldd * (k + j)] = s * rinv[j];
        }
      }
      __syncthreads();
      for (int x = threadIdx.x; x < k * k; x += blockDim.x) {
        int a = x % k, b = x / k;
        T s = T(0);
        for (int j = 0; j < r; ++j) s += Dw[a + (size_t)ldd * (k + j)] * Dw[(k + j) + (size_t)ldd * b];
        Dw[a + (size_t)ldd * b] -= s;
      }
      __syncthreads();
    }
  }
  // ---- the remainder block inverted for the solve (the sketch's place is free), r <= INV_MAX
  if (r > 0 && r <= INV_MAX) {
    T* Db = Dw + k + (size_t)ldd * k;
    if (NWT != NW || r <= 32) fast_invert<T, NWT, 1>(Db, ldd, r, rinv, Y);
    else fast_invert<T, NWT, 2>(Db, ldd, r, rinv, Y);
    for (int x = threadIdx.x; x < r * r; x += blockDim.x) Db[(x % r) + (size_t)ldd * (x / r)] = Y[x];
    if (!fast && threadIdx.x == 0) {     // the pivot sequence as a permutation
      for (int i = 0; i < r; ++i) flags[i] = i;
      for (int j = 0; j < r; ++j) { const int p = piv[j], t = flags[j]; flags[j] = flags[p]; flags[p] = t; }
      for (int i = 0; i < r; ++i) piv[i] = flags[i];
    }
    __syncthreads();
  }
  // ---- outputs
  if (in_smem) {
    for (int x = threadIdx.x; x < e * e; x += blockDim.x) Dg[(x % e) + (size_t)capS * (x / e)] = Dw[x];
    for (int x = threadIdx.x; x < k * r; x += blockDim.x) Tg[(x % k) + (size_t)capS * (x / k)] = Tw[(x % k) + (size_t)ldt * (x / k)];
  }
  for (int j = threadIdx.x; j < e; j += blockDim.x) {
    perm_out[j] = perm[j];
    d.snodes[(size_t)sid * capS + j] = d.nodes[(size_t)sid * capS + perm[j]];
  }
  for (int j = threadIdx.x; j < r; j += blockDim.x) {
    d.piv[(size_t)sid * capS + j] = piv[j];
    Ig[j] = rinv[j];
  }
  if (threadIdx.x == 0) {
    d.kk[sid] = k;
    d.hs[sid] = h;
    work_done += work::interp(k, e) + work::apply(e, k) + (r > 0 ? work::elim(r, k) : 0ull);
    atomicAdd(d.flops, work_done);
    atomicAdd(d.flops + 2, (unsigned long long)((k * r + e * e) * sizeof(T) + 2 * e * sizeof(int)));
  }
}

// Beside a wide kernel this one starts early: what follows both waits for both through the last CTA,
// which ends no sooner than the clusters do, whichever way its segment ended (with no such launch
// before it the wait is none).
template <typename T, int NWT>
__global__ void __launch_bounds__(NWT * 32, NWT == NW ? 4 : 16) sparsify_kernel(LevelDev d, int smem_bytes) {
  sparsify_segment<T, NWT>(d, smem_bytes);
  if (blockIdx.x == gridDim.x - 1) pdl_wait();
}

// W = L^{-1} P A_pd and Z = A_dp U^{-1} for the 32 boundary unknowns x0 .. x0 + 31 of a parent, from
// the factored block A (kp <= 32 RS, in shared memory), posn(x) the place of unknown x in M: four
// columns of W and four rows of Z per warp, lanes over the separator's unknowns, one step per unknown.
// Every shared address is in range whatever its lane's condition: loads may be issued ahead of it.
template <typename T, int RS, class Pos>
__device__ void panel_chunk(T* M, size_t ldp, int Dp, Pos posn, int x0, int ndP, int kp, const T* A, int lda,
                            const int* q, const T* inv, T* Zt) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int CJ = 4;
  const int ldz = kp | 1, nx = min(32, ndP - x0), w0 = CJ * warp;
  for (int x = threadIdx.x; x < 32 * kp; x += blockDim.x) {
    const int r = x & 31, j = x >> 5;
    Zt[r * ldz + j] = M[posn(x0 + min(r, nx - 1)) + ldp * (Dp + j)];
  }
  T s[RS][CJ];
  size_t pc[CJ];
#pragma unroll
  for (int c = 0; c < CJ; ++c) {
    pc[c] = ldp * posn(x0 + min(w0 + c, nx - 1));
#pragma unroll
    for (int t = 0; t < RS; ++t) {
      const int i = min(lane + 32 * t, kp - 1);
      s[t][c] = M[(Dp + q[i]) + pc[c]];
    }
  }
  __syncthreads();                                 // Zt; every entry of W's columns is in registers
  if (w0 < nx) {
    for (int j = 0; j < kp; ++j) {
      T x[CJ];
#pragma unroll
      for (int c = 0; c < CJ; ++c) {
        T v = s[0][c];
#pragma unroll
        for (int t = 1; t < RS; ++t) v = (j >> 5) == t ? s[t][c] : v;
        x[c] = __shfl_sync(0xffffffffu, v, j & 31);
      }
#pragma unroll
      for (int t = 0; t < RS; ++t) {
        const int i = lane + 32 * t;
        if (i > j && i < kp) {
          const T l = A[min(i, kp - 1) + lda * j];
#pragma unroll
          for (int c = 0; c < CJ; ++c) s[t][c] -= l * x[c];
        }
      }
    }
#pragma unroll
    for (int c = 0; c < CJ; ++c)
#pragma unroll
      for (int t = 0; t < RS; ++t)
        if (lane + 32 * t < kp && w0 + c < nx) M[(Dp + lane + 32 * t) + pc[c]] = s[t][c];
    // Z: row z of z U = a, lanes over its entries
#pragma unroll
    for (int c = 0; c < CJ; ++c)
#pragma unroll
      for (int t = 0; t < RS; ++t) s[t][c] = Zt[(w0 + c) * ldz + min(lane + 32 * t, kp - 1)];
    for (int j = 0; j < kp; ++j) {
      T x[CJ];
      const T iv = inv[j];
#pragma unroll
      for (int c = 0; c < CJ; ++c) {
        T v = s[0][c];
#pragma unroll
        for (int t = 1; t < RS; ++t) v = (j >> 5) == t ? s[t][c] : v;
        x[c] = __shfl_sync(0xffffffffu, v, j & 31);
      }
#pragma unroll
      for (int t = 0; t < RS; ++t) {
        const int i = lane + 32 * t;
        if (i > j && i < kp) {
          const T g = A[j + lda * min(i, kp - 1)] * iv;
#pragma unroll
          for (int c = 0; c < CJ; ++c) s[t][c] -= g * x[c];
        }
      }
    }
#pragma unroll
    for (int c = 0; c < CJ; ++c)
#pragma unroll
      for (int t = 0; t < RS; ++t)
        if (lane + 32 * t < kp) Zt[(w0 + c) * ldz + lane + 32 * t] = s[t][c] * inv[min(lane + 32 * t, kp - 1)];
  }
  __syncthreads();
  for (int x = threadIdx.x; x < 32 * kp; x += blockDim.x) {
    const int r = x & 31, j = x >> 5;
    if (r < nx) M[posn(x0 + r) + ldp * (Dp + j)] = Zt[r * ldz + j];
  }
  __syncthreads();
}

// ------------------------------------------------------------ sparsify: one cluster per segment
// On levels of few segments one CTA per segment leaves most SMs idle, and in FP64 the sketch, the
// QR and the dense products of a segment are bound by one SM's FP64 pipe (2 multiply-adds per
// clock).  Here a cluster of C CTAs shares a segment:
//   - rows of the sketch (whole Philox groups of four) are dealt out, each CTA forms and keeps its
//     own (the same sums as in sketch_far);
//   - QR with the rows where they are (row i of the pivot order is local row i / C of CTA i mod C;
//     missing rows are zero): per step every CTA sends its partial products with the pivot column,
//     and one its row i, to all, and after one cluster barrier all take the same decisions from the
//     same numbers, so nothing has to be sent back;
//   - interpolation, transforms and elimination by columns or elements over all CTAs, on the
//     segment's place in global memory, cluster barriers between.
// What bounds it: the pivots' serial chain (a cluster barrier, two block reductions, a FP64 square
// root and a quotient each) and the FP64 pipe of C SMs.  One CTA / cluster, 1023 x 1023 at eps 1e-8:
// Helmholtz, 10 segments of up to 155 unknowns, 33.2 / 3.6 ms; 24 of up to 101, 10.2 / 1.7 ms;
// diffusion, 24 of up to 57, 858 / 535 us.  FP64 only: in FP32 a segment is not bound by a pipe, and the
// clusters' barriers cost more than their SMs give (mixed, levels 6 - 2: 169 / 235, 188 / 230, 183 / 238,
// 142 / 192, 104 / 159 us).
// Columns: warp w of NSW = min(8, ceil(e / 32)) column sets x RG row groups holds set w mod NSW (and
// set w + 8 where e > 256), rows r mod RG = w / NSW; the warps of row group 0 own the columns' state.
namespace cg = cooperative_groups;

struct WideShape {             // sizes that every CTA of the cluster derives alike
  int C, rank, e, NS, NSW, RG, EC;
};

__host__ __device__ inline int wide_rows(int C, int nN, int far_rows, bool whole) {
  const int nr = (nN + C - 1) / C;
  return whole ? nr + (far_rows + C - 1) / C : nr + 4 * (((far_rows + 3) / 4 + C - 1) / C);
}
// Shared memory of a segment of e unknowns with nb neighbours, a sketch chunk of four far unknowns
// at least: exchange buffers (two parities of C sums and a row per column), partial sums of the row
// groups, coefficients, reciprocals, permutation and pivots, neighbour table; then the rows and the
// chunk, whose place the elimination of up to INV_MAX remainders takes later
__host__ __device__ inline size_t wide_bytes(int e, int nb, int C, int halves, int h0, int p_over, int tb) {
  const size_t ec = (size_t)(e + 31) / 32 * 32;
  const size_t fixed = (2 * (C + 1) * ec + ec + (ec > 256 ? ec : 256)) * 8 + (size_t)e * tb + 8 * (size_t)e + 9 * (size_t)nb + 64;
  const int hcap = h0 > 2 * (e + p_over) ? h0 : 2 * (e + p_over);
  const size_t m = wide_rows(C, halves * NEAR_MAX, hcap, false) | 1;
  const size_t y = m * e + 4 * (size_t)halves * (e + m), lu = 2 * INV_MAX * (INV_MAX + 1);
  return fixed + (y > lu ? y : lu) * tb;
}
// whether the segment is the wide kernel's (asked by both kernels)
__device__ __forceinline__ bool wide_takes(const LevelDev& d, const SegCtx& S, int tb) {
  const int halves = d.symmetric ? 1 : 2;
  return d.wide > 1 && S.e <= WIDE_EMAX && (S.e > 32 || halves * S.e * S.nb >= WIDE_MIN) &&
         wide_bytes(S.e, S.nb, d.wide, halves, d.h0, d.p_over, tb) <= (size_t)d.wide_smem;
}

// The QR above; every thread of every CTA calls it.  Yl: mloc rows (pitch ldl) of e columns.  R rows
// go to Rg (global, leading dimension ldr, columns in place) from CTA 0; perm in every CTA.
template <typename T, int MS>
__device__ int wide_qr(cg::cluster_group& cl, const WideShape& W, T* Yl, int ldl, int mloc, int m, double eps, int kstop,
                       double* xch, double* part, T* coef, int* perm, T* Rg, size_t ldr, double* sc, unsigned* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int e = W.e, C = W.C, rank = W.rank, EC = W.EC;
  const int kmax = min(min(m, e), kstop);
  const int set0 = warp % W.NSW, rg = warp / W.NSW;
  const bool on = rg < W.RG, own = on && rg == 0;
  int col[MS], pos[MS];
  bool val[MS];
  T* yc[MS];
  double n1[MS], g2[MS];
  const double tol3z = sqrt(DBL_EPSILON);
#pragma unroll
  for (int t = 0; t < MS; ++t) {
    col[t] = 32 * (set0 + 8 * t) + lane;
    val[t] = on && col[t] < e;
    yc[t] = Yl + ldl * min(col[t], e - 1);
    pos[t] = val[t] ? col[t] : e;
    n1[t] = g2[t] = 0.0;
  }
  int par = 0;
  // sums over the row groups and the CTAs of one value per column; in v[] for the owners
  auto gather_sum = [&](double (&v)[MS], const T* row) {
#pragma unroll
    for (int t = 0; t < MS; ++t)
      if (val[t]) part[rg * EC + col[t]] = v[t];
    __syncthreads();
    double* buf = xch + (size_t)par * (C + 1) * EC;          // C x EC sums, then the row
    if (own) {
#pragma unroll
      for (int t = 0; t < MS; ++t)
        if (val[t]) {
          double q = part[col[t]];
          for (int g = 1; g < W.RG; ++g) q += part[g * EC + col[t]];
          for (int c = 0; c < C; ++c) {
            double* pb = cl.map_shared_rank(buf, c);
            pb[rank * EC + col[t]] = q;
            if (row) pb[C * EC + col[t]] = (double)row[ldl * col[t]];
          }
        }
    }
    cl.sync();
    if (own) {
#pragma unroll
      for (int t = 0; t < MS; ++t)
        if (val[t]) {
          double q[8];
#pragma unroll
          for (int c = 0; c < 8; ++c) q[c] = c < C ? buf[min(c, C - 1) * EC + col[t]] : 0.0;
#pragma unroll
          for (int o = 4; o > 0; o >>= 1)
            if (o < C)
#pragma unroll
              for (int c = 0; c < 4; ++c)
                if (c < o) q[c] += q[c + o];
          v[t] = q[0];
        }
    }
    par ^= 1;
    return buf + C * EC;
  };
  // pivot among the positions >= i: key = position * 65536 + column, the same in every thread
  auto choose = [&](int i) {
    unsigned hi = 0, lo = 0;
#pragma unroll
    for (int t = 0; t < MS; ++t)
      if (own && pos[t] >= i && pos[t] < e) hi = max(hi, bits_hi(n1[t]));
    hi = __reduce_max_sync(0xffffffffu, hi);
#pragma unroll
    for (int t = 0; t < MS; ++t)
      if (own && pos[t] >= i && pos[t] < e && bits_hi(n1[t]) == hi) lo = max(lo, bits_lo(n1[t]));
    lo = __reduce_max_sync(0xffffffffu, lo);
    if (lane == 0) { red[2 * warp] = hi; red[2 * warp + 1] = lo; }
    __syncthreads();
    unsigned long long mx = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) mx = max(mx, ((unsigned long long)red[2 * q] << 32) | red[2 * q + 1]);
    const long long thr = tie_bits((long long)mx);
    unsigned best = 0xffffffffu, first = 0xffffffffu;
#pragma unroll
    for (int t = 0; t < MS; ++t)
      if (own && pos[t] >= i && pos[t] < e) {
        const unsigned key = ((unsigned)pos[t] << 16) | (unsigned)col[t];
        first = min(first, key);
        if (dbits(n1[t]) >= thr) best = min(best, key);
      }
    best = __reduce_min_sync(0xffffffffu, best);
    first = __reduce_min_sync(0xffffffffu, first);
    if (lane == 0) { red[16 + warp] = best; red[24 + warp] = first; }
    __syncthreads();
    best = first = 0xffffffffu;
#pragma unroll
    for (int q = 0; q < 8; ++q) { best = min(best, red[16 + q]); first = min(first, red[24 + q]); }
    return best != 0xffffffffu ? best : first;
  };
  double v[MS];
#pragma unroll
  for (int t = 0; t < MS; ++t) {
    T a = T(0);
    if (val[t])
      for (int r = rg; r < mloc; r += W.RG) { const T y = yc[t][r]; a += y * y; }
    v[t] = (double)a;
  }
  gather_sum(v, nullptr);
#pragma unroll
  for (int t = 0; t < MS; ++t) { n1[t] = unsign(v[t]); g2[t] = tol3z * v[t]; }
  unsigned key = choose(0);
  int k = kmax;
  for (int i = 0; i < kmax; ++i) {
    const int p = (int)(key & 0xffffu), pp = (int)(key >> 16);
#pragma unroll
    for (int t = 0; t < MS; ++t) {
      if (val[t] && col[t] == p) pos[t] = i;
      else if (val[t] && pos[t] == i) pos[t] = pp;
    }
    // local rows of the pivot order from i on: q C + rank >= i
    const int l0 = i > rank ? (i - rank + C - 1) / C : 0;
    const int lr0 = l0 + ((rg - l0) % W.RG + W.RG) % W.RG;
    const T* x = Yl + ldl * p;
#pragma unroll
    for (int t = 0; t < MS; ++t) {
      T a = T(0);
      if (val[t] && pos[t] >= i)
#pragma unroll 4
        for (int r = lr0; r < mloc; r += W.RG) a += x[r] * yc[t][r];
      v[t] = (double)a;
    }
    const double* yrow = gather_sum(v, rank == i % C ? Yl + i / C : nullptr);
#pragma unroll
    for (int t = 0; t < MS; ++t)
      if (own && val[t] && col[t] == p) { sc[0] = v[t]; sc[1] = yrow[p]; }
    __syncthreads();
    if (warp == 0) {
      const T s = (T)sc[0], x0 = (T)sc[1];
      const T normx = qr_norm(s);
      int stop = 0;
      double re = sc[6];
      if (i == 0) {
        re = eps * (double)normx;
        if (normx == T(0)) stop = 2;
      }
      if (!stop && ((double)normx <= re || normx == T(0))) stop = 1;
      const T alpha = x0 >= T(0) ? -normx : normx;
      const T den = s + (x0 >= T(0) ? x0 : -x0) * normx;
      const T c2 = den > T(0) ? T(1) / den : T(0);
      __syncwarp();
      if (lane == 0) {
        sc[2] = (double)alpha;
        sc[3] = (double)(x0 - alpha);
        sc[4] = (double)c2;
        sc[5] = (double)stop;
        if (i == 0) sc[6] = re;
      }
    }
    __syncthreads();
    const int stop = (int)sc[5];
    if (stop) { k = stop == 2 ? 0 : i; break; }
    bool low = false;
    {
      const T alpha = (T)sc[2], v0 = (T)sc[3], c2 = (T)sc[4];
#pragma unroll
      for (int t = 0; t < MS; ++t)
        if (own && val[t]) {
          const bool act = pos[t] > i;
          const T yi = (T)yrow[col[t]];
          const T cj = act ? c2 * ((T)v[t] - alpha * yi) : T(0);
          const T rij = yi - cj * v0;
          coef[col[t]] = cj;
          if (act) {
            if (rank == 0) Rg[i + ldr * col[t]] = rij;
            if (dbits(n1[t]) != 0) {
              const double rd = (double)rij, sn = n1[t] - rd * rd;
              const long long sb = dbits(sn) < 0 ? 0 : dbits(sn);
              if (sb <= dbits(g2[t])) low = true;
              else n1[t] = __longlong_as_double(sb);
            }
          } else if (col[t] == p && rank == 0) {
            Rg[i + ldr * col[t]] = alpha;
          }
        }
    }
    low = __syncthreads_or(low);
    if (i + 1 >= kmax) break;
    const int l1 = i + 1 > rank ? (i + 1 - rank + C - 1) / C : 0;
    const int lr1 = l1 + ((rg - l1) % W.RG + W.RG) % W.RG;
    const T* vc = Yl + ldl * p;
#pragma unroll
    for (int t = 0; t < MS; ++t) {
      double a2 = 0.0;
      if (val[t] && pos[t] > i) {
        const T cj = coef[col[t]];
#pragma unroll 4
        for (int r = lr1; r < mloc; r += W.RG) {
          const T y = yc[t][r] - cj * vc[r];
          yc[t][r] = y;
          if (low) a2 += (double)y * (double)y;
        }
      }
      v[t] = a2;
    }
    if (low) {
      gather_sum(v, nullptr);
#pragma unroll
      for (int t = 0; t < MS; ++t)
        if (own && val[t] && pos[t] > i) { n1[t] = unsign(v[t]); g2[t] = tol3z * v[t]; }
    }
    key = choose(i + 1);       // its barriers also order the update before the next products
  }
  __syncthreads();
#pragma unroll
  for (int t = 0; t < MS; ++t)
    if (own && val[t]) perm[pos[t]] = col[t];
  cl.sync();                   // perm; R in global memory; no CTA still reads another's buffers
  return k;
}

// T = R_1^{-1} R_2 over the cluster's warps: two columns per warp, lanes over the rows, R in global
// memory (column of position b at ldr perm[b]) and, where it fits, R_1 in pool; rinv: k values in
// every CTA.
template <typename T>
__device__ void wide_interp(const WideShape& W, const T* Rg, size_t ldr, int k, const int* perm, T* Tg, size_t ldt, T* rinv,
                            T* pool, size_t room) {
  const int lane = threadIdx.x & 31, e = W.e;
  const bool staged = (size_t)k * k <= room;         // addresses stay below k^2 and k: loads may run ahead
  if (staged)
    for (int b = threadIdx.x >> 5; b < k; b += 8)
      for (int a = lane; a <= b; a += 32) pool[a + k * b] = Rg[a + ldr * perm[b]];
  constexpr int CJ = 2, MK = WIDE_EMAX / 32;
  for (int a = threadIdx.x; a < k; a += blockDim.x) rinv[a] = T(1) / Rg[a + ldr * perm[a]];
  __syncthreads();
  const int nk = (k + 31) / 32;
  for (int j0 = CJ * ((threadIdx.x >> 5) * W.C + W.rank); j0 < e - k; j0 += CJ * 8 * W.C) {
    T s[MK][CJ];
#pragma unroll
    for (int t = 0; t < MK; ++t)
#pragma unroll
      for (int q = 0; q < CJ; ++q) {
        s[t][q] = T(0);
        if (t < nk && lane + 32 * t < k) s[t][q] = Rg[min(lane + 32 * t, k - 1) + ldr * perm[min(k + j0 + q, e - 1)]];
      }
#pragma unroll
    for (int tb = MK - 1; tb >= 0; --tb) {
      if (tb >= nk) continue;
      for (int a = min(32 * tb + 31, k - 1); a >= 32 * tb; --a) {
        const T* ra = staged ? pool + k * a : Rg + ldr * perm[a];
        const T iv = rinv[a];
        T x[CJ];
#pragma unroll
        for (int q = 0; q < CJ; ++q) x[q] = __shfl_sync(0xffffffffu, s[tb][q], a & 31);
#pragma unroll
        for (int t = 0; t <= tb; ++t) {
          const int b = lane + 32 * t;
          if (b < a) {
            const T g = ra[min(b, k - 1)] * iv;
#pragma unroll
            for (int q = 0; q < CJ; ++q) s[t][q] -= g * x[q];
          }
        }
      }
    }
#pragma unroll
    for (int t = 0; t < MK; ++t)
#pragma unroll
      for (int q = 0; q < CJ; ++q)
        if (t < nk && lane + 32 * t < k && j0 + q < e - k)
          Tg[lane + 32 * t + ldt * (j0 + q)] = s[t][q] * rinv[min(lane + 32 * t, k - 1)];
  }
}

// LU with partial pivoting of the n x n block A (global memory, leading dimension lda) by the
// cluster, columns dealt out (column c to CTA c mod C) and held in shared memory: the owner of the
// next pivot column updates it first, finds its pivot and sends the multipliers to all.  Multipliers
// are not interchanged afterwards.  cs: n ceil(n / C) values; mb: 2 (n + 2) doubles.
template <typename T>
__device__ bool wide_lu(cg::cluster_group& cl, const WideShape& W, T* A, size_t lda, int n, int* piv, T* inv, T* cs, double* mb) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, C = W.C, rank = W.rank;
  const int mine = (n - rank + C - 1) / C;
  for (int x = threadIdx.x; x < mine * n; x += blockDim.x) cs[x] = A[x % n + lda * (rank + C * (x / n))];
  cl.sync();                   // cs; every CTA runs, so that its buffers may be written
  bool ok = true;
  // warp 0 of the owner: pivot of column j, multipliers and pivot row to every CTA
  auto prepare = [&](int j) {
    T* c = cs + (size_t)n * (j / C);
    unsigned hi = 0, lo = 0, best = 0xffffffffu;
    for (int r = j + lane; r < n; r += 32) hi = max(hi, abs_hi(c[r]));
    hi = __reduce_max_sync(0xffffffffu, hi);
    for (int r = j + lane; r < n; r += 32)
      if (abs_hi(c[r]) == hi) lo = max(lo, abs_lo(c[r]));
    lo = __reduce_max_sync(0xffffffffu, lo);
    for (int r = j + lane; r < n; r += 32)
      if (abs_hi(c[r]) == hi && abs_lo(c[r]) == lo) best = min(best, (unsigned)r);
    best = __reduce_min_sync(0xffffffffu, best);
    const int p = (int)min(best, (unsigned)(n - 1));
    const T pv = c[p], old = c[j];
    const T iv = (hi | lo) ? T(1) / pv : T(0);
    __syncwarp();
    if (lane == 0) { c[p] = old; c[j] = pv; }
    __syncwarp();
    double* b = mb + (size_t)(j & 1) * (n + 2);
    for (int r = j + 1 + lane; r < n; r += 32) {
      const T l = c[r] * iv;
      c[r] = l;
      for (int q = 0; q < C; ++q) cl.map_shared_rank(b, q)[r] = (double)l;
    }
    if (lane < C) {
      double* pb = cl.map_shared_rank(b, lane);
      pb[n] = (double)p;
      pb[n + 1] = (double)iv;
    }
  };
  if (rank == 0 && warp == 0) prepare(0);
  cl.sync();
  for (int j = 0; j < n; ++j) {
    const double* b = mb + (size_t)(j & 1) * (n + 2);
    const int p = (int)b[n];
    const T iv = (T)b[n + 1];
    if (iv == T(0)) ok = false;
    if (rank == 0 && threadIdx.x == 0) { piv[j] = p; inv[j] = iv; }
    auto column = [&](int c) {
      T* y = cs + (size_t)n * (c / C);
      const T u = y[p], o = y[j];
      __syncwarp();
      for (int r = j + 1 + lane; r < n; r += 32) y[r] = (r == p ? o : y[r]) - (T)b[r] * u;
      __syncwarp();
      if (lane == 0) y[j] = u;
      __syncwarp();
    };
    // the CTA's columns above j, the next pivot column by warp 0 first
    const bool mynext = j + 1 < n && (j + 1) % C == rank;
    const int c0 = j + 1 + ((rank - (j + 1)) % C + C) % C;     // first own column above j
    if (mynext) {
      if (warp == 0) { column(j + 1); prepare(j + 1); }
      else
        for (int c = c0 + C * warp; c < n; c += 7 * C) column(c);
    } else {
      for (int c = c0 + C * warp; c < n; c += 8 * C) column(c);
    }
    cl.sync();
  }
  for (int x = threadIdx.x; x < mine * n; x += blockDim.x) A[x % n + lda * (rank + C * (x / n))] = cs[x];
  return ok;
}

template <typename T>
__global__ void __launch_bounds__(256) sparsify_wide_kernel(LevelDev d) {
  extern __shared__ double sm[];
  __shared__ SegCtx S;
  __shared__ int nearlist[NEAR_MAX];
  __shared__ int nnear_sh, nfar_sh, okf;
  __shared__ double sc[8];
  __shared__ unsigned red[32];
  __shared__ int shi[8];
  pdl_trigger();               // sparsify_kernel, on this level's other segments
  cg::cluster_group cl = cg::this_cluster();
  WideShape W;
  W.C = d.wide;
  W.rank = (int)cl.block_rank();
  const int sid = blockIdx.x / d.wide;
  if (threadIdx.x == 0) seg_context(d, sid, S);
  __syncthreads();
  const int e = S.e, capS = d.capS, rank = W.rank, C = W.C;
  if (!wide_takes(d, S, sizeof(T))) return;          // the whole cluster: sparsify_kernel's
  const bool lead = rank == 0 && threadIdx.x == 0;
  if (lead) atomicMax(d.lstat + LS_EMAX, e);
  if (e == 0) {
    if (lead) { d.kk[sid] = 0; d.hs[sid] = 0; }
    return;
  }
  W.e = e;
  W.NS = (e + 31) / 32;
  W.NSW = min(8, W.NS);
  W.RG = 8 / W.NSW;
  W.EC = 32 * W.NS;
  const size_t ld = d.ldF;
  const T* F1 = static_cast<const T*>(d.F) + (size_t)S.b1 * ld * ld;
  const T* F2 = static_cast<const T*>(d.F) + (size_t)S.b2 * ld * ld;
  T* Dg = static_cast<T*>(d.Dm) + (size_t)sid * capS * capS;
  T* Tg = static_cast<T*>(d.T) + (size_t)sid * capS * capS;
  T* Ykeep = static_cast<T*>(d.Yg) + (size_t)sid * d.Ycap * capS;
  const int halves = d.symmetric ? 1 : 2;
  // shared memory
  char* q = reinterpret_cast<char*>(sm);
  double* xch = reinterpret_cast<double*>(q); q += (size_t)2 * (C + 1) * W.EC * 8;
  double* part = reinterpret_cast<double*>(q); q += (size_t)max(256, W.EC) * 8;
  T* coef = reinterpret_cast<T*>(q); q += (size_t)W.EC * 8;
  T* rinv = reinterpret_cast<T*>(q); q += (size_t)e * sizeof(T);
  int* perm = reinterpret_cast<int*>(q); q += (size_t)e * 4;
  int* piv = reinterpret_cast<int*>(q); q += (size_t)e * 4;
  int* tb_node = reinterpret_cast<int*>(q); q += (size_t)S.nb * 4;
  short* tb_p1 = reinterpret_cast<short*>(q); q += (size_t)S.nb * 2;
  short* tb_p2 = reinterpret_cast<short*>(q); q += (size_t)S.nb * 2;
  unsigned char* tb_nf = reinterpret_cast<unsigned char*>(q); q += S.nb;
  q = reinterpret_cast<char*>(((uintptr_t)q + 15) & ~(uintptr_t)15);
  T* pool = reinterpret_cast<T*>(q);
  const size_t room = ((size_t)d.wide_smem - (size_t)(q - reinterpret_cast<char*>(sm))) / sizeof(T);
  const NbrTab tb{tb_node, tb_p1, tb_p2, tb_nf, true};
  {
    const NbrTab none{nullptr, nullptr, nullptr, nullptr, false};
    for (int f = threadIdx.x; f < S.nb; f += blockDim.x) {
      const Nbr n = nbr_get(d, S, none, f);
      tb_node[f] = n.node;
      tb_p1[f] = (short)n.p1;
      tb_p2[f] = (short)n.p2;
      tb_nf[f] = n.nearf ? 1 : 0;
    }
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    int nn = 0;
    for (int base = 0; base < S.nb; base += 32) {
      const bool isnear = base + lane < S.nb && tb_nf[min(base + lane, S.nb - 1)] != 0;
      const unsigned msk = __ballot_sync(0xffffffffu, isnear);
      const int at = nn + __popc(msk & ((1u << lane) - 1u));
      if (isnear && at < NEAR_MAX) nearlist[at] = base + lane;
      nn += __popc(msk);
    }
    if (lane == 0) {
      if (nn > NEAR_MAX) atomicOr(d.err, ERR_CAPACITY);
      nnear_sh = min(nn, NEAR_MAX);
      nfar_sh = S.nb - nn;
    }
  }
  cl.sync();                   // the lists; every CTA runs, so that its buffers may be written
  const int nnear = nnear_sh, nN = halves * nnear, nF = halves * nfar_sh;
  const int hcap = max(d.h0, 2 * (e + d.p_over)), hmax = min(nF, hcap);
  const bool small = e + d.p_over <= 2 * d.h0;
  int h = min((nF <= d.h0) ? nF : small ? min(hmax, 2 * d.h0) : min(hmax, d.h0), hmax);
  const int nrl = (nN + C - 1) / C;
  auto bget = [&](int t, int f, int c) { return bval_q<T>(d, S, F1, F2, nbr_get(d, S, tb, f), t, c); };
  int k = 0, passes = 0, have = 0;
  unsigned long long work_done = 0;
  while (true) {
    const bool full = h >= nF;
    const int hh = full ? nF : h, m = nN + hh;
    const int mloc = wide_rows(C, nN, hh, full), ldl = mloc | 1;
    T* Yl = pool;
    if (lead && !full) work_done += work::sketch(hh, nF, e);
    for (int x = threadIdx.x; x < ldl * e; x += blockDim.x) Yl[x] = T(0);
    __syncthreads();
    for (int x = threadIdx.x; x < nrl * e; x += blockDim.x) {
      const int a = rank + C * (x % nrl), c = x / nrl;
      if (a < nN) Yl[x % nrl + ldl * c] = bget(a / nnear, nearlist[a % nnear], c);
    }
    if (full) {
      // Phi = I: far row t nfar + j, j the place of the far neighbour among the far ones
      for (int f = threadIdx.x; f < S.nb; f += blockDim.x) {
        int before = 0;
        bool isnear = false;
        for (int a = 0; a < nnear; ++a) {
          if (nearlist[a] < f) ++before;
          if (nearlist[a] == f) isnear = true;
        }
        if (isnear) continue;
        for (int t = 0; t < halves; ++t) {
          const int j = t * nfar_sh + f - before;
          if (j % C == rank)
            for (int c = 0; c < e; ++c) Yl[nrl + j / C + ldl * c] = bget(t, f, c);
        }
      }
    } else {
      // this CTA's groups of four rows: g = rank + C gl; those below `have` were kept
      const int ng = (hh + 3) / 4, ngl = ng > rank ? (ng - rank + C - 1) / C : 0;
      const int kept = have / 4 > rank ? (have / 4 - rank + C - 1) / C : 0, gn = ngl - kept, nr = 4 * gn;
      T* Yr = Yl + nrl + 4 * kept;
      if (gn > 0) {
        const size_t left = room - (size_t)ldl * e;
        const int ch = (int)min((size_t)SK_CHUNK_MAX, left / ((size_t)halves * (e + nr))) & ~(SK_CHUNK - 1);
        const int cw = ch > 0 ? ch : (int)max((size_t)1, min((size_t)SK_CHUNK, left / ((size_t)halves * (e + nr))));
        T* Bc = Yl + (size_t)ldl * e;
        T* Gc = Bc + (size_t)halves * cw * e;
        for (int f0 = 0; f0 < S.nb; f0 += cw) {
          const int nc = min(cw, S.nb - f0), rows = halves * nc;
          for (int x = threadIdx.x; x < nc * e; x += blockDim.x) {
            Bc[x % nc + (size_t)rows * (x / nc)] = bget(0, f0 + x % nc, x / nc);
            if (halves == 2) Bc[nc + x / e + (size_t)rows * (x % e)] = bget(1, f0 + x / e, x % e);
          }
          for (int x = threadIdx.x; x < gn * rows; x += blockDim.x) {
            const int gi = x % gn, row = x / gn, t = row / nc, f = f0 + row % nc;
            float z[4] = {0.f, 0.f, 0.f, 0.f};
            if (!tb_nf[f]) sketch_gauss4(d.seed, d.l, sid, rank + C * (kept + gi), tb_node[f], t, z);
#pragma unroll
            for (int i = 0; i < 4; ++i) Gc[4 * gi + i + (size_t)nr * row] = (T)z[i];
          }
          __syncthreads();
          for (int x = threadIdx.x; x < nr * e; x += blockDim.x) {
            const int rr = x % nr, c = x / nr;
            const T* g = Gc + rr;
            const T* bc = Bc + (size_t)rows * c;
            T y = Yr[rr + ldl * c];
            for (int b0 = 0; b0 < nc; b0 += SK_CHUNK) {
              const int b1 = min(nc, b0 + SK_CHUNK);
              T acc = T(0);
#pragma unroll 4
              for (int row = b0; row < b1; ++row) acc += g[(size_t)nr * row] * bc[row];
              if (halves == 2) {
#pragma unroll 4
                for (int row = nc + b0; row < nc + b1; ++row) acc += g[(size_t)nr * row] * bc[row];
              }
              y += acc;
            }
            Yr[rr + ldl * c] = y;
          }
          __syncthreads();
        }
      }
      // scale; rows past hh are zero; rows that a larger sketch would continue are kept
      const T scl = (T)(1.0 / sqrt((double)hh));
      const bool keep = e > hh - d.p_over;
      for (int x = threadIdx.x; x < 4 * ngl * e; x += blockDim.x) {
        const int lr = x % (4 * ngl), c = x / (4 * ngl), rr = 4 * (rank + C * (lr / 4)) + lr % 4;
        T* y = Yl + nrl + lr + ldl * c;
        T val = lr < 4 * kept ? Ykeep[rr + (size_t)d.Ycap * c] : *y;
        if (rr >= hh) val = T(0);
        if (keep && lr >= 4 * kept && rr < hh) Ykeep[rr + (size_t)d.Ycap * c] = val;
        *y = val * scl;
      }
      if (keep) have = hh & ~3;
    }
    __syncthreads();
    const int kstop = (!full && h < nF) ? max(1, hh - d.p_over + 1) : e;
    k = 0;
    if (m > 0) {
      k = e <= 256 ? wide_qr<T, 1>(cl, W, Yl, ldl, mloc, m, d.eps, kstop, xch, part, coef, perm, Dg, capS, sc, red)
                   : wide_qr<T, 2>(cl, W, Yl, ldl, mloc, m, d.eps, kstop, xch, part, coef, perm, Dg, capS, sc, red);
    } else {
      for (int j = threadIdx.x; j < e; j += blockDim.x) perm[j] = j;
      __syncthreads();
    }
    ++passes;
    if (lead) work_done += work::qr(m, e, k);
    if (!full && k > h - d.p_over && h < nF) {
      h = min(2 * h, hmax);
      continue;
    }
    break;
  }
  const int r = e - k;
  if (k > 0) wide_interp<T>(W, Dg, capS, k, perm, Tg, capS, rinv, pool, room);
  cl.sync();                                          // R is read, T is written
  // ---- transformed diagonal block, in its place in global memory
  const int gt = rank * blockDim.x + threadIdx.x, gs = C * blockDim.x;
  for (int x = gt; x < e * e; x += gs) {
    const int a = x % e, b = x / e, pa = perm[a], pb = perm[b];
    Dg[a + (size_t)capS * b] = F1[(S.s1 + pa) + ld * (S.s1 + pb)] + F2[(S.s2 + pa) + ld * (S.s2 + pb)];
  }
  cl.sync();
  if (k > 0 && r > 0) {
    for (int x = gt; x < e * r; x += gs) {
      const int a = x % e, b = x / e;
      T s = T(0);
#pragma unroll 4
      for (int c = 0; c < k; ++c) s += Dg[a + (size_t)capS * c] * Tg[c + (size_t)capS * b];
      Dg[a + (size_t)capS * (k + b)] -= s;
    }
    cl.sync();
    for (int x = gt; x < r * e; x += gs) {
      const int a = x % r, b = x / r;
      T s = T(0);
#pragma unroll 4
      for (int c = 0; c < k; ++c) s += Tg[c + (size_t)capS * a] * Dg[c + (size_t)capS * b];
      Dg[(k + a) + (size_t)capS * b] -= s;
    }
    cl.sync();
  }
  // ---- remainder
  bool ok = true;
  if (r > 0 && r <= INV_MAX) {
    const int lda = r | 1;
    T* A = pool;
    T* Zt = A + (size_t)r * lda;
    for (int x = threadIdx.x; x < r * r; x += blockDim.x) A[x % r + lda * (x / r)] = Dg[(k + x % r) + (size_t)capS * (k + x / r)];
    __syncthreads();
    ok = r <= 32 ? fast_elim<T, 8, 1>(A, lda, 0, r, piv, rinv, shi, &okf) : fast_elim<T, 8, 2>(A, lda, 0, r, piv, rinv, shi, &okf);
    auto posn = [](int x) { return x; };
    for (int x0 = 32 * rank; x0 < k; x0 += 32 * C) {
      if (r <= 32) panel_chunk<T, 1>(Dg, capS, k, posn, x0, k, r, A, lda, piv, rinv, Zt);
      else panel_chunk<T, 2>(Dg, capS, k, posn, x0, k, r, A, lda, piv, rinv, Zt);
    }
    cl.sync();
    for (int x = gt; x < k * k; x += gs) {
      const int a = x % k, b = x / k;
      T s = T(0);
#pragma unroll 4
      for (int j = 0; j < r; ++j) s += Dg[a + (size_t)capS * (k + j)] * Dg[(k + j) + (size_t)capS * b];
      Dg[a + (size_t)capS * b] -= s;
    }
    if (rank == 0) {
      if (r <= 32) fast_invert<T, 8, 1>(A, lda, r, rinv, Zt);
      else fast_invert<T, 8, 2>(A, lda, r, rinv, Zt);
      for (int x = threadIdx.x; x < r * r; x += blockDim.x) Dg[(k + x % r) + (size_t)capS * (k + x / r)] = Zt[x];
    }
  } else if (r > INV_MAX && k == 0) {
    ok = wide_lu<T>(cl, W, Dg, capS, r, piv, rinv, pool, xch);
  } else if (r > INV_MAX && rank == 0) {
    ok = block_gepp<T>(Dg, capS, k, r, e, piv, rinv, shi, false);
    for (int a = threadIdx.x; a < k; a += blockDim.x)
      for (int j = 0; j < r; ++j) {
        T s = Dg[a + (size_t)capS * (k + j)];
        for (int i2 = 0; i2 < j; ++i2) s -= Dg[a + (size_t)capS * (k + i2)] * Dg[(k + i2) + (size_t)capS * (k + j)];
        Dg[a + (size_t)capS * (k + j)] = s * rinv[j];
      }
    __syncthreads();
    for (int x = threadIdx.x; x < k * k; x += blockDim.x) {
      const int a = x % k, b = x / k;
      T s = T(0);
      for (int j = 0; j < r; ++j) s += Dg[a + (size_t)capS * (k + j)] * Dg[(k + j) + (size_t)capS * b];
      Dg[a + (size_t)capS * b] -= s;
    }
  }
  __syncthreads();
  if (rank != 0) return;
  if (!ok && threadIdx.x == 0) atomicOr(d.err, ERR_SINGULAR);
  for (int j = threadIdx.x; j < e; j += blockDim.x) {
    d.perm[(size_t)sid * capS + j] = perm[j];
    d.snodes[(size_t)sid * capS + j] = d.nodes[(size_t)sid * capS + perm[j]];
  }
  for (int j = threadIdx.x; j < r; j += blockDim.x) {
    d.piv[(size_t)sid * capS + j] = piv[j];
    static_cast<T*>(d.Dinv)[(size_t)sid * capS + j] = rinv[j];
  }
  if (threadIdx.x == 0) {
    d.kk[sid] = k;
    d.hs[sid] = h;
    work_done += work::interp(k, e) + work::apply(e, k) + (r > 0 ? work::elim(r, k) : 0ull);
    atomicAdd(d.lstat + LS_PASSES, passes);
    atomicAdd(d.flops, work_done);
    atomicAdd(d.flops + 2, (unsigned long long)((k * r + e * e) * sizeof(T) + 2 * e * sizeof(int)));
  }
}

// ------------------------------------------------------------ level-L segment tables
__global__ void level_init_L_kernel(LevelDev d) {
  const int nseg = d.g.nseg();
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < nseg * LEAF; x += gridDim.x * blockDim.x) {
    int sid = x / LEAF, t = x % LEAF;
    d.nodes[(size_t)sid * d.capS + t] = d.g.seg_node(sid, t, d.nx);
    if (t == 0) d.cnt[sid] = LEAF;
  }
}

// ------------------------------------------------------------ merge (Sec. 4.3, E_(l))
// Table entry per unknown of the parent's extended block [dP | p]: see MERGE_TABW.
constexpr int TABW = MERGE_TABW;

struct ParentCtx {
  int Ip, Jp, c1, c2, I1, J1, I2, J2, sep, kp;
};

__device__ void parent_ctx(const LevelDev& d, int P, ParentCtx& C) {
  C.Ip = P % d.gp.bx;
  C.Jp = P / d.gp.bx;
  if (d.vcut) { C.I1 = 2 * C.Ip; C.J1 = C.Jp; C.I2 = 2 * C.Ip + 1; C.J2 = C.Jp; }
  else { C.I1 = C.Ip; C.J1 = 2 * C.Jp; C.I2 = C.Ip; C.J2 = 2 * C.Jp + 1; }
  C.c1 = C.I1 + d.g.bx * C.J1;
  C.c2 = C.I2 + d.g.bx * C.J2;
  C.sep = d.g.box_side(C.I1, C.J1, d.vcut ? SIDE_RIGHT : SIDE_TOP);
  C.kp = d.kk[C.sep];
}

// The table is built in two passes: thread 0 lists the runs of entries (a child side's
// skeleton, a junction or corner, the separator skeleton) with their first table index and
// first position in the parent block, then all threads fill the entries.
struct TabRun {
  int kind;            // 0: side of child `child`, 1: corner / junction, 2: separator skeleton
  int n0, cnt, pos;    // first table index, entries, first position in the parent block
  int child, I, J, side;
  int I1, J1, c1, I2, J2, c2;
};
constexpr int TRUN_MAX = 16;

__global__ void merge_table_kernel(LevelDev d) {
  __shared__ TabRun runs[TRUN_MAX];
  __shared__ int nrun_sh, total_sh;
  const int P = blockIdx.x;
  ParentCtx C;
  parent_ctx(d, P, C);
  int* tab = d.ptab + (size_t)P * d.ldFp * TABW;
  const Geo gp = d.gp;
  const int Dp = gp.D();
  if (threadIdx.x == 0) {
    const bool root = gp.bx * gp.by == 1;
    int n = 0, nr = 0;
    auto side_run = [&](int pos, int child, int I, int J, int side) {
      const int sg = d.g.box_side(I, J, side);
      if (sg < 0) return 0;
      TabRun& R = runs[nr++];
      R.kind = 0; R.n0 = n; R.cnt = d.kk[sg]; R.pos = pos; R.child = child; R.I = I; R.J = J; R.side = side;
      n += R.cnt;
      return R.cnt;
    };
    auto corner_run = [&](int pos, int I1, int J1, int c1, int I2, int J2, int c2) {
      const int cid = c1 >= 0 ? d.g.box_corner(I1, J1, c1) : d.g.box_corner(I2, J2, c2);
      if (cid < 0) return 0;
      TabRun& R = runs[nr++];
      R.kind = 1; R.n0 = n; R.cnt = 1; R.pos = pos;
      R.I1 = I1; R.J1 = J1; R.c1 = c1; R.I2 = I2; R.J2 = J2; R.c2 = c2;
      n += 1;
      return 1;
    };
    // sides of P (merged or inherited), then its corners, then the separator skeleton
    for (int side = 0; side < 4 && !root; ++side) {
      if (gp.box_side(C.Ip, C.Jp, side) < 0) continue;
      const int pos = gp.side_pos(side);
      const bool split = d.vcut ? (side == SIDE_BOTTOM || side == SIDE_TOP) : (side == SIDE_LEFT || side == SIDE_RIGHT);
      if (!split) {
        const int child = d.vcut ? (side == SIDE_LEFT ? 1 : 2) : (side == SIDE_BOTTOM ? 1 : 2);
        side_run(pos, child, child == 1 ? C.I1 : C.I2, child == 1 ? C.J1 : C.J2, side);
      } else {
        const int k1 = side_run(pos, 1, C.I1, C.J1, side);
        // junction: vertical cut: bottom -> b1.BR = b2.BL, top -> b1.TR = b2.TL;
        //           horizontal cut: left -> b1.TL = b2.BL, right -> b1.TR = b2.BR
        int jc1, jc2;
        if (d.vcut) { jc1 = side == SIDE_BOTTOM ? C_BR : C_TR; jc2 = side == SIDE_BOTTOM ? C_BL : C_TL; }
        else { jc1 = side == SIDE_LEFT ? C_TL : C_TR; jc2 = side == SIDE_LEFT ? C_BL : C_BR; }
        const int kj = corner_run(pos + k1, C.I1, C.J1, jc1, C.I2, C.J2, jc2);
        side_run(pos + k1 + kj, 2, C.I2, C.J2, side);
      }
    }
    for (int c = 0; c < 4 && !root; ++c) {
      if (gp.box_corner(C.Ip, C.Jp, c) < 0) continue;
      // vertical cut: BL,TL from b1; BR,TR from b2.  horizontal: BL,BR from b1; TL,TR from b2
      const bool from1 = d.vcut ? (c == C_BL || c == C_TL) : (c == C_BL || c == C_BR);
      if (from1) corner_run(gp.corner_pos(c), C.I1, C.J1, c, 0, 0, -1);
      else corner_run(gp.corner_pos(c), 0, 0, -1, C.I2, C.J2, c);
    }
    const int ndP = n;
    {
      TabRun& R = runs[nr++];
      R.kind = 2; R.n0 = n; R.cnt = C.kp; R.pos = Dp;
      n += C.kp;
    }
    nrun_sh = nr;
    total_sh = n;
    d.pcount[2 * P] = ndP;
    d.pcount[2 * P + 1] = C.kp;
    if (C.kp > 0) {
      atomicAdd(d.flops + 1, work::elim(C.kp, ndP));
      const size_t tb = d.fp32 ? sizeof(float) : sizeof(double);
      atomicAdd(d.flops + 3, (unsigned long long)(((size_t)C.kp * C.kp + 2 * (size_t)C.kp * ndP) * tb +
                                                  (size_t)C.kp * sizeof(int)));
    }
    atomicMax(d.lstat + LS_KPMAX, C.kp);
    atomicMax(d.lstat + LS_DPMAX, ndP);
  }
  __syncthreads();
  const int nr = nrun_sh, total = total_sh;
  for (int x = threadIdx.x; x < total; x += blockDim.x) {
    int ri = 0;
    while (ri + 1 < nr && x >= runs[ri + 1].n0) ++ri;
    const TabRun& R = runs[ri];
    const int t = x - R.n0;
    int* e = tab + (size_t)x * TABW;
    if (R.kind == 0) {
      const int sg = d.g.box_side(R.I, R.J, R.side);
      const int q = d.perm[(size_t)sg * d.capS + t];
      const int pc = d.g.side_pos(R.side) + q;
      e[0] = R.pos + t;
      e[1] = e[2] = e[3] = e[4] = e[5] = e[6] = -1;
      e[R.child == 1 ? 1 : 4] = pc;
      e[R.child == 1 ? 2 : 5] = R.side;
      e[R.child == 1 ? 3 : 6] = t;
      e[7] = d.nodes[(size_t)sg * d.capS + q];
    } else if (R.kind == 1) {
      const int cid = R.c1 >= 0 ? d.g.box_corner(R.I1, R.J1, R.c1) : d.g.box_corner(R.I2, R.J2, R.c2);
      e[0] = R.pos;
      e[1] = R.c1 >= 0 ? d.g.corner_pos(R.c1) : -1;
      e[2] = R.c1 >= 0 ? 4 : -1;
      e[3] = 0;
      e[4] = R.c2 >= 0 ? d.g.corner_pos(R.c2) : -1;
      e[5] = R.c2 >= 0 ? 4 : -1;
      e[6] = 0;
      e[7] = d.g.junction_node(cid, d.nx);
    } else {
      // separator skeleton: side RIGHT/TOP of child 1 (owner) = LEFT/BOTTOM of child 2
      const int s1 = d.vcut ? SIDE_RIGHT : SIDE_TOP, s2 = d.vcut ? SIDE_LEFT : SIDE_BOTTOM;
      const int sg = C.sep;
      const int q = d.perm[(size_t)sg * d.capS + t];
      e[0] = Dp + t;
      e[1] = d.g.side_pos(s1) + q; e[2] = s1; e[3] = t;
      e[4] = d.g.side_pos(s2) + q; e[5] = s2; e[6] = t;
      e[7] = d.nodes[(size_t)sg * d.capS + q];
    }
  }
}

// M[a][b] = sum over the children holding both unknowns of the child's block, where the
// block of a segment with itself is its eliminated skeleton block A_ss' (held by the owner
// child: the segment is that child's TOP or RIGHT side) and zero in the other child.
template <typename T>
__global__ void merge_assemble_kernel(LevelDev d) {
  const int P = blockIdx.y;
  const int nM = d.pcount[2 * P] + d.pcount[2 * P + 1];
  const int* tab = d.ptab + (size_t)P * d.ldFp * TABW;
  ParentCtx C;
  parent_ctx(d, P, C);
  const size_t ld = d.ldF, ldp = d.ldFp;
  const T* F1 = static_cast<const T*>(d.F) + (size_t)C.c1 * ld * ld;
  const T* F2 = static_cast<const T*>(d.F) + (size_t)C.c2 * ld * ld;
  const T* Dm = static_cast<const T*>(d.Dm);
  T* M = static_cast<T*>(d.Fp) + (size_t)P * ldp * ldp;
  const long long tot = (long long)nM * nM;
  for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < tot;
       x += (long long)gridDim.x * blockDim.x) {
    int a = (int)(x % nM), b = (int)(x / nM);
    const int* ea = tab + (size_t)a * TABW;
    const int* eb = tab + (size_t)b * TABW;
    T v = T(0);
    for (int ch = 0; ch < 2; ++ch) {
      int pa = ea[1 + 3 * ch], pb = eb[1 + 3 * ch];
      if (pa < 0 || pb < 0) continue;
      int sa = ea[2 + 3 * ch], sb = eb[2 + 3 * ch];
      if (sa == sb && sa < 4) {
        if (sa == SIDE_TOP || sa == SIDE_RIGHT) {
          int I = ch == 0 ? C.I1 : C.I2, J = ch == 0 ? C.J1 : C.J2;
          int sg = d.g.box_side(I, J, sa);
          v += Dm[(size_t)sg * d.capS * d.capS + ea[3 + 3 * ch] + (size_t)d.capS * eb[3 + 3 * ch]];
        }
      } else {
        const T* Fc = ch == 0 ? F1 : F2;
        v += Fc[pa + ld * pb];
      }
    }
    M[ea[0] + ldp * eb[0]] = v;
  }
}

// Separators of more than INV_MAX unknowns: LU of the separator block in global memory with the
// row operations over every column (W = L^{-1} P A_pd), then Z = A_dp U^{-1}; one CTA.
template <typename T>
__device__ void panel_large(const LevelDev& d, T* M, const int* tab, int ndP, int kp, int* piv, T* inv, int* shi) {
  const int nM = ndP + kp, Dp = d.gp.D();
  const size_t ldp = d.ldFp;
  bool ok = true;
  for (int j = 0; j < kp; ++j) {
    const int cj = Dp + j;
    if (threadIdx.x < 32) {
      int lane = threadIdx.x;
      double best = -1.0;
      int bi = kp;
      for (int r = j + lane; r < kp; r += 32) {
        double v = fabs((double)M[(Dp + r) + ldp * cj]);
        if (v > best || (v == best && r < bi)) { best = v; bi = r; }
      }
      for (int o = 16; o > 0; o >>= 1) {
        double ob = __shfl_xor_sync(0xffffffffu, best, o);
        int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
      }
      if (bi >= kp) bi = j;    // only where no entry of the column is a number
      if (lane == 0) { shi[0] = bi; shi[1] = best == 0.0; piv[j] = bi; }
    }
    __syncthreads();
    const int p = shi[0];
    if (shi[1]) { ok = false; if (threadIdx.x == 0) inv[j] = T(0); __syncthreads(); continue; }
    if (p != j) {
      for (int c = threadIdx.x; c < nM; c += blockDim.x) {
        const int pc = tab[(size_t)c * TABW];
        if (pc >= Dp && pc < cj) continue;
        size_t col = ldp * pc;
        T a = M[(Dp + j) + col];
        M[(Dp + j) + col] = M[(Dp + p) + col];
        M[(Dp + p) + col] = a;
      }
      __syncthreads();
    }
    const T ipv = T(1) / M[(Dp + j) + ldp * cj];
    if (threadIdx.x == 0) inv[j] = ipv;
    for (int r = j + 1 + threadIdx.x; r < kp; r += blockDim.x) M[(Dp + r) + ldp * cj] *= ipv;
    __syncthreads();
    const int nr = kp - j - 1;
    // update rows j+1.. over columns: the separator columns j+1..kp-1 and every dP column
    const int ncols = (kp - j - 1) + ndP;
    for (int x = threadIdx.x; x < nr * ncols; x += blockDim.x) {
      int r = j + 1 + x % nr, cc = x / nr;
      int col = cc < kp - j - 1 ? (Dp + j + 1 + cc) : tab[(size_t)(cc - (kp - j - 1)) * TABW];
      M[(Dp + r) + ldp * col] -= M[(Dp + r) + ldp * cj] * M[(Dp + j) + ldp * col];
    }
    __syncthreads();
  }
  if (!ok && threadIdx.x == 0) atomicOr(d.err, ERR_SINGULAR);
  // Z = A_dp U^{-1}: each dP row solved left to right
  for (int a = threadIdx.x; a < ndP; a += blockDim.x) {
    size_t row = tab[(size_t)a * TABW];
    for (int j = 0; j < kp; ++j) {
      T s = M[row + ldp * (Dp + j)];
      for (int i = 0; i < j; ++i) s -= M[row + ldp * (Dp + i)] * M[(Dp + i) + ldp * (Dp + j)];
      M[row + ldp * (Dp + j)] = s * inv[j];
    }
  }
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.aligned;\n" ::: "memory"); }

// Separators of more than INV_MAX unknowns whose factored block fits in shared memory with 32
// boundary rows: shared memory of merge_sides_kernel, and of the LU by a cluster of 8
constexpr int SIDES_MAX = 160;
template <typename T>
__host__ __device__ inline size_t sides_bytes(int kp) {
  const size_t ld = kp | 1;
  return (kp * ld + 32 * ld + kp) * sizeof(T) + 4 * (size_t)kp + 16;
}
template <typename T>
__host__ __device__ inline bool sides_fit(int kp) { return kp <= SIDES_MAX && sides_bytes<T>(kp) <= 216 * 1024; }

// W and Z of those separators, 32 boundary unknowns per CTA: every CTA reads the factored block and
// takes its multipliers through the later interchanges (the stored ones stay where the solve's
// sweeps expect them).  The multiply-adds bound it (kp^2 per boundary unknown), so the boundary
// spreads over as many SMs as it has groups of 32.  One CTA for all (panel_large) / cluster LU and
// this kernel, whole merge: 10 parents, separators up to 140, 8.8 / 0.88 ms; 24, 83, 4.0 / 0.60 ms.
template <typename T>
__global__ void __launch_bounds__(256) merge_sides_kernel(LevelDev d) {
  extern __shared__ double pm_sm[];
  const int P = blockIdx.x;
  const int ndP = d.pcount[2 * P], kp = d.pcount[2 * P + 1];
  if (kp <= INV_MAX || !sides_fit<T>(kp)) return;
  if (32 * (int)blockIdx.y >= ndP) return;
  const int* tab = d.ptab + (size_t)P * d.ldFp * TABW;
  const size_t ldp = d.ldFp;
  T* M = static_cast<T*>(d.Fp) + (size_t)P * ldp * ldp;
  const T* invg = static_cast<const T*>(d.Pinv) + (size_t)P * d.sepcap;
  const int* pivg = d.ppiv + (size_t)P * d.sepcap;
  const int Dp = d.gp.D(), lda = kp | 1;
  T* A = reinterpret_cast<T*>(pm_sm);
  T* Zt = A + (size_t)kp * lda;
  T* inv = Zt + 32 * lda;
  int* q = reinterpret_cast<int*>(inv + kp);
  int* piv = reinterpret_cast<int*>(Zt);             // until the first group
  for (int j = threadIdx.x >> 5; j < kp; j += 8)
    for (int i = threadIdx.x & 31; i < kp; i += 32) A[i + lda * j] = M[(Dp + i) + ldp * (Dp + j)];
  for (int j = threadIdx.x; j < kp; j += blockDim.x) { inv[j] = invg[j]; piv[j] = pivg[j]; }
  __syncthreads();
  if (threadIdx.x < kp) {
    T* c = A + (size_t)lda * threadIdx.x;
    for (int t = threadIdx.x + 1; t < kp; ++t) {
      const int p = piv[t];
      if (p != t) { const T a = c[t]; c[t] = c[p]; c[p] = a; }
    }
  } else if (threadIdx.x == blockDim.x - 1) {
    for (int i = 0; i < kp; ++i) q[i] = i;
    for (int j = 0; j < kp; ++j) { const int p = piv[j], t = q[j]; q[j] = q[p]; q[p] = t; }
  }
  __syncthreads();
  auto posn = [&](int x) { return tab[(size_t)x * TABW]; };
  for (int x0 = 32 * blockIdx.y; x0 < ndP; x0 += 32 * gridDim.y)
    panel_chunk<T, SIDES_MAX / 32>(M, ldp, Dp, posn, x0, ndP, kp, A, lda, q, inv, Zt);
}

// The separator of each parent: LU of its block, W = L^{-1} P A_pd, Z = A_dp U^{-1}, and the block
// replaced by [L~^{-1} \ U^{-1}] for the solve (kp <= INV_MAX).  gridDim.y CTAs (one cluster) share
// a parent: each factors the block for itself (one barrier per pivot, fast_elim) and takes every
// gridDim.y-th group of 32 boundary unknowns, so that on levels of few parents the columns and
// rows spread over SMs; the first writes the inverse, after all have read the block.  What bounds
// it: the kp steps of the three recurrences, about 0.1 us each in FP32 and 0.3 in FP64 (a FP64
// instruction is 64 cycles; four columns share the one that scales U).  Whole merge in FP64 at
// 1023 x 1023, one CTA per parent with the inverses in a kernel of their own and 64 x 64 Schur tiles /
// this and 32 x 32: level 12 1453 / 1190 us, level 9 785 / 611, level 4 327 / 173, level 2 158 / 90.
template <typename T>
__global__ void __launch_bounds__(256) merge_panel_kernel(LevelDev d) {
  extern __shared__ double pm_sm[];
  __shared__ T inv[INV_MAX];
  __shared__ int q[INV_MAX];
  __shared__ int shi[8];
  const int P = blockIdx.x;
  const int ndP = d.pcount[2 * P], kp = d.pcount[2 * P + 1];
  if (kp == 0) return;
  const int* tab = d.ptab + (size_t)P * d.ldFp * TABW;
  const size_t ldp = d.ldFp;
  T* M = static_cast<T*>(d.Fp) + (size_t)P * ldp * ldp;
  T* invg = static_cast<T*>(d.Pinv) + (size_t)P * d.sepcap;
  int* pivg = d.ppiv + (size_t)P * d.sepcap;
  const int Dp = d.gp.D();
  if (kp > INV_MAX) {          // the LU by the cluster, W and Z by merge_sides_kernel, where they fit
    if (sides_fit<T>(kp) && gridDim.y == 8) {
      cg::cluster_group cl = cg::this_cluster();
      WideShape W;
      W.C = (int)gridDim.y;
      W.rank = (int)blockIdx.y;
      double* mb = pm_sm;
      int* piv = reinterpret_cast<int*>(mb + 2 * (kp + 2));
      T* iv = reinterpret_cast<T*>(piv + ((kp + 1) & ~1));
      const bool ok = wide_lu<T>(cl, W, M + Dp + ldp * Dp, ldp, kp, piv, iv, iv + kp, mb);
      __syncthreads();
      if (blockIdx.y == 0) {
        if (!ok && threadIdx.x == 0) atomicOr(d.err, ERR_SINGULAR);
        for (int j = threadIdx.x; j < kp; j += blockDim.x) { invg[j] = iv[j]; pivg[j] = piv[j]; }
      }
    } else if (blockIdx.y == 0) {
      panel_large<T>(d, M, tab, ndP, kp, pivg, invg, shi);
    }
    return;
  }
  const int lda = kp | 1;
  T* A = reinterpret_cast<T*>(pm_sm);
  T* Zt = A + (size_t)kp * lda;
  for (int x = threadIdx.x; x < kp * kp; x += blockDim.x) {
    const int i = x % kp, j = x / kp;
    A[i + lda * j] = M[(Dp + i) + ldp * (Dp + j)];
  }
  __syncthreads();
  cluster_arrive();
  const bool ok = kp <= 32 ? fast_elim<T, 8, 1>(A, lda, 0, kp, q, inv, shi, shi + 6)
                           : fast_elim<T, 8, 2>(A, lda, 0, kp, q, inv, shi, shi + 6);
  for (int x0 = 32 * blockIdx.y; x0 < ndP; x0 += 32 * gridDim.y) {
    auto posn = [&](int x) { return tab[(size_t)x * TABW]; };
    if (kp <= 32) panel_chunk<T, 1>(M, ldp, Dp, posn, x0, ndP, kp, A, lda, q, inv, Zt);
    else panel_chunk<T, 2>(M, ldp, Dp, posn, x0, ndP, kp, A, lda, q, inv, Zt);
  }
  cluster_wait();
  if (blockIdx.y != 0) return;
  if (!ok && threadIdx.x == 0) atomicOr(d.err, ERR_SINGULAR);
  if (kp <= 32) fast_invert<T, 8, 1>(A, lda, kp, inv, Zt);
  else fast_invert<T, 8, 2>(A, lda, kp, inv, Zt);
  for (int x = threadIdx.x; x < kp * kp; x += blockDim.x) M[(Dp + x % kp) + ldp * (Dp + x / kp)] = Zt[x];
  for (int j = threadIdx.x; j < kp; j += blockDim.x) { invg[j] = inv[j]; pivg[j] = q[j]; }
}

// Schur update of the parent's boundary block: M[dP, dP] -= Z W, 32 x 32 tiles of two warps, each
// thread 4 x 4.  In FP64 the multiply-adds bound it (64 cycles per warp instruction whatever its
// lanes), so tiles are no larger than what pads a boundary of 60 - 100 unknowns little, a warp
// whose 16 rows do not exist skips, and the sum runs over kp entries, not over a multiple of 16.
template <typename T>
__global__ void __launch_bounds__(64) merge_schur_kernel(LevelDev d) {
  constexpr int TS = 32;
  __shared__ T Zs[TS][17];
  __shared__ T Ws[16][TS + 1];
  __shared__ int ra[TS], cb[TS];
  const int P = blockIdx.z;
  const int ndP = d.pcount[2 * P], kp = d.pcount[2 * P + 1];
  if (kp == 0) return;
  const int tiles = (ndP + TS - 1) / TS;
  const int* tab = d.ptab + (size_t)P * d.ldFp * TABW;
  const size_t ldp = d.ldFp;
  T* M = static_cast<T*>(d.Fp) + (size_t)P * ldp * ldp;
  const int Dp = d.gp.D();
  const int tx = threadIdx.x % 8, ty = threadIdx.x / 8;   // 8 x 8 threads, 4 x 4 each
  for (int ti = blockIdx.x; ti < tiles; ti += gridDim.x)
    for (int tj = blockIdx.y; tj < tiles; tj += gridDim.y) {
      __syncthreads();
      {
        const int x = threadIdx.x & 31, i = (threadIdx.x < 32 ? ti : tj) * TS + x;
        (threadIdx.x < 32 ? ra : cb)[x] = i < ndP ? tab[(size_t)i * TABW] : -1;
      }
      __syncthreads();
      const bool live = ti * TS + 16 * (threadIdx.x >> 5) < ndP;   // the warp's 16 rows
      T acc[4][4] = {};
      for (int j0 = 0; j0 < kp; j0 += 16) {
        const int nj = min(16, kp - j0);
        for (int x = threadIdx.x; x < TS * 16; x += 64) {
          const int i = x % TS, j = x / TS;
          Zs[i][j] = (ra[i] >= 0 && j < nj) ? M[ra[i] + ldp * (Dp + j0 + j)] : T(0);
          const int jj = x % 16, c = x / 16;
          Ws[jj][c] = (cb[c] >= 0 && jj < nj) ? M[(Dp + j0 + jj) + ldp * cb[c]] : T(0);
        }
        __syncthreads();
        if (live) {
#pragma unroll 4
          for (int j = 0; j < nj; ++j) {
            T z[4], w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) { z[u] = Zs[ty * 4 + u][j]; w[u] = Ws[j][tx * 4 + u]; }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
              for (int v = 0; v < 4; ++v) acc[u][v] += z[u] * w[v];
          }
        }
        __syncthreads();
      }
      if (live) {
#pragma unroll
        for (int v = 0; v < 4; ++v)
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = ty * 4 + u, c = tx * 4 + v;
            if (ra[i] >= 0 && cb[c] >= 0) M[ra[i] + ldp * cb[c]] -= acc[u][v];
          }
      }
    }
}

// The same update on the tensor cores (mixed path, schur_tc): 3xTF32 mma.sync (helpers above).
// 64 x 64 tile per CTA: warp w owns rows 16 (w % 4) .. +16 and columns 32 (w / 4) .. +32
// (four 16 x 8 accumulator tiles).
__global__ void __launch_bounds__(256) merge_schur_tc_kernel(LevelDev d) {
  __shared__ float Zs[64][17];
  __shared__ float Ws[16][65];
  __shared__ int ra[64], cb[64];
  const int P = blockIdx.z;
  const int ndP = d.pcount[2 * P], kp = d.pcount[2 * P + 1];
  if (kp == 0 || ndP == 0) return;
  const int tiles = (ndP + 63) / 64;
  const int ti = blockIdx.x, tj = blockIdx.y;
  if (ti >= tiles || tj >= tiles) return;
  const int* tab = d.ptab + (size_t)P * d.ldFp * TABW;
  const size_t ldp = d.ldFp;
  float* M = static_cast<float*>(d.Fp) + (size_t)P * ldp * ldp;
  const int Dp = d.gp.D();
  for (int x = threadIdx.x; x < 64; x += blockDim.x) {
    int a = ti * 64 + x, b = tj * 64 + x;
    ra[x] = a < ndP ? tab[(size_t)a * TABW] : -1;
    cb[x] = b < ndP ? tab[(size_t)b * TABW] : -1;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, q = lane & 3;
  const int r0 = 16 * (warp & 3), c0 = 32 * (warp >> 2);
  float acc[4][4] = {};
  for (int j0 = 0; j0 < kp; j0 += 16) {
    for (int x = threadIdx.x; x < 64 * 16; x += blockDim.x) {
      int i = x % 64, j = x / 64;
      Zs[i][j] = (ra[i] >= 0 && j0 + j < kp) ? M[ra[i] + ldp * (Dp + j0 + j)] : 0.f;
      Ws[j][i] = (cb[i] >= 0 && j0 + j < kp) ? M[(Dp + j0 + j) + ldp * cb[i]] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) {
      uint32_t ah[4], al[4];
      split_tf32(Zs[r0 + g][8 * ks + q], ah[0], al[0]);
      split_tf32(Zs[r0 + g + 8][8 * ks + q], ah[1], al[1]);
      split_tf32(Zs[r0 + g][8 * ks + q + 4], ah[2], al[2]);
      split_tf32(Zs[r0 + g + 8][8 * ks + q + 4], ah[3], al[3]);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        uint32_t bh[2], bl[2];
        split_tf32(Ws[8 * ks + q][c0 + 8 * t + g], bh[0], bl[0]);
        split_tf32(Ws[8 * ks + q + 4][c0 + 8 * t + g], bh[1], bl[1]);
        mma_tf32(acc[t], al, bh);
        mma_tf32(acc[t], ah, bl);
        mma_tf32(acc[t], ah, bh);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int t = 0; t < 4; ++t)
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = r0 + g + 8 * (u >> 1), c = c0 + 8 * t + 2 * q + (u & 1);
      if (ra[i] >= 0 && cb[c] >= 0) M[ra[i] + ldp * cb[c]] -= acc[t][u];
    }
}

// Level-(l-1) segment tables: counts and grid nodes (merged sides: [skel 1, junction, skel 2]).
__global__ void seg_merge_kernel(LevelDev d) {
  const Geo gp = d.gp, g = d.g;
  const int sidp = blockIdx.x;
  const bool horiz = sidp < gp.nh();
  int Ip, Jp;
  if (horiz) { Ip = sidp % gp.bx; Jp = sidp / gp.bx + 1; }
  else { int t = sidp - gp.nh(); Ip = t % (gp.bx - 1) + 1; Jp = t / (gp.bx - 1); }
  int* out = d.nodes_up + (size_t)sidp * d.capS_up;
  bool split = d.vcut ? horiz : !horiz;
  int cs1, cs2 = -1, jn = -1;
  if (!split) {
    // horizontal cut at level l: hs_p(Ip,Jp) -> hs(Ip, 2Jp); vertical cut: vs_p(Ip,Jp) -> vs(2Ip, Jp)
    if (horiz) cs1 = Ip + g.bx * (2 * Jp - 1);
    else cs1 = g.nh() + (2 * Ip - 1) + (g.bx - 1) * Jp;
  } else if (horiz) {   // vertical cut: hs_p(Ip,Jp) -> hs(2Ip,Jp), c(2Ip+1,Jp), hs(2Ip+1,Jp)
    cs1 = 2 * Ip + g.bx * (Jp - 1);
    cs2 = 2 * Ip + 1 + g.bx * (Jp - 1);
    jn = g.junction_node((2 * Ip + 1 - 1) + (g.bx - 1) * (Jp - 1), d.nx);
  } else {              // horizontal cut: vs_p(Ip,Jp) -> vs(Ip,2Jp), c(Ip,2Jp+1), vs(Ip,2Jp+1)
    cs1 = g.nh() + (Ip - 1) + (g.bx - 1) * (2 * Jp);
    cs2 = g.nh() + (Ip - 1) + (g.bx - 1) * (2 * Jp + 1);
    jn = g.junction_node((Ip - 1) + (g.bx - 1) * (2 * Jp + 1 - 1), d.nx);
  }
  const int k1 = d.kk[cs1];
  for (int t = threadIdx.x; t < k1; t += blockDim.x)
    out[t] = d.nodes[(size_t)cs1 * d.capS + d.perm[(size_t)cs1 * d.capS + t]];
  int n = k1;
  if (cs2 >= 0) {
    if (threadIdx.x == 0) out[n] = jn;
    ++n;
    const int k2 = d.kk[cs2];
    for (int t = threadIdx.x; t < k2; t += blockDim.x)
      out[n + t] = d.nodes[(size_t)cs2 * d.capS + d.perm[(size_t)cs2 * d.capS + t]];
    n += k2;
  }
  if (threadIdx.x == 0) d.cnt_up[sidp] = n;
}

// ------------------------------------------------------------ solve
constexpr int SC = 16;      // right-hand sides per solve pass (register accumulators per thread)
constexpr int DCAP = 512;   // parent boundaries up to this size are staged in shared memory

// out(a, c, acc) for a < nout, c < nc with acc = sum_j A(a, j) v[j + ldv c]: one thread per
// (row, right-hand side) pair, so that short products (a few rows, as in the finest levels)
// still spread over the CTA; v is read from shared memory, A from shared or global memory.
template <typename T, class Row, class Out>
__device__ __forceinline__ void gemv_pairs(int nout, int nin, Row row, size_t sj, const T* v, int ldv, int nc,
                                           Out out) {
  for (int x = threadIdx.x; x < nout * nc; x += blockDim.x) {
    const int a = x % nout, c = x / nout;
    const T* Aa = row(a);   // global or shared memory: plain (generic) loads
    const T* vc = v + (size_t)ldv * c;
    T acc = T(0);
#pragma unroll 4
    for (int j = 0; j < nin; ++j) acc += Aa[j * sj] * vc[j];
    out(a, c, acc);
  }
}

// Triangular sweeps on the SC columns held in shared memory (one warp per column).
template <typename T>
__device__ __forceinline__ void lower_sweep(T* y, int ldy, int n, const T* LU, size_t ldl, const int* pv, int nc) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int c = warp; c < nc; c += nw) {
    T* yy = y + (size_t)ldy * c;
    for (int j = 0; j < n; ++j) {
      const int p = pv[j];
      __syncwarp();
      if (p != j && lane == 0) { T t = yy[j]; yy[j] = yy[p]; yy[p] = t; }
      __syncwarp();
      const T yj = yy[j];
      for (int i = j + 1 + lane; i < n; i += 32) yy[i] -= LU[i + ldl * j] * yj;
    }
    __syncwarp();
  }
}

template <typename T>
__device__ __forceinline__ void upper_sweep(T* y, int ldy, int n, const T* LU, size_t ldl, const T* iv, int nc) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int c = warp; c < nc; c += nw) {
    T* yy = y + (size_t)ldy * c;
    for (int j = n - 1; j >= 0; --j) {
      __syncwarp();
      const T yj = yy[j] * iv[j];
      __syncwarp();
      if (lane == 0) yy[j] = yj;
      for (int i = lane; i < j; i += 32) yy[i] -= LU[i + ldl * j] * yj;
    }
    __syncwarp();
  }
}


// Triangular blocks of order up to INV_MAX are inverted by the factorization, so that the solve
// applies them as one product per right-hand side instead of a sequential sweep: [L\U] becomes
// [L~^{-1}\U^{-1}] with L~ the multipliers after all later interchanges, and the pivot sequence
// becomes the permutation q, (P b)_i = b_{q_i}.
// v[:, c] = L~^{-1} v[q, c] (lower) or U^{-1} v[:, c] (upper) for c < nc, n <= INV_MAX, A the
// inverted block (ld lda) in shared or global memory.  NT threads (the CTA), each holding at
// most INV_MAX x 16 / NT outputs.
template <typename T, bool LOWER, int NT = 256>
__device__ __forceinline__ void tri_apply(T* v, int ldv, int n, const T* A, size_t lda, const int* q, int nc) {
  constexpr int PER = (INV_MAX * 16 + NT - 1) / NT;   // outputs per thread (nc <= 16)
  T acc[PER];
#pragma unroll
  for (int t = 0; t < PER; ++t) {
    const int x = threadIdx.x + NT * t;
    acc[t] = T(0);
    if (x < n * nc) {
      const int i = x % n, c = x / n;
      const T* vc = v + (size_t)ldv * c;
      T s;
      if constexpr (LOWER) {
        s = vc[q[i]];
        for (int k = 0; k < i; ++k) s += A[i + lda * k] * vc[q[k]];
      } else {
        s = T(0);
        for (int k = i; k < n; ++k) s += A[i + lda * k] * vc[k];
      }
      acc[t] = s;
    }
  }
  __syncthreads();
#pragma unroll
  for (int t = 0; t < PER; ++t) {
    const int x = threadIdx.x + NT * t;
    if (x < n * nc) v[(x % n) + (size_t)ldv * (x / n)] = acc[t];
  }
  __syncthreads();
}

template <typename T>
__device__ __forceinline__ void gather_panel(T* dst, int nr, int ncl, const T* src, size_t ldsrc,
                                             const int* rowidx, size_t colbase) {
  // dst[i + nr * j] = src[rowidx(i) + ldsrc * (colbase + j)]; independent loads, coalesced per column
  for (int x = threadIdx.x; x < nr * ncl; x += blockDim.x) {
    const int i = x % nr, j = x / nr;
    dst[x] = src[(size_t)rowidx[i] + ldsrc * (colbase + j)];
  }
}

// The right-hand sides of a launch are split into gridDim.y groups (one CTA per group and
// segment or separator: more CTAs where a level has few segments); this CTA's group becomes
// columns 0 .. nc-1 of X.  False when the group is empty.
template <typename T>
__device__ __forceinline__ bool rhs_group(T*& X, int& nc, const VecLayout& lay) {
  const int per = (nc + (int)gridDim.y - 1) / (int)gridDim.y, c0 = (int)blockIdx.y * per;
  if (c0 >= nc) return false;
  X += (size_t)c0 * (size_t)lay.cs;
  nc = nc - c0 < per ? nc - c0 : per;
  return true;
}

// ---- level solves of segments and separators of at most INV_MAX unknowns.
//
// What bounds them: latency.  A level is two dependent launches per direction, each a chain of a
// gather, two or three short products and a scatter.  So everything the factorization left is
// staged before the wait on the preceding kernel, the products are three barriers apart, results
// go from registers to the solve vector, and a thread holds one row and V right-hand sides (16
// bytes): a multiply-add of the product costs 1/V loads of the matrix entry and one 16-byte load
// of V vector entries instead of two loads each.
template <typename T> struct RhsVec;
template <> struct RhsVec<float> { static constexpr int V = 4; using type = float4; };
template <> struct RhsVec<double> { static constexpr int V = 2; using type = double2; };
__device__ __forceinline__ void axpy(float4& y, float a, const float4& x) {
  y.x += a * x.x; y.y += a * x.y; y.z += a * x.z; y.w += a * x.w;
}
__device__ __forceinline__ void axpy(double2& y, double a, const double2& x) { y.x += a * x.x; y.y += a * x.y; }
__device__ __forceinline__ float4 vzero(float) { return make_float4(0.f, 0.f, 0.f, 0.f); }
__device__ __forceinline__ double2 vzero(double) { return make_double2(0.0, 0.0); }
__device__ __forceinline__ float4 vsub(const float4& a, const float4& b) {
  return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
}
__device__ __forceinline__ double2 vsub(const double2& a, const double2& b) { return make_double2(a.x - b.x, a.y - b.y); }

// The CTA's right-hand sides: of the launch's nc (<= 16), groups of V, gridDim.y CTAs each taking
// as many groups; lg = log2 of the groups rounded up to a power of two.  False: none left.
template <typename T>
__device__ __forceinline__ bool rhs_vec_group(T*& X, int& nc, int& lg, const VecLayout& lay) {
  constexpr int V = RhsVec<T>::V;
  const int tot = (nc + V - 1) / V, per = (tot + (int)gridDim.y - 1) / (int)gridDim.y, g0 = (int)blockIdx.y * per;
  if (g0 >= tot) return false;
  X += (size_t)(g0 * V) * (size_t)lay.cs;
  nc = min(nc - g0 * V, per * V);
  const int g = (nc + V - 1) / V;
  lg = g > 4 ? 3 : g > 2 ? 2 : g > 1 ? 1 : 0;
  return true;
}

// V right-hand sides of one node.  FP32: the chunked vector, whose 16 places per node always exist
// (places past nc are carried along and never read out); FP64: columns, those past nc zero.
__device__ __forceinline__ float4 rhs_load(const float* X, const VecLayout&, int node, int g, int) {
  return reinterpret_cast<const float4*>(X + (size_t)node * 16)[g];
}
__device__ __forceinline__ double2 rhs_load(const double* X, const VecLayout& lay, int node, int g, int nc) {
  double2 v;
  v.x = 2 * g < nc ? X[lay.at(node, 2 * g)] : 0.0;
  v.y = 2 * g + 1 < nc ? X[lay.at(node, 2 * g + 1)] : 0.0;
  return v;
}
__device__ __forceinline__ void rhs_store(float* X, const VecLayout&, int node, int g, int, const float4& v) {
  reinterpret_cast<float4*>(X + (size_t)node * 16)[g] = v;
}
__device__ __forceinline__ void rhs_store(double* X, const VecLayout& lay, int node, int g, int nc, const double2& v) {
  if (2 * g < nc) X[lay.at(node, 2 * g)] = v.x;
  if (2 * g + 1 < nc) X[lay.at(node, 2 * g + 1)] = v.y;
}
__device__ __forceinline__ void rhs_sub_atomic(float* X, const VecLayout&, int node, int g, int, const float4& v) {
  atomicAdd(reinterpret_cast<float4*>(X + (size_t)node * 16) + g, make_float4(-v.x, -v.y, -v.z, -v.w));
}
__device__ __forceinline__ void rhs_sub_atomic(double* X, const VecLayout& lay, int node, int g, int nc, const double2& v) {
  if (2 * g < nc) atomicAdd(X + lay.at(node, 2 * g), -v.x);
  if (2 * g + 1 < nc) atomicAdd(X + lay.at(node, 2 * g + 1), -v.y);
}

// rows x (groups of right-hand sides): node rows into dst (pitch 16 values); FP32 reads a node's
// groups with neighbouring threads, FP64 neighbouring rows of a column
template <typename T, int NT, class Node>
__device__ __forceinline__ void team_gather(const T* X, const VecLayout& lay, int nc, int lg, int n, Node node, T* dst) {
  using Vt = typename RhsVec<T>::type;
  const int tid = threadIdx.x, G = (nc + RhsVec<T>::V - 1) / RhsVec<T>::V;
  if constexpr (sizeof(T) == 4) {
    for (int x = tid; x < n << lg; x += NT) {
      const int a = x >> lg, g = x & ((1 << lg) - 1);
      if (g < G) reinterpret_cast<Vt*>(dst + 16 * a)[g] = rhs_load(X, lay, node(a), g, nc);
    }
  } else {
    for (int g = tid >> 5; g < G; g += NT / 32)
      for (int a = tid & 31; a < n; a += 32) reinterpret_cast<Vt*>(dst + 16 * a)[g] = rhs_load(X, lay, node(a), g, nc);
  }
}

// for every row a < n and group g: acc = sum over j in [j0(a), j1(a)) of A[a + ld j] v[j][g], then out
template <typename T, int NT, class J0, class J1, class Out>
__device__ __forceinline__ void team_product(int n, int nc, int lg, const T* A, int ld, const T* v, J0 j0, J1 j1, Out out) {
  using Vt = typename RhsVec<T>::type;
  const int tid = threadIdx.x, G = (nc + RhsVec<T>::V - 1) / RhsVec<T>::V;
  for (int x = tid; x < n << lg; x += NT) {
    const int a = x >> lg, g = x & ((1 << lg) - 1);
    if (g >= G) continue;
    Vt acc = vzero(T(0));
    const int je = j1(a);
#pragma unroll 4
    for (int j = j0(a); j < je; ++j) axpy(acc, A[a + ld * j], reinterpret_cast<const Vt*>(v + 16 * j)[g]);
    out(a, g, acc);
  }
}

// Shared memory of one segment of up to e unknowns: 2 panels of k r <= (e / 2)^2 values, the r x r
// block, e rows of right-hand sides and r more, e nodes and r permutation entries
__host__ __device__ inline size_t seg_team_bytes(int e, int tb) {
  const size_t pc = (size_t)(e / 2 + 1) * (e / 2 + 1);
  return ((2 * pc + (size_t)e * e + 32 * (size_t)e) * tb + 8 * (size_t)e + 15) / 16 * 16;
}
// ... of one separator of up to kp unknowns with up to nd boundary unknowns: the kp x nd panel (odd
// pitch), the kp x kp block, kp rows of right-hand sides twice, nd rows (backward; and 256 partial
// vectors), kp + 2 nd table entries and kp permutation entries
__host__ __device__ inline size_t sep_team_bytes(int kp, int nd, int tb) {
  return ((size_t)(kp | 1) * nd + (size_t)kp * kp + 32 * (size_t)kp + 16 * (size_t)nd) * tb + 256 * 16 + 4 * (2 * (size_t)kp + 2 * (size_t)nd) + 64;
}

// Forward, per segment: b_r -= T^T b_s; y_r = L^{-1} P b_r; b_s -= Z y_r.
// Backward, per segment: x_r = U^{-1} (y_r - W x_s); x_s -= T x_r.
// What bounds it: the chain of staging, three small products and the scattered stores, in FP64 also the
// pipe.  All level solves of one solve, seg/sep_solve_kernel / these: mixed 1023 x 1023, 16 right-hand
// sides, 634 / 324 us; mixed 255 x 255, 5, 279 / 100 us; FP64 1023 x 1023, 16, 2030 / 1540 us.
template <typename T, int NT>
__global__ void __launch_bounds__(NT) seg_team_kernel(LevelDev d, SolveCaps cap, T* X, int nc, VecLayout lay, int bwd) {
  pdl_trigger();
  extern __shared__ float4 tsm4[];
  const int sid = blockIdx.x, tid = threadIdx.x;
  int lg = 0;
  const bool some = rhs_vec_group(X, nc, lg, lay);
  const int e = some ? d.cnt[sid] : 0, k = some ? d.kk[sid] : 0;
  int r = e - k;
  if (e > cap.vrows) { if (tid == 0) atomicOr(d.err, ERR_CAPACITY); r = 0; }
  if (r == 0) { pdl_wait(); return; }
  const int capS = d.capS;
  T* S = reinterpret_cast<T*>(tsm4);                     // skeleton rows, then remainder rows, pitch 16
  T* R = S + 16 * k;
  T* Yb = S + 16 * e;                                    // the new remainder rows
  T* Ts = Yb + 16 * r;                                   // forward: T^T, rows permuted (r x k); backward: T (k x r)
  T* Ps = Ts + k * r;                                    // forward: Z (k x r); backward: W (r x k)
  T* LU = Ps + k * r;                                    // r x r
  int* nds = reinterpret_cast<int*>(LU + r * r);
  int* q = nds + e;
  const int* snodes = d.snodes + (size_t)sid * capS;     // nodes in [skeleton | remainder] order
  const int* piv = d.piv + (size_t)sid * capS;
  const T* Tm = static_cast<const T*>(d.T) + (size_t)sid * capS * capS;
  const T* Dg = static_cast<const T*>(d.Dm) + (size_t)sid * capS * capS;
  const int lane = tid & 31, w = tid >> 5;
  constexpr int NWT = NT / 32;
  for (int a = tid; a < e; a += NT) nds[a] = snodes[a];
  for (int a = tid; a < r; a += NT) q[a] = piv[a];
  __syncthreads();
  for (int j = w; j < r; j += NWT) {
    for (int i = lane; i < r; i += 32) LU[i + r * j] = Dg[(k + i) + (size_t)capS * (k + j)];
    if (!bwd) {
      const int jq = q[j];
      for (int i = lane; i < k; i += 32) {
        Ts[j + r * i] = Tm[i + (size_t)capS * jq];
        Ps[i + k * j] = Dg[i + (size_t)capS * (k + j)];
      }
    } else {
      for (int i = lane; i < k; i += 32) Ts[i + k * j] = Tm[i + (size_t)capS * j];
    }
  }
  if (bwd)
    for (int j = w; j < k; j += NWT)
      for (int i = lane; i < r; i += 32) Ps[i + r * j] = Dg[(k + i) + (size_t)capS * j];
  pdl_wait();
  using Vt = typename RhsVec<T>::type;
  team_gather<T, NT>(X, lay, nc, lg, e, [&](int a) { return nds[(a < k || bwd) ? a : k + q[a - k]]; }, S);
  __syncthreads();
  auto zero = [](int) { return 0; };
  // remainder rows less their skeleton part (forward in pivot order)
  team_product<T, NT>(r, nc, lg, bwd ? Ps : Ts, r, S, zero, [&](int) { return k; }, [&](int a, int g, const Vt& acc) {
    Vt* v = reinterpret_cast<Vt*>(R + 16 * a) + g;
    *v = vsub(*v, acc);
  });
  __syncthreads();
  // the inverted triangle (forward: unit lower, diagonal not stored)
  team_product<T, NT>(r, nc, lg, LU, r, R, [&](int a) { return bwd ? a : 0; }, [&](int a) { return bwd ? r : a; },
                      [&](int a, int g, Vt acc) {
                        if (!bwd) axpy(acc, T(1), reinterpret_cast<const Vt*>(R + 16 * a)[g]);
                        reinterpret_cast<Vt*>(Yb + 16 * a)[g] = acc;
                        rhs_store(X, lay, nds[k + a], g, nc, acc);
                      });
  if (k == 0) return;
  __syncthreads();
  // skeleton rows less their remainder part
  team_product<T, NT>(k, nc, lg, bwd ? Ts : Ps, k, Yb, zero, [&](int) { return r; }, [&](int a, int g, const Vt& acc) {
    rhs_store(X, lay, nds[a], g, nc, vsub(reinterpret_cast<const Vt*>(S + 16 * a)[g], acc));
  });
}

// Separator of each parent: forward y_p = L^{-1} P b_p, then b_dP -= Z y_p added atomically
// (a boundary unknown is shared by up to four parents; the order of their contributions is
// not fixed; FP32: four right-hand sides per atomic); backward x_p = U^{-1} (y_p - W x_dP), the sum
// over the boundary split over the threads that kp rows leave idle.
template <typename T, int NT>
__global__ void __launch_bounds__(NT) sep_team_kernel(LevelDev d, SolveCaps cap, T* X, int nc, VecLayout lay, int bwd) {
  pdl_trigger();
  extern __shared__ float4 tsm4[];
  using Vt = typename RhsVec<T>::type;
  const int P = blockIdx.x, tid = threadIdx.x;
  int lg = 0;
  const bool some = rhs_vec_group(X, nc, lg, lay);
  const int ndP = d.pcount[2 * P];
  int kp = some ? d.pcount[2 * P + 1] : 0;
  if (kp > cap.yrows || ndP > cap.drows) { if (tid == 0) atomicOr(d.err, ERR_CAPACITY); kp = 0; }
  if (kp == 0) { pdl_wait(); return; }
  const int* tab = d.ptab + (size_t)P * d.ldFp * TABW;
  const size_t ldp = d.ldFp;
  const T* M = static_cast<const T*>(d.Fp) + (size_t)P * ldp * ldp;
  const int Dp = d.gp.D();
  const int* piv = d.ppiv + (size_t)P * d.sepcap;
  Vt* part = reinterpret_cast<Vt*>(tsm4);                // 256 partial vectors (backward)
  T* y = reinterpret_cast<T*>(part + 256);               // kp rows, pitch 16
  T* y2 = y + 16 * kp;
  T* xd = y2 + 16 * kp;                                  // ndP rows (backward)
  T* LU = xd + 16 * ndP;                                 // kp x kp
  const int ldw = kp | 1;
  T* Pn = LU + kp * kp;                                  // forward: Z (ndP x kp); backward: W (kp x ndP, pitch ldw)
  int* pos = reinterpret_cast<int*>(Pn + (size_t)ldw * ndP);
  int* node = pos + ndP;                                 // boundary, then separator
  int* q = node + ndP + kp;
  for (int x = tid; x < ndP + kp; x += NT) {
    if (x < ndP) pos[x] = tab[(size_t)x * TABW];
    node[x] = tab[(size_t)x * TABW + 7];
  }
  for (int a = tid; a < kp; a += NT) q[a] = piv[a];
  __syncthreads();
  const int lane = tid & 31, w = tid >> 5;
  constexpr int NWT = NT / 32;
  for (int j = w; j < kp; j += NWT) {
    for (int i = lane; i < kp; i += 32) LU[i + kp * j] = M[(Dp + i) + ldp * (Dp + j)];
    if (!bwd)
      for (int i = lane; i < ndP; i += 32) Pn[i + ndP * j] = M[pos[i] + ldp * (Dp + j)];
  }
  if (bwd)
    for (int b = w; b < ndP; b += NWT)
      for (int i = lane; i < kp; i += 32) Pn[i + ldw * b] = M[(Dp + i) + ldp * pos[b]];
  pdl_wait();
  team_gather<T, NT>(X, lay, nc, lg, kp, [&](int a) { return node[ndP + (bwd ? a : q[a])]; }, y);
  if (bwd) team_gather<T, NT>(X, lay, nc, lg, ndP, [&](int b) { return node[b]; }, xd);
  __syncthreads();
  auto zero = [](int) { return 0; };
  if (!bwd) {
    team_product<T, NT>(kp, nc, lg, LU, kp, y, zero, [](int a) { return a; }, [&](int a, int g, Vt acc) {
      axpy(acc, T(1), reinterpret_cast<const Vt*>(y + 16 * a)[g]);
      reinterpret_cast<Vt*>(y2 + 16 * a)[g] = acc;
      rhs_store(X, lay, node[ndP + a], g, nc, acc);
    });
    __syncthreads();
    team_product<T, NT>(ndP, nc, lg, Pn, ndP, y2, zero, [&](int) { return kp; }, [&](int b, int g, const Vt& acc) {
      rhs_sub_atomic(X, lay, node[b], g, nc, acc);
    });
  } else {
    // y_p - W x_dP: (kp rows x groups) outputs, each summed by 2^ls threads
    const int G = (nc + RhsVec<T>::V - 1) / RhsVec<T>::V, n = kp << lg;
    int ls = 0;
    while (ls < 4 && (n << (ls + 1)) <= NT) ++ls;
    for (int x0 = 0; x0 < n << ls; x0 += NT) {
      const int x = x0 + tid, o = x >> ls, s = x & ((1 << ls) - 1), a = o >> lg, g = o & ((1 << lg) - 1);
      Vt acc = vzero(T(0));
      if (a < kp && g < G) {
#pragma unroll 4
        for (int b = s; b < ndP; b += 1 << ls) axpy(acc, Pn[a + ldw * b], reinterpret_cast<const Vt*>(xd + 16 * b)[g]);
      }
      part[tid] = acc;
      __syncwarp();
      if (s == 0 && a < kp && g < G) {
        Vt t = reinterpret_cast<const Vt*>(y + 16 * a)[g];
        for (int i = 0; i < 1 << ls; ++i) t = vsub(t, part[tid + i]);
        reinterpret_cast<Vt*>(y + 16 * a)[g] = t;
      }
      __syncwarp();
    }
    __syncthreads();
    team_product<T, NT>(kp, nc, lg, LU, kp, y, [](int a) { return a; }, [&](int) { return kp; }, [&](int a, int g, const Vt& acc) {
      rhs_store(X, lay, node[ndP + a], g, nc, acc);
    });
  }
}

// The same for levels with larger segments or separators.
// Forward, per segment: b_r -= T^T b_s; y_r = L^{-1} P b_r; b_s -= Z y_r.
// Backward, per segment: x_r = U^{-1} (y_r - W x_s); x_s -= T x_r.
template <typename T, int NT>
__global__ void __launch_bounds__(NT, NT == 256 ? 4 : 16) seg_solve_kernel(LevelDev d, SolveCaps cap, T* X, int nc, VecLayout lay, int bwd) {
  pdl_trigger();
  extern __shared__ double smd[];
  if (!rhs_group(X, nc, lay)) { pdl_wait(); return; }
  const int sid = blockIdx.x;
  const int e = d.cnt[sid], k = d.kk[sid], r = e - k;
  if (r == 0 || e == 0) { pdl_wait(); return; }
  if (e > cap.vrows) { if (threadIdx.x == 0) atomicOr(d.err, ERR_CAPACITY); pdl_wait(); return; }
  const int capS = d.capS;
  T* v = reinterpret_cast<T*>(smd);                      // e x SC, [skeleton | remainder]
  T* LUsm = v + (size_t)cap.vrows * SC;                  // r x r LU (when r <= lucap)
  T* Psm = LUsm + (size_t)cap.lucap * cap.lucap;         // two k x r panels (when k r <= pcap)
  T* invs = Psm + 2 * (size_t)cap.pcap;
  int* pivs = reinterpret_cast<int*>(invs + cap.lucap);
  int* nds = pivs + cap.lucap;                           // the segment's nodes (vrows)
  const bool staged = r <= cap.lucap;
  const bool pstaged = (size_t)k * r <= (size_t)cap.pcap;
  const int* snodes = d.snodes + (size_t)sid * capS;     // nodes in [skeleton | remainder] order
  const int* piv = d.piv + (size_t)sid * capS;
  const T* Tm = static_cast<const T*>(d.T) + (size_t)sid * capS * capS;
  const T* Dg = static_cast<const T*>(d.Dm) + (size_t)sid * capS * capS;
  const T* inv = static_cast<const T*>(d.Dinv) + (size_t)sid * capS;
  // factor data first (it overlaps the preceding kernel), the right-hand side after the wait
  if (staged) {
    for (int x = threadIdx.x; x < r * r; x += blockDim.x)
      LUsm[x] = Dg[(k + x % r) + (size_t)capS * (k + x / r)];
    for (int x = threadIdx.x; x < r; x += blockDim.x) { invs[x] = inv[x]; pivs[x] = piv[x]; }
  }
  // panels: T (k x r, ld capS) and Z = D[0:k, k:e] (forward) or W = D[k:e, 0:k] (backward)
  T* Ts = Psm;              // k x r, ld k
  T* Ps = Psm + cap.pcap;   // forward: Z as k x r (ld k); backward: W as r x k (ld r)
  if (pstaged && k > 0) {
    for (int x = threadIdx.x; x < k * r; x += blockDim.x) {
      const int i = x % k, j = x / k;
      Ts[x] = Tm[i + (size_t)capS * j];
      if (!bwd) Ps[x] = Dg[i + (size_t)capS * (k + j)];
    }
    if (bwd)
      for (int x = threadIdx.x; x < r * k; x += blockDim.x) Ps[x] = Dg[(k + x % r) + (size_t)capS * (x / r)];
  }
  for (int a = threadIdx.x; a < e; a += blockDim.x) nds[a] = snodes[a];
  __syncthreads();
  pdl_wait();
  for (int x = threadIdx.x; x < e * nc; x += blockDim.x) {
    int a = x % e, c = x / e;
    v[x] = X[lay.at(nds[a], c)];
  }
  __syncthreads();
  const T* LUs = staged ? LUsm : Dg + k + (size_t)capS * k;
  const size_t ldl = staged ? (size_t)r : (size_t)capS;
  const T* ivs = staged ? invs : inv;
  const int* pvs = staged ? pivs : piv;
  const T* Tp = pstaged ? Ts : Tm;
  const size_t ldt = pstaged ? (size_t)k : (size_t)capS;
  T* vs = v;          // skeleton part
  T* vr = v + k;      // remainder part
  if (!bwd) {
    if (k > 0) {      // b_r -= T^T b_s: row a of T^T is column a of T
      gemv_pairs<T>(r, k, [&](int a) { return Tp + ldt * a; }, 1, vs, e, nc,
                    [&](int a, int c, T acc) { vr[a + e * c] -= acc; });
      __syncthreads();
    }
    if (r <= INV_MAX) tri_apply<T, true, NT>(vr, e, r, LUs, ldl, pvs, nc);
    else lower_sweep<T>(vr, e, r, LUs, ldl, pvs, nc);
    __syncthreads();
    if (k > 0) {      // b_s -= Z y_r
      const T* Zp = pstaged ? Ps : Dg + (size_t)capS * k;
      const size_t ldz = pstaged ? (size_t)k : (size_t)capS;
      gemv_pairs<T>(k, r, [&](int a) { return Zp + a; }, ldz, vr, e, nc,
                    [&](int a, int c, T acc) { vs[a + e * c] -= acc; });
    }
  } else {
    if (k > 0) {      // y_r -= W x_s
      const T* Wp = pstaged ? Ps : Dg + k;
      const size_t ldw = pstaged ? (size_t)r : (size_t)capS;
      gemv_pairs<T>(r, k, [&](int a) { return Wp + a; }, ldw, vs, e, nc,
                    [&](int a, int c, T acc) { vr[a + e * c] -= acc; });
      __syncthreads();
    }
    if (r <= INV_MAX) tri_apply<T, false, NT>(vr, e, r, LUs, ldl, pvs, nc);
    else upper_sweep<T>(vr, e, r, LUs, ldl, ivs, nc);
    __syncthreads();
    if (k > 0) {      // x_s -= T x_r
      gemv_pairs<T>(k, r, [&](int a) { return Tp + a; }, ldt, vr, e, nc,
                    [&](int a, int c, T acc) { vs[a + e * c] -= acc; });
    }
  }
  __syncthreads();
  for (int x = threadIdx.x; x < e * nc; x += blockDim.x) {
    int a = x % e, c = x / e;
    X[lay.at(nds[a], c)] = v[x];
  }
}

// Separator of each parent: forward y_p = L^{-1} P b_p, then b_dP -= Z y_p added atomically
// (a boundary unknown is shared by up to four parents; the order of their contributions is
// not fixed); backward x_p = U^{-1} (y_p - W x_dP).
template <typename T, int NT>
__global__ void __launch_bounds__(NT, NT == 256 ? 4 : 16) sep_solve_kernel(LevelDev d, SolveCaps cap, T* X, int nc, VecLayout lay, int bwd) {
  pdl_trigger();
  extern __shared__ double smd[];
  if (!rhs_group(X, nc, lay)) { pdl_wait(); return; }
  const int P = blockIdx.x;
  const int ndP = d.pcount[2 * P], kp = d.pcount[2 * P + 1];
  if (kp == 0) { pdl_wait(); return; }
  if (kp > cap.yrows) { if (threadIdx.x == 0) atomicOr(d.err, ERR_CAPACITY); pdl_wait(); return; }
  const int* tab = d.ptab + (size_t)P * d.ldFp * TABW;
  const size_t ldp = d.ldFp;
  const T* M = static_cast<const T*>(d.Fp) + (size_t)P * ldp * ldp;
  const T* inv = static_cast<const T*>(d.Pinv) + (size_t)P * d.sepcap;
  const int Dp = d.gp.D();
  const int* piv = d.ppiv + (size_t)P * d.sepcap;
  const int ub = cap.lucap * cap.lucap > cap.qcap ? cap.lucap * cap.lucap : cap.qcap;
  T* y = reinterpret_cast<T*>(smd);                     // kp x SC
  T* U = y + (size_t)cap.yrows * SC;                    // union: LU block / panel
  T* xd = U + ub;                                       // drows x SC (backward)
  T* invs = xd + (size_t)cap.drows * SC;
  int* pivs = reinterpret_cast<int*>(invs + cap.lucap);
  int* rows_sm = pivs + cap.lucap;                      // 2 * drows
  int* ynode = rows_sm + 2 * cap.drows;                 // the separator skeleton's nodes (yrows)
  const bool staged = kp <= cap.lucap;
  const bool dstage = ndP <= cap.drows;
  const int ldw = ndP | 1;                              // odd pitch of the staged W^T panel
  const bool pstaged = dstage && (size_t)ldw * kp <= (size_t)cap.qcap;
  if (dstage) {
    for (int x = threadIdx.x; x < ndP; x += blockDim.x) {
      rows_sm[x] = tab[(size_t)x * TABW];
      rows_sm[cap.drows + x] = tab[(size_t)x * TABW + 7];
    }
  }
  auto rowpos = [&](int a) { return dstage ? rows_sm[a] : tab[(size_t)a * TABW]; };
  auto rownode = [&](int a) { return dstage ? rows_sm[cap.drows + a] : tab[(size_t)a * TABW + 7]; };
  if (staged) for (int x = threadIdx.x; x < kp; x += blockDim.x) { invs[x] = inv[x]; pivs[x] = piv[x]; }
  for (int a = threadIdx.x; a < kp; a += blockDim.x) ynode[a] = tab[(size_t)(ndP + a) * TABW + 7];
  const size_t ldl = staged ? (size_t)kp : ldp;
  const T* ivs = staged ? invs : inv;
  const int* pvs = staged ? pivs : piv;
  auto stage_lu = [&]() {
    if (staged)
      for (int x = threadIdx.x; x < kp * kp; x += blockDim.x) U[x] = M[(Dp + x % kp) + ldp * (Dp + x / kp)];
  };
  // factor data first (it overlaps the preceding kernel): the LU block (forward) or the W^T
  // panel (backward); the solve vector after the wait
  T* Wt = U;                                            // W^T panel, pitch ldw
  if (!bwd) stage_lu();
  else if (pstaged) {
    __syncthreads();                                    // rows_sm
    for (int x = threadIdx.x; x < ndP * kp; x += blockDim.x) {
      const int j = x % kp, b = x / kp;
      Wt[b + (size_t)ldw * j] = M[(Dp + j) + ldp * rows_sm[b]];
    }
  }
  __syncthreads();          // ynode, rows_sm
  pdl_wait();
  for (int x = threadIdx.x; x < kp * nc; x += blockDim.x) {
    int a = x % kp, c = x / kp;
    y[x] = X[lay.at(ynode[a], c)];
  }
  __syncthreads();          // y (and the LU block) are read by other threads below
  if (!bwd) {
    if (kp <= INV_MAX) tri_apply<T, true, NT>(y, kp, kp, staged ? U : M + Dp + ldp * Dp, ldl, pvs, nc);
    else lower_sweep<T>(y, kp, kp, staged ? U : M + Dp + ldp * Dp, ldl, pvs, nc);
    __syncthreads();
    // b_dP -= Z y_p, Z = M[dP rows, separator columns]
    if (pstaged) {
      gather_panel<T>(U, ndP, kp, M, ldp, rows_sm, Dp);
      __syncthreads();
    }
    gemv_pairs<T>(ndP, kp,
                  [&](int a) { return pstaged ? U + a : M + rowpos(a) + ldp * Dp; },
                  pstaged ? (size_t)ndP : ldp, y, kp, nc,
                  [&](int a, int c, T acc) { atomicAdd(X + lay.at(rownode(a), c), -acc); });
  } else {
    if (dstage) {
      for (int x = threadIdx.x; x < ndP * nc; x += blockDim.x) {
        int b = x % ndP, c = x / ndP;
        xd[x] = X[lay.at(rows_sm[cap.drows + b], c)];
      }
    }
    __syncthreads();
    // y_p -= W x_dP, one thread per (row a, right-hand side c)
    for (int x = threadIdx.x; x < kp * nc; x += blockDim.x) {
      const int a = x % kp, c = x / kp;
      T acc = T(0);
      if (pstaged) {
        const T* wa = Wt + (size_t)ldw * a;
        const T* xc = xd + (size_t)ndP * c;
#pragma unroll 4
        for (int b = 0; b < ndP; ++b) acc += wa[b] * xc[b];
      } else if (dstage) {
        const T* xc = xd + (size_t)ndP * c;
        for (int b = 0; b < ndP; ++b) acc += M[(Dp + a) + ldp * rows_sm[b]] * xc[b];
      } else {
        for (int b = 0; b < ndP; ++b) acc += M[(Dp + a) + ldp * rowpos(b)] * X[lay.at(rownode(b), c)];
      }
      y[a + kp * c] -= acc;
    }
    __syncthreads();
    stage_lu();             // the panel is consumed: U takes the LU block
    __syncthreads();
    if (kp <= INV_MAX) tri_apply<T, false, NT>(y, kp, kp, staged ? U : M + Dp + ldp * Dp, ldl, pvs, nc);
    else upper_sweep<T>(y, kp, kp, staged ? U : M + Dp + ldp * Dp, ldl, ivs, nc);
  }
  __syncthreads();
  for (int x = threadIdx.x; x < kp * nc; x += blockDim.x) {
    int a = x % kp, c = x / kp;
    X[lay.at(ynode[a], c)] = y[x];
  }
}


}  // namespace

// Clusters per segment and their shared memory (0: none): FP64, levels of more than 16 unknowns per
// side whose segments leave SMs idle.  Up to 8 CTAs a segment, two per SM at most; one per SM where
// there is room for that, with all of the shared memory, else half of it.  Largest segments by
// wide_bytes at the default h0 and p, without neighbours / with six sides of neighbours: 8 CTAs with
// all of it (up to 19 segments on 152 SMs) 267 / 257 symmetric, 256 / 251 with both halves of B; with
// half of it (up to 38) 171 / 162 and 161 / 155; 4 CTAs (up to 76) 138 / 131 and 128 / 123; 2 (up to
// 152) 99 / 97 and 94 / 91.  A larger segment stays with one CTA.
void sparsify_wide_plan(const LevelPlan& p, LevelDev* d) {
  d->wide = d->wide_smem = 0;
  const int n = p.g.nseg(), sms = sm_count();
  if (d->fp32 || p.capS <= 16 || n == 0) return;
  int C = 8;
  while (C > 1 && n * C > 2 * sms) C /= 2;
  if (C == 1) return;
  d->wide = C;
  d->wide_smem = n * C <= sms ? 216 * 1024 : 108 * 1024;
}

// The sizes below follow the layout of sparsify_kernel.
size_t sparsify_smem_need(int e, int symmetric, int h0, int p_over, int tbytes, int chunk) {
  const size_t halves = symmetric ? 1 : 2;
  const size_t hcap = (size_t)(h0 > 2 * (e + p_over) ? h0 : 2 * (e + p_over));
  const size_t mmax = halves * NEAR_MAX + hcap;
  const size_t un = std::max((size_t)chunk * halves * (e + hcap), (size_t)e * e);
  return sparsify_smem_small(e, tbytes) + (un + (mmax + 1) * e + sparsify_t_values(e)) * tbytes +
         sparsify_smem_stage(e, symmetric, tbytes);
}

// segments of at most 32 unknowns also stage their B block (<= 6 sides of e + 8 corners)
size_t sparsify_smem_stage(int e, int symmetric, int tbytes) {
  const size_t halves = symmetric ? 1 : 2;
  return e <= 32 ? (halves * (6 * (size_t)e + 8) * e + 4) * tbytes : 0;
}

size_t sparsify_smem_min(int e, int symmetric, int h0, int p_over, int tbytes) {
  const size_t halves = symmetric ? 1 : 2;
  const size_t hcap = (size_t)(h0 > 2 * (e + p_over) ? h0 : 2 * (e + p_over));
  return sparsify_smem_small(e, tbytes) + halves * (e + hcap) * tbytes;
}

int sm_count() {
  int dev = 0, v = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
  return v > 0 ? v : 1;
}

size_t sparsify_smem_budget(int fp32, int capS, int ctas) {
  if (ctas < 1) return 0;
  int dev = 0, per_sm = 0, reserved = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
  cudaFuncAttributes fa{};
  cudaError_t e;
  const int threads = (capS <= 16 ? NW_SMALL : NW) * 32;
  if (capS <= 16)
    e = fp32 ? cudaFuncGetAttributes(&fa, sparsify_kernel<float, NW_SMALL>)
             : cudaFuncGetAttributes(&fa, sparsify_kernel<double, NW_SMALL>);
  else
    e = fp32 ? cudaFuncGetAttributes(&fa, sparsify_kernel<float, NW>)
             : cudaFuncGetAttributes(&fa, sparsify_kernel<double, NW>);
  if (e != cudaSuccess) { cudaGetLastError(); return 0; }
  // no more CTAs than the register file holds: shared memory beyond that buys nothing
  const int regs = fa.numRegs > 0 ? fa.numRegs : 64;
  const int by_regs = 65536 / (regs * threads);
  if (by_regs >= 1 && ctas > by_regs) ctas = by_regs;
  const long long share = ((long long)per_sm / ctas) & ~255LL;   // allocation granularity
  const long long dyn = share - reserved - (long long)fa.sharedSizeBytes;
  return dyn > 0 ? (size_t)(dyn & ~255LL) : 0;
}

void launch_level_init_L(const LevelDev& d, cudaStream_t s) {
  int n = d.g.nseg() * LEAF;
  if (n == 0) return;
  note_launch();
  level_init_L_kernel<<<(n + 255) / 256, 256, 0, s>>>(d);
}

template <typename T>
static void sparsify_launch(const LevelDev& d0, const LevelPlan& p, cudaStream_t s) {
  int smem = (int)p.spars_smem;
  LevelDev d = d0;
  // few segments in FP64: a cluster each (the predictor and eps = 0 stay with one CTA)
  if (d.pred_mode != PRED_OFF || d.eps == 0.0) d.wide = 0;
  if (d.use_order && d.g.nseg() > 0) {
    note_launch();
    seg_order_kernel<<<1, 1024, 0, s>>>(d.cnt, d.g.nseg(), d.order);
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 0;
  if constexpr (sizeof(T) == 8) if (d.wide > 1) {
    cfg.gridDim = dim3(d.g.nseg() * d.wide);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = d.wide_smem;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = d.wide;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.numAttrs = 1;
    note_launch();
    cudaLaunchKernelEx(&cfg, smem_allowed<sparsify_wide_kernel<T>>(), d);
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
  }
  cfg.gridDim = dim3(d.g.nseg());
  cfg.dynamicSmemBytes = smem;
  note_launch();
  auto run = [&](auto kernel, int threads) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    cfg.blockDim = dim3(threads);
    cudaLaunchKernelEx(&cfg, kernel, d, smem);
  };
  if (d.capS <= 16) run(smem_allowed<sparsify_kernel<T, NW_SMALL>>(), NW_SMALL * 32);   // two warps each, many segments per SM
  else run(smem_allowed<sparsify_kernel<T, NW>>(), NW * 32);
}

void launch_sparsify(const LevelDev& d, const LevelPlan& p, cudaStream_t s) {
  if (d.g.nseg() == 0) return;
  if (d.fp32) sparsify_launch<float>(d, p, s);
  else sparsify_launch<double>(d, p, s);
}

template <typename T>
static void merge_launch(const LevelDev& d, const LevelPlan& p, cudaStream_t s) {
  const int np = d.gp.nbox();
  note_launch();
  merge_table_kernel<<<np, 128, 0, s>>>(d);
  {
    long long nmax = (long long)p.ldFp;
    int gx = (int)((nmax * nmax + 255) / 256);
    if (gx > 256) gx = 256;
    dim3 grid(gx, np);
    note_launch();
    merge_assemble_kernel<T><<<grid, 256, 0, s>>>(d);
  }
  {
    // the factored block and the larger of its inverse and the 32 boundary rows in work.  At most
    // two parents per SM: a cluster of up to 8 CTAs per parent (more never helps: 256 boundary
    // unknowns), else one
    const size_t kb = (size_t)std::min(p.sepcap, INV_MAX), lda = kb | 1;
    int pm = (int)(sizeof(T) * (kb * lda + std::max(kb * kb, 32 * lda)));
    int cl = 1;
    if (np <= 2 * sm_count())
      while (cl < 8 && 32 * cl < p.ldFp) cl *= 2;
    // larger separators: the cluster's columns of the block, two multiplier buffers, pivots
    const bool sides = cl == 8 && p.sepcap > INV_MAX;
    if (sides) {
      const size_t km = std::min(p.sepcap, SIDES_MAX);
      pm = std::max(pm, (int)(sizeof(T) * (km * ((km + 7) / 8) + km) + 16 * (km + 2) + 4 * (km + 2)));
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(np, cl);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = pm;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = cl;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    note_launch();
    cudaLaunchKernelEx(&cfg, smem_allowed<merge_panel_kernel<T>>(), d);
    if (sides) {
      int ks = std::min(p.sepcap, SIDES_MAX);
      while (!sides_fit<T>(ks)) --ks;
      const int sb = (int)sides_bytes<T>(ks);
      note_launch();
      smem_allowed<merge_sides_kernel<T>>()<<<dim3(np, std::min((p.ldFp + 31) / 32, 48)), 256, sb, s>>>(d);
    }
  }
  note_launch();
  if (d.schur_tc && d.fp32) {
    const int tiles = (p.ldFp + 63) / 64;
    merge_schur_tc_kernel<<<dim3(tiles, tiles, np), 256, 0, s>>>(d);
  } else {
    // tiles by the geometric bound (most are empty at the coarse levels), at most 32 x 32 of them
    const int tiles = std::min((p.ldFp + 31) / 32, 32);
    merge_schur_kernel<T><<<dim3(tiles, tiles, np), 64, 0, s>>>(d);
  }
  if (d.l > 1 && d.gp.nseg() > 0) {
    note_launch();
    seg_merge_kernel<<<d.gp.nseg(), 128, 0, s>>>(d);
  }
}

void launch_merge(const LevelDev& d, const LevelPlan& p, cudaStream_t s) {
  if (d.fp32) merge_launch<float>(d, p, s);
  else merge_launch<double>(d, p, s);
}

bool level_solve_caps(const LevelDev& d, const int* lmax, SolveCaps* out) {
  // lmax: the level counters, LS_EMAX / LS_KPMAX / LS_DPMAX first
  auto mn = [](long long a, long long b) { return a < b ? a : b; };
  auto mx = [](long long a, long long b) { return a > b ? a : b; };
  const long long TB = d.fp32 ? 4 : 8, budget = 200 * 1024;
  SolveCaps sc{};
  sc.vrows = (int)mx(lmax[0], 1);
  sc.yrows = (int)mx(lmax[1], 1);
  sc.drows = (int)mn(lmax[2], DCAP);
  sc.lucap = (int)mn(mx(lmax[0], lmax[1]), RSTAGE);
  long long seg_fixed = 0, sep_fixed = 0;
  for (;;) {
    // segment: v, LU block, reciprocal pivots, pivots (panels come on top)
    seg_fixed = TB * ((long long)sc.vrows * SC + (long long)sc.lucap * sc.lucap + sc.lucap) +
                4LL * (sc.lucap + sc.vrows) + 16;
    // separator: y, xd, reciprocal pivots, pivots, boundary rows (the LU block / panel union on top)
    sep_fixed = TB * ((long long)sc.yrows * SC + (long long)sc.drows * SC + sc.lucap) +
                4LL * (sc.lucap + 2 * sc.drows + sc.yrows) + 16;
    const long long lu = TB * (long long)sc.lucap * sc.lucap;
    if (seg_fixed <= budget && sep_fixed + lu <= budget) break;
    if (sc.lucap > 8) sc.lucap /= 2;
    else if (sc.lucap > 0) sc.lucap = 0;
    else if (sc.drows > 0) sc.drows /= 2;
    else return false;              // the right-hand-side blocks alone exceed the budget
  }
  // a segment panel is k x r <= (e/2)^2; a separator panel |dP| x kp
  sc.pcap = (int)mx(0, mn((long long)(sc.vrows / 2 + 1) * (sc.vrows / 2 + 1), (budget - seg_fixed) / (2 * TB)));
  sc.qcap = (int)mx(0, mn((long long)(sc.drows | 1) * sc.yrows, (budget - sep_fixed) / TB));
  sc.seg_smem = (size_t)(seg_fixed + 2 * TB * sc.pcap);
  // CTA widths before any tuning: 2-warp segment CTAs where segments have at most 32 unknowns
  sc.seg_nt = d.capS <= 32 ? 64 : 256;
  sc.sep_nt = 256;
  // FP64: right-hand sides over more CTAs on levels of few segments or separators (1799 -> 1617 us
  // of level solves at 1023^2 with 16: a CTA's FP64 pipe is the limit there); FP32 stays on one
  // (336 against 343 us)
  sc.seg_split = sc.sep_split = 1;
  if (!d.fp32) {
    while (sc.seg_split < 8 && 2 * sc.seg_split * d.g.nseg() <= sm_count()) sc.seg_split *= 2;
    while (sc.sep_split < 8 && 2 * sc.sep_split * d.gp.nbox() <= sm_count()) sc.sep_split *= 2;
  }
  sc.sep_smem = (size_t)(sep_fixed + TB * mx((long long)sc.lucap * sc.lucap, sc.qcap));
  // the forms for at most INV_MAX unknowns, where all of a segment or separator fits
  sc.seg_team = lmax[0] <= INV_MAX;
  sc.sep_team = lmax[1] <= INV_MAX && lmax[2] <= DCAP &&
                sep_team_bytes(sc.yrows, (int)lmax[2], (int)TB) <= (size_t)budget;
  if (sc.sep_team) sc.drows = (int)lmax[2];
  if (sc.seg_team) {
    // measured (level solves of one solve): FP32 1023^2 with 16 right-hand sides 324 us with two
    // warps per segment, 423 with eight; FP64 1632 and 1542
    sc.seg_nt = d.fp32 ? 64 : 256;
    sc.seg_smem = seg_team_bytes(sc.vrows, (int)TB);
  }
  if (sc.sep_team) sc.sep_smem = sep_team_bytes(sc.yrows, sc.drows, (int)TB);
  *out = sc;
  return true;
}

template <typename T>
static void level_solve(const LevelDev& d, const SolveCaps& sc, T* X, int nrhs, VecLayout lay, int bwd, cudaStream_t s) {
  for (int c0 = 0; c0 < nrhs; c0 += SC) {
    const int nc = nrhs - c0 < SC ? nrhs - c0 : SC;
    T* Xc = X + (size_t)(c0 / SC) * lay.chunk;
    auto go = [&](auto kern, int n, int split, int threads, size_t smem) {
      note_launch();
      launch_pdl(kern, dim3(n, split < nc ? split : nc), dim3(threads), smem, s, d, sc, Xc, nc, lay, bwd);
    };
    auto seg_go = [&]() {
      const int n = d.g.nseg();
      if (n == 0) return;
      if (sc.seg_team) {
        if (sc.seg_nt == 64) go(smem_allowed<seg_team_kernel<T, 64>>(), n, sc.seg_split, 64, sc.seg_smem);
        else go(smem_allowed<seg_team_kernel<T, 256>>(), n, sc.seg_split, 256, sc.seg_smem);
      } else if (sc.seg_nt == 64) {       // 2-warp CTAs: four times as many resident per SM
        go(smem_allowed<seg_solve_kernel<T, 64>>(), n, sc.seg_split, 64, sc.seg_smem);
      } else {
        go(smem_allowed<seg_solve_kernel<T, 256>>(), n, sc.seg_split, 256, sc.seg_smem);
      }
    };
    auto sep_go = [&]() {
      const int n = d.gp.nbox();
      if (sc.sep_team) {
        if (sc.sep_nt == 64) go(smem_allowed<sep_team_kernel<T, 64>>(), n, sc.sep_split, 64, sc.sep_smem);
        else go(smem_allowed<sep_team_kernel<T, 256>>(), n, sc.sep_split, 256, sc.sep_smem);
      } else if (sc.sep_nt == 64) {
        go(smem_allowed<sep_solve_kernel<T, 64>>(), n, sc.sep_split, 64, sc.sep_smem);
      } else {
        go(smem_allowed<sep_solve_kernel<T, 256>>(), n, sc.sep_split, 256, sc.sep_smem);
      }
    };
    if (!bwd) { seg_go(); sep_go(); }
    else { sep_go(); seg_go(); }
  }
}

void launch_level_solve_fwd(const LevelDev& d, const SolveCaps& c, void* X, int nrhs, VecLayout lay, cudaStream_t s) {
  if (d.fp32) level_solve<float>(d, c, static_cast<float*>(X), nrhs, lay, 0, s);
  else level_solve<double>(d, c, static_cast<double*>(X), nrhs, lay, 0, s);
}

void launch_level_solve_bwd(const LevelDev& d, const SolveCaps& c, void* X, int nrhs, VecLayout lay, cudaStream_t s) {
  if (d.fp32) level_solve<float>(d, c, static_cast<float*>(X), nrhs, lay, 1, s);
  else level_solve<double>(d, c, static_cast<double*>(X), nrhs, lay, 1, s);
}

}  // namespace spalu
