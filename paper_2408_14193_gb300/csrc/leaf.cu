// Leaf-interior elimination (Sec. 4.3, first step: L_(L+1)^{-1} A U_(L+1)^{-1} = diag(I, A^(L)))
// and the leaf part of the tree-ordered solve (Eq. (WV)).
//
// The 225 x 225 interior block A_II of a 15 x 15 leaf is banded in the natural in-leaf order
// (x fastest, lower and upper bandwidth 15).  Gaussian elimination with partial pivoting
// (pivot = largest |a_ij| in the column, ties -> lowest row) runs in LAPACK band storage
// (kl = ku = 15, 46 rows incl. the fill of the row interchanges) in FP64: it performs exactly
// the operations of dense partial-pivoting LU on the nonzeros.  The Schur complement
// S_b = A_dI A_II^{-1} A_Id onto the 60 side unknowns needs A_II^{-1} only at the ring of
// interior nodes next to the sides (every side unknown couples to one interior node), so it
// comes from 60 solves with unit right-hand sides.
//
// The LU works on a window of band columns in shared memory (LAPACK band layout); each final
// column leaves it as three 16-value records (L multipliers and pivot offset; reciprocal
// pivot and U above the diagonal; U entries 16..30 that interchanges create), which the sweeps
// stage 16 columns at a time as contiguous runs.
//
// GB300 mapping: FP64 runs at 2 FMA per clock per SM, so every FP64 warp instruction must
// carry 32 useful lanes.  The solves therefore give one thread to one (leaf, right-hand side)
// column and sweep the band with a register window (the interchanges stay inside it); the
// reciprocal pivots are stored once, and the upper sweep runs at the bandwidth the
// interchanges actually produced (15 when there were none).
#include <algorithm>
#include <cstdio>

#include "spalu_internal.h"

namespace spalu {
namespace {

constexpr int KV = KL + KU;   // row of the diagonal in band storage
constexpr int NQ = 4 * LEAF;  // side unknowns of a leaf
constexpr int LPC = 2;        // leaves per CTA of the factor kernel
constexpr int FTH = 128;      // threads of the factor kernel (64 per leaf)
constexpr int QL = 64;        // column slots per leaf in the sweep buffer (60 used by the factor)

__device__ __forceinline__ int leaf_frontal_pos(int vx, int vy, int x0, int y0) {
  const int w = LEAF;
  if (vy == y0 - 1 && vx >= x0 && vx < x0 + w) return vx - x0;                  // bottom
  if (vy == y0 + w && vx >= x0 && vx < x0 + w) return w + vx - x0;              // top
  if (vx == x0 - 1 && vy >= y0 && vy < y0 + w) return 2 * w + vy - y0;          // left
  if (vx == x0 + w && vy >= y0 && vy < y0 + w) return 3 * w + vy - y0;          // right
  if (vx == x0 - 1 && vy == y0 - 1) return 4 * w + C_BL;
  if (vx == x0 + w && vy == y0 - 1) return 4 * w + C_BR;
  if (vx == x0 - 1 && vy == y0 + w) return 4 * w + C_TL;
  if (vx == x0 + w && vy == y0 + w) return 4 * w + C_TR;
  return -1;
}

// side unknown q (0..59: BOTTOM, TOP, LEFT, RIGHT, 15 each): grid node and the local index of
// its interior neighbour
__device__ __forceinline__ void side_unknown(int q, int x0, int y0, int* vx, int* vy, int* m) {
  int s = q / LEAF, t = q % LEAF;
  switch (s) {
    case SIDE_BOTTOM: *vx = x0 + t; *vy = y0 - 1; *m = t; break;
    case SIDE_TOP: *vx = x0 + t; *vy = y0 + LEAF; *m = t + LEAF * (LEAF - 1); break;
    case SIDE_LEFT: *vx = x0 - 1; *vy = y0 + t; *m = LEAF * t; break;
    default: *vx = x0 + LEAF; *vy = y0 + t; *m = LEAF * t + LEAF - 1; break;
  }
}

__device__ __forceinline__ double csr_entry(const int* rowptr, const int* colind, const double* val, int r, int c) {
  for (int p = rowptr[r]; p < rowptr[r + 1]; ++p)
    if (colind[p] == c) return val[p];
  return 0.0;
}

// side unknowns ordered by the position of their interior neighbour (so that the solves of
// one warp can start late: L^{-1} P e_m vanishes above row m - 15)
__constant__ int c_qorder[NQ];
__constant__ int c_qstart[2];   // first sweep step of the two solve warps of a leaf

// Read-only view of one leaf's factor records in precision T (written by an earlier kernel,
// read through the read-only path).
template <typename T>
struct Band {
  const T* __restrict__ lr;     // NI x 16: L(j+1+r, j) at r, pivot offset at 15
  const T* __restrict__ ur;     // NI x 16: 1/U_jj at 0, U(j-r, j) at r <= 15
  const T* __restrict__ ux;     // NI x 16: U(j-r, j) at r - 16 for r >= 16
  __device__ __forceinline__ T l(int r, int j) const { return __ldg(lr + 16 * j + r - 1); }   // L(j+r, j)
  __device__ __forceinline__ T u(int r, int j) const {                                        // U(j-r, j)
    return r < 16 ? __ldg(ur + 16 * j + r) : __ldg(ux + 16 * j + r - 16);
  }
  __device__ __forceinline__ int p(int j) const { return j + (int)__ldg(lr + 16 * j + 15); }
  __device__ __forceinline__ T dinv(int j) const { return __ldg(ur + 16 * j); }
};

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem));
}
// L2 policy for data read once per pass (the factor records of the sweeps): first to be evicted,
// so that the solve vector, written and read back within the pass, stays in L2
__device__ __forceinline__ unsigned long long evict_first_policy() {
  unsigned long long p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(p));
  return p;
}
__device__ __forceinline__ void cp_async16_ef(void* smem, const void* gmem, unsigned long long pol) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem), "l"(pol));
}

// 16 consecutive values of shared memory (16-byte aligned) into registers, 128-bit loads
template <typename T, int N>
__device__ __forceinline__ void lds_vec(const T* p, T (&v)[N]) {
  if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int i = 0; i < N / 4; ++i) {
      const float4 q = reinterpret_cast<const float4*>(p)[i];
      v[4 * i] = q.x; v[4 * i + 1] = q.y; v[4 * i + 2] = q.z; v[4 * i + 3] = q.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
      const double2 q = reinterpret_cast<const double2*>(p)[i];
      v[2 * i] = q.x; v[2 * i + 1] = q.y;
    }
  }
}

// Warp-staged variants of the two sweeps for the leaf Schur kernel: every lane of the warp
// takes part (act = this lane owns a column), the warp starts its forward sweep at the same
// column j0, and the records of the next 16 columns are copied into a double-buffered per-warp
// stage with 16-byte cp.async while the current 16 columns are swept.  A stage holds 16
// records of 16 values: the L records of columns jb..jb+15, or the U records of columns
// NI-1-t0 down to NI-16-t0.  Upper bandwidth <= 15 (no interchange widened U).
template <typename T>
struct WarpStage {
  T* v;      // 2 x 16 x 16, 16-byte aligned
};

template <typename T>
__device__ __forceinline__ void stage_L(const WarpStage<T>& w, int buf, const T* lr, int jb, int lane) {
  constexpr int EPC = 16 / sizeof(T), CPR = 16 / EPC;   // values per chunk, chunks per record
  T* v = w.v + buf * 256;
  for (int x = lane; x < 16 * CPR; x += 32) {
    const int u = x / CPR, k = x % CPR, j = jb + u;
    if (j < NI) cp_async16(v + u * 16 + k * EPC, lr + (size_t)16 * j + k * EPC);
  }
  cp_async_commit();
}

template <typename T>
__device__ __forceinline__ void stage_U(const WarpStage<T>& w, int buf, const T* ur, int t0, int lane) {
  constexpr int EPC = 16 / sizeof(T), CPR = 16 / EPC;
  T* v = w.v + buf * 256;
  for (int x = lane; x < 16 * CPR; x += 32) {
    const int u = x / CPR, k = x % CPR, j = NI - 1 - (t0 + u);
    if (j >= 0) cp_async16(v + u * 16 + k * EPC, ur + (size_t)16 * j + k * EPC);
  }
  cp_async_commit();
}

template <typename T, class In, class Out>
__device__ __forceinline__ void sweep_L_staged(const WarpStage<T>& w, const T* lr, int j0, bool act, In in,
                                               Out out) {
  const int lane = threadIdx.x & 31;
  T W[16];
#pragma unroll
  for (int r = 0; r < 16; ++r) W[r] = (act && j0 + r < NI) ? in(j0 + r) : T(0);
  const int nb = (NI - j0 + 15) / 16;
  stage_L(w, 0, lr, j0, lane);
  for (int blk = 0; blk < nb; ++blk) {
    if (blk + 1 < nb) { stage_L(w, (blk + 1) & 1, lr, j0 + 16 * (blk + 1), lane); cp_async_wait<1>(); }
    else cp_async_wait<0>();
    __syncwarp();
    const T* S = w.v + (blk & 1) * 256;
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      const int j = j0 + 16 * blk + u;
      if (j < NI) {
        T lv[16];
        lds_vec(S + u * 16, lv);
        const int dsw = (int)lv[15];   // the same for the whole warp (one leaf)
        T a = W[u], b = a;
        if (dsw != 0) {
#pragma unroll
          for (int r = 1; r < 16; ++r)
            if (r == dsw) { b = W[(u + r) & 15]; W[(u + r) & 15] = a; }
          W[u] = b;
        }
#pragma unroll
        for (int r = 1; r < 16; ++r) W[(u + r) & 15] -= lv[r - 1] * b;
        if (act) out(j, b);
        W[u] = (act && j + 16 < NI) ? in(j + 16) : T(0);
      }
    }
    __syncwarp();
  }
}

template <typename T, class In, class Out>
__device__ __forceinline__ void sweep_U_staged(const WarpStage<T>& w, const T* ur, bool act, In in, Out out) {
  const int lane = threadIdx.x & 31;
  T V[16];
#pragma unroll
  for (int r = 0; r < 16; ++r) V[r] = act ? in(NI - 1 - r) : T(0);
  const int nb = (NI + 15) / 16;
  stage_U(w, 0, ur, 0, lane);
  for (int blk = 0; blk < nb; ++blk) {
    if (blk + 1 < nb) { stage_U(w, (blk + 1) & 1, ur, 16 * (blk + 1), lane); cp_async_wait<1>(); }
    else cp_async_wait<0>();
    __syncwarp();
    const T* S = w.v + (blk & 1) * 256;
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      const int t = 16 * blk + u;
      if (t < NI) {
        const int j = NI - 1 - t;
        T uv[16];
        lds_vec(S + u * 16, uv);
        const T x = V[u] * uv[0];
        if (act) out(j, x);
#pragma unroll
        for (int r = 1; r < 16; ++r) V[(u + r) & 15] -= uv[r] * x;
        V[u] = (act && j - 16 >= 0) ? in(j - 16) : T(0);
      }
    }
    __syncwarp();
  }
}

// The backward sweep of the leaf Schur kernel in FP32 with the y rows of the next block staged
// too: row j of the warp's 32 columns is one 128-byte run of the sweep buffer (ybw + j QL),
// written by this warp's forward sweep; the refill of step u of block blk reads row j - 16 from
// the stage of block blk + 1 instead of a global load outstanding at the warp barriers.
// Rows below j0 (where this warp's forward sweep started) are zero.
template <typename T, class Out>
__device__ __forceinline__ void sweep_U_staged_y(const WarpStage<T>& w, T* ys, const T* ur, const T* ybw, int j0,
                                                 bool act, Out out) {
  const int lane = threadIdx.x & 31;
  T V[16];
#pragma unroll
  for (int r = 0; r < 16; ++r) V[r] = (act && NI - 1 - r >= j0) ? ybw[(size_t)(NI - 1 - r) * QL + lane] : T(0);
  auto stage_y = [&](int buf, int blk) {   // rows of block blk (no commit: stage_U commits)
    T* Y = ys + buf * 512;
    for (int x = lane; x < 16 * 8; x += 32) {
      const int u = x >> 3, k = x & 7, j = NI - 1 - 16 * blk - u;
      if (j >= j0) cp_async16(Y + u * 32 + 4 * k, ybw + (size_t)j * QL + 4 * k);
    }
  };
  const int nb = (NI + 15) / 16;
  stage_y(0, 1);
  stage_U(w, 0, ur, 0, lane);
  for (int blk = 0; blk < nb; ++blk) {
    if (blk + 1 < nb) {
      stage_y((blk + 1) & 1, blk + 2);
      stage_U(w, (blk + 1) & 1, ur, 16 * (blk + 1), lane);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncwarp();
    const T* S = w.v + (blk & 1) * 256;
    const T* Ys = ys + (blk & 1) * 512 + lane;
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      const int t = 16 * blk + u;
      if (t < NI) {
        const int j = NI - 1 - t;
        T uv[16];
        lds_vec(S + u * 16, uv);
        const T x = V[u] * uv[0];
        if (act) out(j, x);
#pragma unroll
        for (int r = 1; r < 16; ++r) V[(u + r) & 15] -= uv[r] * x;
        V[u] = (act && j - 16 >= j0) ? Ys[u * 32] : T(0);
      }
    }
    __syncwarp();
  }
}

// Forward sweep y = L^{-1} P x for one column held by this thread.  in(j) gives x_j,
// out(j, y) receives y_j for j = j0..NI-1 (x_j = 0 for j < j0 is assumed).
template <typename T, class BandT, class In, class Out>
__device__ __forceinline__ void sweep_L(const BandT& B, int j0, In in, Out out) {
  T W[16];
#pragma unroll
  for (int r = 0; r < 16; ++r) W[r] = (j0 + r < NI) ? in(j0 + r) : T(0);
  for (int t0 = 0; j0 + t0 < NI; t0 += 16) {
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      const int j = j0 + t0 + u;
      if (j < NI) {
        const int dsw = B.p(j) - j;     // 0..15: the interchange stays in the window
        T a = W[u], b = a;
        if (__any_sync(__activemask(), dsw != 0)) {   // skipped when no lane interchanges
#pragma unroll
          for (int r = 1; r < 16; ++r)
            if (r == dsw) { b = W[(u + r) & 15]; W[(u + r) & 15] = a; }
          W[u] = b;
        }
#pragma unroll
        for (int r = 1; r < 16; ++r) W[(u + r) & 15] -= B.l(r, j) * b;
        out(j, b);
        W[u] = (j + 16 < NI) ? in(j + 16) : T(0);
      }
    }
  }
}

// Backward sweep x = U^{-1} y (upper bandwidth < KUW) for one column: in(j) gives y_j,
// out(j, x) receives x_j for j = NI-1 .. 0.
template <typename T, int KUW, class BandT, class In, class Out>
__device__ __forceinline__ void sweep_U(const BandT& B, In in, Out out) {
  T V[KUW];
#pragma unroll
  for (int r = 0; r < KUW; ++r) V[r] = (NI - 1 - r >= 0) ? in(NI - 1 - r) : T(0);
  constexpr int RMAX = KUW - 1 < KV ? KUW - 1 : KV;
  for (int t0 = 0; t0 < NI; t0 += KUW) {
#pragma unroll
    for (int u = 0; u < KUW; ++u) {
      const int t = t0 + u;
      if (t < NI) {
        const int j = NI - 1 - t;
        const T x = V[u] * B.dinv(j);
        out(j, x);
#pragma unroll
        for (int r = 1; r <= RMAX; ++r) V[(u + r) & (KUW - 1)] -= B.u(r, j) * x;
        V[u] = (j - KUW >= 0) ? in(j - KUW) : T(0);
      }
    }
  }
}

// ---- leaf factorization, kernel A: band LU (the dgbtf2 sequence: pivot = largest |entry| of
// the column inside the band, ties -> lowest row; interchanges applied to the columns the U
// factor can reach; multipliers scaled by the reciprocal pivot) of one leaf per CTA, in FP64,
// on a sliding window of WS band columns in shared memory: column c sits in slot c mod WS.
// One barrier per pivot: at step j a half-warp holds a column (lanes over the 15 rows below j) and
// applies interchange and rank-1 update to it; warp 0 takes column j + 1, which it keeps in
// registers, finds its pivot, scales it and leaves it ready for the next step, while the other
// warps finish the columns from j + 3 on.  The last warp also stores column j - 1, final since
// the barrier, and refills its slot with column j + 31 (first touched at step j + 1) from the
// gathered nonzeros (leaf_band5_kernel), loaded a step ahead.
// What bounds it: with few leaves the chain from pivot to pivot (an update, three warp
// reductions, a FP64 reciprocal of about 370 cycles, the scaling); with many the FP64 pipe (18
// instructions of 64 cycles a step, half of them the reciprocal's).
// Also zeroes the leaf's frontal block, where `couple` is set puts the couplings that it owns there
// (the Schur kernel over the band rows subtracts from them), and records the upper bandwidth reached.
constexpr int WS = 32;       // window columns (> KV)

template <typename T>
__device__ __forceinline__ void own_couplings(const LeafDev& d, int b, int tid, T* F) {
  const int nx = d.nx, x0 = (b % d.g.bx) * (LEAF + 1), y0 = (b / d.g.bx) * (LEAF + 1);
  // original couplings owned by this box: its TOP and RIGHT sides (it is their lower /
  // left box) with their end junctions, and the diagonal of its BL junction.
  //   task 0..14 TOP row -> TOP, TL, TR   15..29 RIGHT row -> RIGHT, BR, TR
  //   30 TL row -> TOP   31 TR row -> TOP, RIGHT   32 BR row -> RIGHT   33 BL row -> BL
  if (tid < 2 * LEAF + 4) {
    int vx, vy;
    if (tid < LEAF) { vx = x0 + tid; vy = y0 + LEAF; }
    else if (tid < 2 * LEAF) { vx = x0 + LEAF; vy = y0 + tid - LEAF; }
    else if (tid == 30) { vx = x0 - 1; vy = y0 + LEAF; }
    else if (tid == 31) { vx = x0 + LEAF; vy = y0 + LEAF; }
    else if (tid == 32) { vx = x0 + LEAF; vy = y0 - 1; }
    else { vx = x0 - 1; vy = y0 - 1; }
    if (vx >= 0 && vx < nx && vy >= 0 && vy < d.ny) {
      const int row = vx + nx * vy;
      const int pi = leaf_frontal_pos(vx, vy, x0, y0);
      for (int p = d.rowptr[row]; p < d.rowptr[row + 1]; ++p) {
        int c = d.colind[p];
        int pj = leaf_frontal_pos(c % nx, c / nx, x0, y0);
        if (pj < 0) continue;
        const bool on_top = pj >= LEAF && pj < 2 * LEAF;
        const bool on_right = pj >= 3 * LEAF && pj < 4 * LEAF;
        bool take;
        if (tid < LEAF) take = on_top || pj == 4 * LEAF + C_TL || pj == 4 * LEAF + C_TR;
        else if (tid < 2 * LEAF) take = on_right || pj == 4 * LEAF + C_BR || pj == 4 * LEAF + C_TR;
        else if (tid == 30) take = on_top;
        else if (tid == 31) take = on_top || on_right;
        else if (tid == 32) take = on_right;
        else take = (pj == pi);
        if (take) F[pi + (size_t)d.ldF * pj] += (T)d.val[p];
      }
    }
  }
}

// The leaf matrices' nonzeros by column, gathered from the CSR once for all leaves (one thread
// per leaf, column and stencil offset, every lookup independent), so that the LU's window
// refills read them with plain loads issued a step ahead instead of searching the CSR on the
// critical path of every step.
__global__ void leaf_band5_kernel(LeafDev d) {
  const int nbox = d.g.nbox();
  const long long n = (long long)nbox * NI * 5;
  for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < n; x += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(x % 5), c = (int)((x / 5) % NI), b = (int)(x / (5 * NI));
    const int o = k == 0 ? -LEAF : k == 1 ? -1 : k == 2 ? 0 : k == 3 ? 1 : LEAF;
    const int i = c + o;
    double v = 0.0;
    if (i >= 0 && i < NI && (o == 0 || o == LEAF || o == -LEAF || i / LEAF == c / LEAF)) {
      const int x0 = (b % d.g.bx) * (LEAF + 1), y0 = (b / d.g.bx) * (LEAF + 1);
      v = csr_entry(d.rowptr, d.colind, d.val, (x0 + i % LEAF) + d.nx * (y0 + i / LEAF),
                    (x0 + c % LEAF) + d.nx * (y0 + c / LEAF));
    }
    d.band5[x] = v;
  }
}

template <typename T, int LUW>
__global__ void __launch_bounds__(32 * LUW) leaf_lu_kernel(LeafDev d, int couple) {
  constexpr int LUT = 32 * LUW;
  __shared__ double W[LDAB * WS];
  __shared__ double rps[4];    // of the last pivots: reciprocal, offset, whether zero
  __shared__ int offs[4], zeros[4];
  const int b = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const Geo g = d.g;
  {
    T* F = reinterpret_cast<T*>(d.F) + (size_t)b * d.ldF * d.ldF;
    const int D = g.D();
    for (int e = tid; e < D * D; e += LUT) F[(e % D) + (size_t)d.ldF * (e / D)] = T(0);
  }
  T* lrg = reinterpret_cast<T*>(d.lrec) + (size_t)b * NI * 16;
  T* urg = reinterpret_cast<T*>(d.urec) + (size_t)b * NI * 16;
  T* uxg = reinterpret_cast<T*>(d.uext) + (size_t)b * NI * 16;
  // band row r of column c of A_II: A(c + r - KV, c), nonzero for the five stencil offsets only
  const double* b5 = d.band5 + (size_t)b * NI * 5;
  auto assemble = [&](int r, int c) -> double {
    const int o = r - KV;
    const int k = o == -LEAF ? 0 : o == -1 ? 1 : o == 0 ? 2 : o == 1 ? 3 : o == LEAF ? 4 : -1;
    return (c < NI && k >= 0) ? b5[5 * c + k] : 0.0;
  };
  auto w = [&](int i, int c) -> double& { return W[(KV + i - c) + LDAB * (c & (WS - 1))]; };
  for (int x = tid; x < LDAB * WS; x += LUT) W[x] = assemble(x % LDAB, x / LDAB);
  // pivot of column c: a is its entry in row c + lane (lanes 0 .. 15 of warp 0)
  auto pivot = [&](int c, double a) {
    const int km = min(KL, NI - 1 - c);
    const bool in = lane <= km;
    const unsigned ah = (unsigned)((unsigned long long)__double_as_longlong(a) >> 32) & 0x7fffffffu;
    const unsigned al = (unsigned)(unsigned long long)__double_as_longlong(a);
    const unsigned hi = __reduce_max_sync(0xffffffffu, in ? ah : 0u);
    const unsigned lo = __reduce_max_sync(0xffffffffu, in && ah == hi ? al : 0u);
    const int p = (int)__reduce_min_sync(0xffffffffu, in && ah == hi && al == lo ? (unsigned)lane : 31u) & 15;
    const bool zero = (hi | lo) == 0u;
    const double pv = __shfl_sync(0xffffffffu, a, p), a0 = __shfl_sync(0xffffffffu, a, 0);
    const double rp = zero ? 0.0 : 1.0 / pv;
    const double v = lane == 0 ? pv : lane == p ? a0 : a;
    if (in) w(c + min(lane, km), c) = lane == 0 || zero ? v : v * rp;
    if (lane == 0) { rps[c & 3] = rp; offs[c & 3] = p; zeros[c & 3] = zero ? 1 : 0; }
  };
  // the last warp's rows of a stored or refilled column: lane, lane + 32
  auto stencil = [](int t) {
    const int o = t - KV;
    return o == -LEAF ? 0 : o == -1 ? 1 : o == 0 ? 2 : o == 1 ? 3 : o == LEAF ? 4 : -1;
  };
  const int k0 = stencil(lane), k1 = stencil(lane + 32);
  double n0 = 0.0, n1 = 0.0;   // column j + 31's entries at step j
  auto fetch = [&](int c) {
    const double* q = b5 + 5 * min(c, NI - 1);
    n0 = k0 >= 0 ? q[k0] : 0.0;
    n1 = k1 >= 0 ? q[k1] : 0.0;
  };
  auto store = [&](int c, int t) {
    const T v = (T)W[t + LDAB * (c & (WS - 1))];
    if (t > KV) lrg[16 * c + (t - KV - 1)] = v;                  // L(c+1+r, c), r = t - KV - 1
    else if (t == KV) {
      lrg[16 * c + 15] = (T)offs[c & 3];                         // pivot offset 0..15, exact in T
      urg[16 * c] = (T)rps[c & 3];
      uxg[16 * c + 15] = T(0);
    } else if (t > KV - 16) urg[16 * c + (KV - t)] = v;          // U(c-r, c), r = KV - t <= 15
    else uxg[16 * c + (KV - 16 - t)] = v;                        // U(c-r, c), r = 16..30
  };
  __syncthreads();
  if (warp == 0) pivot(0, w(min(lane, KL), 0));
  if (warp == LUW - 1) fetch(WS);
  __syncthreads();
  int ju = 0, kureach = KU;
  bool ok = true, swapped = false;
  const int r = lane & 15, half = lane >> 4;
  for (int j = 0; j < NI; ++j) {
    const int km = min(KL, NI - 1 - j), jp = offs[j & 3];
    const bool zero = zeros[j & 3] != 0;
    if (zero) ok = false;
    swapped |= jp != 0;
    ju = max(ju, min(j + KU + jp, NI - 1));
    kureach = max(kureach, ju - j);
    // row j + 1 + r (lane 15: only kept, for the pivot of column j + 1)
    const int i = min(j + 1 + r, NI - 1);
    const double m = r < km && !zero ? w(min(i, j + KL), j) : 0.0;
    auto update = [&](int c) {               // column c <= ju; the new entry of row i
      const double a = w(i, c), u = w(j + jp, c), o = w(j, c);
      __syncwarp();
      double v = a;
      if (r < km && !zero) {
        v = (r + 1 == jp ? o : a) - m * u;
        w(i, c) = v;
      }
      if (r == 15) w(j, c) = u;
      return v;
    };
    if (warp == 0) {
      if (j + 1 < NI) {
        const double v = update(min(j + 1 + half, NI - 1));
        __syncwarp();
        pivot(j + 1, v);
      }
    } else {
      if (warp == LUW - 1 && j > 0) {
        store(j - 1, lane);
        if (lane + 32 < LDAB) store(j - 1, lane + 32);
        if (j - 1 + WS < NI) {
          W[lane + LDAB * ((j - 1) & (WS - 1))] = n0;
          if (lane + 32 < LDAB) W[lane + 32 + LDAB * ((j - 1) & (WS - 1))] = n1;
          fetch(j + WS);
        }
        __syncwarp();
      }
      for (int c = j + 3 + 2 * (warp - 1); c <= ju; c += 2 * (LUW - 1)) update(min(c + half, ju));
    }
    __syncthreads();
  }
  if (warp == LUW - 1) {
    store(NI - 1, lane);
    if (lane + 32 < LDAB) store(NI - 1, lane + 32);
  }
  if (couple) own_couplings<T>(d, b, tid, reinterpret_cast<T*>(d.F) + (size_t)b * d.ldF * d.ldF);
  if (!ok && tid == 0) atomicOr(d.err, ERR_SINGULAR);
  if (tid == 0) {
    const int ku = min(kureach, KV);
    d.kur[b] = ku;
    atomicMax(d.kumax, swapped && ku < 16 ? 16 : ku);   // <= 15: no leaf made an interchange
  }
}

// ---- leaf factorization, kernel B: the Schur complement onto the sides from the ring of
// A_II^{-1} (one thread per side unknown q: a band solve with the unit vector of its interior
// neighbour, the factor read from global memory), then the original couplings this box owns.
// Two leaves per 128-thread CTA.
template <typename T>
__global__ void __launch_bounds__(FTH) leaf_schur_kernel(LeafDev d) {
  __shared__ double qa[LPC][NQ], qc[LPC][NQ];
  __shared__ int qm[LPC][NQ], qex[LPC][NQ];
  const int sub = threadIdx.x / 64;
  const int tid = threadIdx.x % 64;
  const int b = blockIdx.x * LPC + sub;
  const int nbox = d.g.nbox();
  const bool live = b < nbox;
  const Geo g = d.g;
  const int I = live ? b % g.bx : 0, J = live ? b / g.bx : 0;
  const int x0 = I * (LEAF + 1), y0 = J * (LEAF + 1);
  const int nx = d.nx;
  T* F = reinterpret_cast<T*>(d.F) + (size_t)(live ? b : 0) * d.ldF * d.ldF;
  if (live) {
    for (int q = tid; q < NQ; q += 64) {
      int vx, vy, m;
      side_unknown(q, x0, y0, &vx, &vy, &m);
      const bool exists = vx >= 0 && vx < nx && vy >= 0 && vy < d.ny;
      qm[sub][q] = m;
      qex[sub][q] = exists ? 1 : 0;
      double a = 0.0, c = 0.0;
      if (exists) {
        const int node = vx + nx * vy;
        const int mnode = (x0 + m % LEAF) + nx * (y0 + m / LEAF);
        a = csr_entry(d.rowptr, d.colind, d.val, node, mnode);
        c = csr_entry(d.rowptr, d.colind, d.val, mnode, node);
      }
      qa[sub][q] = a;
      qc[sub][q] = c;
      reinterpret_cast<T*>(d.cpl)[(size_t)b * NQ + q] = (T)c;   // A(m, side unknown q), 0 outside the grid
    }
  }
  __syncthreads();
  __shared__ __align__(16) T stv[FTH / 32][512];
  __shared__ __align__(16) T sty[FTH / 32][sizeof(T) == 4 ? 1024 : 4];   // FP32: y rows of the U sweep
  if (live && d.kur[b] <= 15) {     // warp-staged sweeps (all lanes; lanes >= NQ only stage)
    const bool act = tid < NQ;
    const int q = act ? c_qorder[tid] : 0;
    const int j0 = c_qstart[tid >> 5];
    const WarpStage<T> ws{stv[threadIdx.x >> 5]};
    const T* lr = reinterpret_cast<const T*>(d.lrec) + (size_t)b * NI * 16;
    const T* ur = reinterpret_cast<const T*>(d.urec) + (size_t)b * NI * 16;
    T* yb = reinterpret_cast<T*>(d.ybuf) + (size_t)b * NI * QL;
    T* Gb = d.G ? reinterpret_cast<T*>(d.G) + (size_t)b * NI * NQ : nullptr;
    const int mq = act ? qm[sub][q] : -1;
    const T cq = (act && qex[sub][q]) ? (T)qc[sub][q] : T(0);
    sweep_L_staged<T>(ws, lr, j0, act, [&](int j) { return j == mq ? cq : T(0); },
                      [&](int j, T y) { yb[(size_t)j * QL + tid] = y; });
    const size_t ldF = d.ldF;
    auto yin = [&](int j) { return j < j0 ? T(0) : yb[(size_t)j * QL + tid]; };
    auto ring_out = [&](int j, T x) {
      if (Gb) Gb[(size_t)j * NQ + q] = x;                   // column q of A_II^{-1} A_Id
      const int lx = j % LEAF, ly = j / LEAF;
      if (ly == 0 && qex[sub][lx]) F[lx + ldF * q] = -(T)qa[sub][lx] * x;
      if (ly == LEAF - 1 && qex[sub][LEAF + lx]) F[(LEAF + lx) + ldF * q] = -(T)qa[sub][LEAF + lx] * x;
      if (lx == 0 && qex[sub][2 * LEAF + ly]) F[(2 * LEAF + ly) + ldF * q] = -(T)qa[sub][2 * LEAF + ly] * x;
      if (lx == LEAF - 1 && qex[sub][3 * LEAF + ly]) F[(3 * LEAF + ly) + ldF * q] = -(T)qa[sub][3 * LEAF + ly] * x;
    };
    if constexpr (sizeof(T) == 4)
      sweep_U_staged_y<T>(ws, sty[threadIdx.x >> 5], ur, yb + 32 * (tid >> 5), j0, act, ring_out);
    else
      sweep_U_staged<T>(ws, ur, act, yin, ring_out);
  } else if (live && tid < NQ) {    // widened U: sweeps reading the band from global memory
    const int q = c_qorder[tid];
    const int j0 = c_qstart[tid >> 5];
    Band<T> Bd{reinterpret_cast<const T*>(d.lrec) + (size_t)b * NI * 16,
               reinterpret_cast<const T*>(d.urec) + (size_t)b * NI * 16,
               reinterpret_cast<const T*>(d.uext) + (size_t)b * NI * 16};
    T* yb = reinterpret_cast<T*>(d.ybuf) + (size_t)b * NI * QL;
    T* Gb = d.G ? reinterpret_cast<T*>(d.G) + (size_t)b * NI * NQ : nullptr;
    const int mq = qm[sub][q];
    const T cq = qex[sub][q] ? (T)qc[sub][q] : T(0);
    sweep_L<T>(Bd, j0, [&](int j) { return j == mq ? cq : T(0); },
               [&](int j, T y) { yb[(size_t)j * QL + tid] = y; });
    const size_t ldF = d.ldF;
    auto yin = [&](int j) { return j < j0 ? T(0) : yb[(size_t)j * QL + tid]; };
    auto ring_out = [&](int j, T x) {
      if (Gb) Gb[(size_t)j * NQ + q] = x;                   // column q of A_II^{-1} A_Id
      const int lx = j % LEAF, ly = j / LEAF;
      if (ly == 0 && qex[sub][lx]) F[lx + ldF * q] = -(T)qa[sub][lx] * x;
      if (ly == LEAF - 1 && qex[sub][LEAF + lx]) F[(LEAF + lx) + ldF * q] = -(T)qa[sub][LEAF + lx] * x;
      if (lx == 0 && qex[sub][2 * LEAF + ly]) F[(2 * LEAF + ly) + ldF * q] = -(T)qa[sub][2 * LEAF + ly] * x;
      if (lx == LEAF - 1 && qex[sub][3 * LEAF + ly]) F[(3 * LEAF + ly) + ldF * q] = -(T)qa[sub][3 * LEAF + ly] * x;
    };
    sweep_U<T, 32>(Bd, yin, ring_out);
  }
  __syncthreads();
  const bool active = live;
  if (active) own_couplings<T>(d, b, tid, F);
}

// ---------------------------------------------------------------- solve
// One thread per (leaf, right-hand side).  Forward (leaf part of W~): X[I] <- A_II^{-1} X[I];
// the side unknowns are updated afterwards by sep_update_fwd_kernel.  Backward (leaf part of
// V~): X[I] <- X[I] - A_II^{-1} (A_Id x_d).
constexpr int SLOT = 16;   // right-hand-side slots per leaf and launch
constexpr int SWPB = 4;    // warps per CTA of the solve sweeps (two leaves per warp)

// Per-warp shared-memory stage of leaf_solve_kernel (values of T).  L phase, two buffers of:
// for each of the warp's two leaves 16 L records and (FP32 forward) the right-hand-side rows
// of the next block; backward also the leaves' 60 side values x_d and coupling coefficients.
// U phase, two buffers of: KUW columns of KUW values (the U record, and for KUW = 32 its
// extension) and (FP32) the KUW rows y of the next block and (FP32 backward) the KUW rows of x
// this block updates.  Rows hold 16 values (the right-hand sides); the pads put the two
// leaves of a warp on different banks.
template <typename T, int KUW, bool bwd>
struct SolveStage {
  static constexpr int EPC = 16 / (int)sizeof(T);      // values per 16-byte chunk
  static constexpr int CPR = SLOT / EPC;                // chunks per 16-value record
  static constexpr bool CHKV = sizeof(T) == 4;          // FP32: the chunked solve vector
  static constexpr bool XPF = !bwd && CHKV;
  static constexpr bool YPF = CHKV;
  static constexpr bool XOPF = bwd && CHKV;
  static constexpr int LSTP = SLOT * SLOT + EPC;
  static constexpr int USTP = KUW * KUW + EPC;
  static constexpr int XSTP = SLOT * SLOT + 16;
  static constexpr int YSTP = KUW * SLOT + 16;
  static constexpr int XDSTP = NQ * SLOT + 16;
  static constexpr int bufL = 2 * (LSTP + (XPF ? XSTP : 0));
  static constexpr int bufU = 2 * (USTP + (YPF ? YSTP : 0) + (XOPF ? YSTP : 0));
  static constexpr int xdsz = bwd ? 2 * XDSTP + 2 * 64 : 0;
  static constexpr int warpsz = 2 * bufL + xdsz > 2 * bufU ? 2 * bufL + xdsz : 2 * bufU;
  static constexpr size_t bytes = (size_t)SWPB * warpsz * sizeof(T);
};

// Band sweeps, one warp per two leaves x 16 right-hand sides, thread (leaf, rhs): forward
// x_I = U^{-1} L^{-1} P b_I; backward x_I -= U^{-1} L^{-1} P (A_Id x_d).
// - Warp-synchronous: a warp stages the factor records of its own two leaves for the next
//   block of 16 (L) or KUW (U) steps with 16-byte cp.async (L2 evict-first: read once per
//   pass) into its double-buffered stage while it sweeps the current block; no CTA barrier.
// - Forward: y = L^{-1} P b overwrites b in the solve vector (row j is written at step j,
//   after the last read of b_j) and the U sweep reads it back from there, so the intermediate
//   costs no scratch traffic and stays in L2 between the sweeps.  Backward: x_I is needed
//   until the last step, so y goes through the sweep buffer.
// - Backward input: (A_Id x_d)_j is nonzero on the leaf's boundary rows only, one term per
//   side the node touches: the coupling coefficient (stored by the factorization) times the
//   side value, both staged once per warp.
// - FP32: the solve vector is chunked (a node's 16 right-hand sides are one 64-byte run); the
//   right-hand-side rows of the next L block, the y rows of the next U block and (backward)
//   the rows a U block updates are staged with the records, so no global load is
//   outstanding at a warp barrier.  FP64 reads them directly.
// - KUW = 16 is launched only when no leaf made an interchange (the step has no swap).
// All lanes run the sweep arithmetic (lanes without a right-hand side or leaf on values that
// are never stored), so the warp votes and barriers are full-warp.
template <typename T, int KUW, bool bwd>
__global__ void __launch_bounds__(SWPB * 32) leaf_solve_kernel(LeafDev d, T* X, int nrhs, VecLayout lay) {
  pdl_trigger();
  extern __shared__ float4 lsm4[];
  using St = SolveStage<T, KUW, bwd>;
  constexpr int EPC = St::EPC, CPR = St::CPR;
  constexpr int LSTP = St::LSTP, USTP = St::USTP, XSTP = St::XSTP, YSTP = St::YSTP, XDSTP = St::XDSTP;
  constexpr int bufL = St::bufL, bufU = St::bufU;
  constexpr int RMAX = KUW - 1 < KV ? KUW - 1 : KV;
  constexpr bool CHK = St::CHKV, XPF = St::XPF, YPF = St::YPF, XOPF = St::XOPF;
  constexpr bool PIV = KUW > 16;
  constexpr int RPC = SLOT * CPR;                     // chunks of one leaf's 16 records
  constexpr int CPC = (KUW / SLOT) * CPR;             // chunks of one U column
  static_assert(RPC % 32 == 0 && (KUW * CPC) % 32 == 0, "a leaf's stage is a whole number of warp copies");
  const int lane = threadIdx.x & 31;
  const int sub = lane >> 4, c = lane & 15;
  const int nbox = d.g.nbox();
  const int b0 = (blockIdx.x * SWPB + (threadIdx.x >> 5)) * 2;   // the warp's first leaf
  if (b0 >= nbox) return;                             // whole warp: no leaf
  const int b = b0 + sub;
  const bool act = b < nbox && c < nrhs;
  T* stg = reinterpret_cast<T*>(lsm4) + (size_t)(threadIdx.x >> 5) * St::warpsz;
  const T* lrec = reinterpret_cast<const T*>(d.lrec);
  const T* urec = reinterpret_cast<const T*>(d.urec);
  const T* uext = reinterpret_cast<const T*>(d.uext);
  const unsigned long long pol = evict_first_policy();
  const int bx = d.g.bx, nx = d.nx;
  const int bb = b < nbox ? b : nbox - 1;
  // the warp's two leaves (the second clamped) and the grid nodes of their interiors' (0, 0)
  const int bl0 = b0, bl1 = b0 + 1 < nbox ? b0 + 1 : b0;
  const int og0 = (bl0 % bx) * (LEAF + 1) + nx * ((bl0 / bx) * (LEAF + 1));
  const int og1 = (bl1 % bx) * (LEAF + 1) + nx * ((bl1 / bx) * (LEAF + 1));
  auto bl = [&](int s) { return s ? bl1 : bl0; };
  auto og = [&](int s) { return s ? og1 : og0; };
  const int o0 = og(sub);                             // this lane's leaf
  auto node_of = [&](int j) { return o0 + j % LEAF + nx * (j / LEAF); };
  T* yb = reinterpret_cast<T*>(d.ybuf) + (size_t)bb * NI * QL;   // backward only, rows of 16
  T* Xc = X + (size_t)c * lay.cs;
  const long long rs = lay.rs;
  auto xat = [&](int node) -> T& {
    if constexpr (CHK) return X[(size_t)node * SLOT + c];
    else return Xc[(size_t)(node * rs)];
  };
  // chunk k (4 values) of the 16-value row of grid node `node` (FP32 chunked vector)
  auto node_chunk = [&](T* dst, int node, int k) { cp_async16(dst, X + (size_t)node * SLOT + 4 * k); };

  // ---- backward input: side values x_d (60 per leaf: BOTTOM, TOP, LEFT, RIGHT, 15 each, the
  //      grid neighbours of the boundary rows) and their coupling coefficients
  T* xd = stg + 2 * bufL;                             // [leaf][q][16], pitch XDSTP
  T* cf = xd + 2 * XDSTP;                             // [leaf][q], pitch 64
  auto side_node = [&](int s, int q) {
    const int t = q % LEAF, o = og(s);
    switch (q / LEAF) {
      case SIDE_BOTTOM: return o - nx + t;
      case SIDE_TOP: return o + LEAF * nx + t;
      case SIDE_LEFT: return o - 1 + nx * t;
      default: return o + LEAF + nx * t;
    }
  };
  if constexpr (bwd) {
    // a side exists unless the leaf touches the grid boundary there (coefficient 0)
    for (int x = lane; x < 2 * NQ; x += 32) {
      const int s = x / NQ, q = x % NQ;
      cf[s * 64 + q] = reinterpret_cast<const T*>(d.cpl)[(size_t)bl(s) * NQ + q];
    }
    __syncwarp();
  }
  // (A_Id x_d)_j of row j = (lx, ly), terms in the order of the CSR columns
  auto cplin = [&](int lx, int ly) -> T {
    const T* xs = xd + sub * XDSTP + c;
    const T* cs = cf + sub * 64;
    T v = T(0);
    if (ly == 0) v += cs[lx] * xs[lx * SLOT];
    if (lx == 0) v += cs[2 * LEAF + ly] * xs[(2 * LEAF + ly) * SLOT];
    if (lx == LEAF - 1) v += cs[3 * LEAF + ly] * xs[(3 * LEAF + ly) * SLOT];
    if (ly == LEAF - 1) v += cs[LEAF + lx] * xs[(LEAF + lx) * SLOT];
    return v;
  };

  // ---- L sweep: y = L^{-1} P x, blocks of 16 steps.  Stage of block blk: its records and
  //      (FP32 forward) right-hand-side rows blk * 16 + 16 .. + 31, the refills of its steps.
  auto issue_L_rec = [&](int blk, int buf) {
    T* S = stg + (size_t)buf * bufL;
    const int j0 = blk * SLOT;
    const int nch = (NI - j0 < SLOT ? NI - j0 : SLOT) * CPR;
#pragma unroll
    for (int i = 0; i < 2 * RPC / 32; ++i) {
      const int s = i / (RPC / 32), k = lane + 32 * (i % (RPC / 32));
      if (k < nch) cp_async16_ef(S + s * LSTP + k * EPC, lrec + ((size_t)bl(s) * NI + j0) * SLOT + k * EPC, pol);
    }
  };
  auto issue_L_x = [&](int blk, int buf) {
    if constexpr (XPF) {
      T* S = stg + (size_t)buf * bufL + 2 * LSTP;
#pragma unroll
      for (int i = 0; i < 2 * SLOT * 4 / 32; ++i) {
        const int s = i / (SLOT * 4 / 32), u = (lane + 32 * (i % (SLOT * 4 / 32))) / 4, k = lane % 4;
        const int r = blk * SLOT + SLOT + u;
        if (r < NI) node_chunk(S + s * XSTP + u * SLOT + 4 * k, og(s) + r % LEAF + nx * (r / LEAF), k);
      }
    }
    cp_async_commit();
  };
  const int nbl = (NI + SLOT - 1) / SLOT;
  issue_L_rec(0, 0);
  pdl_wait();                             // the solve vector is written by the preceding kernel
  if constexpr (bwd) {
    if constexpr (CHK) {
      for (int x = lane; x < 2 * NQ * 4; x += 32) {
        const int s = x / (NQ * 4), q = (x / 4) % NQ, k = x % 4;
        T* dst = xd + s * XDSTP + q * SLOT + 4 * k;
        if (cf[s * 64 + q] != T(0)) node_chunk(dst, side_node(s, q), k);
        else *reinterpret_cast<float4*>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    } else {
      for (int q = 0; q < NQ; ++q) {
        const T a = cf[sub * 64 + q];
        xd[sub * XDSTP + q * SLOT + c] = (act && a != T(0)) ? xat(side_node(sub, q)) : T(0);
      }
    }
  }
  issue_L_x(0, 0);
  T W[16];
  if constexpr (bwd) {
    cp_async_wait<0>();
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 16; ++r) W[r] = cplin(r % LEAF, r / LEAF);
  } else {
#pragma unroll
    for (int r = 0; r < 16; ++r) W[r] = act ? xat(node_of(r)) : T(0);
  }
  for (int blk = 0; blk < nbl; ++blk) {
    if (blk + 1 < nbl) {
      issue_L_rec(blk + 1, (blk + 1) & 1);
      issue_L_x(blk + 1, (blk + 1) & 1);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncwarp();
    const T* S = stg + (size_t)(blk & 1) * bufL + sub * LSTP;
    const T* xs = stg + (size_t)(blk & 1) * bufL + 2 * LSTP + sub * XSTP + c;
    int lx = (blk * SLOT) % LEAF, node = node_of(blk * SLOT);   // grid node of step j
    int rx = (blk * SLOT + SLOT) % LEAF, ry = (blk * SLOT + SLOT) / LEAF;   // row j + 16 (backward)
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      const int j = blk * SLOT + u;
      if (j < NI) {
        T lv[16];
        lds_vec(S + u * SLOT, lv);
        T bv = W[u];
        if constexpr (PIV) {
          const int dsw = (int)lv[15];     // 0..15: the interchange stays in the window
          if (__any_sync(0xffffffffu, dsw != 0)) {
            const T a = bv;
#pragma unroll
            for (int r = 1; r < 16; ++r)
              if (r == dsw) { bv = W[(u + r) & 15]; W[(u + r) & 15] = a; }
          }
        }
#pragma unroll
        for (int r = 1; r < 16; ++r) W[(u + r) & 15] -= lv[r - 1] * bv;
        if (act) {
          if constexpr (!bwd) xat(node) = bv;    // y_j over b_j
          else yb[(size_t)j * SLOT + c] = bv;
        }
        T nv = T(0);
        if (j + 16 < NI) {
          if constexpr (bwd) nv = cplin(rx, ry);
          else if constexpr (XPF) nv = xs[u * SLOT];
          else nv = act ? xat(node_of(j + 16)) : T(0);
        }
        W[u] = nv;
        const bool wrap = lx == LEAF - 1;
        lx = wrap ? 0 : lx + 1;
        node += wrap ? nx - (LEAF - 1) : 1;
        if constexpr (bwd) {
          const bool rw = rx == LEAF - 1;
          rx = rw ? 0 : rx + 1;
          ry += rw ? 1 : 0;
        }
      }
    }
    __syncwarp();
  }

  // ---- U sweep: x = U^{-1} y, blocks of KUW steps from the bottom.  Stage of block blk: its
  //      U columns, (FP32) the y rows of block blk + 1 (the refills of its steps) and
  //      (FP32 backward) the x rows of block blk.
  auto issue_U = [&](int blk, int buf) {
    T* S = stg + (size_t)buf * bufU;
    const int t0 = blk * KUW;
#pragma unroll
    for (int i = 0; i < 2 * KUW * CPC / 32; ++i) {
      const int s = i / (KUW * CPC / 32), rem = lane + 32 * (i % (KUW * CPC / 32)), u = rem / CPC, k = rem % CPC;
      const int j = NI - 1 - (t0 + u);
      if (j >= 0) {
        const size_t rec = ((size_t)bl(s) * NI + j) * SLOT;
        const T* src = k < CPR ? urec + rec + k * EPC : uext + rec + (k - CPR) * EPC;
        cp_async16_ef(S + s * USTP + u * KUW + k * EPC, src, pol);
      }
    }
    if constexpr (YPF) {
      T* Y = S + 2 * USTP;
#pragma unroll
      for (int i = 0; i < 2 * KUW * 4 / 32; ++i) {
        const int s = i / (KUW * 4 / 32), u = (lane + 32 * (i % (KUW * 4 / 32))) / 4, k = lane % 4;
        const int r = NI - 1 - (t0 + KUW + u);
        if (r >= 0) {
          if constexpr (bwd)
            cp_async16(Y + s * YSTP + u * SLOT + 4 * k,
                       reinterpret_cast<const T*>(d.ybuf) + ((size_t)bl(s) * NI * QL + (size_t)r * SLOT) + 4 * k);
          else
            node_chunk(Y + s * YSTP + u * SLOT + 4 * k, og(s) + r % LEAF + nx * (r / LEAF), k);
        }
      }
    }
    if constexpr (XOPF) {
      T* XO = S + 2 * USTP + 2 * YSTP;
#pragma unroll
      for (int i = 0; i < 2 * KUW * 4 / 32; ++i) {
        const int s = i / (KUW * 4 / 32), u = (lane + 32 * (i % (KUW * 4 / 32))) / 4, k = lane % 4;
        const int r = NI - 1 - (t0 + u);
        if (r >= 0) node_chunk(XO + s * YSTP + u * SLOT + 4 * k, og(s) + r % LEAF + nx * (r / LEAF), k);
      }
    }
    cp_async_commit();
  };
  // (FP64 forward) row j - KUW from row j: KUW = 15 q + m, so q leaf rows down and m nodes
  // left, one more row down (and LEAF nodes right) when fewer than m nodes are left of j
  constexpr int QD = KUW / LEAF, MD = KUW % LEAF;
  const int nbu = (NI + KUW - 1) / KUW;
  T V[KUW];
#pragma unroll
  for (int r = 0; r < KUW; ++r)
    V[r] = (act && NI - 1 - r >= 0) ? (bwd ? yb[(size_t)(NI - 1 - r) * SLOT + c] : xat(node_of(NI - 1 - r))) : T(0);
  issue_U(0, 0);
  for (int blk = 0; blk < nbu; ++blk) {
    if (blk + 1 < nbu) { issue_U(blk + 1, (blk + 1) & 1); cp_async_wait<1>(); }
    else cp_async_wait<0>();
    __syncwarp();
    const T* S = stg + (size_t)(blk & 1) * bufU + sub * USTP;
    const T* ys = stg + (size_t)(blk & 1) * bufU + 2 * USTP + sub * YSTP + c;
    const T* xo = stg + (size_t)(blk & 1) * bufU + 2 * USTP + 2 * YSTP + sub * YSTP + c;
    const int jt = NI - 1 - blk * KUW;
    int lx = jt % LEAF, node = node_of(jt);      // grid node of step j (descending)
#pragma unroll
    for (int u = 0; u < KUW; ++u) {
      const int t = blk * KUW + u;
      if (t < NI) {
        const int j = NI - 1 - t;
        T uv[KUW];
        lds_vec(S + u * KUW, uv);
        const T x = V[u] * uv[0];
        if (act) {
          if constexpr (!bwd) xat(node) = x;
          else if constexpr (XOPF) xat(node) = xo[u * SLOT] - x;
          else xat(node) -= x;
        }
#pragma unroll
        for (int r = 1; r <= RMAX; ++r) V[(u + r) & (KUW - 1)] -= uv[r] * x;
        T nv = T(0);
        if (j - KUW >= 0) {
          if constexpr (YPF) nv = ys[u * SLOT];
          else if constexpr (bwd) nv = act ? yb[(size_t)(j - KUW) * SLOT + c] : T(0);
          else nv = act ? xat(node - QD * nx - MD + (lx < MD ? LEAF - nx : 0)) : T(0);
        }
        V[u] = nv;
        const bool wrap = lx == 0;
        lx = wrap ? LEAF - 1 : lx - 1;
        node -= wrap ? nx - (LEAF - 1) : 1;
      }
    }
    __syncwarp();
  }
}

// ---- FP64 leaf sweeps over the band rows: few right-hand sides, or few leaves.
//
// A half-warp owns one leaf and its 16 lanes own the 16 rows of the sweep window (row j in lane
// j mod 16), so a step is one shuffle and one multiply-add per right-hand side for all 15 rows
// at once, instead of 15 multiply-adds in a thread that owns a whole column.  R right-hand sides
// run side by side in a warp; the others are other warps (gridDim.y).
// What bounds it: a FP64 warp instruction occupies an SM sub-partition for 64 cycles however few
// of its lanes are active (measured: 64.1 cycles with 1 to 32 lanes, 67 from one to the next
// that needs it).  Per two leaves and pair of steps (one of L, one of U) this form issues
// 2 R + 1 of them for R right-hand sides, leaf_solve_kernel 31 for any number up to 16.
// Forward + backward launch, before and after: 63^2, 1 right-hand side 294 + 314 -> 53 + 62 us;
// 255^2, 5: 312 + 343 -> 62 + 72 us; 1023^2, 4: 894 + 1029 -> 340 + 386 us; with interchanges
// (1023^2 Helmholtz, 8) 1959 + 2138 -> 1093 + 1235 us.
// The U sweep scales the column by its reciprocal pivot (once per step, off the chain) instead of
// the running value, and the solution rows once per 16 steps.
// The right-hand sides (backward: A_Id x_d) are brought into shared memory first and the sweeps
// run in place there; a lane reads and writes only rows j = lane mod 16, so the sweeps need no
// barrier.  The records come straight from global memory, one block of 16 steps ahead (a
// half-warp reads a record as one contiguous run).  Every address is valid whether or not its
// value is used: shared loads under a condition may be issued ahead of it.
constexpr int RWPB = 4;                                // warps per CTA
constexpr int RNB = 15;                                // blocks of 16 rows (the last holds one)
constexpr int RROW = 16 * (RNB + 1);                   // rows of a right-hand side and a block of zeros
template <int R>
__host__ __device__ constexpr int row_leaf_pitch() { return R * RROW + (R % 2 == 0 ? 16 : 0); }
template <int R>
__host__ __device__ constexpr size_t row_smem() { return (size_t)RWPB * 2 * row_leaf_pitch<R>() * sizeof(double); }

// Records of block blk, lane l's slot of each: every address lies inside the leaf's records (the
// last block repeats its one column, a block number past either end is clamped), so the loads
// need no condition; the sweeps use only the columns that exist.
__device__ __forceinline__ void rows_load_L(const double* lr, int blk, int l, double (&v)[16]) {
  const int bk = min(max(blk, 0), RNB - 1);
#pragma unroll
  for (int u = 0; u < 16; ++u) v[u] = __ldg(lr + 16 * min(16 * bk + u, NI - 1) + ((l - u + 31) & 15));
}
__device__ __forceinline__ void rows_load_U(const double* ur, int blk, int l, double (&v)[16]) {
  const int bk = min(max(blk, 0), RNB - 1);
#pragma unroll
  for (int u = 0; u < 16; ++u) v[u] = __ldg(ur + 16 * min(16 * bk + u, NI - 1) + ((u - l + 16) & 15));
}

// y = L^{-1} P y in place (y: R columns of RROW values, rows >= NI zero; rows before block b0 stay
// as they are).  lv holds block b0.
template <int R, bool PIV>
__device__ __forceinline__ void rows_sweep_L(const double* lr, double* y, double (&lv)[16], int b0) {
  const int lane = threadIdx.x & 31, l = lane & 15, hb = lane & 16;
  double W[R];
#pragma unroll
  for (int c = 0; c < R; ++c) W[c] = y[c * RROW + 16 * b0 + l];
#pragma unroll 1
  for (int blk = b0; blk < RNB; ++blk) {
    double ln[16], nx[R], fin[R];
    rows_load_L(lr, blk + 1, l, ln);
#pragma unroll
    for (int c = 0; c < R; ++c) {
      nx[c] = y[c * RROW + 16 * (blk + 1) + l];        // past the last block: the zeros
      fin[c] = 0.0;
    }
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      if (16 * blk + u < NI) {
        int dsw = 0;
        if constexpr (PIV) dsw = (int)__shfl_sync(0xffffffffu, lv[u], hb | u);   // pivot offset 0..15
        const double m = l == u ? 0.0 : lv[u];
#pragma unroll
        for (int c = 0; c < R; ++c) {
          double b;
          if constexpr (PIV) {
            const int s = (u + dsw) & 15;
            const double a = __shfl_sync(0xffffffffu, W[c], hb | u);
            b = __shfl_sync(0xffffffffu, W[c], hb | s);
            if (l == s) W[c] = a;                      // the interchanged row; lane u retires below
          } else {
            b = __shfl_sync(0xffffffffu, W[c], hb | u);
          }
          W[c] -= m * b;
          if (l == u) { fin[c] = b; W[c] = nx[c]; }
        }
      }
    }
#pragma unroll
    for (int c = 0; c < R; ++c) y[c * RROW + 16 * blk + l] = fin[c];
#pragma unroll
    for (int u = 0; u < 16; ++u) lv[u] = ln[u];
  }
}

// y = U^{-1} y in place; WIDE: upper bandwidth up to 30 (a second window of 16 rows).
template <int R, bool WIDE>
__device__ __forceinline__ void rows_sweep_U(const double* ur, const double* ux, double* y) {
  const int lane = threadIdx.x & 31, l = lane & 15, hb = lane & 16;
  constexpr int AHEAD = WIDE ? 2 : 1;
  double uv[16], xv[16], V[R], V1[R];
  rows_load_U(ur, RNB - 1, l, uv);
  if constexpr (WIDE) rows_load_U(ux, RNB - 1, l, xv);
  // the last block holds row NI - 1 (lane 0); the other lanes start one block down
  const int top = l == 0 ? RNB - 1 : RNB - 2;
#pragma unroll
  for (int c = 0; c < R; ++c) {
    V[c] = y[c * RROW + 16 * top + l];
    V1[c] = WIDE ? y[c * RROW + 16 * (top - 1) + l] : 0.0;
  }
#pragma unroll 1
  for (int blk = RNB - 1; blk >= 0; --blk) {
    double un[16], xn[16], nx[R], fin[R], dself = 0.0;
    rows_load_U(ur, blk - 1, l, un);
    if constexpr (WIDE) rows_load_U(ux, blk - 1, l, xn);
    // rows above the first do not exist: the zero block stands for them
    const int nb = blk >= AHEAD ? blk - AHEAD : RNB;
#pragma unroll
    for (int c = 0; c < R; ++c) {
      nx[c] = y[c * RROW + 16 * nb + l];
      fin[c] = 0.0;
    }
#pragma unroll
    for (int u = 15; u >= 0; --u) {
      if (16 * blk + u < NI) {
        const double dinv = __shfl_sync(0xffffffffu, uv[u], hb | u);
        if (l == u) dself = uv[u];
        const double g = l == u ? 0.0 : uv[u] * dinv;
        double g1 = 0.0;
        if constexpr (WIDE) g1 = xv[u] * dinv;         // slot r - 16; lane u: r = 16
#pragma unroll
        for (int c = 0; c < R; ++c) {
          const double v = __shfl_sync(0xffffffffu, V[c], hb | u);
          V[c] -= g * v;
          if constexpr (WIDE) V1[c] -= g1 * v;
          if (l == u) {
            fin[c] = v;
            if constexpr (WIDE) { V[c] = V1[c]; V1[c] = nx[c]; }
            else V[c] = nx[c];
          }
        }
      }
    }
#pragma unroll
    for (int c = 0; c < R; ++c) y[c * RROW + 16 * blk + l] = fin[c] * dself;   // rows >= NI stay zero
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      uv[u] = un[u];
      if constexpr (WIDE) xv[u] = xn[u];
    }
  }
}

template <int R, bool WIDE, bool bwd>
__global__ void __launch_bounds__(RWPB * 32) leaf_rows_kernel(LeafDev d, double* X, int nrhs, VecLayout lay) {
  extern __shared__ float4 lsm4[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane >> 4, l = lane & 15;
  const int nbox = d.g.nbox();
  // a warp without a leaf and a half-warp without one repeat the last leaf and store nothing
  const int bq = (blockIdx.x * RWPB + warp) * 2 + sub;
  const bool live = bq < nbox;
  const int b = live ? bq : nbox - 1;
  const int c0 = blockIdx.y * R;
  double* y = reinterpret_cast<double*>(lsm4) + (2 * warp + sub) * row_leaf_pitch<R>();
  const double* lr = reinterpret_cast<const double*>(d.lrec) + (size_t)b * NI * 16;
  const double* ur = reinterpret_cast<const double*>(d.urec) + (size_t)b * NI * 16;
  const double* ux = reinterpret_cast<const double*>(d.uext) + (size_t)b * NI * 16;
  const int nx = d.nx;
  const int o = (b % d.g.bx) * (LEAF + 1) + nx * ((b / d.g.bx) * (LEAF + 1));
  double lv[16];
  rows_load_L(lr, 0, l, lv);                           // the factor's: overlaps the preceding kernel
  pdl_enter();
  // rows l, l + 16, ... of the right-hand sides (backward: of A_Id x_d, the terms of a row in the
  // order of the CSR columns; a coefficient of 0 may stand for a side outside the grid, so nothing is
  // read for it)
#pragma unroll 1
  for (int blk = 0; blk < RNB + 1; ++blk) {
    const int jr = 16 * blk + l, j = min(jr, NI - 1);
    const int lx = j % LEAF, ly = j / LEAF, own = o + lx + nx * ly;
    const bool in = jr < NI;
    double v[R];
    if constexpr (!bwd) {
#pragma unroll
      for (int c = 0; c < R; ++c) {
        const int cc = min(c0 + c, nrhs - 1);
        const double xv = X[lay.at(own, cc)];
        v[c] = (in && c0 + c < nrhs) ? xv : 0.0;
      }
    } else {
      const double* cp = reinterpret_cast<const double*>(d.cpl) + (size_t)b * NQ;
#pragma unroll
      for (int c = 0; c < R; ++c) v[c] = 0.0;
      auto term = [&](bool on, int q, int nb) {
        const double a = on ? __ldg(cp + q) : 0.0;
        if (a != 0.0) {
#pragma unroll
          for (int c = 0; c < R; ++c) {
            const double xv = X[lay.at(nb, min(c0 + c, nrhs - 1))];
            v[c] += a * xv;
          }
        }
      };
      if (in) {
        term(ly == 0, lx, o - nx + lx);
        term(lx == 0, 2 * LEAF + ly, o - 1 + nx * ly);
        term(lx == LEAF - 1, 3 * LEAF + ly, o + LEAF + nx * ly);
        term(ly == LEAF - 1, LEAF + lx, o + LEAF * nx + lx);
      }
    }
#pragma unroll
    for (int c = 0; c < R; ++c) y[c * RROW + jr] = v[c];
  }
  rows_sweep_L<R, WIDE>(lr, y, lv, 0);
  rows_sweep_U<R, WIDE>(ur, ux, y);
  if (!live) return;
#pragma unroll 1
  for (int j = l; j < NI; j += 16) {
    const int node = o + j % LEAF + nx * (j / LEAF);
#pragma unroll
    for (int c = 0; c < R; ++c)
      if (c0 + c < nrhs) {
        double* x = X + lay.at(node, c0 + c);
        if constexpr (!bwd) *x = y[c * RROW + j];
        else *x -= y[c * RROW + j];
      }
  }
}

// ---- leaf factorization, kernel B in FP64: the sweeps over the band rows, R of the 60 columns per
// half-warp.  The columns are taken in the order of their interior neighbours' rows m and a warp
// starts its L sweep at the block of 16 rows that holds the first of them (15 rows earlier where
// the leaf has interchanges: they move a row up by at most 15).  The leaf's couplings are in F
// already; a column of F takes A_dI times the ring of its solution.
// For grids of few leaves: there the chain of a thread that owns a column bounds the time (31 FP64
// instructions of 64 cycles for a step of L and one of U), here it is 2 R + 1.  At 32 leaves the
// leaf factorization takes 325 us with it and 575 without.  On many leaves both forms
// are bound by the FP64 pipe and this one issues more (the scaled U column, the halves' idle lanes).
template <int R>
__host__ __device__ constexpr int schur_warps() { return R == 2 ? 3 : 2; }          // per CTA
template <int R>
__host__ __device__ constexpr int schur_ctas() { return NQ / (2 * R * schur_warps<R>()); }   // per leaf
template <int R>
__global__ void __launch_bounds__(schur_warps<R>() * 32) leaf_schur_rows_kernel(LeafDev d) {
  static_assert(schur_ctas<R>() * schur_warps<R>() * 2 * R == NQ, "columns dealt out evenly");
  extern __shared__ float4 lsm4[];
  __shared__ double qa[NQ], qc[NQ];
  __shared__ int qm[NQ], qex[NQ];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane >> 4, l = lane & 15;
  const int b = blockIdx.x / schur_ctas<R>(), part = blockIdx.x % schur_ctas<R>();
  const int nx = d.nx, x0 = (b % d.g.bx) * (LEAF + 1), y0 = (b / d.g.bx) * (LEAF + 1);
  const double* lr = reinterpret_cast<const double*>(d.lrec) + (size_t)b * NI * 16;
  const double* ur = reinterpret_cast<const double*>(d.urec) + (size_t)b * NI * 16;
  const double* ux = reinterpret_cast<const double*>(d.uext) + (size_t)b * NI * 16;
  for (int q = threadIdx.x; q < NQ; q += blockDim.x) {
    int vx, vy, m;
    side_unknown(q, x0, y0, &vx, &vy, &m);
    const bool exists = vx >= 0 && vx < nx && vy >= 0 && vy < d.ny;
    double a = 0.0, c = 0.0;
    if (exists) {
      const int node = vx + nx * vy, mnode = (x0 + m % LEAF) + nx * (y0 + m / LEAF);
      a = csr_entry(d.rowptr, d.colind, d.val, node, mnode);
      c = csr_entry(d.rowptr, d.colind, d.val, mnode, node);
    }
    qm[q] = m;
    qex[q] = exists ? 1 : 0;
    qa[q] = a;
    qc[q] = c;
    if (part == 0) reinterpret_cast<double*>(d.cpl)[(size_t)b * NQ + q] = c;   // 0 outside the grid
  }
  double* y = reinterpret_cast<double*>(lsm4) + (2 * warp + sub) * row_leaf_pitch<R>();
  for (int x = l; x < R * RROW; x += 16) y[x] = 0.0;
  __syncthreads();
  const int first = (part * schur_warps<R>() + warp) * 2 * R;    // place of the warp's first column
  const int q0 = first + sub * R;                                // ... of the half-warp's
  if (l < R) {
    const int q = c_qorder[q0 + l];
    y[l * RROW + qm[q]] = qc[q];
  }
  __syncwarp();
  const bool piv = *d.kumax > 15;                                // some leaf made an interchange
  const int m0 = qm[c_qorder[first]], b0 = (piv ? max(m0 - 15, 0) : m0) / 16;
  double lv[16];
  rows_load_L(lr, b0, l, lv);
  if (piv) rows_sweep_L<R, true>(lr, y, lv, b0);
  else rows_sweep_L<R, false>(lr, y, lv, b0);
  if (d.kur[b] > 15) rows_sweep_U<R, true>(ur, ux, y);
  else rows_sweep_U<R, false>(ur, ux, y);
  __syncwarp();
  double* F = reinterpret_cast<double*>(d.F) + (size_t)b * d.ldF * d.ldF;
#pragma unroll 1
  for (int c = 0; c < R; ++c) {
    const int q = c_qorder[q0 + c];
    if (!qex[q]) continue;
    for (int r = l; r < NQ; r += 16)
      if (qex[r]) F[r + (size_t)d.ldF * q] -= qa[r] * y[c * RROW + qm[r]];
  }
}

// Backward leaf step of the mixed path on grids of few leaves: x_I -= G x_d with
// G = A_II^{-1} A_Id (FP32, stored by the factorization) and x_d the 60 side unknowns of the
// leaf.  One leaf per CTA: G is staged in shared memory by cp.async while x_d is gathered,
// then thread j forms row j of G x_d for all right-hand sides of the chunk (up to 16) and
// updates the interior unknown j.  225 independent rows per leaf instead of one sequential
// sweep pair: on a grid of few leaves the sweeps' step latency, not traffic, bounds the time.
constexpr int GTH = 256;
constexpr int GRC = 16;                          // right-hand sides per launch
__global__ void __launch_bounds__(GTH, 3) leaf_bwd_g_kernel(LeafDev d, float* X, int nrhs, VecLayout lay) {
  pdl_trigger();
  extern __shared__ float4 gsm4[];
  float* Gs = reinterpret_cast<float*>(gsm4);    // NI x NQ
  float* xd = Gs + NI * NQ;                      // NQ x GRC
  const int b = blockIdx.x;
  const float* Gg = reinterpret_cast<const float*>(d.G) + (size_t)b * NI * NQ;
  for (int i = threadIdx.x; i < NI * NQ / 4; i += GTH) cp_async16(Gs + 4 * i, Gg + 4 * i);
  cp_async_commit();
  pdl_wait();              // G is the factorization's; the solve vector is the preceding kernel's
  const int I = b % d.g.bx, J = b / d.g.bx;
  const int x0 = I * (LEAF + 1), y0 = J * (LEAF + 1);
  const int nx = d.nx;
  for (int i = threadIdx.x; i < NQ * GRC; i += GTH) {
    const int q = i / GRC, c = i % GRC;
    int vx, vy, m;
    side_unknown(q, x0, y0, &vx, &vy, &m);
    const bool ex = c < nrhs && vx >= 0 && vx < nx && vy >= 0 && vy < d.ny;
    xd[i] = ex ? X[lay.at(vx + nx * vy, c)] : 0.f;
  }
  cp_async_wait<0>();
  __syncthreads();
  const int j = threadIdx.x;
  if (j >= NI) return;
  float acc[GRC];
#pragma unroll
  for (int c = 0; c < GRC; ++c) acc[c] = 0.f;
  const float4* gr = reinterpret_cast<const float4*>(Gs + j * NQ);
  const float4* x4 = reinterpret_cast<const float4*>(xd);
#pragma unroll 3
  for (int k = 0; k < NQ / 4; ++k) {
    const float4 g = gr[k];
    const float gq[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
    for (int t = 0; t < 4; ++t) {
#pragma unroll
      for (int c4 = 0; c4 < GRC / 4; ++c4) {
        const float4 v = x4[(4 * k + t) * (GRC / 4) + c4];
        acc[4 * c4 + 0] += gq[t] * v.x;
        acc[4 * c4 + 1] += gq[t] * v.y;
        acc[4 * c4 + 2] += gq[t] * v.z;
        acc[4 * c4 + 3] += gq[t] * v.w;
      }
    }
  }
  const int node = (x0 + j % LEAF) + nx * (y0 + j / LEAF);
#pragma unroll
  for (int c = 0; c < GRC; ++c)
    if (c < nrhs) X[lay.at(node, c)] -= acc[c];
}

// b_u -= sum over interior neighbours j of A_uj t_j, for every separator node u.  One thread
// per (separator node, right-hand side); separator nodes are enumerated in closed form: the
// R full separator rows (y = 16 r + 15) first, then the C separator columns (x = 16 q + 15) of
// the remaining rows.
template <typename T>
__global__ void sep_update_fwd_kernel(LeafDev d, T* X, int nrhs, VecLayout lay) {
  pdl_enter();
  const int nx = d.nx, ny = d.ny;
  const int R = (ny + 1) / (LEAF + 1) - 1, C = (nx + 1) / (LEAF + 1) - 1;
  const long long nrow = (long long)R * nx;
  const long long nsep = nrow + (long long)(ny - R) * C;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nsep * nrhs;
       e += (long long)gridDim.x * blockDim.x) {
    // consecutive threads: consecutive nodes (column-major vectors) or right-hand sides
    const bool cin = lay.cs == 1;
    const long long sidx = cin ? e / nrhs : e % nsep;
    const int c = (int)(cin ? e % nrhs : e / nsep);
    int ux, uy;
    if (sidx < nrow) {
      uy = (int)(sidx / nx) * (LEAF + 1) + LEAF;
      ux = (int)(sidx % nx);
    } else {
      const long long t = sidx - nrow;
      const int yy = (int)(t / C);
      ux = (int)(t % C) * (LEAF + 1) + LEAF;
      uy = (yy / LEAF) * (LEAF + 1) + yy % LEAF;
    }
    const int u = ux + nx * uy;
    T acc = T(0);
    for (int p = d.rowptr[u]; p < d.rowptr[u + 1]; ++p) {
      const int v = d.colind[p];
      const int vx = v % nx, vy = v / nx;
      const bool vsep = ((vx + 1) % (LEAF + 1) == 0) || ((vy + 1) % (LEAF + 1) == 0);
      if (!vsep) {
        T a;
        if constexpr (sizeof(T) == 4) a = d.fval[p]; else a = d.val[p];
        acc += a * X[lay.atc(v, c)];
      }
    }
    X[lay.atc(u, c)] -= acc;
  }
}

// The same update for the chunked FP32 vector (a node's 16 right-hand sides contiguous): one
// thread per separator node and all 16 right-hand sides, so that the row's CSR entries are
// read and classified once instead of once per right-hand side, and the neighbour values move
// as four 16-byte loads.  Same operations in the same order for every right-hand side.
__global__ void sep_update_fwd16_kernel(LeafDev d, float* X) {
  pdl_enter();
  const int nx = d.nx, ny = d.ny;
  const int R = (ny + 1) / (LEAF + 1) - 1, C = (nx + 1) / (LEAF + 1) - 1;
  const long long nrow = (long long)R * nx;
  const long long nsep = nrow + (long long)(ny - R) * C;
  for (long long sidx = blockIdx.x * (long long)blockDim.x + threadIdx.x; sidx < nsep;
       sidx += (long long)gridDim.x * blockDim.x) {
    int ux, uy;
    if (sidx < nrow) {
      uy = (int)(sidx / nx) * (LEAF + 1) + LEAF;
      ux = (int)(sidx % nx);
    } else {
      const long long t = sidx - nrow;
      const int yy = (int)(t / C);
      ux = (int)(t % C) * (LEAF + 1) + LEAF;
      uy = (yy / LEAF) * (LEAF + 1) + yy % LEAF;
    }
    const int u = ux + nx * uy;
    float4 acc[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int p = d.rowptr[u]; p < d.rowptr[u + 1]; ++p) {
      const int v = d.colind[p];
      const int vx = v % nx, vy = v / nx;
      const bool vsep = ((vx + 1) % (LEAF + 1) == 0) || ((vy + 1) % (LEAF + 1) == 0);
      if (!vsep) {
        const float a = d.fval[p];
        const float4* xv = reinterpret_cast<const float4*>(X + (size_t)v * 16);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 t = xv[q];
          acc[q].x += a * t.x; acc[q].y += a * t.y; acc[q].z += a * t.z; acc[q].w += a * t.w;
        }
      }
    }
    float4* xu = reinterpret_cast<float4*>(X + (size_t)u * 16);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float4 t = xu[q];
      t.x -= acc[q].x; t.y -= acc[q].y; t.z -= acc[q].z; t.w -= acc[q].w;
      xu[q] = t;
    }
  }
}

// side unknowns sorted by the in-leaf index of their interior neighbour, and the first
// sweep step of each of the two warps that solve for them
void qorder_tables(int* ord, int* start) {
  int m[NQ];
  for (int q = 0; q < NQ; ++q) {
    int s = q / LEAF, t = q % LEAF;
    m[q] = s == SIDE_BOTTOM ? t : s == SIDE_TOP ? t + LEAF * (LEAF - 1) : s == SIDE_LEFT ? LEAF * t : LEAF * t + LEAF - 1;
    ord[q] = q;
  }
  for (int a = 1; a < NQ; ++a)
    for (int b2 = a; b2 > 0 && (m[ord[b2]] < m[ord[b2 - 1]] || (m[ord[b2]] == m[ord[b2 - 1]] && ord[b2] < ord[b2 - 1])); --b2) {
      int t = ord[b2]; ord[b2] = ord[b2 - 1]; ord[b2 - 1] = t;
    }
  for (int w = 0; w < 2; ++w) {
    int mn = NI;
    for (int l = 32 * w; l < 32 * w + 32 && l < NQ; ++l) mn = m[ord[l]] < mn ? m[ord[l]] : mn;
    start[w] = mn - KL > 0 ? mn - KL : 0;
  }
}

}  // namespace


cudaError_t leaf_init_tables() {
  int ord[NQ], start[2];
  qorder_tables(ord, start);
  cudaError_t e = cudaMemcpyToSymbol(c_qorder, ord, sizeof(ord));
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_qstart, start, sizeof(start));
  return e;
}

template <int R>
static void leaf_schur_rows_go(const LeafDev& d, cudaStream_t s) {
  const int smem = (int)(2 * schur_warps<R>() * row_leaf_pitch<R>() * sizeof(double));
  cudaFuncSetAttribute(leaf_schur_rows_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  leaf_schur_rows_kernel<R><<<d.g.nbox() * schur_ctas<R>(), schur_warps<R>() * 32, smem, s>>>(d);
}

// Columns per half-warp of the FP64 Schur kernel over the band rows, or 0 for the one with a thread per
// column.  Leaf factorization, 2 / 5 / thread per column: 16 leaves 321 / 400 / 575 us, 64 375 / 407 /
// 577, 128 433 / 417 / 578, 256 571 / 572 / 585 (with interchanges 802 / 792 / 872), 1024 1489 / 1210 /
// 1175, 4096 5559 / 4313 / 3838.
static int schur_rows_width(int nbox) {
  const int sms = sm_count();
  return 2 * nbox <= sms ? 2 : nbox <= 2 * sms ? 5 : 0;
}

template <int LUW>
static void leaf_lu_go(const LeafDev& d, int couple, cudaStream_t s) {
  if (d.fp32) leaf_lu_kernel<float, LUW><<<d.g.nbox(), 32 * LUW, 0, s>>>(d, couple);
  else leaf_lu_kernel<double, LUW><<<d.g.nbox(), 32 * LUW, 0, s>>>(d, couple);
}

// Warps per leaf LU.  Leaf factorization with 2 / 3 / 5: 32 leaves 276 / - / 222 us, 256 521 / - / 470;
// 1024 1162 / 1128 / 1150, 4096 3846 / 3822 / 3875 (more CTAs per SM, a smaller last wave).  Two
// warps with five barriers a pivot: 32 leaves 325 us, 256 572, 1024 1175, 4096 3838.
static int lu_warps(int nbox) { return nbox <= 2 * sm_count() ? 5 : 3; }

void launch_leaf_factor(const LeafDev& d, cudaStream_t s) {
  const int nbox = d.g.nbox();
  note_launch();
  {
    const long long n = (long long)nbox * NI * 5;
    long long blocks = (n + 255) / 256;
    if (blocks > 152 * 64) blocks = 152 * 64;
    leaf_band5_kernel<<<(int)blocks, 256, 0, s>>>(d);
  }
  note_launch();
  const int R = d.fp32 ? 0 : schur_rows_width(nbox);
  if (lu_warps(nbox) == 5) leaf_lu_go<5>(d, R > 0, s);
  else leaf_lu_go<3>(d, R > 0, s);
  note_launch();
  if (d.fp32) leaf_schur_kernel<float><<<(nbox + LPC - 1) / LPC, FTH, 0, s>>>(d);
  else if (R == 2) leaf_schur_rows_go<2>(d, s);
  else if (R == 5) leaf_schur_rows_go<5>(d, s);
  else leaf_schur_kernel<double><<<(nbox + LPC - 1) / LPC, FTH, 0, s>>>(d);
}

template <typename T, int KUW>
static void leaf_solve_go(const LeafDev& d, T* X, int nrhs, VecLayout lay, int bwd, cudaStream_t s) {
  const int grid = (d.g.nbox() + 2 * SWPB - 1) / (2 * SWPB);
  note_launch();
  if (!bwd) {
    const int smem = (int)SolveStage<T, KUW, false>::bytes;
    cudaFuncSetAttribute(leaf_solve_kernel<T, KUW, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    launch_pdl(leaf_solve_kernel<T, KUW, false>, dim3(grid), dim3(SWPB * 32), smem, s, d, X, nrhs, lay);
  } else {
    const int smem = (int)SolveStage<T, KUW, true>::bytes;
    cudaFuncSetAttribute(leaf_solve_kernel<T, KUW, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    launch_pdl(leaf_solve_kernel<T, KUW, true>, dim3(grid), dim3(SWPB * 32), smem, s, d, X, nrhs, lay);
  }
}

template <int R, bool WIDE>
static void leaf_rows_go(const LeafDev& d, double* X, int nrhs, VecLayout lay, int bwd, cudaStream_t s) {
  const dim3 grid((d.g.nbox() + 2 * RWPB - 1) / (2 * RWPB), (nrhs + R - 1) / R);
  const int smem = (int)row_smem<R>();
  note_launch();
  if (!bwd) {
    cudaFuncSetAttribute(leaf_rows_kernel<R, WIDE, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    launch_pdl(leaf_rows_kernel<R, WIDE, false>, grid, dim3(RWPB * 32), smem, s, d, X, nrhs, lay);
  } else {
    cudaFuncSetAttribute(leaf_rows_kernel<R, WIDE, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    launch_pdl(leaf_rows_kernel<R, WIDE, true>, grid, dim3(RWPB * 32), smem, s, d, X, nrhs, lay);
  }
}

// Right-hand sides per warp of the FP64 sweeps over the band rows, or 0 for the sweeps over columns
// (leaf_solve_kernel).  Times in units of one FP64 warp instruction per step pair (7.2 us per
// launch at 2 GHz): a form costs the larger of its latency with one warp per SM sub-partition and
// its instructions x warps per sub-partition x the measured overhead of issuing them.  Measured
// for 1 .. 16 right-hand sides on 31^2 .. 1023^2: the column form wins at 1023^2 from 12 up
// (893 against 908 us forward) and at 511^2 at 16 (328 against 338 us), never below 511^2.
static int leaf_rows_width(int nbox, int nrhs, bool wide) {
  const double sub = 4.0 * sm_count(), pairs = (nbox + 1) / 2;
  auto cost = [&](double lat, double instr, double over, double warps) {
    return std::max(lat, instr * over * warps / sub);
  };
  const double col = wide ? cost(64, 46, 1.75, pairs) : cost(42, 31, 1.18, pairs);
  const double r1 = wide ? cost(12, 5, 1.4, pairs * nrhs) : cost(7.4, 3, 1.4, pairs * nrhs);
  const double r2 = wide ? cost(16, 8, 1.4, pairs * ((nrhs + 1) / 2)) : cost(11, 5, 1.4, pairs * ((nrhs + 1) / 2));
  if (col <= r1 && col <= r2) return 0;
  return r1 <= r2 ? 1 : 2;
}

// The FP32 solve vector is always chunked (VecLayout{16, 1, 16 N}: a node's 16 right-hand
// sides contiguous, every chunk 64-byte aligned); the FP32 forward sweep stages its rows as such.
void launch_leaf_solve(const LeafDev& d, void* Xv, int nrhs, VecLayout lay, int bwd, int kumax, cudaStream_t s) {
  if (bwd && d.fp32 && d.G) {
    const int smem = (int)(sizeof(float) * (NI * NQ + NQ * GRC));
    cudaFuncSetAttribute(leaf_bwd_g_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    for (int c0 = 0; c0 < nrhs; c0 += GRC) {
      const int nc = nrhs - c0 < GRC ? nrhs - c0 : GRC;
      note_launch();
      launch_pdl(leaf_bwd_g_kernel, dim3(d.g.nbox()), dim3(GTH), smem, s, d,
                 static_cast<float*>(Xv) + (size_t)(c0 / GRC) * lay.chunk, nc, lay);
    }
    return;
  }
  for (int c0 = 0; c0 < nrhs; c0 += SLOT) {
    const int nc = nrhs - c0 < SLOT ? nrhs - c0 : SLOT;
    if (d.fp32) {
      float* Xc = static_cast<float*>(Xv) + (size_t)(c0 / SLOT) * lay.chunk;
      if (kumax <= 15) leaf_solve_go<float, 16>(d, Xc, nc, lay, bwd, s);
      else leaf_solve_go<float, 32>(d, Xc, nc, lay, bwd, s);
    } else {
      double* Xc = static_cast<double*>(Xv) + (size_t)(c0 / SLOT) * lay.chunk;
      const int R = leaf_rows_width(d.g.nbox(), nc, kumax > 15);
      if (R == 1 && kumax <= 15) leaf_rows_go<1, false>(d, Xc, nc, lay, bwd, s);
      else if (R == 1) leaf_rows_go<1, true>(d, Xc, nc, lay, bwd, s);
      else if (R == 2 && kumax <= 15) leaf_rows_go<2, false>(d, Xc, nc, lay, bwd, s);
      else if (R == 2) leaf_rows_go<2, true>(d, Xc, nc, lay, bwd, s);
      else if (kumax <= 15) leaf_solve_go<double, 16>(d, Xc, nc, lay, bwd, s);
      else leaf_solve_go<double, 32>(d, Xc, nc, lay, bwd, s);
    }
  }
}

void launch_sep_update_fwd(const LeafDev& d, void* X, int nrhs, VecLayout lay, cudaStream_t s) {
  const int R = (d.ny + 1) / (LEAF + 1) - 1, C = (d.nx + 1) / (LEAF + 1) - 1;
  long long n = ((long long)R * d.nx + (long long)(d.ny - R) * C) * nrhs;
  if (n <= 0) return;
  int blocks = (int)((n + 255) / 256);
  if (blocks > 152 * 32) blocks = 152 * 32;
  if (blocks < 1) blocks = 1;
  note_launch();
  if (d.fp32 && lay.cs == 1 && lay.rs == 16) {   // the chunked FP32 vector: a thread per node
    const long long nsep = n / nrhs;
    int b16 = (int)((nsep + 255) / 256);
    if (b16 > 152 * 32) b16 = 152 * 32;
    if (b16 < 1) b16 = 1;
    for (int c0 = 0; c0 < nrhs; c0 += 16) {       // one launch per chunk of 16 right-hand sides
      if (c0 > 0) note_launch();
      launch_pdl(sep_update_fwd16_kernel, dim3(b16), dim3(256), 0, s, d,
                 static_cast<float*>(X) + (size_t)(c0 / 16) * lay.chunk);
    }
  } else if (d.fp32) {
    launch_pdl(sep_update_fwd_kernel<float>, dim3(blocks), dim3(256), 0, s, d, static_cast<float*>(X), nrhs, lay);
  } else {
    launch_pdl(sep_update_fwd_kernel<double>, dim3(blocks), dim3(256), 0, s, d, static_cast<double*>(X), nrhs, lay);
  }
}

}  // namespace spalu
