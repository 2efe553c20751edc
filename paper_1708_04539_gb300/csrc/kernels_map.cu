// Index-map kernels (HBM/latency bound): the value scatter into the
// supernodal storage, the gather of Ainv_{C,C} for a supernode (the
// operand of Algorithm 1 steps 3 and 5), the scatter-subtract of a Schur
// complement into the ancestors (supernodal LU), panel copies, and the
// extraction of the selected entries (Algorithm 1 step 6, Theorem 2).
#include "device.cuh"

#include <type_traits>

namespace pselinv {

namespace {

constexpr int kThreads = 256;
constexpr int kTile = 32;

__device__ __forceinline__ bool map_in_range(const SymDev& S, int64_t rb, int p, int q) {
  const int bp = S.rows_blk[rb + p];
  const int bq = S.rows_blk[rb + q];
  const int b = bp >= bq ? bq : bp;
  if (b < 0) return false;
  const int64_t base = S.blk_rel[b] - S.blk_pb[b];
  if (base + p < 0 || base + p >= S.relidx_size || base + q < 0 || base + q >= S.relidx_size)
    return false;
  const int64_t slot = map_slot(S, rb, p, q);
  return slot >= 0 && slot < S.storage;
}

template <typename T>
__global__ void __launch_bounds__(kThreads)
scatter_values_kernel(SymDev S, const T* __restrict__ vals, T* store, int64_t total) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = e / S.nnz, p = e - b * S.nnz;
    store[b * S.storage + S.value_map[p]] = vals[e];
  }
}

__device__ __forceinline__ unsigned long long abs_bits_of(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}

// One 32 x 32 tile of G_K = Ainv(R_K, R_K) (column-major, ld = c) per task.
// Entries below or on the block diagonal are read down panel columns; the
// ones above it come from U^T panels and are read along their rows, so each
// half of the tile is loaded with the lane index running over the
// contiguous direction and transposed through shared memory.

template <typename T>
__global__ void __launch_bounds__(kThreads)
gather_kernel(SymDev S, const T* __restrict__ store, T* out, const int64_t* __restrict__ gofs,
              const SnTask* __restrict__ tasks, int ntasks, const int64_t* __restrict__ mofs,
              unsigned long long* maxbase) {
  __shared__ T tile[kTile][kTile + 1];
  const int lx = threadIdx.x & 31, ly = threadIdx.x >> 5;
  for (int t = blockIdx.x; t < ntasks; t += gridDim.x) {
    const SnTask task = tasks[t];
    const int K = task.K;
    const int c = S.sn_c[K];
    const int64_t rb = S.rows_ptr[K];
    const T* src = store + (int64_t)task.inst * S.storage;
    T* G = out + gofs[t];
    const int p0 = task.a * kTile, q0 = task.b * kTile;
    // pass 1: lane runs over p (rows): lower/diagonal entries
    for (int r = ly; r < kTile; r += kThreads / 32) {
      const int p = p0 + lx, q = q0 + r;
      if (p < c && q < c && S.rows_blk[rb + p] >= S.rows_blk[rb + q]) {
        if (S.check && !map_in_range(S, rb, p, q)) {
          set_error(S.err, DEV_CHECK, K);
          tile[r][lx] = sc_zero(T());
        } else {
          tile[r][lx] = src[map_slot(S, rb, p, q)];
        }
      }
    }
    // pass 2: lane runs over q (columns): entries from U^T panels
    for (int r = ly; r < kTile; r += kThreads / 32) {
      const int p = p0 + r, q = q0 + lx;
      if (p < c && q < c && S.rows_blk[rb + p] < S.rows_blk[rb + q]) {
        if (S.check && !map_in_range(S, rb, p, q)) {
          set_error(S.err, DEV_CHECK, K);
          tile[lx][r] = sc_zero(T());
        } else {
          tile[lx][r] = src[map_slot(S, rb, p, q)];
        }
      }
    }
    __syncthreads();
    for (int r = ly; r < kTile; r += kThreads / 32) {
      const int p = p0 + lx, q = q0 + r;
      if (p < c && q < c) G[p + (int64_t)q * c] = tile[r][lx];
    }
    if constexpr (sizeof(T) == 8) {
      if (mofs) {
        // row maxima (warp 0: lane = row p) and column maxima (warp 1: lane = column q)
        unsigned long long* mrow = maxbase + mofs[t];
        if (ly == 0 && p0 + lx < c) {
          unsigned long long m = 0;
          for (int q = 0; q < kTile && q0 + q < c; q++) m = max(m, abs_bits_of((double)tile[q][lx]));
          atomicMax(mrow + p0 + lx, m);
        } else if (ly == 1 && q0 + lx < c) {
          unsigned long long m = 0;
          for (int p = 0; p < kTile && p0 + p < c; p++) m = max(m, abs_bits_of((double)tile[lx][p]));
          atomicMax(mrow + c + q0 + lx, m);
        }
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// general patterns (C_L != C_U)
// ---------------------------------------------------------------------------
// Slot of Ainv(x, y) for x = R_U(K)[p] in supernode I (block bp of R_U(K))
// and y = R_L(K)[q] in supernode J (block bq of R_L(K)), on the pattern of
// (L+U)^T: the diagonal block of J (I == J), the U^T panel of J (rows
// R_U(J), I > J) or the L panel of I (rows R_L(I), I < J).  ok = false when
// a checked read falls outside the maps or the storage.
__device__ __forceinline__ int64_t gen_slot(const SymDev& S, int64_t rbL, int64_t rbU, int p,
                                            int q, bool& ok) {
  const int bq = S.rows_blk[rbL + q], bp = S.urows_blk[rbU + p];
  const int J = S.blk_sn[bq], I = S.ublk_sn[bp];
  int64_t ri;
  if (I >= J) {
    ri = S.blk_rel[bq] - S.blk_q0[bq] + p;  // x in J (local) or its position in R_U(J)
  } else {
    ri = S.ublk_rel[bp] - S.ublk_q0[bp] + q;  // position of y in R_L(I)
  }
  if (S.check && (ri < 0 || ri >= S.relidx_size)) {
    ok = false;
    return 0;
  }
  const int64_t r = S.relidx[ri];
  int64_t slot;
  if (I == J) {
    slot = S.sn_off[J] + r + (int64_t)(S.lrows[rbL + q] - S.sn_first[J]) * S.sn_width[J];
  } else if (I > J) {
    const int sJ = S.sn_width[J];
    slot = S.sn_off[J] + (int64_t)sJ * sJ + (int64_t)S.sn_c[J] * sJ + r +
           (int64_t)(S.lrows[rbL + q] - S.sn_first[J]) * S.sn_cu[J];
  } else {
    const int sI = S.sn_width[I];
    slot = S.sn_off[I] + (int64_t)sI * sI + r +
           (int64_t)(S.urows[rbU + p] - S.sn_first[I]) * S.sn_c[I];
  }
  if (S.check && (slot < 0 || slot >= S.storage)) ok = false;
  return slot;
}

// One 32 x 32 tile of G_K = Ainv(R_U(K), R_L(K)) per task: entries with I >= J
// are read down the columns of J's blocks (lanes along p), the others along
// the columns of I's L panel (lanes along q), transposed through shared memory.
template <typename T>
__global__ void __launch_bounds__(kThreads)
gather_general_kernel(SymDev S, const T* __restrict__ store, T* out,
                      const int64_t* __restrict__ gofs, const SnTask* __restrict__ tasks,
                      int ntasks) {
  __shared__ T tile[kTile][kTile + 1];
  const int lx = threadIdx.x & 31, ly = threadIdx.x >> 5;
  for (int t = blockIdx.x; t < ntasks; t += gridDim.x) {
    const SnTask task = tasks[t];
    const int K = task.K;
    const int cl = S.sn_c[K], cu = S.sn_cu[K];
    const int64_t rbL = S.rows_ptr[K], rbU = S.urows_ptr[K];
    const T* src = store + (int64_t)task.inst * S.storage;
    T* G = out + gofs[t];
    const int p0 = task.a * kTile, q0 = task.b * kTile;
    for (int r = ly; r < kTile; r += kThreads / 32) {
      const int p = p0 + lx, q = q0 + r;
      if (p < cu && q < cl &&
          S.ublk_sn[S.urows_blk[rbU + p]] >= S.blk_sn[S.rows_blk[rbL + q]]) {
        bool ok = true;
        const int64_t slot = gen_slot(S, rbL, rbU, p, q, ok);
        if (!ok) set_error(S.err, DEV_CHECK, K);
        tile[r][lx] = ok ? src[slot] : sc_zero(T());
      }
    }
    for (int r = ly; r < kTile; r += kThreads / 32) {
      const int p = p0 + r, q = q0 + lx;
      if (p < cu && q < cl &&
          S.ublk_sn[S.urows_blk[rbU + p]] < S.blk_sn[S.rows_blk[rbL + q]]) {
        bool ok = true;
        const int64_t slot = gen_slot(S, rbL, rbU, p, q, ok);
        if (!ok) set_error(S.err, DEV_CHECK, K);
        tile[lx][r] = ok ? src[slot] : sc_zero(T());
      }
    }
    __syncthreads();
    for (int r = ly; r < kTile; r += kThreads / 32) {
      const int p = p0 + lx, q = q0 + r;
      if (p < cu && q < cl) G[p + (int64_t)q * cu] = tile[r][lx];
    }
    __syncthreads();
  }
}

// Slot of the Schur update of entry (i, m), i = R_L(K)[p] in supernode I, m =
// R_U(K)[q] in J: the diagonal block (I == J), the L panel of J (I > J: position
// of i in R_L(J) from the map of R_U(K)'s block) or the U^T panel of I (I < J:
// position of m in R_U(I)).  ok = false when a checked map read is out of range.
__device__ __forceinline__ int64_t schur_slot_general(const SymDev& S, int64_t rbL, int64_t rbU, int p,
                                                      int q, bool& ok) {
  const int bp = S.rows_blk[rbL + p], bq = S.urows_blk[rbU + q];
  const int I = S.blk_sn[bp], J = S.ublk_sn[bq];
  const int i = S.lrows[rbL + p], m = S.urows[rbU + q];
  if (I == J) {
    const int sI = S.sn_width[I], f = S.sn_first[I];
    return S.sn_off[I] + (i - f) + (int64_t)(m - f) * sI;
  }
  const int64_t ri = I > J ? S.ublk_rel[bq] - S.ublk_q0[bq] + p : S.blk_rel[bp] - S.blk_q0[bp] + q;
  if (S.check && (ri < 0 || ri >= S.relidx_size)) {
    ok = false;
    return 0;
  }
  if (I > J) {
    const int sJ = S.sn_width[J];
    return S.sn_off[J] + (int64_t)sJ * sJ + S.relidx[ri] + (int64_t)(m - S.sn_first[J]) * S.sn_c[J];
  }
  const int sI = S.sn_width[I];
  return S.sn_off[I] + (int64_t)sI * sI + (int64_t)S.sn_c[I] * sI + S.relidx[ri] +
         (int64_t)(i - S.sn_first[I]) * S.sn_cu[I];
}

// store(R_L(K), R_U(K)) -= Sc (c_L x c_U, column-major; atomic: supernodes
// of one level may update the same ancestors); slots as above.
template <typename T>
__global__ void __launch_bounds__(kThreads)
scatter_sub_general_kernel(SymDev S, T* store, const T* __restrict__ src,
                           const int64_t* __restrict__ sofs, const SnTask* __restrict__ tasks,
                           int ntasks) {
  const int lx = threadIdx.x & 31, ly = threadIdx.x >> 5;
  for (int t = blockIdx.x; t < ntasks; t += gridDim.x) {
    const SnTask task = tasks[t];
    const int K = task.K;
    const int cl = S.sn_c[K], cu = S.sn_cu[K];
    const int64_t rbL = S.rows_ptr[K], rbU = S.urows_ptr[K];
    T* dst = store + (int64_t)task.inst * S.storage;
    const T* Sc = src + sofs[t];
    const int p0 = task.a * kTile, q0 = task.b * kTile;
    for (int r = ly; r < kTile; r += kThreads / 32) {
      const int p = p0 + lx, q = q0 + r;
      if (p >= cl || q >= cu) continue;
      bool ok = true;
      const int64_t slot = schur_slot_general(S, rbL, rbU, p, q, ok);
      if (S.check && (slot < 0 || slot >= S.storage)) ok = false;
      if (!ok) {
        set_error(S.err, DEV_CHECK, K);
        continue;
      }
      atomic_add_s(dst + slot, scale_s(Sc[p + (int64_t)q * cl], -1.0));
    }
  }
}

// store(R_K, R_K) -= Sc (atomic: siblings of one level update shared
// ancestors); ASSIGN: store(R_K, R_K) = Sc (the import of a gathered block);
// LOWER: the entries p >= q only (a symmetric Sc).  Entry (p, q), x = R_K[p]
// in supernode I, y = R_K[q] in J, lies in J's diagonal block or L panel
// (I >= J: the column's storage base + the relative index of p) or in I's
// U^T panel (I < J: the row's base + the relative index of q); the bases of
// the tile's 32 rows and columns are staged in shared memory once, so an
// entry costs one index load, one value load and one store or atomic.
template <typename T, bool ASSIGN = false, bool LOWER = false>
__global__ void __launch_bounds__(kThreads)
scatter_sub_kernel(SymDev S, T* store, const T* __restrict__ src, const int64_t* __restrict__ sofs,
                   const SnTask* __restrict__ tasks, int ntasks) {
  __shared__ int64_t cdiag[kTile], cpan[kTile], crel[kTile], rpan[kTile], rrel[kTile];
  __shared__ int csn[kTile], rsn[kTile];
  const int tid = threadIdx.x, lx = tid & 31, ly = tid >> 5;
  for (int t = blockIdx.x; t < ntasks; t += gridDim.x) {
    const SnTask task = tasks[t];
    const int K = task.K;
    const int c = S.sn_c[K];
    const int64_t rb = S.rows_ptr[K];
    T* dst = store + (int64_t)task.inst * S.storage;
    const T* Sc = src + sofs[t];
    const int p0 = task.a * kTile, q0 = task.b * kTile;
    if (tid < kTile) {
      const int q = q0 + tid;
      if (q < c) {
        cdiag[tid] = S.col_diag[rb + q];
        cpan[tid] = S.col_pan[rb + q];
        crel[tid] = S.col_rel[rb + q];
        csn[tid] = S.col_sn[rb + q];
      }
    } else if (tid < 2 * kTile) {
      const int pl = tid - kTile, p = p0 + pl;
      if (p < c) {
        rpan[pl] = S.row_pan[rb + p];
        rrel[pl] = S.row_rel[rb + p];
        rsn[pl] = S.row_sn[rb + p];
      }
    }
    __syncthreads();
    for (int r = ly; r < kTile; r += kThreads / 32) {
      const int p = p0 + lx, q = q0 + r;  // lanes along p: Sc is column major
      if (p >= c || q >= c || (LOWER && p < q)) continue;
      const bool col_side = rsn[lx] >= csn[r];
      const int64_t ri = col_side ? crel[r] + p : rrel[lx] + q;
      if (S.check && (ri < 0 || ri >= S.relidx_size)) {
        set_error(S.err, DEV_CHECK, K);
        continue;
      }
      const int64_t slot =
          (col_side ? (rsn[lx] == csn[r] ? cdiag[r] : cpan[r]) : rpan[lx]) + S.relidx[ri];
      if (S.check && (slot < 0 || slot >= S.storage)) {
        set_error(S.err, DEV_CHECK, K);
        continue;
      }
      const T v = Sc[p + (int64_t)q * c];
      if (ASSIGN)
        dst[slot] = v;
      else
        atomic_add_s(dst + slot, scale_s(v, -1.0));
    }
    __syncthreads();
  }
}

// Schur complement of one supernode's FP64 panels subtracted straight from
// the ancestors: a task computes the TS x TS tile (tp, tq) of TL TU^T over K
// range [k0, k1) and subtracts it atomically (so a K split costs nothing but
// atomics), the storage bases of the tile's rows and columns staged as in
// scatter_sub_kernel.  The product is never stored, and a level needs one
// launch for what were a product and a scatter.  256 threads, (TS / 16)^2
// outputs each; the FP64 pipe (19 cycles per warp operation and SM) is the
// bound of a task: 32 x 32 x 32 takes it 10 us, 16 x 16 x 32 2.5 us, so levels
// of little work use the small tile (see add_schur_scatter).
template <typename T, int TS, bool LOWER, bool GENERAL>
__global__ void __launch_bounds__(kThreads)
schur_scatter_kernel(SymDev S, T* store, const SchurDesc* __restrict__ descs,
                     const SchurTask* __restrict__ tasks, int ntasks) {
  constexpr int TM = TS / 16, BK = 32, NL = TS * BK / kThreads;
  __shared__ T sa[BK][TS], sb[BK][TS];
  __shared__ int64_t cdiag[TS], cpan[TS], crel[TS], rpan[TS], rrel[TS];
  __shared__ int csn[TS], rsn[TS];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  for (int t = blockIdx.x; t < ntasks; t += gridDim.x) {
    const SchurTask task = tasks[t];
    const SchurDesc d = descs[task.d];
    const T* __restrict__ A = (const T*)d.TL;
    const T* __restrict__ B = (const T*)d.TU;
    const int K = d.K, c = d.c, cu = d.cu;
    const int p0 = task.tp * TS, q0 = task.tq * TS;
    const int64_t rbL = S.rows_ptr[K], rbU = GENERAL ? S.urows_ptr[K] : rbL;
    T ra[NL], rb[NL];
    auto load = [&](int k0) {
#pragma unroll
      for (int i = 0; i < NL; i++) {
        const int e = tid + i * kThreads, m = e % TS, k = k0 + e / TS;
        const bool in = k < task.k1;
        ra[i] = in && p0 + m < c ? A[p0 + m + (int64_t)k * c] : sc_zero(T());
        rb[i] = in && q0 + m < cu ? B[q0 + m + (int64_t)k * cu] : sc_zero(T());
      }
    };
    load(task.k0);
    if (!GENERAL) {
      if (tid < TS) {
        if (q0 + tid < c) {
          cdiag[tid] = S.col_diag[rbL + q0 + tid];
          cpan[tid] = S.col_pan[rbL + q0 + tid];
          crel[tid] = S.col_rel[rbL + q0 + tid];
          csn[tid] = S.col_sn[rbL + q0 + tid];
        }
      } else if (tid < 2 * TS) {
        const int m = tid - TS;
        if (p0 + m < c) {
          rpan[m] = S.row_pan[rbL + p0 + m];
          rrel[m] = S.row_rel[rbL + p0 + m];
          rsn[m] = S.row_sn[rbL + p0 + m];
        }
      }
    }
    T acc[TM][TM];
#pragma unroll
    for (int i = 0; i < TM; i++)
#pragma unroll
      for (int j = 0; j < TM; j++) acc[i][j] = sc_zero(T());
    for (int k0 = task.k0; k0 < task.k1; k0 += BK) {
      __syncthreads();
#pragma unroll
      for (int i = 0; i < NL; i++) {
        const int e = tid + i * kThreads;
        sa[e / TS][e % TS] = ra[i];
        sb[e / TS][e % TS] = rb[i];
      }
      __syncthreads();
      if (k0 + BK < task.k1) load(k0 + BK);
      const int kn = min(BK, task.k1 - k0);
#pragma unroll 4
      for (int k = 0; k < kn; k++) {
        T a[TM], b[TM];
#pragma unroll
        for (int i = 0; i < TM; i++) a[i] = sa[k][tx + 16 * i];
#pragma unroll
        for (int j = 0; j < TM; j++) b[j] = sb[k][ty + 16 * j];
#pragma unroll
        for (int i = 0; i < TM; i++)
#pragma unroll
          for (int j = 0; j < TM; j++) acc[i][j] = fma_s(a[i], b[j], acc[i][j]);
      }
    }
    T* dst = store + (int64_t)d.inst * S.storage;
#pragma unroll
    for (int i = 0; i < TM; i++)
#pragma unroll
      for (int j = 0; j < TM; j++) {
        const int pl = tx + 16 * i, ql = ty + 16 * j, p = p0 + pl, q = q0 + ql;
        if (p >= c || q >= cu || (LOWER && p < q)) continue;
        int64_t slot = 0;
        bool ok = true;
        if (GENERAL) {
          slot = schur_slot_general(S, rbL, rbU, p, q, ok);
        } else {
          const bool col_side = rsn[pl] >= csn[ql];
          const int64_t ri = col_side ? crel[ql] + p : rrel[pl] + q;
          if (S.check && (ri < 0 || ri >= S.relidx_size)) ok = false;
          if (ok)
            slot = (col_side ? (rsn[pl] == csn[ql] ? cdiag[ql] : cpan[ql]) : rpan[pl]) +
                   S.relidx[ri];
        }
        if (S.check && (slot < 0 || slot >= S.storage)) ok = false;
        if (!ok) {
          set_error(S.err, DEV_CHECK, K);
          continue;
        }
        atomic_add_s(dst + slot, scale_s(acc[i][j], -1.0));
      }
    __syncthreads();
  }
}

// D(i, j) = D(j, i) for i < j of the diagonal block of each task's
// supernode: 32 x 32 tiles of the upper triangle staged through shared
// memory (coalesced on both sides)
template <typename T>
__global__ void __launch_bounds__(kThreads)
mirror_lower_kernel(SymDev S, T* store, const SnTask* __restrict__ tasks, int ntasks) {
  __shared__ T tile[kTile][kTile + 1];
  const int lx = threadIdx.x & 31, ly = threadIdx.x >> 5;
  for (int t = blockIdx.x; t < ntasks; t += gridDim.x) {
    const SnTask task = tasks[t];
    const int s = S.sn_width[task.K];
    T* D = store + (int64_t)task.inst * S.storage + S.sn_off[task.K];
    const int nb = (s + kTile - 1) / kTile;
    for (int bj = 0; bj < nb; bj++)
      for (int bi = 0; bi <= bj; bi++) {
        // source: rows bj*32.., columns bi*32.. (on or below the diagonal)
        for (int r = ly; r < kTile; r += kThreads / 32) {
          const int row = bj * kTile + lx, col = bi * kTile + r;
          if (row < s && col < s) tile[r][lx] = D[row + (int64_t)col * s];
        }
        __syncthreads();
        // destination: rows bi*32.., columns bj*32.., entries above the diagonal
        for (int r = ly; r < kTile; r += kThreads / 32) {
          const int row = bi * kTile + lx, col = bj * kTile + r;
          if (row < s && col < s && row < col) D[row + (int64_t)col * s] = tile[lx][r];
        }
        __syncthreads();
      }
  }
}

template <typename T>
__global__ void __launch_bounds__(kThreads)
copy_kernel(const CopySeg* __restrict__ segs, int nseg) {
  for (int s = blockIdx.y; s < nseg; s += gridDim.y) {
    const CopySeg g = segs[s];
    const T* a = (const T*)g.src;
    T* b = (T*)g.dst;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < g.count;
         e += (int64_t)gridDim.x * blockDim.x)
      b[e] = a[e];
  }
}

template <typename T>
__global__ void __launch_bounds__(kThreads)
extract_kernel(SymDev S, const T* __restrict__ store, T* out) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < S.nnz;
       p += (int64_t)gridDim.x * blockDim.x)
    out[p] = store[S.out_map[p]];
}

// Pole-expansion consumers (a weighted sum over the instances of a batch).
// out[p] = sum_b w_b Ainv_b at entry p of pattern(A).
template <typename T>
__global__ void __launch_bounds__(kThreads)
weighted_sum_kernel(SymDev S, const T* __restrict__ store, int nb, const T* __restrict__ w,
                    T* out) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < S.nnz;
       p += (int64_t)gridDim.x * blockDim.x) {
    const int64_t slot = S.out_map[p];
    T acc = sc_zero(T());
    for (int b = 0; b < nb; b++) acc = add_s(acc, mul_s(w[b], store[b * S.storage + slot]));
    out[p] = acc;
  }
}

// Partial sums of sum_b w_b sum_p B[p] Ainv_b(j, i) for entry p = (i, j) of
// pattern(A) (tslot[p] = storage slot of the transposed entry): a fixed grid
// and a fixed reduction order, so the result does not depend on timing.
constexpr int kTraceBlocks = 1024;
template <typename T>
__global__ void __launch_bounds__(kThreads)
trace_partial_kernel(SymDev S, const T* __restrict__ store, int nb, const T* __restrict__ w,
                     const T* __restrict__ B, const int64_t* __restrict__ tslot, T* partial) {
  __shared__ T red[kThreads];
  T acc = sc_zero(T());
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < S.nnz;
       p += (int64_t)gridDim.x * blockDim.x) {
    const int64_t slot = tslot[p];
    T x = sc_zero(T());
    for (int b = 0; b < nb; b++) x = add_s(x, mul_s(w[b], store[b * S.storage + slot]));
    acc = add_s(acc, mul_s(B[p], x));
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int h = kThreads / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] = add_s(red[threadIdx.x], red[threadIdx.x + h]);
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

template <typename T>
__global__ void __launch_bounds__(kThreads) trace_final_kernel(const T* __restrict__ partial, T* out) {
  __shared__ T red[kThreads];
  T acc = sc_zero(T());
  for (int i = threadIdx.x; i < kTraceBlocks; i += kThreads) acc = add_s(acc, partial[i]);
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int h = kThreads / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] = add_s(red[threadIdx.x], red[threadIdx.x + h]);
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0];
}

// Algorithm 1 steps 3-5 of an FP64 level in one launch: nothing of G is
// stored.  A task owns the tile [r0, r0 + nr) x [j0, j0 + nw) of one
// supernode's outputs.
//   side 0 (step 3): X = -G(r, :) Lhat(:, j) into Ainv(R_U, K), and step 4's
//     share of these rows, Ainv_KK(:, j) -= Uhat(:, r) X, atomically (D_K
//     written there by the normalisation);
//   side 1 (step 5): -G(:, r)^T Uhat^T(:, j) into Ainv(K, R_L)^T.
// A symmetric A has side 0 only and writes its tile to both panels.  The
// contraction runs in chunks of kLevelK, software pipelined: while a chunk is
// multiplied, the next one's entries of G are on their way from the
// ancestors' blocks (storage bases per position, as in scatter_sub_kernel) and
// the bases of the one after.  Entries of G stored along r are read with
// lanes along r, the others with lanes along k; most chunks hold only one
// kind.  Tiles of few outputs split the contraction over `kg` groups of
// threads.
// Small levels are bound by latency (launch, task, bases, relative index,
// value, then the chain of FP64 operations at 64 cycles each), larger ones by
// the FP64 pipe (17 cycles per warp operation and SM, 1.18 TFLOP/s: 24^3
// upwind's levels of 700 Mflop run at 1.06).  Tiles of 32 x 16 and 32 x 32 with 256
// threads were slower at every size (five 2D grids: 2.38, 2.56, 2.81 ms), without
// the pipelining 2.66; a kernel that held all of G of a supernode took 2.45 with
// the levels that did not fit on the product launches (sweep 3.67 -> 2.92).
// Five CTAs per SM (95 registers) against four: 3.76 / 3.96 ms on 24^3 upwind;
// complex values spill at five.
template <typename T>
__global__ void __launch_bounds__(kLevelThreads, sizeof(T) == 8 ? 5 : 4)
small_level_kernel(SymDev S, T* store, const T* __restrict__ nf, const LevelTask* __restrict__ tasks,
                   int nbatch, int sym) {
  constexpr int NT = kLevelThreads, TP = kLevelTile;
  constexpr int NG = TP * kLevelK / NT, NB = NG, NC = TP * TP / NT;
  extern __shared__ __align__(16) unsigned char small_smem[];
  __shared__ int64_t rdiag[TP], rpan[TP], rrel[TP];
  __shared__ int64_t kdiag[2][kLevelK], kpan[2][kLevelK], krel[2][kLevelK];
  __shared__ int rsn[TP], ksn[2][kLevelK];
  const LevelTask t = tasks[blockIdx.x];
  const int tid = threadIdx.x;
  const int nr = t.nr, nw = t.nw, s = t.s;
  const bool side = t.side != 0;
  const int kt = side ? t.cu : t.c;  // length of the contraction
  const int kc = min(kt, kLevelK), ldr = nr | 1, ldw = nw | 1, si = min(s, kLevelK);
  T* const sG = reinterpret_cast<T*>(small_smem);  // [k][r]
  T* const sB = sG + kc * ldr;                     // [k][j]
  T* const sU = sB + kc * ldw;                     // [i][r]
  T* const sX = sU + si * ldr;                     // [j][r], and the partial sums of kg groups
  const unsigned mr = (65536u + nr - 1) / nr;      // e / nr = e mr >> 16 for e < 2048
  // bases of the positions of R_U (rows of G) and R_L (its columns): of the
  // tile's r and of the contraction's k
  const int64_t* const g_kpan = side ? S.row_pan + t.ru : S.col_pan + t.rl;
  const int64_t* const g_krel = side ? S.row_rel + t.ru : S.col_rel + t.rl;
  const int32_t* const g_ksn = side ? S.row_sn + t.ru : S.col_sn + t.rl;
  const int O = nr * nw;
  const int kg = O * 2 <= NT ? min(min(NT / O, 8), kt) : 1;
  const int g = kg > 1 ? tid / O : 0;
  // outputs of the warp's threads (uniform over the warp: out-of-range lanes
  // repeat the last output)
  const int wbase = tid & ~31;
  const int cnt = kg > 1 ? (g < kg) : (wbase < O ? (O - wbase + NT - 1) / NT : 0);
  int er[NC], ej[NC];
#pragma unroll
  for (int i = 0; i < NC; i++) {
    const int e = min((kg > 1 ? tid - g * O : tid) + i * NT, O - 1);
    ej[i] = (int)(e * mr >> 16);
    er[i] = e - ej[i] * nr;
  }
  for (int inst = blockIdx.y; inst < nbatch; inst += gridDim.y) {
    const int64_t base = (int64_t)inst * S.storage;
    const T* const src = store + base;
    const int64_t so = base + t.off, lo = so + (int64_t)s * s, uo = lo + (int64_t)t.c * s;
    const T* const B = nf + (side ? uo : lo) + (int64_t)t.j0 * kt;
    const T* const U4 = nf + (sym ? lo : uo) + t.r0;
    const int ld4 = t.cu;
    int64_t t_diag = 0, t_pan = 0, t_rel = 0;
    int t_sn = 0;
    T breg[NB], va[NG], vb[NG];  // vb: entries stored along k
    unsigned have = 0;           // entries of va (bits 0 ..) and vb (bits 16 ..) in flight
    auto load_bases = [&](int k0) {
      const int k = k0 + tid;
      if (tid >= kc || k >= kt) return;
      t_pan = g_kpan[k];
      t_rel = g_krel[k];
      t_sn = g_ksn[k];
      if (!side) t_diag = S.col_diag[t.rl + k];
    };
    auto store_bases = [&](int buf) {
      if (tid >= kc) return;
      kpan[buf][tid] = t_pan;
      krel[buf][tid] = t_rel;
      ksn[buf][tid] = t_sn;
      kdiag[buf][tid] = t_diag;
    };
    auto load_b = [&](int k0) {
      const int kn = min(kc, kt - k0);
      const unsigned mk = (65536u + kn - 1) / kn;
#pragma unroll
      for (int i = 0; i < NB; i++) {
        const int e = tid + i * NT, j = (int)(e * mk >> 16), k = e - j * kn;
        if (j < nw) breg[i] = B[k0 + k + (int64_t)j * kt];
      }
    };
    // the chunk's entries of G into registers: (r, k) is stored with r's block
    // (contiguous along k) or with k's (contiguous along r)
    auto slot_of = [&](bool with_r, int r, int k, int k0, int buf) -> int64_t {
      const int64_t ri = with_r ? rrel[r] + k0 + k : krel[buf][k] + t.r0 + r;
      if (S.check && (ri < 0 || ri >= S.relidx_size)) return -1;
      const bool dg = rsn[r] == ksn[buf][k];
      return (with_r ? (dg ? rdiag[r] : rpan[r]) : (dg ? kdiag[buf][k] : kpan[buf][k])) +
             S.relidx[ri];
    };
    auto gather = [&](int k0, int buf) {
      const int kn = min(kc, kt - k0), n = nr * kn;
      const unsigned mk = (65536u + kn - 1) / kn;
      // positions ascend with the supernodes: side 0 stores (r, k) with r where
      // k's supernode is the later one, side 1 where it is not the earlier one
      const int rf = rsn[0], rl = rsn[nr - 1], kf = ksn[buf][0], kl = ksn[buf][kn - 1];
      const bool any_r = side ? rf <= kl : kl > rf, any_k = side ? rl > kf : kf <= rl;
      int64_t slot[2 * NG];
      have = 0;
#pragma unroll
      for (int u = 0; u < 2 * NG; u++) {
        const bool with_r = u >= NG;
        slot[u] = -1;
        if (with_r ? !any_r : !any_k) continue;
        const int e = tid + (u % NG) * NT;
        if (e >= n) continue;
        const int hi = (int)(e * (with_r ? mk : mr) >> 16), lw = e - hi * (with_r ? kn : nr);
        const int r = with_r ? hi : lw, k = with_r ? lw : hi;
        const int a = rsn[r], b = ksn[buf][k];
        if ((side ? a <= b : b > a) != with_r) continue;
        slot[u] = slot_of(with_r, r, k, k0, buf);
        if (S.check && (slot[u] < 0 || slot[u] >= S.storage)) {
          set_error(S.err, DEV_CHECK, t.K);
          slot[u] = 0;
        }
        have |= 1u << (with_r ? 16 + u - NG : u);
      }
#pragma unroll
      for (int u = 0; u < NG; u++) {
        if (slot[u] >= 0) va[u] = src[slot[u]];
        if (slot[NG + u] >= 0) vb[u] = src[slot[NG + u]];
      }
    };
    load_bases(0);
    load_b(0);
    if (tid < nr) {
      rpan[tid] = (side ? S.col_pan + t.rl : S.row_pan + t.ru)[t.r0 + tid];
      rrel[tid] = (side ? S.col_rel + t.rl : S.row_rel + t.ru)[t.r0 + tid];
      rsn[tid] = (side ? S.col_sn + t.rl : S.row_sn + t.ru)[t.r0 + tid];
      if (side) rdiag[tid] = S.col_diag[t.rl + t.r0 + tid];
    }
    if (!side)
      for (int e = tid; e < nr * si; e += NT) {
        const int i = (int)(e * mr >> 16), r = e - i * nr;
        sU[i * ldr + r] = U4[r + (int64_t)i * ld4];
      }
    store_bases(0);
    __syncthreads();
    gather(0, 0);
    load_bases(kc);
    T acc[NC];
#pragma unroll
    for (int i = 0; i < NC; i++) acc[i] = sc_zero(T());
    for (int k0 = 0, buf = 0; k0 < kt; k0 += kc, buf ^= 1) {
      const int kn = min(kc, kt - k0);
      const unsigned mk = (65536u + kn - 1) / kn;
#pragma unroll
      for (int i = 0; i < NB; i++) {
        const int e = tid + i * NT, j = (int)(e * mk >> 16), k = e - j * kn;
        if (j < nw) sB[k * ldw + j] = breg[i];
      }
#pragma unroll
      for (int u = 0; u < NG; u++) {
        const int e = tid + u * NT;
        if (have >> u & 1) {
          const int k = (int)(e * mr >> 16), r = e - k * nr;
          sG[k * ldr + r] = va[u];
        }
        if (have >> (16 + u) & 1) {
          const int r = (int)(e * mk >> 16), k = e - r * kn;
          sG[k * ldr + r] = vb[u];
        }
      }
      store_bases(buf ^ 1);
      __syncthreads();
      if (k0 + kc < kt) {
        gather(k0 + kc, buf ^ 1);
        load_b(k0 + kc);
        load_bases(k0 + 2 * kc);
      }
      auto dots = [&](auto count) {
        constexpr int C = decltype(count)::value;
        const T* pg = sG + g * ldr;
        const T* pb = sB + g * ldw;
#pragma unroll 4
        for (int k = g; k < kn; k += kg) {
#pragma unroll
          for (int i = 0; i < C; i++) acc[i] = fma_s(pg[er[i]], pb[ej[i]], acc[i]);
          pg += kg * ldr;
          pb += kg * ldw;
        }
      };
      if (cnt == 1) dots(std::integral_constant<int, 1>());
      else if (cnt == 2) dots(std::integral_constant<int, 2>());
      __syncthreads();
    }
    if (kg > 1) {
      if (g < kg) sX[tid] = acc[0];
      __syncthreads();
      if (tid < O)
        for (int i = 1; i < kg; i++) acc[0] = add_s(acc[0], sX[i * O + tid]);
      __syncthreads();
    }
    {
      const int ldo = side ? t.c : t.cu;
      T* out = store + (side != (S.general != 0) ? uo : lo) + t.r0 + (int64_t)t.j0 * ldo;
      T* out2 = store + uo + t.r0 + (int64_t)t.j0 * ldo;
#pragma unroll
      for (int i = 0; i < NC; i++) {
        const int e = tid + i * NT;
        if (e >= O) break;
        const int j = (int)(e * mr >> 16), r = e - j * nr;
        const T x = scale_s(acc[i], -1.0);
        out[r + (int64_t)j * ldo] = x;
        if (sym) out2[r + (int64_t)j * ldo] = x;
        sX[j * ldr + r] = x;
      }
    }
    if (!side) {
      // step 4: i0 .. i0 + in - 1 of the diagonal block's rows at a time
      for (int i0 = 0; i0 < s; i0 += si) {
        const int in = min(si, s - i0);
        if (i0 > 0) {
          __syncthreads();
          for (int e = tid; e < nr * in; e += NT) {
            const int i = (int)(e * mr >> 16), r = e - i * nr;
            sU[i * ldr + r] = U4[r + (int64_t)(i0 + i) * ld4];
          }
        }
        __syncthreads();
        const unsigned mi = (65536u + in - 1) / in;
        const int n4 = in * nw, rg = n4 * 2 <= NT ? min(min(NT / n4, 4), nr) : 1;
        T* const D = store + so + i0 + (int64_t)t.j0 * s;
        for (int e4 = tid; e4 < n4 * rg; e4 += NT) {
          const int grp = rg > 1 ? e4 / n4 : 0, e = e4 - grp * n4;
          const int j = (int)(e * mi >> 16), i = e - j * in;
          T a = sc_zero(T()), b = sc_zero(T());
          const T* pu = sU + i * ldr;
          const T* px = sX + j * ldr;
          int r = grp;
          for (; r + rg < nr; r += 2 * rg) {
            a = fma_s(pu[r], px[r], a);
            b = fma_s(pu[r + rg], px[r + rg], b);
          }
          if (r < nr) a = fma_s(pu[r], px[r], a);
          atomic_add_s(D + i + (int64_t)j * s, scale_s(add_s(a, b), -1.0));
        }
      }
    }
    __syncthreads();
  }
}

int grid_for(int64_t n) {
  const int64_t g = (n + kThreads - 1) / kThreads;
  return (int)(g < 152 * 16 ? (g > 0 ? g : 1) : 152 * 16);
}

}  // namespace

void launch_scatter_values(int dtype, const SymDev& S, const void* values, void* store,
                           int nbatch, cudaStream_t st) {
  const int64_t total = (int64_t)nbatch * S.nnz;
  if (total == 0) return;
  if (dtype == DT_F64)
    scatter_values_kernel<double><<<grid_for(total), kThreads, 0, st>>>(S, (const double*)values,
                                                                      (double*)store, total);
  else
    scatter_values_kernel<cdouble><<<grid_for(total), kThreads, 0, st>>>(
        S, (const cdouble*)values, (cdouble*)store, total);
}

size_t small_level_smem(int dtype, const LevelTask& t) {
  const int kt = t.side ? t.cu : t.c, kc = kt < kLevelK ? kt : kLevelK, si = t.s < kLevelK ? t.s : kLevelK;
  const int ldr = t.nr | 1, ldw = t.nw | 1;
  // the partial sums of kg <= 8 groups (at most 256 of them) share the tile X
  const int part = 8 * t.nr * t.nw < 256 ? 8 * t.nr * t.nw : 256;
  const int x = ldr * t.nw > part ? ldr * t.nw : part;
  return (size_t)(kc * ldr + kc * ldw + si * ldr + x) * (dtype == DT_F64 ? 8 : 16);
}

void launch_small_level(int dtype, const SymDev& S, void* store, const void* nf,
                        const LevelTask* tasks, int ntasks, int nbatch, size_t smem, int sym,
                        cudaStream_t st) {
  if (ntasks <= 0) return;
  const dim3 grid((unsigned)ntasks, (unsigned)(nbatch < 65535 ? nbatch : 65535));
  if (dtype == DT_F64)
    small_level_kernel<double><<<grid, kLevelThreads, smem, st>>>(
        S, (double*)store, (const double*)nf, tasks, nbatch, sym);
  else
    small_level_kernel<cdouble><<<grid, kLevelThreads, smem, st>>>(
        S, (cdouble*)store, (const cdouble*)nf, tasks, nbatch, sym);
}

void launch_gather(int dtype, const SymDev& S, const void* store, void* out, const int64_t* gofs,
                   const SnTask* tasks, int ntasks, cudaStream_t st, const int64_t* mofs,
                   unsigned long long* maxbase) {
  if (ntasks <= 0) return;
  const int grid = ntasks < 152 * 8 ? ntasks : 152 * 8;
  if (dtype == DT_F64)
    gather_kernel<double><<<grid, kThreads, 0, st>>>(S, (const double*)store, (double*)out, gofs,
                                                     tasks, ntasks, mofs, maxbase);
  else
    gather_kernel<cdouble><<<grid, kThreads, 0, st>>>(S, (const cdouble*)store, (cdouble*)out,
                                                      gofs, tasks, ntasks, nullptr, nullptr);
}

void launch_scatter_sub(int dtype, const SymDev& S, void* store, const void* src,
                        const int64_t* sofs, const SnTask* tasks, int ntasks, bool lower,
                        cudaStream_t st) {
  if (ntasks <= 0) return;
  const int grid = ntasks < 152 * 8 ? ntasks : 152 * 8;
  if (dtype == DT_F64) {
    if (lower)
      scatter_sub_kernel<double, false, true><<<grid, kThreads, 0, st>>>(
          S, (double*)store, (const double*)src, sofs, tasks, ntasks);
    else
      scatter_sub_kernel<double><<<grid, kThreads, 0, st>>>(S, (double*)store,
                                                            (const double*)src, sofs, tasks, ntasks);
  } else {
    if (lower)
      scatter_sub_kernel<cdouble, false, true><<<grid, kThreads, 0, st>>>(
          S, (cdouble*)store, (const cdouble*)src, sofs, tasks, ntasks);
    else
      scatter_sub_kernel<cdouble><<<grid, kThreads, 0, st>>>(
          S, (cdouble*)store, (const cdouble*)src, sofs, tasks, ntasks);
  }
}

namespace {
template <typename T, int TS>
void schur_launch_t(const SymDev& S, void* store, const SchurDesc* descs, const SchurTask* tasks,
                    int ntasks, bool lower, cudaStream_t st) {
  if (S.general)
    schur_scatter_kernel<T, TS, false, true><<<ntasks, kThreads, 0, st>>>(S, (T*)store, descs, tasks,
                                                                          ntasks);
  else if (lower)
    schur_scatter_kernel<T, TS, true, false><<<ntasks, kThreads, 0, st>>>(S, (T*)store, descs, tasks,
                                                                          ntasks);
  else
    schur_scatter_kernel<T, TS, false, false><<<ntasks, kThreads, 0, st>>>(S, (T*)store, descs,
                                                                           tasks, ntasks);
}
}  // namespace

void launch_schur_scatter(int dtype, const SymDev& S, void* store, const SchurDesc* descs,
                          const SchurTask* tasks, int ntasks, int tile, bool lower,
                          cudaStream_t st) {
  if (ntasks <= 0) return;
  if (dtype == DT_F64) {
    if (tile == 16) schur_launch_t<double, 16>(S, store, descs, tasks, ntasks, lower, st);
    else schur_launch_t<double, 32>(S, store, descs, tasks, ntasks, lower, st);
  } else {
    if (tile == 16) schur_launch_t<cdouble, 16>(S, store, descs, tasks, ntasks, lower, st);
    else schur_launch_t<cdouble, 32>(S, store, descs, tasks, ntasks, lower, st);
  }
}

void launch_mirror_lower(int dtype, const SymDev& S, void* store, const SnTask* tasks, int ntasks,
                         cudaStream_t st) {
  if (ntasks <= 0) return;
  const int grid = ntasks < 152 * 8 ? ntasks : 152 * 8;
  if (dtype == DT_F64)
    mirror_lower_kernel<double><<<grid, kThreads, 0, st>>>(S, (double*)store, tasks, ntasks);
  else
    mirror_lower_kernel<cdouble><<<grid, kThreads, 0, st>>>(S, (cdouble*)store, tasks, ntasks);
}

void launch_gather_general(int dtype, const SymDev& S, const void* store, void* out,
                           const int64_t* gofs, const SnTask* tasks, int ntasks, cudaStream_t st) {
  if (ntasks <= 0) return;
  const int grid = ntasks < 152 * 8 ? ntasks : 152 * 8;
  if (dtype == DT_F64)
    gather_general_kernel<double><<<grid, kThreads, 0, st>>>(S, (const double*)store,
                                                             (double*)out, gofs, tasks, ntasks);
  else
    gather_general_kernel<cdouble><<<grid, kThreads, 0, st>>>(S, (const cdouble*)store,
                                                              (cdouble*)out, gofs, tasks, ntasks);
}

void launch_scatter_sub_general(int dtype, const SymDev& S, void* store, const void* src,
                                const int64_t* sofs, const SnTask* tasks, int ntasks,
                                cudaStream_t st) {
  if (ntasks <= 0) return;
  const int grid = ntasks < 152 * 8 ? ntasks : 152 * 8;
  if (dtype == DT_F64)
    scatter_sub_general_kernel<double><<<grid, kThreads, 0, st>>>(
        S, (double*)store, (const double*)src, sofs, tasks, ntasks);
  else
    scatter_sub_general_kernel<cdouble><<<grid, kThreads, 0, st>>>(
        S, (cdouble*)store, (const cdouble*)src, sofs, tasks, ntasks);
}

void launch_scatter_set(int dtype, const SymDev& S, void* store, const void* src,
                        const int64_t* sofs, const SnTask* tasks, int ntasks, cudaStream_t st) {
  if (ntasks <= 0) return;
  const int grid = ntasks < 152 * 8 ? ntasks : 152 * 8;
  if (dtype == DT_F64)
    scatter_sub_kernel<double, true><<<grid, kThreads, 0, st>>>(
        S, (double*)store, (const double*)src, sofs, tasks, ntasks);
  else
    scatter_sub_kernel<cdouble, true><<<grid, kThreads, 0, st>>>(
        S, (cdouble*)store, (const cdouble*)src, sofs, tasks, ntasks);
}

void launch_copy(int dtype, const CopySeg* segs, int nseg, int per_seg, cudaStream_t st) {
  if (nseg <= 0) return;
  dim3 grid(per_seg > 0 ? per_seg : 8, nseg < 65535 ? nseg : 65535);
  if (dtype == DT_F64)
    copy_kernel<double><<<grid, kThreads, 0, st>>>(segs, nseg);
  else
    copy_kernel<cdouble><<<grid, kThreads, 0, st>>>(segs, nseg);
}

void launch_extract(int dtype, const SymDev& S, const void* store, int inst, void* out,
                    cudaStream_t st) {
  if (S.nnz == 0) return;
  if (dtype == DT_F64)
    extract_kernel<double><<<grid_for(S.nnz), kThreads, 0, st>>>(
        S, (const double*)store + (int64_t)inst * S.storage, (double*)out);
  else
    extract_kernel<cdouble><<<grid_for(S.nnz), kThreads, 0, st>>>(
        S, (const cdouble*)store + (int64_t)inst * S.storage, (cdouble*)out);
}

void launch_weighted_sum(int dtype, const SymDev& S, const void* store, int nb, const void* w,
                         void* out, cudaStream_t st) {
  if (S.nnz == 0) return;
  if (dtype == DT_F64)
    weighted_sum_kernel<double><<<grid_for(S.nnz), kThreads, 0, st>>>(
        S, (const double*)store, nb, (const double*)w, (double*)out);
  else
    weighted_sum_kernel<cdouble><<<grid_for(S.nnz), kThreads, 0, st>>>(
        S, (const cdouble*)store, nb, (const cdouble*)w, (cdouble*)out);
}

void launch_trace(int dtype, const SymDev& S, const void* store, int nb, const void* w,
                  const void* B, const int64_t* tslot, void* partial, void* out, cudaStream_t st) {
  if (dtype == DT_F64) {
    trace_partial_kernel<double><<<kTraceBlocks, kThreads, 0, st>>>(
        S, (const double*)store, nb, (const double*)w, (const double*)B, tslot, (double*)partial);
    trace_final_kernel<double><<<1, kThreads, 0, st>>>((const double*)partial, (double*)out);
  } else {
    trace_partial_kernel<cdouble><<<kTraceBlocks, kThreads, 0, st>>>(
        S, (const cdouble*)store, nb, (const cdouble*)w, (const cdouble*)B, tslot,
        (cdouble*)partial);
    trace_final_kernel<cdouble><<<1, kThreads, 0, st>>>((const cdouble*)partial, (cdouble*)out);
  }
}

size_t trace_partial_bytes() { return (size_t)kTraceBlocks * 16; }

}  // namespace pselinv
