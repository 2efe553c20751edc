// Dense block kernels in FP64 / complex128:
//   * a batched, persistent GEMM over a task list (the block products of
//     Algorithm 1 steps 2-5 and of the supernodal LU),
//   * the panel steps of the blocked LU without pivoting of diagonal blocks
//     and of their triangular inverses.
//
// On GB300 the FP64 rate is the same for DFMA and the FP64 MMA path (about
// 4 flop/clk/SM), so the FP64 GEMM is a register-tiled SIMT DFMA kernel:
// it saturates the FP64 pipe with a 16x16 thread grid and 4x4 (real) or
// 2x2 (complex) outputs per thread.
#include <algorithm>
#include <type_traits>

#include "device.cuh"

namespace pselinv {

namespace {

constexpr int kThreads = 256;

template <typename T, int BM, int BN, int BK>
struct GemmSmem {
  T a[BK][BM];
  T b[BK][BN];
};

template <typename T, int BM, int BN, int BK>
__global__ void __launch_bounds__(kThreads)
gemm_kernel(const GemmDesc* __restrict__ descs, const GemmTask* __restrict__ tasks, int ntasks) {
  constexpr int TM = BM / 16, TN = BN / 16;
  __shared__ GemmSmem<T, BM, BN, BK> sm;
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  for (int t = blockIdx.x; t < ntasks; t += gridDim.x) {
    const GemmTask task = tasks[t];
    const GemmDesc d = descs[task.d];
    const T* __restrict__ A = (const T*)d.A;
    const T* __restrict__ B = (const T*)d.B;
    T* __restrict__ C = (T*)d.C;
    const int m0 = task.tm * BM, n0 = task.tn * BN;
    int kchunk = (d.K + d.ksplit - 1) / d.ksplit;
    kchunk = (kchunk + BK - 1) / BK * BK;
    int kb = task.ks * kchunk;
    int ke = min(d.K, kb + kchunk);
    if (d.tri & GEMM_TRI_LOWER_B) kb = max(kb, n0);
    if (d.tri & GEMM_TRI_UPPER_A) kb = max(kb, m0);
    if (d.tri & GEMM_TRI_UPPER_B) ke = min(ke, n0 + BN);
    if (d.tri & GEMM_TRI_LOWER_A) ke = min(ke, m0 + BM);
    T acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; i++)
#pragma unroll
      for (int j = 0; j < TN; j++) acc[i][j] = sc_zero(T());
    // the next K tile is loaded into registers while the current one is
    // used from shared memory
    constexpr int NA = BM * BK / kThreads, NB = BK * BN / kThreads;
    T ra[NA], rb[NB];
    auto load_tiles = [&](int k0) {
#pragma unroll
      for (int q = 0; q < NA; q++) {
        const int e = tid + q * kThreads;
        int mm, kk;
        if (d.transA) { kk = e % BK; mm = e / BK; } else { mm = e % BM; kk = e / BM; }
        const int m = m0 + mm, k = k0 + kk;
        T v = sc_zero(T());
        if (m < d.M && k < ke)
          v = d.transA ? A[k + (int64_t)m * d.lda] : A[m + (int64_t)k * d.lda];
        ra[q] = v;
      }
#pragma unroll
      for (int q = 0; q < NB; q++) {
        const int e = tid + q * kThreads;
        int kk, nn;
        if (d.transB) { nn = e % BN; kk = e / BN; } else { kk = e % BK; nn = e / BK; }
        const int n = n0 + nn, k = k0 + kk;
        T v = sc_zero(T());
        if (n < d.N && k < ke)
          v = d.transB ? B[n + (int64_t)k * d.ldb] : B[k + (int64_t)n * d.ldb];
        rb[q] = v;
      }
    };
    if (kb < ke) load_tiles(kb);
    for (int k0 = kb; k0 < ke; k0 += BK) {
#pragma unroll
      for (int q = 0; q < NA; q++) {
        const int e = tid + q * kThreads;
        if (d.transA) sm.a[e % BK][e / BK] = ra[q]; else sm.a[e / BM][e % BM] = ra[q];
      }
#pragma unroll
      for (int q = 0; q < NB; q++) {
        const int e = tid + q * kThreads;
        if (d.transB) sm.b[e / BN][e % BN] = rb[q]; else sm.b[e % BK][e / BK] = rb[q];
      }
      __syncthreads();
      if (k0 + BK < ke) load_tiles(k0 + BK);
#pragma unroll
      for (int kk = 0; kk < BK; kk++) {
        T av[TM], bv[TN];
#pragma unroll
        for (int i = 0; i < TM; i++) av[i] = sm.a[kk][tx + 16 * i];
#pragma unroll
        for (int j = 0; j < TN; j++) bv[j] = sm.b[kk][ty + 16 * j];
#pragma unroll
        for (int i = 0; i < TM; i++)
#pragma unroll
          for (int j = 0; j < TN; j++) acc[i][j] = fma_s(av[i], bv[j], acc[i][j]);
      }
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < TM; i++) {
      const int m = m0 + tx + 16 * i;
      if (m >= d.M) continue;
#pragma unroll
      for (int j = 0; j < TN; j++) {
        const int n = n0 + ty + 16 * j;
        if (n >= d.N) continue;
        T* c = C + m + (int64_t)n * d.ldc;
        const T v = scale_s(acc[i][j], d.alpha);
        if (d.atomic) {
          atomic_add_s(c, v);
        } else if (d.beta != 0.0) {
          *c = add_s(v, scale_s(*c, d.beta));
        } else {
          *c = v;
        }
      }
    }
  }
}

// Panel step of the blocked LU without pivoting of the supernodes' diagonal
// blocks (right-looking, panels of 32 columns; the trailing update A22 -=
// L21 U12 is a GEMM launch of its own).  A task {inst, K, j0, line0} factors
// the w x w pivot block at (j0, j0), w = min(32, s - j0), in registers and
// eliminates 32 G "lines" beside it.  The lines of a panel, in order:
//   nl rows of L21 (X U11 = A21), nl columns of U12 (L11 Y = A12): the rest of
//      the diagonal block (s > 32: nl = s - j0 - w, in place);
//   for a narrow supernode (s <= 32, one panel; solve = 1) instead the c rows
//      of its L panel and the cu rows of its U^T panel, so that its triangular
//      solves need no inverse and no launch of their own (symmetric values: no
//      U^T lines, an L line's unscaled entries are the row of U^T).  Levels with
//      sliced panel solves leave them to those (solve = 0): 64 lines a block
//      instead of 64 + c + cu (20 complex shifts of a 16^3 operator, a level of
//      660 tasks: 352 -> 242 us);
//   w unit rows and w unit columns: U11^{-1} and L11^{-1} into winv.
// Every task of a panel factors the pivot block again (the FP64 pipe takes
// 64 cycles per warp instruction whatever the mask, so the pivot block's
// chain, not its work, is what a panel waits for, and a second launch would
// wait for it twice).  The task with line0 = 0 stores the factored block in
// `piv` (column j of the matrix at piv + 32 (inst n + j)); unpack_pivots moves
// it into the storage once nobody reads the unfactored block any more.
// Threads: warp 0 runs the pivot chain alone on its scheduler: an FP64
// instruction of a chain takes 64 cycles on an idle SM, 133 while the other
// three schedulers keep the pipe full and 366 when its own does too.  Warps
// 1-3 hold the pivot block (row = lane, columns 3 jj + (warp & 3) - 1),
// warps 4 g + 1 .. 4 g + 3 the lines 32 (g - 1) .. of the task (line = lane,
// entries along the panel in registers).  Step k, one block barrier: warp 0
// updates column k + 1, computes its reciprocal and the scaled column of L;
// the others apply step k to the columns behind it and publish row k + 1,
// column k + 2 and the lines' entries k + 1.
// P > 1: 32 / P lines a team and P lanes a line, columns dealt over 3 P lanes.  The
// lines' instructions share three schedulers with the pivot block's (a wide
// block's 32 lines: 22 FP64 instructions a warp in the first step), and a launch
// of a few blocks leaves most SMs idle: 8 lines a task there, 16 where 8 would
// give more than one task per SM (256 wide block, one panel: real 25.1 -> 22.0 us,
// complex 57 -> 49; 127^2 grid solve 1.93 -> 1.77 ms, 40^3 upwind 16.9 -> 16.1).
// Bound: the pivot chain (three dependent FP64 operations, a reciprocal and a
// barrier per column) and, about as long, the FP64 pipe.
template <typename T>
__device__ __forceinline__ T shfl_t(T v, int src);
template <>
__device__ __forceinline__ double shfl_t(double v, int src) {
  return __shfl_sync(0xffffffffu, v, src);
}
template <>
__device__ __forceinline__ cdouble shfl_t(cdouble v, int src) {
  return {__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src)};
}
// 1 / d in integers, as the pivot chain waits for it and an FP64 instruction
// takes 64 to 133 cycles there (three of them: 27.1 us a panel of a wide block;
// this: 25.1).  y = Y 2^-24: the FP32 reciprocal of the mantissa's
// leading bits; its residual e = 1 - m y (|e| < 2^-21, units 2^-76) is exact,
// and y (1 + e + e^2) is one third-order step of the Householder family, off by
// e^3 < 2^-63; then rounded to nearest.  Half a unit of the last place and 2^-62
// over 3 10^7 random and near-power-of-two mantissas with y moved by a unit
// either way.  Numbers near the ends of the range, zeros and non-finite ones
// take the division.
__device__ __forceinline__ double rcp_s(double d) {
  const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
  const uint32_t E = (hi >> 20) & 0x7FFu;
  if (E < 64u || E > 1982u) return 1.0 / d;
  float yf;
  asm("rcp.approx.ftz.f32 %0, %1;"
      : "=f"(yf)
      : "f"(__uint_as_float(0x3F800000u | (((hi << 3) | (lo >> 29)) & 0x7FFFFFu))));
  yf = fminf(fmaxf(yf, 0.5f), 0.99999994f);
  const uint32_t Y = (__float_as_uint(yf) & 0x7FFFFFu) | 0x800000u;
  const uint64_t M = ((uint64_t)((hi & 0xFFFFFu) | 0x100000u) << 32) | lo;
  const int64_t e = -(int64_t)(M * Y);  // 2^76 - M Y, which fits 64 bits
  const int64_t eh = (int32_t)(e >> 32);
  const int64_t c = e + ((eh * eh) >> 12);
  const int64_t yc = (int64_t)(int32_t)(c >> 32) * (int64_t)Y +
                     (int64_t)(((uint64_t)(uint32_t)c * Y) >> 32);  // units 2^-68
  const uint64_t r = ((uint64_t)Y << 40) + (uint64_t)(yc >> 4);       // units 2^-64
  const uint64_t bits = ((uint64_t)(2044u - E) << 52) + (r >> 11) + ((r >> 10) & 1u);
  return __longlong_as_double((long long)(bits | ((uint64_t)(hi & 0x80000000u) << 32)));
}
__device__ __forceinline__ cdouble rcp_s(cdouble b) {
  const int ex = (__double2hiint(b.x) >> 20) & 0x7FF, ey = (__double2hiint(b.y) >> 20) & 0x7FF;
  const int e = max(ex, ey);
  if (e < 640 || e > 1400) return div_s(sc_one(cdouble()), b);  // |b|^2 could leave the range
  const double r = rcp_s(fma(b.x, b.x, b.y * b.y));
  return {b.x * r, -b.y * r};
}
__device__ __forceinline__ double fnma_s(double a, double b, double c) { return fma(-a, b, c); }
__device__ __forceinline__ cdouble fnma_s(cdouble a, cdouble b, cdouble c) {
  return {fma(-a.x, b.x, fma(a.y, b.y, c.x)), fma(-a.x, b.y, fma(-a.y, b.x, c.y))};
}

constexpr int kLuW = kLuPanel;  // panel width
// lines of a task: G teams of 32 / P lines, P lanes a line
template <int G, int P>
constexpr int kLuLines = 32 / P * G;
template <typename T, int G, int P>
__global__ void __launch_bounds__(128 * (G + 1))
lu_panel_kernel(SymDev S, T* store, T* winv, T* piv, const LuTask* __restrict__ tasks, int solve,
                int sym) {
  constexpr int kThr = 128 * (G + 1), kLines = kLuLines<G, P>;
  extern __shared__ __align__(16) unsigned char lu_smem[];
  T(*Dd)[kLuW + 1] = reinterpret_cast<T(*)[kLuW + 1]>(lu_smem);  // A11, then the rows of U11
  T(*Ls)[kLuW + 1] = Dd + kLuW;                                  // scaled columns of L11
  T(*X)[kLuW + 1] = Ls + kLuW;                                   // lines (unscaled)
  T* R = reinterpret_cast<T*>(X + kLines);                       // reciprocals of the pivots
  T(*Cn)[kLuW] = reinterpret_cast<T(*)[kLuW]>(R + kLuW);         // the chain's next column
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int team = warp >> 2, q = (warp & 3) - 1;  // q = -1: the chain (warp 0) or idle
  const LuTask task = tasks[blockIdx.x];
  const int K = task.K, j0 = task.j0, s = S.sn_width[K], c = S.sn_c[K];
  const int w = min(kLuW, s - j0), rest = s - j0 - w;
  const bool narrow = s <= kLuW && solve;
  T* D = store + (int64_t)task.inst * S.storage + S.sn_off[K];
  T* W = winv + (int64_t)task.inst * S.w_stride + S.w_off[K];
  // line ranges and addresses: entry k of L line i at Lb[i + k ldl], of U line i
  // at Ub[i us + k uk]
  const int cu = S.general ? S.sn_cu[K] : c;
  const int nl = narrow ? c : rest, nu = narrow ? (sym ? 0 : cu) : rest;
  T* Lb = narrow ? D + s * s : D + (j0 + w) + (int64_t)j0 * s;
  const int64_t ldl = narrow ? c : s;
  T* Ub = narrow ? D + s * s + (int64_t)c * s : D + j0 + (int64_t)(j0 + w) * s;
  const int64_t us = narrow ? 1 : s, uk = narrow ? cu : 1;
  const int nlines = nl + nu + 2 * w;

  for (int e = tid; e < kLuW * kLuW; e += kThr) {
    const int i = e & (kLuW - 1), j = e / kLuW;
    // symmetric values: a narrow block's upper triangle is its lower one's
    const int si = sym && narrow && i < j ? j : i, sj = sym && narrow && i < j ? i : j;
    Dd[i][j] = i < w && j < w ? D[(j0 + si) + (int64_t)(j0 + sj) * s] : sc_zero(T());
    Ls[i][j] = sc_zero(T());
  }
  // lines: lanes along the lines (contiguous), except the columns of U12 of a
  // wide block, contiguous along k
  for (int e = tid; e < kLines * kLuW; e += kThr) {
    const int i = e % kLines, k = e / kLines, l = task.line0 + i;
    if (l >= nlines || k >= w) {
      X[i][k] = sc_zero(T());
    } else if (l < nl) {
      X[i][k] = Lb[l + k * ldl];
    } else if (l < nl + nu) {
      if (narrow) X[i][k] = Ub[(l - nl) * us + k * uk];
    } else {
      const int u = l - nl - nu;  // unit row u, or unit column u - w
      X[i][k] = (u < w ? u : u - w) == k ? sc_one(T()) : sc_zero(T());
    }
  }
  if (!narrow)
    for (int e = tid; e < kLines * kLuW; e += kThr) {
      const int k = e & 31, i = e >> 5, l = task.line0 + i;
      if (l >= nl && l < nl + nu && k < w) X[i][k] = Ub[(l - nl) * us + k * uk];
    }
  __syncthreads();
  if (warp == 0) {
    T v = Dd[lane][0], l = sc_zero(T());
    for (int k = 0; k < w; k++) {
      // column k is final (rows >= k): its reciprocal and column of L11
      if (k > 0) v = fnma_s(l, Dd[k - 1][k], k == 1 ? Dd[lane][1] : Cn[k & 1][lane]);
      const T p = shfl_t(v, k);
      const T r = rcp_s(p);
      l = mul_s(v, r);
      Ls[lane][k] = l;
      if (lane == 0) {
        R[k] = r;
        Dd[k][k] = p;
        if (is_zero(p)) set_error(S.err, DEV_ZERO_PIVOT, S.sn_first[K] + j0 + k);
      }
      __syncthreads();
    }
  } else if (q < 0 || (team > 0 && task.line0 + 32 / P * (team - 1) >= nlines)) {
    for (int k = 0; k < w; k++) __syncthreads();  // a scheduler's spare warp, or no lines left
  } else {
    const T* sm = reinterpret_cast<const T*>(lu_smem);
    constexpr int kEither = 0, kPivot = 1, kLine = 2;
    // the pivot block's warps (one lane a row), a team's (PL lanes a line), or
    // both from one loop: complex values at one lane a line, whose two copies
    // would be slower (pole solve 17.0 against 16.8 ms; real values the other way
    // round: 8^3 x 64 DG 48.95 against 49.3)
    auto eliminate = [&](auto who, auto lanes) {
      constexpr int kWho = decltype(who)::value;
      const bool piv = kWho == kEither ? team == 0 : kWho == kPivot;
      constexpr int PL = decltype(lanes)::value;
      constexpr int kCyc = 3 * PL, kCols = (kLuW + kCyc - 1) / kCyc;
      // row of Dd or of X; first column (columns qq, qq + kCyc, ...)
      const int row = piv ? lane : 32 / PL * (team - 1) + lane % (32 / PL);
      const int qq = q + 3 * (lane / (32 / PL));
      // a line's multiplier and coefficients: L lines (and unit rows) x_k r_k
      // and row k of U11, U lines (and unit columns) x_k and column k of L11
      const int line = task.line0 + row;
      const bool is_l = !piv && (line < nl || (line >= nl + nu && line < nl + nu + w));
      const bool from_u = piv || is_l;  // coefficients from the rows of U11
      const int cbase = from_u ? 0 : kLuW * (kLuW + 1);
      const int cj = from_u ? 1 : kLuW + 1, ck = from_u ? kLuW + 1 : 1;  // strides along j and k
      const bool warp_l = __any_sync(0xffffffffu, is_l);
      // a[jj] holds column kCyc (t + jj) + qq in round t (columns past the panel
      // hold values nobody uses)
      T a[kCols];
#pragma unroll
      for (int jj = 0; jj < kCols; jj++) {
        const int j = min(kCyc * jj + qq, kLuW - 1);
        a[jj] = piv ? Dd[row][j] : X[row][j];
      }
      const int nr = (w + kCyc - 1) / kCyc;
      for (int t = 0; t < nr; t++) {
        const int nj = nr - t;  // columns of this lane still in the panel
#pragma unroll
        for (int kk = 0; kk < kCyc; kk++) {
          const int k = kCyc * t + kk;
          if (k >= w) break;
          __syncthreads();  // row k of U11, column k of L11, r_k and x_k are in place
          // (rows <= k of the pivot block are final and published: their lanes run along)
          T m = piv ? Ls[lane][k] : X[row][k];
          if (warp_l) {
            const T ml = mul_s(m, R[k]);
            if (is_l) m = ml;
          }
          const T* cp = sm + cbase + (kCyc * t + qq) * cj + k * ck;
          // the pivot block's warps publish column k + 2 for the chain (which
          // has column k + 1 itself), the lines their entry k + 1
          const int ahead = piv ? 2 : 1;
          if (qq - kk >= ahead) {
            a[0] = fnma_s(m, cp[0], a[0]);
            if (qq - kk == ahead) {
              if (piv) Cn[k & 1][lane] = a[0];
              else X[row][k + 1] = a[0];
            }
          }
          if (nj > 1 && qq + kCyc - kk >= ahead) {
            a[1] = fnma_s(m, cp[kCyc * cj], a[1]);
            if (qq + kCyc - kk == ahead) {
              if (piv) Cn[k & 1][lane] = a[1];
              else X[row][k + 1] = a[1];
            }
          }
          // (jumps out: a predicated-off FP64 instruction still takes its 64 cycles)
#pragma unroll
          for (int jj = 2; jj < kCols; jj++) {
            if (jj >= nj) break;
            a[jj] = fnma_s(m, cp[kCyc * jj * cj], a[jj]);
          }
          if (piv && lane == k + 1) {  // row k + 1 of U11 right of its diagonal is final
#pragma unroll
            for (int jj = 0; jj < kCols; jj++) {
              const int j = kCyc * (t + jj) + qq;
              if (jj < nj && j > k + 1) Dd[k + 1][j] = a[jj];
            }
          }
        }
#pragma unroll
        for (int jj = 0; jj + 1 < kCols; jj++) a[jj] = a[jj + 1];
      }
    };
    using One = std::integral_constant<int, 1>;
    if constexpr (P == 1 && sizeof(T) == 16) {
      eliminate(std::integral_constant<int, kEither>(), One());
    } else {
      if (team == 0) eliminate(std::integral_constant<int, kPivot>(), One());
      else eliminate(std::integral_constant<int, kLine>(), std::integral_constant<int, P>());
    }
  }
  __syncthreads();
  if (task.line0 == 0) {
    T* Pv = piv + ((int64_t)task.inst * S.n + S.sn_first[K] + j0) * kLuW;
    for (int e = tid; e < w * w; e += kThr) {
      const int i = e % w, j = e / w;
      Pv[i + j * kLuW] = i <= j ? Dd[i][j] : Ls[i][j];
    }
  }
  for (int e = tid; e < kLines * kLuW; e += kThr) {
    const int i = e % kLines, k = e / kLines, l = task.line0 + i;
    if (l >= nlines || k >= w) continue;
    const T x = X[i][k];
    if (l < nl) {
      Lb[l + k * ldl] = mul_s(x, R[k]);
      if (sym && narrow) D[s * s + (int64_t)c * s + l + (int64_t)k * c] = x;
    } else if (l < nl + nu) {
      if (narrow) Ub[(l - nl) * us + k * uk] = x;
    } else {
      const int u = l - nl - nu;
      if (u < w)  // row u of U11^{-1}
        W[(int64_t)s * s + (j0 + u) + (int64_t)(j0 + k) * s] = k < u ? sc_zero(T()) : mul_s(x, R[k]);
      else  // column u - w of L11^{-1}
        W[(j0 + k) + (int64_t)(j0 + u - w) * s] = k < u - w ? sc_zero(T()) : x;
    }
  }
  if (!narrow)
    for (int e = tid; e < kLines * kLuW; e += kThr) {
      const int k = e & 31, i = e >> 5, l = task.line0 + i;
      if (l >= nl && l < nl + nu && k < w) Ub[(l - nl) * us + k * uk] = X[i][k];
    }
}

// The factored pivot blocks (piv, see lu_panel_kernel) into the diagonal
// blocks of the storage: one thread per entry.
template <typename T>
__global__ void __launch_bounds__(kThreads)
unpack_pivots_kernel(SymDev S, T* store, const T* __restrict__ piv, int64_t total) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t g = e / kLuW, b = g / S.n;
    const int i = (int)(e - g * kLuW), col = (int)(g - b * S.n);
    const int K = S.sn_of[col], s = S.sn_width[K], j = col - S.sn_first[K];
    const int j0 = j & ~(kLuW - 1);
    if (i < min(kLuW, s - j0))
      store[b * S.storage + S.sn_off[K] + (j0 + i) + (int64_t)j * s] = piv[e];
  }
}

// Row-panel product C(m, n) = alpha sum_k op(A)(m, k) op(B)(k, n) (+ beta
// C, or atomically added), one thread per row m and columns j0 .. j0 +
// NW - 1, k over the task's K chunk [kb, ke).  TRI = 1 (op(B) lower
// triangular, zero for k < n) or 2 (upper, zero for k > n): square op(B);
// in the diagonal block (k in [j0, j0 + NW)) only the triangle is
// multiplied, the other k of the chunk run over all NW columns.  An upper
// op(A) (GEMM_TRI_UPPER_A, with a lower op(B)) starts every warp at its
// first row.  Lanes past M read row M - 1 and columns past N read column
// N - 1 (in bounds; never stored).  FP64 throughput is the bound: the loads
// of op(B) are warp-uniform, those of A coalesced along m (or, transposed,
// one row per lane reused from L1).
template <typename T, int NW, int TRI>
__device__ __forceinline__ void rows_task(const GemmDesc& d, int m, int warp_m0, int j0, int kb,
                                          int ke) {
  const T* __restrict__ B = (const T*)d.B;
  const int mm = min(m, d.M - 1);
  const T* __restrict__ Ar = (const T*)d.A + (d.transA ? (int64_t)mm * d.lda : (int64_t)mm);
  const int64_t ak = d.transA ? 1 : d.lda;
  const int nlast = d.N - 1;
  const int64_t sk = d.transB ? d.ldb : 1, sn = d.transB ? 1 : d.ldb;
  auto bval = [&](int k, int q) { return B[(int64_t)k * sk + (int64_t)min(j0 + q, nlast) * sn]; };
  T acc[NW];
#pragma unroll
  for (int q = 0; q < NW; q++) acc[q] = sc_zero(T());
  // k in [k0, k1) over all NW columns, the operands of k + 1 loaded while
  // those of k are multiplied (a warp alone on its FP64 unit stays busy)
  auto full_range = [&](int k0, int k1) {
    if (k0 >= k1) return;
    T an = Ar[(int64_t)k0 * ak], bn[NW];
#pragma unroll
    for (int q = 0; q < NW; q++) bn[q] = bval(k0, q);
    for (int k = k0; k < k1; k++) {
      const T a = an;
      T b[NW];
#pragma unroll
      for (int q = 0; q < NW; q++) b[q] = bn[q];
      if (k + 1 < k1) {
        an = Ar[(int64_t)(k + 1) * ak];
#pragma unroll
        for (int q = 0; q < NW; q++) bn[q] = bval(k + 1, q);
      }
#pragma unroll
      for (int q = 0; q < NW; q++) acc[q] = fma_s(a, b[q], acc[q]);
    }
  };
  if (TRI == 1) {
    const int kstart = max(kb, (d.tri & GEMM_TRI_UPPER_A) ? max(j0, warp_m0) : j0);
#pragma unroll
    for (int kk = 0; kk < NW; kk++) {
      const int k = j0 + kk;
      if (k < kstart || k >= ke) continue;
      const T a = Ar[(int64_t)k * ak];
#pragma unroll
      for (int q = 0; q <= kk; q++) acc[q] = fma_s(a, bval(k, q), acc[q]);
    }
    full_range(max(j0 + NW, kstart), ke);
  } else if (TRI == 2) {
    full_range(kb, min(j0, ke));
#pragma unroll
    for (int kk = 0; kk < NW; kk++) {
      const int k = j0 + kk;
      if (k < kb || k >= ke) continue;
      const T a = Ar[(int64_t)k * ak];
#pragma unroll
      for (int q = kk; q < NW; q++) acc[q] = fma_s(a, bval(k, q), acc[q]);
    }
  } else {
    full_range(kb, ke);
  }
  if (m >= d.M) return;
  T* __restrict__ C = (T*)d.C + m;
#pragma unroll
  for (int q = 0; q < NW; q++) {
    const int n = j0 + q;
    if (n >= d.N) break;
    T v = scale_s(acc[q], d.alpha);
    if (d.atomic) {
      atomic_add_s(C + (int64_t)n * d.ldc, v);
      continue;
    }
    if (d.beta != 0.0) v = add_s(v, scale_s(C[(int64_t)n * d.ldc], d.beta));
    C[(int64_t)n * d.ldc] = v;
  }
}

template <typename T, int TRI>
__device__ __forceinline__ void rows_dispatch(const GemmDesc& d, int nw, int m, int warp_m0, int j0,
                                              int kb, int ke) {
  if (nw == 4)
    rows_task<T, 4, TRI>(d, m, warp_m0, j0, kb, ke);
  else
    rows_task<T, 8, TRI>(d, m, warp_m0, j0, kb, ke);
}

// Tasks {d, row block, column chunk, NW + 16 x K chunk index}
template <typename T>
__global__ void __launch_bounds__(kRowsBlock)
rows_gemm_kernel(const GemmDesc* __restrict__ descs, const GemmTask* __restrict__ tasks, int ntasks) {
  for (int t = blockIdx.x; t < ntasks; t += gridDim.x) {
    const GemmTask task = tasks[t];
    const GemmDesc d = descs[task.d];
    const int m = task.tm * kRowsBlock + (int)threadIdx.x;
    const int warp_m0 = m & ~31;
    if (warp_m0 >= d.M) continue;  // whole warp past the last row
    const int j0 = task.tn * kRowsChunk, nw = task.ks & 15, kc = task.ks >> 4;
    const int kchunk = (d.K + d.ksplit - 1) / d.ksplit;
    const int kb = kc * kchunk, ke = min(d.K, kb + kchunk);
    if (d.tri & GEMM_TRI_LOWER_B)
      rows_dispatch<T, 1>(d, nw, m, warp_m0, j0, kb, ke);
    else if (d.tri & GEMM_TRI_UPPER_B)
      rows_dispatch<T, 2>(d, nw, m, warp_m0, j0, kb, ke);
    else
      rows_dispatch<T, 0>(d, nw, m, warp_m0, j0, kb, ke);
  }
}

template <typename T, int BM, int BN, int BK>
void gemm_launch_t(const GemmDesc* descs, const GemmTask* tasks, int ntasks, int grid,
                   cudaStream_t st) {
  if (ntasks <= 0) return;
  gemm_kernel<T, BM, BN, BK><<<grid, kThreads, 0, st>>>(descs, tasks, ntasks);
}

}  // namespace

int gemm_tile_m(int dtype, int cfg) {
  if (cfg == GEMM_16x16) return 16;
  if (cfg == GEMM_128x64) return dtype == DT_F64 ? 128 : 64;
  if (cfg == GEMM_32x32) return 32;
  return dtype == DT_F64 ? 64 : 32;
}
int gemm_tile_n(int dtype, int cfg) {
  if (cfg == GEMM_16x16) return 16;
  if (cfg == GEMM_128x64) return dtype == DT_F64 ? 64 : 32;
  if (cfg == GEMM_32x32) return dtype == DT_F64 ? 32 : 16;
  return dtype == DT_F64 ? 64 : 32;
}

void launch_gemm(int dtype, int cfg, const GemmDesc* descs, const GemmTask* tasks, int ntasks,
                 int grid, cudaStream_t st) {
  if (cfg == GEMM_ROWS) {
    if (ntasks <= 0) return;
    if (dtype == DT_F64)
      rows_gemm_kernel<double><<<grid, kRowsBlock, 0, st>>>(descs, tasks, ntasks);
    else
      rows_gemm_kernel<cdouble><<<grid, kRowsBlock, 0, st>>>(descs, tasks, ntasks);
    return;
  }
  if (dtype == DT_F64) {
    switch (cfg) {
      case GEMM_16x16: gemm_launch_t<double, 16, 16, 32>(descs, tasks, ntasks, grid, st); break;
      case GEMM_32x32: gemm_launch_t<double, 32, 32, 16>(descs, tasks, ntasks, grid, st); break;
      case GEMM_128x64: gemm_launch_t<double, 128, 64, 8>(descs, tasks, ntasks, grid, st); break;
      default: gemm_launch_t<double, 64, 64, 16>(descs, tasks, ntasks, grid, st); break;
    }
  } else {
    switch (cfg) {
      case GEMM_16x16: gemm_launch_t<cdouble, 16, 16, 32>(descs, tasks, ntasks, grid, st); break;
      case GEMM_32x32: gemm_launch_t<cdouble, 32, 16, 16>(descs, tasks, ntasks, grid, st); break;
      case GEMM_128x64: gemm_launch_t<cdouble, 64, 32, 8>(descs, tasks, ntasks, grid, st); break;
      default: gemm_launch_t<cdouble, 32, 32, 16>(descs, tasks, ntasks, grid, st); break;
    }
  }
}

namespace {
template <typename T, int G, int P>
constexpr int lu_smem_bytes() {
  return (int)sizeof(T) * ((2 * kLuW + kLuLines<G, P>) * (kLuW + 1) + 3 * kLuW);
}
template <typename T, int G, int P>
void lu_launch_t(const SymDev& S, void* store, void* winv, void* piv, const LuTask* tasks,
                 int ntasks, bool solve, bool sym, cudaStream_t st) {
  lu_panel_kernel<T, G, P><<<ntasks, 128 * (G + 1), lu_smem_bytes<T, G, P>(), st>>>(
      S, (T*)store, (T*)winv, (T*)piv, tasks, solve ? 1 : 0, sym ? 1 : 0);
}
template <typename T>
void lu_dispatch_t(const SymDev& S, void* store, void* winv, void* piv, const LuTask* tasks,
                   int ntasks, int lines, bool solve, bool sym, cudaStream_t st) {
  switch (lines) {
    case 8: lu_launch_t<T, 1, 4>(S, store, winv, piv, tasks, ntasks, solve, sym, st); break;
    case 16: lu_launch_t<T, 1, 2>(S, store, winv, piv, tasks, ntasks, solve, sym, st); break;
    case 32: lu_launch_t<T, 1, 1>(S, store, winv, piv, tasks, ntasks, solve, sym, st); break;
    default: lu_launch_t<T, kLuGroups, 1>(S, store, winv, piv, tasks, ntasks, solve, sym, st); break;
  }
}
template <typename T, int G, int P>
cudaError_t lu_prepare_t() {
  return cudaFuncSetAttribute(lu_panel_kernel<T, G, P>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              lu_smem_bytes<T, G, P>());
}
}  // namespace

void launch_lu_panel(int dtype, const SymDev& S, void* store, void* winv, void* piv,
                     const LuTask* tasks, int ntasks, int lines, bool solve, bool sym,
                     cudaStream_t st) {
  if (ntasks <= 0) return;
  if (dtype == DT_F64)
    lu_dispatch_t<double>(S, store, winv, piv, tasks, ntasks, lines, solve, sym, st);
  else
    lu_dispatch_t<cdouble>(S, store, winv, piv, tasks, ntasks, lines, solve, sym, st);
}

void launch_unpack_pivots(int dtype, const SymDev& S, void* store, const void* piv, int nbatch,
                          cudaStream_t st) {
  const int64_t total = (int64_t)nbatch * S.n * kLuW;
  if (total == 0) return;
  const int grid = (int)std::min<int64_t>((total + kThreads - 1) / kThreads, 152 * 16);
  if (dtype == DT_F64)
    unpack_pivots_kernel<double><<<grid, kThreads, 0, st>>>(S, (double*)store, (const double*)piv,
                                                            total);
  else
    unpack_pivots_kernel<cdouble><<<grid, kThreads, 0, st>>>(S, (cdouble*)store,
                                                             (const cdouble*)piv, total);
}

cudaError_t prepare_dense_kernels() {
  cudaError_t e = lu_prepare_t<cdouble, 1, 1>();
  if (e == cudaSuccess) e = lu_prepare_t<cdouble, kLuGroups, 1>();
  return e;
}

namespace {
// FP64 pipe throughput: kPeakChains independent fused multiply-add chains
// per thread (enough to hide the pipe's latency), `iters` rounds; the sum is
// stored so that nothing is optimised away.
constexpr int kPeakChains = 8;
__global__ void __launch_bounds__(kThreads)
fp64_peak_kernel(double* out, int iters, double a, double b) {
  double x[kPeakChains];
#pragma unroll
  for (int j = 0; j < kPeakChains; j++) x[j] = threadIdx.x * 1e-3 + j;
  for (int i = 0; i < iters; i++) {
#pragma unroll
    for (int j = 0; j < kPeakChains; j++) x[j] = fma(x[j], a, b);
  }
  double sum = 0.0;
#pragma unroll
  for (int j = 0; j < kPeakChains; j++) sum += x[j];
  out[blockIdx.x * (int64_t)blockDim.x + threadIdx.x] = sum;
}
}  // namespace

int fp64_peak_grid(int sms) { return sms * 8; }

// flops of one launch of the FP64 peak loop over `grid` CTAs
double launch_fp64_peak(double* out, int grid, int iters, cudaStream_t st) {
  fp64_peak_kernel<<<grid, kThreads, 0, st>>>(out, iters, 0.999999, 1e-7);
  return 2.0 * kPeakChains * (double)iters * (double)grid * kThreads;
}

}  // namespace pselinv
