// Device body of the fused ASE-DF face sweep (shared by the one-problem kernel and the
// batched persistent kernel).  See ase_df_sweep.cu for the algorithm.
#pragma once

#include <cuda_runtime.h>

#include "ase_df_device.cuh"
#include "ase_df_fixed.cuh"
#include "ase_df_internal.cuh"

namespace asedf {
namespace {


// Branch of Algorithm 1 capped at order R, from the 2K face strengths of a cell's
// stencil, s[m+K-1] = sigma_{m-1/2} (m = -K+1..K).  Stencil sums use one fixed
// association, symmetric under mirroring: A3 = left + right,
// A5 = (s_-3/2 + s_-1/2) + (s_1/2 + s_3/2), A7 = A5 + (s_-5/2 + s_5/2),
// A9 = A7 + (s_-7/2 + s_7/2).  Smooth iff A < sigma_thres; else alpha = sigma_thres / A.
struct Branch {
  int m;          // R..5 odd: linear m-th order; 0: WENOZ-AO(5,3)+DF; 3: linear 3; -3: DF-damped 3
  double a3[3];   // alpha of S3_{-1}, S3_0, S3_1 (fallback)
  double a5;      // alpha of S5 (fallback) / of S3_0 (DF-damped order 3)
};

template <int R>
__device__ __forceinline__ Branch linear_branch() {
  return Branch{R, {1.0, 1.0, 1.0}, 1.0};
}

template <int R>
__device__ __forceinline__ Branch select_branch(const double* s, double thres) {
  constexpr int K = (R - 1) / 2;
  Branch b = linear_branch<R>();
  // Smooth data without FP64 arithmetic: if every one of the 2K <= 8 strengths is at most
  // thres/16 (compared as unsigned bit patterns, so negative values and NaN fail), each
  // stencil sum is at most 8 thres/16 = thres/2 also after rounding (rounded addition is
  // monotone in its operands), so every sum is below thres and the branch is linear order R.
  const unsigned long long lim = smooth_limit(thres);
  unsigned long long mx = (unsigned long long)dbits(s[0]);
#pragma unroll
  for (int t = 1; t < 2 * K; ++t) mx = max(mx, (unsigned long long)dbits(s[t]));
  if (mx <= lim) return b;
  const double sm12 = s[K - 1], sp12 = s[K];  // sigma_{-1/2}, sigma_{1/2}
  if (R == 3) {
    const double A = sm12 + sp12;
    if (lt_pos(A, thres)) { b.m = 3; } else { b.m = -3; b.a5 = thres / A; }
    return b;
  }
  const double sm32 = s[K - 2], sp32 = s[K + 1];
  const double A5 = (sm32 + sm12) + (sp12 + sp32);
  if (!lt_pos(A5, thres)) {
    b.m = 0;
    const double A3m = sm32 + sm12, A30 = sm12 + sp12, A3p = sp12 + sp32;
    b.a3[0] = lt_pos(A3m, thres) ? 1.0 : thres / A3m;
    b.a3[1] = lt_pos(A30, thres) ? 1.0 : thres / A30;
    b.a3[2] = lt_pos(A3p, thres) ? 1.0 : thres / A3p;
    b.a5 = thres / A5;
    return b;
  }
  b.m = 5;
  if (R >= 7) {
    const double A7 = A5 + (s[K - 3] + s[K + 2]);
    if (lt_pos(A7, thres)) {
      b.m = 7;
      if (R >= 9) {
        const double A9 = A7 + (s[K - 4] + s[K + 3]);
        if (lt_pos(A9, thres)) b.m = 9;
      }
    }
  }
  return b;
}

// Histogram slot of a branch (kBranchSlots order): linear 9, 7, 5 -> 0, 1, 2; the
// WENOZ-AO(5,3)+DF fallback -> 3; linear 3 -> 4; DF-damped 3 -> 5.
__device__ __forceinline__ int branch_slot(int m) {
  return m >= 5 ? (9 - m) / 2 : (m == 0 ? 3 : (m == 3 ? 4 : 5));
}

// Linear M-cell value at point p: v points at W_0, with W_t at v[t*vs].
template <int M>
__device__ __forceinline__ double lin_eval(const double* v, int vs, const double* w) {
  constexpr int H = (M - 1) / 2;
  double acc = w[4 - H] * v[-H * vs];
#pragma unroll
  for (int t = -H + 1; t <= H; ++t) acc = fma(w[4 + t], v[t * vs], acc);
  return acc;
}

// WENOZ-AO(5,3) with DF damping (Sec. 3.2) of one component, at NP points p0..p0+NP-1.
// v points at W_0 (stride vs).
template <int NP>
__device__ __forceinline__ void weno_eval(const double* v, int vs, const Branch& br,
                                          const Tables& T, int p0, double* out) {
  double beta[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double* vk = v + (k - 2) * vs;  // sub-stencil S3_{k-1}: offsets k-2 .. k
    const double c1 = T.cq[k][0][0] * vk[0] + T.cq[k][0][1] * vk[vs] + T.cq[k][0][2] * vk[2 * vs];
    const double c2 = T.cq[k][1][0] * vk[0] + T.cq[k][1][1] * vk[vs] + T.cq[k][1][2] * vk[2 * vs];
    // int_{-1}^{0} (p')^2 + (p'')^2 for p = c0 + c1 xi + c2 xi^2
    beta[k] = c1 * (c1 - 2.0 * c2) + (16.0 / 3.0) * c2 * c2;
  }
  const double b5 = (beta[0] + 4.0 * beta[1] + beta[2]) * (1.0 / 6.0) + fabs(beta[0] - beta[2]);
  const double tau = (fabs(b5 - beta[0]) + fabs(b5 - beta[1]) + fabs(b5 - beta[2])) * (1.0 / 3.0);
  const double tau2 = tau * tau;
  const double e5 = b5 + T.eps;
  const double w5 = T.d5 * (1.0 + tau2 / (e5 * e5));
  double w3[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double e = beta[k] + T.eps;
    w3[k] = T.d3[k] * (1.0 + tau2 / (e * e));
  }
  const double inv = 1.0 / (w5 + w3[0] + w3[1] + w3[2]);
  const double g5 = (w5 * inv) / T.d5;
  double g3[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) g3[k] = w3[k] * inv - g5 * T.d3[k];
  const double W0 = v[0];
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    const int p = p0 + q;
    const double P5 = fma(br.a5, lin_eval<5>(v, vs, T.lin[1][p]) - W0, W0);
    double P = g5 * P5;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double* vk = v + (k - 2) * vs;
      const double u = T.sub[k][p][0] * vk[0] + T.sub[k][p][1] * vk[vs] + T.sub[k][p][2] * vk[2 * vs];
      P = fma(g3[k], fma(br.a3[k], u - W0, W0), P);
    }
    out[q] = P;
  }
}

// Value of the chosen polynomial of one component at NP points p0.. (Algorithm 1).
template <int R, int NP>
__device__ __forceinline__ void recon_eval(const double* v, int vs, const Branch& br,
                                           const Tables& T, int p0, double* out) {
  if (br.m == R) {
#pragma unroll
    for (int q = 0; q < NP; ++q) out[q] = lin_eval<R>(v, vs, T.lin[(R - 3) / 2][p0 + q]);
    return;
  }
  if (R == 3) {  // DF-damped 3rd order
#pragma unroll
    for (int q = 0; q < NP; ++q) out[q] = fma(br.a5, lin_eval<3>(v, vs, T.lin[0][p0 + q]) - v[0], v[0]);
    return;
  }
  if (R >= 9 && br.m == 7) {
#pragma unroll
    for (int q = 0; q < NP; ++q) out[q] = lin_eval<(R >= 7 ? 7 : 3)>(v, vs, T.lin[2][p0 + q]);
    return;
  }
  if (R >= 7 && br.m == 5) {
#pragma unroll
    for (int q = 0; q < NP; ++q) out[q] = lin_eval<5>(v, vs, T.lin[1][p0 + q]);
    return;
  }
  if (R >= 5) weno_eval<NP>(v, vs, br, T, p0, out);
}

// Gauss-point values (tangential reconstruction, Sec. 2.1) of the order-R linear
// branch, using the reflection symmetry of the centred stencil: the points eta and
// -1 - eta share E = w_0 W_0 + sum e_t (W_t + W_-t) and differ in the sign of
// O = sum o_t (W_t - W_-t).  Used for G >= 3, where it saves FMAs over G dot products.
template <int R, int G>
__device__ __forceinline__ void lin_gauss_sym(const double* v, int vs, const Tables& T, double* out) {
  constexpr int K = (R - 1) / 2;
  double S[K + 1], D[K + 1];
#pragma unroll
  for (int t = 1; t <= K; ++t) {
    S[t] = v[t * vs] + v[-t * vs];
    D[t] = v[t * vs] - v[-t * vs];
  }
#pragma unroll
  for (int g = 0; g < (G + 1) / 2; ++g) {
    double E = T.se[g][0] * v[0];
#pragma unroll
    for (int t = 1; t <= K; ++t) E = fma(T.se[g][t], S[t], E);
    if (2 * g + 1 == G) {
      out[g] = E;  // middle point
    } else {
      double O = T.so[g][1] * D[1];
#pragma unroll
      for (int t = 2; t <= K; ++t) O = fma(T.so[g][t], D[t], O);
      out[g] = E + O;
      out[G - 1 - g] = E - O;
    }
  }
}

// Tangential reconstruction at the G Gauss points (points 2..G+1 of the tables).
template <int R, int G>
__device__ __forceinline__ void tang_eval(const double* v, int vs, const Branch& br, const Tables& T,
                                          double* out) {
  if (G >= 3 && br.m == R) {
    lin_gauss_sym<R, G>(v, vs, T, out);
    return;
  }
  recon_eval<R, G>(v, vs, br, T, 2, out);
}

// Tile of the face kernels: TN faces along the sweep on TT lines.  The Lax-Friedrichs sweep
// uses 8 x 64 in 2D (measured on GB300 against 16 x 32, 16 x 16, 32 x 16 and 8 x 32: 1.4 %
// faster than 16 x 32 at order 9, from the smaller share of halo lines); 255 faces in 1D (256
// reconstructing cells: phase 1 gives every one of the 256 threads one cell).
// A 1D sweep of fewer than one 255-face tile per SM takes tiles of 31 faces in CTAs of 32
// threads (Tile<R, 1, 1, 31, 32>): FP64 issues at 2 instructions per cycle per SM, so one
// CTA of 256 threads on a 200-cell problem runs its FP64 work on one SM, 16 us per sweep.
template <int R, int DIM, int TT_ = (DIM == 2) ? 64 : 1, int TN_ = (DIM == 2) ? 8 : 255, int NT_ = 256>
struct Tile {
  static constexpr int K = (R - 1) / 2;
  static constexpr int C = (DIM == 1) ? 3 : 4;
  static constexpr int KT = (DIM == 2) ? K : 0;
  static constexpr int G = (DIM == 2) ? (R == 3 ? 1 : K) : 1;
  static constexpr int TN = TN_;                     // faces along the sweep
  static constexpr int TT = TT_;                     // lines
  static constexpr int NT = NT_;                     // threads
  static constexpr int NA = TN + 1 + 2 * K;          // staged cells along the sweep
  static constexpr int NB = TT + 2 * KT;             // staged lines
  static constexpr int NQ = TN + 1;                  // cells reconstructed along the sweep
  static constexpr int NSN = TN + 2 * K;             // normal faces staged per line
  static constexpr int NST = TT + 2 * K;             // tangential faces staged per column
  // queue of deferred fallback items (defer_item) and its two counters, after the arrays
  static constexpr int QCAP = (NQ * NB > TN * TT) ? NQ * NB : TN * TT;
  static constexpr size_t queue_offset =
      (size_t)C * NB * NA + 2 * (size_t)C * NB * NQ + (size_t)NB * NSN + (DIM == 2 ? (size_t)NQ * NST : 0);
  static constexpr size_t smem_doubles = queue_offset + ((size_t)QCAP + 2 + 1) / 2;
  // 2D sweeps, after the queue: a word of fast cells per staged line and per line of faces (fix_fast)
  static constexpr size_t fast_offset = smem_doubles;
  static constexpr size_t split_offset = smem_doubles + (DIM == 2 ? ((size_t)NB + TT + 1) / 2 : 0);
  // 2D tiles of 16 lines, last: the states [2][G][C] and terms [5][G] of every face and the
  // branches (5 words) of its columns (sweep_tile)
  static constexpr bool split = DIM == 2 && TT == 16;
  static constexpr size_t sweep_doubles = split_offset + (split ? (size_t)(2 * C + 5) * G * TN * TT + 5 * NQ * TT : 0);
};

// Quotient and remainder by a tile's run-time line count n (at most 127) of an index below 2^13, by
// a multiplication: with m = ceil(2^20 / n), i m / 2^20 exceeds i / n by less than 2^13 / 2^20 <
// 1 / n.  An integer division by a run-time number costs some 25 instructions, and the staging
// and item loops do one per element.
struct LineDiv {
  unsigned int m;
  int n;
  __device__ __forceinline__ explicit LineDiv(int n_) : m(((1u << 20) + n_ - 1) / n_), n(n_) {}
  __device__ __forceinline__ void split(int i, int& q, int& r) const {
    q = (int)(((unsigned int)i * m) >> 20);
    r = i - q * n;
  }
};

// Deferral of the work items whose branch is the WENOZ-AO(5,3)+DF fallback.  Its arithmetic
// (smoothness indicators, nonlinear weights, four sub-polynomials) is several times that of
// a linear branch, so a warp holding one such item among linear ones would run the long path
// with most lanes idle.  A deferred item goes to a queue in shared memory, which every thread
// of the CTA works through after the linear items.  The lanes of a warp that defer reserve
// their slots together: one ballot, one shared-memory atomic by the first of them, and each
// lane's rank among them.  Returns whether this lane deferred its item.
__device__ __forceinline__ bool defer_item(bool defer, int item, int* queue, unsigned int* count) {
  const unsigned int active = __activemask();
  const unsigned int m = __ballot_sync(active, defer);
  if (m == 0u) return false;
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(m) - 1;
  unsigned int base = 0u;
  if (lane == leader) base = atomicAdd(count, (unsigned int)__popc(m));
  base = __shfl_sync(active, base, leader);
  if (defer) queue[base + __popc(m & ((1u << lane) - 1u))] = item;
  return defer;
}

// Whether most of a cell's energy is kinetic (p' = E - |m|^2 / (2 rho) below 2^-9 E) or its values lie
// beyond 2^+-60: p' then amplifies the rounding of a state by E / p', the strengths of a fast, even
// stream are that rounding, and the stencils that hold the cell keep to FP64.  From the high words of
// rho, m, E; in FP32, whose few units in 2^-20 do not matter to the rule, the two momenta alike.
__device__ __forceinline__ bool fix_fast(int rho, int mx, int my, int e) {
  auto f = [](int hi) {  // |x| truncated to 20 bits (0 below 2^-63)
    const int b = (hi & 0x7fffffff) - (896 << 20);
    return b < (64 << 20) ? 0.0f : b >= (188 << 20) ? 1e19f : __int_as_float(b << 3);
  };
  const float r = f(rho), u = f(mx), v = f(my), en = f(e);
  return !(r > 0.0f && en > 0.0f && fmaxf(fmaxf(r, en), fmaxf(u, v)) < 1e18f) ||
         __fadd_rn(__fmul_rn(u, u), __fmul_rn(v, v)) > 2.0f * (1.0f - 1.0f / 512.0f) * r * en;
}

// One tile: faces a0 .. a0+TN-1 along the sweep on lines b0 .. b0+tt-1, 1 <= tt <= TT
// (threadIdx.x is the worker index); smem holds Tile<R, DIM, TT>::sweep_doubles doubles,
// laid out for TT lines whatever tt is.
//
// 2D flows of order 5 and more with a front in both directions (some x-face and some y-face strength
// beyond smooth_limit, below which every branch is linear) take the linear branch of order R of both
// reconstructions in fixed point on the integer units (ase_df_fixed.cuh), stencil by stencil where its
// values span few binades and no cell of it is fast (fix_fast); the FP64 pipe is left to the Gauss
// points.  What a face gets depends on its own stencils alone, not on the tile.  The other branches
// run in FP64 in second passes over queues of such cells and faces.
// FP64 -> fixed point: Configuration 3 512^2 order 5, one step, 1235 -> 1000 us; the 1600 x 800 order-9 jet
// residual 3564 -> 2375 us; 64 mixed problems 13.1 -> 10.4 ms.  One exponent per tile measured 950 us, 2410 us and 10.6
// ms: it converts a value once, but cuts off the digits of values far below the tile's largest.
// Flows without a front in both directions stay in FP64 to the bit: their strengths are differences of two
// reconstructions that agree to rounding (1e-12 made of 1e-16 parts on a fine smooth grid), so
// any other rounding of a state, however exact, shows in the fifth digit of the strengths; with a
// front across one direction only (a wall, a tube), the other direction's strengths are such.
template <int R, int DIM, int DIR, int TT_ = (DIM == 2) ? 64 : 1, int TN_ = (DIM == 2) ? 8 : 255, int NT_ = 256>
__device__ __forceinline__ void sweep_tile(const GridInfo& g, const SweepArgs& args, const Tables& T, int a0,
                                           int b0, int tt, double* smem) {
  using TL = Tile<R, DIM, TT_, TN_, NT_>;
  constexpr int K = TL::K, C = TL::C, KT = TL::KT, G = TL::G;
  constexpr int TN = TL::TN, TT = TL::TT, NT = TL::NT;
  constexpr int NA = TL::NA, NB = TL::NB, NQ = TL::NQ, NSN = TL::NSN, NST = TL::NST;
  constexpr int NI = (DIR == 0) ? 1 : 2;  // normal momentum component
  constexpr int TI = (DIR == 0) ? 2 : 1;  // tangential momentum component
  // 2D loops over components and Gauss points stay rolled, their states in local memory: unrolled,
  // the branches of all components and two forms of four points made 760 KB of code, far beyond
  // the instruction cache (190 KB now; 64^2 order-7 run of 4 steps 435 -> 404 us).  1D unrolls its
  // components: there the chain of one cell bounds the tile.
  // So do 64-line tiles of order 3, whose branches are short: 4 steps at 230^2 582 -> 549 us, 256^2 650 -> 632;
  // a 1024^2 residual 497 -> 501.
  constexpr bool kFix = DIM == 2 && R >= 5;  // fixed point (ase_df_fixed.cuh)
  constexpr bool kFlat = TL::split || NT == 32;
  constexpr int kCU = (DIM == 1 || (R == 3 && !TL::split)) ? C : 1, kLU = kFlat ? 1 : C;
  // Products of the Gauss points on the integer units (ase_df_imul.cuh), where the tile has the
  // warps to fill the FP64 pipe: the 1024^2 order-9 step 7393 -> 6466 us, the 65537-cell order-9
  // residual 41.1 -> 39.0 us.  The 32-thread tiles and those of up to 8 lines (two CTAs of a few warps'
  // work on an SM) are bound by latency and keep the FP64 instruction: 64^2 order-7 runs 324 us, 332 with
  // the integer form; 128^2 ones 619 and 577 us.
  const bool ints = NT > 32 && (!TL::split || tt > 8);

  double* sW = smem;                       // [C][NB][NA]
  double* sQP = sW + C * NB * NA;          // [C][NB][NQ] value at xi = 0
  double* sQM = sQP + C * NB * NQ;         // [C][NB][NQ] value at xi = -1
  double* sSn = sQM + C * NB * NQ;         // [NB][NSN]
  double* sSt = sSn + NB * NSN;            // [NQ][NST]

  const int n = (DIR == 0) ? g.nx : g.ny;       // cells along the sweep
  const int mlin = (DIR == 0) ? g.ny : g.nx;    // lines
  const int tid = threadIdx.x;
  const int nb = tt + 2 * KT;  // staged lines of this tile (<= NB)

  const double ts = stage_time(args.st, args.tfrac, args.st->dt);  // for time-dependent ghosts
  __shared__ unsigned int hist_s[kBranchSlots];
  const bool counting = args.hist != nullptr;
  if (counting && tid < kBranchSlots) hist_s[tid] = 0u;
  // queue of deferred fallback items: phase 1 (cells) and phase 2 (faces) share the slots
  int* s_queue = reinterpret_cast<int*>(smem + TL::queue_offset);
  unsigned int* s_qn = reinterpret_cast<unsigned int*>(s_queue + TL::QCAP);
  if (tid < 2) s_qn[tid] = 0u;
  // fixed point: the fast cells of the staged lines (bit aa of word bb), then of each line's 2K+1 lines
  unsigned int* s_fast = reinterpret_cast<unsigned int*>(smem + TL::fast_offset);
  const bool front = kFix && args.front != nullptr && args.front[0] != 0u && args.front[1] != 0u;
  const unsigned long long limit = smooth_limit(g.thres);
  // ---- staging: consecutive threads take consecutive addresses along the direction in which the
  // arrays are contiguous (the sweep for x-faces, the lines for y-faces) ----
  static_assert(NA * NB < (1 << 13) && NB < 128, "LineDiv range");
  const LineDiv dnb(nb);
  const int sta = (DIR == 0) ? 1 : g.nx, stb = (DIR == 0) ? g.nx : 1;
  // a tile whose halo lies inside the grid needs none of the boundary's index maps
  const bool inside = a0 - 1 - K >= 0 && a0 + TN - 1 + K < n && (DIM == 1 || (b0 - KT >= 0 && b0 + tt + KT <= mlin));
  // cell averages: cells a0-1-K .. a0+TN-1+K, lines b0-KT .. b0+tt+KT-1
  // (16-line tiles and those of 32 threads: one component of a cell per thread, which loads one value instead
  // of three or four in turn; a sweep of 2000 cells in 31-face tiles is 0.5 us shorter)
  const int staged = nb * NA;
  for (int k = tid; k < (kFlat ? C * staged : staged); k += NT) {
    const int c0 = kFlat ? (k >= staged) + (k >= 2 * staged) + (k >= 3 * staged) : 0;
    const int cn = kFlat ? c0 + 1 : C, idx = k - c0 * staged;
    int bb, aa;
    if (DIR == 0) { aa = idx % NA; bb = idx / NA; }
    else dnb.split(idx, aa, bb);
    const int a = a0 - 1 - K + aa, b = b0 - KT + bb;
    double* dst = sW + bb * NA + aa;
    if (inside) {
      const double* src = args.W + (size_t)b * stb + (size_t)a * sta;
#pragma unroll kLU
      for (int c = c0; c < cn; ++c) {
        dst[c * NB * NA] = __ldg(src + (size_t)c * g.nx * g.ny);
      }
    } else {
      const int i = (DIR == 0) ? a : b, j = (DIR == 0) ? b : a;
#pragma unroll (DIM == 1 && !kFlat ? C : 1)
      for (int c = c0; c < cn; ++c) {
        dst[c * NB * NA] = fetch_w(g, args.W, c, i, j, ts);
      }
    }
  }
  if (front)
    for (int bb = tid; bb < nb; bb += NT) s_fast[bb] = 0u;
  bool rough = false;  // a strength beyond the limit below which every branch is linear of order R
  // normal face strengths: faces a0-K .. a0+TN-1+K of every staged line
  for (int idx = tid; idx < nb * NSN; idx += NT) {
    int fa, bb;
    if (DIR == 0) { fa = idx % NSN; bb = idx / NSN; }
    else dnb.split(idx, fa, bb);
    const int f = a0 - K + fa, b = b0 - KT + bb;
    double v;
    if (inside) v = __ldg(args.s_norm + ((DIR == 0) ? (size_t)b * (g.nx + 1) + f : (size_t)f * g.nx + b));
    else v = (DIR == 0) ? sigma_x_at(g, args.s_norm, f, b) : sigma_y_at(g, args.s_norm, f, b);
    sSn[bb * NSN + fa] = v;
    rough |= is_front(v, limit);
  }
  // tangential face strengths of the reconstructing cells' columns: faces b0-K+1 .. b0+tt+K-1
  if (DIM == 2) {
    const int nst = tt + 2 * K - 1;
    const LineDiv dst(nst);
    for (int idx = tid; idx < NQ * nst; idx += NT) {
      int qa, fb;
      if (DIR == 0) { qa = idx % NQ; fb = idx / NQ; }
      else dst.split(idx, qa, fb);
      const int f = b0 - K + 1 + fb, a = a0 - 1 + qa;
      double v;
      if (inside) v = __ldg(args.s_tan + ((DIR == 0) ? (size_t)f * g.nx + a : (size_t)a * (g.nx + 1) + f));
      else v = (DIR == 0) ? sigma_y_at(g, args.s_tan, f, a) : sigma_x_at(g, args.s_tan, f, a);
      sSt[qa * NST + fb] = v;
      rough |= is_front(v, limit);
    }
  }
  rough = __syncthreads_or(rough);
  // a tile without such a strength needs no branch choice
  auto branch = [&](const double* s) { return rough ? select_branch<R>(s, g.thres) : linear_branch<R>(); };

  // ---- phase 1: normal reconstruction of cells a0-1 .. a0+TN-1 on all staged lines ----
  // Interior cells serve a face on each side and are evaluated at both xi = 0 and xi = -1; the
  // two end cells serve one tile face each (qa = 0: its xi = 0 value, the left state of face
  // a0; qa = NQ-1: its xi = -1 value).
  bool fast = false;  // whether a staged cell is fast
  if constexpr (kFix) {
    if (front) {
      const int* hi = reinterpret_cast<const int*>(sW) + 1;
      for (int idx = tid; idx < nb * NA; idx += NT)
        if (fix_fast(hi[2 * idx], hi[2 * (NB * NA + idx)], hi[2 * (2 * NB * NA + idx)], hi[2 * (3 * NB * NA + idx)])) {
          atomicOr(&s_fast[idx / NA], 1u << idx % NA);
          fast = true;
        }
      fast = __syncthreads_or(fast);
      if (fast)  // read after phase 1
        for (int tb = tid; tb < tt; tb += NT) {
          unsigned int m = 0u;
          for (int l = 0; l <= 2 * K; ++l) m |= s_fast[tb + l];
          s_fast[NB + tb] = m;
        }
    }
  }
  // fixed point for a stencil that starts at staged cell qa of line (of lines) k, of branch m
  auto fixed = [&](int m, int k, int qa) {
    return front && m == R && !(fast && (s_fast[k] >> qa & ((1u << (2 * K + 1)) - 1u)) != 0u);
  };
  // The end cells come last in the work list and evaluate one point; fallback cells (in a flow with a
  // front: those of any branch but the order-R linear one) are deferred (defer_item) and done in a
  // second pass.  There, and in 1D, the end cells evaluate both points like the others, one of them not
  // read: two lanes of a warp would run the same long chain once more after the others'.  A 16-line tile without a branch choice gives each component of a cell a thread.
  const bool comps = TL::split && !rough;
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    const int cells = NQ * nb;
    const int count = (pass == 0) ? (comps ? C * cells : cells) : (int)s_qn[0];
    for (int k = tid; k < count; k += NT) {
      const int c0 = comps ? (k >= cells) + (k >= 2 * cells) + (k >= 3 * cells) : 0, cn = comps ? c0 + 1 : C;
      const int it = (pass == 0) ? k - c0 * cells : s_queue[k];
      int qa, bb, pt;  // pt -1: an interior cell, both points; 0 / 1: an end cell, one point
      if (it < (NQ - 2) * nb) {
        if (DIR == 0) { qa = 1 + it % (NQ - 2); bb = it / (NQ - 2); }
        else { dnb.split(it, qa, bb); ++qa; }
        pt = -1;
      } else {
        dnb.split(it - (NQ - 2) * nb, pt, bb);  // pt 0: cell qa = 0 at xi = 0; 1: qa = NQ-1 at xi = -1
        qa = pt * (NQ - 1);
        if (DIM == 1 || pass == 1) pt = -1;  // both points (below)
      }
      const Branch br = branch(sSn + bb * NSN + qa);
      if (R >= 5 && rough && pass == 0 && defer_item(front ? br.m != R : br.m == 0, it, s_queue, &s_qn[0]))
        continue;
      const bool fix = fixed(br.m, bb, qa);
      if (pt < 0) {
#pragma unroll kCU
        for (int c = c0; c < cn; ++c) {
          const double* v = sW + (c * NB + bb) * NA + qa + K;  // W_0 of this cell
          double out[2];
          if (!kFix || !(fix && fix_normal<R, 2>(v, 1, out))) recon_eval<R, 2>(v, 1, br, T, 0, out);
          sQP[(c * NB + bb) * NQ + qa] = out[0];
          sQM[(c * NB + bb) * NQ + qa] = out[1];
        }
      } else {
        double* dst = pt ? sQM : sQP;
#pragma unroll kCU
        for (int c = c0; c < cn; ++c) {
          const double* v = sW + (c * NB + bb) * NA + qa + K;
          double out[1];
          if (!kFix || !(fix && fix_normal<R, 1>(v, pt ? -1 : 1, out))) recon_eval<R, 1>(v, 1, br, T, pt, out);
          dst[(c * NB + bb) * NQ + qa] = out[0];
        }
      }
    }
    __syncthreads();  // pass 0: the queue is complete; last pass: phase 1 is done
    if (s_qn[0] == 0u || pass == 1) break;
    const int nq = (int)s_qn[0];
    if (nq * C > NT) continue;
    // a short queue: one component of a cell per thread.  The fallback of one component is some
    // 200 dependent FP64 instructions, and the tile waits for its slowest thread (Sod tube of 200
    // cells, first sweep 42.7 -> 19.6 us, later ones 11.7 -> 10.6); a long queue keeps one thread per cell, which chooses
    // the branch (and divides for its DF factors) once.
    for (int k = tid; k < nq * C; k += NT) {
      const int it = s_queue[k / C], c = k % C;
      int bb, qa;
      if (it < (NQ - 2) * nb) {
        if (DIR == 0) { qa = 1 + it % (NQ - 2); bb = it / (NQ - 2); }
        else { dnb.split(it, qa, bb); ++qa; }
      } else {
        dnb.split(it - (NQ - 2) * nb, qa, bb);
        qa *= NQ - 1;
      }
      double out[2];  // an end cell's value at its outer face is formed too and not read
      const Branch br = select_branch<R>(sSn + bb * NSN + qa, g.thres);
      const double* v = sW + (c * NB + bb) * NA + qa + K;
      if (kFix) recon_eval<R, 2>(v, 1, br, T, 0, out);
      else weno_eval<2>(v, 1, br, T, 0, out);  // 1D: nothing else is queued
      sQP[(c * NB + bb) * NQ + qa] = out[0];
      sQM[(c * NB + bb) * NQ + qa] = out[1];
    }
    __syncthreads();
    break;
  }

  // Gauss-point values of component cs / 2 of the state on side cs % 2 of a face, its branch bt
  auto tang_point = [&](int cs, int fa, int tb, const Branch& bt, double* out) {
    const int qa = fa + (cs & 1);
    const double* v = ((cs & 1) == 0 ? sQP : sQM) + ((cs >> 1) * NB + tb + K) * NQ + qa;
    if (!kFix || !(fixed(bt.m, NB + tb, qa) && fix_gauss<R, G>(v, NQ, out))) tang_eval<R, G>(v, NQ, bt, T, out);
  };
  // ---- phase 2: faces ----
  // 2D: faces with a fallback tangential reconstruction on either side (in a flow with a front: with any
  // but the order-R linear one) are deferred.
  if constexpr (TL::split) {
    // Tiles of up to 16 lines, on grids that give an SM one or two of them: a face per thread would
    // leave half or more of the CTA idle while a quarter of the SM's FP64 unit works on chains of some
    // 100 dependent instructions.  So (component, side) pairs of a face, then its Gauss points, then
    // the components of its sums go to threads of their own, in the same arithmetic and order.
    constexpr int NF = TN * TT;
    double* sP = smem + TL::split_offset;  // [2][G][C][NF] states
    double* sX = sP + 2 * G * C * NF;      // [G][5][NF]: alL, alR, ps, pu, strength
    static_assert(sizeof(Branch) == 5 * sizeof(double), "sB");
    Branch* sB = reinterpret_cast<Branch*>(sX + 5 * G * NF);  // [TT][NQ] branches of the columns
    const int faces = TN * tt;
    const LineDiv dtt(tt);
    auto face_of = [&](int it, int& fa, int& tb) {
      if (DIR == 0) { fa = it % TN; tb = it / TN; }
      else dtt.split(it, fa, tb);
      return a0 + fa <= n && b0 + tb < mlin;
    };
    if (rough) {
      for (int it = tid; it < NQ * tt; it += NT) sB[it] = select_branch<R>(sSt + (it % NQ) * NST + it / NQ, g.thres);
      __syncthreads();
    }
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
      const int nf = (pass == 0) ? faces : (int)s_qn[1];
      for (int k = tid; k < 2 * C * nf; k += NT) {
        int cs = 0, kf = k;
        while (kf >= nf) { kf -= nf; ++cs; }
        const int it = (pass == 0) ? kf : s_queue[kf];
        int fa, tb;
        if (!face_of(it, fa, tb)) continue;
        Branch bt = linear_branch<R>();
        if (rough) bt = sB[tb * NQ + fa + (cs & 1)];
        if (rough && pass == 0) {
          const int m2 = sB[tb * NQ + fa + 1 - (cs & 1)].m;  // the other side's
          const bool later = R >= 5 && (front ? bt.m != R || m2 != R : bt.m == 0 || m2 == 0);
          if (defer_item(later && cs == 0, it, s_queue, &s_qn[1]) || later) continue;
        }
        if (counting && cs < 2) {
          atomicAdd(&hist_s[branch_slot(select_branch<R>(sSn + (tb + KT) * NSN + fa + cs, g.thres).m)], 1u);
          atomicAdd(&hist_s[branch_slot(bt.m)], 1u);
        }
        double out[G];
        tang_point(cs, fa, tb, bt, out);
#pragma unroll
        for (int q = 0; q < G; ++q) sP[(((cs & 1) * G + q) * C + (cs >> 1)) * NF + it] = out[q];
      }
      __syncthreads();
      if (s_qn[1] == 0u) break;
    }
    for (int k = tid; k < G * faces; k += NT) {
      int q = 0, it = k;
      while (it >= faces) { it -= faces; ++q; }
      int fa, tb;
      if (!face_of(it, fa, tb)) continue;
      double qa[C], qb[C], a[C], b[C], sg;
#pragma unroll
      for (int c = 0; c < C; ++c) {
        qa[c] = sP[(q * C + c) * NF + it];
        qb[c] = sP[((G + q) * C + c) * NF + it];
      }
      const double* ca = sW + (tb + KT) * NA + fa + K;
      LfTerms t;
      if (lf_point_terms<C, NI, TI, true>(qa, qb, ca, ca + 1, NB * NA, g.gg1, T.hgw[q], ints, a, b, t, sg)) {
        atomicOr(&args.st->flags, 0x2u);
        if (counting) atomicAdd(&hist_s[kBranchSlots - 1], 1u);
#pragma unroll
        for (int c = 0; c < C; ++c) {
          sP[(q * C + c) * NF + it] = a[c];
          sP[((G + q) * C + c) * NF + it] = b[c];
        }
      }
      const double x[5] = {t.alL, t.alR, t.ps, t.pu, sg};
#pragma unroll
      for (int j = 0; j < 5; ++j) sX[(q * 5 + j) * NF + it] = x[j];
    }
    __syncthreads();
    for (int k = tid; k < (C + 1) * faces; k += NT) {
      int c = 0, it = k;
      while (it >= faces) { it -= faces; ++c; }
      int fa, tb;
      if (!face_of(it, fa, tb)) continue;
      const int f = a0 + fa, b = b0 + tb;
      double sum = 0.0;
#pragma unroll
      for (int q = 0; q < G; ++q) {
        const double* x = sX + q * 5 * NF + it;
        if (c == C) sum += x[4 * NF];
        else sum = lf_add<C, NI>(c, sP[(q * C + c) * NF + it], sP[((G + q) * C + c) * NF + it],
                                 LfTerms{x[0], x[NF], x[2 * NF], x[3 * NF]}, g.gm1_hgw[q], sum);
      }
      if (c < C) {
        if (DIR == 0) args.F[((size_t)c * g.ny + b) * (g.nx + 1) + f] = sum;
        else args.F[((size_t)c * (g.ny + 1) + f) * g.nx + b] = sum;
      } else {
        const double sface = (G == 1) ? sum : sum * (1.0 / G);
        if (kFix && args.front_out != nullptr && is_front(sface, limit)) *args.front_out = 1u;
        args.s_out[(DIR == 0) ? (size_t)b * (g.nx + 1) + f : (size_t)f * g.nx + b] = sface;
      }
    }
  } else {
  const LineDiv dtt(tt);
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    const int count = (pass == 0) ? TN * tt : (int)s_qn[1];
    for (int k = tid; k < count; k += NT) {
      const int it = (pass == 0) ? k : s_queue[k];
      int fa, tb;
      if (DIR == 0) { fa = it % TN; tb = it / TN; }
      else dtt.split(it, fa, tb);
      const int f = a0 + fa, b = b0 + tb;
      if (f > n || b >= mlin) continue;
      Branch bt[2];
      if (DIM == 2) {
        bt[0] = branch(sSt + fa * NST + tb);  // the columns of the two states
        bt[1] = branch(sSt + (fa + 1) * NST + tb);
        if (rough && pass == 0) {
          const bool defer = front ? bt[0].m != R || bt[1].m != R : bt[0].m == 0 || bt[1].m == 0;
          if (R >= 5 && defer_item(defer, it, s_queue, &s_qn[1])) continue;
        }
      }
      double st[2][G][C];
      if (counting) {
#pragma unroll
        for (int side = 0; side < 2; ++side) {  // the normal branch as phase 1 chose it, the tangential one
          const Branch bn = select_branch<R>(sSn + (tb + KT) * NSN + fa + side, g.thres);
          atomicAdd(&hist_s[branch_slot(bn.m)], 1u);
          if (DIM == 2) atomicAdd(&hist_s[branch_slot(bt[side].m)], 1u);
        }
      }
      // left state: cell f-1 (plus face); right: cell f (minus face)
      if constexpr (DIM == 2) {
#pragma unroll (R == 3 ? 2 * C : 1)
        for (int cs = 0; cs < 2 * C; ++cs) {
          double out[G];
          tang_point(cs, fa, tb, (cs & 1) == 0 ? bt[0] : bt[1], out);
#pragma unroll
          for (int q = 0; q < G; ++q) st[cs & 1][q][cs >> 1] = out[q];
        }
      } else {
#pragma unroll
        for (int c = 0; c < C; ++c) {
          st[0][0][c] = sQP[c * NQ + fa];
          st[1][0][c] = sQM[c * NQ + fa + 1];
        }
      }
      // cell averages either side of the face (read by a Gauss point only if it falls back)
      const double* ca = sW + (tb + KT) * NA + fa + K;
      const double* cb = ca + 1;
      double Fs[C];
#pragma unroll
      for (int c = 0; c < C; ++c) Fs[c] = 0.0;
      double ssum = 0.0;
      unsigned int nfb = 0u;
#pragma unroll 1
      for (int q = 0; q < G; ++q) {
        double sg;
        nfb += lf_point_acc<C, NI, TI, (NT > 32)>(st[0][q], st[1][q], ca, cb, NB * NA, g.gm1, g.gg1, T.hgw[q],
                                                  g.gm1_hgw[q], ints, Fs, sg) ? 1u : 0u;
        ssum += sg;
      }
      if (nfb) {
        atomicOr(&args.st->flags, 0x2u);
        if (counting) atomicAdd(&hist_s[kBranchSlots - 1], nfb);
      }
      const double sface = (G == 1) ? ssum : ssum * (1.0 / G);
      if (kFix && args.front_out != nullptr && is_front(sface, limit)) *args.front_out = 1u;
      if (DIR == 0) {
#pragma unroll
        for (int c = 0; c < C; ++c) args.F[((size_t)c * g.ny + b) * (g.nx + 1) + f] = Fs[c];
        args.s_out[(size_t)b * (g.nx + 1) + f] = sface;
      } else {
#pragma unroll
        for (int c = 0; c < C; ++c) args.F[((size_t)c * (g.ny + 1) + f) * g.nx + b] = Fs[c];
        args.s_out[(size_t)f * g.nx + b] = sface;
      }
    }
    if (DIM == 1 || pass == 1) break;
    __syncthreads();  // the queue is complete
    if (s_qn[1] == 0u) break;
  }
  }
  if (counting) {
    __syncthreads();
    if (tid < kBranchSlots && hist_s[tid]) atomicAdd(&args.hist[tid], (unsigned long long)hist_s[tid]);
  }
}

}  // namespace
}  // namespace asedf
