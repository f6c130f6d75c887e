// GFD least-squares fits (Sec. 3.1 item 7), mu(I) closure (Sec. 2.2-2.3) and
// the explicit update (Sec. 3.1 items 8, 10).
//
// One thread per particle. A thread walks its stencil once, accumulating the
// 31 distinct moments of the Taylor rows (the 9x9 Gram matrix has only 31
// different entries) and the right-hand sides A^T b of all fields; it then
// factors the Gram matrix (Cholesky) and solves. Stencils whose Gram matrix is
// too ill-conditioned for the normal equations (relative pivot below the
// threshold, or fewer than 9 rows) are queued for a separate FP64 pivoted-QR
// kernel, the same algorithm the paper names (QR least squares).
//
// FP64 mode: the sums over the rows in 64-bit fixed point (fixed_rows.cuh;
// plain FP64 rows for the particles that do not fit it, for
// lp_fit_derivatives with mirror factors other than -1, 0 and 1, and for
// lp_fit_derivatives_noalloc), the factor, the solves and the rest in FP64.
// MIXED mode: moments, right-hand sides and the Cholesky factor in FP32 on the
// scaled, centred offsets, followed by one FP64 refinement sweep (residual
// r = b - A c and A^T r in FP64, correction solved with the FP32 factor).
//
// Time levels of one step: pass 1 fits u, v, w at time n and sets
// V^{n+1} = V^n + dt V^n div u^n; pass 2 fits |gdot|^n and V^{n+1} and forms
// the acceleration with V^{n+1}, its gradient and phi^{n+1} = 1/V^{n+1}.
#include "fit_bodies.cuh"

namespace lp {

// ------------------------------------------------------------ pass 1

// ------------------------------------------------------------ pass 2

// ------------------------------------------------------------ kernels

template <int PREC, bool PER>
__global__ void __launch_bounds__(kMaxBlock) k_pass1(const StepArgs A) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < A.n) pass1_body<PREC, PER>(A, s);
}

// pivoted-QR fallback of pass 1 (grid-stride over the queued particles)
__global__ void __launch_bounds__(64) k_pass1_fallback(const StepArgs A) {
  const int cnt = min(*A.fb_count, A.fb_cap);
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < cnt; t += gridDim.x * blockDim.x)
    pass1_fallback_item(A, t);
  if (blockIdx.x == 0 && threadIdx.x == 0 && cnt > 0)
    atomicAdd(&A.dg->n_fallback, (unsigned long long)cnt);
}

// pivoted-QR fallback of pass 2: gradients of |gdot|^n and V^{n+1}
__global__ void __launch_bounds__(64) k_pass2_fallback(const StepArgs A) {
  const int cnt = min(*A.fb_count, A.fb_cap);
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < cnt; t += gridDim.x * blockDim.x)
    pass2_fallback_item(A, t);
}

// float-float kernels: 128 threads per block, at most 128 registers so that
// 4 blocks (16 warps) share an SM
constexpr int kFFBlock = 128;
// Fit threads take the particles of each group of kRowGroup in order of
// stencil size: a warp's lanes then have similar row counts and fewer idle
// at the end of the row loops. perm[g kRowGroup + t] is the particle of rank
// t in group g by (rows, index); the arithmetic of each particle is
// unchanged, only the thread that does it.
#ifndef LP_ROW_GROUP
#define LP_ROW_GROUP 128
#endif
#ifndef LP_PASS2_BLOCKS
#define LP_PASS2_BLOCKS 4
#endif
constexpr int kRowGroup = LP_ROW_GROUP;
__global__ void __launch_bounds__(kRowGroup) k_row_order(int n, const int32_t* __restrict__ cnt,
                                                         int32_t* __restrict__ perm) {
  __shared__ uint32_t key[kRowGroup];
  const int base = blockIdx.x * kRowGroup, t = threadIdx.x, s = base + t;
  key[t] = s < n ? ((uint32_t)min(max(cnt[s], 0), 0xffff) << 16) | (uint32_t)t : 0xffffffffu;
  __syncthreads();
  // bitonic sort of the 128 keys, ascending (past-the-end keys sort last)
  for (int k = 2; k <= kRowGroup; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      const int p = t ^ j;
      if (p > t) {
        const uint32_t a = key[t], b = key[p];
        if ((a > b) == ((t & k) == 0)) {
          key[t] = b;
          key[p] = a;
        }
      }
      __syncthreads();
    }
  if (s < n) perm[s] = base + (int)(key[t] & 0xffffu);
}
__device__ __forceinline__ int fit_particle(const StepArgs& A) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  return (A.perm && t < A.n) ? A.perm[t] : t;
}

// FP64 with fixed-point rows (fixed_rows.cuh). 786,000 particles, per step:
// moments and factor 0.58 ms, right-hand sides and solves 0.77 ms, pass 2
// 0.64 ms; with the rows in FP64, on whose pipe they were bound (91 % busy),
// pass 1 took 5.58 and pass 2 2.66 ms. Now the FP64 pipe (factor, solves,
// closure) is 57 % busy and the warps issue in 0.40 to 0.44 of the cycles. 3 blocks of 128 threads at 168
// registers, or WIDE: 4 blocks at 128 registers, whose few spilled values (8
// to 156 bytes a thread) cost less than the fourth block gives once there are
// more particles than 3 blocks per SM take at a time. LP_FP64 steps with 3 and
// with 4 blocks: 8,000 particles 944 and 977 us (4 steps), 17,000 964 and 976,
// 64,000 1640 and 1573, 227,000 3789 and 3585, 402,000 6017 and 5591. The
// right-hand sides of pass 1 stay at 3: 27 sums and the solve of three fields
// spill 430 bytes (402,000: 5641 with 4).
constexpr int kFxBlock = 128;
constexpr int kFxWide = 3 * 152 * kFxBlock;  // particles that 3 blocks per SM hold
__global__ void k_fx_split(const StepArgs A) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < A.n) fx_split_state_body(A, s);
}
__global__ void k_fx_split_p1(const StepArgs A) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < A.n) fx_split_p1_body(A, s);
}
template <bool PER, bool GH, bool WIDE>
__global__ void __launch_bounds__(kFxBlock, WIDE ? 4 : 3) k_gram_fx(const StepArgs A) {
  const int s = fit_particle(A);
  if (s < A.n) gram_fx_body<PER, GH>(A, s);
}
template <bool PER>
__global__ void __launch_bounds__(kFxBlock, 3) k_pass1_fx(const StepArgs A) {
  const int s = fit_particle(A);
  if (s < A.n) pass1_fx_body<PER>(A, s);
}
template <bool PER, bool GH, bool WIDE>
__global__ void __launch_bounds__(kFxBlock, WIDE ? 4 : 3) k_pass2_fx(const StepArgs A) {
  const int s = fit_particle(A);
  pass2_body<kFixedRows, PER, GH>(A, s, s < A.n);
}
// Few particles: four or two lanes to a particle (k_*_fx_lanes). 8,000
// particles, one thread each, are 250 warps, fewer than the chip has
// schedulers, and each row waits for its gathers; the lanes take a quarter or
// half of the rows each. Four LP_FP64 steps with a thread, two and four lanes
// each (us): 512 particles 869, -, 715; 8,000 939, -, 786; 14,000 -, 831, 822;
// 17,000 959, 890, 1039; 22,000 1059, 992, -; 26,000 1084, 1036, 1102; 31,000
// 1138, 1246, -. The lines: what one wave of the lanes' blocks takes at 12
// warps per SM.
constexpr int kFxSplit4 = 3 * 152 * kFxSlots;
constexpr int kFxSplit2 = 6 * 152 * kFxSlots;
// (particle of rank t, or -1)
struct FxParticles {
  const StepArgs& A;
  __device__ __forceinline__ int operator()(int t) const {
    return t < A.n ? (A.perm ? A.perm[t] : t) : -1;
  }
};
template <bool PER, bool GH, int P>
__global__ void __launch_bounds__(P * kFxSlots, 12 / P) k_gram_fx_lanes(const StepArgs A) {
  gram_fx_lanes<PER, GH, P>(A, FxParticles{A});
}
template <bool PER, int P>
__global__ void __launch_bounds__(P * kFxSlots, 12 / P) k_pass1_fx_lanes(const StepArgs A) {
  pass1_fx_lanes<PER, P>(A, FxParticles{A});
}
template <bool PER, bool GH, int P>
__global__ void __launch_bounds__(P * kFxSlots, 12 / P) k_pass2_fx_lanes(const StepArgs A) {
  pass2_fx_lanes<PER, GH, P>(A, FxParticles{A});
}
int fx_lane_blocks(int n) { return (n + kFxSlots - 1) / kFxSlots; }
template <bool PER, bool GH>
void launch_gram_fx(const StepArgs& A, int nf, int b, cudaStream_t st) {
  if (A.n <= kFxSplit4)
    k_gram_fx_lanes<PER, GH, 4><<<fx_lane_blocks(A.n), 4 * kFxSlots, 0, st>>>(A);
  else if (A.n <= kFxSplit2)
    k_gram_fx_lanes<PER, GH, 2><<<fx_lane_blocks(A.n), 2 * kFxSlots, 0, st>>>(A);
  else if (A.n > kFxWide) k_gram_fx<PER, GH, true><<<nf, b, 0, st>>>(A);
  else k_gram_fx<PER, GH, false><<<nf, b, 0, st>>>(A);
}
template <bool PER>
void launch_pass1_fx(const StepArgs& A, int nf, int b, cudaStream_t st) {
  if (A.n <= kFxSplit4)
    k_pass1_fx_lanes<PER, 4><<<fx_lane_blocks(A.n), 4 * kFxSlots, 0, st>>>(A);
  else if (A.n <= kFxSplit2)
    k_pass1_fx_lanes<PER, 2><<<fx_lane_blocks(A.n), 2 * kFxSlots, 0, st>>>(A);
  else k_pass1_fx<PER><<<nf, b, 0, st>>>(A);
}
template <bool PER, bool GH>
void launch_pass2_fx(const StepArgs& A, int nf, int b, cudaStream_t st) {
  if (A.n <= kFxSplit4)
    k_pass2_fx_lanes<PER, GH, 4><<<fx_lane_blocks(A.n), 4 * kFxSlots, 0, st>>>(A);
  else if (A.n <= kFxSplit2)
    k_pass2_fx_lanes<PER, GH, 2><<<fx_lane_blocks(A.n), 2 * kFxSlots, 0, st>>>(A);
  else if (A.n > kFxWide) k_pass2_fx<PER, GH, true><<<nf, b, 0, st>>>(A);
  else k_pass2_fx<PER, GH, false><<<nf, b, 0, st>>>(A);
}
// the particles that the fixed-point rows left to the plain FP64 rows
constexpr int kSlowBlocks = 4 * 152;
template <bool PER>
__global__ void __launch_bounds__(64) k_pass1_slow(const StepArgs A) {
  const int cnt = min(A.slow_count[0], A.n);
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < cnt; t += gridDim.x * blockDim.x)
    pass1_body<LP_FP64, PER>(A, A.slow[t]);
}
template <bool PER>
__global__ void __launch_bounds__(64) k_pass2_slow(const StepArgs A) {
  const int cnt = min(A.slow_count[1], A.n);
  const int lane = threadIdx.x & 31;
  // a warp at a time, so that every lane calls the body
  for (int b = (blockIdx.x * blockDim.x + threadIdx.x) & ~31; b < cnt; b += gridDim.x * blockDim.x) {
    const int t = b + lane;
    pass2_body<LP_FP64, PER>(A, t < cnt ? A.slow[t] : 0, t < cnt);
  }
}

// (PER: periodic axes, offsets take their nearest image)
template <bool PER>
__global__ void __launch_bounds__(kFFBlock, 4) k_gram_ff(const StepArgs A) {
  const int s = fit_particle(A);
  if (s < A.n) gram_ff_body<PER>(A, s);
}

template <bool PER>
__global__ void __launch_bounds__(kFFBlock, 4) k_pass1_ff_rows(const StepArgs A) {
  const int s = fit_particle(A);
  if (s < A.n) pass1_ff_rows_body<PER>(A, s);
}
__global__ void __launch_bounds__(kFFBlock) k_pass1_ff_solve(const StepArgs A) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < A.n) pass1_ff_solve_body(A, s);
}

__global__ void k_split_state(const StepArgs A) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < A.n) split_state_body(A, s);
}

// rows of the entries with a ghost (free surface), ahead of the main kernels:
// a fixed grid strides over the list of particles that have such entries
// (only they have work), so that a warp's lanes are all busy
constexpr int kTwinBlocks = 4 * 152;
template <bool PER>
__global__ void k_gram_twins(const StepArgs A) {
  const int cnt = min(*A.gcount, A.n);
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < cnt; t += gridDim.x * blockDim.x)
    gram_twins_body<PER>(A, A.glist[t]);
}
template <bool PER>
__global__ void k_pass2_twins(const StepArgs A) {
  const int cnt = min(*A.gcount, A.n);
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < cnt; t += gridDim.x * blockDim.x)
    pass2_twins_body<PER>(A, A.glist[t]);
}

__global__ void k_split_p1(const StepArgs A) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < A.n) split_p1_body(A, s);
}

template <int PREC, bool PER>
__global__ void __launch_bounds__(kMaxBlock) k_pass2(const StepArgs A) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  pass2_body<PREC, PER>(A, s, s < A.n);
}

template <bool PER>
__global__ void __launch_bounds__(kFFBlock, LP_PASS2_BLOCKS) k_pass2_ff(const StepArgs A) {
  const int s = fit_particle(A);
  pass2_body<LP_MIXED_FF, PER>(A, s, s < A.n);
}

// ------------------------------------------------ lp_fit_derivatives

__device__ __forceinline__ void write_coeffs(const FitArgs& F, int s, int f, const double* c) {
  const double ih = F.inv_h, ih2 = ih * ih;
  double* o = F.coeffs + ((int64_t)s * F.nf + f) * kNB;
#pragma unroll
  for (int q = 0; q < kNB; ++q) o[q] = c[q] * (q < 3 ? ih : ih2);
}

// fields are processed in groups of 4 right-hand sides per sweep
template <int PREC>
__device__ __forceinline__ void fit_body(const FitArgs& F, int s) {
  const int n = F.n;
  const int m = min(F.cnt[s], F.cap);
  const double xi = F.x[s], yi = F.y[s], zi = F.z[s];
  const double ih = F.inv_h;
  using T = typename std::conditional<PREC == LP_FP64, double, float>::type;
  Moments<T> M;
  M.zero();
  int rows = 0;  // entries with an index in range
  for (int k = 0; k < m; ++k) {
    const uint32_t code = (uint32_t)F.nbr[(int64_t)k * n + s];
    const int j = code & ~kMirrorBit;
    if ((unsigned)j >= (unsigned)n) continue;  // stale or corrupt stencil entry
    const double zj = (code >> 31) ? F.f2 - F.z[j] : F.z[j];
    M.add(T((F.x[j] - xi) * ih), T((F.y[j] - yi) * ih), T((zj - zi) * ih));
    ++rows;
  }
  T L[kTri];
  M.gram(L);
  const bool ok = chol9(L, PREC == LP_FP64 ? T(1e-9) : T(1e-4)) && rows >= kNB;
  if (!ok) {
    const int slot = atomicAdd(F.fb_count, 1);
    if (slot < F.fb_cap) F.fb_list[slot] = s;
    else atomicOr(&F.dg->flags, (unsigned)LP_FLAG_OVERFLOW);
    return;
  }
  for (int f0 = 0; f0 < F.nf; f0 += 4) {
    const int nf = min(4, F.nf - f0);
    T R[4][kNB];
    double si[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      si[f] = f < nf ? F.fields[f0 + f][s] : 0.0;
#pragma unroll
      for (int c = 0; c < kNB; ++c) R[f][c] = T(0);
    }
    for (int k = 0; k < m; ++k) {
      const uint32_t code = (uint32_t)F.nbr[(int64_t)k * n + s];
      const int j = code & ~kMirrorBit;
      if ((unsigned)j >= (unsigned)n) continue;  // stale or corrupt stencil entry
      const bool mir = code >> 31;
      const double zj = mir ? F.f2 - F.z[j] : F.z[j];
      T a[kNB];
      taylor_row(T((F.x[j] - xi) * ih), T((F.y[j] - yi) * ih), T((zj - zi) * ih), a);
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        if (f < nf) {
          double vj = F.fields[f0 + f][j];
          if (mir) vj *= F.msign[f0 + f];
          const T b = T(vj - si[f]);
#pragma unroll
          for (int c = 0; c < kNB; ++c) R[f][c] += b * a[c];
        }
      }
    }
    double c[4][kNB];
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      chol9_solve(L, R[f]);
#pragma unroll
      for (int q = 0; q < kNB; ++q) c[f][q] = (double)R[f][q];
    }
    if (PREC == LP_MIXED) {
      // one FP64 refinement step
      double g[4][kNB];
#pragma unroll
      for (int f = 0; f < 4; ++f)
#pragma unroll
        for (int q = 0; q < kNB; ++q) g[f][q] = 0.0;
      for (int k = 0; k < m; ++k) {
        const uint32_t code = (uint32_t)F.nbr[(int64_t)k * n + s];
        const int j = code & ~kMirrorBit;
        if ((unsigned)j >= (unsigned)n) continue;  // stale or corrupt stencil entry
        const bool mir = code >> 31;
        const double zj = mir ? F.f2 - F.z[j] : F.z[j];
        double a[kNB];
        taylor_row((F.x[j] - xi) * ih, (F.y[j] - yi) * ih, (zj - zi) * ih, a);
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          if (f < nf) {
            double vj = F.fields[f0 + f][j];
            if (mir) vj *= F.msign[f0 + f];
            double r = vj - si[f];
#pragma unroll
            for (int q = 0; q < kNB; ++q) r -= a[q] * c[f][q];
#pragma unroll
            for (int q = 0; q < kNB; ++q) g[f][q] += a[q] * r;
          }
        }
      }
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        chol9_solve(L, g[f]);
#pragma unroll
        for (int q = 0; q < kNB; ++q) c[f][q] += g[f][q];
      }
    }
    for (int f = 0; f < nf; ++f) write_coeffs(F, s, f0 + f, c[f]);
  }
}
template <int PREC>
__global__ void __launch_bounds__(kBlock) k_fit(const FitArgs F) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < F.n) fit_body<PREC>(F, s);
}
__device__ __forceinline__ int fit_thread(const FitArgs& F) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  return (F.perm && t < F.n) ? F.perm[t] : t;
}

// Poorly conditioned stencils (a relative pivot below 2^-7 in FP64, 2^-10 in
// float-float) that the normal equations still take. Rounding is amplified by
// up to 1 / pivot^2 there (2.5e-11 of the largest derivative for a stencil of
// nine entries), so they take the QR fit where they are few: 0.15 % (2^-7) and
// one in 100,000 (2^-10) of the sweep lattice. Surfaces of lattices with little
// jitter, and all of a sheet of two layers, are such stencils, and a QR fit
// costs many times the normal equations (3 ns in FP64, 1.2 in float-float). With all
// of them by QR (120 ns a fit then) 1.0 M particles of 10 to 18 entries a stencil,
// three fields, took 7.6 to 10 ms in FP64 and 7.3 to 8.4 in float-float; plain
// FP64 rows for every particle took 3.1 to 4.7, float-float sums 1.1 to 1.4.
// So above ill_room (lp_fit_derivatives sets it) none does: they take the plain
// FP64 rows, or keep the float-float fit. The line is on their number, so that
// which stencils take which path does not depend on the order of the threads.
// The QR fit's rank is relative to the largest column (1e-8), the pivots here to
// their own, so that a stencil whose columns' lengths differ by 2^8 or more
// (spacings far from h, or unequal) is not one of them: the QR fit might leave
// columns out.
constexpr int kQrSpreadBits = 16;  // of the squared lengths
__device__ __forceinline__ int ill_by_qr(const FitArgs& F) {
  const int c = F.ill ? *F.ill_count : 0;
  return c <= F.ill_room ? c : 0;
}
__device__ __forceinline__ void push_ill(const FitArgs& F, int s) {
  F.ill[atomicAdd(F.ill_count, 1)] = s;  // (each particle once: n entries at most)
}

// ---- lp_fit_derivatives in FP64 with the rows in fixed point (as the step's
// pass 1, fixed_rows.cuh): records of the positions, moments and factor, then
// the fields in groups of up to three. 170,000 particles, three fields: 1.61 ms
// with FP64 rows, 0.40 now.
constexpr uint8_t kFxSlow = 255;
__global__ void k_fit_fx_split(const FitArgs F, const StepArgs A) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= F.n) return;
  FxRec* R = reinterpret_cast<FxRec*>(A.XU);
  fx_position(A, F.x[s], F.y[s], F.z[s], R[s]);
}
// an entry that may only look near along z (the sums over the fields check all
// stencils; this one is for those refused before them)
__device__ __forceinline__ bool fit_far_in_z(const FitArgs& F, const StepArgs& A, int s, int m) {
  for (int k = 0; k < m; ++k) {
    const uint32_t code = (uint32_t)F.nbr[(int64_t)k * F.n + s];
    const int j = code & ~kMirrorBit;
    if ((unsigned)j >= (unsigned)F.n) continue;  // stale or corrupt stencil entry
    const double d = ((code >> 31) ? F.f2 - F.z[j] : F.z[j]) - F.z[s];
    if (!(fabs(d) * A.K.fx_turn < kFxNear)) return true;
  }
  return false;
}
__global__ void __launch_bounds__(kFxBlock, 3) k_fit_gram_fx(const FitArgs F, const StepArgs A) {
  const int s = fit_thread(F);
  if (s >= F.n) return;
  const int64_t n = F.n;
  const int m = min(F.cnt[s], F.cap);
  double L[kTri];
  int rows = 0;
  const int sh = fx_shift(A, s, m);
  bool fits = sh >= 0, resolved = false;
  if (fits) {
    long long H[31];
    double mo[31];
    fits = fx_moment_rows<false, false, true, 1>(A, s, m, 0, H, &rows, sh);
    resolved = fx_resolved(H);
    fx_moment_values<true>(A.K, H, sh, mo);
    gram_of_moments(mo, L);
  }
  bool even = false;  // the columns' lengths
  if (fits) {
    int lo = __double2hiint(L[0]), hi = lo;
#pragma unroll
    for (int j = 1; j < kNB; ++j) {
      lo = min(lo, __double2hiint(L[tri(j, j)]));
      hi = max(hi, __double2hiint(L[tri(j, j)]));
    }
    even = hi - lo < kQrSpreadBits << 20;
  }
  bool ill = false;
  const bool ok = fits && fx_chol9(L, 1e-9, &ill) && rows >= kNB;
  ill = ill || !resolved;  // (QR needs no moments: it does for these as well)
  A.kx[s] = ok && !ill ? sh : kFxSlow;
  if (!ok && fits && (resolved || rows < kNB) && !fit_far_in_z(F, A, s, m)) {
    const int slot = atomicAdd(F.fb_count, 1);
    if (slot < F.fb_cap) F.fb_list[slot] = s;
    else atomicOr(&F.dg->flags, (unsigned)LP_FLAG_OVERFLOW);
    return;
  }
  if (!ok || (ill && !even)) {
    fx_push(A, s, 0);
    return;
  }
  if (ill) {
    push_ill(F, s);
    return;
  }
#pragma unroll
  for (int k = 0; k < kTri; ++k) A.fac[k * n + s] = L[k];
}
// the group's fields as records
template <int NF>
__global__ void k_fit_fx_fields(const FitArgs F, const StepArgs A, int f0) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= F.n) return;
  FxRec& r = reinterpret_cast<FxRec*>(A.XU)[s];
  float v[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    const double w = F.fields[f0 + f][s];
    fx_field(w, &r.m[f], &r.e[f]);
    v[f] = fx_float(w);
  }
  A.fs[s] = make_float4(v[0], v[1], v[2], fx_coarse(F.z[s], fx_ref(A).z, A.K.fx_turn));
}
template <int NF>
__global__ void __launch_bounds__(kFxBlock, 3) k_fit_rhs_fx(const FitArgs F, const StepArgs A,
                                                            int f0) {
  const int s = fit_thread(F);
  if (s >= F.n) return;
  const int sh = A.kx[s];
  if (sh == kFxSlow) return;  // queued for the plain rows or the QR fit
  const int64_t n = F.n;
  const int m = min(F.cnt[s], F.cap);
  int sgn[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) sgn[f] = (int)F.msign[f0 + f];
  double R[NF][kNB];
  if (!fx_rhs<NF, false, false, true, true>(A, s, m, sgn, nullptr, R, sh)) {
    A.kx[s] = kFxSlow;  // (all of its fields)
    fx_push(A, s, 0);
    return;
  }
  {
    double L[kTri];
#pragma unroll
    for (int k = 0; k < kTri; ++k) L[k] = A.fac[k * n + s];
#pragma unroll
    for (int f = 0; f < NF; ++f) fx_chol9_solve(L, R[f]);
  }
#pragma unroll
  for (int f = 0; f < NF; ++f) write_coeffs(F, s, f0 + f, R[f]);
}
__global__ void __launch_bounds__(64) k_fit_slow(const FitArgs F, const StepArgs A) {
  const int cnt = min(A.slow_count[0], F.n);
  const int all = cnt + (ill_by_qr(F) ? 0 : *F.ill_count);
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < all; t += gridDim.x * blockDim.x)
    fit_body<LP_FP64>(F, t < cnt ? A.slow[t] : F.ill[t - cnt]);
}

// ---- lp_fit_derivatives in float-float (LP_MIXED_FF): positions relative
// to the first particle in units of h (with the floor-mirror height) and the
// fields are split once per particle; the moments, the Cholesky factor and
// the right-hand sides then run on FP32 pairs as in the step's pass 1, with
// the same pivot test and the same pivoted-QR fallback.
__global__ void k_fit_split_ff(const FitArgs F) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= F.n) return;
  const double ox = F.x[0], oy = F.y[0], oz = F.z[0], ih = F.inv_h;
  const ff fx = ff_of((F.x[s] - ox) * ih), fy = ff_of((F.y[s] - oy) * ih);
  const ff fz = ff_of((F.z[s] - oz) * ih), fm = ff_of((F.f2 - F.z[s] - oz) * ih);
  F.xs[s].xh = make_float4(fx.h, fy.h, fz.h, fm.h);
  F.xs[s].xl = make_float4(fx.l, fy.l, fz.l, fm.l);
  for (int f = 0; f < F.nf; ++f) {
    const ff v = ff_of(F.fields[f][s]);
    F.fs[(int64_t)f * F.n + s] = make_float2(v.h, v.l);
  }
}

__global__ void __launch_bounds__(128, 4) k_fit_gram_ff(const FitArgs F) {
  const int s = fit_thread(F);
  if (s >= F.n) return;
  const int n = F.n;
  const int m = min(F.cnt[s], F.cap);
  const float4 hi = F.xs[s].xh, lo = F.xs[s].xl;
  const StepConsts K0{};  // no periodic axes
  ff mo[31];
#pragma unroll
  for (int q = 0; q < 31; ++q) mo[q] = {0.f, 0.f};
  int rows = 0;  // entries with an index in range
  // the neighbour's position one row ahead, its stencil code two rows ahead
  float4 jh = make_float4(0.f, 0.f, 0.f, 0.f), jl = jh;
  auto fetch = [&](uint32_t code) {
    int j = code & ~kMirrorBit;
    if ((unsigned)j >= (unsigned)n) j = s;  // never read outside the arrays (row skipped)
    jh = F.xs[j].xh;
    jl = F.xs[j].xl;
  };
  uint32_t code = m > 0 ? (uint32_t)F.nbr[s] : 0u;
  uint32_t nxt = m > 1 ? (uint32_t)F.nbr[(int64_t)n + s] : 0u;
  if (m > 0) fetch(code);
  for (int k = 0; k < m; ++k) {
    const uint32_t c0 = code;
    const float4 h0 = jh, l0 = jl;
    if (k + 1 < m) {
      code = nxt;
      fetch(code);
      if (k + 2 < m) nxt = (uint32_t)F.nbr[(int64_t)(k + 2) * n + s];
    }
    const int j = c0 & ~kMirrorBit;
    if ((unsigned)j >= (unsigned)n) continue;  // stale or corrupt stencil entry
    ff_moments_add(mo, ff_row_of<false>(hi, lo, h0, l0, c0, K0));
    ++rows;
  }
  ff G[kTri];
  ff_gram_fo(mo, G);
#pragma unroll
  for (int k = 0; k < kTri; ++k) G[k] = ff_norm(G[k]);
  bool ill = false;
  const bool ok = ff_chol9(G, 1e-4f, &ill) && rows >= kNB;
  // (at 2^-7, as in FP64, the QR fits of 2.0 M particles of the sweep cost 0.5 ms)
  if (ok && ill) {  // the QR fit overwrites the float-float one
    float shortest = INFINITY, longest = 0.f;  // the columns' squared lengths, from the factor
#pragma unroll
    for (int j = 0; j < kNB; ++j) {
      float d = 1.f / (G[tri(j, j)].h * G[tri(j, j)].h);
#pragma unroll
      for (int k = 0; k < j; ++k) d += G[tri(j, k)].h * G[tri(j, k)].h;
      shortest = fminf(shortest, d);
      longest = fmaxf(longest, d);
    }
    if (shortest * (float)(1 << kQrSpreadBits) > longest) push_ill(F, s);
  }
  if (!ok) {
    const int slot = atomicAdd(F.fb_count, 1);
    if (slot < F.fb_cap) F.fb_list[slot] = s;
    else atomicOr(&F.dg->flags, (unsigned)LP_FLAG_OVERFLOW);
    F.lf[s] = make_float2(-1.f, 0.f);  // 1/L_00 > 0 for a factored stencil
    return;
  }
#pragma unroll
  for (int k = 0; k < kTri; ++k) F.lf[(int64_t)k * n + s] = make_float2(G[k].h, G[k].l);
}

// Right-hand sides and solves of the float-float fit for the field group
// f0 .. f0 + NG - 1 (one launch per group): the group's NG x 9 sums stay in
// registers, and the neighbour's position and field values are loaded one
// row ahead of the arithmetic (its stencil code two rows ahead), as in the
// step's row kernels.
// (NG = 2: a last group of an odd field count holds one field, and its second
// solve runs on zero sums; 3 blocks of 168 registers, as at 128 the sums spill)
template <int NG>
__global__ void __launch_bounds__(128, 3) k_fit_rhs_ff(const FitArgs F, int f0) {
  const int s = fit_thread(F);
  if (s >= F.n) return;
  if (!(F.lf[s].x > 0.f)) return;  // queued for the pivoted-QR fit
  const int n = F.n;
  const int m = min(F.cnt[s], F.cap);
  const int ng = min(NG, F.nf - f0);
  const float4 hi = F.xs[s].xh, lo = F.xs[s].xl;
  const StepConsts K0{};
  ff R[NG][kNB], si[NG];
  float sg[NG];
#pragma unroll
  for (int f = 0; f < NG; ++f) {
    const float2 v = f < ng ? F.fs[(int64_t)(f0 + f) * n + s] : make_float2(0.f, 0.f);
    si[f] = ff{v.x, v.y};
    sg[f] = f < ng ? (float)F.msign[f0 + f] : 0.f;
#pragma unroll
    for (int q = 0; q < kNB; ++q) R[f][q] = {0.f, 0.f};
  }
  float4 jh = make_float4(0.f, 0.f, 0.f, 0.f), jl = jh;
  float2 jv[NG];
  auto fetch = [&](uint32_t code) {
    int j = code & ~kMirrorBit;
    if ((unsigned)j >= (unsigned)n) j = s;  // never read outside the arrays (row skipped)
    jh = F.xs[j].xh;
    jl = F.xs[j].xl;
#pragma unroll
    for (int f = 0; f < NG; ++f)
      jv[f] = f < ng ? F.fs[(int64_t)(f0 + f) * n + j] : make_float2(0.f, 0.f);
  };
  uint32_t code = m > 0 ? (uint32_t)F.nbr[s] : 0u;
  uint32_t nxt = m > 1 ? (uint32_t)F.nbr[(int64_t)n + s] : 0u;
  if (m > 0) fetch(code);
  for (int k = 0; k < m; ++k) {
    const uint32_t c0 = code;
    const float4 h0 = jh, l0 = jl;
    float2 v0[NG];
#pragma unroll
    for (int f = 0; f < NG; ++f) v0[f] = jv[f];
    if (k + 1 < m) {
      code = nxt;
      fetch(code);
      if (k + 2 < m) nxt = (uint32_t)F.nbr[(int64_t)(k + 2) * n + s];
    }
    const int j = c0 & ~kMirrorBit;
    if ((unsigned)j >= (unsigned)n) continue;  // stale or corrupt stencil entry
    const bool mir = c0 >> 31;
    ff a[kNB];
    ff_taylor(ff_row_of<false>(hi, lo, h0, l0, c0, K0), a);
#pragma unroll
    for (int f = 0; f < NG; ++f) {
      if (f < ng) {
        const float sj = mir ? sg[f] : 1.f;  // the field at a floor mirror
        const ff b = ff_diff(sj * v0[f].x, sj * v0[f].y, si[f].h, si[f].l);
#pragma unroll
        for (int q = 0; q < kNB; ++q) ff_acc(R[f][q], b, a[q]);
      }
    }
  }
  // one field at a time: the joint solve of a 2-D array of sums makes the
  // compiler keep them in local memory
  ff_chol_solve<1>(F.lf + s, n, R + 0);
  if (NG > 1) ff_chol_solve<1>(F.lf + s, n, R + 1);
  const double ih = F.inv_h, ih2 = ih * ih;
#pragma unroll
  for (int f = 0; f < NG; ++f) {
    if (f < ng) {
      double* o = F.coeffs + ((int64_t)s * F.nf + f0 + f) * kNB;
#pragma unroll
      for (int q = 0; q < kNB; ++q) o[q] = ff_to_double(R[f][q]) * (q < 3 ? ih : ih2);
    }
  }
}

// Pivoted-QR fits of the queued particles, the same algorithm as
// qr_pivoted_solve (pivot: the largest remaining norm, ties to the lower
// column; rank by 1e-8; basic solution).
//
// Few: a warp for each, a lane holding rows lane and lane + 32 of [A | B] in
// registers, and every column norm and reflection a sum over the warp. What
// bounds it is one warp's chain on the FP64 pipe, 75 cycles an instruction, so
// the sums of a column's norms, or of its reflections, are taken together: each
// step halves the number of values a lane holds (9 additions for 8 sums instead
// of 40), rows past the 32nd and absent fields are skipped, and a lane takes the
// back substitution of one field. A call with one QR fit of 12 to 48 rows takes
// 45 us longer than one without; with a sum at a time 75 to 90.
// Many: a thread for each, its matrix in local memory (fit_qr_item). Particles
// with six entries, all refused, LP_FP64, three fields: 8,000 take 147 us
// (1046 with a warp each, summed one at a time), 1.0 M 5.8 ms (120). The line,
// two waves of warps: 1,728 fits of six entries take 131 us with a thread each
// and 166 with a warp (LP_MIXED_FF 119 and 154); with 48 entries a wave of
// thread fits takes 200 us, one of 608 warp fits 45.
template <int N>
__device__ __forceinline__ void warp_sums(double* v, int lane) {
  constexpr int P = N > 8 ? 8 : (N > 4 ? 8 : (N > 2 ? 4 : N));
  double w[P];
#pragma unroll
  for (int i = 0; i < P; ++i) w[i] = i < N ? v[i] : 0.0;
  int bit = 16;
#pragma unroll
  for (int h = P / 2; h >= 1; h >>= 1) {
    const bool up = lane & bit;
#pragma unroll
    for (int i = 0; i < h; ++i)
      w[i] = (up ? w[i + h] : w[i]) + __shfl_xor_sync(0xffffffffu, up ? w[i] : w[i + h], bit);
    bit >>= 1;
  }
#pragma unroll
  for (; bit; bit >>= 1) w[0] += __shfl_xor_sync(0xffffffffu, w[0], bit);
#pragma unroll
  for (int i = 0; i < P; ++i) {  // (value i lies in the lanes with these bits)
    int src = 0;
#pragma unroll
    for (int h = P / 2, b = 16; h >= 1; h >>= 1, b >>= 1) src |= (i & h) ? b : 0;
    if (i < N) v[i] = __shfl_sync(0xffffffffu, w[0], src);
  }
  if constexpr (N > P) warp_sums<N - P>(v + P, lane);
}
// (two: there are rows past the 32nd)
template <int K>
__device__ __forceinline__ bool qr_column(double (*a)[kNB], double (*b)[4], int nf, bool two,
                                          int* perm, double* rdiag, int lane) {
  // row index of a[h]: lane + 32 h; rows above K are done
  const bool in = lane >= K;
  constexpr int J = kNB - K;  // columns left
  double s[J + 3];            // (J norms, or J - 1 columns and 4 fields)
#pragma unroll
  for (int j = 0; j < J; ++j) s[j] = in ? a[0][K + j] * a[0][K + j] : 0.0;
  if (two) {
#pragma unroll
    for (int j = 0; j < J; ++j) s[j] += a[1][K + j] * a[1][K + j];
  }
  warp_sums<J>(s, lane);
  int best = K;
  double bestn = -1.0;
#pragma unroll
  for (int j = 0; j < J; ++j)
    if (s[j] > bestn) { bestn = s[j]; best = K + j; }
  const double alpha = sqrt(bestn);
  if (alpha == 0.0 || !(bestn >= 0.0)) {  // (a NaN norm never wins: all columns are NaN)
    rdiag[K] = bestn >= 0.0 ? 0.0 : __longlong_as_double(0x7ff8000000000000ll);
    return false;
  }
#pragma unroll
  for (int j = K + 1; j < kNB; ++j)
    if (j == best) {
#pragma unroll
      for (int h = 0; h < 2; ++h) { const double t = a[h][K]; a[h][K] = a[h][j]; a[h][j] = t; }
      const int t = perm[K]; perm[K] = perm[j]; perm[j] = t;
    }
  const double akk = __shfl_sync(0xffffffffu, a[0][K], K);
  const double sgn = akk >= 0.0 ? 1.0 : -1.0;
  const double v0 = lane == K ? akk + sgn * alpha : (in ? a[0][K] : 0.0), v1 = a[1][K];
  const double f = 1.0 / (bestn + fabs(akk) * alpha);  // 2 / v.v
#pragma unroll
  for (int j = 1; j < J; ++j) s[j - 1] = v0 * a[0][K + j];
#pragma unroll
  for (int q = 0; q < 4; ++q) s[J - 1 + q] = q < nf ? v0 * b[0][q] : 0.0;
  if (two) {
#pragma unroll
    for (int j = 1; j < J; ++j) s[j - 1] += v1 * a[1][K + j];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < nf) s[J - 1 + q] += v1 * b[1][q];
  }
  warp_sums<J + 3>(s, lane);
#pragma unroll
  for (int j = 1; j < J; ++j) {
    s[j - 1] *= f;
    a[0][K + j] -= s[j - 1] * v0;
    if (two) a[1][K + j] -= s[j - 1] * v1;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (q < nf) {
      s[J - 1 + q] *= f;
      b[0][q] -= s[J - 1 + q] * v0;
      if (two) b[1][q] -= s[J - 1 + q] * v1;
    }
  rdiag[K] = -sgn * alpha;
  return true;
}
// one fit by a warp (pk: its shared codes)
__device__ __forceinline__ void fit_qr_warp(const FitArgs& F, int s, uint32_t* pk, int lane) {
  const int n = F.n;
  const int m = min(F.cnt[s], F.cap);
  const double xi = F.x[s], yi = F.y[s], zi = F.z[s];
  // rows are packed: an entry whose index is out of range is dropped and the
  // rows after it move up; lanes past the last row hold zeros
  pk[lane] = pk[lane + 32] = ~kMirrorBit;
  __syncwarp();
  int rows = 0;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int k = lane + 32 * h;
    const uint32_t c = k < m ? (uint32_t)F.nbr[(int64_t)k * n + s] : ~kMirrorBit;
    const bool in = (c & ~kMirrorBit) < (uint32_t)n;
    const unsigned all = __ballot_sync(0xffffffffu, in);
    if (in) pk[rows + __popc(all & ((1u << lane) - 1u))] = c;
    rows += __popc(all);
  }
  __syncwarp();
  const bool two = rows > 32;
  uint32_t code[2];
  double row[2][kNB];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    code[h] = pk[lane + 32 * h];
    const int j = code[h] & ~kMirrorBit;
#pragma unroll
    for (int q = 0; q < kNB; ++q) row[h][q] = 0.0;
    if ((unsigned)j < (unsigned)n) {
      const double zj = (code[h] >> 31) ? F.f2 - F.z[j] : F.z[j];
      taylor_row((F.x[j] - xi) * F.inv_h, (F.y[j] - yi) * F.inv_h, (zj - zi) * F.inv_h, row[h]);
    }
  }
  for (int f0 = 0; f0 < F.nf; f0 += 4) {
    const int nf = min(4, F.nf - f0);
    double a[2][kNB], b[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int j = code[h] & ~kMirrorBit;
#pragma unroll
      for (int q = 0; q < kNB; ++q) a[h][q] = row[h][q];
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        b[h][f] = 0.0;
        if (f < nf && (unsigned)j < (unsigned)n) {
          double vj = F.fields[f0 + f][j];
          if (code[h] >> 31) vj *= F.msign[f0 + f];
          b[h][f] = vj - F.fields[f0 + f][s];
        }
      }
    }
    int perm[kNB];
    double rd[kNB];
#pragma unroll
    for (int q = 0; q < kNB; ++q) { perm[q] = q; rd[q] = 0.0; }
    qr_column<0>(a, b, nf, two, perm, rd, lane) && qr_column<1>(a, b, nf, two, perm, rd, lane) &&
        qr_column<2>(a, b, nf, two, perm, rd, lane) &&
        qr_column<3>(a, b, nf, two, perm, rd, lane) &&
        qr_column<4>(a, b, nf, two, perm, rd, lane) &&
        qr_column<5>(a, b, nf, two, perm, rd, lane) &&
        qr_column<6>(a, b, nf, two, perm, rd, lane) &&
        qr_column<7>(a, b, nf, two, perm, rd, lane) &&
        qr_column<8>(a, b, nf, two, perm, rd, lane);
    int rank = 0;
    bool run = true;
#pragma unroll
    for (int q = 0; q < kNB; ++q) {
      run = run && fabs(rd[q]) > 1e-8 * fabs(rd[0]);  // (NaN: the columns before it count)
      rank += run;
    }
    double y[kNB];  // of field f0 + lane
#pragma unroll
    for (int k = kNB - 1; k >= 0; --k) {
      double v = 0.0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const double t = __shfl_sync(0xffffffffu, b[0][q], k);
        if (q == lane) v = t;
      }
#pragma unroll
      for (int j = k + 1; j < kNB; ++j) {
        const double t = __shfl_sync(0xffffffffu, a[0][j], k);
        if (j < rank) v -= t * y[j];  // (past the rank it may be NaN)
      }
      y[k] = k < rank ? v / rd[k] : 0.0;
    }
    if (lane < nf) {
      double* o = F.coeffs + ((int64_t)s * F.nf + f0 + lane) * kNB;
#pragma unroll
      for (int k = 0; k < kNB; ++k)
        o[perm[k]] = y[k] * (perm[k] < 3 ? F.inv_h : F.inv_h * F.inv_h);
    }
  }
  __syncwarp();  // (pk is reused)
}
// one fit by a thread
__device__ __noinline__ void fit_qr_item(const FitArgs& F, int s) {
  double Am[LP_MAX_CAP * kNB], Bm[LP_MAX_CAP * 4], C[4 * kNB];
  const int n = F.n;
  const int m = min(F.cnt[s], F.cap);
  const double xi = F.x[s], yi = F.y[s], zi = F.z[s];
  for (int f0 = 0; f0 < F.nf; f0 += 4) {
    const int nf = min(4, F.nf - f0);
    int rows = 0;  // (packed, as above)
    for (int k = 0; k < m; ++k) {
      const uint32_t code = (uint32_t)F.nbr[(int64_t)k * n + s];
      const int j = code & ~kMirrorBit;
      if ((unsigned)j >= (unsigned)n) continue;  // stale or corrupt stencil entry
      const bool mir = code >> 31;
      const double zj = mir ? F.f2 - F.z[j] : F.z[j];
      taylor_row((F.x[j] - xi) * F.inv_h, (F.y[j] - yi) * F.inv_h, (zj - zi) * F.inv_h,
                 &Am[rows * kNB]);
      for (int f = 0; f < nf; ++f) {
        double vj = F.fields[f0 + f][j];
        if (mir) vj *= F.msign[f0 + f];
        Bm[rows * nf + f] = vj - F.fields[f0 + f][s];
      }
      ++rows;
    }
    qr_pivoted_solve(rows, Am, nf, Bm, C);
    for (int f = 0; f < nf; ++f) write_coeffs(F, s, f0 + f, C + f * kNB);
  }
}
constexpr int kQrWarpFits = 1216;
__global__ void __launch_bounds__(64) k_fit_fallback(const FitArgs F) {
  const int cnt = min(*F.fb_count, F.fb_cap);
  const int all = cnt + ill_by_qr(F);
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31;
  __shared__ uint32_t packed[2][LP_MAX_CAP];
  if (all <= kQrWarpFits) {
    for (int t = tid >> 5; t < all; t += nth >> 5)
      fit_qr_warp(F, t < cnt ? F.fb_list[t] : F.ill[t - cnt], packed[threadIdx.x >> 5], lane);
  } else {
    for (int t = tid; t < all; t += nth) fit_qr_item(F, t < cnt ? F.fb_list[t] : F.ill[t - cnt]);
  }
  // (those of the normal equations' choice count: the refused ones)
  if (tid == 0 && cnt > 0) atomicAdd(&F.dg->n_fallback, (unsigned long long)cnt);
}

// ---------------------------------------------------------- lp_mui_stress

__global__ void k_mui_stress(int64_t n, ColMui mui, double phi_c, double phi_min,
                             double phi_max, double alpha, double beta,
                             const double* __restrict__ V, const double* __restrict__ gu,
                             double* gdot, double* gnorm, double* P, double* eta,
                             int8_t* regime) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double* G = gu + 9 * i;
  const double div = (G[0] + G[4]) + G[8];
  const double d3 = div * (1.0 / 3.0);
  const double gxx = G[0] - d3, gyy = G[4] - d3, gzz = G[8] - d3;
  const double gxy = 0.5 * (G[1] + G[3]), gxz = 0.5 * (G[2] + G[6]), gyz = 0.5 * (G[5] + G[7]);
  const double gn =
      sqrt(0.5 * (gxx * gxx + gyy * gyy + gzz * gzz + 2.0 * (gxy * gxy + gxz * gxz + gyz * gyz)));
  if (gdot) {
    double* o = gdot + 6 * i;
    o[0] = gxx; o[1] = gyy; o[2] = gzz; o[3] = gxy; o[4] = gxz; o[5] = gyz;
  }
  if (gnorm) gnorm[i] = gn;
  const double phi = 1.0 / V[i];
  double p, e;
  int r;
  if (phi <= phi_min) {
    r = 0; p = 0.0; e = 0.0;
  } else if (phi <= phi_max) {
    r = 1;
    const double a = phi_c - phi_min;
    const double q = (2.0 * a * mui.d * gn) / (phi_c - phi);
    p = mui.rho_s * q * q;
    const Closure cl = closure_at(phi, mui, phi_c, phi_min);
    e = mui.rho_s * cl.N * gn;  // mu(I) P / |gdot|
  } else {
    r = 2; p = mui.rho_s * (alpha + beta * phi); e = 0.0;
  }
  if (P) P[i] = p;
  if (eta) eta[i] = e;
  if (regime) regime[i] = (int8_t)r;
}

// ------------------------------------------------------------- launchers

void launch_pass1(int prec, const StepArgs& A, cudaStream_t st, int bs) {
  bs = spread_block(A.n, bs);
  const int sb = spread_block(A.n, 256);  // of the splitting kernels
  const int nb = (A.n + bs - 1) / bs;
  const bool per = A.K.periodic != 0;
  if (prec == LP_FP64) {
    k_fx_split<<<(A.n + sb - 1) / sb, sb, 0, st>>>(A);
    if (A.perm) k_row_order<<<(A.n + kRowGroup - 1) / kRowGroup, kRowGroup, 0, st>>>(A.n, A.cnt, const_cast<int32_t*>(A.perm));
    const int b = bs < kFxBlock ? bs : kFxBlock;
    const int nf = (A.n + b - 1) / b;
    if (per) {
      if (A.K.free_surface) launch_gram_fx<true, true>(A, nf, b, st);
      else launch_gram_fx<true, false>(A, nf, b, st);
      launch_pass1_fx<true>(A, nf, b, st);
      k_pass1_slow<true><<<kSlowBlocks, 64, 0, st>>>(A);
    } else {
      if (A.K.free_surface) launch_gram_fx<false, true>(A, nf, b, st);
      else launch_gram_fx<false, false>(A, nf, b, st);
      launch_pass1_fx<false>(A, nf, b, st);
      k_pass1_slow<false><<<kSlowBlocks, 64, 0, st>>>(A);
    }
  } else if (prec == LP_MIXED) {
    if (per) k_pass1<LP_MIXED, true><<<nb, bs, 0, st>>>(A);
    else k_pass1<LP_MIXED, false><<<nb, bs, 0, st>>>(A);
  } else {
    k_split_state<<<(A.n + sb - 1) / sb, sb, 0, st>>>(A);
    if (A.perm) k_row_order<<<(A.n + kRowGroup - 1) / kRowGroup, kRowGroup, 0, st>>>(A.n, A.cnt, const_cast<int32_t*>(A.perm));
    const int b = bs < kFFBlock ? bs : kFFBlock;
    const int nf = (A.n + b - 1) / b;
    if (per) {
      if (A.K.free_surface) k_gram_twins<true><<<kTwinBlocks, 128, 0, st>>>(A);
      k_gram_ff<true><<<nf, b, 0, st>>>(A);
      k_pass1_ff_rows<true><<<nf, b, 0, st>>>(A);
    } else {
      if (A.K.free_surface) k_gram_twins<false><<<kTwinBlocks, 128, 0, st>>>(A);
      k_gram_ff<false><<<nf, b, 0, st>>>(A);
      k_pass1_ff_rows<false><<<nf, b, 0, st>>>(A);
    }
    k_pass1_ff_solve<<<nf, b, 0, st>>>(A);
  }
  k_pass1_fallback<<<152, 64, 0, st>>>(A);
}
void launch_pass2(int prec, const StepArgs& A, cudaStream_t st, int bs) {
  bs = spread_block(A.n, bs);
  const int sb = spread_block(A.n, 256);  // of the splitting kernels
  if (prec == LP_MIXED_FF) {
    k_split_p1<<<(A.n + sb - 1) / sb, sb, 0, st>>>(A);
    if (A.K.free_surface) {
      if (A.K.periodic) k_pass2_twins<true><<<kTwinBlocks, 128, 0, st>>>(A);
      else k_pass2_twins<false><<<kTwinBlocks, 128, 0, st>>>(A);
    }
  }
  if (prec == LP_FP64) k_fx_split_p1<<<(A.n + sb - 1) / sb, sb, 0, st>>>(A);
  k_pass2_fallback<<<152, 64, 0, st>>>(A);
  const int nb = (A.n + bs - 1) / bs;
  const bool per = A.K.periodic != 0;
  if (prec == LP_FP64) {
    const int b = bs < kFxBlock ? bs : kFxBlock;
    const int nf = (A.n + b - 1) / b;
    if (per) {
      if (A.K.free_surface) launch_pass2_fx<true, true>(A, nf, b, st);
      else launch_pass2_fx<true, false>(A, nf, b, st);
      k_pass2_slow<true><<<kSlowBlocks, 64, 0, st>>>(A);
    } else {
      if (A.K.free_surface) launch_pass2_fx<false, true>(A, nf, b, st);
      else launch_pass2_fx<false, false>(A, nf, b, st);
      k_pass2_slow<false><<<kSlowBlocks, 64, 0, st>>>(A);
    }
  } else if (prec == LP_MIXED) {
    if (per) k_pass2<LP_MIXED, true><<<nb, bs, 0, st>>>(A);
    else k_pass2<LP_MIXED, false><<<nb, bs, 0, st>>>(A);
  } else {
    const int b = bs < kFFBlock ? bs : kFFBlock;
    if (per) k_pass2_ff<true><<<(A.n + b - 1) / b, b, 0, st>>>(A);
    else k_pass2_ff<false><<<(A.n + b - 1) / b, b, 0, st>>>(A);
  }
}
void launch_fit(int prec, const FitArgs& F, cudaStream_t st) {
  const int bs = spread_block(F.n, kBlock);
  const int nb = (F.n + bs - 1) / bs;
  if (F.perm)
    k_row_order<<<(F.n + kRowGroup - 1) / kRowGroup, kRowGroup, 0, st>>>(
        F.n, F.cnt, const_cast<int32_t*>(F.perm));
  if (prec == LP_FP64 && F.rows) {
    const StepArgs& A = *F.rows;
    const int sb = spread_block(F.n, 256), ns = (F.n + sb - 1) / sb;
    k_fit_fx_split<<<ns, sb, 0, st>>>(F, A);
    k_fit_gram_fx<<<nb, bs, 0, st>>>(F, A);
    for (int f0 = 0; f0 < F.nf;) {
      const int left = F.nf - f0, g = left == 4 ? 2 : (left < 3 ? left : 3);
      if (g == 3) {
        k_fit_fx_fields<3><<<ns, sb, 0, st>>>(F, A, f0);
        k_fit_rhs_fx<3><<<nb, bs, 0, st>>>(F, A, f0);
      } else if (g == 2) {
        k_fit_fx_fields<2><<<ns, sb, 0, st>>>(F, A, f0);
        k_fit_rhs_fx<2><<<nb, bs, 0, st>>>(F, A, f0);
      } else {
        k_fit_fx_fields<1><<<ns, sb, 0, st>>>(F, A, f0);
        k_fit_rhs_fx<1><<<nb, bs, 0, st>>>(F, A, f0);
      }
      f0 += g;
    }
    k_fit_slow<<<kSlowBlocks, 64, 0, st>>>(F, A);
  } else if (prec == LP_FP64) {
    k_fit<LP_FP64><<<nb, bs, 0, st>>>(F);
  } else if (prec == LP_MIXED) {
    k_fit<LP_MIXED><<<nb, bs, 0, st>>>(F);
  } else {
    k_fit_split_ff<<<(F.n + 255) / 256, 256, 0, st>>>(F);
    k_fit_gram_ff<<<nb, bs, 0, st>>>(F);
    for (int f0 = 0; f0 < F.nf; f0 += 2) k_fit_rhs_ff<2><<<nb, bs, 0, st>>>(F, f0);
  }
  k_fit_fallback<<<2 * 152, 64, 0, st>>>(F);
}
void launch_mui_stress(int64_t n, const ColMui& m, const lp_eos& e, const double* V,
                       const double* gu, double* gdot, double* gnorm, double* P, double* eta,
                       int8_t* regime, cudaStream_t st) {
  k_mui_stress<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, m, e.phi_c, e.phi_min, e.phi_max,
                                                            e.alpha, e.beta, V, gu, gdot, gnorm,
                                                            P, eta, regime);
}

}  // namespace lp
