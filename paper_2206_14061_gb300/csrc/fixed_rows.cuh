// Stencil rows in 64-bit fixed point: the sums of the LP_FP64 fits.
//
// GB300 issues FP64 at about 1.7 lanes per SM and clock, against 118 for FP32
// and 25 for 32 x 32 + 64-bit integer multiply-adds (measured). A stencil's
// sums took 82 FP64 operations per row in pass 1 and 36 in pass 2, and bound
// the FP64 step (pass 1 5.6 ms, pass 2 2.7 ms on 786,000 particles). Every
// factor of those sums is bounded once the row's scale is known, so here they
// run in fixed point on the integer and FP32 pipes and only the 9 x 9
// factor and solves stay FP64.
//
// A factor v is held as h + l, h a 28-bit integer and l the rest of it in
// units of h, |l| <= 1/2, as a float. A product a b enters its sum as
//   a.h b.h                       exact, one 32 x 32 + 64-bit multiply-add
//   round(a.h b.l + a.l b.h)      FP32, to an integer (a.l b.l is below 1/4)
// so a term errs by 2^-54 of the largest possible one (rms; the FP32 operations,
// on 28-bit values, put the most at 2^-51), where an FP64 sum rounds at 2^-53 of
// the running sum in every row. The sums are
// exact, so their order does not matter, and 64 rows of 2^56 cannot overflow
// them. (Keeping the second part as a float sum, moved into the integer one
// every fourth row, is as fast and errs by 2^-50.) About 8 cycles per
// accumulation and scheduler; an FP64 multiply-add takes about 75.
//
// Positions are integers X = x 2^k modulo 2^64, with r 2^k in (2^59, 2^60]
// for the stencil radius r (a quarter of it in lp_fit_derivatives, see
// kFxMostShift): the conversion is exact for all but the last bits
// of tiny coordinates, and differences of neighbours are exact whatever the
// distance from the origin (the modular wrap cancels). As entries of a stencil
// may be anywhere (held stencils, a caller's own lists), the offsets are also
// taken in FP32 in units of the wrap, to see one that only looks near. Field
// values (u, v, w; |gdot|, V) are aligned per stencil to its largest value, and
// their differences shifted up to fill the range; the scales come from a first
// walk over FP32 copies.
//
// What does not fit (offsets beyond about the radius, which only stencils held
// fixed over several steps or a caller's own can have; stencils thin along an
// axis or small against the radius, see fx_resolved; fields whose differences
// are not finite or are below 2^-90; non-finite positions) is queued for a
// kernel that runs the plain FP64 rows. Where all particles are, a step takes 3
// to 9 % longer than with those rows alone (640,000 particles in a sheet
// compressed to 0.1: 6.89 and 6.35 ms; 2.07 in fixed point, wrong in the twelfth
// digit).
#pragma once

#include "lp_internal.cuh"

namespace lp {

// round(v 2^k) modulo 2^64 (0 for non-finite v, which callers sort out)
__host__ __device__ __forceinline__ unsigned long long fx_of(double v, int k) {
#ifdef __CUDA_ARCH__
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
#else
  unsigned long long b;
  __builtin_memcpy(&b, &v, sizeof b);
#endif
  const int e = (int)((b >> 52) & 0x7ff);
  const unsigned long long m = (b & 0xfffffffffffffull) | (e ? 0x10000000000000ull : 0ull);
  const int sh = e - 1075 + k;
  const unsigned long long left = sh < 64 ? m << (sh & 63) : 0ull;
  const int t = -sh - 1;  // right shift by -sh, rounded
  const unsigned long long right = t < 64 ? ((m >> (t & 63)) + 1ull) >> 1 : 0ull;
  const unsigned long long r = sh >= 0 ? left : right;
  return (b >> 63) ? 0ull - r : r;
}

// One particle of the rows: fixed-point position (with the coarse coordinates,
// see fx_coarse, that choose the nearest image and tell far entries; xf is NaN
// if one of the three is) and the
// field values of the pass as signed significands (53 bits, the top one at bit
// 58) with their exponents, so that a row aligns a value to its stencil's scale
// with one shift. A value is m 2^(e - 58).
struct __align__(64) FxRec {
  unsigned long long X, Y, Z;
  float xf, yf;
  long long m[3];
  short e[4];
};
__device__ __forceinline__ void fx_field(double v, long long* m, short* e) {
  const long long b = __double_as_longlong(v);
  const int x = (int)((b >> 52) & 0x7ff);
  // (subnormal values count as 0: they are queued by the scale walk)
  const long long t = x ? ((b & 0xfffffffffffffll) | 0x10000000000000ll) << 6 : 0ll;
  *m = b < 0 ? -t : t;
  *e = (short)(x - 1023);
}

struct FxV {  // value h + l; hf = float(h)
  int h;
  float hf, l;
};
// (multiply-adds on 64-bit sums as one instruction each)
__device__ __forceinline__ long long fx_mad(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
__device__ __forceinline__ FxV fx_split(unsigned long long D) {
  FxV v;
  v.h = (int)((D + 0x80000000ull) >> 32);
  v.hf = (float)v.h;
  v.l = __fmul_rn((float)(int)(unsigned)D, 0x1p-32f);
  return v;
}
// product of two values, rounded to an integer in units of h h
__device__ __forceinline__ long long fx_mul(const FxV& a, const FxV& b) {
  const float c = __fmaf_rn(a.l, b.hf, __fmul_rn(a.hf, b.l));
  return fx_mad(a.h, b.h, (long long)__float2int_rn(c));
}
// a product as a factor again: units 2^sq
__device__ __forceinline__ FxV fx_quad(long long Q, int sq, float qs) {
  FxV v;
  v.h = (int)((Q + (1ll << (sq - 1))) >> sq);
  v.hf = (float)v.h;
  v.l = __fmul_rn((float)(int)((unsigned)Q - ((unsigned)v.h << sq)), qs);
  return v;
}
__device__ __forceinline__ void fx_acc(long long& H, const FxV& a, const FxV& b) {
  const int c = __float2int_rn(__fmaf_rn(a.l, b.hf, __fmul_rn(a.hf, b.l)));
  H = fx_mad(a.h, b.h, H) + (long long)c;
}
// A coordinate in units of the wrap 2^(64 - k), from that of the first
// particle; NaN from 2^20 on. Its errors (the rounding of both coordinates of
// a difference, and of the mirror plane) are below 0.16, so a difference below
// kFxNear is one of less than half a wrap, and every offset that the range
// takes (1/14 of a wrap) is below it.
constexpr float kFxNear = 0.25f;
__device__ __forceinline__ float fx_coarse(double v, double ref, double turn) {
  const float c = __double2float_rn(__dmul_rn(__dsub_rn(v, ref), turn));
  return fabsf(c) < 0x1p20f ? c : __int_as_float(0x7fffffff);
}
__device__ __forceinline__ double pow2_of(int e) {  // 2^e, a normal double
  return __longlong_as_double((long long)(1023 + e) << 52);
}

// offsets of entry j of a particle at `me` (PER: nearest images)
// (SH: shifted up by sh). True if the entry is near along x and y: the offsets
// are below half a wrap, so the fixed-point ones are the true ones. (Along z:
// fx_rhs_rows, from the copy that its first walk reads anyway.)
template <bool PER, bool SH>
__device__ __forceinline__ bool fx_offsets(const StepConsts& K, int sh, const FxRec& me,
                                           unsigned long long Xj, unsigned long long Yj,
                                           unsigned long long Zj, float xf, float yf, bool mir,
                                           unsigned long long* D) {
  D[0] = Xj - me.X;
  D[1] = Yj - me.Y;
  D[2] = (mir ? K.fx_F2 - Zj : Zj) - me.Z;
  float dx = xf - me.xf, dy = yf - me.yf;
  if (PER) {
    if (fabsf(dx) > K.fx_hLx) {
      D[0] -= dx > 0.f ? K.fx_Lx : 0ull - K.fx_Lx;
      dx -= copysignf(2.f * K.fx_hLx, dx);
    }
    if (fabsf(dy) > K.fx_hLy) {
      D[1] -= dy > 0.f ? K.fx_Ly : 0ull - K.fx_Ly;
      dy -= copysignf(2.f * K.fx_hLy, dy);
    }
  }
  if (SH) {
#pragma unroll
    for (int a = 0; a < 3; ++a) D[a] <<= sh;
  }
  return fabsf(dx) < kFxNear && fabsf(dy) < kFxNear;  // (false for NaN)
}

// row loop state: the neighbour's position one row ahead, its code two rows ahead
struct FxPosLoad {
  ulonglong2 xy;
  ulonglong2 zf;  // Z and the two floats
  __device__ __forceinline__ void fetch(const FxRec* R, uint32_t j, int n, int s) {
    if (j >= (uint32_t)n) j = (uint32_t)s;  // never read outside the arrays (row skipped)
    const ulonglong2* p = reinterpret_cast<const ulonglong2*>(R + j);
    xy = p[0];
    zf = p[1];
  }
  __device__ __forceinline__ float xf() const { return __uint_as_float((unsigned)zf.y); }
  __device__ __forceinline__ float yf() const { return __uint_as_float((unsigned)(zf.y >> 32)); }
};

__device__ __forceinline__ void fx_rec_pos(FxRec& r, const FxRec* R, int s) {
  FxPosLoad p;
  const ulonglong2* q = reinterpret_cast<const ulonglong2*>(R + s);
  p.xy = q[0];
  p.zf = q[1];
  r.X = p.xy.x; r.Y = p.xy.y; r.Z = p.zf.x;
  r.xf = p.xf(); r.yf = p.yf();
}

__device__ __forceinline__ void fx_push(const StepArgs& A, int s, int list) {
  A.slow[atomicAdd(&A.slow_count[list], 1)] = s;  // each particle once per list of n
}

// FP32 copy of a field for the scale walk: 0 only for 0, so that a tiny value
// cannot pass for it
__device__ __forceinline__ float fx_float(double v) {
  const float f = __double2float_rn(v);
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  return (fabsf(f) < 0x1p-100f && (b << 1)) ? copysignf(0x1p-100f, (b >> 63) ? -1.f : 1.f) : f;
}

// the first particle's coordinates (0 for one that is not finite)
struct FxRef {
  double x, y, z;
};
__device__ __forceinline__ FxRef fx_ref(const StepArgs& A) {
  FxRef o{A.x[0], A.y[0], A.z[0]};
  if (!isfinite(o.x)) o.x = 0.0;
  if (!isfinite(o.y)) o.y = 0.0;
  if (!isfinite(o.z)) o.z = 0.0;
  return o;
}
// the position half of a record; the z's coarse coordinate is returned
__device__ __forceinline__ float fx_position(const StepArgs& A, double x, double y, double z,
                                             FxRec& r) {
  const int k = A.K.fx_k;
  r.X = fx_of(x, k); r.Y = fx_of(y, k); r.Z = fx_of(z, k);
  const FxRef o = fx_ref(A);
  const float xf = fx_coarse(x, o.x, A.K.fx_turn), zf = fx_coarse(z, o.z, A.K.fx_turn);
  r.yf = fx_coarse(y, o.y, A.K.fx_turn);
  r.xf = r.yf == r.yf && zf == zf ? xf : r.yf + zf;
  return zf;
}
// records of pass 1: positions, u, v, w
__device__ __forceinline__ void fx_split_state_body(const StepArgs& A, int s) {
  FxRec* R = reinterpret_cast<FxRec*>(A.XU);
  FxRec r;
  const float zf = fx_position(A, A.x[s], A.y[s], A.z[s], r);
  const double u = A.u[s], v = A.v[s], w = A.w[s];
  fx_field(u, &r.m[0], &r.e[0]);
  fx_field(v, &r.m[1], &r.e[1]);
  fx_field(w, &r.m[2], &r.e[2]);
  r.e[3] = 0;
  R[s] = r;
  A.fs[s] = make_float4(fx_float(u), fx_float(v), fx_float(w), zf);
}
// fields of pass 2: |gdot|^n and the V of its fit
__device__ __forceinline__ void fx_split_p1_body(const StepArgs& A, int s) {
  FxRec* R = reinterpret_cast<FxRec*>(A.XU);
  const double g = A.p1[P1_GN * A.n + s], v = A.K.euler ? A.V[s] : A.p1[P1_VN * A.n + s];
  longlong2 m;
  long long mg, mv;
  short eg, ev;
  fx_field(g, &mg, &eg);
  fx_field(v, &mv, &ev);
  m.x = mg; m.y = mv;
  *reinterpret_cast<longlong2*>(&R[s].m[0]) = m;
  *reinterpret_cast<short2*>(&R[s].e[0]) = make_short2(eg, ev);
  A.fs[s] = make_float4(fx_float(g), fx_float(v), 0.f, 0.f);
}

// A position is rounded to a unit, 2^-58 of the largest radius or less; near the
// origin that loses bits of the coordinate, which a shift brings up: after 6 bits
// to 2^-53 of the stencil's largest offset, as much as FP64 loses. (Up to 12 were
// taken: stencils of a thousandth of the largest radius around the origin erred
// by 1.3e-14 of the largest coefficient, where FP64 rows give 1.5e-15.)
constexpr int kFxMostShift = 6;
// Stencils whose radius is not known (lp_fit_derivatives): the shift that
// brings a particle's largest offset into (fx_lim / 2, fx_lim], from a walk over
// the positions; -1 if the offsets are too large, or so small that the shift
// would reach below the positions' resolution.
__device__ __forceinline__ int fx_shift(const StepArgs& A, int s, int m) {
  const int n = A.n;
  const FxRec* R = reinterpret_cast<const FxRec*>(A.XU);
  FxRec me;
  fx_rec_pos(me, R, s);
  unsigned big = 0;
  constexpr int kChunk = 4;
  for (int k0 = 0; k0 < m; k0 += kChunk) {
    uint32_t cd[kChunk];
    FxPosLoad p[kChunk];
#pragma unroll
    for (int t = 0; t < kChunk; ++t)
      cd[t] = k0 + t < m ? (uint32_t)A.nbr[(int64_t)(k0 + t) * n + s] : ~kMirrorBit;
#pragma unroll
    for (int t = 0; t < kChunk; ++t) p[t].fetch(R, cd[t] & A.K.fx_mask, n, s);
#pragma unroll
    for (int t = 0; t < kChunk; ++t) {
      if ((cd[t] & A.K.fx_mask) >= (uint32_t)n) continue;
      unsigned long long D[3];
      fx_offsets<false, false>(A.K, 0, me, p[t].xy.x, p[t].xy.y, p[t].zf.x, 0.f, 0.f,
                               cd[t] >> 31, D);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int h = (int)(D[a] >> 32);
        big = max(big, (unsigned)(h ^ (h >> 31)));
      }
    }
  }
  // (+ 1: the integer parts are rounded)
  const unsigned lim = (unsigned)A.K.fx_lim;
  if (big + 1u > lim) return -1;
  int sh = max(__clz((int)(big + 1u)) - __clz((int)lim), 0);
  if (((big + 1u) << sh) > lim) --sh;
  return sh <= kFxMostShift ? sh : -1;
}

// The 31 moments of a stencil (order of ff_moments_add) in units of the
// lattice spacing. GH: flagged entries (kGhostBit) also stand for their point
// reflection, so they add their even moments twice and no odd ones. False: the
// row does not fit the fixed-point range.
// rows: the entries with an index in range. SH: offsets are shifted up by sh,
// which fx_shift chose for the particle's largest one.
// P lanes of a particle take every P-th entry each (sub: the lane's first
// one); the sums are whole numbers, so that adding the lanes' sums gives the
// bits of one lane taking all (P = 1).
template <bool PER, bool GH, bool SH, int P>
__device__ __forceinline__ bool fx_moment_rows(const StepArgs& A, int s, int m, int sub,
                                               long long* H, int* rows, int sh) {
  const int n = A.n;
  const FxRec* R = reinterpret_cast<const FxRec*>(A.XU);
  const StepConsts& K = A.K;
  const uint32_t mask = K.fx_mask;
  FxRec me;
  fx_rec_pos(me, R, s);
#pragma unroll
  for (int q = 0; q < 31; ++q) H[q] = 0;
  unsigned big = 0;  // the largest magnitude of an offset
  int in_range = m;
  bool bad = !(me.xf == me.xf);
  uint32_t code = sub < m ? (uint32_t)A.nbr[(int64_t)sub * n + s] : 0u;
  uint32_t nxt = sub + P < m ? (uint32_t)A.nbr[(int64_t)(sub + P) * n + s] : 0u;
  FxPosLoad X;
  X.fetch(R, code & mask, n, s);
  for (int k = sub; k < m; k += P) {
    const uint32_t c0 = code;
    const bool live = (c0 & mask) < (uint32_t)n;  // (else: stale or corrupt stencil entry)
    unsigned long long D[3];
    const bool near =
        fx_offsets<PER, SH>(K, sh, me, X.xy.x, X.xy.y, X.zf.x, X.xf(), X.yf(), c0 >> 31, D);
    bad = bad || (live && !near);
    if (k + P < m) {  // (the position is taken: its registers hold the next one)
      code = nxt;
      X.fetch(R, code & mask, n, s);
      if (k + 2 * P < m) nxt = (uint32_t)A.nbr[(int64_t)(k + 2 * P) * n + s];
    }
    if (!live) {
      --in_range;
      continue;
    }
    FxV d[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      d[a] = fx_split(D[a]);
      big = max(big, (unsigned)(d[a].h ^ (d[a].h >> 31)));
    }
    long long Q[6] = {fx_mul(d[0], d[0]), fx_mul(d[1], d[1]), fx_mul(d[2], d[2]),
                      fx_mul(d[0], d[1]), fx_mul(d[0], d[2]), fx_mul(d[1], d[2])};
    FxV q[6];
#pragma unroll
    for (int t = 0; t < 6; ++t) q[t] = fx_quad(Q[t], K.fx_sq, K.fx_qs);
    FxV w[6];  // the first factor of the even moments (twice for a flagged entry)
    const bool twin = GH && (c0 & kGhostBit);
#pragma unroll
    for (int t = 0; t < 6; ++t) {
      w[t] = q[t];
      if (twin) {
        w[t].h <<= 1; w[t].hf *= 2.f; w[t].l *= 2.f;
        Q[t] <<= 1;
      }
      H[t] += Q[t];
    }
    if (twin) {
#pragma unroll
      for (int a = 0; a < 3; ++a) d[a] = FxV{0, 0.f, 0.f};
    }
    // q: 0 xx, 1 yy, 2 zz, 3 xy, 4 xz, 5 yz
    fx_acc(H[6], d[0], q[0]);   fx_acc(H[7], d[1], q[1]);
    fx_acc(H[8], d[2], q[2]);   fx_acc(H[9], d[1], q[0]);
    fx_acc(H[10], d[2], q[0]); fx_acc(H[11], d[0], q[1]);
    fx_acc(H[12], d[2], q[1]); fx_acc(H[13], d[0], q[2]);
    fx_acc(H[14], d[1], q[2]); fx_acc(H[15], d[2], q[3]);
    fx_acc(H[16], w[0], q[0]); fx_acc(H[17], w[1], q[1]);
    fx_acc(H[18], w[2], q[2]); fx_acc(H[19], w[0], q[3]);
    fx_acc(H[20], w[0], q[4]); fx_acc(H[21], w[1], q[3]);
    fx_acc(H[22], w[1], q[5]); fx_acc(H[23], w[2], q[4]);
    fx_acc(H[24], w[2], q[5]); fx_acc(H[25], w[0], q[1]);
    fx_acc(H[26], w[0], q[2]); fx_acc(H[27], w[1], q[2]);
    fx_acc(H[28], w[0], q[5]); fx_acc(H[29], w[1], q[4]);
    fx_acc(H[30], w[2], q[3]);
  }
  *rows = in_range;
  return !(bad || big > (unsigned)K.fx_lim);
}
// The error of a sum is a few units per row whatever its value (a term errs by
// up to 2^5 units, 2^2 typically), so a stencil thin along an axis, or small
// against the radius, has sums with few good bits: with one axis compressed to
// 0.1 the derivatives err by 5e-12 of the largest instead of 3e-15, at 0.01 by
// 5e-8, and no relative pivot shows it, as those do not depend on the columns'
// scale. False if the squared length of a quadratic column is below 2^50 units;
// the particle then takes the plain rows. At the line errors are two to three
// times those of FP64 rows (1.2e-15 and 4e-16 rms of the largest derivative on
// a lattice compressed to 0.35; 2e-14 and 9e-15 in a corner of one). The least
// such length of a jittered lattice at the usual radius of 2.2 spacings: 2^53
// in the bulk, 2^50.4 in corners, where the radius is least favourable to its
// power of two. (The linear columns are at least as well resolved.)
constexpr int kFxLeastBits = 50;
__device__ __forceinline__ bool fx_resolved(const long long* H) {
  long long least = min(min(H[16], H[17]), H[18]);
  least = min(least, min(min(H[25], H[26]), H[27]));
  return least >= 1ll << kFxLeastBits;
}
template <bool SH>
__device__ __forceinline__ void fx_moment_values(const StepConsts& K, const long long* H, int sh,
                                                 double* mo) {
  double g2 = K.fx_g2, g3 = K.fx_g3, g4 = K.fx_g4;
  if (SH) {
    g2 *= pow2_of(-2 * sh);
    g3 *= pow2_of(-3 * sh);
    g4 *= pow2_of(-4 * sh);
  }
#pragma unroll
  for (int t = 0; t < 31; ++t) {
    const double g = t < 6 ? g2 : (t < 16 ? g3 : g4);
    mo[t] = (double)H[t] * g;
  }
}
template <bool PER, bool GH, bool SH = false>
__device__ __forceinline__ bool fx_moments(const StepArgs& A, int s, int m, double* mo,
                                           int* rows, int sh = 0) {
  long long H[31];
  if (!fx_moment_rows<PER, GH, SH, 1>(A, s, m, 0, H, rows, sh) || !fx_resolved(H)) return false;
  fx_moment_values<SH>(A.K, H, sh, mo);
  return true;
}

__device__ __forceinline__ void gram_of_moments(const double* mo, double* L) {
  Moments<double> M;
  M.xx = mo[0]; M.yy = mo[1]; M.zz = mo[2]; M.xy = mo[3]; M.xz = mo[4]; M.yz = mo[5];
  M.xxx = mo[6]; M.yyy = mo[7]; M.zzz = mo[8]; M.xxy = mo[9]; M.xxz = mo[10]; M.xyy = mo[11];
  M.yyz = mo[12]; M.xzz = mo[13]; M.yzz = mo[14]; M.xyz = mo[15];
  M.xxxx = mo[16]; M.yyyy = mo[17]; M.zzzz = mo[18]; M.xxxy = mo[19]; M.xxxz = mo[20];
  M.xyyy = mo[21]; M.yyyz = mo[22]; M.xzzz = mo[23]; M.yzzz = mo[24]; M.xxyy = mo[25];
  M.xxzz = mo[26]; M.yyzz = mo[27]; M.xxyz = mo[28]; M.xyyz = mo[29]; M.xyzz = mo[30];
  M.gram(L);
}

// Right-hand sides A^T b of NF fields in column order, in units of the lattice
// spacing; sgn: the factor (-1, 0, 1) of a field at a floor mirror; GH: bG is
// the right-hand side of a flagged entry's ghost row. False: a field does not
// fit (the caller queues the particle).
// kb: the fields' scales. P, sub: as in fx_moment_rows; with P > 1 every lane
// of the warp must call it. ZC: the copies of the fields hold the coarse z;
// entries that are far along it do not fit either.
template <int NF, bool PER, bool GH, bool SH, bool ZC, int P>
__device__ __forceinline__ bool fx_rhs_rows(const StepArgs& A, int s, int m, int sub,
                                            const int* sgn, const double* bG, long long (*H)[kNB],
                                            int* kb, int sh) {
  const int n = A.n;
  const FxRec* R = reinterpret_cast<const FxRec*>(A.XU);
  const StepConsts& K = A.K;
  const uint32_t mask = K.fx_mask;
  // the scale of each field: its largest difference in this stencil, in FP32
  unsigned mx[NF];
  float mf[NF], zi = 0.f, f2 = 0.f;
  bool near = true;
  {
    const float4 v = A.fs[s];
    if (ZC) {  // (f2: the mirror of z is f2 - z)
      zi = v.w;
      f2 = fx_coarse(2.0 * K.floor_z, 2.0 * fx_ref(A).z, K.fx_turn);
    }
    const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      mf[f] = vv[f];
      mx[f] = 0u;
      if (GH) mx[f] = __float_as_uint(fx_float(bG[f])) & 0x7fffffffu;
    }
  }
  constexpr int kChunk = 4;
  for (int k0 = sub; k0 < m; k0 += kChunk * P) {
    uint32_t cd[kChunk];
    float4 v[kChunk];
#pragma unroll
    for (int t = 0; t < kChunk; ++t)
      cd[t] = k0 + t * P < m ? (uint32_t)A.nbr[(int64_t)(k0 + t * P) * n + s] : ~kMirrorBit;
#pragma unroll
    for (int t = 0; t < kChunk; ++t) {
      const uint32_t j = cd[t] & mask;
      v[t] = A.fs[j < (uint32_t)n ? j : (uint32_t)s];
    }
#pragma unroll
    for (int t = 0; t < kChunk; ++t) {
      if ((cd[t] & mask) >= (uint32_t)n) continue;
      const float vv[4] = {v[t].x, v[t].y, v[t].z, v[t].w};
      const bool mir = cd[t] >> 31;
      if (ZC) near = near && fabsf((mir ? f2 - v[t].w : v[t].w) - zi) < kFxNear;
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        const float d = (mir ? (float)sgn[f] * vv[f] : vv[f]) - mf[f];
        mx[f] = max(mx[f], __float_as_uint(d) & 0x7fffffffu);
      }
    }
  }
#pragma unroll
  for (int o = 1; o < P; o <<= 1)
#pragma unroll
    for (int f = 0; f < NF; ++f) mx[f] = max(mx[f], __shfl_xor_sync(0xffffffffu, mx[f], o));
  // kb: differences are held as b 2^kb; et: values as v 2^(58 - et), exact for
  // all but values far below the largest; lsh: from the second to the first
  int et[NF], lsh[NF];
  bool fits = true;
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    // a bound on the FP64 differences: the FP32 copies err by 2^-24 each
    const float d = __uint_as_float(mx[f]) * (1.f + 0x1p-20f);
    float B = __fmaf_rn(fabsf(mf[f]), 0x1p-22f, d);
    const float V = __fmaf_rn(fabsf(mf[f]), 1.f + 0x1p-20f, d);  // and on the values
    if (GH && K.free_surface) B *= 2.f;  // b +- bG
    fits = fits && B < 0x1p120f && !(B > 0.f && B < 0x1p-90f);
    const int eb = (int)((__float_as_uint(B) + 0x007fffffu) >> 23) - 127;
    const int ev = (int)((__float_as_uint(V) + 0x007fffffu) >> 23) - 127;
    kb[f] = B > 0.f ? 60 - eb : 0;
    et[f] = B > 0.f ? ev : 0;
    lsh[f] = B > 0.f ? ev - eb + 2 : 0;  // (>= 0: B <= 4 V)
  }
  if (!fits) {
    if (P == 1) return false;
    m = 0;  // (the lanes stay together)
  }
  FxRec me;
  fx_rec_pos(me, R, s);
  unsigned long long U[NF], G[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    U[f] = (unsigned long long)(R[s].m[f] >> min(max(et[f] - R[s].e[f], 0), 63));
    G[f] = GH ? fx_of(bG[f], kb[f]) : 0ull;
  }
#pragma unroll
  for (int f = 0; f < NF; ++f)
#pragma unroll
    for (int q = 0; q < kNB; ++q) H[f][q] = 0;
  uint32_t code = sub < m ? (uint32_t)A.nbr[(int64_t)sub * n + s] : 0u;
  uint32_t nxt = sub + P < m ? (uint32_t)A.nbr[(int64_t)(sub + P) * n + s] : 0u;
  FxPosLoad X;
  longlong2 f01, f23;  // m[0], m[1]; m[2], exponents
  auto fetch = [&](uint32_t c) {
    const uint32_t j = c & mask;
    X.fetch(R, j, n, s);
    const longlong2* r = reinterpret_cast<const longlong2*>(&R[j < (uint32_t)n ? j : (uint32_t)s].m[0]);
    f01 = r[0];
    f23 = r[1];
  };
  fetch(code);
  for (int k = sub; k < m; k += P) {
    const uint32_t c0 = code;
    const bool live = (c0 & mask) < (uint32_t)n;  // (else: stale or corrupt stencil entry)
    const bool mir = c0 >> 31;
    unsigned long long D[3], u[NF];
    fx_offsets<PER, SH>(K, sh, me, X.xy.x, X.xy.y, X.zf.x, X.xf(), X.yf(), mir, D);
    {
      const long long mj[3] = {f01.x, f01.y, f23.x};
      const int ej[3] = {(int)(short)f23.y, (int)f23.y >> 16, (int)(short)(f23.y >> 32)};
#pragma unroll
      for (int f = 0; f < NF; ++f)
        u[f] = (unsigned long long)(mj[f] >> min(max(et[f] - ej[f], 0), 63));
    }
    if (k + P < m) {
      code = nxt;
      fetch(code);
      if (k + 2 * P < m) nxt = (uint32_t)A.nbr[(int64_t)(k + 2 * P) * n + s];
    }
    if (!live) continue;
    if (mir) {
#pragma unroll
      for (int f = 0; f < NF; ++f) u[f] = sgn[f] < 0 ? 0ull - u[f] : (sgn[f] ? u[f] : 0ull);
    }
    FxV a[kNB];
#pragma unroll
    for (int t = 0; t < 3; ++t) a[t] = fx_split(D[t]);
    a[3] = fx_quad(fx_mul(a[0], a[0]), K.fx_sq, K.fx_qs);
    a[4] = fx_quad(fx_mul(a[1], a[1]), K.fx_sq, K.fx_qs);
    a[5] = fx_quad(fx_mul(a[2], a[2]), K.fx_sq, K.fx_qs);
    a[6] = fx_quad(fx_mul(a[0], a[1]), K.fx_sq, K.fx_qs);
    a[7] = fx_quad(fx_mul(a[0], a[2]), K.fx_sq, K.fx_qs);
    a[8] = fx_quad(fx_mul(a[1], a[2]), K.fx_sq, K.fx_qs);
    const bool twin = GH && (c0 & kGhostBit);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const unsigned long long d = (u[f] - U[f]) << lsh[f];
      // a ghost row is T(-offset) with right-hand side bG: with the entry's own
      // row, linear terms take b - bG and quadratic ones b + bG
      const FxV bl = fx_split(twin ? d - G[f] : d);
#pragma unroll
      for (int q = 0; q < 3; ++q) fx_acc(H[f][q], bl, a[q]);
      const FxV bq = GH ? fx_split(twin ? d + G[f] : d) : bl;
#pragma unroll
      for (int q = 3; q < kNB; ++q) fx_acc(H[f][q], bq, a[q]);
    }
  }
  return fits && near;
}
template <int NF, bool SH>
__device__ __forceinline__ void fx_rhs_values(const StepConsts& K, const long long (*H)[kNB],
                                              const int* kb, int sh, double (*R9)[kNB]) {
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    const double ub = pow2_of(32 - kb[f]);
    double ul = ub * K.fx_lin, uq = ub * K.fx_quad;
    if (SH) {
      ul *= pow2_of(-sh);
      uq *= pow2_of(-2 * sh);
    }
#pragma unroll
    for (int q = 0; q < kNB; ++q) {
      R9[f][q] = (double)H[f][q] * (q < 3 ? ul : (q < 6 ? 0.5 * uq : uq));
    }
  }
}
template <int NF, bool PER, bool GH, bool ZC, bool SH = false>
__device__ __forceinline__ bool fx_rhs(const StepArgs& A, int s, int m, const int* sgn,
                                       const double* bG, double (*R9)[kNB], int sh = 0) {
  long long H[NF][kNB];
  int kb[NF];
  if (!fx_rhs_rows<NF, PER, GH, SH, ZC, 1>(A, s, m, 0, sgn, bG, H, kb, sh)) return false;
  fx_rhs_values<NF, SH>(A.K, H, kb, sh, R9);
  return true;
}

// Runs with few particles: P lanes to a particle for the rows; the block's
// first warp then takes a particle a lane for what follows them.
constexpr int kFxSlots = 32;  // particles of a block of P * 32 threads
template <int NV>
struct FxShared {
  long long H[NV][kFxSlots];
  int kb[3][kFxSlots];
  int fits[kFxSlots];
};
// the lanes' sums added (whole numbers), to column slot of the shared ones
template <int P, int NV>
__device__ __forceinline__ void fx_lanes_store(FxShared<NV>& S, int slot, int sub, long long* H,
                                               bool fits) {
  int ok = fits;
#pragma unroll
  for (int o = 1; o < P; o <<= 1) ok &= __shfl_xor_sync(0xffffffffu, ok, o);
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    long long v = H[q];
#pragma unroll
    for (int o = 1; o < P; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (q % P == sub) S.H[q][slot] = v;
  }
  if (sub == 0) S.fits[slot] = ok;
}

// right-hand sides from a column of the shared sums
template <int NV>
__device__ __forceinline__ void fx_shared_values(const StepConsts& K, const FxShared<NV>& S,
                                                 int col, double (*R9)[kNB]) {
  constexpr int NF = NV / kNB;
  long long H[NF][kNB];
  int kb[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    kb[f] = S.kb[f][col];
#pragma unroll
    for (int q = 0; q < kNB; ++q) H[f][q] = S.H[f * kNB + q][col];
  }
  fx_rhs_values<NF, false>(K, H, kb, 0, R9);
}

}  // namespace lp
