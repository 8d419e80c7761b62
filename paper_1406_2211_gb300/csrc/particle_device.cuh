// Device code of the Lagrangian-side kernels (see particle_kernels.cu for
// the description): helpers, the kernel bodies, and the per-box kernels.
// Included by particle_kernels.cu (per-box launches) and particle_batch.cu
// (launches over many boxes); everything here has internal linkage.
#pragma once
#include <cooperative_groups.h>

#include "lb_device.cuh"
#include "philox.cuh"

namespace lbc {
namespace {


// ------------------------------------------------------------ launch caches
// Launch quantities that depend on the device (SM count, occupancy) are
// cached per device ordinal, so one process may drive GPUs of different
// sizes.
constexpr int MAX_DEVICES = 64;

// ------------------------------------------------------------ 1-D stencils
// phi_4 (Peskin): (3 - 2|r| + sqrt(1 + 4|r| - 4r^2))/8 on |r| <= 1,
//                 (5 - 2|r| - sqrt(-7 + 12|r| - 4r^2))/8 on 1 <= |r| <= 2
template <typename C> __device__ inline C phi4_inner(C a) {
  return (C(3) - C(2) * a + sqrt(fmax(C(0), C(1) + C(4) * a - C(4) * a * a))) * C(0.125);
}
template <typename C> __device__ inline C phi4_outer(C a) {
  return (C(5) - C(2) * a - sqrt(fmax(C(0), C(-7) + C(12) * a - C(4) * a * a))) * C(0.125);
}
// phi_3 (App. A): (1 + sqrt(1 - 3r^2))/3 on |r| <= 1/2,
//                 (5 - 3|r| - sqrt(-2 + 6|r| - 3r^2))/6 on 1/2 <= |r| <= 3/2
template <typename C> __device__ inline C phi3_inner(C a) {
  return (C(1) + sqrt(fmax(C(0), C(1) - C(3) * a * a))) / C(3);
}
template <typename C> __device__ inline C phi3_outer(C a) {
  return (C(5) - C(3) * a - sqrt(fmax(C(0), C(-2) + C(6) * a - C(3) * a * a))) / C(6);
}

// base node b and weights of nodes b + k along one axis for position X
template <int ST, typename C>
__device__ inline void stencil_1d(double X, int& b, C (&w)[4]) {
  if (ST == 0) {                       // trilinear: nodes floor(X), +1
    const double fl = floor(X);
    b = (int)fl;
    const C t = (C)(X - fl);
    w[0] = C(1) - t; w[1] = t; w[2] = C(0); w[3] = C(0);
  } else if (ST == 1) {                // four-point: floor(X) - 1 .. + 2
    const double fl = floor(X);
    b = (int)fl - 1;
    const C t = (C)(X - fl);           // r_k = t + 1 - k
    w[0] = phi4_outer<C>(C(1) + t);
    w[1] = phi4_inner<C>(t);
    w[2] = phi4_inner<C>(C(1) - t);
    w[3] = phi4_outer<C>(C(2) - t);
  } else {                             // three-point: round(X) - 1 .. + 1
    const double fl = floor(X + 0.5);
    b = (int)fl - 1;
    const C t = (C)(X - fl);           // in [-1/2, 1/2)
    w[0] = phi3_outer<C>(C(1) + t);
    w[1] = phi3_inner<C>(fabs(t));
    w[2] = phi3_outer<C>(C(1) - t);
    w[3] = C(0);
  }
}

template <int ST> __host__ __device__ constexpr int nodes_1d() { return ST == 0 ? 2 : (ST == 1 ? 4 : 3); }

// FP32 weights of the stencil whose floor node is fl, for the fraction t in
// [0, 1) (three-point stencil: fl = floor(X + 1/2), t = frac(X + 1/2))
template <int ST>
__device__ inline void stencil_weights_f32(int fl, float t, int& b, float (&w)[4]) {
  if (ST == 0) {
    b = fl;
    w[0] = 1.0f - t; w[1] = t; w[2] = 0.0f; w[3] = 0.0f;
  } else if (ST == 1) {
    b = fl - 1;
    w[0] = phi4_outer<float>(1.0f + t);
    w[1] = phi4_inner<float>(t);
    w[2] = phi4_inner<float>(1.0f - t);
    w[3] = phi4_outer<float>(2.0f - t);
  } else {                             // t - 1/2 in [-1/2, 1/2): X - round(X)
    b = fl - 1;
    const float r = t - 0.5f;
    w[0] = phi3_outer<float>(1.0f + r);
    w[1] = phi3_inner<float>(fabsf(r));
    w[2] = phi3_outer<float>(1.0f - r);
    w[3] = 0.0f;
  }
}

// v[q] by selects (the array stays in registers)
template <typename T, int N>
__device__ __forceinline__ T pick(const T (&v)[N], int q) {
  T r = v[0];
#pragma unroll
  for (int e = 1; e < N; ++e) r = q == e ? v[e] : r;
  return r;
}

// ------------------------------------------------------------ FP64 values without FP64 work
// The bit pattern of (double)n for 0 < n < 2^31 (integer operations).
__device__ inline long long dbl_bits_of(int n) {
  const int e = 31 - __clz(n);                             // n = 1.f 2^e
  const unsigned long long f = ((unsigned long long)n << (52 - e)) & ((1ull << 52) - 1ull);
  return (long long)(((unsigned long long)(1023 + e) << 52) | f);
}

// x as the unevaluated sum hi + lo of two floats, read off its bit pattern
// with integer operations: hi is x cut to 24 significant bits, lo the other
// 29 bits, rounded to 24 by the conversion, so |x - hi - lo| <= 2^-48 |x|.
// |x| < 2^-126 (zero included) gives 0 + 0; |x| must be below 2^128.
__device__ inline void split_df(double x, float& hi, float& lo) {
  const unsigned long long u = static_cast<unsigned long long>(__double_as_longlong(x));
  const uint32_t w1 = (uint32_t)(u >> 32), w0 = (uint32_t)u;
  const uint32_t sign = w1 & 0x80000000u;
  const int e = (int)((w1 >> 20) & 0x7FFu);              // biased FP64 exponent
  if (e < 897) {
    hi = 0.0f;
    lo = 0.0f;
    return;
  }
  hi = __uint_as_float(sign | ((uint32_t)(e - 896) << 23) | ((w1 & 0xFFFFFu) << 3) | (w0 >> 29));
  const int le = e - 1075 + 127;                          // biased exponent of 2^(e - 1075)
  const float scale = le >= 1 ? __uint_as_float((uint32_t)le << 23) : 0.0f;
  lo = __uint_as_float(__float_as_uint(__uint2float_rn(w0 & 0x1FFFFFFFu) * scale) | sign);
}

// s = fl(a + b) and the rounding error a + b - s exactly (Knuth's TwoSum)
__device__ inline float two_sum(float a, float b, float& err) {
  const float s = __fadd_rn(a, b);
  const float bv = __fsub_rn(s, a);
  const float av = __fsub_rn(s, bv);
  err = __fadd_rn(__fsub_rn(a, av), __fsub_rn(b, bv));
  return s;
}

// Double-float arithmetic (value h + l, |l| <= ulp(h) / 2) on the FP32 pipe
struct dflt {
  float h, l;
};
__device__ inline dflt df_add(dflt a, dflt b) {
  float e;
  const float s = two_sum(a.h, b.h, e);
  e += a.l + b.l;
  const float h = s + e;
  return dflt{h, e - (h - s)};
}
__device__ inline dflt df_mul(dflt a, dflt b) {
  const float p = a.h * b.h;
  float e = fmaf(a.h, b.h, -p);                 // exact residue of the product
  e = fmaf(a.h, b.l, fmaf(a.l, b.h, e));
  const float h = p + e;
  return dflt{h, e - (h - p)};
}
__device__ inline dflt df_of(double x) {
  dflt r;
  split_df(x, r.h, r.l);
  return r;
}

// A stencil base (x, y, z), each in -2^20 .. 2^20 - 1, as three signed
// 21-bit fields of one 64-bit word (bits 0-20, 22-42, 43-63)
__device__ inline unsigned long long pack_base(int x, int y, int z) {
  return ((unsigned long long)(x & 0x1FFFFF)) | ((unsigned long long)(y & 0x1FFFFF) << 22) |
         ((unsigned long long)(z & 0x1FFFFF) << 43);
}
__device__ inline int base_x(unsigned long long u) { return (int)((long long)(u << 43) >> 43); }
__device__ inline int base_y(unsigned long long u) { return (int)((long long)(u << 21) >> 43); }
__device__ inline int base_z(unsigned long long u) { return (int)((long long)u >> 43); }

// The stencil of X given as hi + lo (split_df) in FP32 alone: floor of hi,
// and the fraction (hi - floor(hi)) + lo brought into [0, 1).
template <int ST>
__device__ inline void stencil_1d_df(float xh, float xl, int& b, float (&w)[4]) {
  float fl = floorf(xh);
  float t = (xh - fl) + xl;
  if (ST == 2) t += 0.5f;
  if (t < 0.0f) { fl -= 1.0f; t += 1.0f; }
  if (t >= 1.0f) { fl += 1.0f; t -= 1.0f; }
  stencil_weights_f32<ST>((int)fl, t, b, w);
}

// ------------------------------------------------------------ periodic helpers
// X into [0, n) for X in (-n, 2n): the same result as r = fmod(X, n), + n if
// negative, - n if that rounded up to n, without the FP64 fmod.  The tests
// are taken on the bit pattern (non-negative doubles order as their
// patterns; -0 counts as 0), so only a coordinate that crosses the boundary
// spends FP64 work.
__device__ inline double wrap_axis(double X, int n, bool periodic) {
  if (!periodic) return X;
  const long long un = dbl_bits_of(n);
  constexpr long long NEG_ZERO = (long long)0x8000000000000000ull;
  long long u = __double_as_longlong(X);
  if (u < 0 && u != NEG_ZERO) {                // X < 0
    X += (double)n;
    u = __double_as_longlong(X);
  } else if (u >= un) {                        // X >= n
    X -= (double)n;
    u = __double_as_longlong(X);
  }
  if (u >= un) X -= (double)n;
  return X;
}

// minimum image of a separation d (|d| < 1.5 n); ties at |d| = n/2 are kept,
// as rint(d/n) = 0 there
__device__ inline double min_image(double d, int n, bool periodic) {
  if (!periodic) return d;
  const double h = 0.5 * n;
  if (d > h) d -= n;
  else if (d < -h) d += n;
  return d;
}

__device__ inline uint32_t key_of(const Geom& g, double x, double y, double z) {
  int ix = wrap_int((int)floor(x), g.nx), iy = wrap_int((int)floor(y), g.ny);
  int iz = (int)floor(z);
  if (g.walls) iz = iz < 0 ? 0 : (iz >= g.nz ? g.nz - 1 : iz);
  else iz = wrap_int(iz, g.nz);
  return (uint32_t)tile_of(g, ix, iy, iz);
}

// Markers keep their bins while they are within half a cell of their home
// tile: over a step they then stay within the one cell the spreading's
// neighbour search allows (they move far less than half a cell per step);
// otherwise the next step re-sorts.
__device__ inline bool near_home(const Geom& g, uint32_t home, const double (&r)[3]) {
  const int n3[3] = {g.nx, g.ny, g.nz};
  const bool per[3] = {true, true, !g.walls};
  const int t = (int)home;
  const int tt[3] = {t % g.ntx, (t / g.ntx) % g.nty, t / (g.ntx * g.nty)};
  bool inside = true;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int lo = tt[c] * TILE, w = min(lo + TILE, n3[c]) - lo;
    if (per[c] && n3[c] <= 3 * TILE) continue;      // the search covers the axis
    double dd = r[c] - (double)lo;
    if (per[c]) {
      const double h = 0.5 * n3[c];
      if (dd < -h) dd += n3[c];
      else if (dd >= h) dd -= n3[c];
    }
    inside = inside && dd >= -0.5 && dd < (double)w + 0.5;
  }
  return inside;
}

// The same two decisions from the float splits of the coordinates (FP32
// compute: no FP64 work).  floor(x) is exact for |x| < 2^24; the home test
// may differ from the FP64 one within float rounding of the half-cell
// margins, which only moves a re-binning by a step.
__device__ inline int floor_df(double x) {
  float h, l;
  split_df(x, h, l);
  float fl = floorf(h);
  if (fl == h && l < 0.0f) fl -= 1.0f;
  return (int)fl;
}
__device__ inline uint32_t key_of_f(const Geom& g, double x, double y, double z) {
  int ix = wrap_int(floor_df(x), g.nx), iy = wrap_int(floor_df(y), g.ny);
  int iz = floor_df(z);
  if (g.walls) iz = iz < 0 ? 0 : (iz >= g.nz ? g.nz - 1 : iz);
  else iz = wrap_int(iz, g.nz);
  return (uint32_t)tile_of(g, ix, iy, iz);
}
__device__ inline bool near_home_f(const Geom& g, uint32_t home, const double (&r)[3]) {
  const int n3[3] = {g.nx, g.ny, g.nz};
  const bool per[3] = {true, true, !g.walls};
  const int t = (int)home;
  const int tt[3] = {t % g.ntx, (t / g.ntx) % g.nty, t / (g.ntx * g.nty)};
  bool inside = true;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int lo = tt[c] * TILE, w = min(lo + TILE, n3[c]) - lo;
    if (per[c] && n3[c] <= 3 * TILE) continue;      // the search covers the axis
    float h, l;
    split_df(r[c], h, l);
    float dd = (h - (float)lo) + l;
    if (per[c]) {
      const float hn = 0.5f * n3[c];
      if (dd < -hn) dd += n3[c];
      else if (dd >= hn) dd -= n3[c];
    }
    inside = inside && dd >= -0.5f && dd < (float)w + 0.5f;
  }
  return inside;
}

// ------------------------------------------------------------ drift / forces
constexpr int BONDS_AT_ONCE = 2;

// One marker's sub-step (see DriftArgs): writes its new position, velocity,
// intrinsic force and key, and returns the position, velocity and force.
template <typename C>
__device__ __forceinline__ void drift_one(const PartArgs& __restrict__ p,
                                          const DriftArgs& __restrict__ d, long long i,
                                          double (&r2)[3], double (&v)[3], C (&F)[3]) {
  const long long M = p.M;
  const Geom& g = p.g;
  const int n3[3] = {g.nx, g.ny, g.nz};
  const bool per[3] = {true, true, !g.walls};
  // intermediate positions are left unwrapped (they stay within a cell of
  // the box); only the final position is wrapped, and bond vectors use the
  // minimum image, so no FP64 work is spent on wrapping in between
  // with FP32 compute the two pre-drifts are taken as one (dt_pre0 + dt_pre)
  // v: one FP64 rounding instead of two
  constexpr bool F32 = sizeof(C) == 4;
  const double dt_pre01 = F32 ? d.dt_pre0 + d.dt_pre : 0.0;
  double r1[3];
  if (d.at_force_point) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      v[c] = d.vel_in[c * M + i];
      r1[c] = d.pos_in[c * M + i];
    }
  } else {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      v[c] = d.vel_in[c * M + i];
      r1[c] = F32 ? d.pos_in[c * M + i] + dt_pre01 * v[c]
                  : (d.pos_in[c * M + i] + d.dt_pre0 * v[c]) + d.dt_pre * v[c];
    }
  }
  F[0] = F[1] = F[2] = C(0);
  if (d.compute_force) {
    const C* ext = static_cast<const C*>(d.ext);
    const C* kr = static_cast<const C*>(d.nbr_kr);
    for (int c = 0; c < 3; ++c) F[c] = ext[c * M + i];
    const int bbeg = d.nbr_start[i], bend = d.nbr_start[i + 1];
    // FP32 compute: the marker's position as hi + lo floats (split_df)
    float r1h[3] = {0.0f, 0.0f, 0.0f}, r1l[3] = {0.0f, 0.0f, 0.0f};
    if (F32 && bend > bbeg)
#pragma unroll
      for (int c = 0; c < 3; ++c) split_df(r1[c], r1h[c], r1l[c]);
    // two bonds at a time: their indices, constants and partner positions
    // are loaded together (a marker's bonds are one dependent chain
    // otherwise), the forces are added in bond order
    for (int b0 = bbeg; b0 < bend; b0 += BONDS_AT_ONCE) {
      long long jn[BONDS_AT_ONCE];
      C kn[BONDS_AT_ONCE], r0n[BONDS_AT_ONCE];
      double r0sq[BONDS_AT_ONCE], rjn[BONDS_AT_ONCE][3];
#pragma unroll
      for (int q = 0; q < BONDS_AT_ONCE; ++q) {
        const int b = b0 + q < bend ? b0 + q : b0;       // past the end: the first one again
        jn[q] = d.nbr_j[b];
        kn[q] = kr[2 * b];
        r0n[q] = kr[2 * b + 1];
        r0sq[q] = d.nbr_r0sq[b];
      }
#pragma unroll
      for (int q = 0; q < BONDS_AT_ONCE; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c) rjn[q][c] = d.pos_in[c * M + jn[q]];
      if (!d.at_force_point) {
#pragma unroll
        for (int q = 0; q < BONDS_AT_ONCE; ++q)
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const double vj = d.vel_in[c * M + jn[q]];
            rjn[q][c] = F32 ? rjn[q][c] + dt_pre01 * vj : (rjn[q][c] + d.dt_pre0 * vj) + d.dt_pre * vj;
          }
      }
#pragma unroll
      for (int q = 0; q < BONDS_AT_ONCE; ++q) {
        if (b0 + q >= bend) break;
        const C k = kn[q], r0 = r0n[q];
        C ec[3];
        C dist, D;
        if constexpr (F32) {
          // The bond vector e = r_j - r_i and |e|^2 - r0^2 in double-float
          // arithmetic on the FP32 pipe: e as eh + el (TwoSum of the highs
          // plus the difference of the lows; the minimum image subtracts n
          // from eh exactly), |e|^2 as the exact products eh^2 (FMA residue)
          // plus 2 eh el, summed with TwoSum against r0^2 = hi + lo.  The
          // result matches the FP64 difference of squares to about 2^-46 |e|^2.
          float eh[3], el[3], P[3], PE[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const double rj = rjn[q][c];
            float jh, jl, err;
            split_df(rj, jh, jl);
            float sh = two_sum(jh, -r1h[c], err);
            float t = err + (jl - r1l[c]);
            float h = sh + t;                      // renormalised pair h + l
            float l = t - (h - sh);
            if (per[c]) {
              const float half = 0.5f * (float)n3[c];
              int shift = 0;
              if (h > half || (h == half && l > 0.0f)) shift = -1;
              else if (h < -half || (h == -half && l < 0.0f)) shift = 1;
              if (shift != 0) {
                const float hs = h + (float)(shift * n3[c]);   // exact (Sterbenz)
                h = hs + l;
                l = l - (h - hs);
              }
            }
            eh[c] = h;
            el[c] = l;
            ec[c] = h;
            P[c] = h * h;
            PE[c] = fmaf(h, h, -P[c]) + 2.0f * h * l;
          }
          float e1, e2, e3, r0h, r0l;
          const float S1 = two_sum(P[0], P[1], e1);
          const float S2 = two_sum(S1, P[2], e2);
          split_df(r0sq[q], r0h, r0l);
          const float S3 = two_sum(S2, -r0h, e3);
          D = S3 + (((e1 + e2) + e3) + ((PE[0] + PE[1]) + PE[2]) - r0l);
          dist = sqrtf(S2);
        } else {
          double dist2 = 0.0;
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const double e = min_image(rjn[q][c] - r1[c], n3[c], per[c]);
            ec[c] = (C)e;
            dist2 += e * e;
          }
          // the difference of squares in FP64: bonds sit near their rest
          // length, where |d| - r0 formed directly would lose most digits
          dist = sqrt((C)dist2);
          D = (C)(dist2 - r0sq[q]);
        }
        // stretch |d| - r0 = (|d|^2 - r0^2) / (|d| + r0)
        const C stretch = D / (dist + r0);
        const C mag = k * stretch / dist;
        for (int c = 0; c < 3; ++c) F[c] += ec[c] * mag;
      }
    }
    const int body = d.rigid.nbodies > 0 ? d.rigid.body_of[i] : -1;
    if (body >= 0) {
      // tether to the body's best-fit frame: F = -k (y - X - R q), the
      // difference taken at its minimum image; plus the body's share of
      // the repulsion
      const double* fr = d.rigid.frames + 12 * body;
      const double q[3] = {d.rigid.ref[i], d.rigid.ref[M + i], d.rigid.ref[2 * M + i]};
      // the marker's share of the repulsion: with FP32 compute a float
      // division (an FP64 one is a long sequence on the FP64 pipe)
      const int cnt = d.rigid.count[body];
      const float inv_nf = F32 ? 1.0f / (float)cnt : 0.0f;
      const double inv_n = F32 ? 0.0 : 1.0 / (double)cnt;
#pragma unroll
      if constexpr (F32) {
        // dev = (r1 - X_b) - R q in double-float arithmetic (FP32 pipe)
        const dflt qd[3] = {df_of(q[0]), df_of(q[1]), df_of(q[2])};
        const float kf = (float)d.rigid.k;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          dflt e = df_add(df_of(r1[c]), dflt{0.0f, 0.0f});
          const dflt xb = df_of(fr[c]);
          e = df_add(e, dflt{-xb.h, -xb.l});
          dflt rq = df_mul(df_of(fr[3 + 3 * c]), qd[0]);
          rq = df_add(rq, df_mul(df_of(fr[4 + 3 * c]), qd[1]));
          rq = df_add(rq, df_mul(df_of(fr[5 + 3 * c]), qd[2]));
          e = df_add(e, dflt{-rq.h, -rq.l});
          if (per[c]) {
            const float half = 0.5f * (float)n3[c];
            if (e.h > half || (e.h == half && e.l > 0.0f)) e = df_add(dflt{e.h - (float)n3[c], 0.0f}, dflt{e.l, 0.0f});
            else if (e.h < -half || (e.h == -half && e.l < 0.0f)) e = df_add(dflt{e.h + (float)n3[c], 0.0f}, dflt{e.l, 0.0f});
          }
          F[c] += (C)(-kf * (e.h + e.l)) + (C)d.rigid.frep[3 * body + c] * (C)inv_nf;
        }
      } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const double site = fr[c] + fr[3 + 3 * c] * q[0] + fr[4 + 3 * c] * q[1] + fr[5 + 3 * c] * q[2];
          const double dev = min_image(r1[c] - site, n3[c], per[c]);
          F[c] += (C)(-d.rigid.k * dev + d.rigid.frep[3 * body + c] * inv_n);
        }
      }
    }
    if (d.fint_out) {
      C* fo = static_cast<C*>(d.fint_out);
      for (int c = 0; c < 3; ++c) fo[c * M + i] = F[c];
    }
  }
  // (a zero kick or post-drift leaves v and r unchanged: skipped, FP64 work
  // being scarce)
  if (d.dt_kick != 0.0) {
    const double kick = d.dt_kick * d.inv_mass[i];
#pragma unroll
    for (int c = 0; c < 3; ++c) v[c] += kick * (double)F[c];
  }
  if (d.at_force_point && d.dt_post == 0.0) {
#pragma unroll
    for (int c = 0; c < 3; ++c) r2[c] = r1[c];          // stored wrapped
  } else {
#pragma unroll
    for (int c = 0; c < 3; ++c)
      r2[c] = wrap_axis(d.dt_post != 0.0 ? r1[c] + d.dt_post * v[c] : r1[c], n3[c], per[c]);
  }
  if (d.pos_out)
    for (int c = 0; c < 3; ++c) d.pos_out[c * M + i] = r2[c];
  if (d.vel_out)
    for (int c = 0; c < 3; ++c) d.vel_out[c * M + i] = v[c];
  if (d.write_key) {
    d.key_out[i] = F32 ? key_of_f(g, r2[0], r2[1], r2[2]) : key_of(g, r2[0], r2[1], r2[2]);
    d.idx_out[i] = (uint32_t)i;
    if (i == 0 && d.clear_flags) {       // the flags of the previous step
      d.clear_flags[0] = 0;
      d.clear_flags[1] = 0;
    }
    if (d.home && !(F32 ? near_home_f(g, d.home[i], r2) : near_home(g, d.home[i], r2))) *d.need = 1;
  }
}

template <typename C>
__global__ void __launch_bounds__(128) drift_kernel(const PartArgs p, const DriftArgs d) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= p.M) return;
  double r2[3], v[3];
  C F[3];
  drift_one<C>(p, d, i, r2, v, F);
}

// ------------------------------------------------------------ rigid bodies
constexpr int FRAME_THREADS = 256;

// block-wide sum of n values per thread (shared scratch sh[n][ROW])
template <int NV, int ROW>
__device__ inline void block_sum(double (&v)[NV], double (*sh)[ROW]) {
  for (int k = 0; k < NV; ++k) sh[k][threadIdx.x] = v[k];
  __syncthreads();
  for (int w = FRAME_THREADS / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
      for (int k = 0; k < NV; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
    __syncthreads();
  }
  for (int k = 0; k < NV; ++k) v[k] = sh[k][0];
  __syncthreads();
}

// One block per body: the markers at their pre-drifted positions r1 (the
// drift's own formula), unwrapped around the first marker r0 as
// y = r0 + d, d = min_image(r1 - r0); X = their mean, R = polar factor of
// A = sum (y - X) q^T by the scaled Newton iteration
// R <- (g R + (g R)^-T) / 2, g = |det R|^(-1/3) (converges to the
// orthogonal factor, a proper rotation while det A > 0).  One pass over the
// markers: with m = mean(d), X = r0 + m and A = sum d q^T - m (sum q)^T
// (the offsets d are below two radii, so no large coordinate enters the
// sums).  The iteration is a chain of FP64 operations, so nine lanes hold one
// matrix element each and exchange them by shuffles (one thread doing all of
// it, with a cube root per iteration, took most of the kernel); the scale is
// applied in the first iteration and while det R is above SCALE_DET.  After an
// iteration det R >= 1, and for a compact body it is 1 to second order in the
// deviation from a rotation, where the plain iteration R <- (R + R^-T) / 2
// converges as fast.  The A of a rod or a disc has singular values of the
// square of its aspect ratio: unscaled, the largest would only be halved per
// iteration, and a plate of 2^-30 of its width would not converge in 40.  The
// sums of the block are taken by sixteen threads per value.  500 bodies of 400
// markers: 45 -> 17 us.
constexpr double SCALE_DET = 2.0;
template <bool DF>
__global__ void __launch_bounds__(FRAME_THREADS)
rigid_frames_kernel(const PartArgs p, const DriftArgs d) {
  constexpr int ROW = FRAME_THREADS + 8;       // (padded: the rows of a warp fall on other banks)
  __shared__ double sh[15][ROW];
  __shared__ double accs[15];
  const RigidArgs& rg = d.rigid;
  const int b = blockIdx.x;
  const long long M = p.M;
  const Geom& g = p.g;
  const int n3[3] = {g.nx, g.ny, g.nz};
  const bool per[3] = {true, true, !g.walls};
  const int f = rg.first[b], cnt = rg.count[b];
  double r0[3];
  for (int c = 0; c < 3; ++c) {
    const double v = d.vel_in[c * M + f];
    r0[c] = DF ? d.pos_in[c * M + f] + (d.dt_pre0 + d.dt_pre) * v
               : (d.pos_in[c * M + f] + d.dt_pre0 * v) + d.dt_pre * v;
  }
  // sums: d (3), q (3), d q^T (9)
  if constexpr (DF) {
    // FP32 compute: the same sums in double-float arithmetic on the FP32
    // pipe.  d = (x_i - x_0) + dt (v_i - v_0): the position difference from
    // the float splits of the FP64 positions (TwoSum of the highs), the
    // velocity term in float (|dt (v_i - v_0)| << 1, float rounding of v
    // adds below 2^-24 |v| dt to it); the minimum image subtracts n exactly.
    const float dtf = (float)(d.dt_pre0 + d.dt_pre);
    dflt x0[3];
    float v0[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      x0[c] = df_of(d.pos_in[c * M + f]);
      float vl;
      split_df(d.vel_in[c * M + f], v0[c], vl);
    }
    dflt sd[15];
#pragma unroll
    for (int v = 0; v < 15; ++v) sd[v] = dflt{0.0f, 0.0f};
    for (int k = threadIdx.x; k < cnt; k += FRAME_THREADS) {
      const long long i = f + k;
      dflt dv[3], q[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const dflt xi = df_of(d.pos_in[c * M + i]);
        float vh, vl;
        split_df(d.vel_in[c * M + i], vh, vl);
        dflt e = df_add(xi, dflt{-x0[c].h, -x0[c].l});
        e = df_add(e, dflt{dtf * (vh - v0[c]), 0.0f});
        if (per[c]) {
          const float half = 0.5f * (float)n3[c];
          if (e.h > half || (e.h == half && e.l > 0.0f)) e = df_add(dflt{e.h - (float)n3[c], 0.0f}, dflt{e.l, 0.0f});
          else if (e.h < -half || (e.h == -half && e.l < 0.0f)) e = df_add(dflt{e.h + (float)n3[c], 0.0f}, dflt{e.l, 0.0f});
        }
        dv[c] = e;
        q[c] = df_of(rg.ref[c * M + i]);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        sd[c] = df_add(sd[c], dv[c]);
        sd[3 + c] = df_add(sd[3 + c], q[c]);
      }
#pragma unroll
      for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) sd[6 + 3 * r + c] = df_add(sd[6 + 3 * r + c], df_mul(dv[r], q[c]));
    }
    // block sum in double-float (the scratch as float pairs): sixteen
    // consecutive threads per value, then a butterfly over them
    float2 (*sh2)[ROW] = reinterpret_cast<float2 (*)[ROW]>(sh);
#pragma unroll
    for (int v = 0; v < 15; ++v) sh2[v][threadIdx.x] = make_float2(sd[v].h, sd[v].l);
    __syncthreads();
    const int val = threadIdx.x >> 4, part = threadIdx.x & 15;
    dflt sum{0.0f, 0.0f};
    if (val < 15)
      for (int q = part; q < FRAME_THREADS; q += 16) {
        const float2 e = sh2[val][q];
        sum = df_add(sum, dflt{e.x, e.y});
      }
#pragma unroll
    for (int off = 8; off > 0; off >>= 1)
      sum = df_add(sum, dflt{__shfl_xor_sync(0xffffffffu, sum.h, off), __shfl_xor_sync(0xffffffffu, sum.l, off)});
    if (val < 15 && part == 0) accs[val] = (double)sum.h + (double)sum.l;
  } else {
  double acc[15];
#pragma unroll
  for (int v = 0; v < 15; ++v) acc[v] = 0.0;
  for (int k = threadIdx.x; k < cnt; k += FRAME_THREADS) {
    const long long i = f + k;
    double dv[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double v = d.vel_in[c * M + i];
      const double r1 = (d.pos_in[c * M + i] + d.dt_pre0 * v) + d.dt_pre * v;
      dv[c] = min_image(r1 - r0[c], n3[c], per[c]);
    }
    const double q[3] = {rg.ref[i], rg.ref[M + i], rg.ref[2 * M + i]};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      acc[c] += dv[c];
      acc[3 + c] += q[c];
    }
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c) acc[6 + 3 * r + c] += dv[r] * q[c];
  }
  block_sum<15, ROW>(acc, sh);
  if (threadIdx.x == 0)
    for (int v = 0; v < 15; ++v) accs[v] = acc[v];
  }
  __syncthreads();
  if (threadIdx.x >= 32) return;
  // lane 3 r + c holds element (r, c) (lanes beyond 8 repeat element (2, 2))
  constexpr unsigned full = 0xffffffffu;
  const int lane = threadIdx.x, el = lane < 9 ? lane : 8;
  const int r = el / 3, c = el - 3 * r;
  const int r1 = r == 2 ? 0 : r + 1, r2 = r == 0 ? 2 : r - 1;
  const int c1 = c == 2 ? 0 : c + 1, c2 = c == 0 ? 2 : c - 1;
  const double mr = accs[r] / cnt;
  double R = accs[6 + el] - mr * accs[3 + c];
  // cofactor of the lane's element, and the determinant
  auto cofactor = [&](double v) {
    const double p = __shfl_sync(full, v, 3 * r1 + c1), q = __shfl_sync(full, v, 3 * r2 + c2);
    const double s = __shfl_sync(full, v, 3 * r1 + c2), t = __shfl_sync(full, v, 3 * r2 + c1);
    return p * q - s * t;
  };
  auto det_of = [&](double v, double cof) {
    const double p = v * cof;
    return __shfl_sync(full, p, 0) + __shfl_sync(full, p, 1) + __shfl_sync(full, p, 2);
  };
  double cof = cofactor(R);
  double det = det_of(R, cof);
  const bool ok = det > 0.0;
  for (int it = 0; ok && it < 40; ++it) {
    double from = R, other;
    if (it == 0 || det > SCALE_DET) {
      const double g = 1.0 / cbrt(det);           // the scaled matrix g R has determinant 1
      from = g * R;
      other = g * g * cof;
    } else {
      other = cof / det;
    }
    R = 0.5 * (from + other);
    if (__all_sync(full, fabs(R - from) < 1e-15)) break;
    cof = cofactor(R);
    det = det_of(R, cof);
  }
  if (!ok) {
    if (lane == 0) *rg.status = 2;
    R = r == c ? 1.0 : 0.0;
  }
  double* out = rg.frames + 12 * b;
  if (lane < 9) {
    out[3 + el] = R;
    if (c == 0) out[r] = pick(r0, r) + mr;
  }
}

// one warp per body: the lanes take the other bodies in strides of 32; a
// float screen drops pairs whose centres are farther apart than the reach
// r_b + r_c + 1 by more than the float rounding of the centres can explain,
// and the remaining pairs are evaluated in double.  The lane sums are
// combined by a fixed butterfly, so the result does not depend on
// scheduling.
constexpr int REPULSION_THREADS = 128;

__device__ inline float min_image_f(float d, int n, bool periodic) {
  if (!periodic) return d;
  const float h = 0.5f * n;
  if (d > h) d -= n;
  else if (d < -h) d += n;
  return d;
}

__global__ void __launch_bounds__(REPULSION_THREADS)
rigid_repulsion_kernel(const PartArgs p, const RigidArgs rg) {
  const int b = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (b >= rg.nbodies) return;                   // whole warps leave together
  const Geom& g = p.g;
  const int n3[3] = {g.nx, g.ny, g.nz};
  const bool per[3] = {true, true, !g.walls};
  const double* Xb = rg.frames + 12 * b;
  const float xb[3] = {(float)Xb[0], (float)Xb[1], (float)Xb[2]};
  const double rb = rg.radius[b];
  // centres lie within a few box extents L of the origin, so rounding them
  // and their separation to float moves the distance by a few 1e-7 L; the
  // screen keeps a margin well above that
  const float slack = 1e-3f + 4e-6f * (float)max(g.nx, max(g.ny, g.nz));
  double Fb[3] = {0.0, 0.0, 0.0};
  for (int c2 = lane; c2 < rg.nbodies; c2 += 32) {
    if (c2 == b) continue;
    const double* Xc = rg.frames + 12 * c2;
    const double rc = rg.radius[c2];
    const float reach = (float)(rb + rc) + 1.0f + slack;
    float d2f = 0.0f;
    for (int c = 0; c < 3; ++c) {
      const float e = min_image_f((float)Xc[c] - xb[c], n3[c], per[c]);
      d2f += e * e;
    }
    if (d2f > reach * reach) continue;
    double dv[3], d2 = 0.0;
    for (int c = 0; c < 3; ++c) {
      dv[c] = min_image(Xc[c] - Xb[c], n3[c], per[c]);
      d2 += dv[c] * dv[c];
    }
    const double dist = sqrt(d2);
    const double gap = dist - (rb + rc);
    if (gap < 1.0 && dist > 0.0) {
      const double mag = rg.krep * (1.0 - gap) / dist;      // pushes b away from c2
      for (int c = 0; c < 3; ++c) Fb[c] -= mag * dv[c];
    }
  }
  for (int off = 16; off > 0; off >>= 1)
    for (int c = 0; c < 3; ++c) Fb[c] += __shfl_xor_sync(0xffffffffu, Fb[c], off);
  if (lane == 0)
    for (int c = 0; c < 3; ++c) rg.frep[3 * b + c] = Fb[c];
}



// ------------------------------------------------------------ radix sort
// Stable LSD radix sort with digits of at most 8 bits.  Each block owns
// SORT_BLOCK consecutive elements; per-block digit counts, one exclusive
// scan over (digit, block), and a stable scatter that ranks equal digits in
// element order (warp match within rounds of 256 elements).  The number of
// passes is odd, so the keys written to the b buffers end up sorted in the
// a buffers, which keep the previous result when the sort is skipped.
// Every kernel of the sort returns at once when *need == 0 (the markers are
// still in their bins, see the drift).
constexpr int SORT_THREADS = 256;
constexpr int SORT_ITEMS = 8;
constexpr int SORT_BLOCK = SORT_THREADS * SORT_ITEMS;



__device__ inline bool skip(const int* need) { return need != nullptr && *need == 0; }

__global__ void __launch_bounds__(SORT_THREADS)
sort_hist_kernel(const uint32_t* __restrict__ keys, long long M, int shift, uint32_t mask, int* hist,
                 int nblocks, const int* need) {
  if (skip(need)) return;
  __shared__ int cnt[256];
  cnt[threadIdx.x] = 0;
  __syncthreads();
  const long long base = (long long)blockIdx.x * SORT_BLOCK;
  for (int r = 0; r < SORT_ITEMS; ++r) {
    const long long e = base + r * SORT_THREADS + threadIdx.x;
    if (e < M) atomicAdd(&cnt[(keys[e] >> shift) & mask], 1);   // shared, integer
  }
  __syncthreads();
  hist[threadIdx.x * nblocks + blockIdx.x] = cnt[threadIdx.x];
}

// exclusive scan of n ints in place, one block of 1024 threads: each thread
// sums a contiguous chunk, the chunk sums are scanned with warp shuffles
__global__ void __launch_bounds__(1024) scan_kernel(int* data, int n, const int* need) {
  if (skip(need)) return;
  __shared__ int wsum[32];
  const int per = (n + 1023) / 1024;
  const int lo = threadIdx.x * per;
  int sum = 0;
  for (int k = 0; k < per; ++k) {
    const int e = lo + k;
    if (e < n) sum += data[e];
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int incl = sum;
  for (int off = 1; off < 32; off <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += v;
  }
  if (lane == 31) wsum[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    int w = wsum[lane];
    for (int off = 1; off < 32; off <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, w, off);
      if (lane >= off) w += v;
    }
    wsum[lane] = w;                      // inclusive over warps
  }
  __syncthreads();
  int run = incl - sum + (wid > 0 ? wsum[wid - 1] : 0);
  for (int k = 0; k < per; ++k) {
    const int e = lo + k;
    if (e < n) {
      const int v = data[e];
      data[e] = run;
      run += v;
    }
  }
}

__global__ void __launch_bounds__(SORT_THREADS)
sort_scatter_kernel(const uint32_t* __restrict__ kin, const uint32_t* __restrict__ vin,
                    uint32_t* __restrict__ kout, uint32_t* __restrict__ vout, long long M, int shift,
                    uint32_t mask, const int* __restrict__ hist, int nblocks, const int* need) {
  if (skip(need)) return;
  constexpr int W = SORT_THREADS / 32;
  __shared__ int base_cnt[256];          // elements of each digit already placed
  __shared__ int wcnt[W][256];           // this round: count per warp and digit
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  base_cnt[threadIdx.x] = 0;
  const long long base = (long long)blockIdx.x * SORT_BLOCK;
  for (int r = 0; r < SORT_ITEMS; ++r) {
    for (int k = threadIdx.x; k < W * 256; k += SORT_THREADS) (&wcnt[0][0])[k] = 0;
    __syncthreads();
    const long long e = base + r * SORT_THREADS + threadIdx.x;
    const bool valid = e < M;
    const uint32_t key = valid ? kin[e] : 0u;
    const int dig = valid ? (int)((key >> shift) & mask) : 256;
    const unsigned peers = __match_any_sync(0xffffffffu, dig);
    const int rank = __popc(peers & ((1u << lane) - 1u));
    if (valid && rank == 0) wcnt[warp][dig] = __popc(peers);
    __syncthreads();
    if (valid) {
      int off = base_cnt[dig] + rank;
      for (int w = 0; w < warp; ++w) off += wcnt[w][dig];
      const int pos = hist[dig * nblocks + blockIdx.x] + off;
      kout[pos] = key;
      vout[pos] = vin[e];
    }
    __syncthreads();
    {
      int add = 0;
      for (int w = 0; w < W; ++w) add += wcnt[w][threadIdx.x];
      base_cnt[threadIdx.x] += add;
    }
    __syncthreads();
  }
}



// after a sort: tile ranges [tb, te) of the sorted keys (tiles without
// markers get an empty range), the home tile of every marker, and the
// "bins changed" flag
__global__ void bins_clear_kernel(int ntiles, int* __restrict__ tb, int* __restrict__ te,
                                  const int* need, int* brick_count) {
  if (skip(need)) return;
  if (brick_count && blockIdx.x == 0 && threadIdx.x == 0) *brick_count = 0;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < ntiles; t += gridDim.x * blockDim.x) {
    tb[t] = 0;
    te[t] = 0;
  }
}

__global__ void bins_kernel(long long M, const uint32_t* __restrict__ keys,
                            const uint32_t* __restrict__ idx, int* __restrict__ tb,
                            int* __restrict__ te, uint32_t* __restrict__ home, const int* need,
                            int* changed) {
  if (skip(need)) return;
  const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (k == 0 && changed) *changed = 1;
  if (k >= M) return;
  const uint32_t t = keys[k];
  if (k == 0 || keys[k - 1] != t) tb[t] = (int)k;
  if (k == M - 1 || keys[k + 1] != t) te[t] = (int)(k + 1);
  home[idx[k]] = t;
}


// The whole re-binning of up to SORT_CLUSTER_MAX markers in one launch: one
// thread-block cluster whose blocks exchange their digit counts through
// distributed shared memory and meet at the cluster's hardware barrier, so a
// step carries one gated launch instead of eleven (three radix passes of
// histogram, scan and scatter, and two for the bins).  Each block owns a
// contiguous run of the elements; a pass is the same stable counting sort by
// one digit as above (equal digits in element order), so the order is that of
// any stable sort by key.  Then the tile ranges, home tiles and flags as
// bins_kernel writes them.  Skipped 2 us (the eleven launches 25 us per step);
// with work to do 18 us for 12 500 markers, 54 us for 100 000, 80 us for
// 200 000 (eleven launches: 91, 103, 104 us), growing by 0.3 us per thousand:
// the line at 2^18 markers is where the two meet.
constexpr int SORT_CLUSTER_THREADS = 1024;

__global__ void __launch_bounds__(SORT_CLUSTER_THREADS)
sort_cluster_kernel(long long M, int passes, int width, const uint32_t* kin,
                    const uint32_t* vin, uint32_t* ka, uint32_t* va, uint32_t* kb, uint32_t* vb,
                    int ntiles, int* tb, int* te, uint32_t* home, const int* need, int* changed,
                    int* brick_count) {
  if (skip(need)) return;                  // the same word for every block of the cluster
  namespace cg = cooperative_groups;
  const cg::cluster_group cluster = cg::this_cluster();
  constexpr int W = SORT_CLUSTER_THREADS / 32;
  __shared__ int cnt[256];                 // this block's digit counts (read by the others)
  __shared__ int base[256];                // where the block's next element of a digit goes
  __shared__ int wcnt[W][256];             // a round's counts per warp and digit
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int rank = (int)cluster.block_rank(), nb = (int)cluster.num_blocks();
  const int bins = 1 << width;
  const uint32_t mask = (uint32_t)bins - 1u;
  const long long run = (M + nb - 1) / nb;
  const long long lo = rank * run < M ? rank * run : M, hi = lo + run < M ? lo + run : M;
  for (int p = 0; p < passes; ++p) {
    // pass p reads the given input (p = 0), then a and b in turn
    const uint32_t* k0 = p == 0 ? kin : ((p & 1) ? ka : kb);
    const uint32_t* v0 = p == 0 ? vin : ((p & 1) ? va : vb);
    uint32_t* k1 = (p & 1) ? kb : ka;
    uint32_t* v1 = (p & 1) ? vb : va;
    const int shift = width * p;
    if (t < 256) cnt[t] = 0;
    __syncthreads();
    for (long long e = lo + t; e < hi; e += SORT_CLUSTER_THREADS)
      atomicAdd(&cnt[(__ldcg(k0 + e) >> shift) & mask], 1);          // shared, integer
    cluster.sync();
    // exclusive scan over (digit, block): thread d sums its digit
    int before = 0, total = 0;
    if (t < bins)
      for (int r = 0; r < nb; ++r) {
        const int c = *cluster.map_shared_rank(&cnt[t], r);
        if (r < rank) before += c;
        total += c;
      }
    int incl = total;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += u;
    }
    if (t < 256 && lane == 31) wcnt[0][warp] = incl;
    __syncthreads();
    if (t < 256) {
      int first = incl - total + before;
      for (int w = 0; w < warp; ++w) first += wcnt[0][w];
      base[t] = first;
    }
    cluster.sync();                        // the counts have been read (and base, wcnt written)
    for (long long r0 = lo; r0 < hi; r0 += SORT_CLUSTER_THREADS) {
      for (int k = t; k < W * bins; k += SORT_CLUSTER_THREADS) wcnt[k >> width][k & (bins - 1)] = 0;
      __syncthreads();
      const long long e = r0 + t;
      const bool valid = e < hi;
      const uint32_t key = valid ? __ldcg(k0 + e) : 0u;
      const int dig = valid ? (int)((key >> shift) & mask) : 256;
      const unsigned peers = __match_any_sync(0xffffffffu, dig);
      const int at = __popc(peers & ((1u << lane) - 1u));
      if (valid && at == 0) wcnt[warp][dig] = __popc(peers);
      __syncthreads();
      // a digit's counts over the warps become offsets, and its base moves on
      if (t < bins) {
        int sum = base[t];
        for (int w = 0; w < W; ++w) {
          const int c = wcnt[w][t];
          wcnt[w][t] = sum;
          sum += c;
        }
        base[t] = sum;
      }
      __syncthreads();
      if (valid) {
        const int pos = wcnt[warp][dig] + at;
        k1[pos] = key;
        v1[pos] = __ldcg(v0 + e);
      }
      __syncthreads();
    }
    cluster.sync();                        // the pass is written
  }
  for (long long q = (long long)rank * SORT_CLUSTER_THREADS + t; q < ntiles;
       q += (long long)nb * SORT_CLUSTER_THREADS) {
    tb[q] = 0;
    te[q] = 0;
  }
  cluster.sync();
  for (long long k = lo + t; k < hi; k += SORT_CLUSTER_THREADS) {
    const uint32_t key = __ldcg(ka + k);
    if (k == 0 || __ldcg(ka + k - 1) != key) tb[key] = (int)k;
    if (k == M - 1 || __ldcg(ka + k + 1) != key) te[key] = (int)(k + 1);
    home[__ldcg(va + k)] = key;
  }
  if (rank == 0 && t == 0) {
    if (changed) *changed = 1;
    if (brick_count) *brick_count = 0;
  }
}

// Few markers: the whole re-binning in one block and one launch (a no-op
// while no marker left its bin), so a small box's step carries one gated
// launch instead of the radix passes and the bins.  A stable LSD sort of the
// (key, index) pairs by one key bit per pass in shared memory (each thread
// owns a contiguous run of elements; a block-wide prefix sum of its zero
// bits places them), which gives the same order as any stable sort by key,
// then the tile ranges, home tiles and flags as bins_kernel writes them.
constexpr int SMALL_SORT_THREADS = 1024;

__device__ __forceinline__ void small_sort_body(int n, int key_bits, const uint32_t* __restrict__ kin,
                                                const uint32_t* __restrict__ vin, uint32_t* __restrict__ ka,
                                                uint32_t* __restrict__ va, int ntiles,
                                                int* __restrict__ tb, int* __restrict__ te,
                                                uint32_t* __restrict__ home, const int* need,
                                                int* changed, int* brick_count, uint32_t* ssort) {
  if (skip(need)) return;
  __shared__ int wsum[SMALL_SORT_THREADS / 32];
  const unsigned full = 0xffffffffu;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  constexpr int NW = SMALL_SORT_THREADS / 32;
  uint32_t* k0 = ssort;
  uint32_t* v0 = ssort + n;
  uint32_t* k1 = ssort + 2 * n;
  uint32_t* v1 = ssort + 3 * n;
  for (int i = t; i < n; i += SMALL_SORT_THREADS) {
    k0[i] = kin[i];
    v0[i] = vin[i];
  }
  for (int q = t; q < ntiles; q += SMALL_SORT_THREADS) {
    tb[q] = 0;
    te[q] = 0;
  }
  __syncthreads();
  const int per = (n + SMALL_SORT_THREADS - 1) / SMALL_SORT_THREADS;
  const int lo = min(t * per, n), hi = min(lo + per, n);
  for (int bit = 0; bit < key_bits; ++bit) {
    int zeros = 0;
    for (int i = lo; i < hi; ++i) zeros += ((k0[i] >> bit) & 1u) == 0u;
    int incl = zeros;                  // inclusive scan of the zeros over the block
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int v = __shfl_up_sync(full, incl, off);
      if (lane >= off) incl += v;
    }
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    if (w == 0) {
      int sw = wsum[lane];
#pragma unroll
      for (int off = 1; off < NW; off <<= 1) {
        const int v = __shfl_up_sync(full, sw, off);
        if (lane >= off) sw += v;
      }
      wsum[lane] = sw;
    }
    __syncthreads();
    const int zeros_before = incl - zeros + (w > 0 ? wsum[w - 1] : 0);
    const int total_zeros = wsum[NW - 1];
    int z = zeros_before, o = total_zeros + (lo - zeros_before);
    for (int i = lo; i < hi; ++i) {
      const uint32_t key = k0[i];
      const int dst = ((key >> bit) & 1u) ? o++ : z++;
      k1[dst] = key;
      v1[dst] = v0[i];
    }
    __syncthreads();
    uint32_t* tk = k0; k0 = k1; k1 = tk;
    uint32_t* tv = v0; v0 = v1; v1 = tv;
  }
  for (int i = t; i < n; i += SMALL_SORT_THREADS) {
    const uint32_t key = k0[i];
    ka[i] = key;
    va[i] = v0[i];
    if (i == 0 || k0[i - 1] != key) tb[key] = i;
    if (i == n - 1 || k0[i + 1] != key) te[key] = i + 1;
    home[v0[i]] = key;
  }
  if (t == 0) {
    if (changed) *changed = 1;
    if (brick_count) *brick_count = 0;
  }
}

__global__ void __launch_bounds__(SMALL_SORT_THREADS)
small_sort_bins_kernel(int n, int key_bits, const uint32_t* __restrict__ kin,
                       const uint32_t* __restrict__ vin, uint32_t* __restrict__ ka,
                       uint32_t* __restrict__ va, int ntiles, int* __restrict__ tb,
                       int* __restrict__ te, uint32_t* __restrict__ home, const int* need,
                       int* changed, int* brick_count) {
  extern __shared__ uint32_t ssort[];
  small_sort_body(n, key_bits, kin, vin, ka, va, ntiles, tb, te, home, need, changed,
                  brick_count, ssort);
}



// ------------------------------------------------------------ gather + couple
// acc + sign h c: a 16-bit population's scaling and its part of a sum in one
// explicit operation.  Left to the compiler each kernel contracts products and
// sums in its own way (a bounced population comes out of a branch, which some
// kernels sum inside and some behind), while every variant of the
// interpolation, batched or not, has to give the same bits.
__device__ inline float add_pop(float acc, int sign, float h, float c) {
  return __fmaf_rn(sign > 0 ? h : -h, c, acc);
}

// j and 1 / rho at node (x, y, z)
template <typename S, bool WALLS>
__device__ inline void node_base(const GatherArgs& a, const Geom& g, int x, int y, int z,
                                 typename Store<S>::C (&j)[3], typename Store<S>::C& inv) {
  using C = typename Store<S>::C;
  C rd = C(0), j0 = C(0), j1 = C(0), j2 = C(0);
  if constexpr (sizeof(S) == 2) {
    float h[Q], bb[Q];
    uint32_t bounced;
    pull_raw<S, WALLS>(static_cast<const S*>(a.pops), g, a.bb_bot, a.bb_top, x, y, z, h, bb, bounced);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      float v = h[i], c = float(w_of(i)) * a.scale16;
      if (WALLS && cz_of(i)) {         // a value of its own, wall term included
        v = (bounced >> i) & 1u ? __fmaf_rn(v, c, bb[i]) : __fmul_rn(v, c);
        c = 1.0f;
      }
      rd = add_pop(rd, 1, v, c);
      if (cx_of(i)) j0 = add_pop(j0, cx_of(i), v, c);
      if (cy_of(i)) j1 = add_pop(j1, cy_of(i), v, c);
      if (cz_of(i)) j2 = add_pop(j2, cz_of(i), v, c);
    }
  } else {
    C f[Q];
    pull_cell<S, WALLS>(static_cast<const S*>(a.pops), g, a.bb_bot, a.bb_top, a.scale16, x, y, z, f);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const C v = f[i];
      rd += v;
      if (cx_of(i)) j0 += C(cx_of(i)) * v;
      if (cy_of(i)) j1 += C(cy_of(i)) * v;
      if (cz_of(i)) j2 += C(cz_of(i)) * v;
    }
  }
  j[0] = j0; j[1] = j1; j[2] = j2;
  inv = C(1) / (rv<C>(a.rho0_pop) + rd);
}

// do the stencil nodes b .. b + SN - 1 lie within [lo - 3, hi + 3] of the
// home tile (periodic wrap)?
template <int SN>
__device__ inline bool stencil_near_home(int b, int lo, int hi, int n, bool periodic) {
  if (periodic && n <= 3 * TILE) return true;     // the search window spans the axis
  int d = b - lo;
  if (periodic) {
    if (d < -n / 2) d += n;
    else if (d >= n - n / 2) d -= n;
  }
  return d >= -3 && d + SN - 1 <= hi - lo + 3;
}

// Gather and coupling update, one marker (sorted slot k) per thread.  The
// work of a thread is a chain of dependent memory accesses (slot, particle,
// stencil, node data, force tile, claims), so what does not depend on the
// chain is issued with it: the particle's own data is read before the node
// loop, the eight trilinear nodes are unrolled (their loads are in flight
// together), and a tile is claimed with one atomic exchange.
constexpr int GATHER_THREADS = 128;

// one cached node: j (3) and 1 / rho, stored as one 16-byte (float) or two
// 16-byte (double) vectors
__device__ inline void cache_load(const float* p, float (&j)[3], float& inv) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  j[0] = v.x; j[1] = v.y; j[2] = v.z; inv = v.w;
}
__device__ inline void cache_load(const double* p, double (&j)[3], double& inv) {
  const double2 v0 = reinterpret_cast<const double2*>(p)[0];
  const double2 v1 = reinterpret_cast<const double2*>(p)[1];
  j[0] = v0.x; j[1] = v0.y; j[2] = v1.x; inv = v1.y;
}
__device__ inline void cache_store(float* p, const float (&j)[3], float inv) {
  *reinterpret_cast<float4*>(p) = make_float4(j[0], j[1], j[2], inv);
}
__device__ inline void cache_store(double* p, const double (&j)[3], double inv) {
  reinterpret_cast<double2*>(p)[0] = make_double2(j[0], j[1]);
  reinterpret_cast<double2*>(p)[1] = make_double2(j[2], inv);
}

// fluid velocity at one stencil node from its j and 1 / rho:
// (((j + c1 F1) + cg g) + c2 F2) / rho (F1, F2 where their tile flags are set)
template <typename C>
__device__ __forceinline__ void node_velocity(const GatherArgs& a, long long cell, int tile, C (&j)[3],
                                              C inv, const C (&cgg)[3], C (&nv)[3]) {
  // each force 4-vector is loaded together with its tile's flag (it lies
  // inside the field either way) and used only where the flag is set, so
  // the two loads are not one after the other
  const C* F1 = static_cast<const C*>(a.F1);
  const C* F2 = static_cast<const C*>(a.F2);
  C f1x = C(0), f1y = C(0), f1z = C(0), f2x = C(0), f2y = C(0), f2z = C(0);
  bool on1 = false, on2 = false;
  if (F1) {
    on1 = a.flag1[tile] != 0;
    load_force(F1, cell, f1x, f1y, f1z);
  }
  if (F2) {
    on2 = a.flag2[tile] != 0;
    load_force(F2, cell, f2x, f2y, f2z);
  }
  if (on1) {
    const C c1 = rv<C>(a.c1);
    j[0] += c1 * f1x; j[1] += c1 * f1y; j[2] += c1 * f1z;
  }
  j[0] += cgg[0]; j[1] += cgg[1]; j[2] += cgg[2];
  if (on2) {
    const C c2 = rv<C>(a.c2);
    j[0] += c2 * f2x; j[1] += c2 * f2y; j[2] += c2 * f2z;
  }
  nv[0] = j[0] * inv; nv[1] = j[1] * inv; nv[2] = j[2] * inv;
}
// the same times the node's weight wt, added to own
template <typename C>
__device__ __forceinline__ void node_add(const GatherArgs& a, long long cell, int tile, C wt,
                                         C (&j)[3], C inv, const C (&cgg)[3], C (&own)[3]) {
  C nv[3];
  node_velocity<C>(a, cell, tile, j, inv, cgg, nv);
  own[0] += wt * nv[0]; own[1] += wt * nv[1]; own[2] += wt * nv[2];
}

// fluid velocity at one stencil node (x, y, z) of weight wt, added to own,
// with j and 1 / rho taken from the node-moment field where its tile is
// ready, else pulled from the populations
template <typename S, bool WALLS>
__device__ __forceinline__ void gather_node(const GatherArgs& a, const Geom& g, int x, int y, int z,
                                            typename Store<S>::C wt,
                                            const typename Store<S>::C (&cgg)[3],
                                            typename Store<S>::C (&own)[3]) {
  using C = typename Store<S>::C;
  C j[3], inv;
  const long long cell = z * g.plane + (long long)y * g.pitch + x;
  const int tile = tile_of(g, x, y, z);
  if (a.mom != nullptr && a.mready[tile])
    cache_load(static_cast<const C*>(a.mom) + 4 * cell, j, inv);
  else
    node_base<S, WALLS>(a, g, x, y, z, j, inv);
  node_add<C>(a, cell, tile, wt, j, inv, cgg, own);
}

// the next step's binning from a marker's end-of-step position, drifted on by
// key_ahead (base split: to the next step's force point): its tile key and
// index, and the flag that requests a re-sort (FP32 compute: the float
// splits of the coordinates, as the key-writing drift)
template <typename C>
__device__ __forceinline__ void next_bin(const GatherArgs& a, const Geom& g, long long i,
                                         double (&rn)[3], const double (&vn)[3]) {
  constexpr bool F32 = sizeof(C) == 4;
  if (a.key_ahead != 0.0) {
    const int n3[3] = {g.nx, g.ny, g.nz};
    const bool per[3] = {true, true, !g.walls};
#pragma unroll
    for (int c = 0; c < 3; ++c) rn[c] = wrap_axis(rn[c] + a.key_ahead * vn[c], n3[c], per[c]);
  }
  a.key_out[i] = F32 ? key_of_f(g, rn[0], rn[1], rn[2]) : key_of(g, rn[0], rn[1], rn[2]);
  a.idx_out[i] = (uint32_t)i;
  if (a.home && !(F32 ? near_home_f(g, a.home[i], rn) : near_home(g, a.home[i], rn))) *a.need_next = 1;
}

// the spreading's record of slot k (and its packed base)
template <int ST, typename C>
__device__ __forceinline__ void write_record(const GatherArgs& a, const Geom& g, long long k, const int (&b)[3],
                                             const C (&w)[3][4], const C (&F)[3]) {
  if constexpr (ST == 0) {
    TriRecT<C> r;
    // (periodic coordinates wrapped into the box)
    r.base = pack_base(wrap_int(b[0], g.nx), wrap_int(b[1], g.ny), g.walls ? b[2] : wrap_int(b[2], g.nz));
#pragma unroll
    for (int c = 0; c < 3; ++c) { r.t[c] = w[c][1]; r.F[c] = F[c]; }
    static_cast<TriRecT<C>*>(a.rec)[k] = r;
  } else {
    StencilRecT<C> r;
    r.bx = b[0]; r.by = b[1]; r.bz = b[2]; r.kind = ST;
#pragma unroll
    for (int q = 0; q < 4; ++q) { r.wx[q] = w[0][q]; r.wy[q] = w[1][q]; r.wz[q] = w[2][q]; }
    r.F[0] = F[0]; r.F[1] = F[1]; r.F[2] = F[2];
    r.pad = C(0);
    static_cast<StencilRecT<C>*>(a.rec)[k] = r;
    a.reach[k] = pack_base(b[0], b[1], b[2]);
  }
}

// The lane's stencil nodes (the rows ky = q (mod GL) of lane q of a marker's
// GL lanes; every row for GL = 1) read from the node-moment field in the
// order of the generic loop, with the cell and tile offsets of a row taken
// once: the same sum as there when every node's tile is ready.  Returns
// false if one was not (own is then to be redone by the generic loop; the
// values read here are discarded).
template <typename S, bool WALLS, int SN, int GL>
__device__ __forceinline__ bool gather_field(const GatherArgs& a, const Geom& g, const int (&xs)[SN],
                                             const int (&ys)[SN], const int (&zs)[SN],
                                             const typename Store<S>::C (&w)[3][4], int sub,
                                             const typename Store<S>::C (&cgg)[3],
                                             typename Store<S>::C (&own)[3]) {
  using C = typename Store<S>::C;
  const C* mom = static_cast<const C*>(a.mom);
  bool ok = true;
  int txs[SN];
#pragma unroll
  for (int q = 0; q < SN; ++q) txs[q] = xs[q] >> TILE_SHIFT;
#pragma unroll 1
  for (int kz = 0; kz < SN; ++kz) {
    const int z = pick(zs, kz);
    if (WALLS && z < 0) continue;
    const C wz = pick(w[2], kz);
    const long long cz = z * g.plane;
    const int tz = (z >> TILE_SHIFT) * g.nty;
#pragma unroll 1
    for (int ky = sub; ky < SN; ky += GL) {
      const int y = pick(ys, ky);
      const C wyz = pick(w[1], ky) * wz;
      const long long crow = cz + (long long)y * g.pitch;
      const int trow = (tz + (y >> TILE_SHIFT)) * g.ntx;
#pragma unroll
      for (int kx = 0; kx < SN; ++kx) {
        const long long cell = crow + xs[kx];
        const int tile = trow + txs[kx];
        ok &= a.mready[tile] != 0;
        C j[3], inv;
        cache_load(mom + 4 * cell, j, inv);
        node_add<C>(a, cell, tile, w[0][kx] * wyz, j, inv, cgg, own);
      }
    }
  }
  return ok;
}

// Variants (VAR) of the interpolation:
//   GV_FULL    one lane per marker, no node cache: pulls the populations of
//              two nodes at a time (or reads the node-moment field);
//   GV_LIGHT   the same for launches that read the node-moment field (fewer
//              registers, more markers in flight);
//   GV_CACHED  one lane per marker with the node cache: markers whose cache
//              entry does not hold are refilled by the whole warp first
//              (refill_cache), then every lane reads its nodes from the
//              cache with all loads in flight;
//   GV_GROUP   a group of lanes per marker (gather_group_body): eight for the
//              trilinear stencil, one per node, four for the others;
//   GV_QUAD    (4- and 3-point stencils, 16-bit storage) four lanes per
//              marker, lane q taking the rows ky = q (mod 4) of every plane,
//              their parts summed with a fixed butterfly.  16-bit storage
//              keeps this order of the sum where FP32 and FP64 take the
//              group's: its fluid rounds stochastically, so a force that
//              differs in the last place changes every later step's draws.
//   GV_PULL    GV_GROUP of the 4- and 3-point stencils without the node-moment
//              field
constexpr int GV_FULL = 0, GV_LIGHT = 1, GV_CACHED = 2, GV_GROUP = 3, GV_QUAD = 4, GV_PULL = 5;

// Coupling force F^h of N components from the slip dv = v - u(X), the
// intrinsic force Fi and the random force zeta (compute type)
template <typename C, int N>
__device__ __forceinline__ void couple_force(const GatherArgs& __restrict__ a, C cim, const C (&dv)[N],
                                             const C (&Fi)[N], const C (&zeta)[N], C (&Fh)[N]) {
  const C cs = rv<C>(a.s), crho = rv<C>(a.rho0);
  if (a.kind == 4) {                        // modified EBF, Eq. [modified-ebf]
    // r = 1/(1 + m/rho0) = rho0 im/(rho0 im + 1); 1/(s(1/m + 1/rho0))
    const C r = crho * cim / (crho * cim + C(1));
    const C inv = C(1) / (cs * (cim + C(1) / crho));
#pragma unroll
    for (int c = 0; c < N; ++c) Fh[c] = -dv[c] * inv - r * Fi[c];
  } else {
    const C gam = a.kind == 3 ? crho : rv<C>(a.gamma);   // EBF: rho a^3 / h
    if (a.order == 1) {
#pragma unroll
      for (int c = 0; c < N; ++c) Fh[c] = -gam * dv[c];
      if (a.noise)
#pragma unroll
        for (int c = 0; c < N; ++c) Fh[c] += zeta[c];
    } else {                                // Crank-Nicolson, Eq. [modified-force]
      const C al = gam * cs * cim, be = gam * cs / crho;
      const C D = C(1) + C(0.5) * al + C(0.5) * be;
      if (a.noise) {
#pragma unroll
        for (int c = 0; c < N; ++c) Fh[c] = -((gam * dv[c] + C(0.5) * al * Fi[c]) - zeta[c]) / D;
      } else {
#pragma unroll
        for (int c = 0; c < N; ++c) Fh[c] = -(gam * dv[c] + C(0.5) * al * Fi[c]) / D;
      }
    }
  }
}

// The tile of stencil node q of an axis, or -1 if it carries no weight, lies
// outside the box or repeats an earlier node's tile
template <int SN, typename C>
__device__ __forceinline__ void axis_tiles(int b, const C (&w)[4], int n, bool periodic, int (&tq)[SN]) {
#pragma unroll
  for (int q = 0; q < SN; ++q) {
    int t = -1;
    if (w[q] != C(0)) {
      int node = b + q;
      if (periodic) node = wrap_int(node, n);
      if (node >= 0 && node < n) t = node >> TILE_SHIFT;
    }
#pragma unroll
    for (int e = 0; e < q; ++e) if (tq[e] == t) t = -1;
    tq[q] = t;
  }
}

// the bins are valid while every stencil node lies within three cells of the
// home tile (the reach of the spreading's neighbour search)
template <int SN>
__device__ __forceinline__ bool bins_hold(const Geom& g, int home, const int (&b)[3]) {
  const unsigned t = (unsigned)home, r = t / (unsigned)g.ntx, tz = r / (unsigned)g.nty;
  const int tt[3] = {(int)(t - r * g.ntx), (int)(r - tz * g.nty), (int)tz};
  const int n3[3] = {g.nx, g.ny, g.nz};
  bool ok = true;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int lo = tt[c] * TILE, hi = min(lo + TILE, n3[c]) - 1;
    ok = ok && stencil_near_home<SN>(b[c], lo, hi, n3[c], c < 2 || !g.walls);
  }
  return ok;
}

// Cached variant: the whole warp fills the cache entries of its lanes'
// markers with `want` set.  The lanes take the nodes of those markers side by
// side (trilinear: eight nodes of four markers per round; three-point: one
// marker, four-point: one marker in two rounds), so the 19 loads of a node
// are in flight for 32 nodes at once and neighbouring nodes share sectors.
// When every lane pulled its own marker's nodes one after the other, one
// lane whose base had changed held its warp, and with it the kernel, for as
// long as filling everything: 100 000 markers 36 us per sub-step, 24-26 us with
// the shared refill, of which the kernel's chain of about 2600 instructions per
// warp is what is left.
template <typename S, bool WALLS, int SN>
__device__ __forceinline__ void refill_cache(const GatherArgs& __restrict__ a, const Geom& g,
                                             long long M, long long gid, const int (&b)[3], bool want) {
  using C = typename Store<S>::C;
  constexpr unsigned full = 0xffffffffu;
  constexpr int NN = SN * SN * SN;
  constexpr int PER = NN <= 32 ? 32 / NN : 1;          // markers per round
  const int lane = threadIdx.x & 31;
  C* nc = static_cast<C*>(a.ncache);
  unsigned todo = __ballot_sync(full, want);
  const int r = NN <= 32 ? lane / NN : 0;              // the lane's marker of the round
  while (todo != 0u) {
    unsigned t = todo;
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      if (e < r) t &= t - 1u;                          // drop the markers of other lanes
      todo &= todo - 1u;
    }
    const bool have = t != 0u && r < PER;
    const int src = have ? __ffs(t) - 1 : 0;
    const int bx = __shfl_sync(full, b[0], src), by = __shfl_sync(full, b[1], src),
              bz = __shfl_sync(full, b[2], src);
    const long long kk = gid - lane + src;             // slots follow the lanes
    if (have) {
      for (int node = lane - r * NN; node < NN; node += 32) {
        const int qx = node % SN, qy = (node / SN) % SN, qz = node / (SN * SN);
        const int x = wrap_int(bx + qx, g.nx), y = wrap_int(by + qy, g.ny);
        int z = bz + qz;
        if (!WALLS) z = wrap_int(z, g.nz);
        if (WALLS && (z < 0 || z >= g.nz)) continue;
        C j[3], inv;
        node_base<S, WALLS>(a, g, x, y, z, j, inv);
        cache_store(nc + (node * M + kk) * 4, j, inv);
      }
    }
  }
  __syncwarp();                                        // the entries are read by their owners
}

// Fluid velocity from the cached trilinear nodes, F1 and F2 present or not
// at compile time: the node, force and flag loads of a plane of nodes are
// issued together, then added in node order.
template <typename C, bool HAS1, bool HAS2>
__device__ __forceinline__ void cached_nodes(const GatherArgs& __restrict__ a, const Geom& g, long long M,
                                             long long k, const int (&xs)[2], const int (&ys)[2],
                                             const int (&zs)[2], const C (&w)[3][4], const C (&cgg)[3],
                                             C (&own)[3]) {
  const C* nc = static_cast<const C*>(a.ncache) + 4 * k;
  const C* F1 = static_cast<const C*>(a.F1);
  const C* F2 = static_cast<const C*>(a.F2);
  const C c1 = rv<C>(a.c1), c2 = rv<C>(a.c2);
#pragma unroll
  for (int kz = 0; kz < 2; ++kz) {
    if (zs[kz] < 0) continue;                          // beyond a wall
    C j[4][3], inv[4], f1[4][3], f2[4][3];
    bool on1[4], on2[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int y = ys[q >> 1], x = xs[q & 1];
      cache_load(nc + (4 * kz + q) * M * 4, j[q], inv[q]);
      const long long cell = zs[kz] * g.plane + (long long)y * g.pitch + x;
      const int tile = tile_of(g, x, y, zs[kz]);
      if (HAS1) {
        on1[q] = a.flag1[tile] != 0;
        load_force(F1, cell, f1[q][0], f1[q][1], f1[q][2]);
      }
      if (HAS2) {
        on2[q] = a.flag2[tile] != 0;
        load_force(F2, cell, f2[q][0], f2[q][1], f2[q][2]);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const C wt = w[0][q & 1] * (w[1][q >> 1] * w[2][kz]);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        C v = j[q][c];
        if (HAS1) v = on1[q] ? v + c1 * f1[q][c] : v;
        v += cgg[c];
        if (HAS2) v = on2[q] ? v + c2 * f2[q][c] : v;
        own[c] += wt * (v * inv[q]);
      }
    }
  }
}

// List slots for the tiles claimed by the warp's lanes (nclaim each), one
// atomic per warp: the lane's first slot.  `am`: the lanes taking part (the
// first nact of the warp).
__device__ __forceinline__ int claim_slots(int* nlive, int nclaim, unsigned am, int nact) {
  const int lane = threadIdx.x & 31;
  int incl = nclaim;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int u = __shfl_up_sync(am, incl, off);
    if (lane >= off) incl += u;
  }
  const int total = __shfl_sync(am, incl, nact - 1);
  int base = 0;
  if (lane == nact - 1 && total > 0) base = atomicAdd(nlive, total);
  return __shfl_sync(am, base, nact - 1) + incl - nclaim;
}

// The tile claims of a 4- or 3-point stencil: loops over the distinct tiles per
// axis instead of the SN^3 node combinations: per axis the distinct tiles of
// the nodes with non-zero weight, in node order (at most three: a partial last
// tile and the periodic wrap), their combinations shared out over the
// marker's GL lanes.
template <int SN, int GL, typename C>
__device__ __forceinline__ void claim_wide(const GatherArgs& a, const Geom& g, const int (&b)[3],
                                           const C (&w)[3][4], int sub, bool valid, unsigned am, int nact) {
  const int n3[3] = {g.nx, g.ny, g.nz};
  const bool per[3] = {true, true, !g.walls};
  int tl[3][3], ntl[3];
  uint32_t claimed = 0u;               // bit of the tile combination cid
  int nclaim = 0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    ntl[c] = 0;
    tl[c][0] = tl[c][1] = tl[c][2] = -1;
#pragma unroll
    for (int q = 0; q < SN; ++q) {
      if (w[c][q] == C(0)) continue;
      int node = b[c] + q;
      if (per[c]) node = wrap_int(node, n3[c]);
      if (node < 0 || node >= n3[c]) continue;
      const int t = node >> TILE_SHIFT;
      if (t == tl[c][0] || t == tl[c][1] || t == tl[c][2]) continue;
      if (ntl[c] == 0) tl[c][0] = t;
      else if (ntl[c] == 1) tl[c][1] = t;
      else tl[c][2] = t;
      ++ntl[c];
    }
  }
  // claim the tiles the stencil reaches: the combinations of the axes'
  // tiles, shared out over the marker's lanes
  int cid = 0;
  for (int iz = 0; iz < ntl[2]; ++iz)
    for (int iy = 0; iy < ntl[1]; ++iy)
      for (int ix = 0; ix < ntl[0]; ++ix, ++cid) {
        if (cid % GL != sub || !valid) continue;
        const int tx = pick(tl[0], ix), ty = pick(tl[1], iy), tz = pick(tl[2], iz);
        // most tiles are claimed already: an L2 read (marks only go
        // from 0 to 1 during the gather) spares their atomic
        uint32_t* m = a.mark + (tz * g.nty + ty) * g.ntx + tx;
        if (__ldcg(m) == 0u && atomicExch(m, 1u) == 0u) {
          claimed |= 1u << cid;
          ++nclaim;
        }
      }
  int base = claim_slots(a.nlive, nclaim, am, nact);
  if (claimed != 0u) {
    int cid2 = 0;
    for (int iz = 0; iz < ntl[2]; ++iz)
      for (int iy = 0; iy < ntl[1]; ++iy)
        for (int ix = 0; ix < ntl[0]; ++ix, ++cid2)
          if (claimed & (1u << cid2)) {
            const int tx = pick(tl[0], ix), ty = pick(tl[1], iy), tz = pick(tl[2], iz);
            a.live_tiles[base++] = make_int4((tz * g.nty + ty) * g.ntx + tx, tx, ty, tz);
          }
  }
}

// the body of the gather for thread gid of one box's launch (whole warps of
// one box: gid - lane is a multiple of 32)
template <typename S, bool WALLS, int ST, int VAR>
__device__ __forceinline__ void gather_body(const PartArgs& __restrict__ p,
                                            const GatherArgs& __restrict__ a, long long gid) {
  using C = typename Store<S>::C;
  constexpr int SN = nodes_1d<ST>();
  constexpr int GL = VAR == GV_QUAD ? 4 : 1;       // lanes per marker
  constexpr bool CACHED = VAR == GV_CACHED;
  const Geom& g = p.g;
  const long long M = p.M;
  const int lane = threadIdx.x & 31;
  // the lanes still running: whole groups, the first nact of the warp; with
  // the cache every lane stays (the refill is the whole warp's work), the
  // ones past the last marker on the last marker and without writing
  if (!CACHED && gid / GL >= M) return;
  const bool valid = gid / GL < M;
  const long long k = valid ? gid / GL : M - 1;
  const int sub = (int)(gid % GL);
  const long long i = a.perm ? (long long)a.perm[k] : k;
  const int n3[3] = {g.nx, g.ny, g.nz};
  const bool per[3] = {true, true, !g.walls};
  int4 cb = make_int4(0, 0, 0, 0);
  bool try_reuse = false;
  if (CACHED && a.cache == 2) {
    cb = a.ncache_b[k];
    try_reuse = a.invalidate == nullptr || *a.invalidate == 0;
  }

  // the particle's own data (independent of the gather); with a fused
  // drift this thread first does its marker's drift sub-step
  double v[3] = {0.0, 0.0, 0.0};
  double im = 0.0;
  C Fi[3] = {C(0), C(0), C(0)};
  double X[3];
  const bool at_aux = a.mode == GM_IBM_HALF || a.mode == GM_IBM_FINAL;
  const int home = a.keys ? (int)a.keys[k] : 0;
  if (GL == 1 && a.fused) {
    C F[3];
    im = a.inv_mass[i];
    drift_one<C>(p, a.drift, i, X, v, F);
    if (a.include_int)
#pragma unroll
      for (int c = 0; c < 3; ++c) Fi[c] = F[c];
  } else {
    const C* fint = static_cast<const C*>(a.fint);
    if (a.mode == GM_COUPLE) {
      im = a.inv_mass[i];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        v[c] = a.vel[c * M + i];
        if (a.include_int) Fi[c] = fint[c * M + i];
      }
    } else if (a.mode == GM_IBM_HALF || a.mode == GM_IBM1) {
#pragma unroll
      for (int c = 0; c < 3; ++c) Fi[c] = fint[c * M + i];
    }
    const double* P = at_aux ? a.aux : a.pos;
#pragma unroll
    for (int c = 0; c < 3; ++c) X[c] = P[c * M + i];
  }
  if (valid && k == 0 && sub == 0 && a.clear_next) {      // the next step's flags (read by none now)
    a.clear_next[0] = 0;
    a.clear_next[1] = 0;
  }

  int b[3];
  C w[3][4];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if constexpr (sizeof(C) == 4) {
      float xh, xl;
      split_df(X[c], xh, xl);
      stencil_1d_df<ST>(xh, xl, b[c], w[c]);
    } else {
      stencil_1d<ST, C>(X[c], b[c], w[c]);
    }
  }

  C own[3] = {C(0), C(0), C(0)};
  if (a.mode != GM_IBM1) {
    int xs[SN], ys[SN], zs[SN];
#pragma unroll
    for (int q = 0; q < SN; ++q) {
      xs[q] = wrap_int(b[0] + q, g.nx);
      ys[q] = wrap_int(b[1] + q, g.ny);
      const int zz = b[2] + q;
      zs[q] = WALLS ? ((zz < 0 || zz >= g.nz) ? -1 : zz) : wrap_int(zz, g.nz);
    }
    const C cgg[3] = {rv<C>(a.cgg[0]), rv<C>(a.cgg[1]), rv<C>(a.cgg[2])};
    // node (kx, ky, kz) of slot k sits at nc[((kz SN + ky) SN + kx) M + k] (x 4)
    if constexpr (CACHED) {
      const bool reuse = try_reuse && cb.x == b[0] && cb.y == b[1] && cb.z == b[2];
      const bool want = valid && !reuse;
      if (want) a.ncache_b[k] = make_int4(b[0], b[1], b[2], 0);
      refill_cache<S, WALLS, SN>(a, g, M, gid, b, want);
      if constexpr (SN == 2) {
        if (a.F1 != nullptr) {
          if (a.F2 != nullptr) cached_nodes<C, true, true>(a, g, M, k, xs, ys, zs, w, cgg, own);
          else cached_nodes<C, true, false>(a, g, M, k, xs, ys, zs, w, cgg, own);
        } else {
          if (a.F2 != nullptr) cached_nodes<C, false, true>(a, g, M, k, xs, ys, zs, w, cgg, own);
          else cached_nodes<C, false, false>(a, g, M, k, xs, ys, zs, w, cgg, own);
        }
      } else {
        const C* nc = static_cast<const C*>(a.ncache);
#pragma unroll 1
        for (int kz = 0; kz < SN; ++kz) {
          const int z = pick(zs, kz);
          if (WALLS && z < 0) continue;
          const C wz = pick(w[2], kz);
#pragma unroll 1
          for (int ky = 0; ky < SN; ++ky) {
            const int y = pick(ys, ky);
            const C wyz = pick(w[1], ky) * wz;
#pragma unroll
            for (int kx = 0; kx < SN; ++kx) {
              C j[3], inv;
              cache_load(nc + (((kz * SN + ky) * SN + kx) * M + k) * 4, j, inv);
              const long long cell = z * g.plane + (long long)y * g.pitch + xs[kx];
              node_add<C>(a, cell, tile_of(g, xs[kx], y, z), w[0][kx] * wyz, j, inv, cgg, own);
            }
          }
        }
      }
    } else {
      bool done = false;
      if (a.mom != nullptr) {
        done = gather_field<S, WALLS, SN, GL>(a, g, xs, ys, zs, w, sub, cgg, own);
        if (!done) own[0] = own[1] = own[2] = C(0);
      }
      if (done) {
      } else if (SN == 2) {
#pragma unroll
        for (int kz = 0; kz < SN; ++kz)
#pragma unroll
          for (int ky = 0; ky < SN; ++ky)
#pragma unroll
            for (int kx = 0; kx < SN; ++kx) {
              if (WALLS && zs[kz] < 0) continue;
              const C wt = w[0][kx] * (w[1][ky] * w[2][kz]);
              gather_node<S, WALLS>(a, g, xs[kx], ys[ky], zs[kz], wt, cgg, own);
            }
      } else {
        // the loops are not unrolled: the per-axis nodes and weights are
        // picked by selects, which keeps them in registers
#pragma unroll 1
        for (int kz = 0; kz < SN; ++kz) {
          const int z = pick(zs, kz);
          if (WALLS && z < 0) continue;
          const C wz = pick(w[2], kz);
#pragma unroll 1
          for (int ky = sub; ky < SN; ky += GL) {
            const int y = pick(ys, ky);
            const C wyz = pick(w[1], ky) * wz;
#pragma unroll 2
            for (int kx = 0; kx < SN; ++kx)
              gather_node<S, WALLS>(a, g, pick(xs, kx), y, z, pick(w[0], kx) * wyz, cgg, own);
          }
        }
      }
    }
  }
  const long long wbase = gid - lane;
  const int nact = CACHED || M * GL - wbase >= 32 ? 32 : (int)(M * GL - wbase);
  const unsigned am = nact == 32 ? 0xffffffffu : ((1u << nact) - 1u);
  if (GL > 1) {
#pragma unroll
    for (int off = 1; off < GL; off <<= 1)
#pragma unroll
      for (int c = 0; c < 3; ++c) own[c] += __shfl_xor_sync(am, own[c], off);
  }

  // ---- own marker: coupling / advection update (FP64 integration),
  // stencil record and tile claims
  const double s = a.s.d;
  C Frec[3] = {C(0), C(0), C(0)};
  switch (sub == 0 && valid ? a.mode : -1) {
    case GM_COUPLE: {
      // slip v - u(X) in the compute type (FP64 work being scarce): with
      // FP32 the rounding of v adds at most 2^-24 |v| to it
      C dv[3], zeta[3] = {C(0), C(0), C(0)}, Fh[3];
      for (int c = 0; c < 3; ++c) dv[c] = (C)v[c] - own[c];
      // the random force zeta of this (sub-)step (thermal boxes)
      if (a.noise) {
        C r[4];
        philox_gauss4<C>((uint32_t)i, (uint32_t)(*a.tstep), 8u + (uint32_t)a.substep, 0u,
                         a.tkey0, a.tkey1, r);
        const C za = rv<C>(a.zeta_amp);
        for (int c = 0; c < 3; ++c) zeta[c] = za * r[c];
      }
      couple_force<C, 3>(a, C(im), dv, Fi, zeta, Fh);
      const double kick = s * im;
      double vn[3];
      for (int c = 0; c < 3; ++c) {
        vn[c] = v[c] + kick * (double)(Fh[c] + Fi[c]);
        a.vel[c * M + i] = vn[c];
        if (a.fh_out) static_cast<C*>(a.fh_out)[c * M + i] = Fh[c];
        Frec[c] = -rv<C>(a.rec_weight) * Fh[c];
      }
      // the drift to the next force evaluation (done here once, instead of
      // by every reader of this marker's position)
      if (a.pos_next) {
        // (FP32 compute: the two quarter drifts as one, (post_a + post_b) v)
        const double post_ab = sizeof(C) == 4 ? a.post_a + a.post_b : 0.0;
        double rn[3];
        for (int c = 0; c < 3; ++c) {
          rn[c] = wrap_axis(sizeof(C) == 4 ? X[c] + post_ab * vn[c]
                                           : (X[c] + a.post_a * vn[c]) + a.post_b * vn[c],
                            n3[c], per[c]);
          a.pos_next[c * M + i] = rn[c];
        }
        if (a.key_out) next_bin<C>(a, g, i, rn, vn);
      }
      break;
    }
    case GM_IBM_PREDICT:
      for (int c = 0; c < 3; ++c)
        a.aux[c * M + i] = wrap_axis(a.pos[c * M + i] + s * (double)own[c], n3[c], per[c]);
      break;
    case GM_IBM_HALF:
    case GM_IBM_FINAL:
    case GM_ADVECT:
      for (int c = 0; c < 3; ++c)
        a.pos[c * M + i] = wrap_axis(a.pos[c * M + i] + s * (double)own[c], n3[c], per[c]);
      if (a.mode == GM_IBM_HALF)
        for (int c = 0; c < 3; ++c) Frec[c] = rv<C>(a.rec_weight) * Fi[c];
      break;
    case GM_IBM1:
      for (int c = 0; c < 3; ++c) Frec[c] = rv<C>(a.rec_weight) * Fi[c];
      break;
    default:
      break;
  }
  if (a.rec && (a.mode == GM_COUPLE || a.mode == GM_IBM_HALF || a.mode == GM_IBM1)) {
    if (sub == 0 && valid) {
      write_record<ST>(a, g, k, b, w, Frec);
      if (a.keys && !bins_hold<SN>(g, home, b)) *a.status = 1;
    }
    if constexpr (SN == 2) {
      // trilinear: the 2 x 2 x 2 node combinations, unrolled.  The marker
      // joins the hit list of every tile it reaches; the first to join
      // claims the tile.  All the joins are issued before any of their
      // counts is looked at.
      int tq[3][SN];
#pragma unroll
      for (int c = 0; c < 3; ++c) axis_tiles<SN>(b[c], w[c], n3[c], per[c], tq[c]);
      uint32_t slot[8];
      unsigned joined = 0u;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int tx = tq[0][q & 1], ty = tq[1][(q >> 1) & 1], tz = tq[2][q >> 2];
        slot[q] = 1u;
        if (valid && tx >= 0 && ty >= 0 && tz >= 0) {
          slot[q] = atomicAdd(a.hcnt + (tz * g.nty + ty) * g.ntx + tx, 1u);
          joined |= 1u << q;
        }
      }
      unsigned claimed = 0u;
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (joined & (1u << q)) {
          const int tile = (tq[2][q >> 2] * g.nty + tq[1][(q >> 1) & 1]) * g.ntx + tq[0][q & 1];
          if (slot[q] < (uint32_t)SPREAD_HCAP)
            a.hits[(size_t)tile * SPREAD_HCAP + slot[q]] = (uint32_t)k;
          if (slot[q] == 0u) {
            a.mark[tile] = 1u;
            claimed |= 1u << q;
          }
        }
      int base = claim_slots(a.nlive, __popc(claimed), am, nact);
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (claimed & (1u << q)) {
          const int tx = tq[0][q & 1], ty = tq[1][(q >> 1) & 1], tz = tq[2][q >> 2];
          a.live_tiles[base++] = make_int4((tz * g.nty + ty) * g.ntx + tx, tx, ty, tz);
        }
    } else {
      claim_wide<SN, GL, C>(a, g, b, w, sub, valid, am, nact);
    }
  }
}

// One lane's column of a 4- or 3-point stencil (x fixed; rows ys, planes zs)
// from the node-moment field, two planes of rows with their loads in flight
// together.  The rows lie in the tiles of the first and the last row (else, or
// where a tile is not ready, false is returned and own is to be redone node by
// node), so the ready bytes and force flags are loaded for two tiles a plane.
// HAS: the force field F1 is added.
template <int SN, bool HAS, typename C>
__device__ __forceinline__ bool wide_column(const GatherArgs& __restrict__ a, const Geom& g, int x,
                                            const int (&ys)[SN], const int (&zs)[SN], C wx,
                                            const C (&w)[3][4], const C (&cgg)[3], C (&own)[3]) {
  const C* mom = static_cast<const C*>(a.mom);
  const C* F1 = static_cast<const C*>(a.F1);
  const C c1 = rv<C>(a.c1);
  const int tx = x >> TILE_SHIFT, ty0 = ys[0] >> TILE_SHIFT, ty1 = ys[SN - 1] >> TILE_SHIFT;
  bool ok = true;
#pragma unroll
  for (int q = 1; q < SN - 1; ++q) ok &= (ys[q] >> TILE_SHIFT) == ty0 || (ys[q] >> TILE_SHIFT) == ty1;
  if (!ok) return false;
#pragma unroll 1
  for (int k0 = 0; k0 < SN; k0 += 2) {
    C j[2][SN][3], inv[2][SN], f[2][SN][3];
    bool on[2][2], in[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int z = k0 + h < SN ? pick(zs, k0 + h) : -1;
      in[h] = z >= 0;                                  // a plane of the stencil, not beyond a wall
      on[h][0] = on[h][1] = false;
      if (!in[h]) continue;
      const int t0 = ((z >> TILE_SHIFT) * g.nty + ty0) * g.ntx + tx, t1 = t0 + (ty1 - ty0) * g.ntx;
      ok &= a.mready[t0] != 0 && a.mready[t1] != 0;
      if (HAS) {
        on[h][0] = a.flag1[t0] != 0;
        on[h][1] = a.flag1[t1] != 0;
      }
#pragma unroll
      for (int ky = 0; ky < SN; ++ky) {
        const long long cell = z * g.plane + (long long)ys[ky] * g.pitch + x;
        cache_load(mom + 4 * cell, j[h][ky], inv[h][ky]);
        if (HAS) load_force(F1, cell, f[h][ky][0], f[h][ky][1], f[h][ky][2]);
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (!in[h]) continue;
      const C wxz = wx * pick(w[2], k0 + h);
#pragma unroll
      for (int ky = 0; ky < SN; ++ky) {
        const bool o = HAS && ((ys[ky] >> TILE_SHIFT) == ty0 ? on[h][0] : on[h][1]);
        const C wt = wxz * w[1][ky];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          C v = j[h][ky][c];
          if (HAS) v = o ? v + c1 * f[h][ky][c] : v;
          v += cgg[c];
          own[c] += wt * (v * inv[h][ky]);
        }
      }
    }
  }
  return ok;
}

// The interpolation with a group of lanes per marker, all of its lanes taking
// part in every stage.
//
// Trilinear: eight lanes per marker (every mode; with or without the node
// cache and the fused drift).  Lane q owns node
// (q & 1, (q >> 1) & 1, q >> 2): its cache entry, field entry or 19
// populations are loaded side by side with the other nodes', the node
// velocities are added in node order through shuffles (the same sum as with
// one lane, bit for bit), lanes 0-2 update one component of the marker each,
// and lane q joins the hit list of one tile combination.  A launch of few
// markers lasts as long as one marker's chain of dependent loads, which is
// about one load per stage here (1000 markers, populations pulled: 34 us per
// launch with one lane, whole step of the 64^3 box 66 -> 39 us).
//
// 4- and 3-point stencils (no node cache, no fused drift): four lanes per
// marker, lane q owning the nodes kx = q of every row, so a row of the stencil
// is one contiguous access of the group; the lanes' parts are summed with a
// fixed butterfly.  One lane per marker (or one row per lane) sends 32 lines
// per field load, a group per row about 11: L1's tag lookups fall from 0.44-0.56
// to 0.16-0.26 per cycle and SM, and latency is what is left.
// 41 088 shell markers in 192^3 42 -> 30 us per launch (a row per lane before),
// shell step 387 -> 350 us, one shell in 48^3 58 -> 54 us.
// PULL (4- and 3-point): no node-moment field, the populations are pulled; a
// kernel of its own, so that its registers are not the field reads' (in one
// kernel these spilled, 1.5 % of the shell steps).  IBM, us per step, one node
// after the other and PER nodes in flight: 10 markers in 128^3 125 -> 121
// (4-point), 104 -> 96 (3-point); 1000 markers 137 -> 134, 115 -> 106.
template <typename S, bool WALLS, int ST, bool PULL>
__device__ __forceinline__ void gather_group_body(const PartArgs& __restrict__ p,
                                                const GatherArgs& __restrict__ a, long long gid) {
  using C = typename Store<S>::C;
  constexpr int SN = nodes_1d<ST>();
  constexpr int GL = ST == 0 ? 8 : 4;
  const Geom& g = p.g;
  const long long M = p.M;
  const int lane = threadIdx.x & 31;
  const long long k = gid / GL;
  const int sub = lane & (GL - 1), lead = lane & ~(GL - 1);
  if (k >= M) return;                  // whole groups leave together
  const long long wbase = gid - lane;
  const int nact = GL * M - wbase >= 32 ? 32 : (int)(GL * M - wbase);
  const unsigned am = nact == 32 ? 0xffffffffu : ((1u << nact) - 1u);
  const long long i = a.perm ? (long long)a.perm[k] : k;
  const int n3[3] = {g.nx, g.ny, g.nz};
  const bool per[3] = {true, true, !g.walls};
  const int comp = sub < 3 ? sub : 2;             // the lane's component
  int4 cb = make_int4(0, 0, 0, 0);
  bool try_reuse = false;
  if (ST == 0 && a.cache == 2) {
    cb = a.ncache_b[k];
    try_reuse = a.invalidate == nullptr || *a.invalidate == 0;
  }
  const int home = a.keys ? (int)a.keys[k] : 0;
  const bool at_aux = a.mode == GM_IBM_HALF || a.mode == GM_IBM_FINAL;
  double X[3], vc = 0.0, im = 0.0;
  C Fc = C(0);
  if (ST == 0 && a.fused) {
    double v[3];
    C F[3];
    im = a.inv_mass[i];
    drift_one<C>(p, a.drift, i, X, v, F);
    vc = pick(v, comp);
    if (a.include_int) Fc = pick(F, comp);
  } else {
    const C* fint = static_cast<const C*>(a.fint);
    if (a.mode == GM_COUPLE) {
      im = a.inv_mass[i];
      vc = a.vel[comp * M + i];
      if (a.include_int) Fc = fint[comp * M + i];
    } else if (a.mode == GM_IBM_HALF || a.mode == GM_IBM1) {
      Fc = fint[comp * M + i];
    }
    const double* P = at_aux ? a.aux : a.pos;
#pragma unroll
    for (int c = 0; c < 3; ++c) X[c] = P[c * M + i];
  }
  if (gid == 0 && a.clear_next) {      // the next step's flags (read by none now)
    a.clear_next[0] = 0;
    a.clear_next[1] = 0;
  }
  int b[3];
  C w[3][4];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if constexpr (sizeof(C) == 4) {
      float xh, xl;
      split_df(X[c], xh, xl);
      stencil_1d_df<ST>(xh, xl, b[c], w[c]);
    } else {
      stencil_1d<ST, C>(X[c], b[c], w[c]);
    }
  }
  C own[3] = {C(0), C(0), C(0)};
  if (a.mode != GM_IBM1) {
    if constexpr (ST == 0) {
    const int x = wrap_int(b[0] + (sub & 1), g.nx), y = wrap_int(b[1] + ((sub >> 1) & 1), g.ny);
    int z = b[2] + (sub >> 2);
    if (!WALLS) z = wrap_int(z, g.nz);
    const bool in = !WALLS || (z >= 0 && z < g.nz);
    C nv[3] = {C(0), C(0), C(0)};
    bool reuse = false;
    if (a.cache != 0) {
      reuse = try_reuse && cb.x == b[0] && cb.y == b[1] && cb.z == b[2];
      // every lane of the group has read the entry's base before lane 0
      // replaces it (a lane running behind would take the new base for the
      // base of its old node)
      __syncwarp(am);
      if (sub == 0 && !reuse) a.ncache_b[k] = make_int4(b[0], b[1], b[2], 0);
    }
    if (in) {
      const long long cell = z * g.plane + (long long)y * g.pitch + x;
      const int tile = tile_of(g, x, y, z);
      C* slot = static_cast<C*>(a.ncache) + (sub * M + k) * 4;
      C j[3], inv;
      if (reuse) {
        cache_load(slot, j, inv);
      } else if (a.mom != nullptr && a.cache == 0 && a.mready[tile]) {
        cache_load(static_cast<const C*>(a.mom) + 4 * cell, j, inv);
      } else {
        node_base<S, WALLS>(a, g, x, y, z, j, inv);
        if (a.cache != 0) cache_store(slot, j, inv);
      }
      const C cgg[3] = {rv<C>(a.cgg[0]), rv<C>(a.cgg[1]), rv<C>(a.cgg[2])};
      node_velocity<C>(a, cell, tile, j, inv, cgg, nv);
    }
    // every lane forms the whole sum, in node order
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const bool node_in = !WALLS || (b[2] + (q >> 2) >= 0 && b[2] + (q >> 2) < g.nz);
      const C wt = w[0][q & 1] * (w[1][(q >> 1) & 1] * w[2][q >> 2]);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const C u = __shfl_sync(am, nv[c], lead + q);
        if (node_in) own[c] += wt * u;
      }
    }
    } else {
    // lane q: the nodes kx = q of the rows, row by row
    int ys[SN], zs[SN];
#pragma unroll
    for (int q = 0; q < SN; ++q) {
      ys[q] = wrap_int(b[1] + q, g.ny);
      const int zz = b[2] + q;
      zs[q] = WALLS ? ((zz < 0 || zz >= g.nz) ? -1 : zz) : wrap_int(zz, g.nz);
    }
    const int x = wrap_int(b[0] + sub, g.nx);
    const C wx = pick(w[0], sub);
    const C cgg[3] = {rv<C>(a.cgg[0]), rv<C>(a.cgg[1]), rv<C>(a.cgg[2])};
    if (sub < SN) {
      bool done = false;
      if constexpr (PULL) {
        // the rows of a column share no sectors, so each node is a round trip
        // to L2 or DRAM: the populations of PER nodes in flight together
        constexpr int PER = SN == 4 ? 2 : (sizeof(C) == 4 ? SN : 1);
#pragma unroll 1
        for (int kz = 0; kz < SN; ++kz) {
          const int z = pick(zs, kz);
          if (WALLS && z < 0) continue;
          const C wxz = wx * pick(w[2], kz);
#pragma unroll 1
          for (int k0 = 0; k0 < SN; k0 += PER) {
            C j[PER][3], inv[PER];
#pragma unroll
            for (int h = 0; h < PER; ++h)
              node_base<S, WALLS>(a, g, x, pick(ys, k0 + h), z, j[h], inv[h]);
#pragma unroll
            for (int h = 0; h < PER; ++h) {
              const int y = pick(ys, k0 + h);
              node_add<C>(a, z * g.plane + (long long)y * g.pitch + x, tile_of(g, x, y, z),
                          wxz * pick(w[1], k0 + h), j[h], inv[h], cgg, own);
            }
          }
        }
        done = true;
      } else if (a.mom != nullptr && a.F2 == nullptr)
        done = a.F1 != nullptr ? wide_column<SN, true, C>(a, g, x, ys, zs, wx, w, cgg, own)
                               : wide_column<SN, false, C>(a, g, x, ys, zs, wx, w, cgg, own);
      if (!done) {
        own[0] = own[1] = own[2] = C(0);
#pragma unroll 1
        for (int kz = 0; kz < SN; ++kz) {
          const int z = pick(zs, kz);
          if (WALLS && z < 0) continue;
          const C wxz = wx * pick(w[2], kz);
#pragma unroll 1
          for (int ky = 0; ky < SN; ++ky)
            gather_node<S, WALLS>(a, g, x, pick(ys, ky), z, wxz * pick(w[1], ky), cgg, own);
        }
      }
    }
#pragma unroll
    for (int off = 1; off < GL; off <<= 1)
#pragma unroll
      for (int c = 0; c < 3; ++c) own[c] += __shfl_xor_sync(am, own[c], off);
    }
  }
  // ---- the marker's update, one component per lane
  const double s = a.s.d;
  const C oc = pick(own, comp);
  const int nc = pick(n3, comp);
  const bool pc = comp < 2 || !g.walls;
  C frec = C(0);
  double rn = 0.0;
  if (a.mode == GM_COUPLE) {
    C dv[1] = {(C)vc - oc}, Fi[1] = {Fc}, zeta[1] = {C(0)}, Fh[1];
    if (a.noise) {
      C r[4];
      philox_gauss4<C>((uint32_t)i, (uint32_t)(*a.tstep), 8u + (uint32_t)a.substep, 0u, a.tkey0,
                       a.tkey1, r);
      zeta[0] = rv<C>(a.zeta_amp) * pick(r, comp);
    }
    couple_force<C, 1>(a, C(im), dv, Fi, zeta, Fh);
    const double kick = s * im;
    const double vn = vc + kick * (double)(Fh[0] + Fc);
    frec = -rv<C>(a.rec_weight) * Fh[0];
    const double post_ab = sizeof(C) == 4 ? a.post_a + a.post_b : 0.0;
    const double Xc = pick(X, comp);
    if (a.pos_next)
      rn = wrap_axis(sizeof(C) == 4 ? Xc + post_ab * vn : (Xc + a.post_a * vn) + a.post_b * vn, nc, pc);
    // (the group's lanes have read the marker's state: the shuffles above)
    if (sub < 3) {
      a.vel[sub * M + i] = vn;
      if (a.fh_out) static_cast<C*>(a.fh_out)[sub * M + i] = Fh[0];
      if (a.pos_next) a.pos_next[sub * M + i] = rn;
    }
    if (a.pos_next && a.key_out) {
      double r3[3] = {__shfl_sync(am, rn, lead), __shfl_sync(am, rn, lead + 1),
                      __shfl_sync(am, rn, lead + 2)};
      const double v3[3] = {__shfl_sync(am, vn, lead), __shfl_sync(am, vn, lead + 1),
                            __shfl_sync(am, vn, lead + 2)};
      if (sub == 0) next_bin<C>(a, g, i, r3, v3);
    }
  } else if (a.mode == GM_IBM1) {
    frec = rv<C>(a.rec_weight) * Fc;
  } else {
    if (sub < 3) {
      double* out = a.mode == GM_IBM_PREDICT ? a.aux : a.pos;
      out[sub * M + i] = wrap_axis(a.pos[sub * M + i] + s * (double)oc, nc, pc);
    }
    if (a.mode == GM_IBM_HALF) frec = rv<C>(a.rec_weight) * Fc;
  }
  if (a.rec && (a.mode == GM_COUPLE || a.mode == GM_IBM_HALF || a.mode == GM_IBM1)) {
    const C Frec[3] = {__shfl_sync(am, frec, lead), __shfl_sync(am, frec, lead + 1),
                       __shfl_sync(am, frec, lead + 2)};
    if (sub == 0) {
      write_record<ST>(a, g, k, b, w, Frec);
      if (a.keys && !bins_hold<SN>(g, home, b)) *a.status = 1;
    }
    if constexpr (ST == 0) {
    int tq[3][2];
#pragma unroll
    for (int c = 0; c < 3; ++c) axis_tiles<2>(b[c], w[c], n3[c], per[c], tq[c]);
    const int tx = (sub & 1) ? tq[0][1] : tq[0][0], ty = (sub & 2) ? tq[1][1] : tq[1][0],
              tz = (sub & 4) ? tq[2][1] : tq[2][0];
    const int tile = (tz * g.nty + ty) * g.ntx + tx;
    bool first = false;
    if (tx >= 0 && ty >= 0 && tz >= 0) {
      const uint32_t at = atomicAdd(a.hcnt + tile, 1u);
      if (at < (uint32_t)SPREAD_HCAP) a.hits[(size_t)tile * SPREAD_HCAP + at] = (uint32_t)k;
      first = at == 0u;
      if (first) a.mark[tile] = 1u;
    }
    const unsigned m = __ballot_sync(am, first);
    int base = 0;
    if (lane == 0 && m != 0u) base = atomicAdd(a.nlive, __popc(m));
    base = __shfl_sync(am, base, 0);
    if (first) a.live_tiles[base + __popc(m & ((1u << lane) - 1u))] = make_int4(tile, tx, ty, tz);
    } else {
      claim_wide<SN, GL, C>(a, g, b, w, sub, true, am, nact);
    }
  }
}

// resident blocks per SM a variant is compiled for
template <int ST, int VAR, typename C>
constexpr int gather_resident() {
  if ((VAR == GV_GROUP && ST != 0) || VAR == GV_PULL) return 4;    // two planes of loads in registers
  return VAR != GV_FULL && VAR != GV_QUAD && sizeof(C) == 4 ? 6 : 4;
}

template <typename S, bool WALLS, int ST, int VAR>
__global__ void __launch_bounds__(GATHER_THREADS,
                                  gather_resident<ST, VAR, typename Store<S>::C>())
gather_kernel(const PartArgs p, const GatherArgs a) {
  const long long gid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if constexpr (VAR == GV_GROUP || VAR == GV_PULL)
    gather_group_body<S, WALLS, ST, VAR == GV_PULL>(p, a, gid);
  else gather_body<S, WALLS, ST, VAR>(p, a, gid);
}

// ------------------------------------------------------------ node moments
// The field is filled in bricks of 32 x 4 x 4 cells (eight tiles along x):
// a warp covers 32 consecutive cells of one row, as in the LB step.  The
// bricks are listed at each re-binning with the tiles that lie within one
// tile of a tile holding a marker (periodic in x and y, and in z without
// walls): a marker stays within about a cell of its home tile between
// re-binnings and its stencil reaches two cells beyond its own, so the
// gathers find nearly every node in such a tile; a node in a tile that is
// not ready is pulled from the populations instead.
constexpr int MOM_THREADS = 256;


// one thread per tile, eight consecutive lanes per brick (the row of tiles
// is padded to a multiple of eight)
__device__ __forceinline__ void moment_bricks_body(const Geom& g, const int* __restrict__ tb,
                                                   const int* __restrict__ te, const int* need,
                                                   int2* __restrict__ bricks, int* count,
                                                   uint8_t* __restrict__ ready, long long gid) {
  if (skip(need)) return;
  const int nbx = (g.ntx + 7) >> 3;
  const long long row = 8LL * nbx;
  const long long total = row * g.nty * g.ntz;
  int tx = 0, ty = 0, tz = 0;
  bool needed = false;
  if (gid < total) {
    tx = (int)(gid % row);
    const long long r = gid / row;
    ty = (int)(r % g.nty);
    tz = (int)(r / g.nty);
    if (tx < g.ntx) {
      for (int d = 0; d < 27 && !needed; ++d) {
        const int nx = wrap_int(tx + d % 3 - 1, g.ntx);
        const int ny = wrap_int(ty + (d / 3) % 3 - 1, g.nty);
        int nz = tz + d / 9 - 1;
        if (g.walls) {
          if (nz < 0 || nz >= g.ntz) continue;
        } else {
          nz = wrap_int(nz, g.ntz);
        }
        const int n = (nz * g.nty + ny) * g.ntx + nx;
        needed = te[n] > tb[n];
      }
      if (!needed) ready[(tz * g.nty + ty) * g.ntx + tx] = 0;
    }
  }
  const unsigned bal = __ballot_sync(0xffffffffu, needed);
  const int lane = threadIdx.x & 31;
  if (gid < total && (lane & 7) == 0) {
    const int m = (int)((bal >> lane) & 0xFFu);
    if (m) {
      const int e = atomicAdd(count, 1);
      bricks[e] = make_int2((tz * g.nty + ty) * nbx + tx / 8, m);
    }
  }
}

__global__ void moment_bricks_kernel(const Geom g, const int* __restrict__ tb,
                                     const int* __restrict__ te, const int* need,
                                     int2* __restrict__ bricks, int* count,
                                     uint8_t* __restrict__ ready) {
  moment_bricks_body(g, tb, te, need, bricks, count, ready,
                     blockIdx.x * (long long)blockDim.x + threadIdx.x);
}


// persistent: each block takes the listed bricks in turn, two cells per
// thread along z
template <typename S, bool WALLS>
__device__ __forceinline__ void node_moments_body(const PartArgs& __restrict__ p,
                                                  const GatherArgs& __restrict__ a,
                                                  const int2* __restrict__ bricks, const int* count,
                                                  void* mom, uint8_t* __restrict__ ready, int bid,
                                                  int nblk) {
  using C = typename Store<S>::C;
  const Geom& g = p.g;
  const int nb = *count;
  const int nbx = (g.ntx + 7) >> 3;
  const int t = threadIdx.x;
  C* out = static_cast<C*>(mom);
  for (int e = bid; e < nb; e += nblk) {
    const int2 br = bricks[e];
    const int bx = br.x % nbx, ty = (br.x / nbx) % g.nty, tz = br.x / (nbx * g.nty);
    if (t < 8 && ((br.y >> t) & 1)) ready[(tz * g.nty + ty) * g.ntx + bx * 8 + t] = 1;
    const int x = bx * 32 + (t & 31);
    const int y = ty * TILE + ((t >> 5) & 3);
    if (x >= g.nx || y >= g.ny || !((br.y >> ((t & 31) >> TILE_SHIFT)) & 1)) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int z = tz * TILE + 2 * (t >> 7) + h;
      if (z < g.nz) {
        C j[3], inv;
        node_base<S, WALLS>(a, g, x, y, z, j, inv);
        cache_store(out + 4 * (z * g.plane + (long long)y * g.pitch + x), j, inv);
      }
    }
  }
}

template <typename S, bool WALLS>
__global__ void __launch_bounds__(MOM_THREADS)
node_moments_kernel(const PartArgs p, const GatherArgs a, const int2* __restrict__ bricks,
                    const int* count, void* mom, uint8_t* __restrict__ ready) {
  node_moments_body<S, WALLS>(p, a, bricks, count, mom, ready, blockIdx.x, gridDim.x);
}




// ------------------------------------------------------------ spreading
constexpr int MAXNT = 8;    // neighbour tiles per axis in the table


// does the stencil row b .. b + SN - 1 (periodic wrap) meet [lo, hi]?
template <int SN>
__device__ inline bool axis_reach(int b, int n, bool periodic, int lo, int hi) {
  if (!periodic) return b <= hi && b + SN - 1 >= lo;
  const int off = wrap_int(lo - b, n); // position of lo relative to b, mod n
  return off < SN || off + (hi - lo) >= n;
}

// Weights of one stencil row at the TILE cells lo .. lo + TILE - 1 of an
// axis: nodes b + k (periodic wrap, or dropped outside the box) that land on
// the same cell have their weights added in k order.
template <int SN, typename C>
__device__ inline void tile_weights(int b, const C (&w)[4], int n, bool periodic, int lo,
                                    C (&out)[TILE]) {
  int node[SN];
#pragma unroll
  for (int k = 0; k < SN; ++k) {
    int c = b + k;
    if (periodic) c = wrap_int(c, n);
    else if (c < 0 || c >= n) c = -1;
    node[k] = w[k] == C(0) ? -1 : c - lo;
  }
#pragma unroll
  for (int j = 0; j < TILE; ++j) {
    C acc = C(0);
#pragma unroll
    for (int k = 0; k < SN; ++k) acc += node[k] == j ? w[k] : C(0);
    out[j] = acc;
  }
}

// Offset of a stencil base from the tile origin, b - lo, taken as the
// image in [-n/2, n/2) on a periodic axis.  On an axis of n >= 2 TILE cells
// (or a wall-bounded one) node b + k then sits at local cell e + k of the
// tile if 0 <= e + k < TILE, and no two nodes share a cell.
__device__ inline int tile_offset(int b, int lo, int n, bool periodic) {
  int e = b - lo;
  if (periodic) {
    const int h = n >> 1;
    if (e < -h) e += n;
    else if (e >= n - h) e -= n;
  }
  return e;
}

// the same weights as tile_weights for such an axis: out[j] = w[j - e]
template <int SN, typename C>
__device__ inline void tile_weights_shift(int e, const C (&w)[4], C (&out)[TILE]) {
#pragma unroll
  for (int j = 0; j < TILE; ++j) {
    const int q = j - e;
    C v = C(0);
#pragma unroll
    for (int k = 0; k < SN; ++k) v = q == k ? w[k] : v;
    out[j] = v;
  }
}

// a surviving marker reduced to the current tile: the weights at the tile's
// TILE cells of each axis and its force, each component twice (FP32: the
// operand pairs of the packed multiply-adds).  The z weights stand in the
// order 0, 2, 1, 3: a lane owns the cells z, z + 2.
template <typename C>
struct alignas(16) SpreadHit {
  C wx[TILE], wy[TILE], wz[TILE];
  C F[sizeof(C) == 4 ? 8 : 4];
};

__device__ __forceinline__ void put4(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void put4(double* p, double a, double b, double c, double d) {
  reinterpret_cast<double2*>(p)[0] = make_double2(a, b);
  reinterpret_cast<double2*>(p)[1] = make_double2(c, d);
}

// reduces one marker (base b, per-axis weights w, force F) to the tile at lo
template <int SN, typename C>
__device__ __forceinline__ void reduce_hit(SpreadHit<C>& h, const Geom& g, const int (&b)[3],
                                           const C (&w)[3][4], const C (&F)[3], const int (&lo)[3]) {
  const int n3[3] = {g.nx, g.ny, g.nz};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const bool periodic = d < 2 || !g.walls;
    C wt[TILE];
    // (axes on which a stencil meets a tile only by shifting: see tile_offset)
    if (!periodic || n3[d] >= 2 * TILE)
      tile_weights_shift<SN, C>(tile_offset(b[d], lo[d], n3[d], periodic), w[d], wt);
    else
      tile_weights<SN, C>(b[d], w[d], n3[d], periodic, lo[d], wt);
#pragma unroll
    for (int j = 0; j < TILE; ++j) {
      if (d == 0) h.wx[j] = wt[j];
      else if (d == 1) h.wy[j] = wt[j];
      else h.wz[(j & 1) * 2 + (j >> 1)] = wt[j];
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if (sizeof(C) == 4) h.F[2 * c] = h.F[2 * c + 1] = F[c];
    else h.F[c] = F[c];
  }
}

// the same from the record of a slot
template <int ST, typename C>
__device__ __forceinline__ void reduce_record(SpreadHit<C>& h, const Geom& g, const SpreadArgs& a,
                                              int slot, const int (&lo)[3]) {
  C w[3][4], F[3];
  int b[3];
  if constexpr (ST == 0) {
    const TriRecT<C> r = static_cast<const TriRecT<C>*>(a.rec)[slot];
    b[0] = base_x(r.base); b[1] = base_y(r.base); b[2] = base_z(r.base);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      w[d][0] = C(1) - r.t[d]; w[d][1] = r.t[d]; w[d][2] = w[d][3] = C(0);
      F[d] = r.F[d];
    }
  } else {
    const StencilRecT<C>& r = static_cast<const StencilRecT<C>*>(a.rec)[slot];
    b[0] = r.bx; b[1] = r.by; b[2] = r.bz;
#pragma unroll
    for (int q = 0; q < 4; ++q) { w[0][q] = r.wx[q]; w[1][q] = r.wy[q]; w[2][q] = r.wz[q]; }
#pragma unroll
    for (int d = 0; d < 3; ++d) F[d] = r.F[d];
  }
  reduce_hit<nodes_1d<ST>(), C>(h, g, b, w, F, lo);
}

// A lane's force sums at its cells z and z + 2: a[c] += (wx wy wz) F_c.  FP32
// takes both cells with one paired multiply-add (the same rounding as two
// single ones).
template <typename C>
struct TileSum {
  C a[3][2];
  __device__ void zero() {
#pragma unroll
    for (int c = 0; c < 3; ++c) a[c][0] = a[c][1] = C(0);
  }
  __device__ void add(const SpreadHit<C>& h, int cx, int cy, int cz) {
    const C wxy = h.wx[cx] * h.wy[cy];
    if constexpr (sizeof(C) == 4) {
      const float4 f01 = *reinterpret_cast<const float4*>(&h.F[0]);
      const float2 f2 = *reinterpret_cast<const float2*>(&h.F[4]);
      const float2 f[3] = {make_float2(f01.x, f01.y), make_float2(f01.z, f01.w), f2};
      const float2 w = __fmul2_rn(make_float2(wxy, wxy), *reinterpret_cast<const float2*>(&h.wz[2 * cz]));
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float2 r = __ffma2_rn(w, f[c], make_float2(a[c][0], a[c][1]));
        a[c][0] = r.x;
        a[c][1] = r.y;
      }
    } else {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const C w = wxy * h.wz[2 * cz + q];
#pragma unroll
        for (int c = 0; c < 3; ++c) a[c][q] += w * h.F[c];
      }
    }
  }
};

constexpr int SPREAD_THREADS = 256;
constexpr int SPREAD_WARPS = SPREAD_THREADS / 32;
constexpr int SPREAD_ROUNDS = 4;     // candidate rounds of 32 whose loads are in flight together

// One live tile t (index, tx, ty, tz) by a whole warp, its markers found by a
// search of the markers binned in the neighbour tiles.  Lane l owns the cells
// (l & 3, (l >> 2) & 3, l >> 4) and the same cell two planes up, and keeps
// their force sums in registers; 32 candidates are tested at a time, each
// surviving lane reduces its own marker to the tile, and the warp then adds
// the survivors in candidate order, so the sums are formed in a fixed order
// (no atomics).  stage: 32 hits, hk: 32 SPREAD_ROUNDS slots of this warp.
template <int ST, typename C>
__device__ __forceinline__ void spread_search_tile(const Geom& g, const SpreadArgs& a, const int4& t,
                                                   SpreadHit<C>* stage, int* hk) {
  constexpr int SN = nodes_1d<ST>();
  constexpr unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int cxl = lane & 3, cyl = (lane >> 2) & 3, czl = lane >> 4;
  const bool perz = !g.walls;
  C* F = static_cast<C*>(a.F);
  const int lo[3] = {t.y * TILE, t.z * TILE, t.w * TILE};
  const int hi[3] = {min(lo[0] + TILE, g.nx) - 1, min(lo[1] + TILE, g.ny) - 1, min(lo[2] + TILE, g.nz) - 1};
  const int x = lo[0] + cxl, y = lo[1] + cyl, z0 = lo[2] + czl;
  const bool in0 = x <= hi[0] && y <= hi[1] && z0 <= hi[2];
  const bool in1 = x <= hi[0] && y <= hi[1] && z0 + 2 <= hi[2];
  const long long cell0 = z0 * g.plane + (long long)y * g.pitch + x;
  const long long cell1 = cell0 + 2 * g.plane;
  TileSum<C> sum;
  sum.zero();
  if (a.accumulate && a.flag[t.x]) {
    if (in0) load_force(F, cell0, sum.a[0][0], sum.a[1][0], sum.a[2][0]);
    if (in1) load_force(F, cell1, sum.a[0][1], sum.a[1][1], sum.a[2][1]);
  }
  // axes on which a stencil meets a tile only by shifting (see tile_offset)
  const bool shx = g.nx >= 2 * TILE, shy = g.ny >= 2 * TILE, shz = !perz || g.nz >= 2 * TILE;
  // axes of whole tiles: the neighbour tiles are t - 1, t, t + 1 (wrapped,
  // or clipped at walls), the same list the table holds
  const int n3[3] = {g.nx, g.ny, g.nz}, ntv[3] = {g.ntx, g.nty, g.ntz};
  const int tt[3] = {t.y, t.z, t.w};
  // neighbour tiles per axis: lane q holds entry q of the list (from the
  // table on axes of partial or few tiles)
  int rowv[3], nt[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const bool periodic = d < 2 || perz;
    if (n3[d] % TILE == 0 && (!periodic || ntv[d] >= 3)) {
      const int first = periodic ? tt[d] - 1 : max(tt[d] - 1, 0);
      const int last = periodic ? tt[d] + 1 : min(tt[d] + 1, ntv[d] - 1);
      nt[d] = last - first + 1;
      int v = first + lane;
      if (v < 0) v += ntv[d];
      else if (v >= ntv[d]) v -= ntv[d];
      rowv[d] = lane < nt[d] ? v : -1;
    } else {
      const int* row = a.ntab + (d * a.maxnt + tt[d]) * MAXNT;
      rowv[d] = lane < MAXNT ? row[lane] : -1;
      nt[d] = __popc(__ballot_sync(full, rowv[d] >= 0));
    }
  }
  const int ncand = nt[0] * nt[1] * nt[2];
  // candidate markers: the ranges of the neighbour tiles, flattened; 32
  // neighbour tiles per chunk (one load each), then the candidates in
  // groups of SPREAD_ROUNDS x 32: their reach loads are all issued before
  // any is tested, the hits of the group are listed in candidate order in
  // shared memory, and their stencil records are loaded 32 at a time with
  // one load per lane.  The hits are added in candidate order (markers
  // sorted by tile, neighbour tiles in a fixed order), so the sums do not
  // depend on scheduling.
  for (int qbase = 0; qbase < ncand; qbase += 32) {
    const int q = qbase + lane;
    int qx, qy, qz;
    if (nt[0] == 3 && nt[1] == 3) {    // the usual 3 x 3 x 3 neighbourhood
      qx = q % 3; qy = (q / 3) % 3; qz = (q / 9) & (MAXNT - 1);
    } else {
      qx = q % nt[0]; qy = (q / nt[0]) % nt[1]; qz = (q / (nt[0] * nt[1])) & (MAXNT - 1);
    }
    const int tx = __shfl_sync(full, rowv[0], qx);
    const int ty = __shfl_sync(full, rowv[1], qy);
    const int tz = __shfl_sync(full, rowv[2], qz);
    int cnt = 0, kb = 0;
    if (q < ncand) {
      const int tn = (tz * g.nty + ty) * g.ntx + tx;
      kb = a.tile_begin[tn];
      cnt = a.tile_end[tn] - kb;
    }
    int incl = cnt;                    // inclusive prefix of the counts
    for (int off = 1; off < 32; off <<= 1) {
      const int v = __shfl_up_sync(full, incl, off);
      if (lane >= off) incl += v;
    }
    const int total = __shfl_sync(full, incl, 31);
    for (int cbase = 0; cbase < total; cbase += 32 * SPREAD_ROUNDS) {
      int kk[SPREAD_ROUNDS];
      unsigned long long rr[SPREAD_ROUNDS];
#pragma unroll
      for (int r = 0; r < SPREAD_ROUNDS; ++r) {
        kk[r] = -1;
        rr[r] = 0ull;
        if (cbase + 32 * r >= total) continue;     // warp-uniform: no candidates left
        const int cidx = cbase + 32 * r + lane;
        // owning chunk lane: the first lane whose inclusive prefix exceeds cidx
        int pos = 0;
#pragma unroll
        for (int step = 16; step > 0; step >>= 1) {
          const int v = __shfl_sync(full, incl, pos + step - 1);
          if (v <= cidx) pos += step;
        }
        const int ex = __shfl_sync(full, incl - cnt, pos);
        const int kq = __shfl_sync(full, kb, pos);
        kk[r] = cidx < total ? kq + (cidx - ex) : -1;
        if (kk[r] >= 0) {
          if constexpr (ST == 0) rr[r] = static_cast<const TriRecT<C>*>(a.rec)[kk[r]].base;
          else rr[r] = a.reach[kk[r]];
        }
      }
      int nhit = 0;
#pragma unroll
      for (int r = 0; r < SPREAD_ROUNDS; ++r) {
        if (cbase + 32 * r >= total) break;       // warp-uniform
        bool hit = false;
        if (kk[r] >= 0) {
          const int rvx = base_x(rr[r]), rvy = base_y(rr[r]), rvz = base_z(rr[r]);
          const int e0 = tile_offset(rvx, lo[0], g.nx, true);
          const int e1 = tile_offset(rvy, lo[1], g.ny, true);
          const int e2 = tile_offset(rvz, lo[2], g.nz, perz);
          hit = (shx ? e0 <= hi[0] - lo[0] && e0 + SN - 1 >= 0
                     : axis_reach<SN>(rvx, g.nx, true, lo[0], hi[0])) &&
                (shy ? e1 <= hi[1] - lo[1] && e1 + SN - 1 >= 0
                     : axis_reach<SN>(rvy, g.ny, true, lo[1], hi[1])) &&
                (shz ? e2 <= hi[2] - lo[2] && e2 + SN - 1 >= 0
                     : axis_reach<SN>(rvz, g.nz, perz, lo[2], hi[2]));
        }
        const unsigned m = __ballot_sync(full, hit);
        if (hit) hk[nhit + __popc(m & ((1u << lane) - 1u))] = kk[r];
        nhit += __popc(m);
      }
      __syncwarp();
      for (int hb = 0; hb < nhit; hb += 32) {
        const int nh = min(32, nhit - hb);
        if (lane < nh) reduce_record<ST, C>(stage[lane], g, a, hk[hb + lane], lo);
        __syncwarp();
        for (int src = 0; src < nh; ++src) sum.add(stage[src], cxl, cyl, czl);
        __syncwarp();
      }
    }
  }
  if (in0) store_force(F, cell0, sum.a[0][0], sum.a[1][0], sum.a[2][0]);
  if (in1) store_force(F, cell1, sum.a[0][1], sum.a[1][1], sum.a[2][1]);
  if (lane == 0) {
    a.flag[t.x] = 1;
    // the marks are consumed here, or by the pass over all tiles (spread_flags)
    if (a.accumulate) a.mark[t.x] = 0u;
  }
}

// A field that is not added to: the flags of the tiles no stencil reaches are
// cleared, and the marks consumed (a live tile's flag is set by the warp that
// spreads it: only the other flags are written).  Four tiles per thread and
// access (marks and flags start 256-byte aligned), the remainder one by one.
__device__ __forceinline__ void spread_flags(const Geom& g, const SpreadArgs& a, int bid, int nblk) {
  const int ntiles = g.ntx * g.nty * g.ntz;
  const long long gt = (long long)bid * blockDim.x + threadIdx.x;
  const long long nthreads = (long long)nblk * blockDim.x;
  const long long n4 = ntiles / 4;
  uint4* mark4 = reinterpret_cast<uint4*>(a.mark);
  uchar4* flag4 = reinterpret_cast<uchar4*>(a.flag);
  for (long long q = gt; q < n4; q += nthreads) {
    const uint4 m = mark4[q];
    if ((m.x | m.y | m.z | m.w) == 0u) {
      flag4[q] = make_uchar4(0, 0, 0, 0);
    } else {
      mark4[q] = make_uint4(0u, 0u, 0u, 0u);
      uint8_t* f = a.flag + 4 * q;
      if (!m.x) f[0] = 0;
      if (!m.y) f[1] = 0;
      if (!m.z) f[2] = 0;
      if (!m.w) f[3] = 0;
    }
  }
  for (long long t = 4 * n4 + gt; t < ntiles; t += nthreads) {
    if (a.mark[t] != 0u) a.mark[t] = 0u;
    else a.flag[t] = 0;
  }
}

// Trilinear spreading from the hit lists, one warp per live tile.  Lane l owns
// the cells (l & 3, (l >> 2) & 3, l >> 4) and the same cell two planes up and
// adds the tile's markers in slot order (no atomics).  A tile is a chain of
// four dependent loads (list entry, hits, records, the field it adds to), so
// the chain is pipelined over the warp's tiles: while tile j is summed, the
// records of its next tile, the hits of the one after and the list entry of
// the third are in flight.  The markers are ordered by counting the smaller
// slots (independent shuffles) instead of a sort, and their records are 32
// bytes.  Axes of a single tile (where both nodes of a stencil can meet the
// tile apart) and lists that overflowed take the search.  Bound by issue and
// latency together (11.3 million warp instructions, 0.5 per scheduler and
// cycle at 24 warps per SM):
// 100 000 beads in 256^3 (34 000 live tiles) 34 -> 29 us per launch, 12 500
// beads in 128^3 14.3 -> 10.6 us; half a warp per tile, four cells per lane,
// took 40 us (more instructions per tile, not fewer: both halves wait for the
// longer list), and a tile order that spreads a cluster over the SMs 30 us.
template <typename C>
__device__ __forceinline__ void spread_list_body(const PartArgs& __restrict__ p,
                                                 const SpreadArgs& __restrict__ a, int bid, int nblk) {
  constexpr unsigned full = 0xffffffffu;
  static_assert(SPREAD_HCAP == 32, "one list entry per lane");
  __shared__ SpreadHit<C> shit[SPREAD_WARPS][SPREAD_HCAP];
  __shared__ int shk[SPREAD_WARPS][32 * SPREAD_ROUNDS];
  const Geom& g = p.g;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  SpreadHit<C>* stage = shit[wid];
  const TriRecT<C>* recs = static_cast<const TriRecT<C>*>(a.rec);
  C* F = static_cast<C*>(a.F);
  const int ntiles = g.ntx * g.nty * g.ntz;
  const int cx = lane & 3, cy = (lane >> 2) & 3, cz = lane >> 4;
  const int stride = nblk * SPREAD_WARPS;
  const int j0 = bid * SPREAD_WARPS + wid;
  // (the list has room for every tile: entries are loaded ahead of the count)
  auto entry = [&](int q) { return q < ntiles ? a.live_tiles[q] : make_int4(0, 0, 0, 0); };
  int4 lt = entry(j0), lt1 = entry(j0 + stride), lt2 = entry(j0 + 2 * stride);
  const int nlive = *a.nlive;
  if (bid == 0 && threadIdx.x == 0) *a.nlive_next = 0;    // the next gather's counter (idle now)
  const bool lists = g.ntx > 1 && g.nty > 1 && (g.walls || g.ntz > 1);
  // length of a tile's list (beyond SPREAD_HCAP: the tile takes the search),
  // the lane's entry, and whether the tile's field values are added to
  auto count_of = [&](int q, const int4& t) { return q < nlive ? (int)a.hcnt[t.x] : 0; };
  auto key_of_lane = [&](int q, const int4& t) {      // (entries past the count are not tiles)
    return q < nlive ? a.hits[(size_t)t.x * SPREAD_HCAP + lane] : 0u;
  };
  auto rec_of = [&](int count, uint32_t key) {
    TriRecT<C> r;
    r.base = 0ull;
#pragma unroll
    for (int d = 0; d < 3; ++d) r.t[d] = r.F[d] = C(0);
    if (lane < count && count <= SPREAD_HCAP) r = recs[key];
    return r;
  };
  auto carry_of = [&](int q, const int4& t) { return q < nlive && a.accumulate && a.flag[t.x] != 0; };
  bool overflow = false;
  if (lists) {
    int hc = count_of(j0, lt), hc1 = count_of(j0 + stride, lt1);
    uint32_t key = key_of_lane(j0, lt), key1 = key_of_lane(j0 + stride, lt1);
    bool carry = carry_of(j0, lt), carry1 = carry_of(j0 + stride, lt1);
    TriRecT<C> rec = rec_of(hc, key);
    for (int j = j0; j < nlive; j += stride) {
      const int lo[3] = {lt.y * TILE, lt.z * TILE, lt.w * TILE};
      const bool in0 = lo[0] + cx < g.nx && lo[1] + cy < g.ny && lo[2] + cz < g.nz;
      const bool in1 = in0 && lo[2] + cz + 2 < g.nz;
      const long long cell = (lo[2] + cz) * g.plane + (long long)(lo[1] + cy) * g.pitch + lo[0] + cx;
      // the tile's field values, needed after its markers are staged, and
      // the loads of the warp's next tiles
      TileSum<C> sum;
      sum.zero();
      if (carry) {
        if (in0) load_force(F, cell, sum.a[0][0], sum.a[1][0], sum.a[2][0]);
        if (in1) load_force(F, cell + 2 * g.plane, sum.a[0][1], sum.a[1][1], sum.a[2][1]);
      }
      const TriRecT<C> rec1 = rec_of(hc1, key1);
      const int hc2 = count_of(j + 2 * stride, lt2);
      const uint32_t key2 = key_of_lane(j + 2 * stride, lt2);
      const bool carry2 = carry_of(j + 2 * stride, lt2);
      const int4 lt3 = entry(j + 3 * stride);
      if (hc <= SPREAD_HCAP) {
        // the marker's place: the number of smaller slots in the list
        int rank = 0;
#pragma unroll 4
        for (int q = 0; q < hc; ++q) rank += __shfl_sync(full, key, q) < key ? 1 : 0;
        if (lane < hc) {
          SpreadHit<C>& h = stage[rank];
          // the lower node's cell in the tile: 0 .. 3, or else the node lies
          // one cell before the tile (a marker of the list reaches it)
          const uint32_t b0 = (uint32_t)rec.base, b1 = (uint32_t)(rec.base >> 32);
          const int b[3] = {(int)(b0 & 0x1FFFFFu), (int)(__funnelshift_r(b0, b1, 22) & 0x1FFFFFu),
                            (int)b1 >> 11};
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const int off = b[d] - lo[d];
            const int e = (unsigned)off < (unsigned)TILE ? off : -1;
            const C t0 = C(1) - rec.t[d], t1 = rec.t[d];
            C w[TILE];
#pragma unroll
            for (int q = 0; q < TILE; ++q) w[q] = e == q ? t0 : (e == q - 1 ? t1 : C(0));
            if (d == 0) put4(h.wx, w[0], w[1], w[2], w[3]);
            else if (d == 1) put4(h.wy, w[0], w[1], w[2], w[3]);
            else put4(h.wz, w[0], w[2], w[1], w[3]);
          }
          if constexpr (sizeof(C) == 4) {
            put4(h.F, rec.F[0], rec.F[0], rec.F[1], rec.F[1]);
            h.F[4] = rec.F[2];
            h.F[5] = rec.F[2];
          } else {
            put4(h.F, rec.F[0], rec.F[1], rec.F[2], C(0));
          }
        }
        __syncwarp();
        for (int q = 0; q < hc; ++q) sum.add(stage[q], cx, cy, cz);
        if (in0) store_force(F, cell, sum.a[0][0], sum.a[1][0], sum.a[2][0]);
        if (in1) store_force(F, cell + 2 * g.plane, sum.a[0][1], sum.a[1][1], sum.a[2][1]);
        if (lane == 0) {
          a.flag[lt.x] = 1;
          a.hcnt[lt.x] = 0u;                       // empty for the next gather
          // the marks are consumed here, or by the pass over all tiles below
          if (a.accumulate) a.mark[lt.x] = 0u;
        }
        __syncwarp();
      } else {
        overflow = true;
      }
      lt = lt1; lt1 = lt2; lt2 = lt3;
      hc = hc1; hc1 = hc2;
      key = key1; key1 = key2;
      carry = carry1; carry1 = carry2;
      rec = rec1;
    }
  }
  // the tiles that take the search, in a loop of their own (its registers do
  // not add to the list path's)
  if (overflow || !lists)
    for (int j = j0; j < nlive; j += stride) {
      const int4 t = entry(j);
      if (lists && a.hcnt[t.x] <= (uint32_t)SPREAD_HCAP) continue;
      __syncwarp();
      if (lane == 0) a.hcnt[t.x] = 0u;
      spread_search_tile<0, C>(g, a, t, stage, shk[wid]);
    }
  if (!a.accumulate) spread_flags(g, a, bid, nblk);
}

// Spreading over the live tiles of one box (block bid of its nblk blocks),
// taken from the list the gather built, a warp each: trilinear tiles from their
// hit lists, the others by the search.
template <int ST, typename C>
__device__ __forceinline__ void spread_body(const PartArgs& __restrict__ p,
                                            const SpreadArgs& __restrict__ a, int bid, int nblk) {
  static_assert(TILE == 4 && TILE_CELLS == 64, "cells per lane");
  if constexpr (ST == 0) {
    spread_list_body<C>(p, a, bid, nblk);
  } else {
    __shared__ SpreadHit<C> shit[SPREAD_WARPS][32];
    __shared__ int shk[SPREAD_WARPS][32 * SPREAD_ROUNDS];   // hits of a candidate group, in order
    const Geom& g = p.g;
    const int wid = threadIdx.x >> 5;
    const int ntiles = g.ntx * g.nty * g.ntz;
    const int stride = nblk * SPREAD_WARPS;
    int j = bid * SPREAD_WARPS + wid;
    auto entry = [&](int q) { return q < ntiles ? a.live_tiles[q] : make_int4(0, 0, 0, 0); };
    int4 lt = entry(j);
    const int nlive = *a.nlive;
    if (bid == 0 && threadIdx.x == 0) *a.nlive_next = 0;    // the next gather's counter (idle now)
    for (; j < nlive; j += stride) {
      const int4 lt1 = entry(j + stride);
      spread_search_tile<ST, C>(g, a, lt, shit[wid], shk[wid]);
      lt = lt1;
    }
    if (!a.accumulate) spread_flags(g, a, bid, nblk);
  }
}

// resident blocks per SM the spreading is compiled for: 80 registers without
// spills.  At four blocks (64 registers) the spilled values cost more than the
// warps gain: bead chains 256^3 888 against 892 us per step, 12 500 beads in
// 128^3 285 against 298 us, rigid spheres (four-point) 584 against 606 us.
constexpr int SPREAD_RESIDENT = 3;

template <int ST, typename C>
__global__ void __launch_bounds__(SPREAD_THREADS, SPREAD_RESIDENT)
spread_kernel(const PartArgs p, const SpreadArgs a) {
  spread_body<ST, C>(p, a, blockIdx.x, gridDim.x);
}




// ------------------------------------------------------------ particle momentum
__global__ void __launch_bounds__(256)
particle_momentum_kernel(long long M, const double* __restrict__ vel, const double* __restrict__ mass,
                         double* out3) {
  double acc[3] = {0, 0, 0};
  for (long long i = threadIdx.x; i < M; i += blockDim.x)
    for (int c = 0; c < 3; ++c) acc[c] += mass[i] * vel[c * M + i];
  __shared__ double sh[3][256];
  for (int c = 0; c < 3; ++c) sh[c][threadIdx.x] = acc[c];
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
      for (int c = 0; c < 3; ++c) sh[c][threadIdx.x] += sh[c][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int c = 0; c < 3; ++c) out3[c] = sh[c][0];
}



}  // namespace
}  // namespace lbc
