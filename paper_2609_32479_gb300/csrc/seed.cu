// Analytic seed of Sec. 3.1 on the GPU, in fp64: per track the helix through
// three hits (conformal map), its perigee, and per hit the three residual
// features against that helix (asinh du, asinh dv in the curvilinear frame,
// path length s); plus the decode of the heads' corrections against the seed
// (Sec. 3.3).  A thread fits a track's seed, then the threads of a CTA share the
// hits of its tracks.  Bound by the fp64 pipe (524,288 tracks with the features:
// 7.20 ms with a thread for all of a track's hits and a sine and cosine a Newton
// step, 2.65 ms with rotations and starts from fp32).
//
// Conventions (those of the synthetic track generator): B along +z; a positive
// charge turns clockwise seen from +z; at turning angle a from the perigee the
// direction angle is phi0 - q a, the transverse arc length R a and
// z = z0 + R a cot(theta); the perigee point is (-d0 sin phi0, d0 cos phi0);
// p_T = 0.299792458 B R / 1000 GeV (R in mm, B in T); q/p = q sin(theta) / p_T.
#include <math.h>

#include "trackfit_internal.h"

namespace {

constexpr double C_LIGHT = 0.299792458;
constexpr double TWO_PI = 6.283185307179586476925286766559;
constexpr double PI = 3.1415926535897932384626433832795;
constexpr double QOP_FLOOR = 0.02;   // 1/GeV: floor of the scale-free q/p residual (Sec. 3.3)
constexpr int NEWTON_MAX = 60;
constexpr double PITCH_MIN_MM = 1.0;   // below this pitch z does not choose the helix turn of a hit

// x mod 2 pi in [0, 2 pi)
__device__ __forceinline__ double mod2pi(double x) {
  double r = fmod(x, TWO_PI);
  return r < 0.0 ? r + TWO_PI : r;
}

// fp32 to fp64 and (by truncation) back, for values that are normal in both, on the
// integer pipe: a conversion instruction would take the fp64 pipe, which bounds this
// file (two operations a cycle and SM).
__device__ __forceinline__ double widen(float f) {
  const uint32_t u = __float_as_uint(f);
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
}
__device__ __forceinline__ float narrow(double v) {
  const uint32_t hi = (uint32_t)__double2hiint(v);
  const uint32_t m = __funnelshift_l((uint32_t)__double2loint(v), (hi & 0x7fffffffu) - (896u << 20), 3);
  return __uint_as_float((hi & 0x80000000u) | m);
}
// |v| in (2^-100, 2^100): where the fp32 functions below give normal results
__device__ __forceinline__ bool mid_range(double v) {
  const uint32_t e = ((uint32_t)__double2hiint(v) >> 20) & 0x7ffu;
  return e - 923u < 200u;
}

// 1 / sqrt(v) and 1 / v by STEPS steps of Newton's iteration from the fp32 function of
// the truncated value (relative error below 5e-7; one step leaves below 4e-13, two
// the fp64 rounding); outside mid_range the library's.
template <int STEPS>
__device__ __forceinline__ double rsqrt_n(double v) {
  if (!mid_range(v) || v < 0.0) return rsqrt(v);
  double y = widen(rsqrtf(narrow(v)));
#pragma unroll
  for (int i = 0; i < STEPS; ++i) y = fma(0.5 * y, fma(-v * y, y, 1.0), y);
  return y;
}
template <int STEPS>
__device__ __forceinline__ double rcp_n(double v) {
  if (!mid_range(v)) return 1.0 / v;
  double y = widen(__fdividef(1.0f, narrow(v)));
#pragma unroll
  for (int i = 0; i < STEPS; ++i) y = fma(y, fma(-v, y, 1.0), y);
  return y;
}

// asinh(x) = sign(x) log(1 + t), t = |x| + x^2 / (1 + sqrt(1 + x^2)), with
// log(1 + t) = e log 2 + 2 atanh(r), r = (m - 1) / (m + 1) for 1 + t = m 2^e with
// m in [1/sqrt 2, sqrt 2] (r = t / (2 + t) for small t, without forming 1 + t).
// |r| < 0.172, so the series of atanh to r^13 leaves 1.3e-12 relative at most, the
// reciprocals 4e-13 each: 3e-5 of the fp32 rounding of the feature.
__device__ __forceinline__ double asinh_n(double x) {
  const double ax = fabs(x);
  if (!(ax < 1e9)) return asinh(x);
  const double xx = x * x, w = 1.0 + xx;
  const double t = fma(xx, rcp_n<1>(fma(w, rsqrt_n<1>(w), 1.0)), ax);
  double num = t, den = 2.0 + t, e = 0.0;
  if (t > 0.4) {
    const double u = 1.0 + t;
    int hi = __double2hiint(u), k = (hi >> 20) - 1023;   // u = m 2^k, m in [1, 2)
    hi -= k << 20;
    if (hi >= 0x3ff6a09e) {   // m >= sqrt 2
      hi -= 1 << 20;
      ++k;
    }
    const double m = __hiloint2double(hi, __double2loint(u));
    num = m - 1.0;
    den = m + 1.0;
    e = (double)k * 0.69314718055994530942;
  }
  const double r = num * rcp_n<1>(den), z = r * r;
  double s = 1.0 / 13.0;
  s = fma(s, z, 1.0 / 11.0);
  s = fma(s, z, 1.0 / 9.0);
  s = fma(s, z, 1.0 / 7.0);
  s = fma(s, z, 1.0 / 5.0);
  s = fma(s, z, 1.0 / 3.0);
  return copysign(fma(2.0, fma(r * z, s, r), e), x);
}

// The angle of the vector (c, s) of length len, in [-pi, pi]: twice the angle whose
// tangent is s / (len + c), by the series of atan up to 0.33 (an angle of 0.64; the
// term left out is below 1e-17), beyond that the library.
__device__ __forceinline__ double angle_of(double s, double c, double len) {
  const double t = s * rcp_n<2>(len + c), z = t * t;
  if (!(z < 0.109) || !(len + c > 0.0)) return atan2(s, c);
  double p = 1.0 / 33.0;
#pragma unroll
  for (int k = 31; k >= 3; k -= 2) p = fma(-p, z, 1.0 / (double)k);
  return 2.0 * fma(-p * z, t, t);
}

// sin and cos of a small step: the Taylor series for |d| <= 0.02 (next term 1e-20),
// else the library.
__device__ __forceinline__ void sincos_step(double d, double& s, double& c) {
  const double z = d * d;
  if (z > 4e-4) {
    sincos(d, &s, &c);
    return;
  }
  s = d * fma(z, fma(z, fma(z, -1.0 / 5040.0, 1.0 / 120.0), -1.0 / 6.0), 1.0);
  c = fma(z, fma(z, fma(z, fma(z, 1.0 / 40320.0, -1.0 / 720.0), 1.0 / 24.0), -0.5), 1.0);
}

// The helix of a seed: charge, radius, centre, the unit vector from the centre to
// the perigee, z at the perigee, and what the foot points need of theta.
struct Helix {
  double q, R, cx, cy, ux, uy, z0, st, ct, rcot, inv_rcot, r_st;
  int turns;   // whether z chooses the helix turn of a hit
};

// Perigee of the helix through three hits in path order (Sec. 3.1: the circle
// from the conformal map, whose image of a circle through the first hit is a
// straight line fixed by the images of the other two).  An arc from the perigee to
// a hit is the angle between two vectors from the centre.
__device__ void perigee_from_triplet(const double (&a)[3], const double (&b)[3], const double (&c)[3],
                                     double b_field, double (&pg)[5], Helix& h) {
  const double ax = b[0] - a[0], ay = b[1] - a[1];
  const double bx = c[0] - a[0], by = c[1] - a[1];
  const double na = ax * ax + ay * ay, nb = bx * bx + by * by;
  const double u1 = ax / na, v1 = ay / na, u2 = bx / nb, v2 = by / nb;
  const double det = u1 * v2 - u2 * v1;
  const double ccx = (v2 - v1) / (2.0 * det), ccy = (u1 - u2) / (2.0 * det);
  const double Cx = a[0] + ccx, Cy = a[1] + ccy;
  const double R = sqrt(ccx * ccx + ccy * ccy);
  const double cross = ax * by - ay * bx;
  const double q = cross > 0.0 ? -1.0 : (cross < 0.0 ? 1.0 : 0.0);
  const double dc = sqrt(Cx * Cx + Cy * Cy);
  const double ux = Cx / dc, uy = Cy / dc;
  const double px = Cx - R * ux, py = Cy - R * uy;     // circle point closest to the beam line
  const double cp = -q * uy, sp = q * ux;              // direction of motion there: (cos phi0, sin phi0)
  // turning angle from the perigee (at -u from the centre) to a point v of the circle
  auto arc = [&](double vx, double vy) {
    const double t = -q * angle_of(uy * vx - ux * vy, -(ux * vx + uy * vy), R);
    return R * (t < 0.0 ? t + TWO_PI : t);
  };
  const double s0 = arc(a[0] - Cx, a[1] - Cy), s2 = arc(c[0] - Cx, c[1] - Cy);
  const double cot = (c[2] - a[2]) / (s2 - s0);
  const double st = 1.0 / sqrt(1.0 + cot * cot);
  const double pt = C_LIGHT * b_field * R / 1000.0;
  pg[0] = -px * sp + py * cp;
  pg[1] = a[2] - s0 * cot;
  pg[2] = atan2(sp, cp);
  pg[3] = atan2(1.0, cot);
  pg[4] = q * st / pt;
  h.q = q;
  h.R = R;
  h.cx = Cx;
  h.cy = Cy;
  h.ux = -ux;
  h.uy = -uy;
  h.z0 = pg[1];
  h.st = st;
  h.ct = cot * st;
  h.rcot = R * cot;
  h.inv_rcot = 1.0 / h.rcot;
  h.r_st = R / st;
  h.turns = 2.0 * PI * fabs(h.rcot) > PITCH_MIN_MM;
}

// (du, dv, s) of a hit against the helix: the foot point is the helix point whose
// normal plane holds the hit, found by Newton's method on g(a) = (hit - p(a)) . t(a).
// The start is the hit's transverse angle around the centre counted from the
// perigee into [-pi, pi] (continuous across the perigee), moved by the whole
// turns that bring it closest to the angle of the hit's z, (z - z0) / (R cot theta),
// where the pitch 2 pi R |cot theta| exceeds PITCH_MIN_MM.  du, dv are the hit's
// coordinates along U = z x t / |z x t| and V = t x U at the foot point,
// s = R a / sin(theta) (negative behind the perigee).
//
// The fp64 pipe bounds this.  So the angle is evaluated once: the sine and cosine of
// the direction at the start are the hit's own unit vector from the centre, and each
// step turns them by the small angle of the step.  With w the distance of the hit from the
// foot point along the transverse direction, g'' is sin^2(theta) w and g''' at most about
// R / sin(theta), so after a step d the angle is off by less than d^2 (w + d R / sin(theta)) /
// 2 |g'|: a step that leaves 1e-14 is the last.  (With a step of 1e-5 as the last s was up to
// 5e-9 off for hits 100 mm beside the helix, 2e-8 at 1 m, near fp32's rounding.)
__device__ __forceinline__ void residuals(const Helix& h, double x, double y, double z, double& du, double& dv,
                                          double& s) {
  double hx = x - h.cx, hy = y - h.cy;
  const double hh = hx * hx + hy * hy;
  if (hh == 0.0) {
    hx = h.ux;
    hy = h.uy;
  }
  const double inv = hh == 0.0 ? 1.0 : rsqrt_n<2>(hh);
  double a = -h.q * angle_of(h.ux * hy - h.uy * hx, h.ux * hx + h.uy * hy, hh == 0.0 ? 1.0 : hh * inv);
  if (h.turns) a += TWO_PI * floor(((z - h.z0) * h.inv_rcot - a) * (1.0 / TWO_PI) + 0.5);
  double sphi = -h.q * hx * inv, cphi = h.q * hy * inv;   // p = c + R (-q sin phi, q cos phi)
  const double qR = h.q * h.R, qst = h.q * h.st;
  double rx, ry, rz;
  for (int it = 0;; ++it) {
    rx = x - (h.cx - qR * sphi);
    ry = y - (h.cy + qR * cphi);
    rz = z - fma(h.rcot, a, h.z0);
    if (it == NEWTON_MAX) break;
    const double w = rx * cphi + ry * sphi, g = h.st * w + h.ct * rz;
    // dp/da = (R / sin theta) t;  dt/da = q sin(theta) (sin phi, -cos phi, 0)
    const double dg = qst * (rx * sphi - ry * cphi) - h.r_st, d = -g * rcp_n<1>(dg);
    a += d;
    double sd, cd;
    sincos_step(-h.q * d, sd, cd);   // phi = phi0 - q a
    const double s1 = sphi * cd + cphi * sd;
    cphi = cphi * cd - sphi * sd;
    sphi = s1;
    // one more pass for the residual, then out
    if (d * d * fma(fabs(d), h.r_st, fabs(w)) <= 2e-14 * fabs(dg)) it = NEWTON_MAX - 1;
  }
  // U = (-sin phi, cos phi, 0); V = t x U = (-cos theta cos phi, -cos theta sin phi, sin theta)
  du = ry * cphi - rx * sphi;
  dv = h.st * rz - h.ct * (rx * cphi + ry * sphi);
  s = h.r_st * a;
}

// A CTA takes SEED_TRK tracks: one warp fits the seeds, then all warps take the
// hits of these tracks back to back (only valid hits, so no lane idles on a shorter
// track).
constexpr int SEED_TRK = 32, SEED_NT = 128;

__global__ void __launch_bounds__(SEED_NT) seed_kernel(const float* __restrict__ hits, int hs,
                                                       const int32_t* __restrict__ n_hits, int64_t B, int T,
                                                       double b_field, double min_sep, double* __restrict__ seed,
                                                       float* __restrict__ feats, int fs) {
  __shared__ Helix hel[SEED_TRK];
  __shared__ int cnt[SEED_TRK], end[SEED_TRK];   // hits with features, and their running sum
  const int64_t b0 = blockIdx.x * (int64_t)SEED_TRK;
  const int tid = threadIdx.x;
  if (tid < SEED_TRK) {
    const int64_t b = b0 + tid;
    int m = 0;
    if (b < B) {
      int n = n_hits[b];
      if (n < 0 || n > T) n = 0;   // not a track: no seed
      const float* hb = hits + (size_t)b * T * hs;   // hit t of this track at hb[t * hs]
      // the seed triplet: the first hit, then each first later hit more than min_sep
      // (3-D) from the previous seed hit
      double p3[3][3];
      int np = 0;
      for (int t = 0; t < n && np < 3; ++t) {
        const double p[3] = {(double)hb[t * hs + 0], (double)hb[t * hs + 1], (double)hb[t * hs + 2]};
        bool take = np == 0;
        if (!take) {
          const double(&l)[3] = np == 1 ? p3[0] : p3[1];
          const double dx = p[0] - l[0], dy = p[1] - l[1], dz = p[2] - l[2];
          take = sqrt(dx * dx + dy * dy + dz * dz) > min_sep;
        }
        if (take) {
#pragma unroll
          for (int k = 0; k < 3; ++k)
            if (np == k) {
              p3[k][0] = p[0];
              p3[k][1] = p[1];
              p3[k][2] = p[2];
            }
          ++np;
        }
      }
      double pg[5];
      bool finite = np == 3;
      if (finite) {
        perigee_from_triplet(p3[0], p3[1], p3[2], b_field, pg, hel[tid]);
        for (int k = 0; k < 5; ++k) finite = finite && isfinite(pg[k]);
      } else {
        for (int k = 0; k < 5; ++k) pg[k] = __longlong_as_double(0x7ff8000000000000ll);
      }
      for (int k = 0; k < 5; ++k) seed[b * 5 + k] = pg[k];
      m = finite ? n : 0;
    }
    int e = m;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, e, o);
      if (tid >= o) e += u;
    }
    cnt[tid] = m;
    end[tid] = e;
  }
  if (!feats) return;
  __syncthreads();
  float* fb = feats + (size_t)b0 * T * fs;
  const float* hb = hits + (size_t)b0 * T * hs;
  for (int i = tid; i < end[SEED_TRK - 1]; i += SEED_NT) {
    int k = 0;   // the track that holds hit i
#pragma unroll
    for (int o = SEED_TRK / 2; o > 0; o >>= 1)
      if (end[k + o - 1] <= i) k += o;
    const int row = k * T + i - (end[k] - cnt[k]);
    const float* p = hb + (size_t)row * hs;
    double du, dv, s;
    residuals(hel[k], (double)p[0], (double)p[1], (double)p[2], du, dv, s);
    float* o = fb + (size_t)row * fs;
    o[0] = (float)asinh_n(du);
    o[1] = (float)asinh_n(dv);
    o[2] = (float)s;
  }
  // padding rows, and tracks without a seed
  const int nt = (int)(B - b0 < SEED_TRK ? B - b0 : SEED_TRK);
  for (int i = tid; i < nt * T; i += SEED_NT) {
    const int k = i / T, t = i - k * T;
    if (t < cnt[k]) continue;
    float* o = fb + (size_t)i * fs;
    o[0] = o[1] = o[2] = 0.0f;
  }
}

// out = seed + correction, phi wrapped to (-pi, pi]; q/p from the scale-free
// residual: q/p = q/p_seed + r (|q/p_seed| + 0.02 / GeV)  (Sec. 3.3).
__global__ void decode_kernel(const double* __restrict__ seed, const float* __restrict__ corr, int64_t B,
                              float* __restrict__ out) {
  const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (b >= B) return;
  double v[5];
  for (int k = 0; k < 5; ++k) v[k] = seed[b * 5 + k] + (double)corr[b * 5 + k];
  v[2] = PI - mod2pi(PI - v[2]);
  v[4] = seed[b * 5 + 4] + (double)corr[b * 5 + 4] * (fabs(seed[b * 5 + 4]) + QOP_FLOOR);
  for (int k = 0; k < 5; ++k) out[b * 5 + k] = (float)v[k];
}

}  // namespace

extern "C" int trackfit_seed(const float* hits, int32_t hit_stride, const int32_t* n_hits, int64_t n_tracks,
                             int32_t max_hits, double b_field, double* seed_out, float* features_out,
                             int32_t feat_stride, void* stream) {
  tf_nvtx_range nvtx_range("trackfit_seed");
  if (!hits || !n_hits || !seed_out || n_tracks <= 0 || max_hits < 1 || max_hits > TF_MAX_HITS) {
    return TRACKFIT_ERR_INVALID_ARG;
  }
  if (hit_stride < 3 || (features_out && feat_stride < 3)) return TRACKFIT_ERR_INVALID_ARG;
  if (!(b_field > 0.0) || !isfinite(b_field)) return TRACKFIT_ERR_INVALID_ARG;
  const uintptr_t mis = reinterpret_cast<uintptr_t>(hits) | reinterpret_cast<uintptr_t>(seed_out) |
                        reinterpret_cast<uintptr_t>(n_hits) | reinterpret_cast<uintptr_t>(features_out);
  if (mis & 15u) return TRACKFIT_ERR_INVALID_ARG;
  const unsigned grid = (unsigned)((n_tracks + SEED_TRK - 1) / SEED_TRK);
  seed_kernel<<<grid, SEED_NT, 0, reinterpret_cast<cudaStream_t>(stream)>>>(hits, hit_stride, n_hits, n_tracks, max_hits,
                                                                        b_field, 10.0, seed_out, features_out,
                                                                        feat_stride);
  return cudaPeekAtLastError() == cudaSuccess ? TRACKFIT_OK : TRACKFIT_ERR_CUDA;
}

extern "C" int trackfit_decode(const double* seed, const float* corrections, int64_t n_tracks, float* out_params,
                               void* stream) {
  tf_nvtx_range nvtx_range("trackfit_decode");
  if (!seed || !corrections || !out_params || n_tracks <= 0) return TRACKFIT_ERR_INVALID_ARG;
  const uintptr_t mis = reinterpret_cast<uintptr_t>(seed) | reinterpret_cast<uintptr_t>(corrections) |
                        reinterpret_cast<uintptr_t>(out_params);
  if (mis & 15u) return TRACKFIT_ERR_INVALID_ARG;
  const unsigned grid = (unsigned)((n_tracks + 255) / 256);
  decode_kernel<<<grid, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(seed, corrections, n_tracks, out_params);
  return cudaPeekAtLastError() == cudaSuccess ? TRACKFIT_OK : TRACKFIT_ERR_CUDA;
}
