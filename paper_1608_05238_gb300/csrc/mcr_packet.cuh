// mcr_packet.cuh -- what every 2D transport kernel does to start and to turn a packet, shared so
// that the direct and the record transport follow identical paths.
#pragma once

#include "mcr_internal.h"
#include "mcr_rng.cuh"

namespace mcr {
constexpr unsigned kFull = 0xFFFFFFFFu;

// Volumetric source: smallest i with cdf[i] > floor(r48 * total / 2^48).
__device__ __forceinline__ int pick_pixel(const unsigned long long *__restrict__ cdf, int npix,
                                          unsigned long long total, unsigned w0, unsigned w1) {
  const unsigned long long r48 = ((unsigned long long)w0 << 16) | (unsigned long long)(w1 >> 16);
  const unsigned long long target = __umul64hi(r48 << 16, total);
  int lo = 0, hi = npix - 1;
  while (lo < hi) {
    const int mid = lo + ((hi - lo) >> 1);
    if (__ldg(cdf + mid) > target)
      hi = mid;
    else
      lo = mid + 1;
  }
  return lo;
}

__device__ __forceinline__ float clamp_dx(float v, float dx) { return fminf(fmaxf(v, 0.f), dx); }

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// Launch angle (from +z) of an MCR_ANGULAR_POINT source: the theta in [0, 2 pi) at which the
// integral of its density from 0,
//   F(theta) = (theta + sum_n [c_n sin n theta + s_n (1 - cos n theta)] / n) / (2 pi),
// reaches u; 24 bisection steps resolve theta to the FP32 spacing of [0, 2 pi).  Runs once per
// packet, at launch.
__device__ __forceinline__ float launch_angle(const ProblemDesc &P, float u) {
  const float two_pi = 6.28318530717958648f;
  float lo = 0.f, hi = two_pi;
  const float target = u * two_pi;
  for (int it = 0; it < 24; ++it) {
    const float mid = 0.5f * (lo + hi);
    float F = mid;
    for (int n = 1; n <= P.n_ang; ++n) {
      float sn, cn;
      sincosf(n * mid, &sn, &cn);
      F += (P.ang_c[n - 1] * sn + P.ang_s[n - 1] * (1.f - cn)) / n;
    }
    if (F < target)
      lo = mid;
    else
      hi = mid;
  }
  return 0.5f * (lo + hi);
}

// Launch position, direction and weight of packet `pid` of problem P (nx, nz, dx, key0, key1: its
// fields).  Returns whether the packet starts inside the grid; W0 is +-1, or 0 (and false) for an
// all-zero volumetric source.
__device__ __forceinline__ bool launch_packet(const ProblemDesc &P, unsigned long long pid, int nx, int nz, float dx,
                                              unsigned key0, unsigned key1, int &ix, int &iz, float &fx, float &fz,
                                              float &sx, float &sz, float &W0) {
  W0 = 1.f;
  if (P.kind == kVolume) {
    const int npix = nx * nz;
    const unsigned long long total = __ldg(P.cdf + npix - 1);
    if (total == 0ull) {  // all-zero source: nothing to launch
      W0 = 0.f;
      return false;
    }
    const uint4 r0 = philox4x32_10(pid, 0u, key0, key1);
    const uint4 r1 = philox4x32_10(pid, 1u, key0, key1);
    const int pix = pick_pixel(P.cdf, npix, total, r0.x, r0.y);
    ix = pix % nx;
    iz = pix / nx;
    fx = u01(r1.x) * dx;
    fz = u01(r1.y) * dx;
    sincospif(2.f * u01(r0.z), &sx, &sz);
    W0 = __ldg(P.q + pix) < 0.f ? -1.f : 1.f;
    return true;
  }
  float x = P.x0, z = P.z0;
  sx = P.dir_x;
  sz = P.dir_z;
  if (P.kind == MCR_LINE) {
    const uint4 r0 = philox4x32_10(pid, 0u, key0, key1);
    const float u = u01(r0.x);
    x = fmaf(u, P.x1 - P.x0, P.x0);
    z = fmaf(u, P.z1 - P.z0, P.z0);
  } else if (P.kind == MCR_ISO_POINT) {
    const uint4 r0 = philox4x32_10(pid, 0u, key0, key1);
    sincospif(2.f * u01(r0.z), &sx, &sz);
  } else if (P.kind == MCR_ANGULAR_POINT) {
    const uint4 r0 = philox4x32_10(pid, 0u, key0, key1);
    sincosf(launch_angle(P, u01(r0.z)), &sx, &sz);
  }
  if (!(x >= 0.f && x <= nx * dx && z >= 0.f && z <= nz * dx)) return false;
  ix = min((int)floorf(x / dx), nx - 1);
  iz = min((int)floorf(z / dx), nz - 1);
  fx = clamp_dx(x - ix * dx, dx);
  fz = clamp_dx(z - iz * dx, dx);
  return true;
}

// The 2D HG angle theta_s = 2 atan(c tan(pi U)) (Eq. 7) as a rotation: cos theta_s =
// (cp^2 - c^2 sp^2)/(cp^2 + c^2 sp^2), sin theta_s = 2 c sp cp/(...), (sp, cp) = (sin pi U, cos pi U): the
// same angle without tan's pole at U = 1/2.
__device__ __forceinline__ void hg_rotation(float hg_c, float u, float &cs, float &sn) {
  float sp, cp;
  sincospif(u, &sp, &cp);
  const float a = cp * cp, b = hg_c * hg_c * sp * sp;
  const float inv = 1.f / (a + b);
  cs = (a - b) * inv;
  sn = 2.f * hg_c * sp * cp * inv;
}

// Turn a direction and renormalise it.
__device__ __forceinline__ void rotate(float cs, float sn, float &sx, float &sz) {
  const float nsx = fmaf(sx, cs, sz * sn), nsz = fmaf(sz, cs, -sx * sn);
  const float rn = rsqrtf(fmaf(nsx, nsx, nsz * nsz));
  sx = nsx * rn;
  sz = nsz * rn;
}

__device__ __forceinline__ void scatter_hg(float hg_c, float u, float &sx, float &sz) {
  float cs, sn;
  hg_rotation(hg_c, u, cs, sn);
  rotate(cs, sn, sx, sz);
}

// A packet between two launches (record transport -> its next launch, or -> the direct transport):
// four 16-byte words per slot, word w of slot i at saved[w * n + i].
struct SavedPacket {
  unsigned long long pid;
  float fx, fz, sx, sz, W, tau;
  int ix, iz, prob;
  unsigned flight, nscat, cu1, cu2;
};

__device__ __forceinline__ void save_packet(uint4 *saved, size_t n, size_t i, const SavedPacket &s) {
  auto f = [](float v) { return __float_as_uint(v); };
  saved[i] = make_uint4(f(s.fx), f(s.fz), f(s.sx), f(s.sz));
  saved[n + i] = make_uint4(f(s.W), f(s.tau), (unsigned)s.ix, (unsigned)s.iz);
  saved[2 * n + i] = make_uint4((unsigned)s.pid, (unsigned)(s.pid >> 32), s.flight, s.nscat);
  saved[3 * n + i] = make_uint4(s.cu1, s.cu2, (unsigned)s.prob, 0u);
}

__device__ __forceinline__ SavedPacket load_packet(const uint4 *saved, size_t n, size_t i) {
  const uint4 a = saved[i], b = saved[n + i], c = saved[2 * n + i], d = saved[3 * n + i];
  auto f = [](unsigned v) { return __uint_as_float(v); };
  SavedPacket s;
  s.fx = f(a.x), s.fz = f(a.y), s.sx = f(a.z), s.sz = f(a.w);
  s.W = f(b.x), s.tau = f(b.y), s.ix = (int)b.z, s.iz = (int)b.w;
  s.pid = (unsigned long long)c.x | ((unsigned long long)c.y << 32);
  s.flight = c.z, s.nscat = c.w, s.cu1 = d.x, s.cu2 = d.y, s.prob = (int)d.z;
  return s;
}

}  // namespace mcr
