// mcr3.cuh -- what the 3D transport kernels share: the run's parameters, the launch, the spherical harmonics
// and the scatter (the header of include/mcr3.h has the physics).
#pragma once
#include <math_constants.h>

#include "../../include/mcr3.h"
#include "mcr_internal.h"
#include "mcr_rng.cuh"

namespace mcr {

constexpr unsigned kFull3 = 0xFFFFFFFFu;
constexpr int kMaxC3 = (MCR3_MAX_L + 1) * (MCR3_MAX_L + 1);

struct Transport3Params : RecordParams {
  int nx, ny, nz;
  float dx, g;
  int L, C, Cpad, row_stride;
  const float4 *mu;  // packed (mu_a, mu_s, 1/mu_a, 1/mu_s) per voxel
  unsigned long long *tally;
  const unsigned long long *cdf;  // volumetric source: inclusive prefix of quantised |q|
  const float *q;
  int kind;  // MCR_PENCIL, MCR_ISO_POINT, or -1: volumetric
  float x0, y0, z0, ux0, uy0, uz0;
  unsigned key0, key1;
  unsigned long long first_packet, n_packets;
  unsigned max_scatter, max_events;
  float w_threshold, rr_p, rr_inv_p, qscale;
  float nlm[kMaxC3];  // N_lm (times sqrt 2 for m != 0) at index l^2 + l + |m|
  float rinv[MCR3_MAX_L + 1];  // 1 / k
  unsigned long long *work;
  DevStats *stats;
  unsigned *flags;
};

// Real orthonormal spherical harmonics of the unit direction u into row[c], c = l^2 + l + m:
// Y_lm = N_lm Q_l^|m|(u_z) Re/Im[(u_x + i u_y)^|m|], with P_l^m = (1 - u_z^2)^{m/2} Q_l^m and
// Q_m^m = (2m-1)!!, Q_{m+1}^m = (2m+1) u_z Q_m^m, (l - m) Q_l^m = (2l-1) u_z Q_{l-1}^m - (l+m-1) Q_{l-2}^m.
// Every rounding is spelled out (sh_q, sh_power): the record deposit rebuilds the same bits from the same steps.
__device__ __forceinline__ float sh_q(int l, int m, float uz, float qmm, float q1, float q2, float rinv) {
  if (l == m) return qmm;
  if (l == m + 1) return __fmul_rn(__fmul_rn(2.f * m + 1.f, uz), qmm);
  return __fmul_rn(fmaf(__fmul_rn(2.f * l - 1.f, uz), q1, -__fmul_rn(l + m - 1.f, q2)), rinv);
}
__device__ __forceinline__ void sh_power(float &cr, float &ci, float ux, float uy) {  // (cr + i ci) (u_x + i u_y)
  const float nr = fmaf(cr, ux, -__fmul_rn(ci, uy)), ni = fmaf(ci, ux, __fmul_rn(cr, uy));
  cr = nr;
  ci = ni;
}
__device__ __forceinline__ void sh_row(const Transport3Params &p, float ux, float uy, float uz, float *row) {
  float cr = 1.f, ci = 0.f;  // (u_x + i u_y)^m
  float qmm = 1.f;           // Q_m^m
  for (int m = 0; m <= p.L; ++m) {
    float q2 = 0.f, q1 = qmm;
    for (int l = m; l <= p.L; ++l) {
      const float ql = sh_q(l, m, uz, qmm, q1, q2, p.rinv[l - m]);
      if (l > m) {
        q2 = q1;
        q1 = ql;
      }
      const int c0 = l * l + l;
      const float a = __fmul_rn(p.nlm[c0 + m], ql);
      if (m == 0) {
        row[c0] = a;
      } else {
        row[c0 + m] = __fmul_rn(a, cr);
        row[c0 - m] = __fmul_rn(a, ci);
      }
    }
    sh_power(cr, ci, ux, uy);
    qmm = __fmul_rn(qmm, 2.f * m + 1.f);
  }
}

// cos of a 3D Henyey-Greenstein scattering angle by the inverse CDF at u
__device__ __forceinline__ float hg3_cos(float g, float u) {
  if (fabsf(g) < 1e-6f) return 2.f * u - 1.f;
  const float f = (1.f - g * g) / (1.f - g + 2.f * g * u);
  return fminf(fmaxf((1.f + g * g - f * f) / (2.f * g), -1.f), 1.f);
}

// Turn u by polar cos ct and azimuth 2 pi v about itself, in the orthonormal frame of Duff et al.
// (JCGT 2017), then renormalise.
__device__ __forceinline__ void turn(float &ux, float &uy, float &uz, float ct, float v) {
  const float sgn = uz >= 0.f ? 1.f : -1.f;
  const float a = -1.f / (sgn + uz), b = ux * uy * a;
  const float t1x = 1.f + sgn * ux * ux * a, t1y = sgn * b, t1z = -sgn * ux;
  const float t2x = b, t2y = sgn + uy * uy * a, t2z = -uy;
  const float st = sqrtf(fmaxf(0.f, 1.f - ct * ct));
  float sp, cp;
  sincospif(2.f * v, &sp, &cp);
  float nx = ct * ux + st * (cp * t1x + sp * t2x);
  float ny = ct * uy + st * (cp * t1y + sp * t2y);
  float nz = ct * uz + st * (cp * t1z + sp * t2z);
  const float inv = rsqrtf(nx * nx + ny * ny + nz * nz);
  ux = nx * inv;
  uy = ny * inv;
  uz = nz * inv;
}

__device__ __forceinline__ int pick_voxel(const unsigned long long *__restrict__ cdf, int n, unsigned long long total,
                                          unsigned w0, unsigned w1) {
  const unsigned long long r48 = ((unsigned long long)w0 << 16) | (unsigned long long)(w1 >> 16);
  const unsigned long long target = __umul64hi(r48 << 16, total);
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = lo + ((hi - lo) >> 1);
    if (__ldg(cdf + mid) > target)
      hi = mid;
    else
      lo = mid + 1;
  }
  return lo;
}

__device__ __forceinline__ float clamp3(float v, float dx) { return fminf(fmaxf(v, 0.f), dx); }

// Launch voxel, offsets, direction and weight of packet `pid`; returns whether it starts inside the grid.
__device__ __forceinline__ bool launch3(const Transport3Params &p, unsigned long long pid, int &ix, int &iy, int &iz,
                                        float &fx, float &fy, float &fz, float &ux, float &uy, float &uz, float &W0) {
  const float dx = p.dx;
  const uint4 r0 = philox4x32_10(pid, 0u, p.key0, p.key1);
  float x = p.x0, y = p.y0, z = p.z0;
  int vx = -1, vy = 0, vz = 0;
  W0 = 1.f;
  if (p.kind < 0) {  // volumetric: voxel by |q|, uniform in it, W0 = sign q
    const int nvox = p.nx * p.ny * p.nz;
    const unsigned long long total = __ldg(p.cdf + nvox - 1);
    if (total == 0ull) {  // all-zero source: nothing to launch
      W0 = 0.f;
      x = -1.f;
    } else {
      const int v = pick_voxel(p.cdf, nvox, total, r0.x, r0.y);
      const uint4 r1 = philox4x32_10(pid, 1u, p.key0, p.key1);
      vx = v % p.nx;
      vy = (v / p.nx) % p.ny;
      vz = v / (p.nx * p.ny);
      x = u01(r1.x) * dx;
      y = u01(r1.y) * dx;
      z = u01(r1.z) * dx;
      W0 = __ldg(p.q + v) < 0.f ? -1.f : 1.f;
    }
  }
  if (p.kind == MCR_PENCIL) {
    ux = p.ux0;
    uy = p.uy0;
    uz = p.uz0;
  } else {  // isotropic: cos th = 2u - 1, ph = 2 pi u'
    const float ct = 2.f * u01(r0.z) - 1.f, st = sqrtf(fmaxf(0.f, 1.f - ct * ct));
    float sp, cp;
    sincospif(2.f * u01(r0.w), &sp, &cp);
    ux = st * cp;
    uy = st * sp;
    uz = ct;
  }
  if (vx >= 0) {  // (x, y, z) already the offsets in voxel (vx, vy, vz)
    ix = vx;
    iy = vy;
    iz = vz;
    fx = x;
    fy = y;
    fz = z;
    return true;
  }
  if (!(x >= 0.f && x <= p.nx * dx && y >= 0.f && y <= p.ny * dx && z >= 0.f && z <= p.nz * dx)) return false;
  ix = min((int)floorf(x / dx), p.nx - 1);
  iy = min((int)floorf(y / dx), p.ny - 1);
  iz = min((int)floorf(z / dx), p.nz - 1);
  fx = clamp3(x - ix * dx, dx);
  fy = clamp3(y - iy * dx, dx);
  fz = clamp3(z - iz * dx, dx);
  return true;
}

// A packet between two launches: four 16-byte words per slot, word w of slot i at saved[w * n + i].
struct SavedPacket3 {
  unsigned long long pid;
  float fx, fy, fz, ux, uy, uz, W, tau;
  int ix, iy, iz;
  unsigned flight, nscat;
};
__device__ __forceinline__ void save_packet3(uint4 *saved, size_t n, size_t i, const SavedPacket3 &s) {
  auto f = [](float v) { return __float_as_uint(v); };
  saved[i] = make_uint4(f(s.fx), f(s.fy), f(s.fz), f(s.ux));
  saved[n + i] = make_uint4(f(s.uy), f(s.uz), f(s.W), f(s.tau));
  saved[2 * n + i] = make_uint4((unsigned)s.ix, (unsigned)s.iy, (unsigned)s.iz, s.flight);
  saved[3 * n + i] = make_uint4((unsigned)s.pid, (unsigned)(s.pid >> 32), s.nscat, 0u);
}
__device__ __forceinline__ SavedPacket3 load_packet3(const uint4 *saved, size_t n, size_t i) {
  const uint4 a = saved[i], b = saved[n + i], c = saved[2 * n + i], d = saved[3 * n + i];
  auto f = [](unsigned v) { return __uint_as_float(v); };
  SavedPacket3 s;
  s.fx = f(a.x), s.fy = f(a.y), s.fz = f(a.z), s.ux = f(a.w);
  s.uy = f(b.x), s.uz = f(b.y), s.W = f(b.z), s.tau = f(b.w);
  s.ix = (int)c.x, s.iy = (int)c.y, s.iz = (int)c.z, s.flight = c.w;
  s.pid = (unsigned long long)d.x | ((unsigned long long)d.y << 32), s.nscat = d.z;
  return s;
}

// ---- the record deposit (mcr3_records.cu)
cudaError_t rec_plan3(const Transport3Params &p, int64_t rows, RecordPlan *out);
// As launch_records: record launches; on return `closing` is set for the direct transport that adopts the
// packets left.
cudaError_t launch_records3(const Transport3Params &p, const RecordPlan &pl, unsigned char *buf_a, unsigned char *buf_b,
                            unsigned char *scratch, Transport3Params *closing, RecordInfo *info, cudaStream_t s);

}  // namespace mcr
