// mcr3_records.cu -- the record deposit of the 3D form (see mcr_records.cu for the scheme): records of five
// words (voxel, track weight x 2^q, direction), sorted into tiles of 32 voxels; the deposit rebuilds the
// real spherical harmonics of two records at a time in registers, with the operations of sh_row, and sums
// the rounded products.  Bit-identical to the direct deposit of k_transport3, which it replaces because
// that one spends most of a segment on (L+1)^2 reductions: at 96^3 it takes 57, 68, 162 ps a segment for
// L = 2, 4, 8 (1e7 packets; 50 ps by records at L = 4).
#include "mcr3.cuh"
#include "mcr_records.cuh"

namespace mcr {
namespace {

// The transport is bound by instruction issue (78 % of the slots, ALU 51 %, 32 warps an SM); as in 2D,
// lanes that stopped at a collision wait until fewer than kFlyMin3 are flying.
constexpr int kFlyMin3 = 12;

// The 3D packet of a lane: state, the geometry of its flight, and the steps of its path.  The axes' edges
// are handled as in 2D (set_axis).
struct Packet3 {
  unsigned long long pid = 0;
  float fx = 0.f, fy = 0.f, fz = 0.f, ux = 0.f, uy = 0.f, uz = 1.f, W = 0.f, tau = 0.f;
  float inv_x = 0.f, inv_y = 0.f, inv_z = 0.f, ox = 0.f, oy = 0.f, oz = 0.f;
  int ix = 0, iy = 0, iz = 0;
  unsigned flight = 0, nscat = 0;

  __device__ __forceinline__ void load(const SavedPacket3 &s) {
    pid = s.pid, fx = s.fx, fy = s.fy, fz = s.fz, ux = s.ux, uy = s.uy, uz = s.uz, W = s.W, tau = s.tau;
    ix = s.ix, iy = s.iy, iz = s.iz, flight = s.flight, nscat = s.nscat;
  }
  __device__ __forceinline__ void save(uint4 *saved, size_t n, size_t i) const {
    SavedPacket3 s;
    s.pid = pid, s.fx = fx, s.fy = fy, s.fz = fz, s.ux = ux, s.uy = uy, s.uz = uz, s.W = W, s.tau = tau;
    s.ix = ix, s.iy = iy, s.iz = iz, s.flight = flight, s.nscat = nscat;
    save_packet3(saved, n, i, s);
  }
  __device__ __forceinline__ int voxel(const Transport3Params &p) const { return (iz * p.ny + iy) * p.nx + ix; }
  __device__ __forceinline__ bool inside(const Transport3Params &p) const {
    return (unsigned)ix < (unsigned)p.nx && (unsigned)iy < (unsigned)p.ny && (unsigned)iz < (unsigned)p.nz;
  }
  __device__ __forceinline__ void set_direction(float dx) {
    set_axis(ux, dx, ox, inv_x);
    set_axis(uy, dx, oy, inv_y);
    set_axis(uz, dx, oz, inv_z);
  }
  // The next segment in a voxel with 1/mu_s = imus: its length; hit: it ends in a collision; else the axis
  // of the face it ends on (ties: x, y, z).
  __device__ __forceinline__ float segment(float imus, bool &hit, bool &cx, bool &cy) const {
    const float dist_x = fabsf(ox - fx) * inv_x, dist_y = fabsf(oy - fy) * inv_y, dist_z = fabsf(oz - fz) * inv_z;
    const float d_face = fminf(fminf(dist_x, dist_y), dist_z);
    const float d_coll = tau * imus;  // +inf when mu_s = 0 (NaN when tau is 0 too: a face segment)
    hit = d_coll < d_face;
    cx = dist_x == d_face;
    cy = !cx && dist_y == d_face;
    return fminf(d_coll, d_face);
  }
  __device__ __forceinline__ void advance(float l, float dx) {
    fx = clamp3(fmaf(l, ux, fx), dx);
    fy = clamp3(fmaf(l, uy, fy), dx);
    fz = clamp3(fmaf(l, uz, fz), dx);
  }
  __device__ __forceinline__ void cross(bool cx, bool cy, float dx) {
    const bool cz = !cx && !cy;
    ix += cx ? (ux > 0.f ? 1 : -1) : 0;
    iy += cy ? (uy > 0.f ? 1 : -1) : 0;
    iz += cz ? (uz > 0.f ? 1 : -1) : 0;
    fx = cx ? dx - ox : fx;
    fy = cy ? dx - oy : fy;
    fz = cz ? dx - oz : fz;
  }
};

// ------------------------------------------------------------------------------------- transport
__global__ void __launch_bounds__(256, 4) k_transport3_rec(const __grid_constant__ Transport3Params p) {
  extern __shared__ unsigned hist[];  // records per bin of this block
  after_previous();
  if (*p.flags & kFlagMedium) return;
  const unsigned n_in = p.rec_prev ? p.rec_prev->n_left : 0u;
  const bool fresh = !p.rec_prev || p.rec_prev->fresh;
  if (!n_in && !fresh) return;  // every packet has ended
  const unsigned in_buf = p.rec_prev ? p.rec_prev->buf : 1u;
  if (threadIdx.x == 0) p.rec_hdr->buf = 1u - in_buf;
  const int lane = threadIdx.x & 31;
  const unsigned place = warp_place(p.n_sm);
  const unsigned lanes = gridDim.x * blockDim.x;
  const unsigned in_use = fresh ? (unsigned)min(p.n_packets, (unsigned long long)lanes) : n_in;
  const unsigned enough = max(in_use / 2u, p.tail_max);
  for (int i = threadIdx.x; i < p.n_bins; i += blockDim.x) hist[i] = 0u;
  __syncthreads();

  const float dx = p.dx;
  bool alive = false, exhausted = false, pend = false;
  Packet3 a;
  float4 m = make_float4(0.f, 0.f, CUDART_INF_F, CUDART_INF_F);  // (mu_a, mu_s, 1/mu_a, 1/mu_s) of the voxel
  unsigned cu1 = 0, cu2 = 0, cu3 = 0;
  __shared__ double w_esc[256], w_rr[256], w_kill[256];  // weights of the lane's packets that escaped, ...
  w_esc[threadIdx.x] = w_rr[threadIdx.x] = w_kill[threadIdx.x] = 0.0;
  PacketCounts n;
  auto load_mu = [&]() { m = __ldg(p.mu + a.voxel(p)); };
  auto draw_uniforms = [&](unsigned f) {
    const uint4 r = philox4x32_10(a.pid, f + 1u, p.key0, p.key1);
    cu1 = r.y;
    cu2 = r.z;
    cu3 = r.w;
    return r.x;
  };

  bool carrying = false;  // the lane has a packet, or one whose end is not yet counted
  if (place * 32u + lane < n_in) {
    a.load(load_packet3(p.saved + (size_t)in_buf * 4 * p.n_saved, p.n_saved, place * 32u + lane));
    draw_uniforms(a.flight);
    a.set_direction(dx);
    load_mu();
    alive = carrying = true;
  }
  // the next flight, or the packet's end at the event cap
  auto begin_flight = [&]() {
    if (a.flight >= p.max_events) {
      ++n.evl;
      w_kill[threadIdx.x] += a.W;
      alive = false;
      return;
    }
    ++a.flight;
    ++n.flight;
    a.set_direction(dx);
  };
  auto collide = [&]() {
    pend = false;
    ++n.coll;
    if (a.nscat >= p.max_scatter) {
      ++n.scl;
      w_kill[threadIdx.x] += a.W;
      alive = false;
      return;
    }
    // the next flight's numbers depend on nothing here and are drawn first, beside the scatter's chain
    const unsigned u1 = cu1, u2 = cu2, u3 = cu3;
    a.tau = -logf(u01(draw_uniforms(a.flight + 1u)));
    turn(a.ux, a.uy, a.uz, hg3_cos(p.g, u01(u1)), u01(u3));
    ++a.nscat;
    if (fabsf(a.W) < p.w_threshold) {  // |W0| = 1
      if (u01(u2) < p.rr_p) {
        const float Wn = a.W * p.rr_inv_p;
        w_rr[threadIdx.x] += (double)Wn - (double)a.W;
        a.W = Wn;
        ++n.rrs;
      } else {
        w_rr[threadIdx.x] -= a.W;
        ++n.rrk;
        alive = false;
        return;
      }
    }
    begin_flight();
  };
  // ends of packets, counted for the whole call; true when the launch should pause (as in 2D)
  auto count_ends = [&]() -> bool {
    const unsigned ends = __ballot_sync(kFull, carrying && !alive);
    if (!alive) carrying = false;
    const bool draining = __any_sync(kFull, exhausted);
    unsigned ended = 0u;
    if (lane == 0) {
      if (ends) atomicAdd(p.ended, (unsigned)__popc(ends));
      if (draining) ended = *(volatile unsigned *)p.ended;
    }
    return draining && p.n_packets - __shfl_sync(kFull, ended, 0) <= enough;
  };

  RecordWriter w;
  w.stop = in_use <= enough && !(fresh && p.n_packets > lanes);  // as in 2D
  bool first = p.rec_prev == nullptr;
  for (;;) {
    w.room(p, lane);
    unsigned flying = __ballot_sync(kFull, alive && !pend);
    if (w.stop || __popc(flying) < kFlyMin3) {
      if (pend) collide();
      if (count_ends()) w.stop = true;
      if (w.stop && !first) break;  // (the first packets are launched all the same)
      const unsigned need = __ballot_sync(kFull, !alive && !exhausted);
      if (need) {
        const int leader = __ffs(need) - 1;
        unsigned long long base = 0;
        if (lane == leader && !first) base = atomicAdd(p.work, (unsigned long long)__popc(need)) + p.work_base;
        base = __shfl_sync(kFull, base, leader);
        if (!alive && !exhausted) {
          // the first packets go to the warps by their place
          const unsigned long long g = first ? place * 32u + lane : base + __popc(need & ((1u << lane) - 1u));
          if (g >= p.n_packets) {
            exhausted = true;
          } else {
            a.pid = p.first_packet + g;
            ++n.launch;
            carrying = true;
            float W0;
            const bool inside = launch3(p, a.pid, a.ix, a.iy, a.iz, a.fx, a.fy, a.fz, a.ux, a.uy, a.uz, W0);
            a.W = W0;
            n.w_launch += (int)W0;
            a.flight = a.nscat = 0u;
            if (inside) {
              alive = true;
              a.tau = -logf(u01(draw_uniforms(1u)));
              begin_flight();
              load_mu();
            } else {
              ++n.esc;
              w_esc[threadIdx.x] += a.W;
            }
          }
        }
      }
      first = false;
      if (w.stop) break;
      flying = __ballot_sync(kFull, alive);
      if (!flying) {
        if (__all_sync(kFull, exhausted)) break;
        continue;
      }
    }

    // ---------------------------------------------------------------- one voxel segment
    bool has = false;
    unsigned row = 0u;
    float ts = 0.f;
    if (alive && !pend) {
      bool cx, cy;
      const float l = a.segment(m.w, pend, cx, cy);
      const float em1 = expm1f(-m.x * l);
      const float t = m.x > 0.f ? (-a.W * em1) * m.z : a.W * l;
      a.W = fmaf(a.W, em1, a.W);
      ++n.seg;
      ts = t * p.qscale;
      has = t != 0.f && MCR_GUARD(p.flags, isfinite(t));
      row = (unsigned)a.voxel(p);
      a.tau = fmaxf(fmaf(-m.y, l, a.tau), 0.f);  // (a collision draws a new one)
      a.advance(l, dx);
      if (!pend) {
        a.cross(cx, cy, dx);
        if (a.inside(p)) {
          load_mu();
        } else {
          ++n.esc;
          w_esc[threadIdx.x] += a.W;
          alive = false;
        }
      }
    }
    w.put<true>(p, p.flags, hist, lane, has, row, ts, a.ux, a.uy, a.uz);
  }
  if (w.fill < kRecBlock) w.pad(lane);
  count_ends();
  const unsigned left = __ballot_sync(kFull, alive);
  if (left) {  // the packets left go to the next launch, close together
    unsigned at = 0u;
    if (lane == 0) at = atomicAdd(&p.rec_hdr->n_left, (unsigned)__popc(left));
    at = __shfl_sync(kFull, at, 0) + __popc(left & ((1u << lane) - 1u));
    if (alive && MCR_GUARD(p.flags, at < p.n_saved)) a.save(p.saved + (size_t)(1u - in_buf) * 4 * p.n_saved, p.n_saved, at);
  }
  n.add_to(p.stats, p.flags, lane, w_esc[threadIdx.x], w_rr[threadIdx.x], w_kill[threadIdx.x]);
  __syncthreads();
  for (int i = threadIdx.x; i < p.n_bins; i += blockDim.x)
    if (hist[i]) atomicAdd(p.rec_hist + i, hist[i]);
}

// The last packets of a run, a warp to each (k_transport_tail's scheme).
__global__ void __launch_bounds__(kTailThreads, 2) k_transport3_tail(const __grid_constant__ Transport3Params p) {
  extern __shared__ unsigned hist[];
  after_previous();
  if (*p.flags & kFlagMedium) return;
  const unsigned n_in = p.rec_hdr->n_left;
  if (n_in == 0u || n_in > p.tail_max || *p.work + p.work_base < p.n_packets) return;
  for (int i = threadIdx.x; i < p.n_bins; i += blockDim.x) hist[i] = 0u;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const unsigned n_warps = gridDim.x * (blockDim.x >> 5), in_buf = p.rec_hdr->buf;
  const float dx = p.dx;
  const int stride_y = p.nx, stride_z = p.nx * p.ny;
  __shared__ double w_esc[256], w_rr[256], w_kill[256];  // weights of the lane's packets that escaped, ...
  w_esc[threadIdx.x] = w_rr[threadIdx.x] = w_kill[threadIdx.x] = 0.0;
  PacketCounts n;
  RecordWriter w;
  unsigned i = warp_place(p.n_sm);  // the warp's packet; then the next one not yet taken
  while (i < n_in) {
    Packet3 a;
    a.load(load_packet3(p.saved + (size_t)in_buf * 4 * p.n_saved, p.n_saved, i));
    // this voxel and the next ones along the axes (mu has margins: a voxel's neighbours are always there)
    const float4 *at = p.mu + a.voxel(p);
    float4 m = __ldg(at), mx = m, my = m, mz = m;
    int sx = 1, sy = stride_y, sz = stride_z;
    auto look_ahead = [&]() {
      mx = __ldg(at + sx);
      my = __ldg(at + sy);
      mz = __ldg(at + sz);
    };
    auto set_direction = [&]() {
      a.set_direction(dx);
      sx = a.ux > 0.f ? 1 : -1;
      sy = a.uy > 0.f ? stride_y : -stride_y;
      sz = a.uz > 0.f ? stride_z : -stride_z;
      look_ahead();
    };
    set_direction();
    unsigned first = 0u;  // lane k holds the numbers of flight first + k: tau, the scatter's uniforms, roulette
    float n_tau = 0.f, n_cos = 1.f, n_az = 0.f, n_u = 0.f;
    auto draw_flights = [&]() {
      first = a.flight;
      const uint4 r = philox4x32_10(a.pid, a.flight + lane + 1u, p.key0, p.key1);
      n_tau = -logf(u01(r.x));
      n_cos = hg3_cos(p.g, u01(r.y));
      n_u = u01(r.z);
      n_az = u01(r.w);
    };
    draw_flights();
    bool ended = false;
    while (!ended) {
      w.room(p, lane);  // (before a batch, so that one is never left half written)
      if (w.stop) break;
      unsigned row = 0u;  // the lane's segment of the batch
      float len = 0.f, mua = 0.f, imua = 0.f, u0 = 0.f, u1 = 0.f, u2 = 1.f;
      int cnt = 0;
      float loss = 0.f;  // sum of mu_a l of the batch
      auto flush = [&]() {
        const float em1 = lane < cnt ? expm1f(-mua * len) : 0.f;
        float mine = a.W;
#pragma unroll
        for (int k = 0; k < 32; ++k) {  // (past the batch W + W 0)
          const float e = __shfl_sync(kFull, em1, k);
          mine = k == lane ? a.W : mine;
          a.W = fmaf(a.W, e, a.W);
        }
        const float t = mua > 0.f ? (-mine * em1) * imua : mine * len;
        w.put<true>(p, p.flags, hist, lane, lane < cnt && t != 0.f && MCR_GUARD(p.flags, isfinite(t)), row, t * p.qscale, u0,
                    u1, u2);
        if (lane == 0) n.seg += cnt;
        cnt = 0;
      };
      while (cnt < 32 && !ended) {
        bool hit, inside = true;
        do {  // segments up to a collision, the grid's edge or the end of the batch
          bool cx, cy;
          const float l = a.segment(m.w, hit, cx, cy);
          if (lane == cnt) {
            row = (unsigned)a.voxel(p);
            len = l;
            mua = m.x;
            imua = m.z;
            u0 = a.ux;
            u1 = a.uy;
            u2 = a.uz;
          }
          ++cnt;
          loss = fmaf(m.x, l, loss);
          a.advance(l, dx);
          if (hit) break;
          a.tau = fmaxf(fmaf(-m.y, l, a.tau), 0.f);
          a.cross(cx, cy, dx);
          at += cx ? sx : (cy ? sy : sz);
          m = cx ? mx : (cy ? my : mz);
          inside = a.inside(p);
          if (inside) look_ahead();
        } while (inside && cnt < 32);
        if (!hit) {
          if (inside) continue;
          flush();
          if (lane == 0) {
            ++n.esc;
            w_esc[threadIdx.x] += a.W;
          }
          ended = true;
          continue;
        }
        if (lane == 0) ++n.coll;
        if (a.nscat >= p.max_scatter) {
          flush();
          if (lane == 0) {
            ++n.scl;
            w_kill[threadIdx.x] += a.W;
          }
          ended = true;
          continue;
        }
        const int k = (int)(a.flight - first);
        turn(a.ux, a.uy, a.uz, __shfl_sync(kFull, n_cos, k), __shfl_sync(kFull, n_az, k));
        ++a.nscat;
        // |W| is at least |W at the last flush| (1 - loss): the exact weight is needed only when that does
        // not settle the threshold
        if (!(fabsf(a.W) * (1.f - loss) >= 1.001f * p.w_threshold)) {
          flush();
          if (fabsf(a.W) < p.w_threshold) {
            if (__shfl_sync(kFull, n_u, k) < p.rr_p) {
              const float Wn = a.W * p.rr_inv_p;
              if (lane == 0) {
                w_rr[threadIdx.x] += (double)Wn - (double)a.W;
                ++n.rrs;
              }
              a.W = Wn;
            } else {
              if (lane == 0) {
                w_rr[threadIdx.x] -= a.W;
                ++n.rrk;
              }
              ended = true;
              continue;
            }
          }
        }
        if (a.flight >= p.max_events) {
          flush();
          if (lane == 0) {
            ++n.evl;
            w_kill[threadIdx.x] += a.W;
          }
          ended = true;
          continue;
        }
        ++a.flight;
        if (lane == 0) ++n.flight;
        if (a.flight - first == 32u) draw_flights();
        a.tau = __shfl_sync(kFull, n_tau, (int)(a.flight - first));
        set_direction();
        if (cnt == 0) break;  // flushed: a new batch needs its own room
      }
      if (cnt) flush();
    }
    if (lane == 0) {
      if (ended)
        atomicAdd(p.ended, 1u);
      else  // (the buffer is full: the packets still to come pass straight on)
        a.save(p.saved + (size_t)(1u - in_buf) * 4 * p.n_saved, p.n_saved, atomicAdd(&p.rec_hdr->n_tail_left, 1u));
      i = n_warps + atomicAdd(&p.rec_hdr->tail_next, 1u);
    }
    i = __shfl_sync(kFull, i, 0);
  }
  if (w.fill < kRecBlock) w.pad(lane);
  n.add_to(p.stats, p.flags, lane, w_esc[threadIdx.x], w_rr[threadIdx.x], w_kill[threadIdx.x]);
  __syncthreads();
  if (threadIdx.x == 0) p.rec_hdr->tail_ran = 1u;
  for (int k = threadIdx.x; k < p.n_bins; k += blockDim.x)
    if (hist[k]) atomicAdd(p.rec_hist + k, hist[k]);
}

// ------------------------------------------------------------------------------------- deposit
// The channels l^2 + l +- m of the orders m in [M0, M1), numbered in increasing channel order.
template <int L, int M0, int M1>
struct Orders3 {
  static __host__ __device__ constexpr bool has(int c) {
    int l = 0;
    while ((l + 1) * (l + 1) <= c) ++l;
    const int m = c - l * l - l, am = m < 0 ? -m : m;
    return am >= M0 && am < M1;
  }
  static __host__ __device__ constexpr int count(int c_end) {
    int n = 0;
    for (int c = 0; c < c_end; ++c) n += has(c) ? 1 : 0;
    return n;
  }
  static constexpr int kCount = count((L + 1) * (L + 1));
  static __host__ __device__ constexpr int index(int c) { return count(c); }
  static __host__ __device__ constexpr int channel(int i) {
    int c = 0;
    for (int k = 0;; ++c)
      if (has(c) && k++ == i) return c;
  }
};

struct Harmonics3 {
  float nlm[kMaxC3], rinv[MCR3_MAX_L + 1];
};

// compile-time loop: f(integral_constant<int, B>) ... f(integral_constant<int, E - 1>)
template <int V>
struct Int {
  static constexpr int value = V;
};
template <int B, int E, typename F>
__device__ __forceinline__ void unroll(F f) {
  if constexpr (B < E) {
    f(Int<B>{});
    unroll<B + 1, E>(f);
  }
}

// Bound by instruction issue as the 2D deposit (96^3, L = 4: 36 ms of 2.4e9 records, 15 ps each; L = 8, two
// passes: 11 ms of 3e8).
// The orders m in [M0, M1) of all l <= L (the sums of one pass have to fit in registers: two passes from
// L = 7 on).  Even-numbered channels are summed by SumX, odd ones by SumF (see mcr_records.cuh).
template <int L, int M0, int M1, int MINB, int B>
__global__ void __launch_bounds__(kDepThreads, MINB)
    k_rec_deposit3(const float4 *__restrict__ rec, const float *__restrict__ rec_x, const RecordHeader *hdr,
                   const unsigned *__restrict__ tile_off, const unsigned *__restrict__ unit_off, int n_tiles,
                   int tile_shift, long long n_rows, const __grid_constant__ Harmonics3 h, int Cpad,
                   unsigned long long *__restrict__ tally, unsigned *flags) {
  using O = Orders3<L, M0, M1>;
  constexpr int N = O::kCount, NX = (N + 1) / 2, NF = N / 2;
  extern __shared__ float4 smem[];
  after_previous();
  const int T = 1 << tile_shift;
  DepositBatch<B, true> bt(smem, T);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = lane & 3, g = lane >> 2;
  unsigned char *const my_flush = bt.flush + warp * kFlushBytes;
  const unsigned units = hdr->n_units;
  if (blockIdx.x < units && warp == 0) bt.find(rec, rec_x, tile_off, unit_off, n_tiles, blockIdx.x);
  __syncthreads();
  for (unsigned u = blockIdx.x; u < units; u += gridDim.x) {
    const int tile = (int)bt.unit[0];
    const int n_items = bt.load(rec, rec_x, bt.unit[1], (int)bt.unit[2], T, tile_off, unit_off, n_tiles, u + gridDim.x, units);
    for (int it = warp * 8; it < n_items; it = bt.next_runs()) {
      const unsigned item = it + g < n_items ? bt.items[it + g] : 0u;
      const int s0 = item & 0xFFFu, len = (item >> 12) & 0x7Fu;
      const long long row = ((long long)tile << tile_shift) + (item >> 19);
      const int steps = (int)__reduce_max_sync(kFull, (unsigned)(len + 7) / 8);
      const bool ok = len > 0 && MCR_GUARD(flags, row < n_rows);
      unsigned long long *const dst = tally + (size_t)row * Cpad;
      SumX sx[NX];
      SumF sf[NF > 0 ? NF : 1];
#pragma unroll 1
      for (int k = 0; k < steps; ++k) {
        const int ia = k * 8 + j, ib = ia + 4;
        float ta = 0.f, ax = 0.f, ay = 0.f, az = 1.f, tb = 0.f, bx = 0.f, by = 0.f, bz = 1.f;
        if (ia < len) {
          const int r = bt.idx[s0 + ia];
          const float4 v = bt.rec[r];
          ta = v.y, ax = v.z, ay = v.w, az = bt.rec_x[r];
        }
        if (ib < len) {
          const int r = bt.idx[s0 + ib];
          const float4 v = bt.rec[r];
          tb = v.y, bx = v.z, by = v.w, bz = bt.rec_x[r];
        }
        auto add = [&](auto c, float ya, float yb) {
          constexpr int at = O::index(decltype(c)::value);
          if constexpr (at % 2)
            sf[at / 2].add(__fmul_rn(ta, ya), __fmul_rn(tb, yb));
          else
            sx[at / 2].add(__fmul_rn(ta, ya), __fmul_rn(tb, yb));
        };
        // as sh_row: (u_x + i u_y)^m and Q_l^m by the recurrence in l, for both records
        float ca = 1.f, ia_ = 0.f, cb = 1.f, ib_ = 0.f;
        unroll<0, M1>([&](auto m_) {
          constexpr int m = decltype(m_)::value;
          if constexpr (m >= M0) {
            constexpr float qmm = [] {
              float q = 1.f;
              for (int k = 0; k < m; ++k) q *= 2.f * k + 1.f;
              return q;
            }();
            float a2 = 0.f, a1 = qmm, b2 = 0.f, b1 = qmm;
            unroll<m, L + 1>([&](auto l_) {
              constexpr int l = decltype(l_)::value;
              auto next = [&](float &q2, float &q1, float uz) -> float {
                const float ql = sh_q(l, m, uz, qmm, q1, q2, h.rinv[l - m]);
                if constexpr (l > m) {
                  q2 = q1;
                  q1 = ql;
                }
                return ql;
              };
              constexpr int c0 = l * l + l;
              const float va = __fmul_rn(h.nlm[c0 + m], next(a2, a1, az)), vb = __fmul_rn(h.nlm[c0 + m], next(b2, b1, bz));
              if constexpr (m == 0) {
                add(Int<c0>{}, va, vb);
              } else {
                add(Int<c0 + m>{}, __fmul_rn(va, ca), __fmul_rn(vb, cb));
                add(Int<c0 - m>{}, __fmul_rn(va, ia_), __fmul_rn(vb, ib_));
              }
            });
          }
          sh_power(ca, ia_, ax, ay);
          sh_power(cb, ib_, bx, by);
        });
      }
      // sums of the four lanes, 8 channels a round
      unroll<0, (N + 7) / 8>([&](auto r_) {
        constexpr int r = decltype(r_)::value * 8;
        __syncwarp();
        unroll<0, 8>([&](auto c_) {
          constexpr int c = decltype(c_)::value;
          if constexpr (r + c < N) {
            uint2 v;
            if constexpr (c % 2)
              v = make_uint2(sf[(r + c) / 2].lo, sf[(r + c) / 2].hi);
            else
              v = make_uint2(sx[(r + c) / 2].lo, (unsigned)sx[(r + c) / 2].hi);
            *reinterpret_cast<uint2 *>(my_flush + c * kFlushStride + lane * 8) = v;
          }
        });
        __syncwarp();
        unroll<0, 2>([&](auto q_) {
          constexpr int q = decltype(q_)::value * 4;
          if constexpr (r + q < N) {
            const uint4 v = *reinterpret_cast<const uint4 *>(my_flush + (q + j) * kFlushStride + g * 32);
            const uint4 x = *reinterpret_cast<const uint4 *>(my_flush + (q + j) * kFlushStride + g * 32 + 16);
            const unsigned tl = v.x + v.z + x.x + x.z, th = v.y + v.w + x.y + x.w;
            const long long t = j & 1 ? SumF::value(tl, th, 8u * steps) : SumX::value(tl, th);
            constexpr int k0 = O::channel(r + q), k1 = r + q + 1 < N ? O::channel(r + q + 1) : 0,
                          k2 = r + q + 2 < N ? O::channel(r + q + 2) : 0, k3 = r + q + 3 < N ? O::channel(r + q + 3) : 0;
            const int c = j == 0 ? k0 : j == 1 ? k1 : j == 2 ? k2 : k3;
            if (ok && r + q + j < N) atomicAdd(dst + c, (unsigned long long)t);
          }
        });
      });
    }
    __syncthreads();
  }
}

using DepositKernel3 = void (*)(const float4 *, const float *, const RecordHeader *, const unsigned *, const unsigned *,
                                int, int, long long, Harmonics3, int, unsigned long long *, unsigned *);
struct DepositChoice3 {
  DepositKernel3 pass[2];
  int batch;
  size_t (*bytes)(int T);
};
template <int L, int MINB, int B>
DepositChoice3 one_pass() {
  return {{k_rec_deposit3<L, 0, L + 1, MINB, B>, nullptr}, B, DepositBatch<B, true>::bytes};
}
template <int L, int M, int MINB, int B>
DepositChoice3 two_passes() {
  return {{k_rec_deposit3<L, 0, M, MINB, B>, k_rec_deposit3<L, M, L + 1, MINB, B>}, B, DepositBatch<B, true>::bytes};
}
DepositChoice3 deposit_kernel3(int L) {
  switch (L) {
    case 0: return one_pass<0, 5, 1792>();
    case 1: return one_pass<1, 5, 1792>();
    case 2: return one_pass<2, 5, 1792>();
    case 3: return one_pass<3, 5, 1792>();
    case 4: return one_pass<4, 4, 2304>();
    case 5: return one_pass<5, 4, 2304>();
    case 6: return one_pass<6, 3, 2816>();
    case 7: return two_passes<7, 3, 4, 2304>();
    default: return two_passes<8, 3, 4, 2304>();
  }
}

}  // namespace

cudaError_t rec_plan3(const Transport3Params &p, int64_t rows, RecordPlan *out) {
  RecordPlan pl{};
  cudaError_t e = plan_records(rows, p.n_packets, 0, &pl);
  if (e != cudaSuccess) return e;
  pl.threads = 256;
  int sms = 0, per_sm = 0;
  if ((e = sm_count(&sms)) != cudaSuccess) return e;
  const size_t smem = (size_t)pl.n_coarse * 4;
  if ((e = rec_blocks_per_sm(k_transport3_rec, pl.threads, smem, &per_sm)) != cudaSuccess) return e;
  pl.lanes = (unsigned)(sms * per_sm * pl.threads);
  if ((e = rec_blocks_per_sm(k_transport3_tail, kTailThreads, smem, &per_sm)) != cudaSuccess) return e;
  pl.tail_blocks = sms * per_sm;
  set_launches(&pl, p.n_packets);
  *out = pl;
  return cudaSuccess;
}

cudaError_t launch_records3(const Transport3Params &p, const RecordPlan &pl, unsigned char *buf_a, unsigned char *buf_b,
                            unsigned char *scratch, Transport3Params *closing, RecordInfo *info, cudaStream_t s) {
  const DepositChoice3 dc = deposit_kernel3(p.L);
  const size_t dep_smem = dc.bytes(1 << pl.tile_shift);
  int sms = 0, dep[2] = {0, 0};
  cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  for (int k = 0; k < 2 && dc.pass[k]; ++k)
    if ((e = rec_blocks_per_sm(dc.pass[k], kDepThreads, dep_smem, &dep[k])) != cudaSuccess) return e;
  Harmonics3 h;
  for (int c = 0; c < kMaxC3; ++c) h.nlm[c] = p.nlm[c];
  for (int l = 0; l <= MCR3_MAX_L; ++l) h.rinv[l] = p.rinv[l];
  auto buffers = [&](unsigned char *b) { return reinterpret_cast<float4 *>(b); };
  auto fifth = [&](unsigned char *b) { return reinterpret_cast<float *>(b + record_slots(pl) * 16); };
  Transport3Params q = p;
  const unsigned grid = pl.lanes / pl.threads;
  const size_t smem = (size_t)pl.n_coarse * 4;
  e = record_chain<true>(
      pl, layout(scratch, pl), RecordBuffers{buffers(buf_a), buffers(buf_b), fifth(buf_a), fifth(buf_b)}, q, dc.batch,
      p.work, p.n_packets, p.flags,
      [&]() {
        if (q.rec_prev)
          launch_ahead(k_transport3_rec, grid, pl.threads, smem, s, q);
        else  // (it follows a memset)
          k_transport3_rec<<<grid, pl.threads, smem, s>>>(q);
        launch_ahead(k_transport3_tail, pl.tail_blocks, kTailThreads, smem, s, q);
      },
      [&](const float4 *rec, const float *rec_x, const Scratch &sc) {
        int k = 0;
        for (; k < 2 && dc.pass[k]; ++k)
          launch_ahead(dc.pass[k], sms * dep[k], kDepThreads, dep_smem, s, rec, rec_x, q.rec_hdr, sc.tile_off,
                       sc.dep_unit_off, pl.n_tiles, pl.tile_shift, (long long)pl.rows, h, p.Cpad, p.tally, p.flags);
        return k;
      },
      info, s);
  if (e == cudaSuccess) *closing = q;
  return e;
}

}  // namespace mcr
