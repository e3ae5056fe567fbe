// mcr_records.cu -- the record deposit of the 2D harmonic tally (Sec. 3.1, Eqs. 9-11).
//
// The direct deposit (mcr_transport.cu) adds every segment's 2K+1 products to the pixel's tally row
// at once: 8 (2K+1) bytes of 64-bit reductions per segment through the SM's request interface to L2,
// which bounds it.  Here the transport only writes one 16-byte record per segment -- tally row, track
// weight x 2^q, direction -- and the products are made later, row by row, and summed in registers:
//   1. k_transport_rec follows the packets and appends records to blocks of slots that each warp
//      reserves; it counts them per tile (2^tile_shift neighbouring tally rows) in shared memory.
//      When the record buffer is full it pauses: every lane's packet is saved and the next launch
//      takes it up, so that no launch waits for its longest packets.
//   2. k_rec_scan turns the tile counts into offsets and lists the work units.
//   3. k_rec_sort (one pass, or two for many tiles) moves the records into tile order: a block sorts
//      a batch in shared memory and writes each bin's run to its place in one go.
//   4. k_rec_deposit takes a batch of one tile's records, sorts their indices by row in shared memory,
//      and gives each group of four lanes a run of one row's records: every lane rebuilds the harmonic
//      row of two records at a time (the same complex products as harmonic_row, as packed FP32 pairs)
//      and sums the rounded products in registers; one reduction per coefficient and run follows.
// Every product is rounded exactly as in the direct deposit and integer addition is exact, so the
// tally is bit-identical to it.
//
// Nothing is read back: a call enqueues more record launches than it is likely to need (one that finds
// nothing to do ends at once) and then one direct transport launch that adopts whatever packets are
// left, so the call stays asynchronous and can be captured into a graph.
#include <math_constants.h>

#include <mutex>

#include "mcr_packet.cuh"

namespace mcr {
namespace {

constexpr int kMaxBins = 2048;      // bins of one sorting pass (and counters of one transport block)
constexpr int kMaxTiles = 1 << 17;  // tiles of two passes
constexpr int kSortThreads = 512;
constexpr int kTailThreads = 256;
// The tail takes over at this many packets to one of its warps (256 x 256, K = 16, 1e5 packets, transport:
// 3.9 ms at 1, 3.8 at 2, 3.5 at 4, 4.1 at 8; the 128 registers of two blocks per SM beat three blocks by 0.3 ms).
constexpr unsigned kTailPackets = 4;
constexpr int kSortBatch = 4096;    // records a block sorts at a time
constexpr int kDepThreads = 128;
constexpr int kItem = 64;           // most records of one run (a group of four lanes, two records each)
constexpr int kCurStride = 8;       // words between cursors: one 32-byte sector each
constexpr unsigned kMaxLaunches = 1024;
constexpr unsigned kSegmentsPerPacket = 4096;  // record launches are enqueued for this many per packet

// ------------------------------------------------------------------------------------- transport
// Bound by instruction issue (80 % of the slots, 9.9 warp instructions and 9.8 ps a segment at 256 x 256
// with the SMs full).  Lanes that stopped at a collision wait (`pend`) until fewer than kFlyMin of the
// warp's lanes are still flying; the scatter, the new flight's random numbers and the launch of new packets
// then run for all waiting lanes together (4e6 packets: 22.0, 21.4, 21.1, 25.4 ms at 8, 10, 12, 20).
constexpr int kFlyMin = 12;

// A sum of FP32 weights and, apart, of its rounding errors (Knuth's two-sum): FP64's accuracy for a
// lane's few thousand terms without the FP64 pipe, which is narrow on this part.
struct WeightSum {
  float s = 0.f, e = 0.f;
  __device__ __forceinline__ void add(float v) {
    const float t = s + v, b = t - s;
    e += (s - (t - b)) + (v - b);
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)e; }
};

// The warp's record slots: a block of kRecBlock at a time from the launch's buffer.
struct RecordWriter {
  float4 *out = nullptr;
  unsigned fill = kRecBlock;  // slots of the block in use
  bool stop = false;          // the buffer is full (or the launch should pause): write no more
  // what is left of the block holds a sentinel that the sort skips
  __device__ __forceinline__ void pad(int lane) {
    for (unsigned j = fill + lane; j < kRecBlock; j += 32) out[j] = make_float4(__uint_as_float(kRecSentinel), 0.f, 0.f, 1.f);
  }
  __device__ __forceinline__ void room(const TransportParams &p, int lane) {  // for 32 more records; else stop
    if (stop || fill + 32 <= kRecBlock) return;
    pad(lane);
    unsigned b = 0;
    if (lane == 0) b = atomicAdd(&p.rec_hdr->blocks, 1u);
    b = __shfl_sync(kFull, b, 0);
    stop = b >= p.rec_blocks;
    fill = stop ? kRecBlock : 0u;
    if (!stop) out = p.records + (size_t)b * kRecBlock;
  }
  // the warp's records of one step, in its lanes' order
  __device__ __forceinline__ void put(const TransportParams &p, unsigned *hist, int lane, bool has, unsigned row,
                                      float ts, float ux, float uz) {
    const unsigned who = __ballot_sync(kFull, has);
    if (has && MCR_GUARD(p.flags, (row >> p.bin_shift) < (unsigned)p.n_bins)) {
      out[fill + __popc(who & ((1u << lane) - 1u))] = make_float4(__uint_as_float(row), ts, ux, uz);
      atomicAdd(&hist[row >> p.bin_shift], 1u);
    }
    fill += __popc(who);
  }
};

// A lane's run counters, added to the run's by the warp at the end.
struct PacketCounts {
  unsigned launch = 0, flight = 0, coll = 0, seg = 0, esc = 0, rrk = 0, rrs = 0, scl = 0, evl = 0;
  int w_launch = 0;  // |W0| = 1
  WeightSum w_esc, w_rr, w_kill;
  __device__ void add_to(DevStats *st, unsigned *flags, int lane) const {
    auto add = [&](unsigned long long *dst, unsigned v) {
      const unsigned t = __reduce_add_sync(kFull, v);
      if (lane == 0 && t) atomicAdd(dst, (unsigned long long)t);
      return t;
    };
    auto addw = [&](double *dst, double v) {
      const double t = warp_sum(v);
      if (lane == 0 && t != 0.0) atomicAdd(dst, t);
    };
    add(&st->launched, launch);
    add(&st->flights, flight);
    add(&st->collisions, coll);
    add(&st->segments, seg);
    add(&st->escapes, esc);
    add(&st->rr_kill, rrk);
    add(&st->rr_survive, rrs);
    add(&st->scatter_limit, scl);
    if (add(&st->event_limit, evl) && lane == 0) atomicOr(flags, kFlagEventLimit);
    addw(&st->launched_w, (double)w_launch);
    addw(&st->escaped_w, w_esc.value());
    addw(&st->rr_net_w, w_rr.value());
    addw(&st->killed_w, w_kill.value());
  }
};

// The warps of a grid in an order that spreads the first ones over the SMs and their schedulers (blocks
// b, b + n_sm, ... run on one SM, and a block's warp w on scheduler w mod 4).
__device__ __forceinline__ unsigned warp_place(int n_sm) {
  const unsigned wid = (threadIdx.x >> 5) + blockIdx.x / (unsigned)n_sm;
  return (wid % (blockDim.x >> 5)) * gridDim.x + blockIdx.x;
}

// Per-flight geometry of one axis: the offset of the edge ahead and 1 / |s|.  A nonzero component keeps a
// finite reciprocal (so that 0 x it is 0); a zero one gets infinity, and 0 x infinity = NaN loses every
// comparison of the segment.
__device__ __forceinline__ void set_axis(float s, float dx, float &o, float &inv) {
  inv = __frcp_rn(fabsf(s));
  if (s != 0.f) inv = fminf(inv, 3.402823466e38f);
  o = s > 0.f ? dx : 0.f;
}

template <bool BATCH>
__global__ void __launch_bounds__(256, BATCH ? 3 : 4) k_transport_rec(const __grid_constant__ TransportParams p) {
  extern __shared__ unsigned hist[];  // records per bin of this block
  if (*p.flags & kFlagMedium) return;
  // packets that the previous launch left, and whether there are new ones to launch
  const unsigned n_in = p.rec_prev ? p.rec_prev->n_left : 0u;
  const bool fresh = !p.rec_prev || p.rec_prev->fresh;
  if (!n_in && !fresh) return;  // every packet has ended
  const unsigned in_buf = p.rec_prev ? p.rec_prev->buf : 1u;
  if (threadIdx.x == 0) p.rec_hdr->buf = 1u - in_buf;
  const int lane = threadIdx.x & 31;
  const unsigned place = warp_place(p.n_sm);
  // Once no more than `enough` packets are left the launch pauses, so that the next one packs them into
  // full warps, or the tail runs them.
  const unsigned lanes = gridDim.x * blockDim.x;
  const unsigned in_use = fresh ? (unsigned)min(p.total_packets, (unsigned long long)lanes) : n_in;
  const unsigned enough = max(in_use / 2u, p.tail_max);
  for (int i = threadIdx.x; i < p.n_bins; i += blockDim.x) hist[i] = 0u;
  __syncthreads();

  bool alive = false, exhausted = false, pend = false;
  unsigned long long pid = 0;
  // the lane's problem: per-lane registers in a batch, uniform kernel parameters for a single problem
  const float4 *mu = nullptr;
  int prob = 0, nx = 1, nz = 1;
  float dx = 1.f, hg_c = 1.f, qscale = 1.f;
  unsigned key0 = 0, key1 = 0, row_base = 0;
  auto NX = [&]() { return BATCH ? nx : p.prob[0].nx; };
  auto NZ = [&]() { return BATCH ? nz : p.prob[0].nz; };
  auto DX = [&]() { return BATCH ? dx : p.prob[0].dx; };
  auto HGC = [&]() { return BATCH ? hg_c : p.prob[0].hg_c; };
  auto QS = [&]() { return BATCH ? qscale : p.prob[0].qscale; };
  auto KEY0 = [&]() { return BATCH ? key0 : p.prob[0].key0; };
  auto KEY1 = [&]() { return BATCH ? key1 : p.prob[0].key1; };
  auto MU = [&]() { return BATCH ? mu : p.prob[0].mu; };
  auto ROW = [&]() { return BATCH ? row_base : p.prob[0].row_base; };
  auto take_problem = [&](int pi) {
    if (!BATCH) return;
    const ProblemDesc &P = p.prob[pi];
    prob = pi;
    mu = P.mu;
    nx = P.nx;
    nz = P.nz;
    dx = P.dx;
    hg_c = P.hg_c;
    qscale = P.qscale;
    key0 = P.key0;
    key1 = P.key1;
    row_base = P.row_base;
  };
  // packet state; (ox, oz): the offset of the edge ahead, (inv_ax, inv_az): 1 / |s| per axis, and
  // (mu_a, mu_s, 1/mu_a, 1/mu_s) of the current pixel
  float fx = 0.f, fz = 0.f, sx = 0.f, sz = 1.f, W = 0.f, tau = 0.f;
  float inv_ax = 0.f, inv_az = 0.f, ox = 0.f, oz = 0.f;
  int ix = 0, iz = 0;
  float4 m = make_float4(0.f, 0.f, CUDART_INF_F, CUDART_INF_F);
  unsigned flight = 0, nscat = 0, cu1 = 0, cu2 = 0;
  PacketCounts n;

  auto load_mu = [&]() {
    if (MCR_GUARD(p.flags, (unsigned)ix < (unsigned)NX() && (unsigned)iz < (unsigned)NZ())) m = __ldg(MU() + iz * NX() + ix);
  };
  auto set_direction = [&]() {
    set_axis(sx, DX(), ox, inv_ax);
    set_axis(sz, DX(), oz, inv_az);
  };

  // the packets left by the previous launch, 32 to a warp
  bool carrying = false;  // the lane has a packet, or one whose end is not yet counted
  if (place * 32u + lane < n_in) {
    const SavedPacket s = load_packet(p.saved + (size_t)in_buf * 4 * p.n_saved, p.n_saved, place * 32u + lane);
    take_problem(s.prob);
    pid = s.pid, fx = s.fx, fz = s.fz, sx = s.sx, sz = s.sz, W = s.W, tau = s.tau, ix = s.ix, iz = s.iz;
    flight = s.flight, nscat = s.nscat, cu1 = s.cu1, cu2 = s.cu2;
    set_direction();
    load_mu();
    alive = carrying = true;
  }

  // One pixel segment of a flying packet: advances it, sets pend at a collision, ends the packet at the
  // grid's edge; returns whether there is a record (row, ts and the flight's direction).
  auto segment = [&](unsigned &row, float &ts) -> bool {
    const float dist_x = fabsf(ox - fx) * inv_ax, dist_z = fabsf(oz - fz) * inv_az;
    const float d_edge = fminf(dist_x, dist_z);
    const float d_coll = tau * m.w;  // +inf when mu_s = 0 (NaN when tau is 0 too: an edge segment)
    pend = d_coll < d_edge;
    const float l = fminf(d_coll, d_edge);
    // track weight of the segment: W (1 - e^{-mu_a l}) / mu_a, then W <- W e^{-mu_a l}
    const float em1 = expm1f(-m.x * l);
    const float t = m.x > 0.f ? (-W * em1) * m.z : W * l;
    W = fmaf(W, em1, W);
    ++n.seg;
    ts = t * QS();
    row = ROW() + (unsigned)(iz * NX() + ix);
    tau = fmaxf(fmaf(-m.y, l, tau), 0.f);  // (a collision draws a new one)
    fx = clamp_dx(fmaf(l, sx, fx), DX());
    fz = clamp_dx(fmaf(l, sz, fz), DX());
    if (!pend) {  // step over the edge ahead; ties: x first, z follows as a zero-length segment
      const bool cx = dist_x == d_edge;
      ix += cx ? (sx > 0.f ? 1 : -1) : 0;
      iz += cx ? 0 : (sz > 0.f ? 1 : -1);
      fx = cx ? DX() - ox : fx;
      fz = cx ? fz : DX() - oz;
      if ((unsigned)ix >= (unsigned)NX() || (unsigned)iz >= (unsigned)NZ()) {
        ++n.esc;
        n.w_esc.add(W);
        alive = false;
      } else {
        m = __ldg(MU() + iz * NX() + ix);
      }
    }
    return t != 0.f && MCR_GUARD(p.flags, isfinite(t));
  };
  // The random numbers of free flight f (event f + 1): tau = -ln U, the scatter and roulette uniforms.
  auto draw_flight = [&](unsigned f) {
    const uint4 r = philox4x32_10(pid, f + 1u, KEY0(), KEY1());
    tau = -logf(u01(r.x));
    cu1 = r.y;
    cu2 = r.z;
  };
  // The collision of a packet that stopped at one: scatter, roulette, and the next flight.  The next
  // flight's numbers depend on nothing here and are drawn first, beside the scatter's own chain.
  auto collide = [&]() {
    pend = false;
    ++n.coll;
    if (nscat >= p.max_scatter) {
      ++n.scl;
      n.w_kill.add(W);
      alive = false;
      return;
    }
    const unsigned u1 = cu1, u2 = cu2;
    draw_flight(flight + 1u);
    scatter_hg(HGC(), u01(u1), sx, sz);
    set_direction();
    ++nscat;
    if (fabsf(W) < p.w_threshold) {  // |W0| = 1
      if (u01(u2) < p.rr_p) {
        const float Wn = W * p.rr_inv_p;
        n.w_rr.add(Wn);
        n.w_rr.add(-W);
        W = Wn;
        ++n.rrs;
      } else {
        n.w_rr.add(-W);
        ++n.rrk;
        alive = false;
        return;
      }
    }
    if (flight >= p.max_events) {
      ++n.evl;
      n.w_kill.add(W);
      alive = false;
      return;
    }
    ++flight;
    ++n.flight;
  };

  // Ends of packets, counted for the whole call; true when the launch should pause.  (The count is read
  // only by warps that have found no more packets to launch: the answer takes a round trip to L2.)
  auto count_ends = [&]() -> bool {
    const unsigned ends = __ballot_sync(kFull, carrying && !alive);
    if (!alive) carrying = false;
    const bool draining = __any_sync(kFull, exhausted);
    unsigned ended = 0u;
    if (lane == 0) {
      if (ends) atomicAdd(p.ended, (unsigned)__popc(ends));
      if (draining) ended = *(volatile unsigned *)p.ended;
    }
    return draining && p.total_packets - __shfl_sync(kFull, ended, 0) <= enough;
  };

  RecordWriter w;
  w.stop = in_use <= enough;  // nothing for this kernel to do but launch the first packets
  bool first = p.rec_prev == nullptr;
  for (;;) {
    w.room(p, lane);
    unsigned flying = __ballot_sync(kFull, alive && !pend);
    if (w.stop || __popc(flying) < kFlyMin) {
      if (pend) collide();
      if (count_ends()) w.stop = true;
      if (w.stop && !first) break;  // (the first packets are launched all the same)
      // ------------------------------------------------------------- refill / launch
      const unsigned need = __ballot_sync(kFull, !alive && !exhausted);
      if (need) {
        const int leader = __ffs(need) - 1;
        unsigned long long base = 0;
        if (lane == leader && !first) base = atomicAdd(p.work, (unsigned long long)__popc(need)) + p.work_base;
        base = __shfl_sync(kFull, base, leader);
        if (!alive && !exhausted) {
          // the first packets go to the warps by their place
          const unsigned long long g = first ? place * 32u + lane : base + __popc(need & ((1u << lane) - 1u));
          if (g >= p.total_packets) {
            exhausted = true;
          } else {
            int lo = 0;  // the problem owning launch packet g: smallest pi with prob[pi].end > g
            if (BATCH) {
              int hi = p.n_problems - 1;
              while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (p.prob[mid].end > g)
                  hi = mid;
                else
                  lo = mid + 1;
              }
            }
            const ProblemDesc &P = p.prob[lo];
            pid = P.first_packet + (g - (lo ? p.prob[lo - 1].end : 0ull));
            take_problem(lo);
            ++n.launch;
            carrying = true;
            float W0;
            const bool inside = launch_packet(P, pid, NX(), NZ(), DX(), KEY0(), KEY1(), ix, iz, fx, fz, sx, sz, W0);
            W = W0;
            n.w_launch += (int)W0;
            nscat = 0;
            flight = 0;
            if (!inside) {
              ++n.esc;
              n.w_esc.add(W);
            } else if (p.max_events == 0u) {
              ++n.evl;
              n.w_kill.add(W);
            } else {
              flight = 1;
              ++n.flight;
              alive = true;
              draw_flight(1u);
              set_direction();
              load_mu();
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

    // ---------------------------------------------------------------- one pixel segment
    bool has = false;
    unsigned row = 0u;
    float ts = 0.f;
    if (alive && !pend) has = segment(row, ts);
    w.put(p, hist, lane, has, row, ts, sx, sz);
  }
  if (w.fill < kRecBlock) w.pad(lane);
  count_ends();
  // the packets left go to the next launch, close together
  const unsigned left = __ballot_sync(kFull, alive);
  if (left) {
    unsigned at = 0u;
    if (lane == 0) at = atomicAdd(&p.rec_hdr->n_left, (unsigned)__popc(left));
    at = __shfl_sync(kFull, at, 0) + __popc(left & ((1u << lane) - 1u));
    if (alive && MCR_GUARD(p.flags, at < p.n_saved)) {
      SavedPacket s;
      s.pid = pid, s.fx = fx, s.fz = fz, s.sx = sx, s.sz = sz, s.W = W, s.tau = tau, s.ix = ix, s.iz = iz, s.prob = prob;
      s.flight = flight, s.nscat = nscat, s.cu1 = cu1, s.cu2 = cu2;
      save_packet(p.saved + (size_t)(1u - in_buf) * 4 * p.n_saved, p.n_saved, at, s);
    }
  }
  n.add_to(p.stats, p.flags, lane);
  __syncthreads();
  for (int i = threadIdx.x; i < p.n_bins; i += blockDim.x)
    if (hist[i]) atomicAdd(p.rec_hist + i, hist[i]);
}

// ------------------------------------------------------------------------------------------ tail
// The last packets of a run (256 x 256, 1e3 packets: 6.3 ms with the loop of the direct deposit, 3.4 with the
// one above, 1.2 here; 460 cycles a segment, a chain of dependent instructions).
// A packet that stays in the medium lives for thousands of segments, and once
// there are few packets to a warp the run lasts as long as one packet's chain of segments; a warp with
// one lane in use would take every step of the loop above for it.  So a whole warp follows one packet:
// all lanes take the same steps (no divergence), the lanes draw the numbers of 32 flights at once, and
// what does not steer the packet -- track weights, the weight itself -- is computed for 32 segments at
// once, one per lane, in the same order of operations.  The pixels ahead are loaded a segment early.
__global__ void __launch_bounds__(256, 2) k_transport_tail(const __grid_constant__ TransportParams p) {
  extern __shared__ unsigned hist[];  // records per bin of this block
  if (*p.flags & kFlagMedium) return;
  const unsigned n_in = p.rec_hdr->n_left;
  if (n_in == 0u || n_in > p.tail_max || *p.work + p.work_base < p.total_packets) return;
  for (int i = threadIdx.x; i < p.n_bins; i += blockDim.x) hist[i] = 0u;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const unsigned n_warps = gridDim.x * (blockDim.x >> 5), in_buf = p.rec_hdr->buf;
  PacketCounts n;
  RecordWriter w;
  unsigned i = warp_place(p.n_sm);  // the warp's packet; then the next one not yet taken
  while (i < n_in) {
    SavedPacket s = load_packet(p.saved + (size_t)in_buf * 4 * p.n_saved, p.n_saved, i);
    const ProblemDesc &P = p.prob[s.prob];
    const float4 *const mu = P.mu;
    const int nx = P.nx, nz = P.nz;
    const float dx = P.dx, hg_c = P.hg_c, qscale = P.qscale;
    const unsigned key0 = P.key0, key1 = P.key1, row_base = P.row_base;
    const unsigned long long pid = s.pid;
    float fx = s.fx, fz = s.fz, sx = s.sx, sz = s.sz, W = s.W, tau = s.tau;
    int ix = s.ix, iz = s.iz;
    unsigned flight = s.flight, nscat = s.nscat;
    float inv_ax, inv_az, ox, oz;
    // this pixel and the next ones in x and z (mu has margins: a pixel's neighbours are always there)
    const float4 *at = mu + iz * nx + ix;
    int step_x = 1, step_z = 1, stride_z = nx;
    float4 m = __ldg(at), mx = m, mz = m;
    auto look_ahead = [&]() {
      mx = __ldg(at + step_x);
      mz = __ldg(at + stride_z);
    };
    auto set_direction = [&]() {
      set_axis(sx, dx, ox, inv_ax);
      set_axis(sz, dx, oz, inv_az);
      step_x = sx > 0.f ? 1 : -1;
      step_z = sz > 0.f ? 1 : -1;
      stride_z = sz > 0.f ? nx : -nx;
      look_ahead();
    };
    set_direction();
    unsigned first = 0u;  // lane k holds the numbers of flight first + k: tau, rotation, roulette uniform
    float n_tau = 0.f, n_cs = 1.f, n_sn = 0.f, n_u = 0.f;
    auto draw_flights = [&]() {
      first = flight;
      const uint4 r = philox4x32_10(pid, flight + lane + 1u, key0, key1);
      n_tau = -logf(u01(r.x));
      hg_rotation(hg_c, u01(r.y), n_cs, n_sn);
      n_u = u01(r.z);
    };
    draw_flights();
    bool ended = false;
    while (!ended) {
      w.room(p, lane);  // (before a batch, so that one is never left half written)
      if (w.stop) break;
      unsigned row = 0u;  // the lane's segment of the batch
      float len = 0.f, mua = 0.f, imua = 0.f, ux = 0.f, uz = 1.f;
      int cnt = 0;
      float loss = 0.f;  // sum of mu_a l of the batch
      // the batch's track weights and records; W becomes exact again
      auto flush = [&]() {
        const float em1 = lane < cnt ? expm1f(-mua * len) : 0.f;
        float mine = W;
#pragma unroll
        for (int k = 0; k < 32; ++k) {  // (past the batch W + W 0)
          const float e = __shfl_sync(kFull, em1, k);
          mine = k == lane ? W : mine;
          W = fmaf(W, e, W);
        }
        const float t = mua > 0.f ? (-mine * em1) * imua : mine * len;
        w.put(p, hist, lane, lane < cnt && t != 0.f && MCR_GUARD(p.flags, isfinite(t)), row, t * qscale, ux, uz);
        if (lane == 0) n.seg += cnt;
        cnt = 0;
      };
      while (cnt < 32 && !ended) {
        bool hit, inside = true;
        do {  // segments up to a collision, the grid's edge or the end of the batch
          const float dist_x = fabsf(ox - fx) * inv_ax, dist_z = fabsf(oz - fz) * inv_az;
          const float d_edge = fminf(dist_x, dist_z);
          const float d_coll = tau * m.w;
          hit = d_coll < d_edge;
          const float l = fminf(d_coll, d_edge);
          if (lane == cnt) {
            row = row_base + (unsigned)(iz * nx + ix);
            len = l;
            mua = m.x;
            imua = m.z;
            ux = sx;
            uz = sz;
          }
          ++cnt;
          loss = fmaf(m.x, l, loss);
          fx = clamp_dx(fmaf(l, sx, fx), dx);
          fz = clamp_dx(fmaf(l, sz, fz), dx);
          if (hit) break;
          tau = fmaxf(fmaf(-m.y, l, tau), 0.f);
          const bool cx = dist_x == d_edge;
          ix += cx ? step_x : 0;
          iz += cx ? 0 : step_z;
          at += cx ? step_x : stride_z;
          fx = cx ? dx - ox : fx;
          fz = cx ? fz : dx - oz;
          m = cx ? mx : mz;
          inside = (unsigned)ix < (unsigned)nx && (unsigned)iz < (unsigned)nz;
          if (inside) look_ahead();
        } while (inside && cnt < 32);
        if (!hit) {
          if (inside) continue;
          flush();
          if (lane == 0) {
            ++n.esc;
            n.w_esc.add(W);
          }
          ended = true;
          continue;
        }
        if (lane == 0) ++n.coll;
        if (nscat >= p.max_scatter) {
          flush();
          if (lane == 0) {
            ++n.scl;
            n.w_kill.add(W);
          }
          ended = true;
          continue;
        }
        const int k = (int)(flight - first);
        rotate(__shfl_sync(kFull, n_cs, k), __shfl_sync(kFull, n_sn, k), sx, sz);
        ++nscat;
        // |W| is at least |W at the last flush| (1 - loss): the exact weight is needed only when that does
        // not settle the threshold
        if (!(fabsf(W) * (1.f - loss) >= 1.001f * p.w_threshold)) {
          flush();
          if (fabsf(W) < p.w_threshold) {
            if (__shfl_sync(kFull, n_u, k) < p.rr_p) {
              const float Wn = W * p.rr_inv_p;
              if (lane == 0) {
                n.w_rr.add(Wn);
                n.w_rr.add(-W);
                ++n.rrs;
              }
              W = Wn;
            } else {
              if (lane == 0) {
                n.w_rr.add(-W);
                ++n.rrk;
              }
              ended = true;
              continue;
            }
          }
        }
        if (flight >= p.max_events) {
          flush();
          if (lane == 0) {
            ++n.evl;
            n.w_kill.add(W);
          }
          ended = true;
          continue;
        }
        ++flight;
        if (lane == 0) ++n.flight;
        if (flight - first == 32u) draw_flights();
        tau = __shfl_sync(kFull, n_tau, (int)(flight - first));
        set_direction();
        if (cnt == 0) break;  // flushed: a new batch needs its own room
      }
      if (cnt) flush();
    }
    if (lane == 0) {
      if (ended) {
        atomicAdd(p.ended, 1u);
      } else {  // (the buffer is full: the packets still to come pass straight on)
        const uint4 r = philox4x32_10(pid, flight + 1u, key0, key1);
        s.fx = fx, s.fz = fz, s.sx = sx, s.sz = sz, s.W = W, s.tau = tau, s.ix = ix, s.iz = iz;
        s.flight = flight, s.nscat = nscat, s.cu1 = r.y, s.cu2 = r.z;
        save_packet(p.saved + (size_t)(1u - in_buf) * 4 * p.n_saved, p.n_saved, atomicAdd(&p.rec_hdr->n_tail_left, 1u), s);
      }
      i = n_warps + atomicAdd(&p.rec_hdr->tail_next, 1u);
    }
    i = __shfl_sync(kFull, i, 0);
  }
  if (w.fill < kRecBlock) w.pad(lane);
  n.add_to(p.stats, p.flags, lane);
  __syncthreads();
  if (threadIdx.x == 0) p.rec_hdr->tail_ran = 1u;
  for (int i = threadIdx.x; i < p.n_bins; i += blockDim.x)
    if (hist[i]) atomicAdd(p.rec_hist + i, hist[i]);
}

// ------------------------------------------------------------------------------------- offsets
// Inclusive scan of v over the block (1024 threads); warp_tot: 32 words of shared memory.
__device__ unsigned block_scan(unsigned v, unsigned *warp_tot) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(kFull, v, o);
    if (lane >= o) v += t;
  }
  __syncthreads();
  if (lane == 31) warp_tot[wid] = v;
  __syncthreads();
  if (wid == 0) {
    unsigned t = lane < (int)(blockDim.x >> 5) ? warp_tot[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned u = __shfl_up_sync(kFull, t, o);
      if (lane >= o) t += u;
    }
    warp_tot[lane] = t;
  }
  __syncthreads();
  return v + (wid ? warp_tot[wid - 1] : 0u);
}

// Exclusive scan of f(i), i < n, into off[0, n] by one block of 1024 threads; returns the total.
template <typename F>
__device__ unsigned scan_into(int n, unsigned *off, unsigned *warp_tot, F f) {
  unsigned carry = 0;
  __shared__ unsigned total;
  for (int base = 0; base < n; base += 1024) {
    const int i = base + threadIdx.x;
    const unsigned x = i < n ? f(i) : 0u;
    const unsigned incl = block_scan(x, warp_tot);
    if (i < n) off[i] = carry + incl - x;
    if (threadIdx.x == 1023) total = incl;
    __syncthreads();
    carry += total;
    __syncthreads();
  }
  if (threadIdx.x == 0) off[n] = carry;
  __syncthreads();
  return carry;
}

// Counts per bin -> offsets, cursors and the offsets of the bins' work units (batches of `batch`
// records); clears the counts for the next launch.  n_units: the launch's word for their number.  Also
// settles, for every warp of the next launch alike, what is left to it.
__global__ void __launch_bounds__(1024) k_rec_scan(RecordHeader *hdr, unsigned *n_units, unsigned *hist, int n,
                                                   int batch, unsigned *off, unsigned *cur, unsigned *unit_off,
                                                   const unsigned long long *launched, unsigned long long n_packets) {
  __shared__ unsigned warp_tot[32];
  if (threadIdx.x == 0) {
    if (*launched < n_packets) hdr->fresh = 1u;
    if (hdr->tail_ran == 1u) {  // what the tail left stands in the other buffer
      hdr->n_left = hdr->n_tail_left;
      hdr->buf = 1u - hdr->buf;
      hdr->tail_ran = 2u;
    }
  }
  if (hdr->blocks == 0u) return;
  scan_into(n, off, warp_tot, [&](int i) { return hist[i]; });
  const unsigned units = scan_into(n, unit_off, warp_tot, [&](int i) { return (hist[i] + batch - 1) / batch; });
  for (int i = threadIdx.x; i < n; i += 1024) {
    cur[i * kCurStride] = off[i];
    hist[i] = 0u;
  }
  if (threadIdx.x == 0) *n_units = units;
}

// The last i < n with off[i] <= u (off nondecreasing, off[0] = 0), found by the whole block in two
// rounds of probes (three where n > blockDim.x^2).
__device__ int block_find(const unsigned *__restrict__ off, int n, unsigned u) {
  const int t = threadIdx.x, nt = (int)blockDim.x;
  int a = 0;
  for (int step = n > nt * nt ? nt * nt : (n > nt ? nt : 1);; step = step > nt ? nt : 1) {
    a += (__syncthreads_count(a + t * step < n && __ldg(off + a + t * step) <= u) - 1) * step;
    if (step == 1) return a;
  }
}

// ------------------------------------------------------------------------------------- sort
// One sorting pass: batches of records into bins.  FIRST: the transport's slots (sentinels skipped) into
// bins of 2^shift rows.  Otherwise: one coarse bin's records into its tiles.
// The batch is sorted in shared memory first, so that a bin's records leave as one contiguous run and
// take one cursor update per batch and bin instead of one per record.
template <bool FIRST>
__global__ void __launch_bounds__(kSortThreads, 2)
    k_rec_sort(const float4 *__restrict__ in, float4 *__restrict__ sorted, const RecordHeader *hdr, unsigned max_blocks,
               int shift, int n_bins, unsigned *cursor, unsigned capacity, const unsigned *__restrict__ coarse_off, const unsigned *__restrict__ coarse_unit_off,
               int n_coarse, int coarse_shift, unsigned *flags) {
  constexpr int kPer = kSortBatch / kSortThreads;
  extern __shared__ float4 srec[];                                  // [kSortBatch]
  unsigned *cnt = reinterpret_cast<unsigned *>(srec + kSortBatch);  // [n_bins] counts, then local starts
  unsigned *delta = cnt + n_bins;                                   // [n_bins] global place minus local place
  __shared__ unsigned warp_tot[32];
  const unsigned n = min(hdr->blocks, max_blocks) * kRecBlock;
  const unsigned units = FIRST ? (n + kSortBatch - 1) / kSortBatch : hdr->n_coarse_units;
  for (unsigned u = blockIdx.x; u < units; u += gridDim.x) {
    unsigned lo = u * kSortBatch, hi = min(lo + kSortBatch, n), bin0 = 0;
    unsigned *cur = cursor;
    if (!FIRST) {
      const int c = block_find(coarse_unit_off, n_coarse, u);
      bin0 = (unsigned)c << coarse_shift;
      lo = coarse_off[c] + (u - coarse_unit_off[c]) * kSortBatch;
      hi = min(lo + kSortBatch, coarse_off[c + 1]);
      cur += bin0 * kCurStride;
    }
    for (int i = threadIdx.x; i < n_bins; i += kSortThreads) cnt[i] = 0u;
    __syncthreads();
    float4 r[kPer];
    unsigned bin[kPer], rank[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const unsigned i = lo + k * kSortThreads + threadIdx.x;
      r[k] = i < hi ? __ldcs(in + i) : make_float4(__uint_as_float(kRecSentinel), 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const unsigned row = __float_as_uint(r[k].x);
      bin[k] = row == kRecSentinel ? kRecSentinel : (row >> shift) - bin0;
      if (bin[k] != kRecSentinel && !MCR_GUARD(flags, bin[k] < (unsigned)n_bins)) bin[k] = kRecSentinel;
      rank[k] = bin[k] != kRecSentinel ? atomicAdd(&cnt[bin[k]], 1u) : 0u;
    }
    __syncthreads();
    // local starts by a block scan over the bins, and each bin's place from the global cursor
    constexpr int kBins = kMaxBins / kSortThreads;  // neighbouring bins of one thread
    const int b0 = threadIdx.x * kBins;
    unsigned c[kBins], at[kBins], sum = 0;
#pragma unroll
    for (int k = 0; k < kBins; ++k) {
      c[k] = b0 + k < n_bins ? cnt[b0 + k] : 0u;
      sum += c[k];
    }
#pragma unroll
    for (int k = 0; k < kBins; ++k)
      if (c[k]) at[k] = atomicAdd(cur + (b0 + k) * kCurStride, c[k]);
    unsigned start = block_scan(sum, warp_tot) - sum;
#pragma unroll
    for (int k = 0; k < kBins; ++k) {
      if (b0 + k < n_bins) {
        cnt[b0 + k] = start;
        if (c[k]) delta[b0 + k] = at[k] - start;
      }
      start += c[k];
    }
    __syncthreads();
    const unsigned total = warp_tot[(kSortThreads >> 5) - 1];
#pragma unroll
    for (int k = 0; k < kPer; ++k)
      if (bin[k] != kRecSentinel) srec[cnt[bin[k]] + rank[k]] = r[k];
    __syncthreads();
    for (unsigned i = threadIdx.x; i < total; i += kSortThreads) {
      const float4 v = srec[i];
      const unsigned at = delta[(__float_as_uint(v.x) >> shift) - bin0] + i;
      if (MCR_GUARD(flags, at < capacity)) sorted[at] = v;
    }
    __syncthreads();
  }
}

// Counts per tile of the coarse-sorted records, before the second pass.
__global__ void __launch_bounds__(kSortThreads) k_rec_count(const float4 *__restrict__ rec, const RecordHeader *hdr,
                                                            const unsigned *__restrict__ coarse_off,
                                                            const unsigned *__restrict__ coarse_unit_off, int n_coarse,
                                                            int coarse_shift, int tile_shift, unsigned *tile_hist,
                                                            unsigned *flags) {
  __shared__ unsigned cnt[kMaxBins];
  const int nb = 1 << coarse_shift;
  const unsigned units = hdr->n_coarse_units;
  for (unsigned u = blockIdx.x; u < units; u += gridDim.x) {
    for (int i = threadIdx.x; i < nb; i += kSortThreads) cnt[i] = 0u;
    const int c = block_find(coarse_unit_off, n_coarse, u);
    const unsigned lo = coarse_off[c] + (u - coarse_unit_off[c]) * kSortBatch;
    const unsigned hi = min(lo + kSortBatch, coarse_off[c + 1]), bin0 = (unsigned)c << coarse_shift;
#pragma unroll
    for (int k = 0; k < kSortBatch / kSortThreads; ++k) {
      const unsigned i = lo + k * kSortThreads + threadIdx.x;
      if (i >= hi) continue;
      const unsigned b = (__float_as_uint(__ldg(&rec[i].x)) >> tile_shift) - bin0;
      if (MCR_GUARD(flags, b < (unsigned)nb)) atomicAdd(&cnt[b], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nb; i += kSortThreads)
      if (cnt[i]) atomicAdd(tile_hist + bin0 + i, cnt[i]);
    __syncthreads();
  }
}

// ------------------------------------------------------------------------------------- deposit
// The rounded products round(t 2^q h) (below 2^30 in magnitude) are summed exactly in two 32-bit words
// per coefficient, in two ways that load different pipes (cosines take the first, sines the second):
// SumX converts (XU pipe, 16 lanes a cycle) and keeps the sum modulo 2^32 and the sum of the high
// halves x >> 16, which together determine the 64-bit sum of up to 2^16 terms (the low halves' sum is
// below 2^32);
struct SumX {
  unsigned lo = 0u;
  int hi = 0;
  __device__ __forceinline__ void add(float a, float b) {
    const int x = __float2int_rn(a) + __float2int_rn(b);
    lo += (unsigned)x;
    hi += x >> 16;
  }
  static __device__ __forceinline__ long long value(unsigned lo, unsigned hi) {
    return ((long long)(int)hi << 16) + (long long)(lo - (hi << 16));
  }
};
// SumF splits by FP32 additions (FMA pipe): y + 1.5 2^31 holds k = round(y / 2^8) in its low mantissa
// bits, and (y - 2^8 k) + 1.5 2^23 the rest's nearest integer (|rest| <= 2^7; both steps are exact, and
// ties round to even as y's own rounding does, 2^8 k being even).  The words are the sums of the two bit
// patterns; n terms carry n times the constants' bits and at most n 2^22 (n < 2^9).
struct SumF {
  static constexpr float kHigh = 3221225472.f, kLow = 12582912.f;             // 1.5 2^31, 1.5 2^23
  static constexpr unsigned kHighBits = 0x4F400000u, kLowBits = 0x4B400000u;  // their bits
  unsigned lo = 0u, hi = 0u;
  __device__ __forceinline__ void add(float a, float b) {
    const float ha = __fadd_rn(a, kHigh), hb = __fadd_rn(b, kHigh);
    const float la = __fadd_rn(__fadd_rn(a, __fsub_rn(kHigh, ha)), kLow);
    const float lb = __fadd_rn(__fadd_rn(b, __fsub_rn(kHigh, hb)), kLow);
    hi += __float_as_uint(ha) + __float_as_uint(hb);
    lo += __float_as_uint(la) + __float_as_uint(lb);
  }
  static __device__ __forceinline__ long long value(unsigned lo, unsigned hi, unsigned n) {
    return ((long long)(int)(hi - n * kHighBits) << 8) + (long long)(int)(lo - n * kLowBits);
  }
};

constexpr int kFlushStride = 32 * 8 + 16;  // bytes per coefficient of a warp's flush buffer
constexpr int kFlushBytes = 8 * kFlushStride;

struct DepositSmem {  // dynamic shared memory of k_rec_deposit for tiles of T rows and batches of kDepBatch records
  static size_t bytes(int T, int kDepBatch, bool two) {
    return (size_t)kDepBatch * 16 + (kDepThreads / 32) * kFlushBytes + (size_t)T * 8 +
           (size_t)(kDepBatch / kItem + T) * 4 + 64 + kDepBatch * 4 +
           (two ? (size_t)(kDepThreads / 32) * (kItem / 8) * 32 * 16 : 0);
  }
};

// Orders n0+1 .. n0+KT per pass, coefficient 0 with the first; TWO: two passes, the second starting from
// the powers that the first left in shared memory.
template <int KT, int MINB, int kDepBatch, bool TWO>
__global__ void __launch_bounds__(kDepThreads, MINB)
    k_rec_deposit(const float4 *__restrict__ rec, const RecordHeader *hdr, const unsigned *__restrict__ tile_off,
                  const unsigned *__restrict__ unit_off, int n_tiles, int tile_shift, long long n_rows, int K, int Cpad,
                  unsigned long long *__restrict__ tally, unsigned *flags) {
  extern __shared__ float4 srec[];  // [kDepBatch]
  const int T = 1 << tile_shift;
  unsigned char *flush = reinterpret_cast<unsigned char *>(srec + kDepBatch);
  unsigned *cnt = reinterpret_cast<unsigned *>(flush + (kDepThreads / 32) * kFlushBytes);  // [T] records per row
  unsigned *start = cnt + T;                                                               // [T]
  unsigned *items = start + T;                       // runs: start | length << 12 | row << 19
  unsigned *bucket = items + kDepBatch / kItem + T;  // [16] runs by their number of steps, then places
  unsigned short *idx = reinterpret_cast<unsigned short *>(bucket + 16);  // [kDepBatch] record indices by row
  unsigned short *rank = idx + kDepBatch;                                 // [kDepBatch] place within the row
  float4 *const powers = reinterpret_cast<float4 *>(rank + kDepBatch) + (threadIdx.x >> 5) * (kItem / 8) * 32 + (threadIdx.x & 31);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = lane & 3, g = lane >> 2;
  unsigned char *const my_flush = flush + warp * kFlushBytes;
  const int C = 2 * K + 1;
  const unsigned units = hdr->n_units;
  for (unsigned u = blockIdx.x; u < units; u += gridDim.x) {
    const int tile = block_find(unit_off, n_tiles, u);
    const unsigned lo = tile_off[tile] + (u - unit_off[tile]) * kDepBatch;
    const int n = (int)min((unsigned)kDepBatch, tile_off[tile + 1] - lo);
    // ------------------------------------------------------------- the batch, sorted by row
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += kDepThreads) {
      const unsigned dst = (unsigned)__cvta_generic_to_shared(srec + i);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(rec + lo + i) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll 1
    for (int i = threadIdx.x; i < T; i += kDepThreads) cnt[i] = 0u;
    if (threadIdx.x < 16) bucket[threadIdx.x] = 0u;
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // (small loops throughout: the blocks of an SM are in different phases of this kernel and share its
    // instruction cache)
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += kDepThreads)
      rank[i] = (unsigned short)atomicAdd(&cnt[__float_as_uint(srec[i].x) & (T - 1)], 1u);
    __syncthreads();
    // starts of the rows, and how many runs of how many steps (8 records a step) they make
    if (warp == 0) {
      unsigned carry = 0;
#pragma unroll 1
      for (int b = 0; b < T; b += 32) {
        const int row = b + lane;
        const unsigned c = row < T ? cnt[row] : 0u;
        unsigned v = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned t = __shfl_up_sync(kFull, v, o);
          if (lane >= o) v += t;
        }
        if (row < T) start[row] = carry + v - c;
        carry += __shfl_sync(kFull, v, 31);
        if (c) {
          const unsigned k = (c + kItem - 1) / kItem, len = (c + k - 1) / k;
          atomicAdd(&bucket[(len + 7) / 8], k);
        }
      }
      __syncwarp();
      unsigned v = lane < 16 ? bucket[lane] : 0u;  // longest runs first
      unsigned sum = v;
#pragma unroll
      for (int o = 1; o < 16; o <<= 1) {
        const unsigned t = __shfl_down_sync(kFull, sum, o);
        if (lane + o < 16) sum += t;
      }
      if (lane < 16) bucket[lane] = sum - v;
      if (lane == 0) bucket[15] = sum;  // (no run has 15 steps) their total
    }
    __syncthreads();
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += kDepThreads)
      idx[start[__float_as_uint(srec[i].x) & (T - 1)] + rank[i]] = (unsigned short)i;
    const int n_items = (int)bucket[15];
    __syncthreads();
#pragma unroll 1
    for (int row = threadIdx.x; row < T; row += kDepThreads) {
      const unsigned c = cnt[row];
      if (!c) continue;
      const unsigned k = (c + kItem - 1) / kItem, len = (c + k - 1) / k;
      const unsigned at = atomicAdd(&bucket[(len + 7) / 8], k);
#pragma unroll 1
      for (unsigned q = 0; q < k; ++q)
        items[at + q] = (start[row] + q * len) | (min(len, c - q * len) << 12) | ((unsigned)row << 19);
    }
    __syncthreads();
    // ------------------------------------------------------------- eight runs a warp, four lanes each
    for (int it = warp * 8; it < n_items; it += (kDepThreads / 32) * 8) {
      const unsigned item = it + g < n_items ? items[it + g] : 0u;
      const int s0 = item & 0xFFFu, len = (item >> 12) & 0x7Fu;
      const long long row = ((long long)tile << tile_shift) + (item >> 19);
      const int steps = (int)__reduce_max_sync(kFull, (unsigned)(len + 7) / 8);
      const bool ok = len > 0 && MCR_GUARD(flags, row < n_rows);
      unsigned long long *const dst = tally + (size_t)row * Cpad;
      if (TWO)  // the first pass starts from (cos theta, sin theta), found where the second finds its powers
#pragma unroll 1
        for (int k = 0; k < steps; ++k) {
          const int ia = k * 8 + j, ib = ia + 4;
          float4 a = make_float4(0.f, 0.f, 0.f, 1.f), b = a;
          if (ia < len) a = srec[idx[s0 + ia]];
          if (ib < len) b = srec[idx[s0 + ib]];
          powers[k * 32] = make_float4(a.w, a.z, b.w, b.z);
        }
#pragma unroll 1
      for (int pass = 0; pass < (TWO ? 2 : 1); ++pass) {
        int n0 = pass * KT;
        if (TWO) asm volatile("" : "+r"(n0));  // one copy of the loops for both passes
        SumX sum0, sum_c[KT];
        SumF sum_s[KT];
#pragma unroll 1
        for (int k = 0; k < steps; ++k) {
          const int ia = k * 8 + j, ib = ia + 4;
          float4 a = make_float4(0.f, 0.f, 0.f, 1.f), b = a;
          if (ia < len) a = srec[idx[s0 + ia]];
          if (ib < len) b = srec[idx[s0 + ib]];
          sum0.add(a.y, b.y);
          // (cos n theta, sin n theta) by the complex products of harmonic_row
          float ca = a.w, sa = a.z, cb = b.w, sb = b.z;
          auto turn = [](float &c, float &s, float sx, float sz) {
            const float cn = fmaf(c, sz, -s * sx);
            s = fmaf(s, sz, c * sx);
            c = cn;
          };
          if (TWO) {
            const float4 v = powers[k * 32];
            ca = v.x, sa = v.y, cb = v.z, sb = v.w;
          }
#pragma unroll
          for (int q = 0; q < KT; ++q) {
            sum_c[q].add(__fmul_rn(a.y, ca), __fmul_rn(b.y, cb));
            sum_s[q].add(__fmul_rn(a.y, sa), __fmul_rn(b.y, sb));
            turn(ca, sa, a.z, a.w);
            turn(cb, sb, b.z, b.w);
          }
          if (TWO) powers[k * 32] = make_float4(ca, sa, cb, sb);
        }
        // ----------------------------------------------------------- sums of the four lanes, 16 coefficients a round
        if (!TWO || n0 == 0) {
          sum0.lo += __shfl_xor_sync(kFull, sum0.lo, 1);
          sum0.hi += __shfl_xor_sync(kFull, sum0.hi, 1);
          sum0.lo += __shfl_xor_sync(kFull, sum0.lo, 2);
          sum0.hi += __shfl_xor_sync(kFull, sum0.hi, 2);
          if (j == 0 && ok) atomicAdd(dst, (unsigned long long)SumX::value(sum0.lo, (unsigned)sum0.hi));
        }
        constexpr int kRound = 8;
#pragma unroll
        for (int r = 0; r < 2 * KT; r += kRound) {
          __syncwarp();
#pragma unroll
          for (int c = 0; c < kRound; c += 2) {
            const SumX &x = sum_c[(r + c) / 2];
            const SumF &f = sum_s[(r + c) / 2];
            *reinterpret_cast<uint2 *>(my_flush + c * kFlushStride + lane * 8) = make_uint2(x.lo, (unsigned)x.hi);
            *reinterpret_cast<uint2 *>(my_flush + (c + 1) * kFlushStride + lane * 8) = make_uint2(f.lo, f.hi);
          }
          __syncwarp();
#pragma unroll
          for (int q = 0; q < kRound; q += 4) {
            const uint4 v = *reinterpret_cast<const uint4 *>(my_flush + (q + j) * kFlushStride + g * 32);
            const uint4 w = *reinterpret_cast<const uint4 *>(my_flush + (q + j) * kFlushStride + g * 32 + 16);
            const unsigned tl = v.x + v.z + w.x + w.z, th = v.y + v.w + w.y + w.w;
            const long long t = j & 1 ? SumF::value(tl, th, 8u * steps) : SumX::value(tl, th);
            const int c = 1 + 2 * n0 + r + q + j;
            if (ok && c < C) atomicAdd(dst + c, (unsigned long long)t);
          }
        }
      }
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------------------------- host side
std::mutex g_rec_mu;

// Blocks of `threads` with `smem` bytes that fit on one SM, the kernel opted in to that much.
template <typename K>
cudaError_t rec_blocks_per_sm(K kernel, int threads, size_t smem, int *per_sm) {
  std::lock_guard<std::mutex> lock(g_rec_mu);
  cudaFuncAttributes a;
  cudaError_t e = cudaFuncGetAttributes(&a, kernel);
  if (e != cudaSuccess) return e;
  if ((int)smem > a.maxDynamicSharedSizeBytes) {
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kernel, threads, smem);
  return e != cudaSuccess ? e : (*per_sm < 1 ? cudaErrorInvalidConfiguration : cudaSuccess);
}

cudaError_t sm_count(int *sms) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  return e != cudaSuccess ? e : cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
}

size_t sort_smem(int n_bins) { return (size_t)kSortBatch * 16 + (size_t)n_bins * 8; }

struct Scratch {  // rec_scratch, laid out
  RecordHeader *hdr;
  unsigned *saved_work, *ended;
  unsigned *hist, *off, *cur, *unit_off;                  // bins of the first pass
  unsigned *tile_hist, *tile_off, *tile_cur, *dep_unit_off;  // tiles (the same arrays after a single pass)
  uint4 *saved;  // two buffers, read and written by turns
  size_t zeroed, total;
};
Scratch layout(unsigned char *base, const RecordPlan &pl) {
  Scratch s;
  size_t at = 0;
  auto take = [&](size_t bytes) {
    unsigned char *q = base + at;
    at += (bytes + 255) & ~size_t(255);
    return q;
  };
  s.hdr = reinterpret_cast<RecordHeader *>(take(pl.launches * sizeof(RecordHeader)));
  s.saved_work = reinterpret_cast<unsigned *>(take(4));
  s.ended = reinterpret_cast<unsigned *>(take(4));
  auto words = [&](size_t n) { return reinterpret_cast<unsigned *>(take(n * 4)); };
  const bool two = pl.coarse_shift > 0;
  s.hist = words(pl.n_coarse);
  s.tile_hist = two ? words(pl.n_tiles) : s.hist;
  s.zeroed = at;
  s.off = words(pl.n_coarse + 1);
  s.cur = words((size_t)pl.n_coarse * kCurStride);
  s.unit_off = words(pl.n_coarse + 1);
  s.tile_off = two ? words(pl.n_tiles + 1) : s.off;
  s.tile_cur = two ? words((size_t)pl.n_tiles * kCurStride) : s.cur;
  s.dep_unit_off = two ? words(pl.n_tiles + 1) : s.unit_off;
  s.saved = reinterpret_cast<uint4 *>(take((size_t)pl.lanes * 128));
  s.total = at;
  return s;
}

using DepositKernel = void (*)(const float4 *, const RecordHeader *, const unsigned *, const unsigned *, int, int,
                               long long, int, int, unsigned long long *, unsigned *);
struct DepositChoice {
  DepositKernel kernel;
  int batch;  // records of one unit
  bool two;
};
DepositChoice deposit_kernel(int K) {
  if (K <= 4) return {k_rec_deposit<4, 5, 2048, false>, 2048, false};
  if (K <= 8) return {k_rec_deposit<8, 5, 2048, false>, 2048, false};
  if (K <= 12) return {k_rec_deposit<12, 5, 2048, false>, 2048, false};
  if (K <= 16) return {k_rec_deposit<16, 4, 2560, false>, 2560, false};
  if (K <= 24) return {k_rec_deposit<24, 3, 3072, false>, 3072, false};
  if (K <= 32) return {k_rec_deposit<32, 3, 3072, false>, 3072, false};
  if (K <= 48) return {k_rec_deposit<24, 3, 2304, true>, 2304, true};
  return {k_rec_deposit<32, 3, 2304, true>, 2304, true};
}

}  // namespace

cudaError_t rec_plan(const TransportParams &p, const TransportLaunch &cfg, int64_t rows, uint64_t packets,
                     RecordPlan *out) {
  RecordPlan pl{};
  pl.rows = rows;
  // Tiles of 32 rows (more where they would be over kMaxTiles); over kMaxBins of them are sorted in two
  // passes of about equal width.
  pl.tile_shift = 5;
  while (((rows + (1ll << pl.tile_shift) - 1) >> pl.tile_shift) > kMaxTiles) ++pl.tile_shift;
  if (pl.tile_shift > 12) return cudaErrorInvalidValue;  // (a run's row field has 13 bits)
  pl.n_tiles = (int)((rows + (1ll << pl.tile_shift) - 1) >> pl.tile_shift);
  pl.coarse_shift = 0;
  if (pl.n_tiles > kMaxBins)
    while ((1 << (2 * pl.coarse_shift)) < pl.n_tiles / 8) ++pl.coarse_shift;
  pl.n_coarse = pl.coarse_shift ? (pl.n_tiles + (1 << pl.coarse_shift) - 1) >> pl.coarse_shift : pl.n_tiles;
  // Capacity: 1024 records per packet (one launch holds most runs), 64 MB to 4 GB per buffer.
  uint64_t cap = cfg.record_capacity > 0 ? (uint64_t)cfg.record_capacity : packets * 1024;
  if (cfg.record_capacity <= 0) cap = cap < (1ull << 22) ? (1ull << 22) : cap;
  if (cap > (1ull << 28)) cap = 1ull << 28;
  pl.blocks = (unsigned)((cap + kRecBlock - 1) / kRecBlock);
  const uint64_t want = (packets * kSegmentsPerPacket + (uint64_t)pl.blocks * kRecBlock - 1) / ((uint64_t)pl.blocks * kRecBlock) + 7;
  pl.launches = (unsigned)(want < kMaxLaunches ? want : kMaxLaunches);
  pl.threads = cfg.threads_per_block > 0 ? cfg.threads_per_block : 256;
  int sms = 0, per_sm = 0;
  cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  const size_t smem = (size_t)pl.n_coarse * 4;
  e = p.n_problems > 1 ? rec_blocks_per_sm(k_transport_rec<true>, pl.threads, smem, &per_sm)
                       : rec_blocks_per_sm(k_transport_rec<false>, pl.threads, smem, &per_sm);
  if (e != cudaSuccess) return e;
  if (cfg.blocks_per_sm > 0 && cfg.blocks_per_sm < per_sm) per_sm = cfg.blocks_per_sm;
  pl.lanes = (unsigned)(sms * per_sm * pl.threads);
  if ((e = rec_blocks_per_sm(k_transport_tail, kTailThreads, smem, &per_sm)) != cudaSuccess) return e;
  pl.tail_blocks = sms * per_sm;
  *out = pl;
  return cudaSuccess;
}

size_t rec_buffer_bytes(const RecordPlan &pl) { return (size_t)pl.blocks * kRecBlock * sizeof(float4); }
size_t rec_scratch_bytes(const RecordPlan &pl) { return layout(nullptr, pl).total; }

cudaError_t launch_records(const TransportParams &p, const TransportLaunch &cfg, const RecordPlan &pl, float4 *buf_a,
                           float4 *buf_b, unsigned char *scratch, unsigned long long *tally, cudaStream_t s) {
  const Scratch sc = layout(scratch, pl);
  cudaError_t e = cudaMemsetAsync(scratch, 0, sc.zeroed, s);
  if (e != cudaSuccess) return e;
  int sms = 0, sort1 = 0, sort2 = 0, dep = 0;
  if ((e = sm_count(&sms)) != cudaSuccess) return e;
  const bool two = pl.coarse_shift > 0;
  const size_t smem1 = sort_smem(pl.n_coarse), smem2 = sort_smem(1 << pl.coarse_shift);
  if ((e = rec_blocks_per_sm(k_rec_sort<true>, kSortThreads, smem1, &sort1)) != cudaSuccess) return e;
  if (two && (e = rec_blocks_per_sm(k_rec_sort<false>, kSortThreads, smem2, &sort2)) != cudaSuccess) return e;
  const DepositChoice dc = deposit_kernel(p.K);
  const size_t dep_smem = DepositSmem::bytes(1 << pl.tile_shift, dc.batch, dc.two);
  if ((e = rec_blocks_per_sm(dc.kernel, kDepThreads, dep_smem, &dep)) != cudaSuccess) return e;
  const unsigned capacity = pl.blocks * kRecBlock;
  TransportParams q = p;
  q.order = nullptr;
  q.records = buf_a;
  q.rec_blocks = pl.blocks;
  q.rec_hist = sc.hist;
  q.bin_shift = pl.tile_shift + pl.coarse_shift;
  q.n_bins = pl.n_coarse;
  q.ended = sc.ended;
  q.n_sm = sms;
  q.saved = sc.saved;
  q.n_saved = pl.lanes;
  q.saved_work = sc.saved_work;
  q.tail_max = pl.tail_blocks * (kTailThreads / 32) * kTailPackets;
  q.work_base = pl.lanes;
  // the count at which `work` has launched the last packet
  const unsigned long long to_launch = p.total_packets > q.work_base ? p.total_packets - q.work_base : 0ull;
  const unsigned grid = pl.lanes / pl.threads;
  const size_t smem = (size_t)pl.n_coarse * 4;
  for (unsigned i = 0; i < pl.launches; ++i) {
    RecordHeader *hdr = sc.hdr + i;
    q.rec_hdr = hdr;
    q.rec_prev = i ? hdr - 1 : nullptr;
    if (p.n_problems > 1)
      k_transport_rec<true><<<grid, pl.threads, smem, s>>>(q);
    else
      k_transport_rec<false><<<grid, pl.threads, smem, s>>>(q);
    k_transport_tail<<<pl.tail_blocks, kTailThreads, smem, s>>>(q);
    k_rec_scan<<<1, 1024, 0, s>>>(hdr, two ? &hdr->n_coarse_units : &hdr->n_units, sc.hist, pl.n_coarse,
                                  two ? kSortBatch : dc.batch, sc.off, sc.cur, sc.unit_off, p.work, to_launch);
    k_rec_sort<true><<<sms * sort1, kSortThreads, smem1, s>>>(buf_a, buf_b, hdr, pl.blocks, q.bin_shift, pl.n_coarse,
                                                              sc.cur, capacity, nullptr, nullptr, 0, 0, p.flags);
    if (two) {
      k_rec_count<<<sms * 4, kSortThreads, 0, s>>>(buf_b, hdr, sc.off, sc.unit_off, pl.n_coarse, pl.coarse_shift,
                                                   pl.tile_shift, sc.tile_hist, p.flags);
      k_rec_scan<<<1, 1024, 0, s>>>(hdr, &hdr->n_units, sc.tile_hist, pl.n_tiles, dc.batch, sc.tile_off, sc.tile_cur,
                                    sc.dep_unit_off, p.work, to_launch);
      k_rec_sort<false><<<sms * sort2, kSortThreads, smem2, s>>>(
          buf_b, buf_a, hdr, pl.blocks, pl.tile_shift, 1 << pl.coarse_shift, sc.tile_cur, capacity, sc.off, sc.unit_off, pl.n_coarse, pl.coarse_shift, p.flags);
    }
    dc.kernel<<<sms * dep, kDepThreads, dep_smem, s>>>(two ? buf_a : buf_b, hdr, sc.tile_off, sc.dep_unit_off,
                                                       pl.n_tiles, pl.tile_shift, (long long)pl.rows, p.K, p.Cpad,
                                                       tally, p.flags);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  q.rec_prev = sc.hdr + pl.launches - 1;
  return launch_transport(q, TransportLaunch{0, 0, 1, 0}, s);
}

}  // namespace mcr
