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
//      row of two records at a time (the same complex products as harmonic_row) and sums the rounded
//      products in registers; one reduction per coefficient and run follows.
// Every product is rounded exactly as in the direct deposit and integer addition is exact, so the
// tally is bit-identical to it.
//
// Nothing is read back: a call enqueues more record launches than it is likely to need (one that finds
// nothing to do ends at once) and then one direct transport launch that adopts whatever packets are
// left, so the call stays asynchronous and can be captured into a graph.
//
// 1e7 + 1e7 packets at 256 x 256, K = 32: 871 ms by the direct deposit, 475 to 514 so (a record: transport 10 to
// 14 ps, sort 9 to 10, deposit 22 to 23, the waits of kernels launched ahead included); 1e6 packets at
// 1024 x 1024, K = 64: 211 -> 111 ms.
#include "mcr_records.cuh"

namespace mcr {
namespace {

// ------------------------------------------------------------------------------------- transport
// Bound by instruction issue (80 % of the slots, 9.9 warp instructions and 9.8 ps a segment at 256 x 256
// with the SMs full).  Lanes that stopped at a collision wait (`pend`) until fewer than kFlyMin of the
// warp's lanes are still flying; the scatter, the new flight's random numbers and the launch of new packets
// then run for all waiting lanes together (4e6 packets: 22.0, 21.4, 21.1, 25.4 ms at 8, 10, 12, 20).
constexpr int kFlyMin = 12;

template <bool BATCH>
__global__ void __launch_bounds__(256, BATCH ? 3 : 4) k_transport_rec(const __grid_constant__ TransportParams p) {
  extern __shared__ unsigned hist[];  // records per bin of this block
  after_previous();
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
  __shared__ double w_esc[256], w_rr[256], w_kill[256];  // weights of the lane's packets that escaped, ...
  w_esc[threadIdx.x] = w_rr[threadIdx.x] = w_kill[threadIdx.x] = 0.0;
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
        w_esc[threadIdx.x] += W;
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
      w_kill[threadIdx.x] += W;
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
        w_rr[threadIdx.x] += (double)Wn - (double)W;
        W = Wn;
        ++n.rrs;
      } else {
        w_rr[threadIdx.x] -= W;
        ++n.rrk;
        alive = false;
        return;
      }
    }
    if (flight >= p.max_events) {
      ++n.evl;
      w_kill[threadIdx.x] += W;
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
  // nothing for this kernel to do but launch the first packets, all there are
  w.stop = in_use <= enough && !(fresh && p.total_packets > lanes);
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
              w_esc[threadIdx.x] += W;
            } else if (p.max_events == 0u) {
              ++n.evl;
              w_kill[threadIdx.x] += W;
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
    w.put(p, p.flags, hist, lane, has, row, ts, sx, sz);
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
  n.add_to(p.stats, p.flags, lane, w_esc[threadIdx.x], w_rr[threadIdx.x], w_kill[threadIdx.x]);
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
  after_previous();
  if (*p.flags & kFlagMedium) return;
  const unsigned n_in = p.rec_hdr->n_left;
  if (n_in == 0u || n_in > p.tail_max || *p.work + p.work_base < p.total_packets) return;
  for (int i = threadIdx.x; i < p.n_bins; i += blockDim.x) hist[i] = 0u;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const unsigned n_warps = gridDim.x * (blockDim.x >> 5), in_buf = p.rec_hdr->buf;
  __shared__ double w_esc[256], w_rr[256], w_kill[256];  // weights of the lane's packets that escaped, ...
  w_esc[threadIdx.x] = w_rr[threadIdx.x] = w_kill[threadIdx.x] = 0.0;
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
        w.put(p, p.flags, hist, lane, lane < cnt && t != 0.f && MCR_GUARD(p.flags, isfinite(t)), row, t * qscale, ux, uz);
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
            w_esc[threadIdx.x] += W;
          }
          ended = true;
          continue;
        }
        if (lane == 0) ++n.coll;
        if (nscat >= p.max_scatter) {
          flush();
          if (lane == 0) {
            ++n.scl;
            w_kill[threadIdx.x] += W;
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
                w_rr[threadIdx.x] += (double)Wn - (double)W;
                ++n.rrs;
              }
              W = Wn;
            } else {
              if (lane == 0) {
                w_rr[threadIdx.x] -= W;
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
            w_kill[threadIdx.x] += W;
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
  n.add_to(p.stats, p.flags, lane, w_esc[threadIdx.x], w_rr[threadIdx.x], w_kill[threadIdx.x]);
  __syncthreads();
  if (threadIdx.x == 0) p.rec_hdr->tail_ran = 1u;
  for (int i = threadIdx.x; i < p.n_bins; i += blockDim.x)
    if (hist[i]) atomicAdd(p.rec_hist + i, hist[i]);
}

// ------------------------------------------------------------------------------------- deposit
// Bound by instruction issue: 27 instructions per order and two records, 68 % of the issue slots with the 12 warps
// an SM that the sums' registers leave (FMA pipe 46 %, ALU 28 %, XU 34 % of its cycles); at 256^2, K = 32 some
// 22 ps a record, of which 15 grow with K.
// Orders n0+1 .. n0+KT per pass, coefficient 0 with the first; TWO: two passes, the second starting from
// the powers that the first left in shared memory.
template <int KT, int MINB, int kDepBatch, bool TWO>
__global__ void __launch_bounds__(kDepThreads, MINB)
    k_rec_deposit(const float4 *__restrict__ rec, const RecordHeader *hdr, const unsigned *__restrict__ tile_off,
                  const unsigned *__restrict__ unit_off, int n_tiles, int tile_shift, long long n_rows, int K, int Cpad,
                  unsigned long long *__restrict__ tally, unsigned *flags) {
  extern __shared__ float4 srec[];  // [kDepBatch]
  after_previous();
  const int T = 1 << tile_shift;
  DepositBatch<kDepBatch, false> bt(srec, T);
  const unsigned short *const idx = bt.idx;
  float4 *const powers = reinterpret_cast<float4 *>(bt.rest) + (threadIdx.x >> 5) * (kItem / 8) * 32 + (threadIdx.x & 31);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = lane & 3, g = lane >> 2;
  unsigned char *const my_flush = bt.flush + warp * kFlushBytes;
  const int C = 2 * K + 1;
  const unsigned units = hdr->n_units;
  if (blockIdx.x < units && warp == 0) bt.find(rec, nullptr, tile_off, unit_off, n_tiles, blockIdx.x);
  __syncthreads();
  for (unsigned u = blockIdx.x; u < units; u += gridDim.x) {
    const int tile = (int)bt.unit[0];
    const int n_items = bt.load(rec, nullptr, bt.unit[1], (int)bt.unit[2], T, tile_off, unit_off, n_tiles, u + gridDim.x, units);
    // ------------------------------------------------------------- eight runs a warp, four lanes each
    for (int it = warp * 8; it < n_items; it = bt.next_runs()) {
      const unsigned item = it + g < n_items ? bt.items[it + g] : 0u;
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
using DepositKernel = void (*)(const float4 *, const RecordHeader *, const unsigned *, const unsigned *, int, int,
                               long long, int, int, unsigned long long *, unsigned *);
struct DepositChoice {
  DepositKernel kernel;
  int batch;  // records of one unit
  size_t (*bytes)(int T);
};
template <int KT, int MINB, int B, bool TWO>
DepositChoice deposit_choice() {
  return {k_rec_deposit<KT, MINB, B, TWO>, B, [](int T) {
            return DepositBatch<B, false>::bytes(T) + (TWO ? (size_t)(kDepThreads / 32) * (kItem / 8) * 32 * 16 : 0);
          }};
}
// Orders a pass, blocks per SM that its sums' registers allow, and the batch: as many records as measured best
// (K = 32: 2304 47.4, 2560 46.5, 2816 44.9, 3072 45.1, 3328 48.4, 3840 51.9 ps a segment of the whole run; K = 16:
// 2304 38.8, 2560 38.1, 2816 36.9; two passes of 16 orders at K = 32: 51.6, four of 8: 52.7).
DepositChoice deposit_kernel(int K) {
  if (K <= 4) return deposit_choice<4, 5, 2048, false>();
  if (K <= 8) return deposit_choice<8, 5, 2048, false>();
  if (K <= 12) return deposit_choice<12, 5, 2048, false>();
  if (K <= 16) return deposit_choice<16, 4, 2816, false>();
  if (K <= 24) return deposit_choice<24, 3, 2816, false>();
  if (K <= 32) return deposit_choice<32, 3, 2816, false>();
  if (K <= 48) return deposit_choice<24, 3, 2304, true>();
  return deposit_choice<32, 3, 2304, true>();
}

}  // namespace

cudaError_t rec_plan(const TransportParams &p, const TransportLaunch &cfg, int64_t rows, uint64_t packets,
                     RecordPlan *out) {
  RecordPlan pl{};
  cudaError_t e = plan_records(rows, packets, cfg.record_capacity, &pl);
  if (e != cudaSuccess) return e;
  pl.threads = cfg.threads_per_block > 0 ? cfg.threads_per_block : 256;
  int sms = 0, per_sm = 0;
  if ((e = sm_count(&sms)) != cudaSuccess) return e;
  const size_t smem = (size_t)pl.n_coarse * 4;
  e = p.n_problems > 1 ? rec_blocks_per_sm(k_transport_rec<true>, pl.threads, smem, &per_sm)
                       : rec_blocks_per_sm(k_transport_rec<false>, pl.threads, smem, &per_sm);
  if (e != cudaSuccess) return e;
  if (cfg.blocks_per_sm > 0 && cfg.blocks_per_sm < per_sm) per_sm = cfg.blocks_per_sm;
  pl.lanes = (unsigned)(sms * per_sm * pl.threads);
  if ((e = rec_blocks_per_sm(k_transport_tail, kTailThreads, smem, &per_sm)) != cudaSuccess) return e;
  pl.tail_blocks = sms * per_sm;
  set_launches(&pl, packets);
  *out = pl;
  return cudaSuccess;
}

void rec_set_blocks(RecordPlan *pl, uint64_t packets, unsigned blocks) {
  pl->blocks = blocks;
  set_launches(pl, packets);
}
bool rec_held(const RecordStore &st, uint64_t packets, RecordPlan *pl) {
  if (st.blocks >= pl->blocks) return true;
  // smaller buffers will do where the size wanted was not to be had
  const unsigned least = pl->blocks < kRecLeastBlocks ? pl->blocks : kRecLeastBlocks;
  if (!st.denied || pl->blocks < st.denied || st.blocks < least) return false;
  rec_set_blocks(pl, packets, st.blocks);
  return true;
}
size_t rec_scratch_bytes(const RecordPlan &pl) { return layout(nullptr, pl).total; }

cudaError_t launch_records(const TransportParams &p, const TransportLaunch &cfg, const RecordPlan &pl,
                           unsigned char *buf_a, unsigned char *buf_b, unsigned char *scratch, unsigned long long *tally, RecordInfo *info,
                           cudaStream_t s) {
  const DepositChoice dc = deposit_kernel(p.K);
  const size_t dep_smem = dc.bytes(1 << pl.tile_shift);
  int sms = 0, dep = 0;
  cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  if ((e = rec_blocks_per_sm(dc.kernel, kDepThreads, dep_smem, &dep)) != cudaSuccess) return e;
  TransportParams q = p;
  q.order = nullptr;
  const unsigned grid = pl.lanes / pl.threads;
  const size_t smem = (size_t)pl.n_coarse * 4;
  e = record_chain<false>(
      pl, layout(scratch, pl), RecordBuffers{reinterpret_cast<float4 *>(buf_a), reinterpret_cast<float4 *>(buf_b), nullptr, nullptr}, q, dc.batch, p.work, p.total_packets, p.flags,
      [&]() {
        auto *const rec = p.n_problems > 1 ? k_transport_rec<true> : k_transport_rec<false>;
        if (q.rec_prev)
          launch_ahead(rec, grid, pl.threads, smem, s, q);
        else  // (it follows a memset)
          rec<<<grid, pl.threads, smem, s>>>(q);
        launch_ahead(k_transport_tail, pl.tail_blocks, kTailThreads, smem, s, q);
      },
      [&](const float4 *rec, const float *, const Scratch &sc) {
        launch_ahead(dc.kernel, sms * dep, kDepThreads, dep_smem, s, rec, q.rec_hdr, sc.tile_off, sc.dep_unit_off,
                     pl.n_tiles, pl.tile_shift, (long long)pl.rows, p.K, p.Cpad, tally, p.flags);
        return 1;
      },
      info, s);
  return e != cudaSuccess ? e : launch_transport(q, TransportLaunch{0, 0, 1, 0}, s);
}

}  // namespace mcr
