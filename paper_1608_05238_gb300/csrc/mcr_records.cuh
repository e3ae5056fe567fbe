// mcr_records.cuh -- the parts of the record deposit that the 2D and the 3D form share: the warps' record
// writer, the counters, offsets, sort and batches of the deposit, and the sequence of launches
// (mcr_records.cu has the description).
#pragma once
#include <math_constants.h>

#include <mutex>
#include <utility>

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
constexpr int kSortBatch = 3072;    // records a block sorts at a time (2048: 8 % slower; 4096: 10 %, it spills)
static_assert(kMaxBins % kSortThreads == 0 && kSortBatch % kSortThreads == 0, "every bin and record has a thread");
constexpr int kDepThreads = 128;
constexpr int kItem = 64;           // most records of one run (a group of four lanes, two records each)
constexpr int kCurStride = 8;       // words between cursors: one 32-byte sector each
constexpr unsigned kMaxLaunches = 1024;
constexpr unsigned kSegmentsPerPacket = 4096;  // record launches are enqueued for this many per packet

// The warp's record slots: a block of kRecBlock at a time from the launch's buffer.
struct RecordWriter {
  float4 *out = nullptr;
  float *out_x = nullptr;     // (X: the records' fifth word)
  unsigned fill = kRecBlock;  // slots of the block in use
  bool stop = false;          // the buffer is full (or the launch should pause): write no more
  // what is left of the block holds a sentinel that the sort skips
  __device__ __forceinline__ void pad(int lane) {
    for (unsigned j = fill + lane; j < kRecBlock; j += 32) out[j] = make_float4(__uint_as_float(kRecSentinel), 0.f, 0.f, 1.f);
  }
  __device__ __forceinline__ void room(const RecordParams &p, int lane) {  // for 32 more records; else stop
    if (stop || fill + 32 <= kRecBlock) return;
    pad(lane);
    unsigned b = 0;
    if (lane == 0) b = atomicAdd(&p.rec_hdr->blocks, 1u);
    b = __shfl_sync(kFull, b, 0);
    stop = b >= p.rec_blocks;
    fill = stop ? kRecBlock : 0u;
    if (!stop) {
      out = p.records + (size_t)b * kRecBlock;
      out_x = p.records_x + (size_t)b * kRecBlock;
    }
  }
  // the warp's records of one step, in its lanes' order
  template <bool X = false>
  __device__ __forceinline__ void put(const RecordParams &p, unsigned *flags, unsigned *hist, int lane, bool has,
                                      unsigned row, float ts, float u0, float u1, float u2 = 0.f) {
    const unsigned who = __ballot_sync(kFull, has);
    if (has && MCR_GUARD(flags, (row >> p.bin_shift) < (unsigned)p.n_bins)) {
      const unsigned at = fill + __popc(who & ((1u << lane) - 1u));
      out[at] = make_float4(__uint_as_float(row), ts, u0, u1);
      if (X) out_x[at] = u2;
      atomicAdd(&hist[row >> p.bin_shift], 1u);
    }
    fill += __popc(who);
  }
};

// A lane's run counters, added to the run's by the warp at the end.
struct PacketCounts {
  unsigned launch = 0, flight = 0, coll = 0, seg = 0, esc = 0, rrk = 0, rrs = 0, scl = 0, evl = 0;
  int w_launch = 0;  // |W0| = 1
  __device__ void add_to(DevStats *st, unsigned *flags, int lane, double w_esc, double w_rr, double w_kill) const {
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
    addw(&st->escaped_w, w_esc);
    addw(&st->rr_net_w, w_rr);
    addw(&st->killed_w, w_kill);
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

// The kernels of a run are launched ahead: the blocks of one take the places that those of the one before
// free, and wait here for its end.  Nothing of global memory is touched before this.
// (What a small run spends is mostly the gaps between its 30 to 60 kernels: 1e5 packets into 32^2 pixels
// 1690 -> 1539 us, 1e5 packets into 12^3 voxels, L = 5, 577 -> 475 us.)
__device__ __forceinline__ void after_previous() {
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();  // (the next kernel's blocks wait for this one's end in turn)
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
  after_previous();
  if (threadIdx.x == 0) {
    if (*launched < n_packets) {
      hdr->fresh = 1u;
      hdr->unlaunched = n_packets - *launched;
    }
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
// 9 to 10 ps a record and pass (the copy rate would allow 4.7): the shared-memory and cursor wavefronts take
// 58 to 68 % of the load-store slots, and a block's phases wait at its barriers (two blocks an SM; writing each
// record straight to its place took 21 ps, its 16 bytes being half a sector).
// X: records of five words, the fifth in arrays of its own (in_x, sorted_x).
template <bool FIRST, bool X = false>
__global__ void __launch_bounds__(kSortThreads, 2)
    k_rec_sort(const float4 *__restrict__ in, const float *__restrict__ in_x, float4 *__restrict__ sorted,
               float *__restrict__ sorted_x, const RecordHeader *hdr, unsigned max_blocks, int shift, int n_bins,
               unsigned *cursor, unsigned capacity, const unsigned *__restrict__ coarse_off,
               const unsigned *__restrict__ coarse_unit_off, int n_coarse, int coarse_shift, unsigned *flags) {
  after_previous();
  constexpr int kPer = kSortBatch / kSortThreads;
  extern __shared__ float4 srec[];                                  // [kSortBatch]
  unsigned *cnt = reinterpret_cast<unsigned *>(srec + kSortBatch);  // [n_bins] counts, then local starts
  unsigned *delta = cnt + n_bins;                                   // [n_bins] global place minus local place
  float *srec_x = reinterpret_cast<float *>(delta + n_bins);        // X: [kSortBatch]
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
    float r_x[kPer];
    unsigned bin[kPer], rank[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const unsigned i = lo + k * kSortThreads + threadIdx.x;
      r[k] = i < hi ? __ldcs(in + i) : make_float4(__uint_as_float(kRecSentinel), 0.f, 0.f, 0.f);
      if (X) r_x[k] = i < hi ? __ldcs(in_x + i) : 0.f;
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
      if (bin[k] != kRecSentinel) {
        srec[cnt[bin[k]] + rank[k]] = r[k];
        if (X) srec_x[cnt[bin[k]] + rank[k]] = r_x[k];
      }
    __syncthreads();
    for (unsigned i = threadIdx.x; i < total; i += kSortThreads) {
      const float4 v = srec[i];
      const unsigned at = delta[(__float_as_uint(v.x) >> shift) - bin0] + i;
      if (MCR_GUARD(flags, at < capacity)) {
        sorted[at] = v;
        if (X) sorted_x[at] = srec_x[i];
      }
    }
    __syncthreads();
  }
}

// Counts per tile of the coarse-sorted records, before the second pass.  (The kernel just ahead writes rec
// while this one's blocks may already be resident, so it is read by L2 loads and not by the read-only path,
// which wants data that is constant for as long as the kernel lives.)
__global__ void __launch_bounds__(kSortThreads) k_rec_count(const float4 *rec, const RecordHeader *hdr,
                                                            const unsigned *__restrict__ coarse_off,
                                                            const unsigned *__restrict__ coarse_unit_off, int n_coarse,
                                                            int coarse_shift, int tile_shift, unsigned *tile_hist,
                                                            unsigned *flags) {
  __shared__ unsigned cnt[kMaxBins];
  after_previous();
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
      const unsigned b = (__float_as_uint(__ldcg(&rec[i].x)) >> tile_shift) - bin0;
      if (MCR_GUARD(flags, b < (unsigned)nb)) atomicAdd(&cnt[b], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nb; i += kSortThreads)
      if (cnt[i]) atomicAdd(tile_hist + bin0 + i, cnt[i]);
    __syncthreads();
  }
}

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

// The last i < n with off[i] <= u (off nondecreasing, off[0] = 0), found by one warp.
__device__ __forceinline__ int warp_find(const unsigned *__restrict__ off, int n, unsigned u) {
  const int lane = threadIdx.x & 31;
  int a = 0;
  while (n > 1) {
    const int step = (n + 31) / 32;
    const bool le = lane * step < n && __ldg(off + a + lane * step) <= u;
    const int k = (__popc(__ballot_sync(kFull, le)) - 1) * step;
    a += k;
    n = min(step, n - k);
  }
  return a;
}

// One unit of a deposit: a batch of at most B records of one tile of T rows, in shared memory, its records'
// indices sorted by row and cut into runs of at most kItem records of one row.  The runs are listed longest
// first and taken by eight, one warp after the other, so that the eight have about equal lengths and the
// warps end at about the same time.
// (Of a unit's 60,000 cycles at K = 32 and 31,000 at K = 16, 11,000 went into its preparation, where a warp
// waited for one answer after the other, and 13 % of the rest were spent waiting for the slowest warp.  So a
// thread's rows and ranks stay in registers, the unit to come is found and fetched into L2 beside the scan,
// the runs are listed beside the index and taken as warps get to them: 256^2, K = 32, 47.3 -> 44.9 ps a
// segment in all, K = 16 37.1 -> 36.8, 1024^2, K = 64, 92.5 -> 84.7 with tiles of 64 rows.)
// (Small loops: the blocks of an SM are in different phases of the deposit and share its instruction cache.)
template <int B, bool X>
struct DepositBatch {
  static constexpr int kPer = B / kDepThreads;
  static_assert(B % kDepThreads == 0 && B <= 4096, "a run's first index has 12 bits");
  static_assert(B % (4 * kItem) == 0, "what lies behind the runs is aligned to 16 bytes");
  float4 *rec;             // [B]
  float *rec_x;            // X: [B]
  unsigned char *flush;    // [warps][kFlushBytes]
  unsigned *cnt, *start;   // [T] records per row, first index of the row
  unsigned *items;         // runs: start | length << 12 | row << 19
  unsigned *bucket;        // [16] runs by their number of steps, then places; [16] runs taken
  unsigned *unit;          // the unit to come: tile, first record, records
  unsigned short *idx;     // [B] record indices by row
  void *rest;
  static size_t bytes(int T) {
    return (size_t)B * (X ? 20 : 16) + (kDepThreads / 32) * kFlushBytes + (size_t)T * 8 + (size_t)(B / kItem + T) * 4 + 80 +
           B * 2;
  }
  __device__ __forceinline__ DepositBatch(float4 *smem, int T) {
    rec = smem;
    rec_x = reinterpret_cast<float *>(rec + B);
    flush = reinterpret_cast<unsigned char *>(rec_x + (X ? B : 0));
    cnt = reinterpret_cast<unsigned *>(flush + (kDepThreads / 32) * kFlushBytes);
    start = cnt + T;
    items = start + T;
    bucket = items + B / kItem + T;
    unit = bucket + 17;
    idx = reinterpret_cast<unsigned short *>(bucket + 20);
    rest = idx + B;
  }
  // Unit u, found by one warp and fetched into L2.
  __device__ __forceinline__ void find(const float4 *src, const float *src_x, const unsigned *__restrict__ tile_off,
                                       const unsigned *__restrict__ unit_off, int n_tiles, unsigned u) {
    const int t = warp_find(unit_off, n_tiles, u);
    if ((threadIdx.x & 31) != 0) return;
    const unsigned lo = tile_off[t] + (u - unit_off[t]) * B, n = min((unsigned)B, tile_off[t + 1] - lo);
    unit[0] = (unsigned)t;
    unit[1] = lo;
    unit[2] = n;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src + lo), "r"(n * 16u) : "memory");
    if (X) {  // (whole 16 bytes: the buffer is a multiple of them)
      const unsigned a = lo & ~3u, e = (lo + n + 3u) & ~3u;
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src_x + a), "r"((e - a) * 4u) : "memory");
    }
  }
  // Loads and sorts the n records from lo on; returns the number of runs.  u_next: the unit to come, if below
  // `units`.
  __device__ __forceinline__ int load(const float4 *src, const float *src_x, unsigned lo, int n, int T,
                                      const unsigned *__restrict__ tile_off, const unsigned *__restrict__ unit_off,
                                      int n_tiles, unsigned u_next, unsigned units) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += kDepThreads) {
      const unsigned dst = (unsigned)__cvta_generic_to_shared(rec + i);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src + lo + i) : "memory");
      if (X) {
        const unsigned dst_x = (unsigned)__cvta_generic_to_shared(rec_x + i);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst_x), "l"(src_x + lo + i) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll 1
    for (int i = threadIdx.x; i < T; i += kDepThreads) cnt[i] = 0u;
    if (threadIdx.x < 16) bucket[threadIdx.x] = 0u;
    if (threadIdx.x == 16) bucket[16] = (kDepThreads / 32) * 8;
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    unsigned key[kPer];  // row | rank << 16
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int i = k * kDepThreads + (int)threadIdx.x;
      key[k] = i < n ? __float_as_uint(rec[i].x) & (T - 1) : 0u;
    }
#pragma unroll
    for (int k = 0; k < kPer; ++k)
      if (k * kDepThreads + (int)threadIdx.x < n) key[k] |= atomicAdd(&cnt[key[k]], 1u) << 16;
    __syncthreads();
    if (warp == 0) {  // starts of the rows
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
      }
    } else if (warp == 1) {  // how many runs of how many steps (8 records a step) they make
#pragma unroll 1
      for (int row = lane; row < T; row += 32) {
        const unsigned c = cnt[row];
        if (!c) continue;
        const unsigned k = (c + kItem - 1) / kItem, len = (c + k - 1) / k;
        atomicAdd(&bucket[(len + 7) / 8], k);
      }
      __syncwarp();
      const unsigned v = lane < 16 ? bucket[lane] : 0u;  // longest runs first
      unsigned sum = v;
#pragma unroll
      for (int o = 1; o < 16; o <<= 1) {
        const unsigned t = __shfl_down_sync(kFull, sum, o);
        if (lane + o < 16) sum += t;
      }
      const unsigned total = __shfl_sync(kFull, sum, 0);
      if (lane < 16) bucket[lane] = lane == 15 ? total : sum - v;  // (no run has 15 steps: there stands the total)
    } else if (warp == 2 && u_next < units) {
      find(src, src_x, tile_off, unit_off, n_tiles, u_next);
    }
    __syncthreads();
    if (warp == 3) {
#pragma unroll 1
      for (int row = lane; row < T; row += 32) {
        const unsigned c = cnt[row];
        if (!c) continue;
        const unsigned k = (c + kItem - 1) / kItem, len = (c + k - 1) / k;
        const unsigned at = atomicAdd(&bucket[(len + 7) / 8], k);
#pragma unroll 1
        for (unsigned q = 0; q < k; ++q)
          items[at + q] = (start[row] + q * len) | (min(len, c - q * len) << 12) | ((unsigned)row << 19);
      }
    }
    const int n_items = (int)bucket[15];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int i = k * kDepThreads + (int)threadIdx.x;
      if (i < n) idx[start[key[k] & 0xFFFFu] + (key[k] >> 16)] = (unsigned short)i;
    }
    __syncthreads();
    return n_items;
  }
  // The next eight runs for this warp.
  __device__ __forceinline__ int next_runs() const {
    int it = 0;
    if ((threadIdx.x & 31) == 0) it = (int)atomicAdd(&bucket[16], 8u);
    return __shfl_sync(kFull, it, 0);
  }
};
static_assert(kDepThreads == 128, "four warps share the steps of DepositBatch::load");

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

size_t sort_smem(int n_bins, bool x) { return (size_t)kSortBatch * (x ? 20 : 16) + (size_t)n_bins * 8; }

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

// The most packets that the tail takes.
unsigned tail_packets(const RecordPlan &pl) { return (unsigned)pl.tail_blocks * (kTailThreads / 32) * kTailPackets; }

// Tiles, passes and buffer of a run of `packets` into `rows` tally rows.
cudaError_t plan_records(int64_t rows, uint64_t packets, long long capacity, RecordPlan *out) {
  RecordPlan pl{};
  pl.rows = rows;
  // Tiles of 32 rows, 64 where one pass of the sort does not hold so many (half the bins, runs of twice the
  // length: 1024^2, K = 64, 110 -> 100 ps a segment; 256^2, K = 32, 49.9 -> 53), more where they would be over
  // kMaxTiles; over kMaxBins of them are sorted in two passes of about equal width.
  pl.tile_shift = rows > ((int64_t)kMaxBins << 5) ? 6 : 5;
  while (((rows + (1ll << pl.tile_shift) - 1) >> pl.tile_shift) > kMaxTiles) ++pl.tile_shift;
  if (pl.tile_shift > 12) return cudaErrorInvalidValue;  // (a run's row field has 13 bits)
  pl.n_tiles = (int)((rows + (1ll << pl.tile_shift) - 1) >> pl.tile_shift);
  pl.coarse_shift = 0;
  if (pl.n_tiles > kMaxBins)
    while ((1 << (2 * pl.coarse_shift)) < pl.n_tiles / 8) ++pl.coarse_shift;
  pl.n_coarse = pl.coarse_shift ? (pl.n_tiles + (1 << pl.coarse_shift) - 1) >> pl.coarse_shift : pl.n_tiles;
  // Capacity: 1024 records per packet (one launch holds most runs), 64 MB to 4 GB per buffer.
  uint64_t cap = capacity > 0 ? (uint64_t)capacity : packets * 1024;
  if (capacity <= 0) cap = cap < (1ull << 22) ? (1ull << 22) : cap;
  if (cap > (1ull << 28)) cap = 1ull << 28;
  pl.blocks = (unsigned)((cap + kRecBlock - 1) / kRecBlock);
  *out = pl;
  return cudaSuccess;
}

// The record launches to enqueue, once lanes and tail_blocks are known: those that end on a full buffer, one
// for each halving of the packets in use down to what the tail takes, one more for a buffer left part full.
// The five kernels of a launch with nothing left to do took about 8 us (20,000 packets into 12^3 voxels:
// two runs in 1370 us with eleven launches each, 1212 us with six; launched ahead 1037 us, all direct 1184 us).
void set_launches(RecordPlan *pl, uint64_t packets) {
  const uint64_t slots = (uint64_t)pl->blocks * kRecBlock;
  uint64_t n = (packets * kSegmentsPerPacket + slots - 1) / slots;
  if (n < 4) n = 4;
  for (uint64_t r = packets < pl->lanes ? packets : pl->lanes; r > tail_packets(*pl); r /= 2) ++n;
  ++n;
  pl->launches = (unsigned)(n < kMaxLaunches ? n : kMaxLaunches);
}

size_t record_slots(const RecordPlan &pl) { return (size_t)pl.blocks * kRecBlock; }

struct RecordBuffers {
  float4 *a, *b;
  float *a_x, *b_x;  // X: the fifth words
};

// Launches a kernel ahead of the end of the kernel before it in the stream (see after_previous()).
template <typename... P, typename... A>
void launch_ahead(void (*kernel)(P...), int grid, int block, size_t smem, cudaStream_t s, A &&...args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3((unsigned)grid);
  c.blockDim = dim3((unsigned)block);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = &at;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, kernel, std::forward<A>(args)...);  // (the caller asks cudaGetLastError)
}

// The launches of a run: transport() launches the transport and its tail with the fields of q set here,
// deposit(records, their fifth words, scratch) the deposit of the sorted records, and returns its number of
// kernels.  On return q is set for a direct transport that adopts the packets left.
template <bool X, typename Transport, typename Deposit>
cudaError_t record_chain(const RecordPlan &pl, const Scratch &sc, const RecordBuffers &buf, RecordParams &q, int dep_batch,
                         const unsigned long long *work, unsigned long long total_packets, unsigned *flags,
                         Transport transport, Deposit deposit, RecordInfo *info, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(sc.hdr, 0, sc.zeroed, s);
  if (e != cudaSuccess) return e;
  int sms = 0, sort1 = 0, sort2 = 0;
  if ((e = sm_count(&sms)) != cudaSuccess) return e;
  const bool two = pl.coarse_shift > 0;
  const size_t smem1 = sort_smem(pl.n_coarse, X), smem2 = sort_smem(1 << pl.coarse_shift, X);
  if ((e = rec_blocks_per_sm(k_rec_sort<true, X>, kSortThreads, smem1, &sort1)) != cudaSuccess) return e;
  if (two && (e = rec_blocks_per_sm(k_rec_sort<false, X>, kSortThreads, smem2, &sort2)) != cudaSuccess) return e;
  const unsigned capacity = (unsigned)record_slots(pl);
  q.records = buf.a;
  q.records_x = buf.a_x;
  q.rec_blocks = pl.blocks;
  q.rec_hist = sc.hist;
  q.bin_shift = pl.tile_shift + pl.coarse_shift;
  q.n_bins = pl.n_coarse;
  q.ended = sc.ended;
  q.n_sm = sms;
  q.saved = sc.saved;
  q.n_saved = pl.lanes;
  q.saved_work = sc.saved_work;
  q.tail_max = tail_packets(pl);
  q.work_base = pl.lanes;
  // the count at which `work` has launched the last packet
  const unsigned long long to_launch = total_packets > q.work_base ? total_packets - q.work_base : 0ull;
  for (unsigned i = 0; i < pl.launches; ++i) {
    RecordHeader *hdr = sc.hdr + i;
    q.rec_hdr = hdr;
    q.rec_prev = i ? hdr - 1 : nullptr;
    transport();
    launch_ahead(k_rec_scan, 1, 1024, 0, s, hdr, two ? &hdr->n_coarse_units : &hdr->n_units, sc.hist, pl.n_coarse,
                 two ? kSortBatch : dep_batch, sc.off, sc.cur, sc.unit_off, work, to_launch);
    launch_ahead(k_rec_sort<true, X>, sms * sort1, kSortThreads, smem1, s, buf.a, buf.a_x, buf.b, buf.b_x, hdr,
                 pl.blocks, q.bin_shift, pl.n_coarse, sc.cur, capacity, nullptr, nullptr, 0, 0, flags);
    if (two) {
      launch_ahead(k_rec_count, sms * 4, kSortThreads, 0, s, buf.b, hdr, sc.off, sc.unit_off, pl.n_coarse,
                   pl.coarse_shift, pl.tile_shift, sc.tile_hist, flags);
      launch_ahead(k_rec_scan, 1, 1024, 0, s, hdr, &hdr->n_units, sc.tile_hist, pl.n_tiles, dep_batch, sc.tile_off,
                   sc.tile_cur, sc.dep_unit_off, work, to_launch);
      launch_ahead(k_rec_sort<false, X>, sms * sort2, kSortThreads, smem2, s, buf.b, buf.b_x, buf.a, buf.a_x, hdr,
                   pl.blocks, pl.tile_shift, 1 << pl.coarse_shift, sc.tile_cur, capacity, sc.off, sc.unit_off,
                   pl.n_coarse, pl.coarse_shift, flags);
    }
    info->kernels += 4 + (two ? 3 : 0) + deposit(two ? buf.a : buf.b, two ? buf.a_x : buf.b_x, sc);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  q.rec_prev = sc.hdr + pl.launches - 1;
  info->last = q.rec_prev;
  info->passes = two ? 2 : 1;
  return cudaSuccess;
}

}  // namespace
}  // namespace mcr
