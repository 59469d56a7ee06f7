// Path weights (Claim 1, Alg. 1), the guide table of the CDF search, and the
// sampler with CheckMotif / ListCount and the reduction of X (Alg. 2-5).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <utility>
#include <vector>

#include "tc_internal.cuh"

namespace tc {

// ---------------------------------------------------------------------------
// Weights (Claim 1, Alg. 1): w_e = d1 * d3 for every canonical edge
// e = (u, v, t), the sizes of the window of u's alpha1 list and of v's alpha3
// list, and their exact prefix sum.
//
// The four binary searches per edge of Alg. 1 start from anchors built with
// the lists (tc_graph::x_in, x_out, out2in; independent of delta): each
// window bound is found by a galloping search (doubling steps, then
// bisection) from a position where the list reaches time t, so a window of
// d entries costs O(log d) probes near the anchor instead of O(log deg)
// probes over the whole list.  The anchors' range words give the list's
// bounds (no random load of the destination's offsets), and an exact anchor
// (the list's lower bound of t) is itself the window's bound at t in strict
// mode.  The u side of consecutive edges (one source vertex in time order)
// searches the same list at increasing positions.
//
// The weights pass also sums w over each tile of kWTile edges, the first
// level of the reduce-then-scan that writes the prefix (so w is read once
// more, not twice).
//
// A wedge anchor (3-vertex motif) has one window, at u or at v; the other
// side is the dummy [0, 1), so w_e is the size of that window.

// Resident blocks per SM the weights kernel is compiled for (caps its registers).
#ifndef TC_WEIGHTS_MIN_BLOCKS
#define TC_WEIGHTS_MIN_BLOCKS 8
#endif

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

constexpr int kWThreads = 256;
constexpr int kWItems = 8;
constexpr int kWTile = kWThreads * kWItems;  // edges per tile: the scan's tile

// The window of list [s, f) around time t (beta < 0: before, else after;
// strict or closed at t) as positions [*lo, *hi), searched from an anchor a
// with lower_bound(t) <= a <= upper_bound(t).
template <class TimeAt>
__device__ __forceinline__ void window_from(uint32_t s, uint32_t f, uint32_t a, int beta, int closed, int64_t t,
                                            int64_t delta, TimeAt tt, uint32_t* lo, uint32_t* hi) {
  if (beta < 0) {
    *hi = closed ? gallop<true, int64_t>(s, f, a, t, tt) : gallop<false, int64_t>(s, f, a, t, tt);
    *lo = gallop<false, int64_t>(s, f, *hi, sat_sub(t, delta), tt);
  } else {
    *lo = closed ? gallop<false, int64_t>(s, f, a, t, tt) : gallop<true, int64_t>(s, f, a, t, tt);
    *hi = gallop<true, int64_t>(s, f, *lo, sat_add(t, delta), tt);
  }
}

struct WeightsArgs {
  const OutEdge* out_e;
  const InEdge* in_e;
  const uint32_t* out_off;
  const uint32_t* in_off;
  const uint32_t* out_t32;
  const uint32_t* in_t32;
  const uint2* x_in;  // anchors and their range words
  const uint2* x_out;
  const uint2* out2in;
  const uint32_t* r_self;  // range word of the edge in u's out-list
  int64_t tmin;
  uint64_t m;
  int64_t delta;
  int alpha1, alpha3, beta1, beta3, closed;
  EdgeWin* win;
  uint64_t* w;
  uint64_t* tile_sums;  // sum of w over each tile
  uint32_t* err;
};

// Graphs without 32-bit list times.  Window of side alpha (< 0: the vertex's
// in-list, > 0: its out-list) of canonical edge i = (x, ., t), searched from
// anchor a.
__device__ __forceinline__ void side_window(const WeightsArgs& A, int alpha, int beta, int32_t x, uint32_t a,
                                            int64_t t, uint32_t* lo, uint32_t* hi) {
  if (alpha < 0) {
    auto tt = [&](uint32_t p) -> int64_t { return A.in_e[p].t; };
    window_from(__ldg(A.in_off + x), __ldg(A.in_off + x + 1), a, beta, A.closed, t, A.delta, tt, lo, hi);
  } else {
    auto tt = [&](uint32_t p) -> int64_t { return A.out_e[p].t; };
    window_from(__ldg(A.out_off + x), __ldg(A.out_off + x + 1), a, beta, A.closed, t, A.delta, tt, lo, hi);
  }
}

// Block b takes tile b: the windows and w of its kWTile edges (coalesced:
// edge b kWTile + j 256 + thread), and the tile's sum of w.
__global__ void __launch_bounds__(kWThreads, TC_WEIGHTS_MIN_BLOCKS) k_weights(const __grid_constant__ WeightsArgs A) {
  __shared__ unsigned long long s_warp[kWThreads / 32];
  __shared__ uint32_t s_ovf;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid == 0) s_ovf = 0;
  const uint64_t base = (uint64_t)blockIdx.x * kWTile;
  unsigned long long sum = 0;
  bool ovf = false;
#pragma unroll 1
  for (int j = 0; j < kWItems; j++) {
    const uint64_t i = base + (uint64_t)j * kWThreads + tid;
    if (i >= A.m) break;
    const OutEdge e = A.out_e[i];
    uint32_t lo1 = 0, hi1 = 1, lo3 = 0, hi3 = 1;  // a wedge's unused side is [0, 1)
    // anchors: u's in-list (x_in) or the edge itself in u's out-list; the
    // edge itself in v's in-list (out2in) or v's out-list (x_out)
    if (A.alpha1 != 0)
      side_window(A, A.alpha1, A.beta1, e.src, A.alpha1 < 0 ? __ldg(&A.x_in[i].x) : (uint32_t)i, e.t, &lo1, &hi1);
    if (A.alpha3 != 0)
      side_window(A, A.alpha3, A.beta3, e.dst, A.alpha3 < 0 ? __ldg(&A.out2in[i].x) : __ldg(&A.x_out[i].x), e.t, &lo3,
                  &hi3);
    EdgeWin r;
    r.lo1 = lo1;
    r.d1 = hi1 - lo1;
    r.lo3 = lo3;
    r.d3 = hi3 - lo3;
    A.win[i] = r;
    const unsigned long long wv = (unsigned long long)r.d1 * (unsigned long long)r.d3;
    A.w[i] = wv;
    if (sum + wv < sum) ovf = true;
    sum += wv;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, sum, o);
    if (sum + y < sum) ovf = true;
    sum += y;
  }
  if (lane == 0) s_warp[wid] = sum;
  if (ovf) s_ovf = 1;
  __syncthreads();
  if (tid == 0) {
    unsigned long long t = 0;
    bool o2 = s_ovf != 0;
    for (int v = 0; v < kWThreads / 32; v++) {
      if (t + s_warp[v] < t) o2 = true;
      t += s_warp[v];
    }
    A.tile_sums[blockIdx.x] = t;
    if (o2) atomicOr(A.err, kErrOverflow);
  }
}

// Window of one side on the 32-bit list times, searched from anchor a: the
// list [s, f) from the anchor's range word rw (the offsets of x's list are
// read only where a field is saturated).  exact: a is the list's lower bound
// of t (x_in, x_out), so "time >= t" needs no probe.
// The vertex x (the edge's source, or its destination when dst_side) is
// read from the edge record only then.
__device__ __forceinline__ void side_window_rw(const WeightsArgs& A, int alpha, int beta, uint64_t i, bool dst_side,
                                               uint2 anchor, bool exact, int64_t t, uint32_t* lo, uint32_t* hi) {
  const uint32_t a = anchor.x, rw = anchor.y;
  const uint32_t* off = alpha < 0 ? A.in_off : A.out_off;
  uint32_t s = a - (rw >> 16), f = a + (rw & 0xFFFFu);
  if ((rw >> 16) == kRangeCap || (rw & 0xFFFFu) == kRangeCap) {
    const int2 sd = __ldg(reinterpret_cast<const int2*>(A.out_e + i));  // (src, dst)
    const int32_t x = dst_side ? sd.y : sd.x;
    if ((rw >> 16) == kRangeCap) s = __ldg(off + x);
    if ((rw & 0xFFFFu) == kRangeCap) f = __ldg(off + x + 1);
  }
  const uint32_t* t32 = alpha < 0 ? A.in_t32 : A.out_t32;
  auto tt = [&](uint32_t p) -> int64_t { return (int64_t)__ldg(t32 + p) + A.tmin; };
  if (beta < 0) {
    *hi = (exact && !A.closed) ? a : (A.closed ? gallop<true, int64_t>(s, f, a, t, tt) : gallop<false, int64_t>(s, f, a, t, tt));
    *lo = gallop<false, int64_t>(s, f, *hi, sat_sub(t, A.delta), tt);
  } else {
    *lo = (exact && A.closed) ? a : (A.closed ? gallop<false, int64_t>(s, f, a, t, tt) : gallop<true, int64_t>(s, f, a, t, tt));
    *hi = gallop<true, int64_t>(s, f, *lo, sat_add(t, A.delta), tt);
  }
}

// Block b takes tile b (coalesced: edge b kWTile + j 256 + thread) on the
// 32-bit list times: the edge's time from the 32-bit out-list times, the
// list bounds from the anchors' range words (the edge record and the
// offsets are read only where a word is saturated), an exact anchor's
// bound without a probe, the windows and w written with streaming stores,
// and the tile's sum of w.
__global__ void __launch_bounds__(kWThreads, TC_WEIGHTS_MIN_BLOCKS)
    k_weights_rw(const __grid_constant__ WeightsArgs A) {
  __shared__ unsigned long long s_warp[kWThreads / 32];
  __shared__ uint32_t s_ovf;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid == 0) s_ovf = 0;
  const uint64_t base = (uint64_t)blockIdx.x * kWTile;
  unsigned long long sum = 0;
  bool ovf = false;
#pragma unroll 1
  for (int j = 0; j < kWItems; j++) {
    const uint64_t i = base + (uint64_t)j * kWThreads + tid;
    if (i >= A.m) break;
    const int64_t t = (int64_t)__ldg(A.out_t32 + i) + A.tmin;  // the edge's time (4 bytes, not the record)
    uint32_t lo1 = 0, hi1 = 1, lo3 = 0, hi3 = 1;
    // anchors: u's in-list (x_in, exact) or the edge itself in u's out-list;
    // the edge itself in v's in-list (out2in) or v's out-list (x_out, exact)
    if (A.alpha1 < 0)
      side_window_rw(A, -1, A.beta1, i, false, __ldg(A.x_in + i), true, t, &lo1, &hi1);
    else if (A.alpha1 > 0)
      side_window_rw(A, 1, A.beta1, i, false, make_uint2((uint32_t)i, __ldg(A.r_self + i)), false, t, &lo1, &hi1);
    if (A.alpha3 < 0)
      side_window_rw(A, -1, A.beta3, i, true, __ldg(A.out2in + i), false, t, &lo3, &hi3);
    else if (A.alpha3 > 0)
      side_window_rw(A, 1, A.beta3, i, true, __ldg(A.x_out + i), true, t, &lo3, &hi3);
    __stcs(reinterpret_cast<uint4*>(A.win + i), make_uint4(lo1, hi1 - lo1, lo3, hi3 - lo3));
    const unsigned long long wv = (unsigned long long)(hi1 - lo1) * (unsigned long long)(hi3 - lo3);
    __stcs(reinterpret_cast<unsigned long long*>(A.w + i), wv);
    if (sum + wv < sum) ovf = true;
    sum += wv;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, sum, o);
    if (sum + y < sum) ovf = true;
    sum += y;
  }
  if (lane == 0) s_warp[wid] = sum;
  if (ovf) s_ovf = 1;
  __syncthreads();
  if (tid == 0) {
    unsigned long long t = 0;
    bool o2 = s_ovf != 0;
    for (int v = 0; v < kWThreads / 32; v++) {
      if (t + s_warp[v] < t) o2 = true;
      t += s_warp[v];
    }
    A.tile_sums[blockIdx.x] = t;
    if (o2) atomicOr(A.err, kErrOverflow);
  }
}

static uint64_t weights_tiles(uint64_t m) { return (m + kWTile - 1) / kWTile; }

// Scratch of launch_weights_scan: w (unless the caller keeps it), the tile
// sums, and the tile sums' own scan levels.
size_t weights_scan_scratch_bytes(uint64_t m) {
  const uint64_t T = weights_tiles(m) ? weights_tiles(m) : 1;
  return align256(8 * (m ? m : 1)) + align256(8 * T) + align256(8 * (scan_u64_scratch_words(T) + 1));
}

tc_status launch_weights_scan(const tc_graph* g, const Plan& plan, int64_t delta, EdgeWin* win, uint64_t* prefix,
                              uint64_t* w, void* scratch, uint32_t* d_err, cudaStream_t st) {
  static_assert(kWTile == 2048, "the weights tiles are the scan's tiles");
  const uint64_t m = (uint64_t)g->m;
  if (m == 0) {
    TC_CUDA(cudaMemsetAsync(prefix, 0, sizeof(uint64_t), st));
    return TC_OK;
  }
  if (scan_tile_size() != (uint64_t)kWTile) return set_error(TC_ERR_INVALID_ARG, "scan tile mismatch");
  const uint64_t T = weights_tiles(m);
  if (T > 0x7FFFFFFFull) return set_error(TC_ERR_INVALID_ARG, "too many edges for the weights pass");
  char* p = (char*)scratch;
  uint64_t* wbuf = w ? w : (uint64_t*)p;
  uint64_t* sums = (uint64_t*)(p + align256(8 * m));
  uint64_t* scan_scratch = (uint64_t*)(p + align256(8 * m) + align256(8 * T));
  WeightsArgs A;
  A.out_e = g->out_e;
  A.in_e = g->in_e;
  A.out_off = g->out_off;
  A.in_off = g->in_off;
  A.out_t32 = g->out_t32;
  A.in_t32 = g->in_t32;
  A.x_in = g->x_in;
  A.x_out = g->x_out;
  A.out2in = g->out2in;
  A.r_self = g->r_self;
  A.tmin = g->tmin;
  A.m = m;
  A.delta = delta;
  A.alpha1 = plan.alpha1;
  A.alpha3 = plan.alpha3;
  A.beta1 = plan.beta1;
  A.beta3 = plan.beta3;
  A.closed = plan.closed;
  A.win = win;
  A.w = wbuf;
  A.tile_sums = sums;
  A.err = d_err;
  if (g->out_t32)  // 32-bit list times
    k_weights_rw<<<(unsigned)T, kWThreads, 0, st>>>(A);
  else
    k_weights<<<(unsigned)T, kWThreads, 0, st>>>(A);
  TC_LAUNCHED(1);
  TC_CUDA(cudaGetLastError());
  return scan_u64_from_tile_sums(wbuf, prefix, m, sums, d_err, scan_scratch, scan_u64_scratch_words(T) + 1, st);
}

// ---------------------------------------------------------------------------
// Index layout: [header 256 B][EdgeWin m][guide uint32 (2^gbits + 1)].

int guide_bits(uint64_t m) {
  int b = 0;
  while (b < 32 && (1ull << b) < m) b++;
  return b;
}


size_t index_bytes(uint64_t m) {
  return kIndexHeaderBytes + align256(sizeof(EdgeWin) * m) + sizeof(uint32_t) * ((1ull << guide_bits(m)) + 1);
}

struct IndexView {
  IndexHeader* hdr;
  EdgeWin* win;
  uint32_t* guide;
};

static IndexView index_view(void* index, uint64_t m) {
  char* p = (char*)index;
  IndexView v;
  v.hdr = (IndexHeader*)p;
  v.win = (EdgeWin*)(p + kIndexHeaderBytes);
  v.guide = (uint32_t*)(p + kIndexHeaderBytes + align256(sizeof(EdgeWin) * m));
  return v;
}

// Guide table: bucket b covers r in [b << shift, (b + 1) << shift); guide[b]
// is the edge whose range [prefix[i], prefix[i+1]) holds b << shift (the
// largest i with prefix[i] <= b << shift), the first candidate of the CDF
// search for any r in the bucket; guide[nb] = m - 1.  Filled edge-parallel:
// edge i owns the buckets b with b << shift in its range; a warp shares the
// writes of its 32 edges evenly, so that heavy edges do not serialise.
__global__ void __launch_bounds__(256) k_guide(const uint64_t* __restrict__ prefix, uint32_t m, int gbits,
                                               uint32_t* __restrict__ guide, IndexHeader* hdr, Plan plan,
                                               int64_t delta, uint64_t graph_id, const uint32_t* err) {
  const uint64_t W = prefix[m];
  const int wbits = W ? 64 - __clzll(W - 1) : 0;
  const uint32_t shift = wbits > gbits ? (uint32_t)(wbits - gbits) : 0u;
  const uint32_t nb = W ? (uint32_t)(((W - 1) >> shift) + 1) : 0u;
  const uint64_t low = (1ull << shift) - 1ull;
  auto first_bucket = [&](uint64_t x) { return (uint32_t)((x >> shift) + ((x & low) != 0)); };  // ceil(x / 2^shift)
  const int lane = threadIdx.x & 31;
  const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  for (uint64_t wb = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; wb * 32 < m; wb += warps) {
    const uint64_t i = wb * 32 + lane;
    uint32_t b0 = 0, n = 0;
    if (i < m) {
      b0 = first_bucket(prefix[i]);
      n = first_bucket(prefix[i + 1]) - b0;
    }
    uint32_t incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const uint32_t excl = incl - n;
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    for (uint32_t q0 = 0; q0 < total; q0 += 32) {
      const uint32_t q = q0 + lane;
      // owner: the last lane whose exclusive offset is <= q
      int lo = 0, hi = 31;
#pragma unroll
      for (int step = 0; step < 5; step++) {
        const int mid = (lo + hi + 1) >> 1;
        const uint32_t ex = __shfl_sync(0xffffffffu, excl, mid);
        if (ex <= q) lo = mid; else hi = mid - 1;
      }
      const uint32_t ob0 = __shfl_sync(0xffffffffu, b0, lo);
      const uint32_t oex = __shfl_sync(0xffffffffu, excl, lo);
      if (q < total) guide[ob0 + (q - oex)] = (uint32_t)(wb * 32 + lo);
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (m) guide[nb] = m - 1;
    IndexHeader h;
    h.magic = kIndexMagic;
    h.W = W;
    h.m = m;
    h.shift = shift;
    h.nb = nb;
    h.cls[0] = plan.alpha1;
    h.cls[1] = plan.alpha3;
    h.cls[2] = plan.beta1;
    h.cls[3] = plan.beta3;
    h.closed = plan.closed;
    h.anchor[0] = plan.e1;
    h.anchor[1] = plan.mid;
    h.anchor[2] = plan.e3;
    h.delta = delta;
    h.graph_id = graph_id;
    h.status = err ? *err : 0u;
    *hdr = h;
  }
}

tc_status launch_guide(const tc_graph* g, const Plan& plan, int64_t delta, const uint64_t* prefix, void* index,
                       uint32_t* d_err, cudaStream_t st) {
  IndexView v = index_view(index, (uint64_t)g->m);
  return launch_guide_at(g, plan, delta, prefix, v.hdr, v.guide, d_err, st);
}

size_t proposal_index_bytes(uint64_t m) {
  return kIndexHeaderBytes + sizeof(uint32_t) * ((1ull << guide_bits(m)) + 1);
}

tc_status launch_guide_at(const tc_graph* g, const Plan& plan, int64_t delta, const uint64_t* prefix,
                          IndexHeader* hdr, uint32_t* guide, uint32_t* d_err, cudaStream_t st) {
  const uint64_t m = (uint64_t)g->m;
  IndexView v;
  v.hdr = hdr;
  v.guide = guide;
  const int gb = guide_bits(m);
  uint64_t blocks = (m + 255) / 256;
  const uint64_t cap = (uint64_t)num_sms() * 16;
  if (blocks > cap) blocks = cap;
  if (blocks == 0) blocks = 1;
  k_guide<<<(unsigned)blocks, 256, 0, st>>>(prefix, (uint32_t)m, gb, v.guide, v.hdr, plan, delta, g->id, d_err);
  TC_LAUNCHED(1);
  TC_CUDA(cudaGetLastError());
  return TC_OK;
}

// ---------------------------------------------------------------------------
// Sampler.

struct SamplerArgs {
  const OutEdge* out_e;
  const InEdge* in_e;
  const PairSlot* pair_hash;
  uint32_t hash_mask;
  int hash_shift;
  const int64_t* pair_t;
  const uint32_t* pair_t32;  // pair-list times as t - tmin, or NULL
  int64_t tmin;
  const uint64_t* prefix;
  const IndexHeader* hdr;
  const EdgeWin* win;
  const uint32_t* guide;
  uint64_t seed, offset;
  uint64_t chunk_base;    // index of the chunk's first sample within the call
  uint64_t count;         // samples in the chunk
  OrderView ord;          // the chunk's samples by buckets of their draws (nb = 0: in id order)
  uint32_t m;
  int64_t delta;
  uint64_t graph_id;
  uint64_t* trace;
  SampleSums* sums;
  // proposal mode (h != NULL): the middle edge is drawn from the proposal's
  // prefix and guide (hdr, prefix, guide), the records come from the plain
  // index (win, rec_hdr), and each hit adds X and X^2 to bins[3 h + 0..2]
  const uint16_t* h;
  unsigned long long* bins;
  const uint32_t* hrange;  // proposal: smallest and largest h (in the proposal index header)
  const IndexHeader* rec_hdr;
};

// Times inside the sampler: t - tmin in 32 bits on graphs with 32-bit list
// times (Compact; every time, sum and comparison is then one 32-bit
// operation), else the int64 times.
template <bool Compact>
struct SampleTime {
  typedef uint32_t T;
  static __device__ __forceinline__ T rel(const SamplerArgs& A, int64_t t) { return (uint32_t)t - (uint32_t)A.tmin; }
  static __device__ __forceinline__ T pair(const SamplerArgs& A, uint32_t p) { return __ldg(A.pair_t32 + p); }
  static __device__ __forceinline__ bool beyond(const SamplerArgs& A, T first, T last) {
    return (uint64_t)(last - first) > (uint64_t)A.delta;  // first <= last
  }
  // first + delta; every list time is at most 2^32 - 1
  static __device__ __forceinline__ T end(const SamplerArgs& A, T first) {
    const uint64_t x = (uint64_t)first + (uint64_t)A.delta;  // delta < 2^63
    return x > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)x;
  }
};
template <>
struct SampleTime<false> {
  typedef int64_t T;
  static __device__ __forceinline__ T rel(const SamplerArgs&, int64_t t) { return t; }
  static __device__ __forceinline__ T pair(const SamplerArgs& A, uint32_t p) { return __ldg(A.pair_t + p); }
  static __device__ __forceinline__ bool beyond(const SamplerArgs& A, T first, T last) {
    return (uint64_t)last - (uint64_t)first > (uint64_t)A.delta;
  }
  static __device__ __forceinline__ T end(const SamplerArgs& A, T first) { return sat_add(first, A.delta); }
};

// Positions [*s, *e) of the pair list L_{x,y} (empty when x never sends to
// y) from the pair hash table, one 16-byte slot per probe.
__device__ __forceinline__ void pair_list(const SamplerArgs& A, int32_t x, int32_t y, uint32_t* s, uint32_t* e) {
  *s = *e = 0;
  uint32_t h = pair_slot((uint32_t)x, (uint32_t)y, A.hash_shift);
  for (uint64_t probe = 0; probe <= A.hash_mask; probe++) {
    const uint4 slot = __ldg(reinterpret_cast<const uint4*>(A.pair_hash + h));
    if (slot.x == (uint32_t)x && slot.y == (uint32_t)y) {
      *s = slot.z;
      *e = slot.w;
      return;
    }
    if (slot.x == 0xFFFFFFFFu) return;
    h = (h + 1) & A.hash_mask;
  }
}

// Positions [*a, *b) of the non-empty pair list [s, e) with time in (tlo,
// thi]: the first positions with time > tlo and with time > thi.  Nine in ten
// lists that are found have no entry in the window, most because they end
// before it or begin after it, which their two ends tell at once; both
// bisections of the others halve the same length, so one loop runs them with
// a probe of each in flight.
template <bool Compact>
__device__ __forceinline__ void pair_window(const SamplerArgs& A, uint32_t s, uint32_t e,
                                            typename SampleTime<Compact>::T tlo, typename SampleTime<Compact>::T thi,
                                            uint32_t* a, uint32_t* b) {
  typedef SampleTime<Compact> Tm;
  const typename Tm::T first = Tm::pair(A, s), last = Tm::pair(A, e - 1);
  if (last <= tlo || first > thi) {
    *a = *b = s;
    return;
  }
  uint32_t pa = s, pb = s;
  for (uint32_t len = e - s; len > 1;) {
    const uint32_t half = len >> 1;
    const typename Tm::T va = Tm::pair(A, pa + half - 1), vb = Tm::pair(A, pb + half - 1);
    if (va <= tlo) pa += half;
    if (vb <= thi) pb += half;
    len -= half;
  }
  *a = pa + (Tm::pair(A, pa) <= tlo ? 1u : 0u);
  *b = pb + (Tm::pair(A, pb) <= thi ? 1u : 0u);
}

// ListCount (Alg. 4) over l lists by one merged pass in time order: an
// element of list r extends every increasing tuple of lists 1..r-1 that ends
// strictly earlier, so with acc[r] = number of tuples over lists 1..r seen
// so far, each element of list r adds acc[r-1] (acc[0] = 1).  Elements with
// equal time are handled lists-last-first so that ties never chain.
__device__ uint64_t list_count_merge(const int64_t* __restrict__ pt, const uint32_t* a, const uint32_t* b, int l,
                                     uint32_t* err) {
  uint64_t acc[17];
  uint32_t head[16];
  acc[0] = 1;
  for (int r = 0; r < l; r++) {
    acc[r + 1] = 0;
    head[r] = a[r];
  }
  for (;;) {
    int64_t tau = INT64_MAX;
    bool any = false;
    for (int r = 0; r < l; r++)
      if (head[r] < b[r]) {
        const int64_t x = __ldg(pt + head[r]);
        if (!any || x < tau) tau = x;
        any = true;
      }
    if (!any) break;
    for (int r = l - 1; r >= 0; r--)
      while (head[r] < b[r] && __ldg(pt + head[r]) == tau) {
        const uint64_t s = acc[r + 1] + acc[r];
        if (s < acc[r + 1]) atomicOr(err, kErrOverflow);
        acc[r + 1] = s;
        head[r]++;
      }
  }
  return acc[l];
}

// The same over two lists: for every element of the second, the elements of
// the first that are strictly earlier (a forward pointer; at most 2^64 - 1
// pairs, as both lists have fewer than 2^32 entries).
template <bool Compact>
__device__ __forceinline__ uint64_t list_count_two(const SamplerArgs& A, uint32_t a0, uint32_t b0, uint32_t a1,
                                                   uint32_t b1) {
  typedef SampleTime<Compact> Tm;
  uint64_t c = 0;
  uint32_t p = a0;
  typename Tm::T tp = Tm::pair(A, p);
  for (uint32_t q = a1; q < b1; q++) {
    const typename Tm::T tq = Tm::pair(A, q);
    while (p < b0 && tp < tq) {
      p++;
      if (p < b0) tp = Tm::pair(A, p);
    }
    c += p - a0;
  }
  return c;
}

// ListCount of a gap with two or more lists, over times in (tlo, thi] (kept
// out of line so that its arrays do not weigh on the single-list path).
template <bool Compact>
__device__ __noinline__ uint64_t gap_count_multi(const SamplerArgs& A, const Plan& P, int gp, int32_t up, int32_t u,
                                                int32_t v, int32_t vp, typename SampleTime<Compact>::T tlo,
                                                typename SampleTime<Compact>::T thi, uint32_t* err) {
  auto phi = [&](int role) { return role == 0 ? up : (role == 1 ? u : (role == 2 ? v : vp)); };
  const int l = P.ngap[gp];
  uint32_t a[16], b[16];
  for (int j = 0; j < l; j++) {
    uint32_t s, e;
    pair_list(A, phi(P.gx[gp][j]), phi(P.gy[gp][j]), &s, &e);
    if (s == e) return 0;
    pair_window<Compact>(A, s, e, tlo, thi, &a[j], &b[j]);
    if (a[j] == b[j]) return 0;
  }
  if (l == 2) return list_count_two<Compact>(A, a[0], b[0], a[1], b[1]);
  return list_count_merge(A.pair_t, a, b, l, err);
}

// Product over the gaps of their ListCounts (Alg. 3, 4): gap gp holds the
// non-anchor motif edges of ranks between anchor ranks NG gp and gp + 1, with
// times in (ta[gp], ta[gp + 1]); the last gap runs up to ta[0] + delta
// inclusive.  The anchor times increase strictly, so an open upper bound t
// is the closed bound t - 1.  phi maps path roles (u', u, v, v') to graph
// vertices.
template <int NG, bool Compact>
__device__ __forceinline__ uint64_t gaps_product(const SamplerArgs& A, const Plan& P,
                                                 const typename SampleTime<Compact>::T* ta, int32_t up, int32_t u,
                                                 int32_t v, int32_t vp, uint32_t* err) {
  typedef SampleTime<Compact> Tm;
  auto phi = [&](int role) { return role == 0 ? up : (role == 1 ? u : (role == 2 ? v : vp)); };
  uint64_t X = 1;
#pragma unroll
  for (int gp = 0; gp < NG; gp++) {
    const int l = P.ngap[gp];
    if (l == 0) continue;
    const typename Tm::T tlo = ta[gp];
    const typename Tm::T thi = gp < NG - 1 ? ta[gp + 1] - 1 : Tm::end(A, ta[0]);
    uint64_t c;
    if (l == 1) {  // one list: its length in the window
      uint32_t s, e, a0, b0;
      pair_list(A, phi(P.gx[gp][0]), phi(P.gy[gp][0]), &s, &e);
      if (s == e) return 0;
      pair_window<Compact>(A, s, e, tlo, thi, &a0, &b0);
      c = b0 - a0;
    } else {
      c = gap_count_multi<Compact>(A, P, gp, up, u, v, vp, tlo, thi, err);
    }
    if (c == 0) return 0;
    const uint64_t hi = __umul64hi(X, c);
    if (hi) atomicOr(err, kErrOverflow);
    X *= c;
  }
  return X;
}

// CheckMotif of a wedge (3-vertex motif): base (u, v, t0) and second edge
// to or from y at time tj; the three vertices distinct, t0 < tj <= t0 + delta.
template <bool Compact>
__device__ __forceinline__ uint64_t check_wedge(const SamplerArgs& A, const Plan& P, int32_t y, int32_t u, int32_t v,
                                                typename SampleTime<Compact>::T t0,
                                                typename SampleTime<Compact>::T tj, uint32_t* err, uint32_t* checked) {
  if (u == v || y == u || y == v) return 0;
  if (!(t0 < tj) || SampleTime<Compact>::beyond(A, t0, tj)) return 0;
  ++*checked;
  const typename SampleTime<Compact>::T ta[2] = {t0, tj};
  return gaps_product<2, Compact>(A, P, ta, y, u, v, y, err);
}

// CheckMotif (Alg. 3) of the path (u' -e1- u -e2- v -e3- v'), or of the
// wedge (u' -e1- u -e2- v) / (u -e2- v -e3- v') of a wedge anchor.
template <bool Compact>
__device__ __forceinline__ uint64_t check_motif(const SamplerArgs& A, const Plan& P, int32_t up, int32_t u,
                                                int32_t v, int32_t vp, typename SampleTime<Compact>::T t1,
                                                typename SampleTime<Compact>::T t2,
                                                typename SampleTime<Compact>::T t3, uint32_t* err,
                                                uint32_t* checked) {
  if (P.wedge)
    return P.wedge == 1 ? check_wedge<Compact>(A, P, up, u, v, t2, t1, err, checked)
                        : check_wedge<Compact>(A, P, vp, u, v, t2, t3, err, checked);
  if (up == u || up == v || up == vp || u == v || u == vp || v == vp) return 0;
  // anchor edges ordered by rank must have strictly increasing times
  typename SampleTime<Compact>::T ta[3];  // times of anchor ranks rk[0] < rk[1] < rk[2]
#pragma unroll
  for (int j = 0; j < 3; j++) {
    const int r = P.rk[j];
    ta[j] = r == P.e1 ? t1 : (r == P.mid ? t2 : t3);
  }
  if (!(ta[0] < ta[1] && ta[1] < ta[2])) return 0;
  if (SampleTime<Compact>::beyond(A, ta[0], ta[2])) return 0;
  ++*checked;
  return gaps_product<3, Compact>(A, P, ta, up, u, v, vp, err);
}

// The far vertex and time of the end edge at list position p of an alpha
// list (alpha = 0: a wedge's dummy end, vertex -1).
template <bool Compact>
__device__ __forceinline__ void end_edge(const SamplerArgs& A, int alpha, uint32_t p, int32_t* x,
                                         typename SampleTime<Compact>::T* t) {
  if (alpha != 0) {
    const int4 e = __ldg(reinterpret_cast<const int4*>(alpha < 0 ? (const void*)(A.in_e + p) : (const void*)(A.out_e + p)));
    *x = alpha < 0 ? e.x : e.y;
    *t = SampleTime<Compact>::rel(A, (int64_t)(((uint64_t)(uint32_t)e.w << 32) | (uint32_t)e.z));
  } else {
    *x = -1;
    *t = 0;
  }
}

// Per-thread running sums of a sampling kernel; errors go to the block's word.
struct ThreadSums {
  uint64_t sx = 0;
  unsigned __int128 sx2 = 0;
  uint32_t hits = 0, checked = 0;  // a thread takes fewer than 2^32 samples
  uint32_t* s_err;
  __device__ __forceinline__ explicit ThreadSums(uint32_t* e) : s_err(e) {}
  __device__ __forceinline__ void clear() {
    sx = 0;
    sx2 = 0;
    hits = checked = 0;
  }
  __device__ __forceinline__ void fail(uint32_t bits) { atomicOr(s_err, bits); }
  __device__ __forceinline__ void add(uint64_t X) {
    if (X == 0) return;
    sx += X;
    if (sx < X) fail(kErrOverflow);
    sx2 += (unsigned __int128)X * X;
    hits++;
  }
};

// The index must have been built for this graph, anchor class and delta
// (the weights depend on nothing else); a proposal's records come from the
// plain index.  Returns 0 or the error bits to report.
__device__ __forceinline__ uint32_t index_check(const SamplerArgs& A, const Plan& P) {
  const IndexHeader* H = A.hdr;
  if (H->magic == kIndexMagic && H->status) return H->status;  // the weights pass overflowed
  auto matches = [&](const IndexHeader* X) {
    return X->magic == kIndexMagic && X->cls[0] == P.alpha1 && X->cls[1] == P.alpha3 && X->cls[2] == P.beta1 &&
           X->cls[3] == P.beta3 && X->closed == P.closed && X->delta == A.delta && X->graph_id == A.graph_id;
  };
  return (matches(H) && (A.rec_hdr == nullptr || matches(A.rec_hdr))) ? 0u : kErrIndexMismatch;
}

// Resident blocks of 512 threads per SM the sampler is compiled for (caps its registers).
#ifndef TC_SAMPLE_MIN_BLOCKS
#define TC_SAMPLE_MIN_BLOCKS 3
#endif

// Warp-shuffle reduction of the per-thread sums, one shared atomic per warp
// and one global atomic per block; 128-bit sum of squares with carries,
// overflow of the 64-bit sum flagged.
__device__ __forceinline__ void block_commit(SampleSums* G, uint64_t W, uint64_t sx, unsigned __int128 sx2,
                                             uint64_t hits, uint64_t checked, uint32_t err, uint32_t& s_err,
                                             unsigned long long& s_x, unsigned long long& s_x2lo,
                                             unsigned long long& s_x2hi, unsigned long long& s_hits,
                                             unsigned long long& s_checked) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const uint64_t ox = __shfl_down_sync(0xffffffffu, sx, o);
    const uint64_t olo = __shfl_down_sync(0xffffffffu, (uint64_t)sx2, o);
    const uint64_t ohi = __shfl_down_sync(0xffffffffu, (uint64_t)(sx2 >> 64), o);
    const uint64_t oh = __shfl_down_sync(0xffffffffu, hits, o);
    const uint64_t oc = __shfl_down_sync(0xffffffffu, checked, o);
    const uint32_t oe = __shfl_down_sync(0xffffffffu, err, o);
    const uint64_t nx = sx + ox;
    if (nx < sx) err |= kErrOverflow;
    sx = nx;
    sx2 += ((unsigned __int128)ohi << 64) | olo;
    hits += oh;
    checked += oc;
    err |= oe;
  }
  if ((threadIdx.x & 31) == 0) {
    const unsigned long long old = atomicAdd(&s_x, (unsigned long long)sx);
    if (old + sx < old) err |= kErrOverflow;
    const unsigned long long lo = (uint64_t)sx2;
    const unsigned long long ol = atomicAdd(&s_x2lo, lo);
    const unsigned long long carry = (ol + lo < ol) ? 1ull : 0ull;
    atomicAdd(&s_x2hi, (unsigned long long)(sx2 >> 64) + carry);
    atomicAdd(&s_hits, (unsigned long long)hits);
    atomicAdd(&s_checked, (unsigned long long)checked);
    if (err) atomicOr(&s_err, err);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t e2 = s_err;
    const unsigned long long old = atomicAdd(&G->sum_x, s_x);
    if (old + s_x < old) e2 |= kErrOverflow;
    const unsigned long long ol = atomicAdd(&G->sum_x2_lo, s_x2lo);
    atomicAdd(&G->sum_x2_hi, s_x2hi + ((ol + s_x2lo < ol) ? 1ull : 0ull));
    atomicAdd(&G->hits, s_hits);
    atomicAdd(&G->checked, s_checked);
    G->W = W;
    if (e2) atomicOr(&G->err, e2);
  }
}

// Exhaustive path sum (the proof of Claim 2): path p in [0, W) is the
// (p - prefix[e])-th pair (p1, p3) of middle edge e, p1 major; the sum of
// CheckMotif over all paths is the exact count C, the sum of squares gives
// the exact variance of one sample.
//
// A warp takes runs of consecutive paths (4096, fewer where W would leave warps
// without one: 20,000 edges, 276 us in runs of 4096), lane l every 32nd of them
// from l on: the middle edge and its windows, and the end edge e1, are loaded
// when a lane crosses into the next one (an edge has thousands of paths where
// an exact count takes long), and the pair (p1, p3) is stepped on, so that a
// path costs one coalesced end-edge load and its pair lookup.  Bound by issue
// (67% of the slots at 1e6 edges, 97% of the loads hit L1); 4.0e9 paths of a
// 3e6-edge graph: 24.8 ms, and in runs of a fixed 4096 26.2 ms (41.2 ms with a CDF search, a 64-bit division and both end
// loads per path; 28.5 ms without pair_window's look at the list's ends).
// Four blocks of 256 (64 registers): with five 29.9 ms, with six 33.9 ms.
constexpr uint64_t kPathRun = 4096;  // a multiple of 32
template <bool Compact>
__global__ void __launch_bounds__(256, 4) k_path_sum(const __grid_constant__ SamplerArgs A,
                                                    const __grid_constant__ Plan P, uint64_t length) {
  typedef SampleTime<Compact> Tm;
  const IndexHeader* H = A.hdr;
  const uint64_t W = H->W;
  const uint32_t shift = H->shift;
  __shared__ uint32_t s_err;
  __shared__ unsigned long long s_x, s_x2lo, s_x2hi, s_hits, s_checked;
  if (threadIdx.x == 0) {
    s_err = 0;
    s_x = s_x2lo = s_x2hi = s_hits = s_checked = 0;
  }
  __syncthreads();
  const uint32_t bad = index_check(A, P);
  if (bad) {
    if (threadIdx.x == 0) atomicOr(&A.sums->err, bad);
    return;
  }
  ThreadSums T(&s_err);
  const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  uint64_t hits = 0, checked = 0;  // a thread may take more than 2^32 paths
  for (uint64_t run = warp * length; run < W; run += warps * length) {
    const uint64_t end = W - run < length ? W : run + length;
    uint64_t stop = 0;  // end of the paths of the current middle edge
    uint32_t lo1 = 0, lo3 = 0, d3 = 1, i1 = 0, i3 = 0;
    int32_t u = 0, v = 0, up = 0, vp = 0;
    typename Tm::T t1 = 0, t2 = 0, t3 = 0;
#pragma unroll 1
    for (uint64_t p = run + (threadIdx.x & 31); p < end; p += 32) {
      if (p >= stop) {
        const uint32_t b = (uint32_t)(p >> shift);
        uint32_t lo = __ldg(A.guide + b), hi = __ldg(A.guide + b + 1);
        while (lo < hi) {
          const uint32_t mid = lo + ((hi - lo + 1) >> 1);
          if (__ldg(A.prefix + mid) <= p) lo = mid; else hi = mid - 1;
        }
        if (lo >= A.m) { T.fail(kErrBounds); continue; }
        const EdgeWin wn = A.win[lo];
        const OutEdge e = A.out_e[lo];
        if (wn.d1 == 0 || wn.d3 == 0) { T.fail(kErrBounds); continue; }
        u = e.src;
        v = e.dst;
        t2 = Tm::rel(A, e.t);
        lo1 = wn.lo1;
        lo3 = wn.lo3;
        d3 = wn.d3;
        const uint64_t first = __ldg(A.prefix + lo), j = p - first;
        stop = __ldg(A.prefix + lo + 1);
        if (j >> 32) {
          i1 = (uint32_t)(j / d3);
          i3 = (uint32_t)(j % d3);
        } else {
          i1 = (uint32_t)j / d3;
          i3 = (uint32_t)j - i1 * d3;
        }
        if (lo1 + i1 >= A.m || (uint64_t)lo3 + d3 > A.m) {
          T.fail(kErrBounds);
          stop = 0;
          continue;
        }
        end_edge<Compact>(A, P.alpha1, lo1 + i1, &up, &t1);
      } else {
        i3 += 32;
        if (i3 >= d3) {
          const uint32_t q = i3 / d3;
          i1 += q;
          i3 -= q * d3;
          if (lo1 + i1 >= A.m) {
            T.fail(kErrBounds);
            stop = 0;
            continue;
          }
          end_edge<Compact>(A, P.alpha1, lo1 + i1, &up, &t1);
        }
      }
      end_edge<Compact>(A, P.alpha3, lo3 + i3, &vp, &t3);
      T.add(check_motif<Compact>(A, P, up, u, v, vp, t1, t2, t3, &s_err, &T.checked));
    }
    hits += T.hits;
    checked += T.checked;
    T.hits = T.checked = 0;
  }
  block_commit(A.sums, W, T.sx, T.sx2, hits, checked, 0, s_err, s_x, s_x2lo, s_x2hi, s_hits, s_checked);
}

// The rejection loops: the first attempt is tested in the sampler itself and
// these run only when it is rejected (probability below range / 2^64),
// starting again from attempt 0.
__device__ __noinline__ bool bounded_draw_slow(uint64_t seed, uint64_t s, uint64_t range, uint64_t* out) {
  return bounded_draw_words(seed, s, 0, false, range, out);
}

constexpr uint32_t kSmemBins = 1088;  // per-block bins of the proposal sampler (see k_sample): the 1,025 h of S = 1024
constexpr size_t kSmemBinBytes = 3 * sizeof(unsigned long long) * kSmemBins;

// Adds X and X^2 to bin h: three 64-bit words (sum X, sum X^2 low, high).
__device__ __forceinline__ void bin_add(unsigned long long* bin, uint64_t X) {
  atomicAdd(bin, (unsigned long long)X);
  const unsigned __int128 x2 = (unsigned __int128)X * X;
  const unsigned long long l2 = (uint64_t)x2;
  const unsigned long long old = atomicAdd(bin + 1, l2);
  const unsigned long long carry = (old + l2 < old) ? 1ull : 0ull;
  if ((x2 >> 64) || carry) atomicAdd(bin + 2, (unsigned long long)(x2 >> 64) + carry);
}

// The middle-edge draw of sample s from attempt 0's block o (the later
// attempts run only when it is rejected).
__device__ __forceinline__ bool middle_draw(const SamplerArgs& A, uint64_t s, const uint4& o, uint64_t W,
                                            uint64_t* r2) {
  const uint64_t x = (uint64_t)o.x | ((uint64_t)o.y << 32);
  *r2 = __umul64hi(x, W);
  if (x * W >= W) return true;  // accepted whatever the threshold 2^64 mod W
  uint64_t r;
  if (!bounded_draw_slow(A.seed, s, W, &r)) return false;
  *r2 = r;
  return true;
}

// Lemire's test and draw for a range below 2^32 (two 32 x 64-bit products;
// the same result as lemire_accept); false: the low word lies below the
// range, so the rejection threshold decides.
__device__ __forceinline__ bool draw32(uint32_t xlo, uint32_t xhi, uint32_t range, uint32_t* out) {
  const uint64_t p0 = (uint64_t)xlo * range;
  const uint64_t p1 = (uint64_t)xhi * range + (p0 >> 32);
  *out = (uint32_t)(p1 >> 32);
  return (uint32_t)p1 != 0 || (uint32_t)p0 >= range;
}

// The end edges' draws again with the rejection loop.
__device__ __noinline__ bool end_draw_slow(uint64_t seed, uint64_t s, bool upper, uint32_t range, uint32_t* out) {
  uint64_t r;
  if (!bounded_draw_words(seed, s, 1, upper, range, &r)) return false;
  *out = (uint32_t)r;
  return true;
}

// One sample (Alg. 2, 3) with its middle-edge draw r2: sample index i within
// the call (id offset + i).
template <bool Trace, bool Compact>
__device__ __forceinline__ void sample_one(const SamplerArgs& A, const Plan& P, uint32_t shift, uint64_t i,
                                           uint64_t r2, ThreadSums& T, unsigned long long* sbins = nullptr, uint32_t hmin = 0) {
  const uint64_t s = A.offset + i;
  // middle edge: the unique e with prefix[e] <= r2 < prefix[e + 1]
  const uint32_t b = (uint32_t)(r2 >> shift);
  uint32_t lo = __ldg(A.guide + b), hi = __ldg(A.guide + b + 1);
  while (lo < hi) {
    const uint32_t mid = lo + ((hi - lo + 1) >> 1);
    if (__ldg(A.prefix + mid) <= r2) lo = mid; else hi = mid - 1;
  }
  if (lo >= A.m) { T.fail(kErrBounds); return; }
  const uint4 e = __ldg(reinterpret_cast<const uint4*>(A.win + lo));  // lo1, d1, lo3, d3
  const int4 me = __ldg(reinterpret_cast<const int4*>(A.out_e + lo));  // the middle edge (u, v, t)
  // e1 and e3 from the two halves of block 1, drawn while the two loads are
  // in flight; a draw over one position is 0 and takes none of them (a
  // wedge's dummy end, or a window of one edge)
  const uint4 o = philox4x32_10(make_uint4((uint32_t)s, (uint32_t)(s >> 32), 1u, 0u),
                                make_uint2((uint32_t)A.seed, (uint32_t)(A.seed >> 32)));
  if (e.y == 0 || e.w == 0) { T.fail(kErrBounds); return; }  // index not built from this prefix
  uint32_t r1, r3;
  if (!draw32(o.x, o.y, e.y, &r1) && !end_draw_slow(A.seed, s, false, e.y, &r1)) { T.fail(kErrRng); return; }
  if (!draw32(o.z, o.w, e.w, &r3) && !end_draw_slow(A.seed, s, true, e.w, &r3)) { T.fail(kErrRng); return; }
  const uint32_t p1 = e.x + r1, p3 = e.z + r3;
  if (p1 >= A.m || p3 >= A.m) { T.fail(kErrBounds); return; }
  int32_t up, vp;
  typename SampleTime<Compact>::T t1, t3;
  end_edge<Compact>(A, P.alpha1, p1, &up, &t1);
  end_edge<Compact>(A, P.alpha3, p3, &vp, &t3);
  const typename SampleTime<Compact>::T t2 =
      SampleTime<Compact>::rel(A, (int64_t)(((uint64_t)(uint32_t)me.w << 32) | (uint32_t)me.z));
  const uint64_t X = check_motif<Compact>(A, P, up, me.x, me.y, vp, t1, t2, t3, T.s_err, &T.checked);
  if (A.h && X) {  // exact per-h bins of the proposal estimator (the block's own when it has them)
    const uint32_t hv = __ldg(A.h + lo);
    const bool local = sbins && hv - hmin < kSmemBins;  // an h outside the recorded range goes to global
    bin_add(local ? sbins + 3 * (uint64_t)(hv - hmin) : A.bins + 3 * (uint64_t)hv, X);
  }
  if (Trace) {
    A.trace[4 * i + 0] = lo;
    A.trace[4 * i + 1] = p1;
    A.trace[4 * i + 2] = p3;
    A.trace[4 * i + 3] = X;
  }
  T.add(X);
}

// ---------------------------------------------------------------------------
// Processing order of the samples.  Samples whose middle-edge draws are close
// share windows, edges and pair lists, and lanes with neighbouring draws run
// the same searches, so a call's samples are processed in order of their
// draws.  The draw r = floor(x W / 2^64) is monotone in the 64-bit random
// word x, so the order needs no weights: it is that of x's high word y, which
// is uniform over 2^32.  Each chunk's ids are partitioned into nb = nb1 nb2
// buckets of equal width of y (two passes of nb1 and nb2 buckets, one pass
// for few buckets), and the sampler's block orders one bucket at a time in
// shared memory (sample_bucket).
//
// The bucket sizes are binomial, so every bucket gets a fixed room of its
// mean plus eight standard deviations: a tile reserves its run in a bucket
// with one atomic on the bucket's cursor, and no histogram pass and no scan
// run before the scatter (a histogram over the draws costs a second Philox
// block per sample).  Should a bucket ever overflow its room, the order's
// overflow word is set and the sampler takes the chunk in id order instead:
// the sums are integers and do not depend on the order.
//
// Measured for 1e9 samples of the 300M-edge graph: order passes 7.3 ms (4.1 +
// 3.2) and sampler 24.3 ms, where two counting passes over 16-bit keys with
// their histograms and scans took 12.4 ms and the sampler on that order 52.6
// ms.  A sampler on the order by 20, 24 or 32 bits of the draw, otherwise
// unchanged, took 43.5, 38.7 and 39.0 ms: beyond 24 bits (the bucket and its
// bins here) nothing more is gained.  Each chunk reads the graph once from
// DRAM: in chunks of 2^28 the sampler took 28.9 ms (sample_chunk).
constexpr int kOrderThreads = 512;
constexpr int kOrderItems = 16;
constexpr int kOrderTile = kOrderThreads * kOrderItems;  // 8192
constexpr uint32_t kOrderMaxDigits = 1024;               // buckets of one pass
constexpr uint32_t kOrderMaxDigits2 = 512;               // of a second pass: 9 bits carried from the first
constexpr uint32_t kOrderHeadWords = 64;
// The buckets fill the sampler's tile of 4096 less two standard deviations
// (the one in forty that holds more takes a second, small tile).
constexpr uint32_t kBucketMean = 4096 - 2 * 64;
static_assert(kOrderTile == 1 << 13 && kOrderMaxDigits == 1 << 10 && kOrderMaxDigits2 == 1 << 9,
              "digit, position and carry of a staged element are packed into 32 bits");

// Room of a bucket that holds mean elements of a binomial distribution on
// average.  TC_ORDER_SLACK: standard deviations of room (tests build it small).
#ifndef TC_ORDER_SLACK
#define TC_ORDER_SLACK 8
#endif
static uint32_t bucket_room(uint64_t count, uint64_t buckets) {
  const double mean = (double)count / (double)buckets;
  const double room = mean + TC_ORDER_SLACK * std::sqrt(mean) + 8 * TC_ORDER_SLACK + 1;
  return (uint32_t)(((uint64_t)room + 31) & ~31ull);
}

// Layout of an order of count samples: [head: overflow word, next bucket]
// [cursors of the first pass][bucket sizes][ids by bucket]; scratch: the
// first pass's ids and carried digits.
struct OrderPlan {
  uint32_t nb1, nb2, nb, room1, room;
  size_t head_bytes, ids_off, bytes;   // order buffer
  size_t carry_off, scratch_bytes;     // scratch
};

static OrderPlan order_plan(uint64_t count, uint32_t wave) {
  OrderPlan L;
  // whole waves of buckets while they are few (1e6 samples of the 1e7-edge
  // graph in 456 buckets for 456 resident blocks: 100 us; in 608: 118 us)
  uint64_t nb = std::max<uint64_t>((count + kBucketMean - 1) / kBucketMean, 1);
  if (nb < 16ull * wave) nb = (nb + wave - 1) / wave * wave;
  if (nb <= kOrderMaxDigits) {
    L.nb1 = 1;
    L.nb2 = (uint32_t)nb;
  } else {
    uint64_t d = 1;
    while (d * d < nb) d++;
    L.nb2 = (uint32_t)std::min<uint64_t>(d, kOrderMaxDigits2);
    L.nb1 = (uint32_t)((nb + L.nb2 - 1) / L.nb2);
  }
  L.nb = L.nb1 * L.nb2;
  L.room = bucket_room(count, L.nb);
  L.room1 = L.nb1 > 1 ? bucket_room(count, L.nb1) : 0;
  L.head_bytes = align256(sizeof(uint32_t) * ((size_t)kOrderHeadWords + L.nb1 + L.nb));
  L.ids_off = L.head_bytes;
  L.bytes = L.head_bytes + align256(sizeof(uint32_t) * (size_t)L.nb * L.room);
  L.carry_off = align256(sizeof(uint32_t) * (size_t)L.nb1 * L.room1);
  L.scratch_bytes = L.nb1 > 1 ? L.carry_off + align256(sizeof(uint16_t) * (size_t)L.nb1 * L.room1) : 0;
  return L;
}

size_t order_bytes(uint64_t count, uint32_t wave) { return order_plan(count, wave).bytes; }
size_t order_scratch_bytes(uint64_t count, uint32_t wave) {
  return order_plan(count, wave).scratch_bytes;
}

OrderView order_view(uint64_t count, uint32_t wave, void* order) {
  const OrderPlan L = order_plan(count, wave);
  OrderView v;
  uint32_t* w = (uint32_t*)order;
  v.head = w;
  v.sizes = w + kOrderHeadWords + L.nb1;
  v.ids = (const uint32_t*)((const char*)order + L.ids_off);
  v.nb = L.nb;
  v.room = L.room;
  return v;
}

// Exclusive scan of s_cnt[0 .. 2 kOrderThreads) into s_start, two digits a thread.
__device__ __forceinline__ void order_scan(const uint32_t* s_cnt, uint32_t* s_start, uint32_t* s_warp) {
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const uint32_t c0 = s_cnt[2 * t], c1 = s_cnt[2 * t + 1];
  uint32_t inc = c0 + c1;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) s_warp[wid] = inc;
  __syncthreads();
  uint32_t before = 0;
#pragma unroll
  for (int w = 0; w < kOrderThreads / 32; w++) before += w < wid ? s_warp[w] : 0u;
  const uint32_t ex = before + inc - c0 - c1;
  s_start[2 * t] = ex;
  s_start[2 * t + 1] = ex + c0;
}

// First pass: draws the samples' words y and partitions the ids of a tile of
// 8192 samples by floor(y nb / 2^32).  TwoLevel: the second pass's digit is
// carried along.  The tile is staged in shared memory in digit order, so the
// ids of one digit go out as one run; bound by the Philox block per sample.
template <bool TwoLevel>
__global__ void __launch_bounds__(kOrderThreads) k_order_first(uint64_t seed, uint64_t first, uint64_t count,
                                                              uint32_t nb, uint32_t nb2, uint32_t room,
                                                              uint32_t* __restrict__ cursor,
                                                              uint32_t* __restrict__ ids_out,
                                                              uint16_t* __restrict__ carry_out,
                                                              uint32_t* __restrict__ overflow) {
  __shared__ __align__(16) uint32_t s_cnt[kOrderMaxDigits], s_start[kOrderMaxDigits], s_base[kOrderMaxDigits];
  __shared__ uint32_t s_warp[kOrderThreads / 32];
  __shared__ uint32_t stage[kOrderTile];
  const int t = threadIdx.x;
  s_cnt[t] = s_cnt[t + kOrderThreads] = 0;
  __syncthreads();
  const uint64_t base = (uint64_t)blockIdx.x * kOrderTile;
  const uint32_t n = (uint32_t)(count - base < (uint64_t)kOrderTile ? count - base : (uint64_t)kOrderTile);
  const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
  uint32_t dk[kOrderItems], rk[kOrderItems];  // (digit << 9 | carried digit), rank in the tile's digit
#pragma unroll
  for (int it = 0; it < kOrderItems; it++) {
    const uint32_t j = (uint32_t)it * kOrderThreads + t;
    dk[it] = 0xFFFFFFFFu;
    if (j < n) {
      const uint64_t s = first + base + j;
      const uint32_t y = philox4x32_10(make_uint4((uint32_t)s, (uint32_t)(s >> 32), 0u, 0u), key).y;
      const uint32_t d = __umulhi(y, nb);
      dk[it] = d << 9;
      if (TwoLevel) dk[it] |= __umulhi(y * nb, nb2);  // digit of the remainder: bucket floor(y nb nb2 / 2^32) in all
      rk[it] = atomicAdd(&s_cnt[d], 1u);
    }
  }
  __syncthreads();
  order_scan(s_cnt, s_start, s_warp);
#pragma unroll
  for (int h = 0; h < 2; h++) {
    const int d = t + h * kOrderThreads;
    const uint32_t c = s_cnt[d];
    s_base[d] = c ? atomicAdd(cursor + d, c) : 0u;
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < kOrderItems; it++)
    if (dk[it] != 0xFFFFFFFFu)
      stage[s_start[dk[it] >> 9] + rk[it]] = (dk[it] << 13) | ((uint32_t)it * kOrderThreads + t);
  __syncthreads();
  bool over = false;
  for (uint32_t i = t; i < n; i += kOrderThreads) {
    const uint32_t e = stage[i], d = e >> 22;
    const uint32_t pos = s_base[d] + (i - s_start[d]);
    if (pos < room) {
      const uint64_t g = (uint64_t)d * room + pos;
      ids_out[g] = (uint32_t)base + (e & (kOrderTile - 1));
      if (TwoLevel) carry_out[g] = (uint16_t)((e >> 13) & (kOrderMaxDigits2 - 1));
    } else {
      over = true;
    }
  }
  if (over) *overflow = 1;
}

// Second pass: tile blockIdx.x of the first pass's bucket blockIdx.y, by the carried digit.
struct OrderSecondShared {
  uint32_t cnt[kOrderMaxDigits], start[kOrderMaxDigits], base[kOrderMaxDigits];
  uint32_t warp[kOrderThreads / 32];
  uint32_t id[kOrderTile];
  uint16_t d[kOrderTile];
};
__global__ void __launch_bounds__(kOrderThreads) k_order_second(const uint32_t* __restrict__ cursor1, uint32_t room1,
                                                               const uint32_t* __restrict__ ids_in,
                                                               const uint16_t* __restrict__ carry, uint32_t nb2,
                                                               uint32_t room, uint32_t* __restrict__ sizes,
                                                               uint32_t* __restrict__ ids_out,
                                                               uint32_t* __restrict__ overflow) {
  extern __shared__ __align__(16) unsigned char order_raw[];
  OrderSecondShared& S = *reinterpret_cast<OrderSecondShared*>(order_raw);
  const int t = threadIdx.x;
  const uint32_t seg = blockIdx.y, size1 = min(cursor1[seg], room1), lo = blockIdx.x * kOrderTile;
  if (lo >= size1) return;
  const uint32_t n = min(size1 - lo, (uint32_t)kOrderTile);
  const uint64_t g0 = (uint64_t)seg * room1 + lo;
  S.cnt[t] = S.cnt[t + kOrderThreads] = 0;
  uint32_t id[kOrderItems], dr[kOrderItems];
#pragma unroll
  for (int it = 0; it < kOrderItems; it++) {
    const uint32_t j = (uint32_t)it * kOrderThreads + t;
    dr[it] = 0xFFFFFFFFu;
    if (j < n) {
      id[it] = __ldcs(ids_in + g0 + j);
      dr[it] = (uint32_t)__ldcs(carry + g0 + j) << 16;
    }
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < kOrderItems; it++)
    if (dr[it] != 0xFFFFFFFFu) dr[it] |= atomicAdd(&S.cnt[dr[it] >> 16], 1u);
  __syncthreads();
  order_scan(S.cnt, S.start, S.warp);
  if (t < (int)nb2) {
    const uint32_t c = S.cnt[t];
    S.base[t] = c ? atomicAdd(sizes + (uint64_t)seg * nb2 + t, c) : 0u;
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < kOrderItems; it++)
    if (dr[it] != 0xFFFFFFFFu) {
      const uint32_t p = S.start[dr[it] >> 16] + (dr[it] & 0xFFFFu);
      S.id[p] = id[it];
      S.d[p] = (uint16_t)(dr[it] >> 16);
    }
  __syncthreads();
  bool over = false;
  for (uint32_t i = t; i < n; i += kOrderThreads) {
    const uint32_t d = S.d[i], pos = S.base[d] + (i - S.start[d]);
    if (pos < room)
      ids_out[((uint64_t)seg * nb2 + d) * room + pos] = S.id[i];
    else
      over = true;
  }
  if (over) *overflow = 1;
}

// Writes the order of samples first .. first + count - 1 (at most
// kChunkSamples) into order (order_bytes bytes), using only the given scratch
// of order_scratch_bytes bytes (no allocation).
tc_status order_samples(uint64_t seed, uint64_t first, uint64_t count, uint32_t wave, void* scratch, void* order,
                        cudaStream_t st) {
  TC_CUDA(allow_shared(k_order_second, sizeof(OrderSecondShared)));
  const OrderPlan L = order_plan(count, wave);
  uint32_t* head = (uint32_t*)order;
  uint32_t* cursor1 = head + kOrderHeadWords;
  uint32_t* sizes = cursor1 + L.nb1;
  uint32_t* ids = (uint32_t*)((char*)order + L.ids_off);
  TC_CUDA(cudaMemsetAsync(order, 0, L.head_bytes, st));
  const unsigned tiles = (unsigned)((count + kOrderTile - 1) / kOrderTile);
  if (L.nb1 == 1) {
    k_order_first<false><<<tiles, kOrderThreads, 0, st>>>(seed, first, count, L.nb2, 0, L.room, sizes, ids, nullptr,
                                                          head);
    TC_LAUNCHED(1);
    TC_CUDA(cudaGetLastError());
    return TC_OK;
  }
  uint32_t* ids1 = (uint32_t*)scratch;
  uint16_t* carry = (uint16_t*)((char*)scratch + L.carry_off);
  k_order_first<true><<<tiles, kOrderThreads, 0, st>>>(seed, first, count, L.nb1, L.nb2, L.room1, cursor1, ids1, carry,
                                                       head);
  TC_LAUNCHED(1);
  TC_CUDA(cudaGetLastError());
  const dim3 grid((L.room1 + kOrderTile - 1) / kOrderTile, L.nb1);
  k_order_second<<<grid, kOrderThreads, sizeof(OrderSecondShared), st>>>(cursor1, L.room1, ids1, carry, L.nb2, L.room,
                                                                         sizes, ids, head);
  TC_LAUNCHED(1);
  TC_CUDA(cudaGetLastError());
  return TC_OK;
}

// ---------------------------------------------------------------------------
// The sampler's block works through buckets of samples: it draws r for a
// tile of up to 8 BS of the bucket's samples, orders them by the finer bits
// of their draws in shared memory (a counting sort over 2 BS bins, ranks from
// shared-memory atomics), and its warps then take them in that order, 32 at a
// time from a counter, so that a warp's samples lie on a few neighbouring
// middle edges: their CDF searches take the same steps and their loads fall
// in the same sectors.  Shared memory is kept small, because the searches
// live from the L1 that it leaves: a sample takes its id and the low 32 bits
// of r - r0, r0 the smallest draw of the bucket; where the draws of a bucket
// span more than 32 bits, r is drawn again from the id.
//
// Bound by latency and issue together (ncu, 1e8 samples of the 20M-edge
// graph: issue slots 50% busy, long-scoreboard stalls 13 of 24 cycles, DRAM
// 31%), so by resident warps: 40 registers, which hold 48 warps per SM, spill
// a little and still take 30 ms per 1e9 samples where 64 registers took 38.7
// and 32 registers 41; 12 KB more shared memory per block (an SM's L1 falls
// from 92 to 60 KB) cost 30%, and tiles of 2048 samples 10%.
constexpr int kBucketItems = 8;
template <int BS>
struct TileShared {
  uint32_t id[kBucketItems * BS];
  uint32_t r[kBucketItems * BS];
  uint2 cnt[BS];  // 2 BS bins, later the bins' starts
  uint32_t warp[BS / 32];
  unsigned long long r0;  // the bucket's smallest draw
  uint32_t next;          // next place to take
};
constexpr uint32_t kDrawAgain = 0xFFFFFFFFu;  // instead of r - r0: r is drawn from the id

template <int BS, bool Trace, bool Compact>
__device__ __forceinline__ void sample_bucket(const SamplerArgs& A, const Plan& P, uint64_t W, uint32_t shift,
                                              uint32_t bucket, TileShared<BS>& S, ThreadSums& T,
                                              unsigned long long* sbins, uint32_t hmin) {
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const uint32_t size = min(A.ord.sizes[bucket], A.ord.room);
  const uint2 key = make_uint2((uint32_t)A.seed, (uint32_t)(A.seed >> 32));
  uint32_t* cnt = reinterpret_cast<uint32_t*>(S.cnt);
  // the bucket's words y lie in a range of 2^32 / nb, its draws in one of
  // W / nb + W / 2^32 + 1 (nb <= 2^20 buckets)
  const bool wide = W >= (uint64_t)A.ord.nb << 31;
  for (uint32_t base = 0; base < size; base += kBucketItems * BS) {
    const uint32_t n = min(size - base, (uint32_t)(kBucketItems * BS));
    const uint32_t* ids = A.ord.ids + (uint64_t)bucket * A.ord.room + base;
    S.cnt[t] = make_uint2(0, 0);
    if (t == 0) {
      S.next = 0;
      const uint64_t y0 = (((uint64_t)bucket << 32) + A.ord.nb - 1) / A.ord.nb;  // the bucket's first word
      S.r0 = __umul64hi(y0 << 32, W);
    }
    __syncthreads();
    uint32_t br[kBucketItems];  // bin and rank
#pragma unroll
    for (int it = 0; it < kBucketItems; it++) {
      const uint32_t j = (uint32_t)it * BS + t;
      br[it] = 0xFFFFFFFFu;
      if (j < n) {
        const uint32_t id = __ldcs(ids + j);
        const uint64_t s = A.offset + A.chunk_base + id;
        const uint4 o = philox4x32_10(make_uint4((uint32_t)s, (uint32_t)(s >> 32), 0u, 0u), key);
        const uint64_t x = (uint64_t)o.x | ((uint64_t)o.y << 32);
        S.id[j] = id;
        // (x W mod 2^64 < W: attempt 0 may be rejected)
        S.r[j] = wide || x * W < W ? kDrawAgain : (uint32_t)(__umul64hi(x, W) - S.r0);
        const uint32_t bin = __umulhi(o.y * A.ord.nb, 2 * BS);  // by the position inside the bucket
        br[it] = (bin << 16) | atomicAdd(&cnt[bin], 1u);
      }
    }
    __syncthreads();
    {  // exclusive scan of the bins, two a thread
      const uint2 c = S.cnt[t];
      uint32_t inc = c.x + c.y;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      if (lane == 31) S.warp[wid] = inc;
      __syncthreads();
      uint32_t ex = inc - c.x - c.y;
      for (int w = 0; w < wid; w++) ex += S.warp[w];
      S.cnt[t] = make_uint2(ex, ex + c.x);
    }
    uint32_t id[kBucketItems], r[kBucketItems];
#pragma unroll
    for (int it = 0; it < kBucketItems; it++) {
      id[it] = S.id[it * BS + t];
      r[it] = S.r[it * BS + t];
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kBucketItems; it++)
      if (br[it] != 0xFFFFFFFFu) {
        const uint32_t p = cnt[br[it] >> 16] + (br[it] & 0xFFFFu);
        S.id[p] = id[it];
        S.r[p] = r[it];
      }
    __syncthreads();
    const uint64_t r0 = S.r0;
    for (;;) {
      uint32_t p = 0;
      if (lane == 0) p = atomicAdd(&S.next, 32u);
      p = __shfl_sync(0xffffffffu, p, 0);
      if (p >= n) break;
      p += lane;
      if (p < n) {
        const uint64_t i = A.chunk_base + S.id[p];
        uint64_t r2 = r0 + S.r[p];
        if (S.r[p] == kDrawAgain && !bounded_draw_slow(A.seed, A.offset + i, W, &r2))
          T.fail(kErrRng);
        else
          sample_one<Trace, Compact>(A, P, shift, i, r2, T, sbins, hmin);
      }
    }
    __syncthreads();
  }
}

// Samples [lo, hi) of the chunk in id order.
template <int BS, bool Trace, bool Compact>
__device__ __forceinline__ void sample_ids(const SamplerArgs& A, const Plan& P, uint64_t W, uint32_t shift,
                                           uint64_t lo, uint64_t hi, uint64_t stride, ThreadSums& T,
                                           unsigned long long* sbins, uint32_t hmin) {
  const uint2 key = make_uint2((uint32_t)A.seed, (uint32_t)(A.seed >> 32));
#pragma unroll 1
  for (uint64_t j = lo; j < hi; j += stride) {
    const uint64_t i = A.chunk_base + j, s = A.offset + i;
    const uint4 o = philox4x32_10(make_uint4((uint32_t)s, (uint32_t)(s >> 32), 0u, 0u), key);
    uint64_t r2;
    if (middle_draw(A, s, o, W, &r2))
      sample_one<Trace, Compact>(A, P, shift, i, r2, T, sbins, hmin);
    else
      T.fail(kErrRng);
  }
}

// Proposal mode: a block accumulates the per-h bins of its samples in
// shared memory (kSmemBins consecutive h values from the proposal's
// smallest h) and adds them to the global bins once at its end, instead of
// one global atomic per hit on a few hot bins.
//
// The blocks take the order's buckets one after the other from a counter, and
// a block's warps its samples: buckets on hub edges cost more than others (a
// fixed share per block left the slowest SM 16% behind the mean), and so do
// samples with long lists (with list_count_two, 5e6 samples of a
// motif with two lists in its last gap went from 1.55 to 0.40 ms).
constexpr int kSampleThreads = 512;
template <bool Trace, bool Compact>
__global__ void __launch_bounds__(kSampleThreads, TC_SAMPLE_MIN_BLOCKS) k_sample(const __grid_constant__ SamplerArgs A,
                                                                                const __grid_constant__ Plan P) {
  extern __shared__ __align__(16) unsigned char sample_raw[];  // TileShared (ordered samples), then the bins (proposal mode)
  TileShared<kSampleThreads>& S = *reinterpret_cast<TileShared<kSampleThreads>*>(sample_raw);
  unsigned long long* s_bins =
      reinterpret_cast<unsigned long long*>(sample_raw + (A.ord.nb ? sizeof(TileShared<kSampleThreads>) : 0));
  const IndexHeader* H = A.hdr;
  const uint64_t W = H->W;
  const uint32_t shift = H->shift;
  __shared__ uint32_t s_err, s_item;
  __shared__ unsigned long long s_x, s_x2lo, s_x2hi, s_hits, s_checked;
  if (threadIdx.x == 0) {
    s_err = 0;
    s_x = s_x2lo = s_x2hi = s_hits = s_checked = 0;
  }
  uint32_t hmin = 0;
  bool local_bins = false;
  if (A.h && A.hrange) {
    hmin = A.hrange[0];
    local_bins = A.hrange[1] >= hmin;  // h beyond hmin + kSmemBins - 1 (a wider range) goes to the global bins
    if (local_bins)
      for (uint32_t b = threadIdx.x; b < 3 * kSmemBins; b += blockDim.x) s_bins[b] = 0;
  }
  __syncthreads();
  const uint32_t bad = index_check(A, P);
  if (bad) {
    if (threadIdx.x == 0) atomicOr(&A.sums->err, bad);
    return;
  }
  ThreadSums T(&s_err);
  unsigned long long* bins = local_bins ? s_bins : nullptr;
  if (W && A.ord.nb && A.ord.head[0] == 0) {
    for (;;) {
      if (threadIdx.x == 0) s_item = atomicAdd(A.ord.head + 1, 1u);
      __syncthreads();
      const uint32_t item = s_item;
      if (item >= A.ord.nb) break;
      sample_bucket<kSampleThreads, Trace, Compact>(A, P, W, shift, item, S, T, bins, hmin);
      __syncthreads();
    }
  } else if (W) {  // id order: few samples, or an order that overflowed
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    sample_ids<kSampleThreads, Trace, Compact>(A, P, W, shift, (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, A.count,
                                               stride, T, bins, hmin);
  }
  if (local_bins) {
    __syncthreads();
    for (uint32_t b = threadIdx.x; b < kSmemBins; b += blockDim.x) {
      const unsigned long long x = s_bins[3 * b], lo = s_bins[3 * b + 1], hi = s_bins[3 * b + 2];
      if (!x && !lo && !hi) continue;
      unsigned long long* g = A.bins + 3 * (uint64_t)(hmin + b);
      atomicAdd(g, x);
      const unsigned long long old = atomicAdd(g + 1, lo);
      const unsigned long long carry = (old + lo < old) ? 1ull : 0ull;
      if (hi || carry) atomicAdd(g + 2, hi + carry);
    }
  }
  block_commit(A.sums, W, T.sx, T.sx2, T.hits, T.checked, 0, s_err, s_x, s_x2lo, s_x2hi, s_hits, s_checked);
}

// Diagnostic timing by phase (tc_set_timing): event pairs around the
// launches of a phase, recorded on the launching stream and summed when the
// caller asks.  A call that runs a phase first drops that phase's events of
// the previous call.
static thread_local bool t_timing = false;
static thread_local std::vector<std::pair<cudaEvent_t, cudaEvent_t>> t_events[kNumPhases];

PhaseTimer::PhaseTimer(int phase, cudaStream_t s) : ph(phase), st(s) {
  if (!t_timing) return;
  for (auto& e : t_events[ph]) {
    cudaEventDestroy(e.first);
    cudaEventDestroy(e.second);
  }
  t_events[ph].clear();
}

void PhaseTimer::start() {
  if (!t_timing) return;
  std::pair<cudaEvent_t, cudaEvent_t> e{nullptr, nullptr};
  if (cudaEventCreate(&e.first) != cudaSuccess) return;
  if (cudaEventCreate(&e.second) != cudaSuccess) {
    cudaEventDestroy(e.first);
    return;
  }
  cudaEventRecord(e.first, st);
  t_events[ph].push_back(e);
}

void PhaseTimer::stop() {
  if (t_timing && !t_events[ph].empty()) cudaEventRecord(t_events[ph].back().second, st);
}

void set_timing(bool on) { t_timing = on; }

float last_phase_ms(int phase) {
  if (phase < 0 || phase >= kNumPhases) return 0.f;
  float total = 0.f;
  for (auto& e : t_events[phase]) {
    float ms = 0.f;
    if (cudaEventSynchronize(e.second) == cudaSuccess && cudaEventElapsedTime(&ms, e.first, e.second) == cudaSuccess)
      total += ms;
  }
  return total;
}

float last_sampler_ms() { return last_phase_ms(TC_PHASE_SAMPLE); }

// Scratch and order of a call of k samples in chunks of `chunk`: the last chunk
// is smaller than the others, but its order may hold more rounding.
static void chunk_bytes(uint64_t k, uint64_t chunk, uint32_t wave, size_t* scratch, size_t* order) {
  const uint64_t tail = k % chunk;
  *scratch = std::max(order_scratch_bytes(chunk, wave), tail ? order_scratch_bytes(tail, wave) : (size_t)0);
  *order = std::max(order_bytes(chunk, wave), tail ? order_bytes(tail, wave) : (size_t)0);
}

// Samples a chunk, about 11 bytes each: 2^28 (2.9 GB), or up to 2^30 on graphs
// whose own build took as much scratch.  The pool keeps what it has taken, so
// such a chunk needs no more memory than the process has lent it before, and
// the graphs that gain from reading them once are large (300M edges, 1e9
// samples: 41.1 ms, in chunks of 2^28 45.6 ms).  Growing the pool by 11 GB for
// a call and trimming it afterwards would take 9 and 15 ms.
static uint64_t sample_chunk(uint64_t k, uint64_t m, uint32_t wave) {
  uint64_t chunk = std::min(k, kChunkSamples);
  while (chunk > kSmallChunkSamples) {
    size_t scratch, order;
    chunk_bytes(k, chunk, wave, &scratch, &order);
    if (scratch + order <= kBuildScratchBytes * m) break;
    chunk = std::max(chunk / 2, kSmallChunkSamples);
  }
  return chunk;
}

tc_status launch_sampler(const tc_graph* g, const Plan& plan, int64_t delta, const uint64_t* prefix,
                         const void* index, uint64_t k, uint64_t seed, uint64_t offset, uint64_t* trace,
                         SampleSums* d_sums, cudaStream_t st, const void* qindex, const uint16_t* h,
                         unsigned long long* bins) {
  const uint64_t m = (uint64_t)g->m;
  IndexView v = index_view(const_cast<void*>(index), m);
  const IndexHeader* rec_hdr = nullptr;
  if (h) {  // the proposal's header and guide replace the plain ones
    rec_hdr = v.hdr;
    v.hdr = (IndexHeader*)qindex;
    v.guide = (uint32_t*)((char*)const_cast<void*>(qindex) + kIndexHeaderBytes);
  }
  SamplerArgs A;
  A.out_e = g->out_e;
  A.in_e = g->in_e;
  A.pair_hash = g->pair_hash;
  A.hash_mask = g->hash_mask;
  A.hash_shift = g->hash_shift;
  A.pair_t = g->pair_t;
  A.pair_t32 = g->pair_t32;
  A.tmin = g->tmin;
  A.prefix = prefix;
  A.hdr = v.hdr;
  A.win = v.win;
  A.guide = v.guide;
  A.chunk_base = 0;
  A.count = k;
  A.ord = OrderView{};
  A.m = (uint32_t)m;
  A.seed = seed;
  A.offset = offset;
  A.delta = delta;
  A.graph_id = g->id;
  A.trace = trace;
  A.sums = d_sums;
  A.h = h;
  A.bins = bins;
  A.hrange = h ? (const uint32_t*)((const char*)qindex + kProposalRangeOffset) : nullptr;
  A.rec_hdr = rec_hdr;
  const bool compact = A.pair_t32 != nullptr;
  auto kernel = trace ? (compact ? k_sample<true, true> : k_sample<true, false>)
                      : (compact ? k_sample<false, true> : k_sample<false, false>);
  constexpr size_t kTileBytes = sizeof(TileShared<kSampleThreads>);
  TC_CUDA(allow_shared(kernel, kTileBytes + kSmemBinBytes));
  const uint64_t max_blocks = (uint64_t)num_sms() * blocks_per_sm(kernel, kSampleThreads, kTileBytes + kSmemBinBytes);
  auto run = [&](const OrderView& ord, uint64_t base, uint64_t count) -> tc_status {
    A.ord = ord;
    A.chunk_base = base;
    A.count = count;
    uint64_t blocks = max_blocks;
    const uint64_t need = ord.nb ? ord.nb : (count + kSampleThreads - 1) / kSampleThreads;
    if (need < blocks) blocks = need ? need : 1;
    const size_t dyn = (ord.nb ? kTileBytes : 0) + (h ? kSmemBinBytes : 0);
    kernel<<<(unsigned)blocks, kSampleThreads, dyn, st>>>(A, plan);
    TC_LAUNCHED(1);
    TC_CUDA(cudaGetLastError());
    return TC_OK;
  };
  PhaseTimer timer(TC_PHASE_SAMPLE, st), sort_timer(TC_PHASE_ORDER, st);
  if (k < kOrderedMinSamples) {
    timer.start();
    tc_status s = run(OrderView{}, 0, k);
    timer.stop();
    return s;
  }
  // samples in chunks, each with an order of its own (smaller chunks also when
  // the memory for a large one is not there)
  const uint32_t wave = (uint32_t)max_blocks;
  uint64_t chunk = sample_chunk(k, m, wave);
  size_t scratch = 0;
  char* buf = nullptr;
  for (;;) {
    size_t obytes = 0;
    chunk_bytes(k, chunk, wave, &scratch, &obytes);
    const cudaError_t e = pool_malloc(&buf, scratch + obytes, st);
    if (e == cudaSuccess) break;
    if (e != cudaErrorMemoryAllocation || chunk <= kSmallChunkSamples) return cuda_status(e, "pool_malloc(order)");
    cudaGetLastError();
    chunk = std::max(chunk / 2, kSmallChunkSamples);
  }
  void* order = buf + scratch;
  tc_status s = TC_OK;
  for (uint64_t base = 0; base < k && s == TC_OK; base += chunk) {
    const uint64_t count = (k - base) < chunk ? (k - base) : chunk;
    sort_timer.start();
    s = order_samples(seed, offset + base, count, wave, buf, order, st);
    sort_timer.stop();
    timer.start();
    if (s == TC_OK) s = run(order_view(count, wave, order), base, count);
    timer.stop();
  }
  cudaFreeAsync(buf, st);
  return s;
}

tc_status launch_path_sum(const tc_graph* g, const Plan& plan, int64_t delta, const uint64_t* prefix,
                          const void* index, uint64_t W, SampleSums* d_sums, cudaStream_t st) {
  const uint64_t m = (uint64_t)g->m;
  IndexView v = index_view(const_cast<void*>(index), m);
  SamplerArgs A;
  std::memset(&A, 0, sizeof(A));
  A.out_e = g->out_e;
  A.in_e = g->in_e;
  A.pair_hash = g->pair_hash;
  A.hash_mask = g->hash_mask;
  A.hash_shift = g->hash_shift;
  A.pair_t = g->pair_t;
  A.pair_t32 = g->pair_t32;
  A.tmin = g->tmin;
  A.prefix = prefix;
  A.hdr = v.hdr;
  A.win = v.win;
  A.guide = v.guide;
  A.m = (uint32_t)m;
  A.delta = delta;
  A.graph_id = g->id;
  A.sums = d_sums;
  auto kernel = A.pair_t32 ? k_path_sum<true> : k_path_sum<false>;
  uint64_t blocks = (uint64_t)num_sms() * blocks_per_sm(kernel, 256, 0);
  const uint64_t need = (W + 255) / 256;
  if (need < blocks) blocks = need ? need : 1;
  // as many paths for every warp: runs of at most kPathRun, as many of them
  // for each warp, none of which takes a run more than the others (36,000
  // edges: a count 396 us with runs of a fixed 4096 paths, 332 us so)
  const uint64_t warps = blocks * (256 / 32), round = warps * kPathRun;
  const uint64_t all = std::max<uint64_t>(1, W / round + (W % round != 0)) * warps;
  const uint64_t length = (W / all + (W % all != 0) + 31) & ~31ull;
  kernel<<<(unsigned)blocks, 256, 0, st>>>(A, plan, std::max<uint64_t>(32, length));
  TC_LAUNCHED(1);
  TC_CUDA(cudaGetLastError());
  return TC_OK;
}

// ---------------------------------------------------------------------------
// Batched sampling: one persistent launch over the tiles of many queries
// (graphs, motifs, windows).  Each block takes the next work item from a
// global counter; items are numbered query after query, so a block sees
// its queries in increasing order, keeps per-thread sums while the query
// stays the same and commits them to that query's sums when it changes.
// A query's samples and sums are those of the same query run alone.

struct alignas(16) BatchQuery {
  SamplerArgs A;
  Plan P;
};
static_assert(sizeof(BatchQuery) <= kBatchQueryBytes, "batch record too large");
static_assert(kBatchQueryBytes % 16 == 0, "batch record must be whole 16-byte words");

void batch_query_record(void* h_rec, const tc_graph* g, const Plan& plan, int64_t delta, const uint64_t* prefix,
                        const void* index, uint64_t seed, uint64_t offset, uint64_t chunk_base, uint64_t count,
                        void* order, SampleSums* sums) {
  std::memset(h_rec, 0, kBatchQueryBytes);
  BatchQuery* Q = (BatchQuery*)h_rec;
  const uint64_t m = (uint64_t)g->m;
  IndexView v = index_view(const_cast<void*>(index), m);
  SamplerArgs& A = Q->A;
  A.out_e = g->out_e;
  A.in_e = g->in_e;
  A.pair_hash = g->pair_hash;
  A.hash_mask = g->hash_mask;
  A.hash_shift = g->hash_shift;
  A.pair_t = g->pair_t;
  A.pair_t32 = g->pair_t32;
  A.tmin = g->tmin;
  A.prefix = prefix;
  A.hdr = v.hdr;
  A.win = v.win;
  A.guide = v.guide;
  A.seed = seed;
  A.offset = offset;
  A.chunk_base = chunk_base;
  A.count = count;
  if (order) A.ord = order_view(count, 1, order);
  A.m = (uint32_t)m;
  A.delta = delta;
  A.graph_id = g->id;
  A.sums = sums;
  Q->P = plan;
}

static uint32_t batch_record_group(const void* h_rec, uint32_t tile) {
  const SamplerArgs& A = ((const BatchQuery*)h_rec)->A;
  if (!A.ord.nb) return 0;
  const uint64_t group = (uint64_t)tile * A.ord.nb / (A.count ? A.count : 1);
  return (uint32_t)(group ? group : 1);
}

uint64_t batch_record_items(const void* h_rec, uint32_t tile) {
  const SamplerArgs& A = ((const BatchQuery*)h_rec)->A;
  const uint32_t group = batch_record_group(h_rec, tile);
  return group ? (A.ord.nb + group - 1) / group : (A.count + tile - 1) / tile;
}

// Compact: the records of graphs with 32-bit list times, else those with
// 64-bit times only (a kernel each, so that neither pays for the other's
// registers); a record's items are buckets [j group, (j + 1) group) of its
// order, or tiles of its ids when it has no order or one that overflowed.
template <int BS, bool Compact>
__global__ void __launch_bounds__(BS, (512 * TC_SAMPLE_MIN_BLOCKS) / BS)
    k_sample_batch(const char* __restrict__ records, const uint64_t* __restrict__ tile_begin, uint32_t nq,
                   uint32_t tile, unsigned long long* __restrict__ next_item) {
  extern __shared__ __align__(16) unsigned char batch_raw[];
  TileShared<BS>& S = *reinterpret_cast<TileShared<BS>*>(batch_raw);
  __shared__ BatchQuery s_q;
  __shared__ unsigned long long s_j;
  __shared__ uint32_t s_query;
  __shared__ uint32_t s_err;
  __shared__ unsigned long long s_x, s_x2lo, s_x2hi, s_hits, s_checked;
  if (threadIdx.x == 0) {
    s_err = 0;
    s_x = s_x2lo = s_x2hi = s_hits = s_checked = 0;
  }
  uint32_t cur = 0xFFFFFFFFu;
  bool bad = false;
  ThreadSums T(&s_err);
  for (;;) {
    if (threadIdx.x == 0) {
      const unsigned long long item = atomicAdd(next_item, 1ull);
      uint32_t q = nq;
      if (item < tile_begin[nq]) {  // the last record whose first item is <= item
        uint32_t lo = 0, hi = nq - 1;
        while (lo < hi) {
          const uint32_t mid = (lo + hi + 1) >> 1;
          if (tile_begin[mid] <= item) lo = mid; else hi = mid - 1;
        }
        q = lo;
        s_j = item - tile_begin[q];
      }
      s_query = q;
    }
    __syncthreads();
    const uint32_t q = s_query;
    if (q != cur) {  // block-uniform
      if (cur != 0xFFFFFFFFu && !bad) {
        block_commit(s_q.A.sums, s_q.A.hdr->W, T.sx, T.sx2, T.hits, T.checked, 0, s_err, s_x, s_x2lo, s_x2hi, s_hits,
                     s_checked);
        T.clear();
        if (threadIdx.x == 0) {
          s_err = 0;
          s_x = s_x2lo = s_x2hi = s_hits = s_checked = 0;
        }
        __syncthreads();  // the record is no longer read
      }
      if (q >= nq) break;
      // the records are kBatchQueryBytes apart
      const uint4* src = reinterpret_cast<const uint4*>(records + (uint64_t)q * kBatchQueryBytes);
      uint4* dst = reinterpret_cast<uint4*>(&s_q);
      for (uint32_t w = threadIdx.x; w < sizeof(BatchQuery) / 16; w += BS) dst[w] = src[w];
      __syncthreads();
      cur = q;
      const uint32_t e = index_check(s_q.A, s_q.P);
      bad = e != 0;
      if (bad && threadIdx.x == 0) atomicOr(&s_q.A.sums->err, e);
    }
    const uint64_t W = s_q.A.hdr->W;
    const uint32_t shift = s_q.A.hdr->shift;
    if (!bad && W) {
      const uint64_t j = s_j, nb = s_q.A.ord.nb;
      uint64_t j0 = j * tile, j1 = min(j0 + tile, s_q.A.count);
      bool ordered = false;
      if (nb) {  // as batch_record_group
        const uint64_t gr = max((uint64_t)tile * nb / s_q.A.count, (uint64_t)1);
        const uint64_t b0 = j * gr, b1 = min(b0 + gr, nb);
        ordered = s_q.A.ord.head[0] == 0;
        // (at most 2^28 samples and 2^20 buckets: the products fit)
        j0 = ordered ? b0 : s_q.A.count * b0 / nb;
        j1 = ordered ? b1 : s_q.A.count * b1 / nb;
      }
      if (ordered) {
#pragma unroll 1
        for (uint32_t b = (uint32_t)j0; b < (uint32_t)j1; b++)
          sample_bucket<BS, false, Compact>(s_q.A, s_q.P, W, shift, b, S, T, nullptr, 0);
      } else {
        sample_ids<BS, false, Compact>(s_q.A, s_q.P, W, shift, j0 + threadIdx.x, j1, BS, T, nullptr, 0);
      }
    }
    __syncthreads();
  }
}

template <int BS, bool Compact>
static int batch_blocks_per_sm() {
  static_assert(sizeof(TileShared<BS>) + 1024 <= 48 << 10, "with the static part: more has to be allowed first");
  return blocks_per_sm(k_sample_batch<BS, Compact>, BS, sizeof(TileShared<BS>));
}

int sample_batch_blocks_per_sm(int bs, bool compact) {
  if (bs == 128) return compact ? batch_blocks_per_sm<128, true>() : batch_blocks_per_sm<128, false>();
  if (bs == 256) return compact ? batch_blocks_per_sm<256, true>() : batch_blocks_per_sm<256, false>();
  if (bs == 512) return compact ? batch_blocks_per_sm<512, true>() : batch_blocks_per_sm<512, false>();
  return 0;
}


template <int BS>
static void launch_batch(bool compact, uint32_t tile, unsigned blocks, const char* Q, const uint64_t* d_tile_begin,
                         uint32_t nq, unsigned long long* d_next_item, cudaStream_t st) {
  if (compact)
    k_sample_batch<BS, true><<<blocks, BS, sizeof(TileShared<BS>), st>>>(Q, d_tile_begin, nq, tile, d_next_item);
  else
    k_sample_batch<BS, false><<<blocks, BS, sizeof(TileShared<BS>), st>>>(Q, d_tile_begin, nq, tile, d_next_item);
}

tc_status launch_sample_batch(int bs, bool compact, uint32_t tile, unsigned blocks, const void* d_records,
                              const uint64_t* d_tile_begin, uint32_t nq, unsigned long long* d_next_item,
                              cudaStream_t st) {
  const char* Q = (const char*)d_records;
  if (!sample_batch_blocks_per_sm(bs, compact))
    return set_error(TC_ERR_INVALID_ARG, "batch block size must be 128, 256 or 512");
  if (bs == 128)
    launch_batch<128>(compact, tile, blocks, Q, d_tile_begin, nq, d_next_item, st);
  else if (bs == 256)
    launch_batch<256>(compact, tile, blocks, Q, d_tile_begin, nq, d_next_item, st);
  else
    launch_batch<512>(compact, tile, blocks, Q, d_tile_begin, nq, d_next_item, st);
  TC_LAUNCHED(1);
  TC_CUDA(cudaGetLastError());
  return TC_OK;
}

}  // namespace tc
