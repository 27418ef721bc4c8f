// Fused full-vocabulary draft selection (paper Sec. "Fuse draft selection without changing
// proposals"): one pass over a row of logits yields the spine token (argmax, lowest index among
// equal maxima) and three ordered sibling candidates (top-3 by value; among equal values the higher
// index first), written straight into caller-owned buffers.  The two tie conventions differ on
// purpose and both are kept; the candidates are not de-duplicated against the spine token, so
// candidate 0 repeats the spine token whenever the maximum is unique.
//
// One thread-block cluster per row, the vocabulary split over its CTAs.  The pass over the logits keeps one running
// maximum per thread and nothing else (a packed maximum per two bf16 entries), so it runs at the rate of the loads; the
// third largest of the threads' maxima is reached by three distinct entries and therefore bounds the third-best entry from
// below, and only the few threads whose maximum reaches that bound have their entries looked at again (out of L2, a warp per
// thread).  What they yield goes to a short list, from which four warp-wide selections take the result.  Where many threads
// reach the bound (a constant, masked or coarsely quantised row) the visits would take longer than a second pass, in which
// every thread notes the first and the last place of its maximum: the third largest of the (value, last place) keys is then a
// bound that three threads reach.  If even those hold more than the list takes, every thread ranks its own entries and the
// ranks are merged.  Both orders are
// total, so the result depends neither on the way taken nor on how the row was split (any cluster size gives the same bytes).
// Bound by HBM for large calls, by launch, one round trip and the selection for small ones.  Measured against ranking every
// entry on the way (151,936 entries a row): 1024 rows bf16 76 -> 52 us = 6.0 TB/s, f32 107 -> 97 us = 6.4 TB/s; 40 rows bf16
// 11.0 -> 5.4 us; 600 rows of 20,000 bf16 18.3 -> 8.1 us.  Rows with ties, bf16, 1024 and 8 rows: constant 107 and 9.0 us (one
// thread after the other: 568 and 43.5; ranking everything: 346 and 11.8), 1 % of the entries equal 103 and 7.9 us (272 and 21.4).
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <climits>
#include <cmath>

#include "internal.h"

namespace cg = cooperative_groups;

namespace lumo {

namespace {

constexpr int kSelThreads = 512;

// Both orders become plain unsigned comparisons of 64-bit keys: the high word is the value mapped
// monotonically to an unsigned integer (signed zeros made equal first), the low word the index for the
// candidate list (higher index first among equal values) or its complement for the spine token (lower
// index first).  Distinct indices make all keys of a row distinct; key 0 is below every real key.
using Key = unsigned long long;
__device__ __forceinline__ uint32_t ordered_bits(float v) {
  const uint32_t u = __float_as_uint(v + 0.0f);          // -0.0 + 0.0 = +0.0
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float unordered_bits(uint32_t o) {
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7FFFFFFFu) : ~o);
}
__device__ __forceinline__ Key kmax(Key a, Key b) { return a > b ? a : b; }
__device__ __forceinline__ Key kmin(Key a, Key b) { return a < b ? a : b; }

struct Best {
  Key s;             // spine
  Key t0, t1, t2;    // candidates, best first
  __device__ __forceinline__ void init() { s = t0 = t1 = t2 = 0; }
  __device__ __forceinline__ void push(float v, int i) {
    const Key hi = (Key)ordered_bits(v) << 32;
    s = kmax(s, hi | (0xFFFFFFFFu - (uint32_t)i));
    const Key c = hi | (uint32_t)i;
    const Key x = kmin(t0, c);
    t0 = kmax(t0, c);
    const Key y = kmin(t1, x);
    t1 = kmax(t1, x);
    t2 = kmax(t2, y);
  }
  // top three of two sorted triples
  __device__ __forceinline__ void merge(const Best& o) {
    s = kmax(s, o.s);
    const Key c0 = kmax(t0, o.t0), d0 = kmin(t0, o.t0), c1 = kmax(t1, o.t1), c2 = kmax(t2, o.t2);
    t0 = c0;
    t1 = kmax(d0, c1);
    t2 = kmax(kmin(d0, c1), c2);
  }
};

__device__ __forceinline__ void warp_merge(Best& b) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    Best other;
    other.s = __shfl_xor_sync(0xffffffffu, b.s, o);
    other.t0 = __shfl_xor_sync(0xffffffffu, b.t0, o);
    other.t1 = __shfl_xor_sync(0xffffffffu, b.t1, o);
    other.t2 = __shfl_xor_sync(0xffffffffu, b.t2, o);
    b.merge(other);
  }
}

template <typename T> struct Vec;                       // 16 bytes of logits
template <> struct Vec<float> { static constexpr int n = 4; };
template <> struct Vec<__nv_bfloat16> { static constexpr int n = 8; };
__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }

constexpr int kListCap = 256;                            // entries the short list holds
// Threads of a CTA whose entries are looked at again one thread at a time.  Visits and the second pass cost the same at about
// 130 to 160 threads (1024 rows: 0.1 % equal entries, 130 threads, 92 against 102 us; 0.15 %, 180 threads, 119 against 102; 40
// rows in quarters: 0.25 %, 87 threads, 12.4 against 14 us, 0.5 %, 159 threads, 16.0 against 15.3).
constexpr int kVisitMost = 144;

// Ordered maximum of a thread's entries.
template <typename T> struct RunningMax;
template <> struct RunningMax<float> {
  float m;
  __device__ __forceinline__ RunningMax() : m(-INFINITY) {}
  __device__ __forceinline__ void add(const uint4& w) {
    m = fmaxf(m, fmaxf(fmaxf(__uint_as_float(w.x), __uint_as_float(w.y)), fmaxf(__uint_as_float(w.z), __uint_as_float(w.w))));
  }
  __device__ __forceinline__ float get() const { return m; }
};
template <> struct RunningMax<__nv_bfloat16> {
  __nv_bfloat162 m;
  __device__ __forceinline__ RunningMax() : m(__float2bfloat162_rn(-INFINITY)) {}
  __device__ __forceinline__ void add(const uint4& w) {
    const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&w);
    m = __hmax2(m, __hmax2(__hmax2(p[0], p[1]), __hmax2(p[2], p[3])));
  }
  __device__ __forceinline__ float get() const { return fmaxf(__low2float(m), __high2float(m)); }
};

// Removes the largest of the warp's values (one instance of it) and returns it; lanes without a value hold 0.
__device__ __forceinline__ uint32_t take_max(uint32_t& v, int lane) {
  const uint32_t top = __reduce_max_sync(0xffffffffu, v);
  const int owner = __ffs(__ballot_sync(0xffffffffu, v == top)) - 1;
  if (lane == owner) v = 0;
  return top;
}

// Best of up to 32 * kPer keys held by a warp (value in the high word, index in the low word; 0: none): the spine is the
// largest value with the lowest index, the candidates the three largest keys.  Every lane returns the result.
template <int kPer>
__device__ __forceinline__ Best pick_best(Key (&k)[kPer], bool spine_keys, const Key* spine_k) {
  Best b;
  uint32_t hi = 0;
#pragma unroll
  for (int e = 0; e < kPer; ++e) hi = max(hi, (uint32_t)((spine_keys ? spine_k[e] : k[e]) >> 32));
  const uint32_t top = __reduce_max_sync(0xffffffffu, hi);
  uint32_t lo = 0xFFFFFFFFu;
#pragma unroll
  for (int e = 0; e < kPer; ++e) {
    const Key x = spine_keys ? spine_k[e] : k[e];
    if ((uint32_t)(x >> 32) == top) lo = min(lo, (uint32_t)x);
  }
  b.s = (Key)top << 32 | __reduce_min_sync(0xffffffffu, lo);
  Key* out[3] = {&b.t0, &b.t1, &b.t2};
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    Key mine = 0;
#pragma unroll
    for (int e = 0; e < kPer; ++e) mine = kmax(mine, k[e]);
    const uint32_t h = __reduce_max_sync(0xffffffffu, (uint32_t)(mine >> 32));
    const uint32_t l = __reduce_max_sync(0xffffffffu, (uint32_t)(mine >> 32) == h ? (uint32_t)mine : 0u);
    const Key best = (Key)h << 32 | l;
    *out[r] = best;
#pragma unroll
    for (int e = 0; e < kPer; ++e)
      if (k[e] == best) k[e] = 0;
  }
  return b;
}

template <typename T>
__global__ void __launch_bounds__(kSelThreads, 2)
select_kernel(const T* __restrict__ logits, int V, int32_t* __restrict__ spine, int32_t* __restrict__ cand) {
  constexpr int kWarps = kSelThreads / 32;
  __shared__ uint32_t top3[3 * kWarps];
  __shared__ Key list[kListCap];
  __shared__ int n_list, n_tied;
  __shared__ Best warp_best[kWarps];
  __shared__ Best cta_best;                            // its spine key holds the plain index in the low word
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), nblk = (int)cl.num_blocks();
  const int r = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const T* row = logits + (size_t)r * V;
  constexpr int n = Vec<T>::n;
  // the row's 16-byte units are dealt out to the CTAs in contiguous runs; a ragged head and tail
  // (row start not on a 16-byte boundary, V not a multiple of the unit) are read element by element
  const uintptr_t addr = reinterpret_cast<uintptr_t>(row);
  int head = (int)(((16 - (addr & 15)) & 15) / sizeof(T));
  if (head > V) head = V;
  const int units = (V - head) / n;
  const int tail0 = head + units * n;
  const int per = (units + nblk - 1) / nblk;
  const int u_lo = min(units, rank * per), u_hi = min(units, u_lo + per);
  if (tid == 0) n_list = n_tied = 0;
  pdl_wait();          // the logits (and the outputs) may belong to earlier kernels
  pdl_trigger();
  // ---- one pass: the thread's maximum ---------------------------------------------------------------------
  RunningMax<T> rm;
  constexpr int kU = 8;                                // independent 16-byte loads in flight per thread
  const T* base = row + head;
  auto unit = [&](int u) { return *reinterpret_cast<const uint4*>(base + (size_t)u * n); };
  int u = u_lo + tid;
  for (; u + (kU - 1) * kSelThreads < u_hi; u += kU * kSelThreads) {    // bounded: units of this CTA
    uint4 raw[kU];
#pragma unroll
    for (int k = 0; k < kU; ++k) raw[k] = unit(u + k * kSelThreads);
#pragma unroll
    for (int k = 0; k < kU; ++k) rm.add(raw[k]);
  }
  {
    uint4 raw[kU];
    int got = 0;
#pragma unroll
    for (int k = 0; k < kU; ++k)
      if (u + k * kSelThreads < u_hi) { raw[k] = unit(u + k * kSelThreads); got = k + 1; }
#pragma unroll
    for (int k = 0; k < kU; ++k)
      if (k < got) rm.add(raw[k]);
  }
  float mx = rm.get();
  if (rank == 0) {
    if (tid < head) mx = fmaxf(mx, to_f32(row[tid]));
    if (tid < V - tail0) mx = fmaxf(mx, to_f32(row[tail0 + tid]));
  }
  // ---- bound: the third largest of the threads' maxima -----------------------------------------------------
  {
    uint32_t v = ordered_bits(mx);                     // never 0 (only a NaN would map there)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const uint32_t top = take_max(v, lane);
      if (lane == 0) top3[3 * warp + k] = top;
    }
  }
  __syncthreads();
  float thr;
  {
    uint32_t a = top3[lane], c = lane + 32 < 3 * kWarps ? top3[lane + 32] : 0;
    uint32_t top = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      uint32_t v = max(a, c);
      top = __reduce_max_sync(0xffffffffu, v);
      const int owner = __ffs(__ballot_sync(0xffffffffu, v == top)) - 1;
      if (lane == owner) { if (a == top) a = 0; else c = 0; }
    }
    thr = unordered_bits(top);
  }
  // ---- entries that reach it: those of the threads whose maximum does, looked at again by their whole warp ------
  auto visit = [&](uint32_t who, auto push) {
    for (; who; who &= who - 1) {                                                         // bounded: 32 lanes
      const int t = (warp << 5) + __ffs(who) - 1;
      for (int w = u_lo + t + lane * kSelThreads; w < u_hi; w += 32 * kSelThreads) {      // bounded: units of one thread
        const uint4 raw = unit(w);
        const T* e = reinterpret_cast<const T*>(&raw);
#pragma unroll
        for (int k = 0; k < n; ++k) push(to_f32(e[k]), head + w * n + k);
      }
      if (rank == 0 && lane == 0) {
        if (t < head) push(to_f32(row[t]), t);
        if (t < V - tail0) push(to_f32(row[tail0 + t]), tail0 + t);
      }
    }
  };
  auto key_of = [](float v, int i) { return (Key)ordered_bits(v) << 32 | (uint32_t)i; };
  auto enter = [&](int* count, Key key) {
    const int at = atomicAdd(count, 1);
    if (at < kListCap) list[at] = key;
  };
  auto best_of_list = [&](int listed) {                // by one warp
    constexpr int kPer = kListCap / 32;
    if (listed <= 32) {
      Key k[1] = {lane < listed ? list[lane] : 0};
      return pick_best<1>(k, false, nullptr);
    }
    Key k[kPer];
#pragma unroll
    for (int e = 0; e < kPer; ++e) k[e] = lane + 32 * e < listed ? list[lane + 32 * e] : 0;
    return pick_best<kPer>(k, false, nullptr);
  };
  bool ranked = false;                                 // (uniform) warp 0 has the CTA's result
  if (__syncthreads_count(mx >= thr) <= kVisitMost) {
    visit(__ballot_sync(0xffffffffu, mx >= thr), [&](float v, int i) { if (v >= thr) enter(&n_list, key_of(v, i)); });
    __syncthreads();
    ranked = n_list <= kListCap;
    if (ranked && warp == 0) {
      const Best b = best_of_list(n_list);
      if (lane == 0) cta_best = b;
    }
  }
  if (!ranked) {
    // Many equal entries (a constant, fully masked or coarsely quantised row): the value alone bounds too little.  Every
    // thread looks for its largest value again and notes where it stands first and last; the third largest of the threads'
    // (value, last place) keys bounds the candidates, and at most three threads reach it.
    float tv = -INFINITY;
    int first = -1, last = -1;
    auto note = [&](float v, int i) {                  // ascending places
      if (v > tv || first < 0) first = i;
      if (v >= tv) { tv = v; last = i; }
    };
    if (rank == 0 && tid < head) note(to_f32(row[tid]), tid);
    for (int w = u_lo + tid; w < u_hi; w += kSelThreads) {                               // bounded: units of this CTA
      const uint4 raw = unit(w);
      const T* e = reinterpret_cast<const T*>(&raw);
#pragma unroll
      for (int k = 0; k < n; ++k) note(to_f32(e[k]), head + w * n + k);
    }
    if (rank == 0 && tid < V - tail0) note(to_f32(row[tail0 + tid]), tail0 + tid);
    const Key mine = first < 0 ? 0 : key_of(tv, last);
    {
      Key k[1] = {mine};
      const Key sk[1] = {first < 0 ? 0 : key_of(tv, first)};
      const Best b = pick_best<1>(k, true, sk);
      if (lane == 0) warp_best[warp] = b;
    }
    __syncthreads();
    Key k[3] = {0, 0, 0}, sk[3] = {0, 0, 0};
    if (lane < kWarps) {
      const Best& o = warp_best[lane];
      k[0] = o.t0; k[1] = o.t1; k[2] = o.t2; sk[0] = o.s;
    }
    const Best bound = pick_best<3>(k, true, sk);
    visit(__ballot_sync(0xffffffffu, mine != 0 && mine >= bound.t2), [&](float v, int i) {
      const Key key = key_of(v, i);
      if (key >= bound.t2) enter(&n_tied, key);
    });
    __syncthreads();
    ranked = n_tied <= kListCap;
    if (ranked && warp == 0) {
      Best b = best_of_list(n_tied);
      b.s = bound.s;
      if (lane == 0) cta_best = b;
    }
  }
  if (!ranked) {
    // hundreds of the largest entries in the hands of three threads: every thread ranks its own
    Best b;
    b.init();
    for (int w = u_lo + tid; w < u_hi; w += kSelThreads) {                               // bounded: units of this CTA
      const uint4 raw = unit(w);
      const T* e = reinterpret_cast<const T*>(&raw);
#pragma unroll
      for (int k = 0; k < n; ++k) {
        const float v = to_f32(e[k]);
        if (v >= thr) b.push(v, head + w * n + k);
      }
    }
    if (rank == 0) {
      if (tid < head) b.push(to_f32(row[tid]), tid);
      if (tid < V - tail0) b.push(to_f32(row[tail0 + tid]), tail0 + tid);
    }
    warp_merge(b);
    if (lane == 0) warp_best[warp] = b;
    __syncthreads();
    if (warp == 0) {
      if (lane < kWarps) b = warp_best[lane]; else b.init();
      warp_merge(b);
      b.s = (b.s & 0xFFFFFFFF00000000ull) | (0xFFFFFFFFu - (uint32_t)b.s);
      if (lane == 0) cta_best = b;
    }
  }
  auto write = [&](const Best& b) {
    if (lane != 0) return;
    spine[r] = (int32_t)(uint32_t)b.s;
    cand[3 * r + 0] = (int32_t)(uint32_t)b.t0; cand[3 * r + 1] = (int32_t)(uint32_t)b.t1; cand[3 * r + 2] = (int32_t)(uint32_t)b.t2;
  };
  if (nblk == 1) {
    if (warp == 0) { __syncwarp(); write(cta_best); }
    return;
  }
  cl.sync();
  if (rank == 0 && warp == 0) {
    Key k[3] = {0, 0, 0}, sk[3] = {0, 0, 0};           // a CTA without entries contributes nothing
    if (lane < nblk) {
      const Best* o = cl.map_shared_rank(&cta_best, lane);
      k[0] = o->t0; k[1] = o->t1; k[2] = o->t2;
      sk[0] = o->s;
    }
    write(pick_best<3>(k, true, sk));
  }
  cl.sync();                                           // no CTA leaves while rank 0 may still read it
}

}  // namespace

cudaError_t launch_select(const void* logits, int dtype, int rows, int V, int split, int32_t* spine, int32_t* cand,
                          int sms, bool pdl, cudaStream_t st) {
  static int cache_f[64] = {}, cache_h[64] = {};
  const int cap = dtype == LUMO_BF16 ? max_cluster_ctas(select_kernel<__nv_bfloat16>, kSelThreads, cache_h)
                                     : max_cluster_ctas(select_kernel<float>, kSelThreads, cache_f);
  int cluster = split;
  if (cluster == 0) {
    // Few rows: each over more SMs, as long as a CTA keeps 64 KB to read (the two cluster barriers cost as much as a CTA
    // takes for about that).  Of 168 sizes (1 to 400 rows, 16 to 594 KB a row) 117 are within 4 % of the best split and all
    // within 15 %; us, whole / halves / quarters / eighths / sixteenths: 40 rows of 128 KB 4.9 / 5.1 / 5.0 / 8.0 / 12, 16 of 297
    // KB 6.8 / 6.0 / 5.3 / 4.9 / 8.0, 1 of 297 KB 4.4 / 4.4 / 4.0 / 3.6 / 3.5, 100 of 128 KB 5.8 / 6.4 / 9.0 / 15 / -.
    cluster = cap;
    while (cluster > 1 && (long long)rows * cluster > 2LL * sms) cluster >>= 1;
    const long long row_bytes = (long long)V * (dtype == LUMO_BF16 ? 2 : 4);
    while (cluster > 1 && row_bytes < cluster * 65536LL) cluster >>= 1;
  }
  if (cluster > cap) return cudaErrorInvalidConfiguration;
  if (dtype == LUMO_BF16)
    return launch_cluster_kernel(select_kernel<__nv_bfloat16>, dim3(cluster, rows), dim3(kSelThreads), cluster, 0, st, pdl,
                                 reinterpret_cast<const __nv_bfloat16*>(logits), V, spine, cand);
  return launch_cluster_kernel(select_kernel<float>, dim3(cluster, rows), dim3(kSelThreads), cluster, 0, st, pdl,
                               reinterpret_cast<const float*>(logits), V, spine, cand);
}

}  // namespace lumo
