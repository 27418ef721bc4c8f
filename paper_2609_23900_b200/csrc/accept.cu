// Device-resident acceptance walk: accepted path, its length, the pending token and the final row
// as fixed-shape device products (paper Algorithm 1, "Select one continuation"; Sec. "One
// device-selected path drives native continuation"), so that verify -> select -> commit needs no
// host round trip.  One thread-block cluster per sequence (the vocabulary is split over its CTAs,
// partial results meet through distributed shared memory) walks from the pre-tree state through the
// children of the current node in ascending logical index.
//
//   greedy     accept the child whose token equals argmax of the current target row (lowest token
//              index on ties); otherwise stop, the pending token is that argmax.
//   rejection  child c with token x is accepted iff u_c q_c(x) Z < r(x), r the unnormalised residual
//              target (r = p at first) and Z its sum; a rejection replaces r by (r - Z q_c)+ (accepted
//              mass min(p, q), residual mass proportional to (p - q)+, Appendix "Serving configuration
//              and measurement"); when no child is accepted the pending token is drawn from r / Z by an
//              exponential race argmax_i r_i / e_i over caller-supplied Exp(1) variates.
// Decisions that turn floats into integers use fixed precisions: the acceptance test and the residual
// update in float64 (separate multiply and subtract, no contraction), the residual stored in float32,
// the race keys as correctly rounded float32 quotients; sums are float64 in a fixed order.
//
// What bounds it: the chain of passes over a vocabulary row, each one memory round trip, the float64 conversions and one
// cluster-wide reduction.  Hence: a thread keeps to the same entries in every pass, the residual stays in the CTA's shared
// memory (as the float64 it is used as), the next candidate's proposal row is requested before the reduction that decides
// whether it is needed, and a reduction is one exchange: every CTA stores its partial into all CTAs of the cluster, one cluster barrier, and every warp adds up the
// same values in the same order; the residual at the next candidate's token travels with it.  Measured on 151,936 entries against passes through global
// memory and two barriers per candidate: rejection sampling 1 sequence 26.9 -> 23.4 us, 8 sequences 47.9 -> 36.8 us, 16
// sequences 68 -> 52 us; greedy 16 sequences 18.0 -> 15.5 us.  The race divides few entries, a candidate's uniform and probability
// are asked for ahead of the reduction before its test, proposals are widened by integer instructions, and a pack's place in the
// slice is looked up once: 8 sequences 42.4 -> 34.9 us, 1 sequence 17.2 -> 14.0, 2 of 131,071 entries 26.7 -> 22.6 (other inputs
// than the figures before).
// Staging the target row of the candidate under test too, so that an accepted one costs no wait, gained nothing (8 sequences 42.5 ->
// 42.1, 1 sequence 17.2 -> 17.9): a level's time goes into its passes and reductions.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "internal.h"

namespace cg = cooperative_groups;

namespace lumo {

namespace {

constexpr int kAcceptThreads = 512;
constexpr int kAcceptWarps = kAcceptThreads / 32;
constexpr int kAcceptCluster = 8;       // CTAs per sequence when there are many: the vocabulary is split over a cluster
constexpr int kMaxCluster = 16;
// What one reduction exchanges: the warps' partials within a CTA, the CTAs' partials, and the residual at one token.
struct Exchange {
  union { double warp_sum[kAcceptWarps]; unsigned long long warp_key[kAcceptWarps]; };
  union { double sum[kMaxCluster]; unsigned long long key[kMaxCluster]; };
  double at_token;
};

// A thread takes its entries of a slice in packs of four: neighbouring ones where the rows lie on 16-byte boundaries
// (kVec), else four that are kAcceptThreads apart.  Pack k, place j:
template <bool kVec>
__device__ __forceinline__ int entry_of(int k, int j) {
  return kVec ? 4 * (k * kAcceptThreads + (int)threadIdx.x) + j : (4 * k + j) * kAcceptThreads + (int)threadIdx.x;
}
constexpr int kPack = 4 * kAcceptThreads;          // entries of a pack over the CTA
// whether a slice of n entries (a multiple of four where kVec) has that place
template <bool kVec>
__device__ __forceinline__ bool in_slice(int k, int j, int n) { return entry_of<kVec>(k, kVec ? 0 : j) < n; }
constexpr int kFlight = 5;                         // packs requested together
// where the residual of that entry is kept: neighbouring threads, neighbouring places (no bank conflicts either way)
__device__ __forceinline__ int place_of(int k, int j) { return (4 * k + j) * kAcceptThreads + (int)threadIdx.x; }
template <bool kVec>
__device__ __forceinline__ int place_of_entry(int e) {
  return kVec ? (4 * (e / kPack) + (e & 3)) * kAcceptThreads + (e >> 2) % kAcceptThreads : e;
}
// the packs of a slice, kFlight at a time: load(k, i) for all of a flight, then use(k, i)
template <class Load, class Use>
__device__ __forceinline__ void for_packs(int packs, Load load, Use use) {
  for (int k0 = 0; k0 < packs; k0 += kFlight) {    // bounded: the slice
#pragma unroll
    for (int i = 0; i < kFlight; ++i)
      if (k0 + i < packs) load(k0 + i, i);
#pragma unroll
    for (int i = 0; i < kFlight; ++i)
      if (k0 + i < packs) use(k0 + i, i);
  }
}
// thread that holds entry e of a slice
template <bool kVec>
__device__ __forceinline__ int holder_of(int e) { return kVec ? (e >> 2) % kAcceptThreads : e % kAcceptThreads; }

// row: first entry of the slice; n: its length (a multiple of four where kVec).  Places beyond it hold `none`.
template <bool kVec>
__device__ __forceinline__ float4 load_pack(const float* row, int n, int k, float none) {
  float4 w = make_float4(none, none, none, none);
  if constexpr (kVec) {
    const int e = entry_of<true>(k, 0);
    if (e < n) w = __ldg(reinterpret_cast<const float4*>(row + e));
  } else {
    const int e = entry_of<false>(k, 0);
    if (e < n) w.x = __ldg(row + e);
    if (e + kAcceptThreads < n) w.y = __ldg(row + e + kAcceptThreads);
    if (e + 2 * kAcceptThreads < n) w.z = __ldg(row + e + 2 * kAcceptThreads);
    if (e + 3 * kAcceptThreads < n) w.w = __ldg(row + e + 3 * kAcceptThreads);
  }
  return w;
}
// the same entries on their way into shared memory, for the thread that will use them
template <bool kVec>
__device__ __forceinline__ void stage_row(float* dst, const float* row, int n) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  if constexpr (kVec) {
    for (int e = 4 * (int)threadIdx.x; e < n; e += kPack)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d + 4 * e), "l"(row + e) : "memory");
  } else {
    for (int e = (int)threadIdx.x; e < n; e += kAcceptThreads)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d + 4 * e), "l"(row + e) : "memory");
  }
}
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// (double)f.  The conversion instruction takes 16 lanes a clock and SM, and an update needs three per entry; for a positive
// normal number it is three integer instructions.
__device__ __forceinline__ double widen(float f) {
  const uint32_t u = __float_as_uint(f);
  if (u - 0x00800000u >= 0x7F000000u) return (double)f;        // zero, denormal, negative, infinite, NaN
  return __hiloint2double((int)((u >> 3) + 0x38000000u), (int)(u << 29));
}
__device__ __forceinline__ float rcp_approx(float x) { float y; asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }

struct Cluster {
  cg::cluster_group cl;
  int rank, nblk, lane, warp;
  Exchange* x;          // two, taking turns: what reduction k wrote is overwritten by k + 2, behind barrier k + 1, which no
  int turn;             // thread passes before it has read reduction k
  __device__ __forceinline__ void sync() { if (nblk > 1) cl.sync(); else __syncthreads(); }

  // Sum of v over the cluster; `token_here`: this thread holds the residual at the token asked for (value at_token).
  __device__ __forceinline__ double sum(double v, bool token_here, double at_token, double* token_value) {
    Exchange* mine = x + turn;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) mine->warp_sum[warp] = v;
    const uint32_t who = __ballot_sync(0xffffffffu, token_here);
    if (who) {
      const double t = __shfl_sync(0xffffffffu, at_token, __ffs(who) - 1);
      if (lane < nblk) cl.map_shared_rank(mine, lane)->at_token = t;
    }
    __syncthreads();
    if (warp == 0) {
      v = lane < kAcceptWarps ? mine->warp_sum[lane] : 0.0;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      v = __shfl_sync(0xffffffffu, v, 0);
      if (lane < nblk) cl.map_shared_rank(mine, lane)->sum[rank] = v;
    }
    sync();
    double t = lane < nblk ? mine->sum[lane] : 0.0;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    *token_value = mine->at_token;
    turn ^= 1;
    return __shfl_sync(0xffffffffu, t, 0);
  }
  // index of the largest value (the lowest index among equal ones)
  __device__ __forceinline__ int argmax(float v, int i) {
    Exchange* mine = x + turn;
    const uint32_t bits = ordered(v);
    uint32_t top = __reduce_max_sync(0xffffffffu, bits);
    uint32_t idx = __reduce_min_sync(0xffffffffu, bits == top ? (uint32_t)i : 0xFFFFFFFFu);
    if (lane == 0) mine->warp_key[warp] = (unsigned long long)top << 32 | (0xFFFFFFFFu - idx);
    __syncthreads();
    if (warp == 0) {
      const unsigned long long best = pick(lane < kAcceptWarps ? mine->warp_key[lane] : 0);
      if (lane < nblk) cl.map_shared_rank(mine, lane)->key[rank] = best;
    }
    sync();
    const unsigned long long best = pick(lane < nblk ? mine->key[lane] : 0);
    turn ^= 1;
    return (int)(0xFFFFFFFFu - (uint32_t)best);
  }
  static __device__ __forceinline__ unsigned long long pick(unsigned long long k) {
    const uint32_t top = __reduce_max_sync(0xffffffffu, (uint32_t)(k >> 32));
    return (unsigned long long)top << 32 | __reduce_max_sync(0xffffffffu, (uint32_t)(k >> 32) == top ? (uint32_t)k : 0u);
  }
  static __device__ __forceinline__ uint32_t ordered(float v) {
    const uint32_t u = __float_as_uint(v + 0.0f);          // -0.0 counts as +0.0
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
  }
};

// kMode: 0 greedy, 1 rejection sampling.  kVec: rows on 16-byte boundaries.  RT: what the residual of a slice is kept as in shared memory, beside a staged
// proposal row: float64 (no conversion when it is used again), or float32 where that does not fit; void: neither fits, the
// residual lives in the caller's float32 scratch and the proposal rows are read in place.
template <int kMode, bool kVec, class RT>
__global__ void __launch_bounds__(kAcceptThreads)
accept_kernel(TreeDev t, int N, int Ns, AcceptView a, int lmax, int chunk, int32_t* __restrict__ accepted,
              int32_t* __restrict__ len_out, int32_t* __restrict__ next_token, int32_t* __restrict__ final_node) {
  constexpr bool kShared = !std::is_void_v<RT>;
  using R = std::conditional_t<kShared, RT, float>;
  // this sequence's tree, staged once: the walk's dependent lookups then stay on chip
  __shared__ int32_t parent_child_off[kMaxNodes + 2], child_list[kMaxNodes], slot_map[kMaxNodes], tok_of_node[kMaxNodes];
  __shared__ Exchange xch[2];
  extern __shared__ __align__(16) unsigned char dyn[];     // residual, proposal row (whole packs)
  Cluster c = {cg::this_cluster()};
  c.rank = (int)c.cl.block_rank(); c.nblk = (int)c.cl.num_blocks();
  c.lane = threadIdx.x & 31; c.warp = threadIdx.x >> 5;
  c.x = xch; c.turn = 0;
  const int b = blockIdx.y, tid = threadIdx.x, V = a.V;
  const int v_lo = min(V, c.rank * chunk), n = min(V, v_lo + chunk) - v_lo;     // this CTA's slice of the vocabulary
  for (int e = tid; e < N + 2; e += kAcceptThreads) parent_child_off[e] = t.child_off[(size_t)b * (N + 2) + e];
  pdl_wait();          // everything below may belong to earlier kernels
  pdl_trigger();
  for (int e = tid; e < N; e += kAcceptThreads) {
    child_list[e] = t.child_list[(size_t)b * N + e];
    const int row = t.slot[(size_t)b * N + e];
    slot_map[e] = row;
    tok_of_node[e] = a.token[(size_t)b * Ns + row];
  }
  int32_t* acc = accepted + (size_t)b * lmax;
  if (c.rank == 0)
    for (int e = tid; e < lmax; e += kAcceptThreads) acc[e] = -1;
  c.sync();            // tables staged; every CTA of the cluster runs before anyone stores into it
  R* r;
  if constexpr (kShared) r = reinterpret_cast<R*>(dyn); else r = a.work + (size_t)b * V + v_lo;
  float* q_staged = reinterpret_cast<float*>(dyn + (size_t)((chunk + kPack - 1) / kPack) * kPack * sizeof(R));
  const int packs = (n + kPack - 1) / kPack;
  // (the shared arrays hold whole packs, the scratch exactly the slice)
  auto get = [&](int k, int j) -> R { if constexpr (kShared) return r[place_of(k, j)]; else return r[entry_of<kVec>(k, j)]; };
  auto put = [&](int k, int j, R v) { if constexpr (kShared) r[place_of(k, j)] = v; else if (entry_of<kVec>(k, j) < n) r[entry_of<kVec>(k, j)] = v; };
  auto target = [&](int row) { return a.p_target + ((size_t)b * (Ns + 1) + row) * V + v_lo; };
  int cur = -1, len = 0, nxt = 0;

  for (int step = 0; step <= lmax; ++step) {                 // bounded: a path has at most lmax nodes
    const float* p = target(cur < 0 ? Ns : slot_map[cur]);
    const int c_lo = parent_child_off[cur + 1], c_hi = len < lmax ? parent_child_off[cur + 2] : parent_child_off[cur + 1];
    int took = -1;
    if constexpr (kMode == 0) {
      float bv = -1.f;
      int bi = 0x7fffffff;
      // (The rows the walk may go on with are not asked for ahead.  Eight steps, V = 151,936, one sequence: 22.5 us, with the
      // rows of one, two or three children ahead 24.5, 26.5 and 26.6 where the rows lie in L2, as a softmax leaves them; 28.7
      // against 26.7, 28.7 and 30.7 where they do not.  The same at 8000 to 151,936 entries and 1 to 13 sequences.)
      auto look = [&](float v, int e) { if (v > bv) { bv = v; bi = v_lo + e; } };
      float4 w[kFlight];
      for_packs(packs, [&](int k, int i) { w[i] = load_pack<kVec>(p, n, k, -2.f); },
                [&](int k, int i) {                           // ascending entries
                  look(w[i].x, entry_of<kVec>(k, 0)); look(w[i].y, entry_of<kVec>(k, 1));
                  look(w[i].z, entry_of<kVec>(k, 2)); look(w[i].w, entry_of<kVec>(k, 3));
                });
      nxt = c.argmax(bv, bi);
      for (int ci = c_lo; ci < c_hi; ++ci) {                  // bounded: children of one node
        const int ch = child_list[ci];
        if (tok_of_node[ch] == nxt) { took = ch; break; }
      }
    } else {
      auto proposal = [&](int ch) { return a.q_draft + ((size_t)b * Ns + slot_map[ch]) * V + v_lo; };
      auto request = [&](int ci) {                            // the proposal row of the candidate after next
        if (ci >= c_hi) return;
        if constexpr (kShared) stage_row<kVec>(q_staged, proposal(child_list[ci]), n);
      };
      auto holds = [&](int x) { return x >= v_lo && x < v_lo + n && tid == holder_of<kVec>(x - v_lo); };
      auto token_of = [&](int ci) { return ci < c_hi ? tok_of_node[child_list[ci]] : -1; };
      double at_x = 0.0;                                      // residual at the token under test
      float u_x = 0.f, q_x = 0.f;                             // the candidate's uniform, its proposal's probability of the token
      auto candidate = [&](int ci) {                          // requested ahead of the reduction that the test waits for
        if (ci >= c_hi) return;
        const int ch = child_list[ci];
        u_x = __ldg(a.uniforms + (size_t)b * Ns + slot_map[ch]);
        q_x = __ldg(proposal(ch) - v_lo + tok_of_node[ch]);
      };
      auto finish = [&](const double (&z)[4], int x) {
        const bool here = holds(x);
        return c.sum((z[0] + z[1]) + (z[2] + z[3]), here, here ? (double)r[kShared ? place_of_entry<kVec>(x - v_lo) : x - v_lo] : 0.0, &at_x);
      };
      auto start = [&](int x) {                               // r = p; returns its sum
        double z[4] = {0.0, 0.0, 0.0, 0.0};
        float4 w[kFlight];
        for_packs(packs, [&](int k, int i) { w[i] = load_pack<kVec>(p, n, k, 0.f); },
                  [&](int k, int i) {
                    const float v[4] = {w[i].x, w[i].y, w[i].z, w[i].w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                      const double d = (double)v[j];
                      put(k, j, (R)d);
                      z[j] += d;
                    }
                  });
        return finish(z, x);
      };
      candidate(c_lo);
      request(c_lo);
      double Z = start(token_of(c_lo));
      for (int ci = c_lo; ci < c_hi; ++ci) {                  // bounded: children of one node
        const int ch = child_list[ci];
        const float* q = proposal(ch);
        // every CTA evaluates the same test on the same values
        const double lhs = __dmul_rn(__dmul_rn((double)u_x, (double)q_x), Z);
        if (lhs < at_x) { took = ch; break; }
        if constexpr (kShared) stage_wait();
        double z[4] = {0.0, 0.0, 0.0, 0.0};
        float4 w[kFlight];
        for_packs(packs,
                  [&](int k, int i) {
                    if constexpr (!kShared) w[i] = load_pack<kVec>(q, n, k, 0.f);
                    else if constexpr (kVec) w[i] = *reinterpret_cast<const float4*>(q_staged + entry_of<true>(k, 0));
                    else w[i] = make_float4(q_staged[entry_of<false>(k, 0)], q_staged[entry_of<false>(k, 1)], q_staged[entry_of<false>(k, 2)],
                                            q_staged[entry_of<false>(k, 3)]);
                  },
                  [&](int k, int i) {
                    const float qv[4] = {w[i].x, w[i].y, w[i].z, w[i].w};
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                      if (in_slice<kVec>(k, j, n)) {
                        const double d = __dsub_rn((double)get(k, j), __dmul_rn(Z, widen(qv[j])));
                        const double rd = (double)(float)(d > 0.0 ? d : 0.0);
                        put(k, j, (R)rd);
                        z[j] += rd;
                      }
                  });
        candidate(ci + 1);
        request(ci + 1);
        const int nx = token_of(ci + 1);
        const double Zn = finish(z, nx);
        if (Zn > 0.0) Z = Zn;
        else Z = start(nx);                                   // empty residual: restore the target row
      }
      if (took < 0) {                                          // draw the pending token from r / Z
        const float* noise = a.noise + (size_t)b * V + v_lo;
        float bv = -1.f;
        int bi = 0x7fffffff;
        // Correctly rounded quotients only for entries that may be the largest: what r times an approximate 1 / e (to 2^-21) puts
        // below the warp's best by more than 2^-18 of it is not.  Outside 2^-100 .. 2^100 (denormals, zeros, infinities) all
        // entries are divided.  (All of them always: 9 to 15 thousand cycles of a walk's 30 to 70.)
        float top = 0.f;
        for (int k0 = 0; k0 < packs; k0 += kFlight) {          // bounded: the slice
          float4 w[kFlight];
          float about[4 * kFlight];
#pragma unroll
          for (int i = 0; i < kFlight; ++i)
            if (k0 + i < packs) w[i] = load_pack<kVec>(noise, n, k0 + i, 1.f);
          float best = 0.f;
          uint32_t mine = 0;
#pragma unroll
          for (int i = 0; i < kFlight; ++i) {
            const float nv[4] = {w[i].x, w[i].y, w[i].z, w[i].w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              about[4 * i + j] = 0.f;
              if (k0 + i < packs && in_slice<kVec>(k0 + i, j, n)) {
                mine |= 1u << (4 * i + j);
                about[4 * i + j] = (float)get(k0 + i, j) * rcp_approx(nv[j]);
                best = fmaxf(best, about[4 * i + j]);
              }
            }
          }
          top = fmaxf(top, __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(best))));
          const bool plain = top >= 0x1p-100f && top <= 0x1p100f;
          const float line = top * (1.f - 0x1p-18f);
          uint32_t closer = mine;
#pragma unroll
          for (int i = 0; i < 4 * kFlight; ++i)
            if (plain && about[i] < line) closer &= ~(1u << i);
          while (closer) {                                      // bounded: 20; ascending entries
            const int i = __ffs(closer) - 1, k = k0 + (i >> 2), j = i & 3, e = entry_of<kVec>(k, j);
            closer &= closer - 1;
            const float key = __fdiv_rn((float)get(k, j), __ldg(noise + e));
            if (key > bv) { bv = key; bi = v_lo + e; }
          }
        }
        nxt = c.argmax(bv, bi);
      } else if constexpr (kShared) {
        stage_wait();                                          // the row that turned out not to be needed
      }
    }
    if (took < 0) break;                                       // uniform over the cluster
    if (c.rank == 0 && tid == 0) acc[len] = took;
    cur = took;
    ++len;
  }
  if (c.rank == 0 && tid == 0) { len_out[b] = len; next_token[b] = nxt; final_node[b] = cur; }
  c.sync();                                                    // no CTA leaves while a peer may still store into it
}

}  // namespace

cudaError_t launch_accept(const TreeDev& t, int B, int N, int Ns, const AcceptView& a, int lmax, int32_t* accepted,
                          int32_t* len, int32_t* next_token, int32_t* final_node, int sms, bool pdl, cudaStream_t st) {
  static int cache[64] = {};
  int cluster = max_cluster_ctas(accept_kernel<1, true, double>, kAcceptThreads, cache);
  if (cluster > kAcceptCluster && B * cluster > sms) cluster = kAcceptCluster;   // many sequences: smaller clusters
  while (cluster > 1 && a.V < cluster * kAcceptThreads) cluster >>= 1;           // small vocabularies
  // Many short rejection walks: a reduction costs more the more CTAs meet in it, and clusters that need nearly every SM wait
  // for each other's place; against that stands the longer slice of a CTA.  The line lies where the clusters fill 5/6 of the
  // SMs, or 9/10 where halving eights gives a thread a second pack.  us, whole clusters against halves:
  //   16s  V = 22,988: 7 sequences 17.2 / 19.9, 8 22.4 / 21.9, 9 24.8 / 20.6; V = 11,325: 8 20.0 / 18.3, 9 21.4 / 17.9
  //   8s   V = 8000 (one pack): 15 sequences 19.1 / 19.7, 16 22.1 / 19.0, 20 26.5 / 19.9
  //        V = 13,000: 15 18.2 / 20.9, 16 19.9 / 22.2, 17 23.1 / 24.0, 18 22.3 / 20.9, 24 31.7 / 25.6
  const bool second_pack = cluster <= kAcceptCluster && a.V > cluster / 2 * kPack;
  if (a.mode == 1 && cluster > 4 && B * cluster > (second_pack ? 9 * sms / 10 : 5 * sms / 6) && a.V <= cluster / 2 * 4096) cluster >>= 1;
  const bool vec = (a.V & 3) == 0 && (reinterpret_cast<uintptr_t>(a.p_target) & 15) == 0 &&
                   (a.mode == 0 || ((reinterpret_cast<uintptr_t>(a.q_draft) | reinterpret_cast<uintptr_t>(a.noise)) & 15) == 0);
  const int chunk = ((a.V + cluster - 1) / cluster + 3) & ~3;
  constexpr size_t kSharedMost = 216 * 1024;
  const size_t held = (size_t)((chunk + kPack - 1) / kPack) * kPack;
  auto go = [&](auto mode_c, auto vec_c, auto* r_type) {
    using RT = std::remove_pointer_t<decltype(r_type)>;
    constexpr int kMode = decltype(mode_c)::value;
    auto kern = accept_kernel<kMode, decltype(vec_c)::value, RT>;
    static bool done[kMaxDevices] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    if (!done[dev]) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSharedMost);
      if (e != cudaSuccess) return e;
      done[dev] = true;
    }
    size_t smem = 0;
    if constexpr (kMode == 1 && !std::is_void_v<RT>) smem = held * (sizeof(RT) + 4);
    return launch_cluster_kernel(kern, dim3(cluster, B), dim3(kAcceptThreads), cluster, smem, st, pdl, t, N, Ns, a, lmax, chunk, accepted,
                                 len, next_token, final_node);
  };
  auto pick = [&](auto vec_c) {
    constexpr std::integral_constant<int, 0> greedy;
    constexpr std::integral_constant<int, 1> rejection;
    if (a.mode == 0) return go(greedy, vec_c, (void*)nullptr);
    if (held * 12 <= kSharedMost) return go(rejection, vec_c, (double*)nullptr);
    if (held * 8 <= kSharedMost) return go(rejection, vec_c, (float*)nullptr);
    return go(rejection, vec_c, (void*)nullptr);
  };
  return vec ? pick(std::true_type{}) : pick(std::false_type{});
}

}  // namespace lumo
