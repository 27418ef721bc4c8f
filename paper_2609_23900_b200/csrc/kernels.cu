// sm_100a kernels of the GDN tree verifier: tree convolution, rank-1 tree scan, commit.
//
// Row independence is what the layout is built on: row r of the d_v x d_k state evolves
// alone (S[r,:] <- a S[r,:] + delta_r k^T with delta_r = b (v_r - a S[r,:].k)), so a CTA
// owns 32 rows of one (sequence, value head) and walks the WHOLE tree with them, four lanes
// per row, each lane holding d_k/4 fp32 state values in registers (paper Eq. 2-3; Sec.
// "Path-parallel verification and state lifetime": the working tile keeps the full key
// dimension and is reused along the path instead of being reloaded per node).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <climits>
#include <mutex>
#include <type_traits>

#include "conv_split.h"
#include "internal.h"

namespace lumo {

namespace {

constexpr int kRows = 32;        // state rows per CTA
constexpr int kLanesPerRow = 4;
constexpr int kScanThreads = kRows * kLanesPerRow;   // 128
constexpr int kRingDepth = 6;    // staged node operands in flight

// ---------------------------------------------------------------------------------------
// small helpers
// ---------------------------------------------------------------------------------------
template <typename T> struct Vec4;   // four consecutive elements -> float4
template <> struct Vec4<float> {
  static __device__ __forceinline__ float4 load(const float* p) { return *reinterpret_cast<const float4*>(p); }
};
template <> struct Vec4<__nv_bfloat16> {
  static __device__ __forceinline__ float4 load(const __nv_bfloat16* p) {
    uint2 r = *reinterpret_cast<const uint2*>(p);
    return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xFFFF0000u),
                       __uint_as_float(r.y << 16), __uint_as_float(r.y & 0xFFFF0000u));
  }
};

__device__ __forceinline__ void store_scalar(void* p, size_t i, int dtype, float v) {
  if (dtype == LUMO_BF16) reinterpret_cast<__nv_bfloat16*>(p)[i] = __float2bfloat16_rn(v);
  else reinterpret_cast<float*>(p)[i] = v;
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

__device__ __forceinline__ float ex2_approx(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ float rcp_approx(float x) { float y; asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }

template <typename T> struct Packed4;      // four consecutive elements as loaded
template <> struct Packed4<float> {
  using type = float4;
  static __device__ __forceinline__ float4 unpack(const float4& p) { return p; }
};
template <> struct Packed4<__nv_bfloat16> {
  using type = uint2;
  static __device__ __forceinline__ float4 unpack(const uint2& r) {
    return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xFFFF0000u),
                       __uint_as_float(r.y << 16), __uint_as_float(r.y & 0xFFFF0000u));
  }
};

// The convolution's taps of four neighbouring channels, and the sum over a window of four rows, r0 the oldest: oldest first from
// zero in fp32, the same bits in either form.
template <typename T> struct ConvTaps;
template <> struct ConvTaps<float> {                   // tap j of the channel pairs (0, 1) and (2, 3): packed FMAs
  float2 w[4][2] = {};
  __device__ __forceinline__ void load(const float* p) {
    float4 c[4];                                       // the taps of channel e
#pragma unroll
    for (int e = 0; e < 4; ++e) c[e] = *reinterpret_cast<const float4*>(p + e * 4);
    w[0][0] = make_float2(c[0].x, c[1].x); w[0][1] = make_float2(c[2].x, c[3].x);
    w[1][0] = make_float2(c[0].y, c[1].y); w[1][1] = make_float2(c[2].y, c[3].y);
    w[2][0] = make_float2(c[0].z, c[1].z); w[2][1] = make_float2(c[2].z, c[3].z);
    w[3][0] = make_float2(c[0].w, c[1].w); w[3][1] = make_float2(c[2].w, c[3].w);
  }
  __device__ __forceinline__ void sum(const float4& r0, const float4& r1, const float4& r2, const float4& r3, float2 (&y)[2]) const {
    const float2 zero2 = make_float2(0.f, 0.f);
    y[0] = __ffma2_rn(w[0][0], make_float2(r0.x, r0.y), zero2); y[1] = __ffma2_rn(w[0][1], make_float2(r0.z, r0.w), zero2);
    y[0] = __ffma2_rn(w[1][0], make_float2(r1.x, r1.y), y[0]);  y[1] = __ffma2_rn(w[1][1], make_float2(r1.z, r1.w), y[1]);
    y[0] = __ffma2_rn(w[2][0], make_float2(r2.x, r2.y), y[0]);  y[1] = __ffma2_rn(w[2][1], make_float2(r2.z, r2.w), y[1]);
    y[0] = __ffma2_rn(w[3][0], make_float2(r3.x, r3.y), y[0]);  y[1] = __ffma2_rn(w[3][1], make_float2(r3.z, r3.w), y[1]);
  }
};
template <> struct ConvTaps<__nv_bfloat16> {           // as loaded: a product of two bf16 values and an fp32 sum are one
  uint2 w[4] = {};                                     // instruction (sm_100), where widening both first takes one each
  __device__ __forceinline__ void load(const __nv_bfloat16* p) {
    const uint4 lo = *reinterpret_cast<const uint4*>(p), hi = *reinterpret_cast<const uint4*>(p + 8);
    w[0] = make_uint2(lo.x, lo.y); w[1] = make_uint2(lo.z, lo.w);
    w[2] = make_uint2(hi.x, hi.y); w[3] = make_uint2(hi.z, hi.w);
  }
  static __device__ __forceinline__ unsigned short element(const uint2& p, int i) {
    const uint32_t word = i & 2 ? p.y : p.x;
    return (unsigned short)(i & 1 ? word >> 16 : word & 0xFFFF);
  }
  __device__ __forceinline__ float channel(const uint2 (&r)[4], int e) const {
    float c = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float d;
      asm("fma.rn.f32.bf16 %0, %1, %2, %3;" : "=f"(d) : "h"(element(w[e], j)), "h"(element(r[j], e)), "f"(c));
      c = d;
    }
    return c;
  }
  __device__ __forceinline__ void sum(const uint2& r0, const uint2& r1, const uint2& r2, const uint2& r3, float2 (&y)[2]) const {
    const uint2 r[4] = {r0, r1, r2, r3};
    y[0] = make_float2(channel(r, 0), channel(r, 1));
    y[1] = make_float2(channel(r, 2), channel(r, 3));
  }
};

// one-shot mbarrier for a bulk copy into shared memory
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init1(unsigned long long* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(bar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned long long* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// `bytes` (a multiple of 16) between 16-byte aligned addresses, by one thread; counted on `bar`
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, unsigned long long* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
               ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
// Bounded wait for the first phase: false if it did not complete within 2^20 polls (each may sleep a few us).
__device__ __forceinline__ bool mbar_wait0(unsigned long long* bar) {
  const uint32_t addr = smem_u32(bar);
  for (uint32_t spin = 0; spin < (1u << 20); ++spin) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done) : "r"(addr) : "memory");
    if (done) return true;
  }
  return false;
}

// ---------------------------------------------------------------------------------------
// a1: ancestry-gathered causal depthwise conv (width 4) + SiLU -> recorded operands
// ---------------------------------------------------------------------------------------
// A warp owns a run of kRun consecutive entries of one sequence's visiting order (depth first, built on the host) and
// 128 channels, a lane four of them; the warps of a CTA are the runs of the sequence (up to eight, up to 8 kRun entries)
// times as many channel groups as make eight.  The CTA's rows of x and the three history rows are pulled into shared
// memory by cp.async, every one exactly once and all at once, so that a window costs shared-memory loads only, wherever
// its rows lie in the tree.
//
// An entry takes its four rows from there and is done: nothing is carried from one entry to the next.  (The transposed form,
// which hands a parent's partial sums down, reads a row once instead of four times, but telling the cases apart, starting
// sums over and pairing registers for them cost more: 101 against 76 warp instructions per entry and 128 channels, 48 layers.)
// Every sum takes its taps oldest first from zero in fp32 (bf16 by the mixed fma, fp32 by packed FMAs: two correctly rounded
// lanes per instruction, the same bits as scalar fmaf), bias last, SiLU in fp32, one round-to-nearest-even cast (Sec. "Precompute
// branch histories while preserving arithmetic": tap order and cast points are part of the result).
//
// What bounds it: instruction issue (70 % of the slots; the SiLU alone is 14 instructions per four channels, 8 of them special-
// function operations, whose unit is half busy) with HBM behind it (0.5 to 0.6 of the copy rate by the bytes it cannot do without).
// Kernel times against the transposed form, bf16: 48 layers of 4 x 32 nodes 51.6 -> 41.0 us, 32 x 256 nodes 69.6 -> 61.4, 8 x 64
// nodes 7.8 -> 6.2.  Five or six CTAs per SM instead of four spill: 46.7 and 50.0 us against 44.5; two entries at a time instead
// of eight 44.5.
// fp32 rows take twice the registers: one entry at a time and no window kept is what fits 64 of them without spills (63).  As the
// bf16 form has it, with scalar fmaf (84 bytes spilled), it lost to the transposed form: 8 x 64 nodes of 4096 channels 6.5 (transposed)
// -> 6.9 -> 6.3 us (now), spines of 64 7.3 -> 8.1 -> 7.2, 32 x 256 of 8192 channels 105 -> 115 -> 105; three CTAs per SM with room for
// everything 8.1 us (8 x 64: no longer one wave).  Where a sequence falls into several parts, the window of a part's first entry is
// staged with the part's own rows, so that whoever shares it (in a star everyone) does not go to L1 for it: 32 stars of 256 nodes, fp32,
// 102.5 (transposed) -> 111.5 (fetched by every entry) -> 103.0 us (now), 12 x 140 nodes 22.9 -> 25.1 -> 22.4;
// bf16 stars 61.1 -> 58.4, other trees of several parts within 2 % of before.

// kFused: the three history rows are the ones the previous cycle's accepted path will commit, i.e. the
// last three of [old history ; raw inputs of the accepted nodes], read in place through the path (the
// scan that follows writes them to the history buffer once every CTA of this kernel has finished).
// What the main loop needs of an entry, in one 16-byte load: its physical row, and its window as byte offsets in the tile,
// oldest first, or ~visiting place for a row that another CTA's part holds.
struct alignas(16) ConvEntry { int phys, w0, w1, w2; };

template <typename T, int kRun, bool kFused, class LB>
__device__ __forceinline__ void conv_body(const Shape& s, const TreeDev& t, const LB& lb, const ConvSplit& sp, const FusedPrevT<LB>* fp) {
  extern __shared__ __align__(128) unsigned char conv_smem[];            // [runs * kRun + 3 (+ 3) rows][groups * 128 channels]
  __shared__ ConvEntry s_entry[kConvMaxEntries];
  __shared__ int f_acc[kFusedMaxPath], f_par[kFusedMaxPath], f_phys[kFusedMaxPath];
  __shared__ const T* f_hsrc[3];
  using P4 = typename Packed4<T>::type;                // four elements as loaded
  const int b = blockIdx.y, layer = blockIdx.z;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int seg = (int)blockIdx.x >= sp.slabs ? blockIdx.x / sp.slabs : 0, slab = blockIdx.x - seg * sp.slabs;
  const int entries = sp.runs * kRun, e0 = seg * entries;               // this CTA's part of the visiting order
  const int cbase = slab * (128 << sp.log_groups);                      // and of the channels
  const int row_bytes = (128 << sp.log_groups) * (int)sizeof(T);
  const LayerPtrs& L = lb.l[layer];
  const int32_t* prog_g = t.conv_prog + (size_t)b * s.Ns;
  // The window of the part's first entry lies in other parts; its rows are staged behind the history, for all who share them
  // (a part of a star: every entry).
  int4 before = make_int4(-1, -1, -1, -1);
  if (seg > 0) before = *reinterpret_cast<const int4*>(t.win + ((size_t)b * s.Ns + e0) * 4);
  if (tid < entries) {                                 // descriptor tables: nobody writes them
    const int e = e0 + tid;
    if (e < s.Ns) {
      const int4 w = *reinterpret_cast<const int4*>(t.win + ((size_t)b * s.Ns + e) * 4);
      auto place = [&](int v) {
        if (v < 0) return (entries + 3 + v) * row_bytes;
        if (v >= e0) return (v - e0) * row_bytes;
        return v == before.z ? (entries + 5) * row_bytes : v == before.y ? (entries + 4) * row_bytes : v == before.x ? (entries + 3) * row_bytes : ~v;
      };
      s_entry[tid] = {prog_g[e], place(w.x), place(w.y), place(w.z)};
    }
  }
  pdl_wait();       // x, history and the operand buffers belong to earlier kernels until here
  pdl_trigger();
  const int row = L.state_row[b];
  const bool seq_ok = row >= 0 && row < s.n_state_rows;
  const T* xb = reinterpret_cast<const T*>(L.x) + (size_t)b * s.Ns * s.C + cbase;
  // ---- rows of x in visiting order (padding rows come last and are not read), history rows: a thread keeps to one
  //      16-byte column ------------------------------------------------------------------------------------------------
  constexpr int kVec = 16 / (int)sizeof(T);
  const int log_cols = (sizeof(T) == 2 ? 4 : 5) + sp.log_groups, col = (tid & ((1 << log_cols) - 1)) * kVec;
  const int step = (int)blockDim.x >> log_cols;         // rows per round: a multiple of the runs
  const bool col_ok = cbase + col < s.C;
  unsigned char* mycol = conv_smem + col * (int)sizeof(T);
  if (col_ok) {
    const int live = seq_ok ? min(s.N - e0, entries) : 0;
    const T* src = xb + col;
#pragma unroll 4
    for (int e = tid >> log_cols; e < live; e += step)
      cp_async16(mycol + e * row_bytes, src + (size_t)((uint32_t)prog_g[e0 + e] * (uint32_t)s.C));
    if (seg > 0 && live > 0)
      for (int j = tid >> log_cols; j < 3; j += step) {
        const int v = j == 0 ? before.x : j == 1 ? before.y : before.z;
        if (v >= 0) cp_async16(mycol + (entries + 3 + j) * row_bytes, src + (size_t)((uint32_t)prog_g[v] * (uint32_t)s.C));
      }
  }
  const T* hbase = reinterpret_cast<const T*>(L.conv_hist) + (size_t)(seq_ok ? row : 0) * 3 * s.C;
  if constexpr (kFused) {
    if (warp == 0) {
      const int plen = fp->len[b];
      if (lane < fp->lmax) {                             // every place: the length is still on its way
        const int a = fp->accepted[(size_t)b * fp->lmax + lane];
        const bool ok = a >= 0 && a < fp->N;
        f_acc[lane] = a;
        f_par[lane] = ok ? fp->parent[(size_t)b * fp->N + a] : -2;
        f_phys[lane] = ok ? fp->slot[(size_t)b * fp->N + a] : 0;
      }
      __syncwarp();
      if (lane < 3) {
        // an invalid or empty path commits nothing: the history in memory is the history
        const bool ok = seq_ok && check_path_staged(f_acc, f_par, fp->N, plen, fp->lmax) == LUMO_SEQ_OK;
        const int q = (ok ? plen : 0) + lane;          // index into [old0 old1 old2 x_a0 x_a1 ...]
        const T* xprev = reinterpret_cast<const T*>(fp->lb.l[layer].x) + (size_t)b * fp->Ns * s.C;
        f_hsrc[lane] = q < 3 ? hbase + (size_t)q * s.C : xprev + (size_t)f_phys[q - 3] * s.C;
      }
    }
    __syncthreads();
  }
  if (col_ok)
    for (int j = tid >> log_cols; j < 3; j += step) {
      const T* src = hbase + (size_t)j * s.C;
      if constexpr (kFused) src = f_hsrc[j];
      cp_async16(mycol + (entries + j) * row_bytes, src + cbase + col);
    }
  cp_async_commit();
  // ---- taps and bias of this lane's four channels --------------------------------------------------------------------
  const int run = warp >> sp.log_groups, cg = (warp & (sp.groups - 1)) * 128 + lane * 4, c0 = cbase + cg;
  const bool mine = c0 < s.C;
  ConvTaps<T> taps;
  float2 bias[2] = {};
  if (mine) {
    taps.load(reinterpret_cast<const T*>(L.conv_w) + (size_t)c0 * 4);
    if (L.conv_b) {
      const float4 bv = Packed4<T>::unpack(*reinterpret_cast<const P4*>(reinterpret_cast<const T*>(L.conv_b) + c0));
      bias[0] = make_float2(bv.x, bv.y);
      bias[1] = make_float2(bv.z, bv.w);
    }
  }
  cp_async_wait<0>();
  __syncthreads();
  const int first = e0 + run * kRun, live = seq_ok ? min(s.N - first, kRun) : 0;       // padding rows come last
  const ConvEntry* ent = s_entry + run * kRun;
  const bool elsewhere = __any_sync(0xffffffffu, lane < live && (ent[lane].w0 | ent[lane].w1 | ent[lane].w2) < 0);
  if (!mine) return;
  const bool has_bias = L.conv_b != nullptr;
  const int hkd = s.Hk * s.d;
  T* dst;
  uint32_t dst_stride;
  if (c0 < hkd) { dst = reinterpret_cast<T*>(L.q) + c0; dst_stride = hkd; }
  else if (c0 < 2 * hkd) { dst = reinterpret_cast<T*>(L.k) + (c0 - hkd); dst_stride = hkd; }
  else { dst = reinterpret_cast<T*>(L.v) + (c0 - 2 * hkd); dst_stride = (uint32_t)s.Hv * s.d; }
  dst += (size_t)b * s.Ns * dst_stride;
  const unsigned char* tile = conv_smem + cg * (int)sizeof(T);
  const float2 zero2 = make_float2(0.f, 0.f);
  const unsigned char* own = tile + run * kRun * row_bytes;
  auto put = [&](int phys, float2 y0, float2 y1) {
    T* d = dst + (size_t)((uint32_t)phys * dst_stride);
    if constexpr (sizeof(T) == 2) {
      __nv_bfloat162 h01 = __floats2bfloat162_rn(y0.x, y0.y), h23 = __floats2bfloat162_rn(y1.x, y1.y);
      *reinterpret_cast<uint2*>(d) = make_uint2(*reinterpret_cast<uint32_t*>(&h01), *reinterpret_cast<uint32_t*>(&h23));
    } else {
      *reinterpret_cast<float4*>(d) = make_float4(y0.x, y0.y, y1.x, y1.y);
    }
  };
  auto entries_of_run = [&](auto elsewhere_c) {        // elsewhere: a window reaches into another CTA's part
    auto row = [&](int at) -> P4 { return *reinterpret_cast<const P4*>(tile + at); };
    auto row_anywhere = [&](int at) -> P4 {
      if (at >= 0) return row(at);
      return *reinterpret_cast<const P4*>(xb + cg + (size_t)((uint32_t)prog_g[~at] * (uint32_t)s.C));
    };
    // bf16: eight entries at a time, and a window that reaches elsewhere kept for the siblings behind it in the run.  fp32 has no
    // registers for either: see above.
    constexpr int kAtATime = sizeof(T) == 2 ? 8 : 1;
    [[maybe_unused]] P4 far[3] = {};                   // the last window that reached elsewhere, and the parent it belongs to
    [[maybe_unused]] int of = INT_MIN;
#pragma unroll kAtATime
    for (int rr = 0; rr < live; ++rr) {                // bounded: kRun
      const ConvEntry en = ent[rr];
      const P4 r3 = *reinterpret_cast<const P4*>(own + rr * row_bytes);
      P4 r0, r1, r2;
      if (decltype(elsewhere_c)::value && __builtin_expect((en.w0 | en.w1 | en.w2) < 0, 0)) {    // uniform
        if constexpr (sizeof(T) == 2) {
          if (en.w2 != of) {
            far[0] = row_anywhere(en.w0); far[1] = row_anywhere(en.w1); far[2] = row_anywhere(en.w2);
            of = en.w2;
          }
          r0 = far[0]; r1 = far[1]; r2 = far[2];
        } else {
          r0 = row_anywhere(en.w0); r1 = row_anywhere(en.w1); r2 = row_anywhere(en.w2);
        }
      } else {
        r0 = row(en.w0); r1 = row(en.w1); r2 = row(en.w2);
      }
      float2 y[2];
      taps.sum(r0, r1, r2, r3, y);
      if (has_bias) { y[0] = __fadd2_rn(y[0], bias[0]); y[1] = __fadd2_rn(y[1], bias[1]); }   // bias last
      // SiLU a / (1 + 2^(-a log2 e)) with the hardware exponential and reciprocal (1e-6 relative, far
      // below the rounding of the recorded operand); the multiplies and the add are packed
      const float2 nl2e = make_float2(-1.4426950408889634f, -1.4426950408889634f), one = make_float2(1.f, 1.f);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        float2 ex = __fmul2_rn(y[e], nl2e);
        ex = __fadd2_rn(make_float2(ex2_approx(ex.x), ex2_approx(ex.y)), one);
        y[e] = __fmul2_rn(y[e], make_float2(rcp_approx(ex.x), rcp_approx(ex.y)));
      }
      put(en.phys, y[0], y[1]);
    }
  };
  if (elsewhere) entries_of_run(std::true_type{});
  else entries_of_run(std::false_type{});
  for (int rr = max(live, 0); rr < min(s.Ns - first, kRun); ++rr) put(ent[rr].phys, zero2, zero2);   // padding rows, skipped sequences
}

template <typename T, int kRun, class LB>
__global__ void __launch_bounds__(32 * kConvWarps, 4) conv_kernel(Shape s, TreeDev t, LB lb, ConvSplit sp) {
  conv_body<T, kRun, false, LB>(s, t, lb, sp, nullptr);
}
template <typename T, int kRun, class LB>
__global__ void __launch_bounds__(32 * kConvWarps, 4) conv_fused_kernel(Shape s, TreeDev t, LB lb, ConvSplit sp, FusedPrevT<LB> fp) {
  conv_body<T, kRun, true, LB>(s, t, lb, sp, &fp);
}

// ---------------------------------------------------------------------------------------
// a3: rank-1 tree scan
// ---------------------------------------------------------------------------------------
template <int D, typename T>
struct ScanCfg {
  static constexpr int kChunks = D / 16;            // float4 chunks per lane
  static constexpr int kStageElems = 2 * D + kRows; // k row, q row, v slice
  static constexpr int kStageBytes = kStageElems * (int)sizeof(T);
  static constexpr int kStageXfers = kStageBytes / 16;
  static constexpr int kKXfers = D * (int)sizeof(T) / 16;
};

// dynamic shared memory layout (bytes), computed identically on host and device
struct ScanSmem {
  int ops, slot, params, dcache, snaplist, ring, total;
};
__host__ __device__ inline ScanSmem scan_smem(int N, int max_ops, int n_snap_list, int stage_bytes) {
  ScanSmem m;
  int off = 0;
  m.ops = off;      off += ((max_ops * 4 + 15) / 16) * 16;
  m.slot = off;     off += ((N * 4 + 15) / 16) * 16;
  m.params = off;   off += 5 * N * 4;  off = (off + 15) / 16 * 16;
  m.dcache = off;   off += N * kRows * 4;
  m.snaplist = off; off += ((n_snap_list * 4 + 15) / 16) * 16;
  m.ring = off;     off += kRingDepth * stage_bytes;
  m.total = off;
  return m;
}

template <int D, typename T, class LB>
__global__ void __launch_bounds__(kScanThreads)
scan_kernel(Shape s, TreeDev t, LB lb, float* __restrict__ stack, int n_items) {
  using Cfg = ScanCfg<D, T>;
  constexpr int NCH = Cfg::kChunks;
  extern __shared__ __align__(16) unsigned char smem[];
  const int n_snap_list = s.snapshot_mode == 1 ? s.n_snap : 0;
  const ScanSmem lay = scan_smem(s.N, t.max_ops, n_snap_list, Cfg::kStageBytes);
  int32_t* s_ops = reinterpret_cast<int32_t*>(smem + lay.ops);
  int32_t* s_slot = reinterpret_cast<int32_t*>(smem + lay.slot);   // physical row of each node
  float* p_a = reinterpret_cast<float*>(smem + lay.params);
  float* p_b = p_a + s.N;
  float* p_ks = p_b + s.N;      // multiplies the raw key (1 / norm when normalising)
  float* p_qs = p_ks + s.N;     // multiplies the raw query (scale / norm)
  float* p_kq = p_qs + s.N;     // k_n . q_n with both factors applied
  float* s_dc = reinterpret_cast<float*>(smem + lay.dcache);
  int32_t* s_snap = reinterpret_cast<int32_t*>(smem + lay.snaplist);
  unsigned char* s_ring = smem + lay.ring;

  const int tid = threadIdx.x;
  const int j = tid & 3;               // lane within the row group
  const int rl = tid >> 2;             // local row 0..31
  constexpr int kTiles = D / kRows;
  const int rep = s.Hv / s.Hk;
  float* my_stack = stack + (size_t)blockIdx.x * t.max_levels * (kRows * D);

  for (int item = blockIdx.x; item < n_items; item += gridDim.x) {   // bounded: n_items
    const int tile = item % kTiles;
    const int hv = (item / kTiles) % s.Hv;
    const int b = (item / (kTiles * s.Hv)) % s.B;
    const int layer = item / (kTiles * s.Hv * s.B);
    const LayerPtrs& L = lb.l[layer];
    const int g = hv / rep;
    const int row = L.state_row[b];
    const int r0 = tile * kRows;
    const size_t out_row_stride = (size_t)s.Hv * D;
    __syncthreads();   // previous item's shared memory is no longer in use

    if (row < 0 || row >= s.n_state_rows) {
      // skipped sequence: zero outputs; flag a row outside the pool
      for (int e = tid; e < s.Ns * kRows; e += kScanThreads)
        store_scalar(L.out, ((size_t)b * s.Ns + e / kRows) * out_row_stride + hv * D + r0 + e % kRows,
                     s.out_dtype, 0.f);
      if (L.status && hv == 0 && tile == 0 && tid == 0) L.status[b] = row < 0 ? LUMO_SEQ_OK : LUMO_SEQ_BAD_ROW;
      continue;
    }
    if (L.status && hv == 0 && tile == 0 && tid == 0) L.status[b] = LUMO_SEQ_OK;

    // pre-tree state tile -> registers (issued first so the loads overlap the prologue)
    const float* S0 = L.state + (((size_t)row * s.Hv + hv) * D + r0 + rl) * D;
    float4 S[NCH];
#pragma unroll
    for (int m = 0; m < NCH; ++m) S[m] = *reinterpret_cast<const float4*>(S0 + 16 * m + 4 * j);

    const int nops = t.nops[b];
    const int32_t* ops_g = t.sched + (size_t)b * t.max_ops;
    for (int e = tid; e < nops; e += kScanThreads) s_ops[e] = ops_g[e];
    for (int e = tid; e < s.N; e += kScanThreads) s_slot[e] = t.slot[b * s.N + e];
    for (int e = tid; e < n_snap_list; e += kScanThreads) s_snap[e] = L.snap_nodes[(size_t)b * s.n_snap + e];
    // padding rows: zero outputs
    for (int e = tid; e < s.Ns * kRows; e += kScanThreads) {
      int ps = e / kRows;
      if (t.slot_inv[b * s.Ns + ps] < 0)
        store_scalar(L.out, ((size_t)b * s.Ns + ps) * out_row_stride + hv * D + r0 + e % kRows, s.out_dtype, 0.f);
    }
    // per-node scalars: gates, normalisation factors, k.q
    const T* qg = reinterpret_cast<const T*>(L.q);
    const T* kg = reinterpret_cast<const T*>(L.k);
    const T* vg = reinterpret_cast<const T*>(L.v);
    {
      // eight lanes per node, sixteen nodes in flight per pass; the trip count is uniform over
      // the CTA so that every lane takes part in the shuffles
      const int grp = tid >> 3, gl = tid & 7;
#pragma unroll 2
      for (int n0 = 0; n0 < s.N; n0 += kScanThreads / 8) {
        const int n = n0 + grp;
        const bool live = n < s.N;
        const size_t pr = (size_t)b * s.Ns + (live ? t.slot[b * s.N + n] : 0);
        const T* kr = kg + (pr * s.Hk + g) * D;
        const T* qr = qg + (pr * s.Hk + g) * D;
        float kk = 0.f, qq = 0.f, kq = 0.f;
        if (live) {
#pragma unroll
          for (int c = 0; c < D / 32; ++c) {
            float4 kv = Vec4<T>::load(kr + gl * 4 + 32 * c), qv = Vec4<T>::load(qr + gl * 4 + 32 * c);
            kk += kv.x * kv.x + kv.y * kv.y + kv.z * kv.z + kv.w * kv.w;
            qq += qv.x * qv.x + qv.y * qv.y + qv.z * qv.z + qv.w * qv.w;
            kq += kv.x * qv.x + kv.y * qv.y + kv.z * qv.z + kv.w * qv.w;
          }
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
          kk += __shfl_xor_sync(0xffffffffu, kk, o);
          qq += __shfl_xor_sync(0xffffffffu, qq, o);
          kq += __shfl_xor_sync(0xffffffffu, kq, o);
        }
        if (live && gl == 0) {
          float ks = 1.f, qs = s.scale;
          if (s.l2norm) { ks = rsqrtf(kk + s.l2_eps); qs = s.scale * rsqrtf(qq + s.l2_eps); }
          p_ks[n] = ks; p_qs[n] = qs; p_kq[n] = kq * ks * qs;
          const float2 gates = load_gates(L, s, pr * s.Hv + hv, hv);
          p_a[n] = gates.x;
          p_b[n] = gates.y;
        }
      }
    }
    __syncthreads();

    // operand ring: stage i holds k row, q row and this tile's v slice of op i's node
    auto prefetch = [&](int i) {
      if (i < nops) {
        const int op = s_ops[i];
        const int kind = op >> 24;
        if (kind <= OP_DESCEND) {
          const int n = op & 0xFFFF;
          const size_t pr = (size_t)b * s.Ns + s_slot[n];
          unsigned char* st = s_ring + (i % kRingDepth) * Cfg::kStageBytes;
          const int nx = kind == OP_DESCEND ? Cfg::kKXfers : Cfg::kStageXfers;
          if (tid < nx) {
            const unsigned char* src;
            if (tid < Cfg::kKXfers) src = reinterpret_cast<const unsigned char*>(kg + (pr * s.Hk + g) * D) + tid * 16;
            else if (tid < 2 * Cfg::kKXfers)
              src = reinterpret_cast<const unsigned char*>(qg + (pr * s.Hk + g) * D) + (tid - Cfg::kKXfers) * 16;
            else
              src = reinterpret_cast<const unsigned char*>(vg + (pr * s.Hv + hv) * D + r0) + (tid - 2 * Cfg::kKXfers) * 16;
            cp_async16(st + tid * 16, src);
          }
        }
      }
      cp_async_commit();
    };
#pragma unroll
    for (int i = 0; i < kRingDepth - 1; ++i) prefetch(i);

    for (int i = 0; i < nops; ++i) {                   // bounded: nops <= max_ops
      cp_async_wait<kRingDepth - 2>();
      __syncthreads();
      prefetch(i + kRingDepth - 1);
      const int op = s_ops[i];
      const int kind = op >> 24;
      const int arg = op & 0xFFFF;
      const T* st_k = reinterpret_cast<const T*>(s_ring + (i % kRingDepth) * Cfg::kStageBytes);
      const T* st_q = st_k + D;
      const T* st_v = st_q + D;
      if (kind <= OP_EMIT_DESCEND) {
        const int n = arg;
        float u0 = 0.f, u1 = 0.f, w0 = 0.f, w1 = 0.f;
#pragma unroll
        for (int m = 0; m < NCH; ++m) {
          float4 kv = Vec4<T>::load(st_k + 16 * m + 4 * j);
          float4 qv = Vec4<T>::load(st_q + 16 * m + 4 * j);
          u0 = fmaf(S[m].x, kv.x, u0); u1 = fmaf(S[m].y, kv.y, u1);
          u0 = fmaf(S[m].z, kv.z, u0); u1 = fmaf(S[m].w, kv.w, u1);
          w0 = fmaf(S[m].x, qv.x, w0); w1 = fmaf(S[m].y, qv.y, w1);
          w0 = fmaf(S[m].z, qv.z, w0); w1 = fmaf(S[m].w, qv.w, w1);
        }
        float u = u0 + u1, w = w0 + w1;
        u += __shfl_xor_sync(0xffffffffu, u, 1); w += __shfl_xor_sync(0xffffffffu, w, 1);
        u += __shfl_xor_sync(0xffffffffu, u, 2); w += __shfl_xor_sync(0xffffffffu, w, 2);
        const float a = p_a[n], bt = p_b[n], ks = p_ks[n];
        float vv;
        if constexpr (sizeof(T) == 2) vv = __bfloat162float(st_v[rl]); else vv = st_v[rl];
        const float dl = bt * (vv - a * (ks * u));          // delta = beta (v - R' k)
        const float o = a * (p_qs[n] * w) + dl * p_kq[n];   // o = R q = a R_p q + delta (k.q)
        if (j == 0) {
          const size_t pr = (size_t)b * s.Ns + s_slot[n];
          store_scalar(L.out, pr * out_row_stride + hv * D + r0 + rl, s.out_dtype, o);
          if ((op >> 20) & 1) s_dc[n * kRows + rl] = dl;
        }
        if (kind == OP_EMIT_DESCEND) {
          const float gk = dl * ks;
#pragma unroll
          for (int m = 0; m < NCH; ++m) {
            float4 kv = Vec4<T>::load(st_k + 16 * m + 4 * j);
            S[m].x = fmaf(a, S[m].x, gk * kv.x); S[m].y = fmaf(a, S[m].y, gk * kv.y);
            S[m].z = fmaf(a, S[m].z, gk * kv.z); S[m].w = fmaf(a, S[m].w, gk * kv.w);
          }
        }
      } else if (kind == OP_DESCEND) {
        const int n = arg;
        const float a = p_a[n];
        const float gk = s_dc[n * kRows + rl] * p_ks[n];
#pragma unroll
        for (int m = 0; m < NCH; ++m) {
          float4 kv = Vec4<T>::load(st_k + 16 * m + 4 * j);
          S[m].x = fmaf(a, S[m].x, gk * kv.x); S[m].y = fmaf(a, S[m].y, gk * kv.y);
          S[m].z = fmaf(a, S[m].z, gk * kv.z); S[m].w = fmaf(a, S[m].w, gk * kv.w);
        }
      } else if (kind == OP_PUSH) {
        float* dst = my_stack + ((size_t)arg * kRows + rl) * D;
#pragma unroll
        for (int m = 0; m < NCH; ++m) *reinterpret_cast<float4*>(dst + 16 * m + 4 * j) = S[m];
      } else {  // OP_POP
        const float* src = arg == kPopRoot ? S0 : my_stack + ((size_t)arg * kRows + rl) * D;
#pragma unroll
        for (int m = 0; m < NCH; ++m) S[m] = *reinterpret_cast<const float4*>(src + 16 * m + 4 * j);
      }
      // node states on request: the registers now hold S_n
      if (s.snapshot_mode != 0 && (kind == OP_EMIT_DESCEND || kind == OP_DESCEND)) {
        const int n = arg;
        const int E = s.n_snap;
        if (s.snapshot_mode == 2) {
          float* dst = L.snap_out + ((((size_t)b * E + n) * s.Hv + hv) * D + r0 + rl) * D;
#pragma unroll
          for (int m = 0; m < NCH; ++m) *reinterpret_cast<float4*>(dst + 16 * m + 4 * j) = S[m];
        } else {
          for (int e = 0; e < E; ++e) {          // bounded: E
            if (s_snap[e] != n) continue;
            float* dst = L.snap_out + ((((size_t)b * E + e) * s.Hv + hv) * D + r0 + rl) * D;
#pragma unroll
            for (int m = 0; m < NCH; ++m) *reinterpret_cast<float4*>(dst + 16 * m + 4 * j) = S[m];
          }
        }
      }
    }
    cp_async_wait<0>();
  }
}

// ---- the same walk with every node's operands in shared memory ---------------------------------------
// For trees whose widened keys and queries fit (kStagedSmem): they are staged once per CTA, so the operations need no
// barrier and a warp (eight rows) walks the tree at its own pace.  64 rows per CTA share the staging and the per-node
// scalars.  In the snapshot modes a leaf's state is formed on its way to memory (a S_p + gk k) without disturbing the
// registers, and with every state exported a branching node's state is fetched back from the export instead of a stack.
// Bound by the state writes in the snapshot modes, by instruction latency in small launches.  Measured against the operand
// ring below: every state of 8 layers of 4 x 32 nodes (2.1 GB) 573 -> 415 us, 5 x 17 nodes of two layers 102 -> 86 us; a step
// of a seven-node fp32 tree (d = 64) 11.0 -> 8.3 us on the device.
constexpr int kStagedRows = 64;
constexpr int kStagedThreads = kStagedRows * kLanesPerRow;
constexpr int kStagedSmem = 112 * 1024;      // at least two CTAs per SM

struct StagedSmem { int ops, slot, params, snap, levels, k, q, v, dcache, total; };
__host__ __device__ inline StagedSmem staged_smem(int N, int D, int max_ops, int n_snap_list, int max_levels) {
  StagedSmem m;
  int off = 0;
  auto take = [&](int bytes) { const int at = off; off += (bytes + 15) / 16 * 16; return at; };
  m.k = take(N * D * 4);
  m.q = take(N * D * 4);
  m.v = take(N * kStagedRows * 4);           // values, then outputs
  m.dcache = take(N * kStagedRows * 4);
  m.params = take(5 * N * 4);
  m.ops = take(max_ops * 4);
  m.slot = take(N * 4);
  m.snap = take(n_snap_list * 4);
  m.levels = take(max_levels * (kStagedThreads / 32) * 4);
  m.total = off;
  return m;
}

template <int D, typename T, class LB>
__global__ void __launch_bounds__(kStagedThreads, 3)
scan_staged_kernel(Shape s, TreeDev t, LB lb, float* __restrict__ stack, int n_items) {
  constexpr int NCH = D / 16, kVec = 16 / (int)sizeof(T);
  extern __shared__ __align__(16) unsigned char smem[];
  const int n_snap_list = s.snapshot_mode == 1 ? s.n_snap : 0;
  const StagedSmem lay = staged_smem(s.N, D, t.max_ops, n_snap_list, t.max_levels);
  float* s_k = reinterpret_cast<float*>(smem + lay.k);
  float* s_q = reinterpret_cast<float*>(smem + lay.q);
  float* s_v = reinterpret_cast<float*>(smem + lay.v);
  float* s_dc = reinterpret_cast<float*>(smem + lay.dcache);
  float* p_a = reinterpret_cast<float*>(smem + lay.params);
  float* p_b = p_a + s.N;
  float* p_ks = p_b + s.N;      // multiplies the raw key (1 / norm when normalising)
  float* p_qs = p_ks + s.N;     // multiplies the raw query (scale / norm)
  float* p_kq = p_qs + s.N;     // k_n . q_n with both factors applied
  int32_t* s_ops = reinterpret_cast<int32_t*>(smem + lay.ops);
  int32_t* s_slot = reinterpret_cast<int32_t*>(smem + lay.slot);
  int32_t* s_snap = reinterpret_cast<int32_t*>(smem + lay.snap);

  const int tid = threadIdx.x, warp = tid >> 5;
  const int j = tid & 3;               // lane within the row group
  const int rl = tid >> 2;             // local row
  int32_t* lvl_node = reinterpret_cast<int32_t*>(smem + lay.levels) + warp * t.max_levels;   // node pushed at each level
  constexpr int kTiles = D / kStagedRows;
  const int rep = s.Hv / s.Hk;
  float* my_stack = stack + ((size_t)blockIdx.x * t.max_levels * kStagedRows + rl) * D + 4 * j;

  bool waited = false;
  for (int item = blockIdx.x; item < n_items; item += gridDim.x) {   // bounded: n_items
    const int tile = item % kTiles;
    const int hv = (item / kTiles) % s.Hv;
    const int b = (item / (kTiles * s.Hv)) % s.B;
    const int layer = item / (kTiles * s.Hv * s.B);
    const LayerPtrs& L = lb.l[layer];
    const int g = hv / rep;
    const int r0 = tile * kStagedRows;
    const size_t out_row_stride = (size_t)s.Hv * D;
    __syncthreads();   // previous item's shared memory is no longer in use
    const int nops = t.nops[b];
    for (int e = tid; e < nops; e += kStagedThreads) s_ops[e] = t.sched[(size_t)b * t.max_ops + e];
    for (int e = tid; e < s.N; e += kStagedThreads) s_slot[e] = t.slot[b * s.N + e];
    if (!waited) { pdl_wait(); pdl_trigger(); waited = true; }        // only descriptor tables were read so far
    const int row = L.state_row[b];
    const bool lead = L.status && hv == 0 && tile == 0 && tid == 0;
    if (row < 0 || row >= s.n_state_rows) {
      // skipped sequence: zero outputs; flag a row outside the pool
      for (int e = tid; e < s.Ns * kStagedRows; e += kStagedThreads)
        store_scalar(L.out, ((size_t)b * s.Ns + e / kStagedRows) * out_row_stride + hv * D + r0 + e % kStagedRows, s.out_dtype, 0.f);
      if (lead) L.status[b] = row < 0 ? LUMO_SEQ_OK : LUMO_SEQ_BAD_ROW;
      continue;
    }
    if (lead) L.status[b] = LUMO_SEQ_OK;

    // pre-tree state rows -> registers (issued first so the loads overlap the staging)
    const float* S0 = L.state + (((size_t)row * s.Hv + hv) * D + r0 + rl) * D + 4 * j;
    float4 S[NCH];
#pragma unroll
    for (int m = 0; m < NCH; ++m) S[m] = *reinterpret_cast<const float4*>(S0 + 16 * m);
    for (int e = tid; e < n_snap_list; e += kStagedThreads) s_snap[e] = L.snap_nodes[(size_t)b * s.n_snap + e];
    // padding rows: zero outputs
    if (s.Ns > s.N)
      for (int e = tid; e < s.Ns * kStagedRows; e += kStagedThreads) {
        const int ps = e / kStagedRows;
        if (t.slot_inv[b * s.Ns + ps] < 0)
          store_scalar(L.out, ((size_t)b * s.Ns + ps) * out_row_stride + hv * D + r0 + e % kStagedRows, s.out_dtype, 0.f);
      }
    // gates of this thread's node (a CTA has more threads than a staged tree has nodes)
    if (tid < s.N) {
      const float2 gates = load_gates(L, s, ((size_t)b * s.Ns + t.slot[b * s.N + tid]) * s.Hv + hv, hv);
      p_a[tid] = gates.x;
      p_b[tid] = gates.y;
    }
    __syncthreads();   // slots
    {
      const T* qg = reinterpret_cast<const T*>(L.q) + (size_t)b * s.Ns * s.Hk * D + g * D;
      const T* kg = reinterpret_cast<const T*>(L.k) + (size_t)b * s.Ns * s.Hk * D + g * D;
      const T* vg = reinterpret_cast<const T*>(L.v) + (size_t)b * s.Ns * s.Hv * D + hv * D + r0;
      auto put = [&](float* dst, const T* src) {
        const uint4 w = *reinterpret_cast<const uint4*>(src);
        if constexpr (sizeof(T) == 2) {
          reinterpret_cast<float4*>(dst)[0] = Packed4<T>::unpack(make_uint2(w.x, w.y));
          reinterpret_cast<float4*>(dst)[1] = Packed4<T>::unpack(make_uint2(w.z, w.w));
        } else {
          *reinterpret_cast<float4*>(dst) = *reinterpret_cast<const float4*>(&w);
        }
      };
      constexpr int kKP = D / kVec, kVP = kStagedRows / kVec;       // 16-byte pieces of a row
#pragma unroll 4
      for (int e = tid; e < s.N * kKP; e += kStagedThreads) {
        const int n = e / kKP, c = (e % kKP) * kVec;
        const size_t off = (size_t)((uint32_t)s_slot[n] * (uint32_t)(s.Hk * D)) + c;
        put(s_k + n * D + c, kg + off);
        put(s_q + n * D + c, qg + off);
      }
#pragma unroll 2
      for (int e = tid; e < s.N * kVP; e += kStagedThreads) {
        const int n = e / kVP, c = (e % kVP) * kVec;
        put(s_v + n * kStagedRows + c, vg + (size_t)((uint32_t)s_slot[n] * (uint32_t)(s.Hv * D)) + c);
      }
    }
    __syncthreads();
    {
      // per-node scalars: normalisation factors and k.q, eight lanes per node; the trip count is uniform over the CTA
      // so that every lane takes part in the shuffles
      const int grp = tid >> 3, gl = tid & 7;
      for (int n0 = 0; n0 < s.N; n0 += kStagedThreads / 8) {
        const int n = n0 + grp;
        const bool live = n < s.N;
        float kk = 0.f, qq = 0.f, kq = 0.f;
        if (live) {
#pragma unroll
          for (int c = 0; c < D / 32; ++c) {
            const float4 kv = *reinterpret_cast<const float4*>(s_k + n * D + gl * 4 + 32 * c), qv = *reinterpret_cast<const float4*>(s_q + n * D + gl * 4 + 32 * c);
            kk += kv.x * kv.x + kv.y * kv.y + kv.z * kv.z + kv.w * kv.w;
            qq += qv.x * qv.x + qv.y * qv.y + qv.z * qv.z + qv.w * qv.w;
            kq += kv.x * qv.x + kv.y * qv.y + kv.z * qv.z + kv.w * qv.w;
          }
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
          kk += __shfl_xor_sync(0xffffffffu, kk, o);
          qq += __shfl_xor_sync(0xffffffffu, qq, o);
          kq += __shfl_xor_sync(0xffffffffu, kq, o);
        }
        if (live && gl == 0) {
          float ks = 1.f, qs = s.scale;
          if (s.l2norm) { ks = rsqrtf(kk + s.l2_eps); qs = s.scale * rsqrtf(qq + s.l2_eps); }
          p_ks[n] = ks; p_qs[n] = qs; p_kq[n] = kq * ks * qs;
        }
      }
    }
    __syncthreads();

    // where node n's state goes (nullptr: nowhere); mode 1 may name a node more than once
    auto snap_at = [&](int e) { return L.snap_out + ((((size_t)b * s.n_snap + e) * s.Hv + hv) * D + r0 + rl) * D + 4 * j; };
    auto export_state = [&](int n, const float4 (&X)[NCH]) {
      if (s.snapshot_mode == 2) {
        float* dst = snap_at(n);
#pragma unroll
        for (int m = 0; m < NCH; ++m) *reinterpret_cast<float4*>(dst + 16 * m) = X[m];
      } else {
        for (int e = 0; e < s.n_snap; ++e) {          // bounded: the list
          if (s_snap[e] != n) continue;
          float* dst = snap_at(e);
#pragma unroll
          for (int m = 0; m < NCH; ++m) *reinterpret_cast<float4*>(dst + 16 * m) = X[m];
        }
      }
    };
    int cur = -1;                                      // node whose state the registers hold (-1: the pre-tree state)
#pragma unroll 1
    for (int i = 0; i < nops; ++i) {                   // bounded: nops <= max_ops
      const int op = s_ops[i];
      const int kind = op >> 24;
      const int arg = op & 0xFFFF;
      if (kind <= OP_DESCEND) {
        const int n = arg;
        const float* kr = s_k + n * D + 4 * j;
        const float a = p_a[n], ks = p_ks[n];
        float dl;
        if (kind == OP_DESCEND) {
          dl = s_dc[n * kStagedRows + rl];
        } else {
          const float* qr = s_q + n * D + 4 * j;
          float2 u2 = make_float2(0.f, 0.f), w2 = make_float2(0.f, 0.f);
#pragma unroll
          for (int m = 0; m < NCH; ++m) {
            const float4 kv = *reinterpret_cast<const float4*>(kr + 16 * m), qv = *reinterpret_cast<const float4*>(qr + 16 * m);
            const float2 lo = make_float2(S[m].x, S[m].y), hi = make_float2(S[m].z, S[m].w);
            u2 = __ffma2_rn(lo, make_float2(kv.x, kv.y), u2); u2 = __ffma2_rn(hi, make_float2(kv.z, kv.w), u2);
            w2 = __ffma2_rn(lo, make_float2(qv.x, qv.y), w2); w2 = __ffma2_rn(hi, make_float2(qv.z, qv.w), w2);
          }
          float u = u2.x + u2.y, w = w2.x + w2.y;
          u += __shfl_xor_sync(0xffffffffu, u, 1); w += __shfl_xor_sync(0xffffffffu, w, 1);
          u += __shfl_xor_sync(0xffffffffu, u, 2); w += __shfl_xor_sync(0xffffffffu, w, 2);
          float* vo = s_v + n * kStagedRows + rl;
          dl = p_b[n] * (*vo - a * (ks * u));                   // delta = beta (v - R' k)
          const float o = a * (p_qs[n] * w) + dl * p_kq[n];     // o = R q = a R_p q + delta (k.q)
          __syncwarp();                                         // the row's four lanes have read v
          if (j == 0) *vo = o;
          if ((op >> 20) & 1) {
            if (j == 0) s_dc[n * kStagedRows + rl] = dl;
            __syncwarp();
          }
        }
        // the node's state: in place of its parent's, or (a leaf, snapshots) formed on its way out
        const bool descend = kind != OP_EMIT;
        if (descend || (s.snapshot_mode != 0 && !((op >> 20) & 1))) {
          const float gk = dl * ks;
          const float2 a2 = make_float2(a, a), g2 = make_float2(gk, gk);
          auto child = [&](int m) {
            const float4 kv = *reinterpret_cast<const float4*>(kr + 16 * m);
            const float2 lo = __ffma2_rn(a2, make_float2(S[m].x, S[m].y), __fmul2_rn(g2, make_float2(kv.x, kv.y)));
            const float2 hi = __ffma2_rn(a2, make_float2(S[m].z, S[m].w), __fmul2_rn(g2, make_float2(kv.z, kv.w)));
            return make_float4(lo.x, lo.y, hi.x, hi.y);
          };
          asm volatile("" ::: "memory");                        // the key row is read again instead of being held in registers
          if (descend) {
#pragma unroll
            for (int m = 0; m < NCH; ++m) S[m] = child(m);
            cur = n;
            if (s.snapshot_mode != 0) export_state(n, S);
          } else if (s.snapshot_mode == 2) {
            float* dst = snap_at(n);
#pragma unroll
            for (int m = 0; m < NCH; ++m) *reinterpret_cast<float4*>(dst + 16 * m) = child(m);
          } else {
            for (int e = 0; e < s.n_snap; ++e) {                // bounded: the list
              if (s_snap[e] != n) continue;
              float* dst = snap_at(e);
#pragma unroll
              for (int m = 0; m < NCH; ++m) *reinterpret_cast<float4*>(dst + 16 * m) = child(m);
            }
          }
        }
      } else if (kind == OP_PUSH) {
        if (s.snapshot_mode == 2) {
          if ((tid & 31) == 0) lvl_node[arg] = cur;             // its state has just been exported
          __syncwarp();
        } else {
          float* dst = my_stack + (size_t)arg * kStagedRows * D;
#pragma unroll
          for (int m = 0; m < NCH; ++m) *reinterpret_cast<float4*>(dst + 16 * m) = S[m];
        }
      } else {  // OP_POP
        const float* src = S0;
        if (arg == kPopRoot) cur = -1;
        else if (s.snapshot_mode == 2) { cur = lvl_node[arg]; src = snap_at(cur); }
        else src = my_stack + (size_t)arg * kStagedRows * D;
#pragma unroll
        for (int m = 0; m < NCH; ++m) S[m] = *reinterpret_cast<const float4*>(src + 16 * m);
      }
    }
    __syncthreads();
    // outputs, two rows per thread
#pragma unroll 2
    for (int e = tid; e < s.N * (kStagedRows / 2); e += kStagedThreads) {
      const int n = e / (kStagedRows / 2), c = (e % (kStagedRows / 2)) * 2;
      const float2 o = *reinterpret_cast<const float2*>(s_v + n * kStagedRows + c);
      const size_t i = ((size_t)b * s.Ns + s_slot[n]) * out_row_stride + hv * D + r0 + c;
      if (s.out_dtype == LUMO_BF16) *reinterpret_cast<__nv_bfloat162*>(reinterpret_cast<__nv_bfloat16*>(L.out) + i) = __floats2bfloat162_rn(o.x, o.y);
      else *reinterpret_cast<float2*>(reinterpret_cast<float*>(L.out) + i) = o;
    }
  }
  if (!waited) pdl_wait();
}

// One token of the native recurrence on one state row, held by four lanes (lane j: floats 16 m + 4 j ..):
// S <- alpha S + delta ks k, delta = beta (v - alpha ks S.k).  Packed fp32 FMAs: two correctly rounded lanes per
// instruction, the same bits as the scalar form of the scan.
template <int D, typename T>
__device__ __forceinline__ void commit_token(float4 (&S)[D / 16], const float* k, T v, float2 gates, int l2norm, float l2_eps, int j) {
  constexpr int NCH = D / 16;
  float2 u2 = make_float2(0.f, 0.f), k2 = make_float2(0.f, 0.f);
#pragma unroll
  for (int m = 0; m < NCH; ++m) {
    const float4 kv = *reinterpret_cast<const float4*>(k + 16 * m + 4 * j);
    const float2 lo = make_float2(kv.x, kv.y), hi = make_float2(kv.z, kv.w);
    u2 = __ffma2_rn(make_float2(S[m].x, S[m].y), lo, u2);
    u2 = __ffma2_rn(make_float2(S[m].z, S[m].w), hi, u2);
    k2 = __ffma2_rn(lo, lo, k2);
    k2 = __ffma2_rn(hi, hi, k2);
    if (m == 3) asm volatile("" ::: "memory");   // half of the key row in flight at a time (registers)
  }
  float u = u2.x + u2.y, kk = k2.x + k2.y;
  u += __shfl_xor_sync(0xffffffffu, u, 1); kk += __shfl_xor_sync(0xffffffffu, kk, 1);
  u += __shfl_xor_sync(0xffffffffu, u, 2); kk += __shfl_xor_sync(0xffffffffu, kk, 2);
  float vv;
  if constexpr (sizeof(T) == 2) vv = __bfloat162float(v); else vv = v;
  const float a = gates.x;
  const float ks = l2norm ? rsqrtf(kk + l2_eps) : 1.f;
  const float dl = gates.y * (vv - a * (ks * u));
  const float gk = dl * ks;
  const float2 a2 = make_float2(a, a), g2 = make_float2(gk, gk);
  asm volatile("" ::: "memory");      // the key row is read again instead of being held in 32 registers
#pragma unroll
  for (int m = 0; m < NCH; ++m) {
    const float4 kv = *reinterpret_cast<const float4*>(k + 16 * m + 4 * j);
    const float2 lo = __ffma2_rn(a2, make_float2(S[m].x, S[m].y), __fmul2_rn(g2, make_float2(kv.x, kv.y)));
    const float2 hi = __ffma2_rn(a2, make_float2(S[m].z, S[m].w), __fmul2_rn(g2, make_float2(kv.z, kv.w)));
    S[m] = make_float4(lo.x, lo.y, hi.x, hi.y);
    if (m == 3) asm volatile("" ::: "memory");
  }
}

// ---------------------------------------------------------------------------------------
// a4 + a5: commit - replay the accepted path into the running state, in place, and gather the
// convolution history of the accepted path
// ---------------------------------------------------------------------------------------
// One launch.  The first CTAs of a (sequence, layer) each own ROWS rows of one value head's state: same per-token
// arithmetic as the scan's EMIT_DESCEND without the output, i.e. the "native per-token update" of Algorithm 2 applied
// for the accepted nodes in path order.  The remaining CTAs own 16-byte pieces of channels of the history rows: new
// history = last three rows of [old history ; x of the accepted nodes] (Algorithm 1).
//
// Bound by HBM: every state is read and written once.  What stands between that and the measured time is the chain row
// -> length -> path -> operands -> updates that each CTA goes through, so the state comes by bulk copy into shared
// memory, requested whole before that chain starts (three CTAs keep 192 KB per SM on the way), and the operands of up
// to kCommitChunk accepted nodes are fetched together instead of one node at a time.  Nothing is written unless the path
// is valid.  Measured: 48 layers of batch 4 (805 MB) 160 -> 141 us = 5.7 TB/s, 6 layers of batch 16 116 -> 89 us, one
// layer of batch 8 (a single wave) 15.4 -> 14.7 us.
constexpr int kCommitChunk = 8;   // accepted nodes whose operands are staged at a time

template <int D, typename T, int ROWS>
struct CommitCfg {
  static constexpr int kThreads = ROWS * 4 < 256 ? ROWS * 4 : 256;      // four lanes per row
  static constexpr int kPasses = ROWS * 4 / kThreads;
  static constexpr int kStateBytes = ROWS * D * 4;
  static constexpr int kBytes = kStateBytes + kCommitChunk * (D * 4 + ROWS * (int)sizeof(T));
};

template <int D, typename T, int ROWS, class LB>
__global__ void __launch_bounds__(CommitCfg<D, T, ROWS>::kThreads, ROWS == 32 ? 7 : 3)
commit_kernel(Shape s, TreeDev t, LB lb, const int32_t* __restrict__ accepted,
              const int32_t* __restrict__ len_arr, int lmax, int n_state_ctas) {
  using Cfg = CommitCfg<D, T, ROWS>;
  constexpr int NCH = D / 16, kThreads = Cfg::kThreads;
  constexpr int kTiles = D / ROWS;
  const int b = blockIdx.y, layer = blockIdx.z;
  const LayerPtrs& L = lb.l[layer];
  const int tid = threadIdx.x;
  if (s.wait_first) pdl_wait();
  const int row = L.state_row[b];
  const int len = len_arr[b];
  const bool lead = blockIdx.x == 0 && tid == 0;
  // What this kernel WRITES (state, history, status) may still be read by its predecessor (the scan
  // reads the pre-tree state), so every write sits behind pdl_wait().  What it READS ahead of that wait
  // (state tile, path, operands) must be older than its predecessor: that is so for a small launch right after a
  // verify call, whose own dependency wait orders everything before it.  Otherwise (wait_first) it reads nothing
  // ahead either, and the overlap hides its launch alone.
  if (row < 0) { pdl_wait(); if (lead && L.status) L.status[b] = LUMO_SEQ_OK; return; }
  if (row >= s.n_state_rows) { pdl_wait(); if (lead && L.status) L.status[b] = LUMO_SEQ_BAD_ROW; return; }
  const int32_t* acc = accepted + (size_t)b * lmax;
  // the whole path at once: entry t, its parent and its physical row (one level of dependent loads
  // instead of one per step)
  __shared__ int s_acc[kMaxNodes], s_par[kMaxNodes], s_phys[kMaxNodes];
  const int lcap = len < 0 ? 0 : (len > lmax ? 0 : len);

  if ((int)blockIdx.x >= n_state_ctas) {
    // ---- convolution history ------------------------------------------------------------------
    for (int tt = tid; tt < lcap; tt += kThreads) {       // bounded: lmax
      const int a = acc[tt];
      const bool ok = a >= 0 && a < s.N;
      s_acc[tt] = a;
      s_par[tt] = ok ? t.parent[(size_t)b * s.N + a] : -2;
      s_phys[tt] = ok ? t.slot[b * s.N + a] : 0;
    }
    constexpr int kVec = 16 / (int)sizeof(T);
    const int c0 = ((blockIdx.x - n_state_ctas) * kThreads + tid) * kVec;
    __syncthreads();
    // every exit path passes the dependency wait: a CTA that left without it would let this grid complete
    // (and its own dependent start) while the kernel before it is still running
    if (c0 >= s.C || L.x == nullptr) { pdl_wait(); return; }
    if (check_path_staged(s_acc, s_par, s.N, len, lmax) != LUMO_SEQ_OK || len == 0) { pdl_wait(); return; }
    T* hist = reinterpret_cast<T*>(L.conv_hist) + (size_t)row * 3 * s.C + c0;
    const T* x = reinterpret_cast<const T*>(L.x);
    uint4 v[3];
#pragma unroll
    for (int jj = 0; jj < 3; ++jj) {
      const int q = len + jj;        // index into [old0 old1 old2 x_a0 x_a1 ...]
      const T* src = q < 3 ? hist + (size_t)q * s.C
                           : x + ((size_t)b * s.Ns + s_phys[q - 3]) * s.C + c0;
      v[jj] = *reinterpret_cast<const uint4*>(src);
    }
    pdl_wait();
#pragma unroll
    for (int jj = 0; jj < 3; ++jj) *reinterpret_cast<uint4*>(hist + (size_t)jj * s.C) = v[jj];
    return;
  }

  // ---- state rows ---------------------------------------------------------------------------------
  extern __shared__ __align__(128) unsigned char commit_smem[];
  float* Ss = reinterpret_cast<float*>(commit_smem);                              // [ROWS][D]
  float* Ks = reinterpret_cast<float*>(commit_smem + Cfg::kStateBytes);           // [chunk][D], widened
  T* Vs = reinterpret_cast<T*>(commit_smem + Cfg::kStateBytes + kCommitChunk * D * 4);   // [chunk][ROWS]
  __shared__ float2 s_gate[kCommitChunk];
  __shared__ unsigned long long mbar;
  const int tile = blockIdx.x % kTiles, hv = blockIdx.x / kTiles;
  const int g = hv / (s.Hv / s.Hk);
  const int r0 = tile * ROWS;
  float* Sg = L.state + (((size_t)row * s.Hv + hv) * D + r0) * D;
  if (tid == 0) {
    mbar_init1(&mbar);
    if (lcap > 0) {                                                        // the rows are contiguous
      mbar_expect(&mbar, Cfg::kStateBytes);
      bulk_load(Ss, Sg, Cfg::kStateBytes, &mbar);
    }
  }
  for (int tt = tid; tt < lcap; tt += kThreads) {         // bounded: lmax
    const int a = acc[tt];
    const bool ok = a >= 0 && a < s.N;
    s_acc[tt] = a;
    s_par[tt] = ok ? t.parent[(size_t)b * s.N + a] : -2;
    s_phys[tt] = ok ? t.slot[b * s.N + a] : 0;
  }
  __syncthreads();
  int st = check_path_staged(s_acc, s_par, s.N, len, lmax);
  const T* kg = reinterpret_cast<const T*>(L.k);
  const T* vg = reinterpret_cast<const T*>(L.v);
  // operands of the accepted nodes [t0, t0 + n): widened key rows, this CTA's part of the value rows, gates
  auto stage = [&](int t0, int n) {
    constexpr int kVec = 16 / (int)sizeof(T), kKP = D / kVec, kVP = ROWS / kVec;
    for (int e = tid; e < n * (kKP + kVP); e += kThreads) {                // bounded: <= 2 rounds of bf16
      const int i = e / (kKP + kVP), c = e % (kKP + kVP);
      const size_t pr = (size_t)b * s.Ns + s_phys[t0 + i];
      if (c < kKP) {
        const uint4 w = *reinterpret_cast<const uint4*>(kg + (pr * s.Hk + g) * D + c * kVec);
        float4* dst = reinterpret_cast<float4*>(Ks + i * D + c * kVec);
        if constexpr (sizeof(T) == 2) {
          dst[0] = Packed4<T>::unpack(make_uint2(w.x, w.y));
          dst[1] = Packed4<T>::unpack(make_uint2(w.z, w.w));
        } else {
          dst[0] = *reinterpret_cast<const float4*>(&w);
        }
      } else {
        *reinterpret_cast<uint4*>(Vs + i * ROWS + (c - kKP) * kVec) =
            *reinterpret_cast<const uint4*>(vg + (pr * s.Hv + hv) * D + r0 + (c - kKP) * kVec);
      }
    }
    if (tid < n) s_gate[tid] = load_gates(L, s, ((size_t)b * s.Ns + s_phys[t0 + tid]) * s.Hv + hv, hv);
  };
  const bool go = st == LUMO_SEQ_OK && len > 0;
  if (go) stage(0, len < kCommitChunk ? len : kCommitChunk);
  // the copy is on its way whatever the path turned out to be: nobody leaves before it has landed
  if (lcap > 0 && !mbar_wait0(&mbar)) st = LUMO_SEQ_TIMEOUT;
  if (lead && L.status) { pdl_wait(); L.status[b] = st; }
  if (!go || st != LUMO_SEQ_OK) { pdl_wait(); return; }
  __syncthreads();
  const int j = tid & 3;
  // chunk by chunk (one chunk for all but the deepest trees), the state back to shared memory in between
  for (int t0 = 0; t0 < len; t0 += kCommitChunk) {                         // bounded: lmax / kCommitChunk
    const int n = len - t0 < kCommitChunk ? len - t0 : kCommitChunk;
    if (t0 > 0) {
      __syncthreads();                                                     // the last chunk's operands have been read
      stage(t0, n);
      __syncthreads();
    }
    const bool last = t0 + n == len;
#pragma unroll 1
    for (int ps = 0; ps < Cfg::kPasses; ++ps) {
      const int rl = ps * (kThreads / 4) + (tid >> 2);
      float* Sr = Ss + rl * D + 4 * j;
      float4 S[NCH];
#pragma unroll
      for (int m = 0; m < NCH; ++m) S[m] = *reinterpret_cast<const float4*>(Sr + 16 * m);
#pragma unroll 1
      for (int tt = 0; tt < n; ++tt)
        commit_token<D, T>(S, Ks + tt * D, Vs[tt * ROWS + rl], s_gate[tt], s.l2norm, s.l2_eps, j);
      if (last) {
        pdl_wait();
        float* Gr = Sg + (size_t)rl * D + 4 * j;
#pragma unroll
        for (int m = 0; m < NCH; ++m) *reinterpret_cast<float4*>(Gr + 16 * m) = S[m];
      } else {
#pragma unroll
        for (int m = 0; m < NCH; ++m) *reinterpret_cast<float4*>(Sr + 16 * m) = S[m];
      }
    }
  }
}

// device helper: root-first path ending at node[b]
__global__ void path_from_node_kernel(TreeDev t, int B, int N, const int32_t* __restrict__ node,
                                      int lmax, int32_t* __restrict__ accepted,
                                      int32_t* __restrict__ len, int32_t* __restrict__ status) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  pdl_wait();
  pdl_trigger();
  if (b >= B) return;
  int32_t* acc = accepted + (size_t)b * lmax;
  for (int e = 0; e < lmax; ++e) acc[e] = -1;
  int n = node[b], st = LUMO_SEQ_OK, l = 0;
  if (n != -1) {
    if (n < 0 || n >= N) st = LUMO_SEQ_BAD_NODE;
    else {
      l = t.depth[(size_t)b * N + n];
      if (l > lmax) { st = LUMO_SEQ_BAD_LEN; l = 0; }
      else
        for (int e = l - 1; e >= 0 && n >= 0; --e) { acc[e] = n; n = t.parent[(size_t)b * N + n]; }  // bounded: depth
    }
  }
  len[b] = l;
  if (status) status[b] = st;
}

template <typename F>
cudaError_t dispatch(int d, int in_dtype, F f) {
  if (d == 128 && in_dtype == LUMO_BF16) return f(std::integral_constant<int, 128>{}, __nv_bfloat16{});
  if (d == 128 && in_dtype == LUMO_F32) return f(std::integral_constant<int, 128>{}, float{});
  if (d == 64 && in_dtype == LUMO_BF16) return f(std::integral_constant<int, 64>{}, __nv_bfloat16{});
  if (d == 64 && in_dtype == LUMO_F32) return f(std::integral_constant<int, 64>{}, float{});
  return cudaErrorInvalidValue;
}

}  // namespace

// ---------------------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------------------
// Entries per run: sixteen amortise the window set-up, fewer let a small launch reach more SMs.  Counted are groups of eight
// warps (a warp is one run of 128 channels), however conv_split deals them out to CTAs: a run length is taken when it gives
// every SM sixteen warps.  Convolution and scan together, us, at four / eight / sixteen entries (4096 channels): 4 sequences of
// 60 entries (32 groups of sixteen) 20.5 / 22.2 / 22.1, 12 of 60 30.0 / 28.7 / 30.2, 24 of 28 37.4 / 36.9 / 37.5, 48 of 28
// 59.4 / 60.1 / 57.5.
int conv_rows_per_cta(int C, int Ns, int seqs, int sms) {
  const int slabs = (C / 4 + 255) / 256;
  auto groups = [&](int run) { return (long long)slabs * ((Ns + run - 1) / run) * seqs; };
  if (groups(16) >= 2LL * sms) return 16;
  if (groups(8) >= 2LL * sms) return 8;
  return 4;
}

template <typename K>
static cudaError_t allow_smem_once(K kern, int bytes, bool (&done)[kMaxDevices]) {      // a per-device setting
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  if (done[dev]) return cudaSuccess;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done[dev] = true;
  return e;
}

template <typename T>
static cudaError_t launch_conv_t(const Shape& s, const TreeDev& t, const LayerBatch& lb, const FusedPrev* fp, int sms,
                                 bool pdl, cudaStream_t st) {
  const int seqs = s.B * s.n_layers;
  const int rows = conv_rows_per_cta(s.C, s.Ns, seqs, sms);
  auto go = [&](auto rows_c, auto few_c) {
    constexpr int R = decltype(rows_c)::value;
    constexpr bool kFew = decltype(few_c)::value;
    using LB = std::conditional_t<kFew, FewLayers, LayerBatch>;
    constexpr int kMost = (kConvMaxEntries + 3 * kConvWarps) * 128 * (int)sizeof(T);    // of any split
    const ConvSplit sp = conv_split(s.C, s.Ns, R, seqs, sms);
    const int entries = sp.runs * R;
    const int parts = (s.Ns + entries - 1) / entries;
    const dim3 grid(sp.slabs * parts, s.B, s.n_layers), block(32 * sp.runs * sp.groups);
    const size_t smem = (size_t)(entries + (parts > 1 ? 6 : 3)) * sp.groups * 128 * sizeof(T);   // (several parts: one group)
    auto layers = [&]() -> decltype(auto) { if constexpr (kFew) return few_layers(lb); else return (lb); };
    if constexpr (sizeof(T) == 2) {                               // the fused path serves bf16 operands only
      if (fp) {
        static bool done[kMaxDevices] = {};
        const cudaError_t e = allow_smem_once(conv_fused_kernel<T, R, LB>, kMost, done);
        if (e != cudaSuccess) return e;
        auto prev = [&]() -> decltype(auto) { if constexpr (kFew) return few_layers(*fp); else return (*fp); };
        return launch_kernel(conv_fused_kernel<T, R, LB>, grid, block, smem, st, pdl, s, t, layers(), sp, prev());
      }
    }
    static bool done[kMaxDevices] = {};
    const cudaError_t e = allow_smem_once(conv_kernel<T, R, LB>, kMost, done);
    if (e != cudaSuccess) return e;
    return launch_kernel(conv_kernel<T, R, LB>, grid, block, smem, st, pdl, s, t, layers(), sp);
  };
  auto pick = [&](auto rows_c) { return s.n_layers <= kFewLayers ? go(rows_c, std::true_type{}) : go(rows_c, std::false_type{}); };
  if (rows == 16) return pick(std::integral_constant<int, 16>{});
  if (rows == 8) return pick(std::integral_constant<int, 8>{});
  return pick(std::integral_constant<int, 4>{});
}

cudaError_t launch_conv(const Shape& s, const TreeDev& t, const LayerBatch& lb, int sm_count, bool pdl, cudaStream_t st) {
  if (s.in_dtype == LUMO_BF16) return launch_conv_t<__nv_bfloat16>(s, t, lb, nullptr, sm_count, pdl, st);
  return launch_conv_t<float>(s, t, lb, nullptr, sm_count, pdl, st);
}

cudaError_t launch_conv_fused(const Shape& s, const TreeDev& t, const LayerBatch& lb, const FusedPrev& fp, int sm_count,
                              bool pdl, cudaStream_t st) {
  if (s.in_dtype != LUMO_BF16) return cudaErrorInvalidValue;
  return launch_conv_t<__nv_bfloat16>(s, t, lb, &fp, sm_count, pdl, st);
}

// Trees whose operands fit in shared memory take the staged kernel.
bool scan_staged(const Shape& s, const TreeDev& t) {
  return s.N <= kStagedThreads &&
         staged_smem(s.N, s.d, t.max_ops, s.snapshot_mode == 1 ? s.n_snap : 0, t.max_levels).total <= kStagedSmem;
}

// CTAs of `kern` that an SM holds at `smem` bytes; raises the kernel's shared-memory limit when it has to.  The answer for
// the size last asked for is kept per kernel instance and device: the two calls cost more host time than the launch itself.
struct Occupancy {
  std::atomic<uint64_t> known[kMaxDevices] = {};      // smem << 8 | CTAs
  std::mutex mu;
  int limit[kMaxDevices] = {};                        // only grows, so that a launch prepared for another size still fits
  cudaError_t per_sm(const void* kern, int threads, int smem, int* ctas) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    const uint64_t seen = known[dev].load(std::memory_order_relaxed);
    *ctas = (int)(seen & 0xFF);
    if (seen >> 8 == (uint64_t)smem && *ctas > 0) return cudaSuccess;
    {
      std::lock_guard<std::mutex> lock(mu);
      if (smem > limit[dev]) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        limit[dev] = smem;
      }
    }
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas, kern, threads, smem);
    if (e != cudaSuccess) return e;
    if (*ctas < 1) *ctas = 1;
    known[dev].store((uint64_t)smem << 8 | (uint64_t)*ctas, std::memory_order_relaxed);
    return cudaSuccess;
  }
};

cudaError_t scan_plan(const Shape& s, const TreeDev& t, int sm_count, int* grid, size_t* stack_bytes) {
  return dispatch(s.d, s.in_dtype, [&](auto dc, auto tc) {
    constexpr int D = decltype(dc)::value;
    using T = decltype(tc);
    const int n_snap_list = s.snapshot_mode == 1 ? s.n_snap : 0;
    const bool few = s.n_layers <= kFewLayers, staged = scan_staged(s, t);
    static Occupancy occ[2][2];
    int per_sm = 0, smem, rows;
    cudaError_t e;
    if (staged) {
      rows = kStagedRows;
      smem = staged_smem(s.N, D, t.max_ops, n_snap_list, t.max_levels).total;
      e = occ[1][few].per_sm(few ? (const void*)scan_staged_kernel<D, T, FewLayers> : (const void*)scan_staged_kernel<D, T, LayerBatch>,
                             kStagedThreads, smem, &per_sm);
    } else {
      rows = kRows;
      smem = scan_smem(s.N, t.max_ops, n_snap_list, ScanCfg<D, T>::kStageBytes).total;
      e = occ[0][few].per_sm(few ? (const void*)scan_kernel<D, T, FewLayers> : (const void*)scan_kernel<D, T, LayerBatch>, kScanThreads,
                             smem, &per_sm);
    }
    if (e != cudaSuccess) return e;
    const int items = s.n_layers * s.B * s.Hv * (D / rows), resident = sm_count * per_sm;
    *grid = items < resident ? items : resident;
    // with every state exported the staged kernel needs no stack
    *stack_bytes = staged && s.snapshot_mode == 2 ? 0 : (size_t)*grid * t.max_levels * rows * D * sizeof(float);
    return cudaSuccess;
  });
}

// ---------------------------------------------------------------------------------------
// fixed scratch for callers that cannot allocate (lumo_gdn_tree_scan_static)
// ---------------------------------------------------------------------------------------
// The scan's state stack normally lives in memory the context allocates on first use.  This
// array is the same stack with a fixed capacity, part of the library image on every GPU that
// loads it.  Host code must not pass `g_static_stack` itself to a kernel: on the host the name
// is only a handle for the symbol, so its device address is looked up once per device.
__device__ __align__(256) static float g_static_stack[kStaticStackBytes / sizeof(float)];

cudaError_t static_stack_address(int device, float** ptr) {
  static float* cached[kMaxDevices] = {};
  static std::mutex mu;
  if (device < 0 || device >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (!cached[device]) {
    int cur = -1;
    cudaError_t e = cudaGetDevice(&cur);
    if (e != cudaSuccess) return e;
    if (cur != device) return cudaErrorInvalidDevice;   // the caller makes `device` current first
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_static_stack);
    if (e != cudaSuccess) return e;
    cached[device] = static_cast<float*>(p);
  }
  *ptr = cached[device];
  return cudaSuccess;
}

cudaError_t launch_scan(const Shape& s, const TreeDev& t, const LayerBatch& lb, float* stack,
                        int grid, int sm_count, bool pdl, cudaStream_t st) {
  return dispatch(s.d, s.in_dtype, [&](auto dc, auto tc) {
    constexpr int D = decltype(dc)::value;
    using T = decltype(tc);
    const int n_snap_list = s.snapshot_mode == 1 ? s.n_snap : 0;
    const bool few = s.n_layers <= kFewLayers;
    if (scan_staged(s, t)) {
      const int items = s.n_layers * s.B * s.Hv * (D / kStagedRows);
      // Entering early, the CTAs crowd onto the SMs that the convolution leaves first.  That costs nothing while there is one
      // for each SM at most (seven-node step: 11.0 -> 8.3 us), and more than the launch it hides beyond (2 x 2 layers of
      // 27 nodes with cached states, 256 CTAs: convolution 9 us and scan 52 us alone, 72 us together).
      pdl = pdl && items <= sm_count;
      const StagedSmem lay = staged_smem(s.N, D, t.max_ops, n_snap_list, t.max_levels);
      if (few)
        return launch_kernel(scan_staged_kernel<D, T, FewLayers>, dim3(grid), dim3(kStagedThreads), lay.total, st, pdl, s, t, few_layers(lb), stack, items);
      return launch_kernel(scan_staged_kernel<D, T, LayerBatch>, dim3(grid), dim3(kStagedThreads), lay.total, st, pdl, s, t, lb, stack, items);
    }
    const int items = s.n_layers * s.B * s.Hv * (D / kRows);
    const ScanSmem lay = scan_smem(s.N, t.max_ops, n_snap_list, ScanCfg<D, T>::kStageBytes);
    if (few)
      return launch_kernel(scan_kernel<D, T, FewLayers>, dim3(grid), dim3(kScanThreads), lay.total, st, false, s, t, few_layers(lb), stack, items);
    return launch_kernel(scan_kernel<D, T, LayerBatch>, dim3(grid), dim3(kScanThreads), lay.total, st, false, s, t, lb, stack, items);
  });
}

cudaError_t launch_commit(const Shape& s, const TreeDev& t, const LayerBatch& lb, const int32_t* accepted,
                          const int32_t* len, int lmax, bool with_state, bool with_hist, int sm_count, bool pdl,
                          cudaStream_t st) {
  if (!with_state && !with_hist) return cudaSuccess;
  return dispatch(s.d, s.in_dtype, [&](auto dc, auto tc) {
    constexpr int D = decltype(dc)::value;
    using T = decltype(tc);
    auto go = [&](auto rows_c, auto few_c) {
      constexpr int R = decltype(rows_c)::value;
      using LB = std::conditional_t<decltype(few_c)::value, FewLayers, LayerBatch>;
      using Cfg = CommitCfg<D, T, R>;
      auto kern = commit_kernel<D, T, R, LB>;
      static bool configured[kMaxDevices] = {};            // the shared-memory limit is a per-device setting
      int dev = 0;
      cudaError_t e = cudaGetDevice(&dev);
      if (e != cudaSuccess) return e;
      if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
      if (!configured[dev]) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::kBytes);
        if (e != cudaSuccess) return e;
        configured[dev] = true;
      }
      const int n_state = with_state ? s.Hv * (D / R) : 0;
      const int per_cta = 16 / (int)sizeof(T) * Cfg::kThreads;
      const int n_hist = with_hist ? (s.C + per_cta - 1) / per_cta : 0;
      const dim3 grid(n_state + n_hist, s.B, s.n_layers);
      if constexpr (decltype(few_c)::value)
        return launch_kernel(kern, grid, dim3(Cfg::kThreads), Cfg::kBytes, st, pdl, s, t, few_layers(lb), accepted, len, lmax, n_state);
      else
        return launch_kernel(kern, grid, dim3(Cfg::kThreads), Cfg::kBytes, st, pdl, s, t, lb, accepted, len, lmax, n_state);
    };
    // up to one wave of 32-row CTAs (seven per SM): the shortest chain per CTA; beyond that whole heads, three CTAs per SM
    const long long tiles = (long long)s.n_layers * s.B * s.Hv * (D / 32);
    auto rows = [&](auto rows_c) {
      return s.n_layers <= kFewLayers ? go(rows_c, std::true_type{}) : go(rows_c, std::false_type{});
    };
    return tiles <= 7LL * sm_count ? rows(std::integral_constant<int, 32>{}) : rows(std::integral_constant<int, D>{});
  });
}

cudaError_t launch_path_from_node(const TreeDev& t, int B, int N, const int32_t* node, int lmax,
                                  int32_t* accepted, int32_t* len, int32_t* status, bool pdl, cudaStream_t st) {
  return launch_kernel(path_from_node_kernel, dim3((B + 63) / 64), dim3(64), 0, st, pdl, t, B, N, node, lmax, accepted, len, status);
}

}  // namespace lumo
