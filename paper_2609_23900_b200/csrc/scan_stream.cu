// Tree scan in the solved Gram form on tcgen05, the state streamed through shared memory.
//
// The algebra is the solved Gram form (paper Eq. 2-3, exact; see scan_gram.cu for the symbols):
//
//   A[t,s] = beta_t G(t,s) (k^_s . k^_t),  W[t,s] = G(t,s) (k^_s . q^_t),  M = W (I + A)^-1     along each root path
//   q~_t   = g_t |q scale| q_t - sum_s M[t,s] (beta_s g_s |k scale|) k_s
//   o_t    = S0 q~_t + sum_s M[t,s] beta_s v_s
//
// A, W, M and q~ need keys, queries and gates alone, so they are worked out while the state is on its way, and what is
// left once it has arrived is one conversion to bf16 hi + lo, one product and the read-out.  A persistent CTA goes from
// one (layer, sequence, value head) to the next:
//
//   * the state (64 KB, contiguous) is one bulk copy into shared memory, converted from there to bf16 hi + lo in tensor
//     memory, where it is an operand of the product; its buffer is free again at once, so the next head's state is on its
//     way while this one's groups are worked out.  Key and query rows of the next group are requested as soon as q~ has
//     been formed, its value rows behind the product.
//   * trees of more than 32 nodes are walked in groups of at most 32 (closed under "parent of") with the state kept in
//     tensor memory: it is read and converted once, whatever the size of the tree.
//   * a group takes three products with what they need in between spread over the CTA, eight lanes a node for A, W, M:
//       Gram = [K ; Q] [K ; Q]^T                                    (64 x 64, exact products of bf16 inputs)
//       Q~^T = K^T Mc^T + |q scale| g Q^T    Mc = -M diag(beta g |k scale|) as bf16 hi + lo, the query term in fp32
//       O^T  = S0 Q~ + V^T (M diag(beta))^T  S0 and q~ as hi + lo (three products), M diag(beta) as hi + lo
//     K and V enter as operands just as they lie in memory (MN-major).
//   * kFused: the accepted path of the previous cycle is replayed into the state rows between their arrival and their
//     conversion, with the arithmetic of the commit, and the rows are written back in place.
//
// Bounds it: 48 layers of 4 x 32 nodes, 172.7 us in one-item-at-a-time CTAs, now 122 (504 MB, 0.64 of the copy rate); 32 x 256
// nodes 212 -> 158; 28 nodes, 32 items 7.6 -> 5.5.  A group takes about 8 thousand cycles, two in flight per SM, none of its phases above
// 900; shared memory (operands of the products, look-ups) is the busiest unit.  Two CTAs because of the 64 KB a state lands in.
// Eight computing warps and 32-node groups: 64-node groups would leave one CTA per SM.
//
// The dense products run over all nodes of a group with zero coefficients off the path, so a key or value that is not
// finite is zeroed in its tile and its node marked; the outputs of exactly the nodes with a marked node on their path
// are then NaN.  Non-finite queries and gates reach only the coefficient rows of the node and its descendants.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "internal.h"

namespace lumo {

namespace {

constexpr int kD = 128;
constexpr int kNT = 32;               // nodes of a group at most
constexpr int kWarps = 8;             // that compute, and one more that leads them (below)
constexpr int kThreads = 32 * kWarps;
constexpr uint32_t kStateBytes = kD * kD * 4;

// shared memory map (bytes from a 1024-aligned base)
constexpr int kOffS = 0;                        // state as it lies in memory: [128][128] fp32
constexpr int kOffKQ = 65536;                   // rows 0..31 = K, 32..63 = Q, 2 k-blocks x [64 rows x 128 B], SW128
constexpr int kKQBlock = 8192;
constexpr int kOffQt = kOffKQ + 2 * kKQBlock;   // q~: hi, then lo: [128 columns][32 nodes], 64 B rows, SW64 (MN-major operands)
constexpr int kOffV = kOffQt + 16384;           // V rows, 2 halves of 64 value columns x [32 rows x 128 B], SW128 (MN-major operand)
constexpr int kVBlock = 4096;
constexpr int kOffMb = kOffV + 2 * kVBlock;     // M diag(beta): [32 nodes][32 nodes hi | 32 nodes lo], SW128
constexpr int kOffSmall = kOffMb + 4096;
// before q~ is formed its area holds the scalar part, after the product the outputs on their way out
constexpr int kDumpStride = 33;
constexpr int kOffDump = kOffQt;                // Gram rows [64][33] fp32
constexpr int kAStride = 20;                    // floats per row of A: rows of neighbouring lanes fall into different banks
constexpr int kOffA = kOffDump + 64 * kDumpStride * 4;
constexpr int kOffMc = kOffQt + 12288;          // Mc: [32 nodes][32 nodes hi | 32 nodes lo], SW128
static_assert(kOffA + kNT * kAStride * 4 <= kOffMc, "scalar tables overflow the effective queries' area");
// fused: the accepted path's recorded rows, over the Gram rows once the coefficients have been read from them
constexpr int kOffPrevK = kOffDump, kOffPrevV = kOffDump + kFusedMaxPath * kD * 2;
static_assert(kOffPrevV + kFusedMaxPath * kD * 2 <= kOffA, "recorded rows overflow the Gram rows");

// One (layer, sequence, part of its groups, value head): what is done with one state.
struct Unit {
  int hv, bp, layer;       // value head, sequence << log_parts | part, layer
  int b, row, gi, gend;    // sequence, state row, next group, end of the part's groups
  bool lead;               // the part begins with the sequence's first group (a part may be empty)
};
// One group of a unit, as the CTA needs it: operand rows from the sequence's first physical row on, of the unit's head.
struct Step {
  const unsigned char *k, *q, *v, *out;
  int layer, b, hv, gi;
  int row;
  bool have, fresh, lead;  // there is such a step; the state has to be fetched; first group of the sequence
};
struct Small {
  float4 node[2][kNT];               // alpha, beta, |k scale|, |q scale| of each node; the steps take turns
  float ck[kNT], cq[kNT];            // beta_t g_t |k scale|, g_t |q scale|
  uint32_t bad[2];                   // nodes whose key or value row is not finite; the steps take turns
  uint32_t look[2];                  // set when some |k|^2 is not finite: the key rows are to be looked over
  uint32_t timed_out;
  uint32_t state_missing;            // the wait for a state ran out (kept by the computing warps): its copy may still be on its way
  uint32_t tmem_base;
  unsigned long long mb_state, mb_mma;
  // kept by the leading warp
  Step step[4];                      // step k lies at k mod 4; two steps beyond the one at hand are known
  Unit unit;                         // of the last step looked at
  bool unit_fresh;
  int by_hv, by_bp, by_layer;        // the grid, in heads, sequence parts and layers
  // fused: the accepted path of the sequence at hand
  int plen;                          // accepted nodes to replay (0 when the path is empty or refused)
  int phys[kFusedMaxPath];
  float prev_ks[kFusedMaxPath];      // key normalisation factors
  float2 gates[kFusedMaxPath];       // alpha, beta
};
constexpr int kSmemBytes = kOffSmall + (int)sizeof(Small) + 1024;   // + alignment slack
static_assert(2 * (kSmemBytes + 1024) <= 228 * 1024, "two CTAs must share an SM");
// tensor memory columns
constexpr uint32_t kColS = 0, kColO = 128, kColGram = 192, kColQt = 192;   // state: 64 columns hi, 64 lo
constexpr int kTmemCols = 256;

// roles and exceptions: their code lies out of line, so that the common path is not broken by jumps across it
__device__ __forceinline__ bool rarely(bool b) { return __builtin_expect(b, 0); }
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// 16 bytes, or zeros where `live` is false
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* gmem, bool live) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(gmem), "r"(live ? 16u : 0u) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_but_one() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void mbar_init(unsigned long long* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
// Bounded wait: false if the phase did not complete within the spin limit.
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, uint32_t parity, uint32_t limit) {
  const uint32_t addr = smem_u32(bar);
  for (uint32_t spin = 0; spin < limit; ++spin) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done) : "r"(addr), "r"(parity) : "memory");
    if (done) return true;
  }
  return false;
}
// one thread: the state of one head, counted on `bar`
__device__ __forceinline__ void request_state(uint32_t dst, const float* src, unsigned long long* bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(kStateBytes) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
               ::"r"(dst), "l"(src), "r"(kStateBytes), "r"(smem_u32(bar)) : "memory");
}

// Shared-memory operand descriptor, 128-byte swizzle (kSw 2) or 64-byte swizzle (4), version 1 (sm_100).  K-major: rows of
// 128 B, eight-row groups `sbo` bytes apart, `lbo` unused.  MN-major (the contraction index runs over the rows): 64 (32)
// elements of the M or N dimension per row of 128 (64) bytes, eight-row groups of the contraction index `sbo` bytes apart,
// the next 64 (32) elements `lbo` bytes on.
template <int kSw = 2>
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)(lbo >> 4) << 16;
  d |= (uint64_t)(sbo >> 4) << 32;
  d |= (uint64_t)1 << 46;                           // descriptor version
  d |= (uint64_t)kSw << 61;                         // SWIZZLE_128B or SWIZZLE_64B
  return d;
}
// kind::f16, bf16 x bf16 -> fp32, M = 128; a_mn / b_mn: that operand is MN-major
__host__ __device__ constexpr uint32_t umma_idesc(int N, int a_mn, int b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) | ((uint32_t)(N >> 3) << 17) | ((128u >> 4) << 24);
}
// Products are issued by one lane of a warp that stays together (`lead`: this is the lane): operands and descriptors then live
// in uniform registers.  Issued from a branch of one thread, every operand was moved there first, some 60 cycles a product.
__device__ __forceinline__ void umma(uint32_t lead, uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.b32 p, %4, 0;\nsetp.ne.b32 q, %5, 0;\n"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(lead) : "memory");
}
// the same with A in tensor memory: lane = row, a 32-bit column holds two consecutive elements of the contraction
__device__ __forceinline__ void umma_ta(uint32_t lead, uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.b32 p, %4, 0;\nsetp.ne.b32 q, %5, 0;\n"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate), "r"(lead) : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t lead, unsigned long long* bar) {
  asm volatile("{\n.reg .pred q;\nsetp.ne.b32 q, %1, 0;\n@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n"
               ::"r"(smem_u32(bar)), "r"(lead) : "memory");
}
// 1 in one lane of a warp whose lanes are all here
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t one;
  asm volatile("{\n.reg .pred q;\nelect.sync _|q, 0xFFFFFFFF;\nselp.u32 %0, 1, 0, q;\n}\n" : "=r"(one));
  return one;
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
// 16 lanes x 32 columns: registers 4 n .. 4 n + 3 of lane l are columns 8 n + 2 (l & 3), + 1 of lane l / 4, then of lane 8 + l / 4
__device__ __forceinline__ void tmem_st_16x256b_x4(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory"); }

__device__ __forceinline__ uint32_t sw128_offset(int row, int chunk16) {   // within one [rows x 128 B] block
  return (uint32_t)(row * 128 + ((chunk16 ^ (row & 7)) << 4));
}
__device__ __forceinline__ uint32_t pack_bf16(float2 v) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ float2 unpack_bf16(uint32_t w) { return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u)); }
// fp32 pair -> bf16 hi and lo words (x - hi is exact)
__device__ __forceinline__ void split2(float2 x, uint32_t& hi, uint32_t& lo) {
  hi = pack_bf16(x);
  lo = pack_bf16(__ffma2_rn(make_float2(-1.f, -1.f), unpack_bf16(hi), x));
}
// whether any of the bf16 values in two 16-byte pieces is not finite: zero times it is NaN, and stays in the sum
__device__ __forceinline__ bool any_not_finite(uint4 a, uint4 b) {
  const uint32_t ws[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  const __nv_bfloat162 zero = __floats2bfloat162_rn(0.f, 0.f);
  __nv_bfloat162 sum[2] = {zero, zero};
#pragma unroll
  for (int e = 0; e < 8; ++e) sum[e & 1] = __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&ws[e]), zero, sum[e & 1]);
  const uint32_t nan = *reinterpret_cast<const uint32_t*>(&sum[0]) | *reinterpret_cast<const uint32_t*>(&sum[1]);
  return (nan & 0x7F807F80u) != 0u;
}
// values of a 16-byte piece that are not finite become zero; true if there were any
__device__ __noinline__ bool drop_non_finite(uint4* piece) {
  const uint4 w = *piece;
  uint32_t ws[4] = {w.x, w.y, w.z, w.w};
  bool any = false;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    if ((ws[e] & 0x7F80u) == 0x7F80u) { ws[e] &= 0xFFFF0000u; any = true; }
    if ((ws[e] & 0x7F800000u) == 0x7F800000u) { ws[e] &= 0x0000FFFFu; any = true; }
  }
  *piece = make_uint4(ws[0], ws[1], ws[2], ws[3]);
  return any;
}

// kDrill: a test aid; nothing asynchronous is issued to the tensor core or the state's barrier, and every wait runs out.
template <bool kFused, bool kDrill, class LB>
__device__ __forceinline__ void scan_stream_body(const Shape& s, const TreeDev& t, const LB& lb, int log_parts, const FusedPrevT<LB>* fp) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t sbase = smem_u32(smem);
  Small& sm = *reinterpret_cast<Small*>(smem + kOffSmall);
  float* dump = reinterpret_cast<float*>(smem + kOffDump);
  float* At = reinterpret_cast<float*>(smem + kOffA);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int trow = 32 * (warp & 3) + lane;                      // tensor-memory lane of this thread
  const int t0 = (warp >> 2) * 16;                              // its half of the nodes
  const int r16 = tid >> 4, c16 = tid & 15;                     // operand rows r16 and r16 + 16, 16-byte piece c16 of them
  const uint32_t kq_dst = kOffKQ + (c16 >> 3) * kKQBlock + sw128_offset(r16, c16 & 7);   // row + 16: + 2048; queries: + 4096
  const uint32_t v_dst = kOffV + (c16 >> 3) * kVBlock + sw128_offset(r16, c16 & 7);
  const int sn = tid >> 3, s8 = tid & 7;                        // scalar part: node, and which two entries of its path
  const bool leads = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0) == kWarps;      // the ninth warp
  const int rep = s.Hv / s.Hk;
  const uint32_t rep_mul = 0xFFFFFFFFu / (uint32_t)rep + 1u;    // hv / rep = high word of hv * rep_mul (rep > 1)
  const int out_size = s.out_dtype == LUMO_BF16 ? 2 : 4;
  const uint32_t k_pitch = (uint32_t)s.Hk * kD, v_pitch = (uint32_t)s.Hv * kD;   // elements from one physical row to the next
  constexpr uint32_t spin_limit = kDrill ? 1024 : 1u << 24;
  auto live = [](int meta) { return ((meta >> 16) & 0xFF) != 0; };               // a node, not the rest of the group's table

  // ---- the leading warp looks ahead ------------------------------------------------------------------------------------
  auto advance = [&](Unit& u) {                                 // by the grid
    const int n_bp = s.B << log_parts;
    u.hv += sm.by_hv; u.bp += sm.by_bp; u.layer += sm.by_layer;
    if (u.hv >= s.Hv) { u.hv -= s.Hv; ++u.bp; }
    if (u.bp >= n_bp) { u.bp -= n_bp; ++u.layer; }
  };
  // completes `u` (head, bp and layer given), going on to later units where there is nothing to do; false at the end
  auto open = [&](Unit& u) -> bool {
    while (u.layer < s.n_layers) {                              // bounded: the launch's units
      const LayerPtrs& L = lb.l[u.layer];
      const int part = u.bp & ((1 << log_parts) - 1);
      u.b = u.bp >> log_parts;
      u.row = L.state_row[u.b];
      int first = u.b, last = u.b + 1;
      if (t.st_groups != s.B) { first = t.st_off[u.b]; last = t.st_off[u.b + 1]; }
      u.gi = first + ((part * (last - first)) >> log_parts);
      u.gend = first + (((part + 1) * (last - first)) >> log_parts);
      u.lead = u.gi == first;
      const bool row_ok = u.row >= 0 && u.row < s.n_state_rows;
      if (row_ok && u.gi < u.gend) return true;
      if (!row_ok && part == 0) {                               // skipped sequence: zero outputs
        pdl_wait();
        unsigned char* out = reinterpret_cast<unsigned char*>(L.out) + (((size_t)u.b * s.Ns) * s.Hv + u.hv) * kD * out_size;
        for (int ps = lane >> 3; ps < s.Ns; ps += 4)
          for (int c = (lane & 7) * 16; c < kD * out_size; c += 128) *reinterpret_cast<uint4*>(out + (size_t)ps * v_pitch * out_size + c) = make_uint4(0, 0, 0, 0);
        if (L.status && u.hv == 0 && lane == 0) L.status[u.b] = u.row < 0 ? LUMO_SEQ_OK : LUMO_SEQ_BAD_ROW;
        if constexpr (kFused) {
          int32_t* pst = fp->lb.l[u.layer].status;
          if (pst && u.hv == 0 && lane == 0) pst[u.b] = u.row < 0 ? LUMO_SEQ_OK : LUMO_SEQ_BAD_ROW;
        }
      }
      advance(u);
    }
    return false;
  };
  auto state_of = [&](int layer, int row, int hv) { return lb.l[layer].state + ((size_t)row * s.Hv + hv) * kD * kD; };
  // the step after the last one written, in two parts: which it is, and where its rows lie (a lane per pointer)
  auto look_ahead = [&]() {
    Unit u = sm.unit;
    const bool last = u.layer >= s.n_layers;
    __syncwarp();
    bool fresh = false;
    if (++u.gi >= u.gend && !last) {
      fresh = true;
      advance(u);
      open(u);
    }
    if (lane == 0) { sm.unit = u; sm.unit_fresh = fresh; }
    __syncwarp();
  };
  auto write_step = [&](Step& st) {
    const Unit u = sm.unit;
    const bool have = u.layer < s.n_layers;
    if (lane == 4) {
      st.have = have;
      st.layer = u.layer; st.b = u.b; st.hv = u.hv; st.gi = u.gi; st.row = u.row;
      st.fresh = sm.unit_fresh;
      st.lead = sm.unit_fresh && u.lead;
    }
    if (lane < 4 && have) {
      const LayerPtrs& L = lb.l[u.layer];
      const bool key = lane < 2;
      const unsigned char* base = reinterpret_cast<const unsigned char*>(lane == 0 ? L.k : lane == 1 ? L.q : lane == 2 ? L.v : L.out);
      const int heads = key ? s.Hk : s.Hv, head = key && rep > 1 ? (int)__umulhi((uint32_t)u.hv, rep_mul) : u.hv;
      (&st.k)[lane] = base + (((size_t)u.b * s.Ns) * heads + head) * (kD * (lane == 3 ? out_size : 2));
    }
    __syncwarp();
  };

  // ---- operand rows of a step: this thread's pieces (m0, m1: table words of nodes r16 and r16 + 16) ------------------
  auto request_kq = [&](const Step& st, int m0, int m1) {
    const uint32_t o0 = (uint32_t)(m0 & 0xFFFF) * k_pitch + c16 * 8, o1 = (uint32_t)(m1 & 0xFFFF) * k_pitch + c16 * 8;
    const __nv_bfloat16 *kg = reinterpret_cast<const __nv_bfloat16*>(st.k), *qg = reinterpret_cast<const __nv_bfloat16*>(st.q);
    cp_async16(sbase + kq_dst, kg + o0, live(m0));
    cp_async16(sbase + kq_dst + 4096, qg + o0, live(m0));
    cp_async16(sbase + kq_dst + 2048, kg + o1, live(m1));
    cp_async16(sbase + kq_dst + 4096 + 2048, qg + o1, live(m1));
    cp_async_commit();
  };
  auto request_v = [&](const Step& st, int m0, int m1) {
    const __nv_bfloat16* vg = reinterpret_cast<const __nv_bfloat16*>(st.v) + c16 * 8;
    cp_async16(sbase + v_dst, vg + (uint32_t)(m0 & 0xFFFF) * v_pitch, live(m0));
    cp_async16(sbase + v_dst + 2048, vg + (uint32_t)(m1 & 0xFFFF) * v_pitch, live(m1));
    cp_async_commit();
  };
  // this thread's pieces of rows r16 and r16 + 16 at `at` (have landed): values that are not finite are dropped and noted
  auto drop = [&](uint32_t at, uint32_t* bad) {
    if (drop_non_finite(reinterpret_cast<uint4*>(smem + at))) atomicOr(bad, 1u << r16);
    if (drop_non_finite(reinterpret_cast<uint4*>(smem + at + 2048))) atomicOr(bad, 1u << (r16 + 16));
  };
  // leading warp: gates of node `lane` as stored, and the head's parameters where they are raw
  uint2 gate_words = make_uint2(0, 0);
  float2 gate_par = make_float2(0.f, 0.f);
  bool gate_live = false;
  auto request_gates = [&](const Step& st) {
    const int m = t.st_meta[(size_t)st.gi * kNT + lane];
    const LayerPtrs& L = lb.l[st.layer];
    gate_live = live(m);
    if (gate_live) gate_words = load_gate_words(L, s, ((size_t)st.b * s.Ns + (m & 0xFFFF)) * s.Hv + st.hv);
    if (s.gate_mode == 1) gate_par = make_float2(L.a_log[st.hv], L.dt_bias[st.hv]);
  };
  auto store_gates = [&](float4* nodes) {
    float2 gates = make_float2(1.f, 0.f);
    if (gate_live) gates = finish_gates(gate_words, s, gate_par.x, gate_par.y);
    *reinterpret_cast<float2*>(&nodes[lane].x) = gates;
  };
  // fused, leading warp: the accepted path, a lane per entry, in three dependent steps
  int f_len = 0, f_acc = 0, f_par = -2, f_phys = 0;
  auto path_entries = [&](const Step& w) {
    f_len = fp->len[w.b];
    f_acc = lane < fp->lmax && lane < kFusedMaxPath ? fp->accepted[(size_t)w.b * fp->lmax + lane] : -1;
  };
  auto path_nodes = [&](const Step& w) {
    const bool ok = f_acc >= 0 && f_acc < fp->N;
    f_par = ok ? fp->parent[(size_t)w.b * fp->N + f_acc] : -2;
    f_phys = ok ? fp->slot[(size_t)w.b * fp->N + f_acc] : 0;
  };
  auto path_store = [&](const Step& w) {                        // same order of checks as check_path_staged
    int st = LUMO_SEQ_OK;
    const int before = __shfl_up_sync(0xffffffffu, f_acc, 1);
    if (f_len < 0 || f_len > fp->lmax) st = LUMO_SEQ_BAD_LEN;
    else {
      int mine = LUMO_SEQ_OK;
      if (lane < f_len) {
        if (f_acc < 0 || f_acc >= fp->N) mine = LUMO_SEQ_BAD_NODE;
        else if (lane == 0) mine = f_par != -1 ? LUMO_SEQ_BAD_ROOT : LUMO_SEQ_OK;
        else if (f_par != before) mine = LUMO_SEQ_BAD_LINK;
      }
      const uint32_t wrong = __ballot_sync(0xffffffffu, mine != LUMO_SEQ_OK);
      if (wrong) st = __shfl_sync(0xffffffffu, mine, __ffs(wrong) - 1);
    }
    if (lane < kFusedMaxPath) sm.phys[lane] = f_phys;
    if (lane == 0) {
      sm.plen = st == LUMO_SEQ_OK ? f_len : 0;
      int32_t* pst = fp->lb.l[w.layer].status;
      if (pst && w.hv == 0) pst[w.b] = st;
    }
  };

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&sm.tmem_base)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  if (tid == 0) {
    mbar_init(&sm.mb_state, 1);
    mbar_init(&sm.mb_mma, 1);
    sm.timed_out = sm.state_missing = 0; sm.bad[0] = sm.bad[1] = sm.look[0] = sm.look[1] = 0; sm.plen = 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem_base, tmem_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
  uint32_t ph_mma = 0, k = 0;
  // named barriers: 1 everyone (a product's operands are there, or its result), 2 the computing warps
  auto all = [] { asm volatile("bar.sync 1, %0;\n" ::"n"(kThreads + 32) : "memory"); };
  auto crew = [] { asm volatile("bar.sync 2, %0;\n" ::"n"(kThreads) : "memory"); };

  if (leads) {
    const int n_bp = s.B << log_parts;
    Unit u;
    {
      int h = (int)gridDim.x / s.Hv;
      if (lane == 0) { sm.by_hv = (int)gridDim.x - h * s.Hv; sm.by_bp = h % n_bp; sm.by_layer = h / n_bp; }
      h = (int)blockIdx.x / s.Hv;
      u.hv = (int)blockIdx.x - h * s.Hv; u.bp = h % n_bp; u.layer = h / n_bp;
    }
    __syncwarp();
    const bool any = open(u);
    uint32_t requested = 0;                                     // states asked for (first lane)
    if (lane == 0) {
      sm.unit = u;
      sm.unit_fresh = true;
      // the state is settled before this kernel may enter early; everything else may still be in the making
      if (any && !kDrill) {
        request_state(sbase + kOffS, state_of(u.layer, u.row, u.hv), &sm.mb_state);
        ++requested;
      }
    }
    __syncwarp();
    write_step(sm.step[0]);
    if constexpr (kFused) if (any) { path_entries(sm.step[0]); path_nodes(sm.step[0]); }
    look_ahead();
    write_step(sm.step[1]);
    __syncthreads();
    pdl_wait();
    // a fused launch rewrites the state, which a dependent may request ahead of its own wait: nobody in before it has finished
    if constexpr (!kFused) pdl_trigger();
    if (any) {
      request_gates(sm.step[0]);
      store_gates(sm.node[0]);
      if constexpr (kFused) path_store(sm.step[0]);
    }
    const uint32_t lead = kDrill ? 0u : elect_one();
    uint32_t landed = 0;                                        // states that the others have seen arrive
    for (; sm.step[k & 3].have; ++k) {                          // bounded: the launch's work
      const Step &cur = sm.step[k & 3], &nxt = sm.step[(k + 1) & 3];
      all();                                                    // key and query rows are there
      {
        tc_fence_after();
        const uint64_t d_kq = umma_desc(sbase + kOffKQ, 16, 1024);
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
          const uint64_t o = (uint64_t)(((ks >> 2) * kKQBlock + (ks & 3) * 32) >> 4);
          umma(lead, tmem + kColGram, d_kq + o, d_kq + o, umma_idesc(64, 0, 0), ks ? 1u : 0u);   // rows 64..127 of A: whatever lies behind
        }
        umma_commit(lead, &sm.mb_mma);
      }
      if (lane == 0) {
        sm.bad[(k & 1) ^ 1] = sm.look[(k & 1) ^ 1] = 0;
        int32_t* status = lb.l[cur.layer].status;
        if (cur.lead && cur.hv == 0 && status) status[cur.b] = LUMO_SEQ_OK;
      }
      if constexpr (kFused) {
        if (cur.fresh && lane < sm.plen) {
          const LayerPtrs& PL = fp->lb.l[cur.layer];
          sm.gates[lane] = load_gates(PL, s, ((size_t)cur.b * fp->Ns + sm.phys[lane]) * s.Hv + cur.hv, cur.hv);
        }
        if (nxt.have && nxt.fresh) path_entries(nxt);
      }
      look_ahead();
      write_step(sm.step[(k + 2) & 3]);
      ph_mma ^= 1;                                              // (the Gram rows are waited for by who reads them)
      all();                                                    // coefficient tiles and value rows are there
      {
        tc_fence_after();
        const uint64_t d_k = umma_desc(sbase + kOffKQ, kKQBlock, 1024), d_m = umma_desc(sbase + kOffMc, 16, 1024);
        const uint64_t d_v = umma_desc(sbase + kOffV, kVBlock, 1024), d_b = umma_desc(sbase + kOffMb, 16, 1024);
#pragma unroll
        for (int i = 0; i < 4; ++i)                             // contraction over 2 x 16 nodes, hi then lo
          umma(lead, tmem + kColQt, d_k + (uint64_t)(((i & 1) * 2048) >> 4), d_m + (uint64_t)((i * 32) >> 4), umma_idesc(32, 1, 0), i ? 1u : 0u);
        umma_commit(lead, &sm.mb_mma);
#pragma unroll
        for (int i = 0; i < 4; ++i)                             // V^T (M diag(beta))^T: the state's product is added to it
          umma(lead, tmem + kColO, d_v + (uint64_t)(((i & 1) * 2048) >> 4), d_b + (uint64_t)((i * 32) >> 4), umma_idesc(32, 1, 0), i ? 1u : 0u);
      }
      if constexpr (kFused) if (nxt.have && nxt.fresh) path_nodes(nxt);
      if (!mbar_wait(&sm.mb_mma, ph_mma, spin_limit)) sm.timed_out = 1;
      ph_mma ^= 1;
      all();                                                    // q~ is in tensor memory
      all();                                                    // q~ and the state are operands
      {
        tc_fence_after();
        const uint64_t d_q = umma_desc<4>(sbase + kOffQt, 16, 512);
#pragma unroll
        for (int i = 0; i < 24; ++i) {                          // hi q~hi, hi q~lo, lo q~hi: eight steps of 16 key columns each
          const int term = i >> 3, ks = i & 7;
          umma_ta(lead, tmem + kColO, tmem + kColS + (term == 2 ? 64 : 0) + 8 * ks, d_q + (uint64_t)(((term == 1 ? 8192 : 0) + ks * 1024) >> 4),
                  umma_idesc(32, 0, 1), 1u);
        }
        umma_commit(lead, &sm.mb_mma);
      }
      if (nxt.have) {
        if (nxt.fresh && lane == 0 && !kDrill && !sm.state_missing) {   // (one copy at a time on the barrier)
          request_state(sbase + kOffS, state_of(nxt.layer, nxt.row, nxt.hv), &sm.mb_state);
          ++requested;
        }
        request_gates(nxt);
      }
      if (!mbar_wait(&sm.mb_mma, ph_mma, spin_limit)) sm.timed_out = 1;
      ph_mma ^= 1;
      __syncwarp();
      all();                                                    // the outputs are in tensor memory
      if (cur.fresh && !sm.state_missing) ++landed;
      if (sm.timed_out) {                                       // the same in every thread: report this unit and all that are left
        auto give_up = [&](int layer, int b, bool replayed) {
          const int row = lb.l[layer].state_row[b];
          const int32_t st = row < 0 ? LUMO_SEQ_OK : row >= s.n_state_rows ? LUMO_SEQ_BAD_ROW : LUMO_SEQ_TIMEOUT;
          int32_t* status = lb.l[layer].status;
          if (status) status[b] = st;
          if constexpr (kFused) {
            int32_t* pst = fp->lb.l[layer].status;
            if (pst && !replayed) pst[b] = st;
          }
        };
        if (lane == 0) {
          give_up(cur.layer, cur.b, !(cur.fresh && sm.state_missing));
          if (nxt.have) give_up(nxt.layer, nxt.b, !nxt.fresh);
          Unit u = sm.unit;                                     // of the step after that
          while (u.layer < s.n_layers) {                        // bounded: the launch's units
            give_up(u.layer, u.bp >> log_parts, false);
            advance(u);
          }
        }
        break;
      }
      if (nxt.have) {
        store_gates(sm.node[(k & 1) ^ 1]);
        if constexpr (kFused) if (nxt.fresh) path_store(nxt);
      }
    }
    // nobody leaves before its own copies have landed
    if (lane == 0 && requested > landed) mbar_wait(&sm.mb_state, landed & 1, spin_limit);
  } else {
  __syncthreads();
  uint32_t ph_state = 0;
  int m0 = 0, m1 = 0;                                           // table words of nodes r16 and r16 + 16
  if (sm.step[0].have) {
    const int32_t* tab = t.st_meta + (size_t)sm.step[0].gi * kNT + r16;
    m0 = tab[0];
    m1 = tab[16];
  }
  pdl_wait();
  if constexpr (!kFused) pdl_trigger();
  if (sm.step[0].have) {
    request_kq(sm.step[0], m0, m1);
    request_v(sm.step[0], m0, m1);
  }

  for (; sm.step[k & 3].have; ++k) {                            // bounded: the launch's work
    const Step &cur = sm.step[k & 3], &nxt = sm.step[(k + 1) & 3];
    uint32_t* bad = &sm.bad[k & 1];
    float4* nodes = sm.node[k & 1];
    const bool fresh = cur.fresh;
    const int md = t.st_meta[(size_t)cur.gi * kNT + sn];        // node sn's table word and path (root first)
    const uint4 av = *reinterpret_cast<const uint4*>(t.st_anc + ((size_t)cur.gi * kNT + sn) * 16);
    // ---- operand rows have landed: look them over, hand them to the tensor core --------------------------------------
    cp_async_wait_but_one();                                    // (the value rows may still be on their way)
    fence_async_proxy();
    tc_fence_before();
    all();
    // ---- meanwhile: coefficient tiles cleared, rows without a node zeroed ---------------------------------------------
    *reinterpret_cast<uint4*>(smem + kOffMc + tid * 16) = make_uint4(0, 0, 0, 0);
    *reinterpret_cast<uint4*>(smem + kOffMb + tid * 16) = make_uint4(0, 0, 0, 0);
    if (rarely(cur.lead && s.Ns > s.N)) {
      for (int e = s.N + r16; e < s.Ns; e += 16) {              // padding rows, last in the convolution's visiting order
        const uint32_t ps = (uint32_t)t.conv_prog[(size_t)cur.b * s.Ns + e];
        for (int c = c16 * 16; c < kD * out_size; c += 256) *reinterpret_cast<uint4*>(const_cast<unsigned char*>(cur.out) + (size_t)ps * v_pitch * out_size + c) = make_uint4(0, 0, 0, 0);
      }
    }
    if constexpr (kFused) {
      if (fresh && sm.plen > 0) {
        if (fp->hist_in_kernels && warp == 2) {
          const LayerPtrs& PL = fp->lb.l[cur.layer];
          // The convolution before this kernel read the committed history through the path; now that it has finished, the
          // history itself is brought up to date: the value heads of a sequence share out the channels, a thread moves
          // 16 bytes of all three rows (reads before writes).
          const int chunks = s.C / 8, per_head = (chunks + s.Hv - 1) / s.Hv, plen = sm.plen;
          __nv_bfloat16* hist = reinterpret_cast<__nv_bfloat16*>(lb.l[cur.layer].conv_hist) + (size_t)cur.row * 3 * s.C;
          const __nv_bfloat16* xprev = reinterpret_cast<const __nv_bfloat16*>(PL.x) + (size_t)cur.b * fp->Ns * s.C;
          for (int c = cur.hv * per_head + lane; c < min(chunks, (cur.hv + 1) * per_head); c += 32) {   // bounded: per_head
            uint4 rows3[3];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
              const int q = plen + j;    // index into [old0 old1 old2 x_a0 x_a1 ...]
              const __nv_bfloat16* src = q < 3 ? hist + (size_t)q * s.C : xprev + (size_t)sm.phys[q - 3] * s.C;
              rows3[j] = *reinterpret_cast<const uint4*>(src + c * 8);
            }
#pragma unroll
            for (int j = 0; j < 3; ++j) *reinterpret_cast<uint4*>(hist + (size_t)j * s.C + c * 8) = rows3[j];
          }
        }
      }
    }
    int n0 = 0, n1 = 0;
    const bool n_have = nxt.have;
    if (n_have) {
      const int32_t* tab = t.st_meta + (size_t)nxt.gi * kNT + r16;
      n0 = tab[0];
      n1 = tab[16];
    }
    // ---- Gram rows out of tensor memory; normalisation factors ---------------------------------------------------------
    if ((warp & 3) < 2) {                                       // lanes 0..31 the key rows, 32..63 the query rows
      if (!mbar_wait(&sm.mb_mma, ph_mma, spin_limit)) sm.timed_out = 1;
      tc_fence_after();
      const bool is_q = warp & 1;
      uint32_t r[16];
      tmem_ld16(tmem_lane + kColGram + t0, r);
      tmem_ld_wait();
#pragma unroll
      for (int e = 0; e < 16; ++e) dump[trow * kDumpStride + t0 + e] = __uint_as_float(r[e]);
      if (is_q) {                                               // uniform over the warp: the queries' own columns
        tmem_ld16(tmem_lane + kColGram + kNT + t0, r);
        tmem_ld_wait();
      }
      if ((lane >> 4) == (warp >> 2)) {                         // |k|^2 and |q|^2: the diagonal
        uint32_t d8[8], d4[4], d2[2];
#pragma unroll
        for (int e = 0; e < 8; ++e) d8[e] = lane & 1 ? r[2 * e + 1] : r[2 * e];
#pragma unroll
        for (int e = 0; e < 4; ++e) d4[e] = lane & 2 ? d8[2 * e + 1] : d8[2 * e];
#pragma unroll
        for (int e = 0; e < 2; ++e) d2[e] = lane & 4 ? d4[2 * e + 1] : d4[2 * e];
        const float sq = __uint_as_float(lane & 8 ? d2[1] : d2[0]);
        const float inv = s.l2norm ? rsqrtf(sq + s.l2_eps) : 1.f;
        if (is_q) nodes[lane].w = s.scale * inv;
        else {
          nodes[lane].z = inv;
          if (rarely(!(sq <= 3.4028234e38f))) sm.look[k & 1] = 1;
        }
      }
    }
    ph_mma ^= 1;
    crew();
    // ---- A, W and M along each node's path, eight lanes per node (lane s8: path entries 2 s8, 2 s8 + 1) ----------------
    {
      const int D = (md >> 16) & 0xFF;                          // depth 1..16; 0: no node
      const int Dw = __reduce_max_sync(0xffffffffu, D);
      const uint32_t aw[4] = {av.x, av.y, av.z, av.w};
      const uint32_t half = s8 & 4 ? (s8 & 2 ? av.w : av.z) : (s8 & 2 ? av.y : av.x);
      const uint32_t own = s8 & 1 ? half >> 16 : half;
      const int a0 = own & 0xFF, a1 = (own >> 8) & 0xFF;        // 0 beyond the depth
      const bool in0 = 2 * s8 < D, in1 = 2 * s8 + 1 < D;
      const float4 self = nodes[sn], e0 = nodes[a0], e1 = nodes[a1];       // alpha, beta, |k scale|, |q scale|
      const float kk0 = dump[sn * kDumpStride + a0], kk1 = dump[sn * kDumpStride + a1];
      const float qk0 = dump[(kNT + sn) * kDumpStride + a0], qk1 = dump[(kNT + sn) * kDumpStride + a1];
      const float al0 = in0 ? e0.x : 1.f, al1 = in1 ? e1.x : 1.f;
      // products of alpha over the path entries behind each of the two
      float incl = al0 * al1;
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {
        const float v = __shfl_down_sync(0xffffffffu, incl, o, 8);
        if (s8 + o < 8) incl *= v;
      }
      float G1 = __shfl_down_sync(0xffffffffu, incl, 1, 8);
      if (s8 == 7) G1 = 1.f;
      const float g_t = __shfl_sync(0xffffffffu, incl, 0, 8);   // over the whole path
      const float bk = self.y * self.z, k0 = G1 * al1 * e0.z, k1 = G1 * e1.z;
      float w0 = in0 ? self.w * k0 * qk0 : 0.f, w1 = in1 ? self.w * k1 * qk1 : 0.f;
      *reinterpret_cast<float2*>(At + sn * kAStride + 2 * s8) = make_float2(2 * s8 < D - 1 ? bk * k0 * kk0 : 0.f, 2 * s8 + 1 < D - 1 ? bk * k1 * kk1 : 0.f);
      if (s8 == 0) {
        sm.ck[sn] = bk * g_t;
        sm.cq[sn] = D > 0 ? g_t * self.w : 0.f;
      }
      crew();
      if constexpr (kFused) {
        if (fresh && sm.plen > 0) {                             // recorded key and value rows of the accepted nodes
          const LayerPtrs& PL = fp->lb.l[cur.layer];
          const __nv_bfloat16 *pk = reinterpret_cast<const __nv_bfloat16*>(PL.k), *pv = reinterpret_cast<const __nv_bfloat16*>(PL.v);
          const int g = rep > 1 ? (int)__umulhi((uint32_t)cur.hv, rep_mul) : cur.hv;
          for (int e = tid; e < sm.plen * 32; e += kThreads) {  // bounded: <= 2 rounds
            const int tt = e >> 5, c = e & 15;
            const size_t pr = (size_t)cur.b * fp->Ns + sm.phys[tt];
            if ((e & 16) == 0) cp_async16(sbase + kOffPrevK + tt * 256 + c * 16, pk + (pr * s.Hk + g) * kD + c * 8, true);
            else cp_async16(sbase + kOffPrevV + tt * 256 + c * 16, pv + (pr * s.Hv + cur.hv) * kD + c * 8, true);
          }
        }
      }
      // back substitution over the node's own path: m[j] = W[j] - sum_(i > j) m[i] A[a_i][j]
#pragma unroll
      for (int i4 = 3; i4 >= 0; --i4) {
        if (4 * i4 < Dw) {                                      // uniform over the warp
          float2 row[4];
#pragma unroll
          for (int e = 3; e >= 0; --e) row[e] = *reinterpret_cast<const float2*>(At + ((aw[i4] >> (8 * e)) & 0xFF) * kAStride + 2 * s8);
#pragma unroll
          for (int e = 3; e >= 0; --e) {
            const float m = __shfl_sync(0xffffffffu, e & 1 ? w1 : w0, 2 * i4 + (e >> 1), 8);
            if (4 * i4 + e < D) {                               // (an entry beyond the depth names node 0: not its business)
              w0 = fmaf(-m, row[e].x, w0);
              w1 = fmaf(-m, row[e].y, w1);
            }
          }
        }
      }
      const uint32_t hi_at = sw128_offset(sn, 0), lo_at = sw128_offset(sn, 4);
      auto put = [&](int a, float w, float beta) {
        uint32_t hi, lo;                                        // low half: Mc, high half: M diag(beta)
        split2(make_float2(-w * sm.ck[a], w * beta), hi, lo);
        const uint32_t piece = (uint32_t)((a >> 3) << 4), in_piece = (uint32_t)((a & 7) * 2);
        const uint32_t at_hi = (hi_at ^ piece) + in_piece, at_lo = (lo_at ^ piece) + in_piece;
        *reinterpret_cast<unsigned short*>(smem + kOffMc + at_hi) = (unsigned short)hi;
        *reinterpret_cast<unsigned short*>(smem + kOffMc + at_lo) = (unsigned short)lo;
        *reinterpret_cast<unsigned short*>(smem + kOffMb + at_hi) = (unsigned short)(hi >> 16);
        *reinterpret_cast<unsigned short*>(smem + kOffMb + at_lo) = (unsigned short)(lo >> 16);
      };
      if (in0) put(a0, w0, e0.y);
      if (in1) put(a1, w1, e1.y);
    }
    cp_async_wait_all();                                        // value rows
    if (rarely(any_not_finite(*reinterpret_cast<const uint4*>(smem + v_dst), *reinterpret_cast<const uint4*>(smem + v_dst + 2048)))) drop(v_dst, bad);
    if (rarely(sm.look[k & 1] != 0)) drop(kq_dst, bad);
    fence_async_proxy();
    tc_fence_before();
    all();
    // ---- meanwhile the state: (replayed and) converted to hi and lo in tensor memory, a warp sixteen rows, four lanes a row -------
    if (fresh) {
      if constexpr (kFused) {
        if (sm.plen > 0) {
          for (int tt = warp; tt < sm.plen; tt += kWarps) {      // bounded: <= 2 rounds
            const uint2 w = *reinterpret_cast<const uint2*>(smem + kOffPrevK + tt * 256 + lane * 8);
            const float2 k01 = unpack_bf16(w.x), k23 = unpack_bf16(w.y);
            float kk = fmaf(k01.x, k01.x, fmaf(k01.y, k01.y, fmaf(k23.x, k23.x, k23.y * k23.y)));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) kk += __shfl_xor_sync(0xffffffffu, kk, o);
            if (lane == 0) sm.prev_ks[tt] = s.l2norm ? rsqrtf(kk + s.l2_eps) : 1.f;
          }
        }
      }
      if (mbar_wait(&sm.mb_state, ph_state, spin_limit)) ph_state ^= 1;
      else sm.timed_out = sm.state_missing = 1;
      const int r0 = 32 * (warp & 3) + 16 * (warp >> 2) + (lane >> 2);           // rows r0 and r0 + 8
      const float* base = reinterpret_cast<const float*>(smem + kOffS) + r0 * kD + (lane & 3) * 4;
      const uint32_t to = tmem + ((uint32_t)(32 * (warp & 3) + 16 * (warp >> 2)) << 16) + kColS;
      if constexpr (kFused) {
        const int plen = sm.plen;
        if (plen > 0) crew();
        if (plen > 0 && !sm.state_missing) {                    // (the same in every warp: nothing but a state that is there goes back)
#pragma unroll 1
          for (int r = 0; r < 2; ++r) {                         // eight rows at a time, a lane four columns of each; back to where
            const int first = 32 * (warp & 3) + 16 * (warp >> 2) + 8 * r;        // they were, and to memory
            float* rows = reinterpret_cast<float*>(smem + kOffS) + first * kD + lane * 4;
            float4 x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = *reinterpret_cast<const float4*>(rows + u * kD);
#pragma unroll 1
            for (int tt = 0; tt < plen; ++tt) {                 // bounded: <= 16
              const uint2 w = *reinterpret_cast<const uint2*>(smem + kOffPrevK + tt * 256 + lane * 8);
              const float2 k01 = unpack_bf16(w.x), k23 = unpack_bf16(w.y), ab = sm.gates[tt];
              const float ks = sm.prev_ks[tt];
              float p[8];
#pragma unroll
              for (int u = 0; u < 8; ++u) {
                const float2 d = __ffma2_rn(make_float2(x[u].z, x[u].w), k23, __fmul2_rn(make_float2(x[u].x, x[u].y), k01));
                p[u] = d.x + d.y;
              }
              // eight row sums over 32 lanes: each exchange halves the values a lane carries, so that lanes 4 u' .. 4 u' + 3
              // end with the sum of row u (u' = u with its bits reversed) and work out that row's correction alone
              const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
              float q4[4], q2[2], q1;
#pragma unroll
              for (int i = 0; i < 4; ++i) q4[i] = (b4 ? p[i + 4] : p[i]) + __shfl_xor_sync(0xffffffffu, b4 ? p[i] : p[i + 4], 16);
#pragma unroll
              for (int i = 0; i < 2; ++i) q2[i] = (b3 ? q4[i + 2] : q4[i]) + __shfl_xor_sync(0xffffffffu, b3 ? q4[i] : q4[i + 2], 8);
              q1 = (b2 ? q2[1] : q2[0]) + __shfl_xor_sync(0xffffffffu, b2 ? q2[0] : q2[1], 4);
              q1 += __shfl_xor_sync(0xffffffffu, q1, 2);
              q1 += __shfl_xor_sync(0xffffffffu, q1, 1);
              const int mine = (b4 ? 4 : 0) + (b3 ? 2 : 0) + (b2 ? 1 : 0);
              const float vv = __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(smem + kOffPrevV + tt * 256)[first + mine]);
              const float gk = ab.y * (vv - ab.x * (ks * q1)) * ks;
              const float2 a2 = make_float2(ab.x, ab.x);
#pragma unroll
              for (int u = 0; u < 8; ++u) {
                const float g1 = __shfl_sync(0xffffffffu, gk, (u & 4) * 4 + (u & 2) * 4 + (u & 1) * 4);
                const float2 g2 = make_float2(g1, g1);
                const float2 l2 = __ffma2_rn(a2, make_float2(x[u].x, x[u].y), __fmul2_rn(g2, k01));
                const float2 h2 = __ffma2_rn(a2, make_float2(x[u].z, x[u].w), __fmul2_rn(g2, k23));
                x[u] = make_float4(l2.x, l2.y, h2.x, h2.y);
              }
            }
            float* to_rows = state_of(cur.layer, cur.row, cur.hv) + first * kD + lane * 4;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              *reinterpret_cast<float4*>(to_rows + u * kD) = x[u];
              *reinterpret_cast<float4*>(rows + u * kD) = x[u];
            }
          }
          __syncwarp();
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {                             // 64 key columns at a time
        uint32_t hi[16], lo[16];
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          const float4 x = *reinterpret_cast<const float4*>(base + h * 64 + n * 16), y = *reinterpret_cast<const float4*>(base + 8 * kD + h * 64 + n * 16);
          split2(make_float2(x.x, x.y), hi[4 * n], lo[4 * n]);
          split2(make_float2(x.z, x.w), hi[4 * n + 1], lo[4 * n + 1]);
          split2(make_float2(y.x, y.y), hi[4 * n + 2], lo[4 * n + 2]);
          split2(make_float2(y.z, y.w), hi[4 * n + 3], lo[4 * n + 3]);
        }
        tmem_st_16x256b_x4(to + 32 * h, hi);
        tmem_st_16x256b_x4(to + 64 + 32 * h, lo);
      }
      tmem_st_wait();
      if constexpr (kFused) crew();                             // the recorded rows give way to q~
    }
    // ---- effective queries: lane = key column, a thread sixteen nodes --------------------------------------------------
    {
      const uint32_t q_at = kOffKQ + (trow >> 6) * kKQBlock + 4096 + t0 * 128 + (trow & 7) * 2;
      const int qc = (trow & 63) >> 3;                          // 16-byte piece of this column
      float qv[16];
#pragma unroll
      for (int e = 0; e < 16; ++e)
        qv[e] = __uint_as_float((uint32_t)*reinterpret_cast<const unsigned short*>(smem + q_at + e * 128 + ((qc ^ (e & 7)) << 4)) << 16);
#pragma unroll
      for (int e = 0; e < 16; e += 4) {
        const float4 c = *reinterpret_cast<const float4*>(&sm.cq[t0 + e]);
        qv[e] *= c.x; qv[e + 1] *= c.y; qv[e + 2] *= c.z; qv[e + 3] *= c.w;
      }
      all();
      ph_mma ^= 1;
      tc_fence_after();
      uint32_t r[16];
      tmem_ld16(tmem_lane + kColQt + t0, r);
      tmem_ld_wait();
      uint32_t hi[8], lo[8];
#pragma unroll
      for (int e = 0; e < 8; ++e)
        split2(__fadd2_rn(make_float2(__uint_as_float(r[2 * e]), __uint_as_float(r[2 * e + 1])), make_float2(qv[2 * e], qv[2 * e + 1])), hi[e], lo[e]);
      unsigned char* qt = smem + kOffQt + trow * 64;
      const int c0 = ((t0 >> 3) ^ ((trow >> 1) & 3)) << 4, c1 = (((t0 >> 3) + 1) ^ ((trow >> 1) & 3)) << 4;
      *reinterpret_cast<uint4*>(qt + c0) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
      *reinterpret_cast<uint4*>(qt + c1) = make_uint4(hi[4], hi[5], hi[6], hi[7]);
      *reinterpret_cast<uint4*>(qt + 8192 + c0) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
      *reinterpret_cast<uint4*>(qt + 8192 + c1) = make_uint4(lo[4], lo[5], lo[6], lo[7]);
    }
    fence_async_proxy();
    tc_fence_before();
    all();
    // ---- O^T = S0 Q~ is on its way; the key and query rows are free --------------------------------------------------------
    if (n_have) request_kq(nxt, n0, n1);
    all();
    ph_mma ^= 1;
    tc_fence_after();
    if (sm.timed_out) break;                                    // the same in every thread
    if (n_have) request_v(nxt, n0, n1);                         // the value rows have been read
    // ---- outputs: lane = value row; through shared memory, then a node's row 16 bytes at a time -----------------------
    {
      uint32_t r[16];
      tmem_ld16(tmem_lane + kColO + t0, r);
      tmem_ld_wait();
      if (s.out_dtype == LUMO_BF16) {
        __nv_bfloat16* st = reinterpret_cast<__nv_bfloat16*>(smem + kOffQt) + t0 * kD + trow;
#pragma unroll
        for (int e = 0; e < 16; ++e) st[e * kD] = __float2bfloat16_rn(__uint_as_float(r[e]));
      } else {
        float* st = reinterpret_cast<float*>(smem + kOffQt) + t0 * kD + trow;
#pragma unroll
        for (int e = 0; e < 16; ++e) st[e * kD] = __uint_as_float(r[e]);
      }
    }
    tc_fence_before();
    crew();
    const uint32_t marked = *bad;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int m = h ? m1 : m0, node = r16 + 16 * h;
      if (((m >> 24) & 1) == 0) continue;                       // no node, or another group writes it
      bool gone = false;
      if (marked) {                                             // rare: a node of its path is not finite
        const uint8_t* path = t.st_anc + ((size_t)cur.gi * kNT + node) * 16;
        for (int j = 0; j < ((m >> 16) & 0xFF); ++j) gone = gone || ((marked >> path[j]) & 1u);     // bounded: <= 16
      }
      unsigned char* to = const_cast<unsigned char*>(cur.out) + ((size_t)(uint32_t)(m & 0xFFFF) * v_pitch + c16 * 8) * out_size;
      if (s.out_dtype == LUMO_BF16) {
        uint4 o = *reinterpret_cast<const uint4*>(smem + kOffQt + node * 256 + c16 * 16);
        if (gone) o = make_uint4(0x7FC07FC0u, 0x7FC07FC0u, 0x7FC07FC0u, 0x7FC07FC0u);
        *reinterpret_cast<uint4*>(to) = o;
      } else {
        const float4* st = reinterpret_cast<const float4*>(smem + kOffQt + node * 512 + c16 * 32);
        float4 o0 = st[0], o1 = st[1];
        const float nan = __uint_as_float(0x7FC00000u);
        if (gone) o0 = o1 = make_float4(nan, nan, nan, nan);
        reinterpret_cast<float4*>(to)[0] = o0;
        reinterpret_cast<float4*>(to)[1] = o1;
      }
    }
    m0 = n0; m1 = n1;
  }
  cp_async_wait_all();                                          // nobody leaves before its own copies have landed
  }
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

template <bool kDrill, class LB>
__global__ void __launch_bounds__(kThreads + 32, 2) scan_stream_kernel(Shape s, TreeDev t, LB lb, int log_parts) {
  scan_stream_body<false, kDrill, LB>(s, t, lb, log_parts, nullptr);
}
template <bool kDrill, class LB>
__global__ void __launch_bounds__(kThreads + 32, 2) scan_stream_fused_kernel(Shape s, TreeDev t, LB lb, FusedPrevT<LB> fp) {
  scan_stream_body<true, kDrill, LB>(s, t, lb, 0, &fp);
}

template <bool kDrill, class LB>
cudaError_t launch_t(const Shape& s, const TreeDev& t, const LB& lb, const FusedPrevT<LB>* fp, int sm_count, bool pdl, cudaStream_t st) {
  static bool configured[kMaxDevices] = {};                     // the shared-memory limit is a per-device setting
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  if (!configured[dev]) {
    e = cudaFuncSetAttribute(scan_stream_kernel<kDrill, LB>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(scan_stream_fused_kernel<kDrill, LB>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess) return e;
    configured[dev] = true;
  }
  const int items = s.n_layers * s.B * s.Hv, resident = 2 * sm_count;
  if (fp) return launch_kernel(scan_stream_fused_kernel<kDrill, LB>, dim3(items < resident ? items : resident), dim3(kThreads + 32), kSmemBytes, st, pdl, s, t, lb, *fp);
  // A tree of several groups may be shared by CTAs that fetch the same state: what counts is the longest CTA, in steps
  // (a state's fetch and conversion cost about a third of a step)
  int log_parts = 0;
  if (t.st_groups > s.B) {
    long long best = -1;
    const int per_tree = (t.st_groups + s.B - 1) / s.B;
    for (int lp = 0; lp <= 3 && (1 << lp) <= per_tree; ++lp) {
      const long long waves = (((long long)items << lp) + resident - 1) / resident, cost = waves * (3 * ((per_tree + (1 << lp) - 1) >> lp) + 1);
      if (best < 0 || cost < best) { best = cost; log_parts = lp; }
    }
  }
  const int units = items << log_parts;
  return launch_kernel(scan_stream_kernel<kDrill, LB>, dim3(units < resident ? units : resident), dim3(kThreads + 32), kSmemBytes, st, pdl, s, t, lb, log_parts);
}

}  // namespace

// Where the streamed scan takes the place of the closed form with the tensor-core sum (scan_gram.cu).  Measured at 380 points over
// 4 to 256 nodes and 32 to 4096 items (a state each), launches overlapped, us, closed form / streamed:
//   * groups of 32 alone: always.  16 nodes, 32 items 6.0 / 5.0, 304 14.8 / 10.4, 2048 54.9 / 45.1; 28 nodes 7.0 / 5.3, 16.6 / 11.0, 61.5 / 46.6.
//   * one group of 64 that falls into two or three of 32: nearly always.  As long as the parts of a tree find SMs of their own (64
//     nodes, 72 items 10.6 / 8.8); from the fifth wave on (56 nodes, 2048 items 95.8 / 76.3; 64 nodes 98.8 / 98.4); with fewer than three
//     groups also between (58 nodes, 448 items 26.7 / 25.0; 62 nodes, 148 11.6 / 11.6), where three lose (64 nodes, 148 items 11.3 /
//     12.0, 340 23.9 / 27.9).  One wave of whole trees waits for its longest: two groups each win (50 nodes, 224 items 13.2 / 11.9), a
//     few trees of three turn it (57 nodes, 156 items 12.9 / 13.4), three lose most (64 nodes, 292 items 14.6 / 17.0).
//   * several groups of 64: nearly always (256 nodes, 1024 items 213 / 157; 70 nodes, 224 items 24.4 / 15.5).  Not where the larger
//     tiles make one wave and a tree's halves, on shared SMs, three steps (150 nodes, 84 items 13.4 / 16.7; 96 nodes, two steps, 148
//     items 14.2 / 12.9), nor where they make two and whole trees of six steps put a second CTA on a few SMs (160 nodes, 180 items
//     26.0 / 30.0; 128 nodes, five steps, 176 items 25.2 / 24.7).
// With the commit folded in (whole calls) groups of 32 alone: from the second wave on (8 nodes, 448 items 32.3 / 31.7, 1200 67.4 / 62.6;
// 20 nodes, 1200 75.2 / 69.6), before that from 20 nodes on (20 nodes, 76 items 19.2 / 17.9; 16 nodes 16.5 / 17.6; 8 nodes, 152 17.4 /
// 19.4), never where every CTA has an SM to itself (28 nodes, 64 items 18.4 / 19.6).  Trees that need a second group keep the 64-node
// tile: 34 nodes, 1536 items 118 / 122, 64 nodes 141 / 154.
bool scan_stream_pays(const Shape& s, const TreeDev& t, bool fused, int sm_count) {
  const long long sms = sm_count, items = (long long)s.n_layers * s.B * s.Hv, B = s.B, g32 = t.st_groups;
  const bool apart = 2 * items <= sms, one_wave = items > sms && items <= 2 * sms;
  if (fused) return g32 == B && !apart && (s.N >= 20 || items > 2 * sms);
  if (g32 == B || apart) return true;
  if (t.n_groups == s.B) return one_wave ? g32 == 2 * B : items > 4 * sms || 10 * g32 < 29 * B;
  const long long tiles = (long long)s.n_layers * t.n_groups * s.Hv;
  if (tiles <= 2 * sms) return 12 * g32 <= 49 * B;                // (four groups a tree, but for a few)
  return items <= sms || tiles > 4 * sms || 10 * g32 <= 51 * B;
}

cudaError_t launch_scan_stream(const Shape& s, const TreeDev& t, const LayerBatch& lb, const FusedPrev* fp, int sm_count, bool pdl,
                               cudaStream_t st) {
  auto launch = [&](auto drill) {                               // (the kernels in use do not carry the test aid)
    constexpr bool kDrill = decltype(drill)::value;
    if (s.n_layers > kFewLayers) return launch_t<kDrill>(s, t, lb, fp, sm_count, pdl, st);
    const FewLayers few = few_layers(lb);
    if (!fp) return launch_t<kDrill, FewLayers>(s, t, few, nullptr, sm_count, pdl, st);
    const FusedPrevT<FewLayers> prev = few_layers(*fp);
    return launch_t<kDrill, FewLayers>(s, t, few, &prev, sm_count, pdl, st);
  };
  return s.debug_skip_mma ? launch(std::true_type{}) : launch(std::false_type{});
}

}  // namespace lumo
