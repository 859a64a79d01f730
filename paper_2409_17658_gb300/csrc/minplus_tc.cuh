// minplus_tc.cuh -- one output tile of a (min,+) product on the tensor cores (tcgen05), exact.
//
// Encoding.  A level t in [0, W) is written as the power of two 2^(E - L t) (a bf16 whose exponent field is
// L (W - t) and whose mantissa is zero), anything else -- RD_INF, a value >= W, a tile's padding -- as 0.  Then
//   sum_t enc(A[i][t]) enc(B[t][j]) = sum over the pairs below W of 2^(2E - L (A[i][t] + B[t][j])),
// and with at most 2^(L-1) terms the smallest sum s alone fixes the exponent of the total: the total lies in
// [2^(2E - L s), 2^(2E - L s + L - 1)].  Every product is a power of two and every addend is >= 0, so the fp32
// accumulation may round or truncate: it never falls below the largest term (a power of two itself), and its
// relative error is far below the factor 2 left at the top.  So s is read exactly off the exponent.
//
// A pair with an entry outside the window sums to at least W.  Hence an output with s <= W is decided: it is
// the exact minimum over all pairs.  Any other output is undecided and is computed by the DPX kernel (whole
// tile) or term by term (a few outputs); nothing is assumed about the operands' values.  Entries with bit 14 or
// 15 set (outside the documented range) send the whole tile to the DPX kernel.
//
// Why: the DPX units do 128 add-mins per clock and SM, the tensor cores 4096 bf16 multiply-adds.
#pragma once

#include "rd_internal.cuh"

namespace rd {
namespace tc {

// Geometry.  A pair of CTAs (a cluster of two, cta_group::2) owns a tile of 256 rows x NH x 256 columns: CTA r holds
// rows 128 r .. of A, columns 128 r .. of each 256-column part of B, and the 128 x 256 NH accumulator of its rows in
// TMEM.  16 producer warps load the int16 operands (16-byte loads, one stage ahead in registers), encode them and
// store them in the layout the MMA reads; a 17th warp of CTA 0 issues the MMAs.
//
// Why this split: the operands go through the SM's 128-byte shared memory/L1 path three times (load, store, MMA
// read), so the path, not the tensor core, bounds the tile.  Per 64 terms it carries 384 + 384 + 512 = 1280
// wavefronts against 1024 tensor clocks for NH = 2, and 256 + 256 + 256 = 768 against 512 for NH = 1; one CTA with a
// 128 x 256 tile needs 1152 against 512 (measured: tensor pipe 27 % busy, that path 82 %, N = 16384 in 11.9 ms).
constexpr int kProducers = 512, kThreads = kProducers + 32;
constexpr int kBM = 128, kBN = 256, kBK = 64;                         // one CTA's rows, one part's columns, a stage's terms
constexpr int kBytesA = kBM * kBK * 2, kBytesB = (kBN / 2) * kBK * 2;  // of one CTA; B per part
__host__ __device__ constexpr int stage_bytes(int nh) { return kBytesA + nh * kBytesB; }
__host__ __device__ constexpr int stages(int nh) { return nh == 2 ? 3 : 4; }
__host__ __device__ constexpr int smem_bytes(int nh) { return 1024 + stages(nh) * stage_bytes(nh); }
constexpr int kMostFix = 64;                                          // undecided outputs of 128 x 256 computed term by term
constexpr int64_t kMaxM = (int64_t)65535 * kBM;                       // as the DPX launch
constexpr int64_t kMaxLd = 1 << 23;                                   // strides whose steps fit 32 bits
constexpr int kLookStages = 40;                                       // tiles of fewer stages have no early look
constexpr int64_t kMinK = 64, kMaxK = (int64_t)1 << 19;
constexpr uint32_t kWaitRounds = 1u << 18;                            // bound of every mbarrier wait

// Checked builds (-DRD_CHECKED): what rd_tc_check sets and reads.  Every launch reads the settings and adds to the
// counts.
struct Check {
  uint32_t wait_rounds;  // bound of the waits of a tile (those before the shared memory is given up keep kWaitRounds)
  int32_t hold_at;       // the first pair's MMA warp pauses before this stage, counted from 0 over its tiles (-1: never)
  uint32_t hold_us;      // for so many microseconds, as a warp that is kept from running would
  uint32_t deaf;         // bit r: CTA r of a pair finds nothing in its half of a sample, whatever it holds
  // parts of C written, outputs computed term by term, parts left to the DPX launch, pairs of CTAs that lost their
  // pipeline, tiles left by the early look
  uint32_t decided, fixed, left, lost, early;
};
#ifdef RD_CHECKED
__device__ Check g_check = {kWaitRounds, -1, 0, 0, 0, 0, 0, 0, 0};
__device__ __forceinline__ uint32_t wait_rounds() { return *(volatile uint32_t*)&g_check.wait_rounds; }
__device__ __forceinline__ void count(uint32_t Check::*what, uint32_t n) { atomicAdd(&(g_check.*what), n); }
__device__ __forceinline__ void hold(uint32_t stage) {
  if (blockIdx.x > 1 || (int32_t)stage != *(volatile int32_t*)&g_check.hold_at) return;
  for (uint32_t us = *(volatile uint32_t*)&g_check.hold_us; us > 0; --us) __nanosleep(1000);
}
__device__ __forceinline__ bool deaf(uint32_t rank) { return *(volatile uint32_t*)&g_check.deaf >> rank & 1; }
#else
__device__ __forceinline__ constexpr uint32_t wait_rounds() { return kWaitRounds; }
__device__ __forceinline__ void count(uint32_t Check::*, uint32_t) {}
__device__ __forceinline__ void hold(uint32_t) {}
__device__ __forceinline__ constexpr bool deaf(uint32_t) { return false; }
#endif

// Window and exponent step for sums of at most K terms: 2^(L-1) >= K, and the largest W for which 2^(L-1)
// products of two level-0 codes stay below 2^127: 2 (L W - 127) + L - 1 <= 126.
struct Code {
  uint32_t L, W;
};
__host__ __device__ inline Code code_for(int64_t K) {
  Code c;
  c.L = 7;
  while (((int64_t)1 << (c.L - 1)) < K) ++c.L;
  c.W = (381 - c.L) / (2 * c.L);
  return c;
}

struct Shared {
  uint64_t full[4];   // CTA 0's: a stage is stored in both CTAs (one arrival per producer warp)
  uint64_t empty[4];  // the MMAs that read a stage are done
  uint64_t all;       // every MMA issued so far is done
  int64_t at[2];      // the tile's m0 and n0
  uint32_t tmem;      // the accumulator's TMEM address
  uint32_t bad;       // an operand outside the documented range in either CTA
  uint32_t lost[2];   // a wait ran out in either CTA, in an even or an odd phase of `all`; stays set
  uint32_t look[2];   // the early look: undecided outputs and outputs looked at, both CTAs
  uint32_t vote[2][16];  // a sample's counts by group, from both CTAs; one slot per question in turn
  uint32_t cnt[2];    // undecided outputs of each 128 x 256 part
  uint32_t list[2][kMostFix];
};

// Progress of the pipeline, carried across the tiles that a pair works on.
struct Progress {
  uint32_t st = 0, round = 0;  // next stage, and how often the ring has gone round
  uint32_t all = 0;            // phases of `all` so far
};

__device__ __forceinline__ uint32_t sm_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ uint32_t cta_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t at_rank(const void* p, uint32_t rank) {  // the same variable of another CTA
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(sm_u32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
  cluster_arrive();
  cluster_wait();
}
__device__ __forceinline__ void producers_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kProducers) : "memory"); }
__device__ __forceinline__ void add_at(uint32_t addr, uint32_t v) {
  asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sm_u32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n.reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(sm_u32(b)), "r"(parity)
      : "memory");
  return done;
}
// A wait of phase `all` of the pipeline.  Running out, or finding that another wait has, is reported to both CTAs.
__device__ __forceinline__ void pipe_wait(Shared* s, uint64_t* b, uint32_t parity, uint32_t all) {
  for (uint32_t n = 0; !mbar_try(b, parity); ++n) {
    if (n < 64 || (n < wait_rounds() && !(*(volatile uint32_t*)&s->lost[0] | *(volatile uint32_t*)&s->lost[1]))) continue;
    add_at(at_rank(&s->lost[all & 1], 0), 1);
    add_at(at_rank(&s->lost[all & 1], 1), 1);
    break;
  }
}
// On a barrier of either CTA.  What the arriving warp stored is read by the tensor core alone, each CTA's by its own:
// the proxy fence before the arrival orders that, so the release stays at CTA scope.  (At cluster scope it waits for
// the loads in flight too: N = 16384 took 10.5 ms with such a release in every warp, 7.0 ms in one warp of CTA 1.)
__device__ __forceinline__ void arrive_at(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Once per CTA, all threads of the pair: first the barriers, with an arrival at the cluster barrier (behind whose wait
// the other CTA has started and its barriers are ready), later the accumulator's TMEM columns.
template <int NH>
__device__ __forceinline__ void open(Shared* s) {
  if (threadIdx.x == kProducers) {  // not a thread that the first sample waits for
#pragma unroll
    for (int i = 0; i < stages(NH); ++i) {
      mbar_init(&s->full[i], 2 * kProducers / 32);
      mbar_init(&s->empty[i], 1);
    }
    mbar_init(&s->all, 1);
    s->lost[0] = s->lost[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  cluster_arrive();
}
template <int NH>
__device__ __forceinline__ void take_accumulator(Shared* s) {
  if (threadIdx.x < 32) {
    __syncwarp();  // .aligned: the warp's lanes together, as in every tcgen05 instruction of a whole warp below
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sm_u32(&s->tmem)),
                 "n"(NH * kBN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();  // the other CTA's columns are taken before its first stages are
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// After the last tile, all threads of the pair; no MMA is in flight then.
template <int NH>
__device__ __forceinline__ void close(Shared* s) {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  cluster_sync();
  if (threadIdx.x < 32) {
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(s->tmem), "n"(NH * kBN) : "memory");
  }
}

// A load that stays where it is written (moved together, the loads of a stage cost more registers than there are).
__device__ __forceinline__ uint4 load16(const int16_t* a) {
  uint4 v;
  asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(a));
  return v;
}
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\n"
      "setp.ne.u32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void commit(uint64_t* bar) {  // to the same barrier of both CTAs
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          sm_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t addr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
      "tcgen05.wait::ld.sync.aligned;"  // in one statement: no use of v may move between the two
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(addr)
      : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t addr, uint32_t (&v)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
      : "r"(addr)
      : "memory");
}

// 16 bytes (8 entries) of a matrix row from element e0, RD_INF beyond `len`.
__device__ __forceinline__ uint4 row8(const int16_t* row, int64_t e0, int64_t len) {
  if (e0 + 8 <= len) return __ldg(reinterpret_cast<const uint4*>(row + e0));
  uint32_t w[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint32_t lo = (e0 + 2 * q < len) ? (uint32_t)(uint16_t)row[e0 + 2 * q] : (uint32_t)kInf;
    const uint32_t hi = (e0 + 2 * q + 1 < len) ? (uint32_t)(uint16_t)row[e0 + 2 * q + 1] : (uint32_t)kInf;
    w[q] = lo | (hi << 16);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// Whether a product is worth trying.  A sample of it: 16 groups of one row, 16 columns and 64 terms, spread over its
// rows, columns and terms, 8 from each CTA.  It gives the pairs of entries that are `hits` (both below W, their sum at
// most W), by group, and how many of the 256 outputs have none.  An output stays undecided with probability exp(-hits
// among its K pairs), and a part of 32768 outputs needs nearly all of them decided: 32768 exp(-6.2) = 66.  So a product
// is left to the DPX kernel
//  * where K times the share of hits is below 6.2; if its tiles have an early look, only where it is so by more than the
//    sample's deviation;
//  * if `strict`, where clearly more outputs lack a hit than if the hits were spread evenly, or a quarter lacks one and
//    the groups' hits differ by more than chance: rows, columns or blocks without a small entry, whose outputs stay
//    undecided.
// (The shares of small entries in A and in B alone, asked for before, passed operands in blocks, triangles or stripes of
// 1024 to 2048 rows, which then took 1.1 to 1.55 times the DPX product's time.)
// Only speed hangs on this, as long as both CTAs of a pair get the same answer: each writes what it finds to both, so the
// answer is the same whatever the loads return.  All threads of the pair call it, for the turn-th time; the loads are in
// flight together, so it costs one memory latency.  FIRST: right behind open().
template <bool FIRST>
__device__ __forceinline__ bool worth(const GemmParams& p, uint32_t W, bool strict, Shared* s, uint32_t turn) {
  constexpr int kGroups = 16, kOutputs = 16 * kGroups, kTerms = 64;
  constexpr uint32_t top = 0x80008000u;
  const uint32_t tid = threadIdx.x, lane = tid & 31;
  const uint32_t i = (tid >> 5) * 2 + cta_rank();  // the group; its row's place is another one
  uint32_t* vote = s->vote[turn & 1];              // last read before the barrier of the question in between
  const float need = __fdividef(6.2f * (kOutputs * kTerms), (float)p.K);
  uint32_t hits = 0, any = 0;
  if (tid < 16 * kGroups && p.N >= 8) {
    // 32 bits hold these: K <= kMaxK, N <= ldb <= kMaxLd, M <= kMaxM
    const uint32_t K = (uint32_t)p.K, last = (uint32_t)(p.N - 8) & ~7u;
    const uint32_t M = (uint32_t)p.M;
    // the last summand: offsets without a period, not one residue of the rows only
    const uint32_t row = (((i * 5 + 3) & 15) * M >> 4) + (uint32_t)(0x904d2b2ff239863aull >> 4 * i & (M >= 256 ? 15 : 0));
    uint32_t k = (((lane >> 1) * 16 + i) * K >> 8) & ~3u, col = ((i * (uint32_t)p.N >> 4) & ~7u) + (lane & 1) * 8;
    if (k + 4 > K) k = (K - 4) & ~3u;
    if (col > last) col = last;
    const int16_t* b0 = p.B + (int64_t)k * p.ldb + col;
    uint4 bv[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) bv[t] = __ldg(reinterpret_cast<const uint4*>(b0 + t * p.ldb));
    const uint2 av = __ldg(reinterpret_cast<const uint2*>(p.A + (int64_t)row * p.lda + k));
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const uint32_t a = ((t & 2) ? av.y : av.x) >> (16 * (t & 1)) & 0xFFFFu, b[4] = {bv[t].x, bv[t].y, bv[t].z, bv[t].w};
      // a hit: an entry of B below this.  Entries are below 2^15, so bit 15 of a half of (b | top) - c says b >= c.
      const uint32_t room = (a == 0 ? W : a < W ? W - a + 1 : 0) * 0x00010001u;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t hit = ~((b[q] | top) - room) & top;
        hits += __popc(hit);
        any |= hit >> q;
      }
    }
    hits = __reduce_add_sync(0xFFFFFFFFu, hits);
    any = __reduce_or_sync(0xFFFFFFFFu, (lane & 1) ? any >> 4 : any);  // 8 of the 16 columns in each half's upper byte
    if (deaf(cta_rank())) hits = 0, any = ~0u;
  }
  if (FIRST) cluster_wait();
  if (tid < 16 * kGroups && lane < 2)
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(at_rank(&vote[i], lane)),
                 "r"(hits | (16 - __popc(any & 0xFF00FF00u)) << 16)
                 : "memory");
  cluster_sync();
  const uint32_t v = lane < kGroups ? vote[lane] : 0, mine = v & 0xFFFFu;
  const uint32_t sum = __reduce_add_sync(0xFFFFFFFFu, v), squares = __reduce_add_sync(0xFFFFFFFFu, mine * mine);
  const float found = (float)(sum & 0xFFFFu), none = (float)(sum >> 16), mean = found / kGroups;
  const bool looks = p.K > (kLookStages - 1) * kBK;
  if (!strict) return found >= need || (looks && (need - found) * (need - found) <= found);
  return found >= need && none <= kOutputs * (__expf(-found / kOutputs) + 0.12f) &&
         (none <= 0.25f * kOutputs || (float)squares <= kGroups * mean * (1.3f * mean + 2.f));
}

// One output by its terms, by a whole warp (operands inside [0, RD_INF]: no tile with other entries gets here).
__device__ __forceinline__ int32_t dot(const int16_t* a, const int16_t* b, int64_t ldb, int64_t K) {
  int32_t r = kInf;
  for (int64_t k = threadIdx.x & 31; k < K; k += 32) r = min(r, (int32_t)a[k] + (int32_t)b[k * ldb]);
  return __reduce_min_sync(0xFFFFFFFFu, r);
}

// How the accumulator is read: s = (2E + 127 + L - 1 - exponent field) / L.
struct Decode {
  uint32_t top, inv, W;
  __device__ explicit Decode(const Code& c)
      : top(2 * c.L * c.W - 128 + c.L), inv((65536 + c.L - 1) / c.L), W(c.W) {}  // x / L for x < 256, L <= 20
  __device__ uint32_t operator()(uint32_t bits) const { return ((top - (bits >> 23)) * inv) >> 16; }
};

// A producer thread's share of the stages: where its 16-byte chunks come from and go to.  Of A, two rows (a_next
// elements apart); of B, NB terms (b_next apart) of one column chunk.
struct Feed {
  const int16_t *a, *b;     // the next stage's first chunks
  int32_t a_next, b_next;
  uint32_t a_at, b_at;      // shared memory addresses in stage 0
  uint32_t full;            // CTA 0's first `full` barrier, as a cluster address
  uint32_t w2, step, top2;  // W in both halves; one level in a bf16's bits; level 0 (level W is the code 0)
  uint32_t seen, seen_b[4]; // the bits of all entries; of B's per word where N cuts the chunk
  Progress pr;
};
__device__ __forceinline__ uint4 encode(const Feed& f, const uint4& v) {
  return make_uint4(f.top2 - __vminu2(v.x, f.w2) * f.step, f.top2 - __vminu2(v.y, f.w2) * f.step,
                    f.top2 - __vminu2(v.z, f.w2) * f.step, f.top2 - __vminu2(v.w, f.w2) * f.step);
}
__device__ __forceinline__ void store16(uint32_t at, const uint4& v) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
template <int NH>
struct Chunks {
  static constexpr int A = kBM * kBK / 8 / kProducers, B = kBK * 16 * NH / kProducers;
  static constexpr int kPerRow = 16 * NH, kStepB = kProducers / kPerRow;  // B chunks per term; terms between a thread's
  static_assert(A == 2, "one step between a thread's rows");
};
template <int NH>
__device__ __forceinline__ void stage_free(Feed& f, Shared* s) {  // the MMAs that read the next stage are done
  if (f.pr.round > 0) pipe_wait(s, &s->empty[f.pr.st], (f.pr.round - 1) & 1, f.pr.all);
}
template <int NH>
__device__ __forceinline__ void stage_done(Feed& f) {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
  if ((threadIdx.x & 31) == 0) arrive_at(f.full + f.pr.st * 8);
  if (++f.pr.st == stages(NH)) f.pr.st = 0, ++f.pr.round;
}

// n stages that lie inside the matrices: encoded and stored, each register loaded again, with the next stage, as soon
// as it is free, so that a load has the time of a whole stage to arrive.  CUTS: N may cut a chunk of B.
// The loads in flight need room in the L1 cache, so the ring has 3 (4) stages and not all that fit: with shared memory
// at its largest split N = 16384 took 7.1 ms instead of 5.3.  A second set of registers spills (8.0 ms).
template <int NH, bool CUTS>
__device__ __forceinline__ void feed(Feed& f, Shared* s, const int n) {
  constexpr int NA = Chunks<NH>::A, NB = Chunks<NH>::B, kStepB = Chunks<NH>::kStepB;
  uint4 ra[NA], rb[NB];
#pragma unroll
  for (int h = 0; h < NA; ++h) ra[h] = load16(f.a + (int64_t)(h * f.a_next));
#pragma unroll
  for (int h = 0; h < NB; ++h) rb[h] = load16(f.b), f.b += f.b_next;
  f.a += kBK;
  auto put = [&](const bool again) {
    stage_free<NH>(f, s);
    const uint32_t st = f.pr.st * stage_bytes(NH);
#pragma unroll
    for (int h = 0; h < NA; ++h) {
      f.seen |= ra[h].x | ra[h].y | ra[h].z | ra[h].w;
      store16(f.a_at + st + h * (64 * 128), encode(f, ra[h]));
      if (again) ra[h] = load16(f.a + (int64_t)(h * f.a_next));
    }
#pragma unroll
    for (int h = 0; h < NB; ++h) {
      if (CUTS) {
        f.seen_b[0] |= rb[h].x;
        f.seen_b[1] |= rb[h].y;
        f.seen_b[2] |= rb[h].z;
        f.seen_b[3] |= rb[h].w;
      } else {
        f.seen |= rb[h].x | rb[h].y | rb[h].z | rb[h].w;
      }
      store16(f.b_at + st + h * (kStepB * 128), encode(f, rb[h]));
      if (again) rb[h] = load16(f.b), f.b += f.b_next;
    }
    if (again) f.a += kBK;
    stage_done<NH>(f);
  };
#pragma unroll 1
  for (int i = 1; i < n; ++i) put(true);
  put(false);
}

// A wait ran out in phase `all` - 1 or before: read behind that phase's cluster barrier, and the same in all threads of
// both CTAs, because the next write to the same slot lies behind the next phase's barrier.
__device__ __forceinline__ bool lost_by(const Shared* s, uint32_t all) {
  return *(volatile const uint32_t*)&s->lost[(all - 1) & 1];
}
// Whether the pair's pipeline is intact after its tiles so far.
__device__ __forceinline__ bool usable(const Shared* s, const Progress& pr) { return pr.all == 0 || !lost_by(s, pr.all); }

// The pair's tile at (m0, n0) -- m0 is this CTA's first row, n0 the tile's first column -- over all K terms.  On true,
// this CTA's 128 x 256 NH outputs are in shared memory at buf: row r, 16-byte vector c (columns 8c ..) at
// T[r 32 NH + (c ^ (r & 7))], undecided outputs as RD_INF, those inside M x N counted per 256 columns in s->cnt and the
// first kMostFix listed as row * 512 + column.  False: the DPX kernel has to compute the tile (an entry outside the
// documented range, a wait that ran out, or too little decided: an eighth of the way some of the outputs are
// looked at).  Called by all threads of both CTAs with the same answer; the caller syncs the producers before the
// next call.
//
// A wait that runs out leaves the two CTAs' stages and barrier phases out of step with each other, for good: what was
// waited for may still come.  So it ends the tensor cores' part in this pair (usable): this tile and all later ones are
// the DPX kernel's, no thread waits for long again, and the MMAs already issued are waited for.
template <int NH>
__device__ __forceinline__ bool tile(const GemmParams& p, const int64_t m0, const int64_t n0, const Code code, char* buf,
                                     Shared* s, Progress& pr) {
  constexpr int kGroups = kProducers / 128, kCols = NH * kBN / kGroups;  // a warp's columns of its 32 accumulator rows
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cta_rank();
  const int KT = (int)((p.K + kBK - 1) / kBK);
  // The early look (an eighth of the way) costs 2 us a tile, 8 % of a product at K = 1024; a tile of fewer stages than
  // this that turns out hopeless costs at most 20.
  const int check = KT >= kLookStages ? KT >> 3 : -1;

  if (tid == 0) s->at[0] = m0, s->at[1] = n0;
  if (tid == 0) s->bad = s->look[0] = s->look[1] = s->cnt[0] = s->cnt[1] = 0;
  // whether the early look leaves the tile to the DPX kernel: a share f left open by an eighth of the terms is f^8 at
  // the end, 64 of 32768 at f = 0.46
  auto hopeless = [&](uint32_t all) {
    cluster_sync();  // both CTAs' counts are in
    const bool r = (float)s->look[0] > 0.46f * (float)s->look[1] || lost_by(s, all);
    cluster_sync();  // and read
    return r;
  };

  if (warp == kProducers / 32) {  // the MMA warp
    // Shared memory descriptors (start, leading and stride byte offsets >> 4, version 1, 128-byte swizzle): A K-major,
    // 8-row groups 1024 bytes apart; B N-major, 64-column atoms 8192 bytes apart, 8-term groups 1024.  Instruction
    // descriptor: fp32 accumulator, bf16 operands, B N-major, 256 x 256.
    constexpr uint64_t kDescA =
        ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
    constexpr uint64_t kDescB =
        ((uint64_t)(8192 >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
    constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(kBN >> 3) << 17) |
                                ((uint32_t)((2 * kBM) >> 4) << 24);
    const uint32_t base = sm_u32(buf), tmem = s->tmem;
    const bool issuer = rank == 0 && lane == 0;
    for (int kt = 0; kt < KT; ++kt) {
      if (kt == check) {
        if (issuer) commit(&s->all);
        __syncwarp();
        if (hopeless(++pr.all)) return false;
      }
      if (rank == 0) {
        hold(pr.round * stages(NH) + pr.st);
        pipe_wait(s, &s->full[pr.st], pr.round & 1, pr.all);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (issuer) {
          const uint32_t a0 = base + pr.st * stage_bytes(NH), b0 = a0 + kBytesA;
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk)
#pragma unroll
            for (int h = 0; h < NH; ++h)  // 14 address bits: the CTA's rank in the cluster stands above them
              mma(tmem + h * kBN, kDescA | (((a0 + kk * 32) >> 4) & 0x3FFF),
                  kDescB | (((b0 + h * kBytesB + kk * 2048) >> 4) & 0x3FFF), kIdesc, kt > 0 || kk > 0);
          commit(&s->empty[pr.st]);
        }
        __syncwarp();
      }
      if (++pr.st == stages(NH)) pr.st = 0, ++pr.round;
    }
    if (issuer) commit(&s->all);
    ++pr.all;
    __syncwarp();
    cluster_sync();
    return false;
  }

  // Rows from M on and column chunks from N on repeat ones inside (only outputs outside C see them), so every stage
  // before the last terms is loaded without a branch.  A chunk that N cuts is read whole where a later row of B
  // follows it; its columns from N on are kept out of the range check.
  constexpr int NA = Chunks<NH>::A, NB = Chunks<NH>::B, kStepB = Chunks<NH>::kStepB;
  const int r0 = tid >> 3, ak = (tid & 7) * 8, k0 = tid / Chunks<NH>::kPerRow;
  const int j0 = tid % Chunks<NH>::kPerRow;  // 16 chunks of part 0, 16 of part 1
  int64_t bj = n0 + (j0 >> 4) * kBN + (int)rank * (kBN / 2) + (j0 & 15) * 8;
  if (bj >= p.N) bj = 0;  // N >= 8
  const bool cuts = (p.N & 7) != 0 && p.N < n0 + NH * kBN;  // some chunk of the tile, the same for all its threads
  const int cut = p.N - bj < 8 ? (int)(p.N - bj) : 8;
  const int64_t row_a = m0 + r0 < p.M ? m0 + r0 : p.M - 1, row_b = m0 + r0 + 64 < p.M ? m0 + r0 + 64 : p.M - 1;
  Feed f;
  f.a = p.A + row_a * p.lda + ak;
  f.b = p.B + (int64_t)k0 * p.ldb + bj;
  f.a_next = (int32_t)(row_b - row_a) * (int32_t)p.lda;  // lda, ldb <= kMaxLd
  f.b_next = kStepB * (int32_t)p.ldb;
  // the chunk number within 128 bytes is xored with the row (A) or term (B) modulo 8
  f.a_at = sm_u32(buf) + r0 * 128 + (((ak >> 3) ^ (r0 & 7)) << 4);
  f.b_at = sm_u32(buf) + kBytesA + (j0 >> 3) * 8192 + k0 * 128 + (((j0 & 7) ^ (k0 & 7)) << 4);
  f.full = at_rank(&s->full[0], 0);
  f.w2 = code.W * 0x00010001u;
  f.step = code.L << 7;
  f.top2 = (code.L * code.W << 7) * 0x00010001u;
  f.seen = f.seen_b[0] = f.seen_b[1] = f.seen_b[2] = f.seen_b[3] = 0;
  f.pr = pr;
  // the stage of the last terms: RD_INF in A from K on
  auto feed_last = [&](int kt) {
    uint4 ra[NA], rb[NB];
    const int64_t gk = (int64_t)kt * kBK + ak, b0 = (int64_t)kt * kBK + k0;
#pragma unroll
    for (int h = 0; h < NA; ++h) ra[h] = make_uint4(kInf2, kInf2, kInf2, kInf2);
    if (gk + 8 <= p.K) {
#pragma unroll
      for (int h = 0; h < NA; ++h) ra[h] = load16(f.a + (int64_t)(h * f.a_next));
    } else if (gk < p.K) {
      ra[0] = row8(f.a, 0, p.K - gk);
      ra[1] = row8(f.a + f.a_next, 0, p.K - gk);
    }
#pragma unroll
    for (int h = 0; h < NB; ++h) {
      const int64_t k = b0 + kStepB * h < p.K ? b0 + kStepB * h : p.K - 1;
      rb[h] = cut == 8 ? load16(p.B + k * p.ldb + bj) : row8(p.B + k * p.ldb + bj, 0, cut);
    }
    stage_free<NH>(f, s);
    const uint32_t st = f.pr.st * stage_bytes(NH);
#pragma unroll
    for (int h = 0; h < NA; ++h) {
      f.seen |= ra[h].x | ra[h].y | ra[h].z | ra[h].w;
      store16(f.a_at + st + h * (64 * 128), encode(f, ra[h]));
    }
#pragma unroll
    for (int h = 0; h < NB; ++h) {
      f.seen |= rb[h].x | rb[h].y | rb[h].z | rb[h].w;
      store16(f.b_at + st + h * (kStepB * 128), encode(f, rb[h]));
    }
    stage_done<NH>(f);
  };
  auto drain = [&]() {  // every MMA issued so far is complete
    pipe_wait(s, &s->all, f.pr.all & 1, f.pr.all);
    ++f.pr.all;
    __syncwarp();  // each lane has polled for itself
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  };
  // Behind the cluster barrier after a drain: the MMA warp has issued all it will.  None is in flight afterwards.
  auto settle = [&]() {
    for (uint32_t n = 0; n < kWaitRounds && !mbar_try(&s->all, (f.pr.all - 1) & 1); ++n) {}
  };
  // What the accumulator is read with, computed anew where it is needed: held across the loop it cost spills there.
  struct Reader {
    int row, col0, part;
    uint32_t taddr;
    int64_t rows, cols;  // the tile's rows and columns inside C, from its first ones
    __device__ Reader(const GemmParams& p, Shared* s) {
      int t;
      asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
      const int w = t >> 5;
      row = (w & 3) * 32 + (t & 31);
      col0 = (w >> 2) * kCols;
      part = col0 / kBN;
      taddr = *(volatile uint32_t*)&s->tmem + ((uint32_t)(w & 3) << 21) + (uint32_t)col0;
      rows = p.M - *(volatile int64_t*)&s->at[0];
      cols = p.N - *(volatile int64_t*)&s->at[1];
    }
  };
  auto look = [&]() {
    drain();
    const Reader at(p, s);
    const Decode level(code);
    uint32_t v[8];  // few registers beside the operands in flight
    tmem_ld8(at.taddr, v);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    uint32_t open_n = 0, seen_n = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const bool in = at.row < at.rows && at.col0 + c < at.cols;
      seen_n += in;
      open_n += in && level(v[c]) > code.W;
    }
    open_n = __reduce_add_sync(0xFFFFFFFFu, open_n);
    seen_n = __reduce_add_sync(0xFFFFFFFFu, seen_n);
    if (lane < 2) {
      add_at(at_rank(&s->look[0], lane), open_n);
      add_at(at_rank(&s->look[1], lane), seen_n);
    }
    __syncwarp();
    return hopeless(f.pr.all);
  };
  // whole stages, short of the row of B that no row follows where N cuts a chunk
  const int inside = (int)((p.N & 7) != 0 ? (p.K - 1) / kBK : p.K / kBK);
  int kt = 0;
  for (;;) {
    const int stop = kt < check ? check : KT, n = (stop < inside ? stop : inside) - kt;
    if (n > 0) {
      if (cuts) feed<NH, true>(f, s, n);
      else feed<NH, false>(f, s, n);
      kt += n;
    }
    for (; kt < stop; ++kt) feed_last(kt);
    if (stop == KT) break;
    if (look()) {
      if (lost_by(s, f.pr.all)) settle();
      else if (tid == 0 && rank == 0) count(&Check::early, 1);
      pr = f.pr;
      return false;
    }
  }
#pragma unroll
  for (int e = 0; e < 8; ++e)
    if (e < cut) f.seen |= f.seen_b[e >> 1] & (0xFFFFu << (16 * (e & 1)));
  drain();
  const bool wrong = __any_sync(0xFFFFFFFFu, (f.seen & 0xC000C000u) != 0);
  pr = f.pr;
  if (wrong && lane < 2) add_at(at_rank(&s->bad, lane), 1);
  __syncwarp();
  cluster_sync();  // both CTAs' flags are in; nobody reads a stage any more
  if (lost_by(s, f.pr.all)) {
    settle();
    return false;
  }
  if (s->bad) return false;
  __syncwarp();

  const Reader at(p, s);
  const Decode level(code);
  uint4* T = reinterpret_cast<uint4*>(buf);
  uint32_t mine = 0;
#pragma unroll 1
  for (int c0 = 0; c0 < kCols; c0 += 32) {
    uint32_t v[32];
    tmem_ld32(at.taddr + c0, v);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint32_t o[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const uint32_t x = level(v[q * 8 + e]);
        o[e] = x <= code.W ? x : (uint32_t)kInf;
        if (x > code.W) {
          const int col = at.col0 + c0 + q * 8 + e;
          if (at.row < at.rows && col < at.cols) {
            if (mine < 8) {
              const uint32_t i = atomicAdd(&s->cnt[at.part], 1u);
              if (i < kMostFix) s->list[at.part][i] = (uint32_t)at.row * 512 + col;
            }
            ++mine;
          }
        }
      }
      const int c8 = (at.col0 + c0) / 8 + q;
      T[at.row * (32 * NH) + (c8 ^ (at.row & 7))] =
          make_uint4(o[0] | o[1] << 16, o[2] | o[3] << 16, o[4] | o[5] << 16, o[6] | o[7] << 16);
    }
  }
  if (mine > 8) atomicAdd(&s->cnt[at.part], (uint32_t)kMostFix);  // too many for the list
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  producers_sync();
  return true;
}

}  // namespace tc
}  // namespace rd
