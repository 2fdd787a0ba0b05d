// chym_k2.cu -- large-N step (N > 128): tcgen05 GEMM Y = J X with the CHYM update fused
// into its epilogue, one persistent launch per D and kLaunchSteps Euler-Maruyama steps.
//
// Layouts (device, internal to this path), per context:
//   Xm[c][p]   FP32 master state, column c = r * D + mu, spin p contiguous,
//              leading dimension KP = 128 * MT (MT = ceil(N / 128));
//   Xt[b][t][ct][kc]  BF16 hi (t = 0) / lo (t = 1) split of Xm, double buffered
//              by step parity (b), stored as ready-made B-operand blocks: column
//              tile ct (n = D * RT columns, RT runs) x K chunk kc (32 spins),
//              MN-major canonical layout without swizzle: core matrix = 8 spins x
//              16 bytes (8 consecutive columns), core (col/8, k/8) at
//              (col/8) * 512 + (k/8) * 128.  Columns of a tile are ordered
//              component-major, c_loc = mu * RT + r_loc, so the 8 runs of one
//              component that an epilogue thread finishes form one 16-byte row of
//              a core matrix (one coalesced store per component);
//   Aimg[t][mt][kc]  J (t = 0) and, for real couplings, its BF16 residual
//              (t = 1) as A-operand blocks of 128 rows x 32 K, K-major: core
//              (row/8, k/8) at (row/8) * 512 + (k/8) * 128; for +-1 couplings
//              t = 1 holds J in FP8 e4m3 (exact), 4 KB blocks with core
//              (row/8, k/16) at (row/8) * 256 + (k/16) * 128.
// FP8 mode (+-1 couplings, CHYM_PREC_FP8): the lo half of the split is stored in
// e4m3 instead of BF16, its blocks MN-major with core (col/16, k/8) at
// (col/16) * 512 + (k/8) * 128 (16 columns of one byte per core row), and multiplied
// by the e4m3 image of J with one kind::f8f6f4 product (K = 32) per K chunk at twice
// the BF16 rate.  Both halves carry the scale S = 2^kLoScaleLog2 (exact in BF16), so
// that x_lo S sits in the normal range of e4m3 (|x_lo| <= 2^-9 |x|); the hi and lo
// products add into one FP32 accumulator holding S y, and the epilogue folds 1/S
// into dt eps.  x_lo then keeps 4 significant bits: x = hi + lo within 2^-13 |x|.
// A launch advances every context of its D in the call.  Work is a table of tiles (context,
// M tile mt, column tile ct), dealt to the CTAs once per call: in phases of a few tiles a CTA,
// each advanced by all steps of the launch before the next, the tiles of a phase in lists of
// near-equal cost (costliest first, mt fastest so that the CTAs that run at the same time
// share their column tile's B blocks in L2).  A CTA, one per SM, walks its list of the phase
// once per step; its five roles walk it independently:
//   warp 3  scout: waits until all MT tiles of the column tile have finished the previous
//           step (a counter per column tile in global memory) and clears the tile;
//   warp 0  producer: fills a ring of up to 8 stages with TMA bulk copies of the A / B_hi /
//           B_lo blocks of each K chunk of a cleared tile (mbarrier expect_tx);
//   warp 1  MMA issuer: tcgen05.mma (M = 128, N = n, K = 16), J_hi X_hi +
//           J_hi X_lo (+ J_lo X_hi), FP32 accumulators in TMEM, two of them so
//           that the next tile's products run while the epilogue drains the last;
//   warps 4-11 epilogue: thread = spin (TMEM lane) x half of the tile's runs; it
//           loads its runs' x (global) before the accumulator is ready, then reads
//           Y (tcgen05.ld), applies drift, loss, annealing and Philox noise (text
//           after Eq. 1 and after Fig. 2), writes x back and the new BF16 hi/lo
//           straight into the other buffer (the next step's B blocks).  Per-run
//           quantities (round keys, the rounds of Philox that depend on the run and step
//           only, annealing scale) are staged per warp in shared memory;
//   warp 2  publisher: once every epilogue warp has stored the tile (generic proxy), fences
//           towards the async proxy of the other SMs' TMA and adds 1 to the column tile's
//           counter.
// A column tile depends on its own tiles of the previous step only, so there is no barrier
// over a step: tiles of other column tiles and contexts fill the time of its hand-over.
// (One launch per step and D, graph-replayed, measured: 32 uneven instances 187 us a step,
// N = 250 with 1024 runs 18.5 us; every step paid the launch, the ring's fill, the last
// tile's epilogue, and one D after the other left most SMs idle.)
// The CTAs wait for one another, so only CTAs known to be resident take part: each counts
// itself in; once all have, or 100 us after the first, the first one freezes the count P,
// CTAs that start later exit, and the P present ones share the lists of the absent ones; such a
// launch stops early once enough have come late, and the next one counts again (go_on).
// All waits are bounded; on a timeout the CTA raises the status word, drains its own
// tensor-core and copy work with bounded waits, frees TMEM and returns.
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include <algorithm>
#include <type_traits>
#include <utility>
#include <vector>

#include "chym_internal.cuh"

namespace chym {
namespace {

constexpr int kKc = 32;                        // K chunk (spins) of one stage
constexpr uint32_t kABlock = 128 * kKc * 2;    // bytes of an A block (8 KB)
constexpr uint32_t kCoreK = 128;               // K-direction core stride (both operands)
constexpr uint32_t kCoreMN = (kKc / 8) * 128;  // M/N-direction core stride (512)
constexpr int kMaxStages = 8;
constexpr int kWQ = 2;                         // epilogue warps per TMEM lane quarter
constexpr int kEpiWarps = 4 * kWQ;
constexpr int kUnit = 8;                       // runs of an epilogue unit: a 16-byte core-matrix row of BF16
constexpr int kPiece = 4;                      // runs finished at a time
// Warps 0-3 are the producer, the MMA issuer, the publisher and the scout, the others the
// epilogue.  The helpers' warpgroup hands registers to the epilogue's, which spilled at the
// launch's even share of 168 (16 bytes at D = 4 cost 10 % of a step, 60 at D = 8 13 %: the ring
// leaves the spills little L1).
constexpr int kPubWarp = 2, kScoutWarp = 3, kEpiWarp0 = 4;
constexpr int kThreads = 32 * (kEpiWarp0 + kEpiWarps);
constexpr int kLaunchRegs = 168, kHelperRegs = 64, kEpiRegs = 216;
static_assert(128 * kHelperRegs + 32 * kEpiWarps * kEpiRegs <= kThreads * kLaunchRegs &&
                  kThreads * kLaunchRegs <= 65536, "register split");
constexpr int kAccCols = 256;                  // TMEM columns of one accumulator
constexpr size_t kRingBudget = 192 * 1024;     // shared memory for the stage ring
constexpr int kLaunchSteps = 1024;             // most steps of one launch
constexpr int kCheckSteps = 2;                 // with CTAs missing: steps between looks for late ones
constexpr int kMaxGridY = 65535;
// Phases.  The CTAs of a phase stay within its tiles of one another, so that those that share a
// column tile read it while it is in L2; walking their whole lists they drift apart by up to a
// step.  Two tiles a CTA are the fewest that cover a tile's hand-over: us a step for 1 / 2 / 3 /
// 4 / all, N = 800, D = 4, 65536 runs 1179 / 766 / 792 / 809 / 943; N = 600, D = 3, 16384 runs
// 172 / 110 / 112 / 114 / 120; 125 instances of N = 130..2000, D = 4, 64 runs 278 / 207 / 214 /
// 215 / 218.  Lists shorter than kPhaseMin keep together by themselves, and in phases a context
// whose tiles lie first in some lists and last in others has no slack for its hand-over (30
// instances of N = 176..2000, D = 2..8, 64 runs, D = 2 in two phases: 86, else 74).  A phase costs the
// filling of the CTAs' pipelines once, not worth it for few steps, and leaves CTAs idle where tiles
// are uneven: by the tiles' times phases may be longer than whole lists by kDriftLoss.
constexpr int kPhaseTiles = 2, kPhaseMin = 4;
constexpr int kPhaseSteps = 32;
constexpr double kDriftLoss = 1.1;
// Several D.  Side by side, on shares of the SMs, they hold each other's data out of L2 and end
// apart (the 512 instances of the uneven workload: 1064 us a step, 821 one after the other; their
// D = 4 and 8 alone 601 and 558; 8 instances of 2048 runs 317 and 307, 0.90 by the tiles' times), so
// it has to gain kBesideLoss by those: few tiles of each D, which would leave SMs idle (28
// instances of N = 61..1707, D = 3 and 4, 72 runs, 0.86: 42 steps take 9.44 ms side by side, 9.85 in
// turn; the 30 uneven ones of kPhaseMin, 0.55: 72 and 137 us a step).
constexpr double kBesideLoss = 1.14;
constexpr double kHandOverNs = 4000.0;         // a step's, with one tile a CTA: store, publish, fetch
constexpr double kLaunchNs = 10000.0;          // start and end of a launch
constexpr uint32_t kA8Block = 128 * kKc;       // bytes of an e4m3 A block (4 KB)
constexpr int kLoScaleLog2 = 16;               // FP8 mode: B operands carry 2^16

// Most runs per column tile (n = D * RT <= 256).  Any RT is a multiple of 8 (the epilogue's
// units) with n a multiple of 16: 32 and its multiples, or 16 and 24 from k2_pick_rt.
__host__ __device__ constexpr int k2_rt_max(int D) {
  return D == 1 ? 256 : D == 2 ? 128 : D <= 4 ? 64 : 32;
}

// One large-N context of a launch.
struct K2Desc {
  int D;
  int flag0;               // its first column-tile counter
  const uint8_t* Aimg;
  float* Xm;
  uint8_t* Xt;             // both buffers; buffer b at Xt + b * buf_bytes
  const float* ar;         // per run: 1 + dt (h - 1)
  const uint64_t* seeds;   // per run: Philox key
  const int64_t* koff;     // per run: global step of its (re)seeding
  unsigned long long buf_bytes;  // even: a 256-byte multiple
  int N, KP, MT, KC, CT, RT, n, n_runs, a_terms, sched_kind;
  int lo8;                 // 1: lo half in e4m3 (FP8 mode, +-1 couplings)
  int stall;               // CHYM_FLAG_TEST_STALL: the accumulator-full signal is withheld
  int64_t k0, k_anneal, k_total;  // k0: step of the context when the call began
  float gdt, kdt, edt, neg2ln2s2, inv_ramp;
};

struct K2Tile {
  int desc, mt, ct, pad;
};

// Per-run quantities of one step, staged in shared memory by each epilogue warp for the
// next slots() runs it finishes.  r12[blk] carries the first two Philox rounds as far as
// they depend on the run and the step only (see philox_run), rk the keys of rounds 3..10.
template <int D>
struct __align__(16) RunC {
  static constexpr int kSlots = 32;
  uint4 r12[(D + 3) / 4];
  uint4 rk[4];
  float ar, erp;  // 1 + dt (h - 1), and dt eps alpha_mu of the extra components mu >= 1
};
constexpr int kTileCache = 24;  // tiles of a CTA's list whose descriptors are kept in shared memory

// Where a launch begins: steps taken in this call, and launches that stopped early so far.
struct K2Progress {
  int64_t step;
  int stops, pad;
};

struct K2Launch {
  const K2Desc* descs;
  const K2Tile* tiles;
  int n_tiles;
  const int* cta_begin;   // list of CTA b: tiles [cta_begin[b], cta_begin[b + 1])
  const int* phase_end;   // [CTA][phase]: ends of the phases in its list
  int phases;
  unsigned* sync;         // [0] CTAs arrived (kFrozen: count closed), [1] their number when it was
                          // closed, [2] 2 x checks passed + 1 if stopped at the next (go_on)
  unsigned* flags;        // per column tile: M tiles finished, over all steps of the launch
  K2Progress* progress;   // of this launch and the next, by launch parity
  int launch;             // parity of its index in the call
  int max_stops;          // launches of the call that may stop early
  int64_t total;          // steps of the call
  int stages;             // depth of the ring
  uint32_t stage_stride;  // bytes per stage
  unsigned* status;
  unsigned long long wait_ns;  // limit of every bounded wait
};
constexpr unsigned kFrozen = 0x80000000u;
constexpr unsigned long long kJoinNs = 100000;

__host__ __device__ inline uint32_t b_block_bytes(int n) { return (uint32_t)n * kKc * 2u; }
// bytes of a lo block: BF16, or e4m3 in FP8 mode
__host__ __device__ inline uint32_t b_lo_bytes(int n, int lo8) { return (uint32_t)n * kKc * (lo8 ? 1u : 2u); }
// bytes of one stage of a context: A (and its second term: the BF16 residual of real
// J or the e4m3 J of FP8 mode), B hi and B lo
__host__ __device__ inline uint32_t stage_bytes(int n, int a_terms, int lo8) {
  return kABlock + (a_terms > 1 ? kABlock : lo8 ? kA8Block : 0u) + b_block_bytes(n) + b_lo_bytes(n, lo8);
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint64_t global_timer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait for the completion of phase `parity` of an mbarrier.  Each try_wait
// may suspend the thread for up to kSuspendNs (it resumes as soon as the phase
// completes), so waiting warps do not take issue slots from working ones.
constexpr uint32_t kSuspendNs = 20000;
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, unsigned long long limit_ns) {
  uint64_t t0 = 0;
  for (uint32_t it = 0;; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity), "r"(kSuspendNs)
        : "memory");
    if (done) return true;
    const uint64_t t = global_timer();
    if (it == 0) t0 = t;
    else if (t - t0 > limit_ns) return false;
  }
}
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}
// D (+)= A B on the tensor core, kind::f16 (BF16 operands, FP32 accumulator), issued by one
// elected lane of a converged warp.  The whole warp runs the issue loop: its descriptors
// stay in uniform registers (44 cycles a product of N = 48, 128 of N = 256, the tensor
// core's own rates), while a lone thread's loop moves them there for every product (65 to
// 150 cycles).
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\tsetp.ne.b32 p, %4, 0;\n\telect.sync _|e, 0xffffffff;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}
// D += A B, kind::f8f6f4 (e4m3 operands, K = 32, FP32 accumulator), issued likewise.
__device__ __forceinline__ void mma_f8(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc) {
  asm volatile(
      "{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, 1;\n\t}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc));
}
// Arrival on an mbarrier once the products issued so far are complete; the lane elected for
// them (the same one for every elect.sync of a full warp).
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\t"
      "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}\n" ::"r"(bar)
      : "memory");
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}
// SFU approximations with denormals flushed; no argument or result of the noise
// transform below is denormal, so they equal the non-flushing forms there.
__device__ __forceinline__ float sqrt_ftz(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float lg2_ftz(float x) {
  float r;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ void sincos_ftz(float x, float& s, float& c) {
  asm("sin.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(x));
  asm("cos.approx.ftz.f32 %0, %1;" : "=f"(c) : "f"(x));
}
// Box-Muller on the word pairs of two runs at once (see box_muller_f32 in
// chym_internal.cuh), in paired FP32 arithmetic: z0 = (z0 of run A, of run B), likewise z1;
// the noise scale sigma sqrt(dt) is folded into neg2ln2s2 = -2 ln2 (sigma^2 dt).
__device__ __forceinline__ void box_muller2(uint32_t wrA, uint32_t waA, uint32_t wrB, uint32_t waB,
                                            float neg2ln2s2, float2& z0, float2& z1) {
  const float2 ur = __ffma2_rn(make_float2((float)wrA, (float)wrB),
                               make_float2(2.3283064365386963e-10f, 2.3283064365386963e-10f),
                               make_float2(1.1641532182693481e-10f, 1.1641532182693481e-10f));
  const float2 th = __ffma2_rn(make_float2((float)waA, (float)waB),
                               make_float2(1.4629180792671596e-09f, 1.4629180792671596e-09f),
                               make_float2(-3.1415926528582302f, -3.1415926528582302f));
  const float2 r2 = __fmul2_rn(make_float2(neg2ln2s2, neg2ln2s2), make_float2(lg2_ftz(ur.x), lg2_ftz(ur.y)));
  const float2 r = make_float2(-sqrt_ftz(r2.x), -sqrt_ftz(r2.y));
  float sA, cA, sB, cB;
  sincos_ftz(th.x, sA, cA);
  sincos_ftz(th.y, sB, cB);
  z0 = __fmul2_rn(r, make_float2(cA, cB));
  z1 = __fmul2_rn(r, make_float2(sA, sB));
}
// Philox4x32-10 of the block of spin (group) p of a run at its local step.  Counter (p, blk,
// k_lo, k_hi) and key (k0, k1): round 1 multiplies p (a constant of the thread: mp = M0 p)
// and k_lo, and round 2 the result of k_lo's product, which depends on the run and step
// only.  RunC::r12 holds what is left of both rounds (k' = the round-2 key):
//   x = k_hi ^ k1, y = lo(M1 k_lo) ^ k0', z = hi(M0 c) ^ k1', w = lo(M0 c) with
//   c = hi(M1 k_lo) ^ blk ^ k0.
__device__ __forceinline__ uint4 run_rounds12(uint32_t blk, uint32_t k_lo, uint32_t k_hi, uint32_t k0, uint32_t k1) {
  const uint64_t p1 = (uint64_t)kPhiloxM1 * k_lo;
  const uint64_t p0 = (uint64_t)kPhiloxM0 * ((uint32_t)(p1 >> 32) ^ blk ^ k0);
  return make_uint4(k_hi ^ k1, (uint32_t)p1 ^ (k0 + kPhiloxW0), (uint32_t)(p0 >> 32) ^ (k1 + kPhiloxW1), (uint32_t)p0);
}
template <int D>
__device__ __forceinline__ uint4 philox_run(uint64_t mp, const RunC<D>& rc, int blk) {
  const uint4 t = rc.r12[blk];
  const uint64_t q = (uint64_t)kPhiloxM1 * ((uint32_t)(mp >> 32) ^ t.x);
  uint4 c = make_uint4((uint32_t)(q >> 32) ^ t.y, (uint32_t)q, t.z ^ (uint32_t)mp, t.w);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint4 kk = rc.rk[i];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint64_t p0 = (uint64_t)kPhiloxM0 * c.x, p1 = (uint64_t)kPhiloxM1 * c.z;
      c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ (h ? kk.z : kk.x), (uint32_t)p1,
                     (uint32_t)(p0 >> 32) ^ c.w ^ (h ? kk.w : kk.y), (uint32_t)p0);
    }
  }
  return c;
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// Bounded wait until *p >= want (p: a counter other SMs add to).
__device__ __forceinline__ bool counter_wait(const unsigned* p, unsigned want, unsigned long long limit_ns) {
  uint64_t t0 = 0;
  for (uint32_t it = 0;; ++it) {
    if (ld_acquire(p) >= want) return true;
    if ((it & 15u) == 0u) {
      const uint64_t t = global_timer();
      if (it == 0) t0 = t;
      else if (t - t0 > limit_ns) return false;
    }
  }
}
__device__ __forceinline__ uint32_t ld_acquire_cta(uint32_t p) {
  uint32_t v;
  asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_cta(uint32_t p, uint32_t v) {
  asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async;" ::: "memory"); }

// The accumulator columns of a piece's runs for M components, ld columns apart, for the warp's
// 32 lanes, with the wait in the same asm statement (tcgen05.ld fills its registers
// asynchronously until tcgen05.wait::ld, so the compiler must not see them earlier).  One
// round trip for all of them: a load per run pair and component made the D = 8 step 13 %
// slower.
template <int M>
__device__ __forceinline__ void tmem_ld_piece(uint32_t a, uint32_t ld, float (&y)[4][kPiece]) {
  static_assert(kPiece == 4, "x4 loads");
  uint32_t r[16] = {};
  if constexpr (M == 4)
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%16];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4,%5,%6,%7}, [%17];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8,%9,%10,%11}, [%18];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%12,%13,%14,%15}, [%19];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(a), "r"(a + ld), "r"(a + 2 * ld), "r"(a + 3 * ld)
        : "memory");
  else if constexpr (M == 3)
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%12];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4,%5,%6,%7}, [%13];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8,%9,%10,%11}, [%14];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11])
        : "r"(a), "r"(a + ld), "r"(a + 2 * ld)
        : "memory");
  else if constexpr (M == 2)
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%8];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4,%5,%6,%7}, [%9];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
        : "r"(a), "r"(a + ld)
        : "memory");
  else
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
        : "r"(a)
        : "memory");
#pragma unroll
  for (int m = 0; m < M; ++m)
#pragma unroll
    for (int j = 0; j < kPiece; ++j) y[m][j] = __uint_as_float(r[4 * m + j]);
}

// Streaming access to the master state.  Volatile: a thread reads back what it stored
// itself one step earlier, and volatile asm statements keep their order.
__device__ __forceinline__ float ld_stream(const float* p) {
  float v;
  asm volatile("ld.global.cs.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ void st_stream(float* p, float v) {
  asm volatile("st.global.cs.f32 [%0], %1;" ::"l"(p), "f"(v));
}

// x of a piece's consecutive runs (the first `left` of them exist) and all components at the
// thread's spin; x points at the first run's component 0.
template <int D>
__device__ __forceinline__ void load_piece(const float* x, int KP, int left, bool live, float (&v)[D][kPiece]) {
#pragma unroll
  for (int j = 0; j < kPiece; ++j) {
    const bool ok = live && j < left;
#pragma unroll
    for (int mu = 0; mu < D; ++mu) v[mu][j] = ok ? ld_stream(x + (j * D + mu) * KP) : 0.f;  // 32-bit offsets
  }
}

// Split of a piece's n values of one component, packed: BF16 hi words, BF16 lo words.
template <int n>
__device__ __forceinline__ void split_piece(const float (&v)[n], uint32_t (&hi)[n / 2], uint32_t (&lo)[n / 2]) {
#pragma unroll
  for (int j = 0; j < n / 2; ++j) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
    const float2 hf = __bfloat1622float2(h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(v[2 * j] - hf.x, v[2 * j + 1] - hf.y);
    hi[j] = *reinterpret_cast<const uint32_t*>(&h);
    lo[j] = *reinterpret_cast<const uint32_t*>(&l);
  }
}

// FP8 mode: S bf16(v) and, in lo[0], the n bytes e4m3(S (v - bf16(v))), S = 2^kLoScaleLog2.
// The product by S and the difference are exact, so the pair is scaled as BF16 (one
// instruction for two) and the remainder is one FMA.
template <int n>
__device__ __forceinline__ void split_piece8(const float (&v)[n], uint32_t (&hi)[n / 2], uint32_t (&lo)[n / 2]) {
  constexpr float S = (float)(1u << kLoScaleLog2);
  const __nv_bfloat162 S2 = __floats2bfloat162_rn(S, S);
  uint32_t l = 0;
#pragma unroll
  for (int j = 0; j < n / 2; ++j) {
    const __nv_bfloat162 hs = __hmul2_rn(__floats2bfloat162_rn(v[2 * j], v[2 * j + 1]), S2);
    const float2 hf = __bfloat1622float2(hs);
    hi[j] = *reinterpret_cast<const uint32_t*>(&hs);
    l |= (uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(fmaf(v[2 * j], S, -hf.x), fmaf(v[2 * j + 1], S, -hf.y)),
                                            __NV_SATFINITE, __NV_E4M3)
         << (16 * j);
  }
  lo[0] = l;
}

// Constants of one tile for the epilogue, in registers.
struct EpiTile {
  float* Xm;
  int KP, n_runs, RT, run0;  // run0: the tile's first run
  int p;
  bool live;
  float gdt, kdt, edt, nl2;
  uint32_t acc;              // accumulator of the warp's lanes
  uint64_t mp;               // M0 times the Philox counter of the spin
};

// A piece of one unit: x (in: state before the step, out: after it, zero for absent runs)
// at the thread's spin, from the accumulator columns col.. of each component; writes x back.
template <int D>
__device__ __forceinline__ void advance_piece(const EpiTile& w, const RunC<D>* rc, int run, uint32_t col,
                                              float (&x)[D][kPiece]) {
  // per run: 1 + dt(h-1) - dt gamma |x_p|^2 from the state before the step
  float tl[kPiece];
#pragma unroll
  for (int j = 0; j < kPiece; ++j) {
    float n2 = 0.f;
#pragma unroll
    for (int mu = 0; mu < D; ++mu) n2 = fmaf(x[mu][j], x[mu][j], n2);
    tl[j] = fmaf(-w.gdt, n2, rc[j].ar);
  }
  float* xrow = w.Xm + (size_t)run * D * w.KP + w.p;
  auto block = [&](auto blk_c) {  // components 4 blk .. 4 blk + M - 1, one Philox block
    constexpr int blk = decltype(blk_c)::value, M = D - 4 * blk < 4 ? D - 4 * blk : 4;
    float y[4][kPiece];
    tmem_ld_piece<M>(w.acc + (uint32_t)(4 * blk * w.RT) + col, (uint32_t)w.RT, y);
#pragma unroll
    for (int j = 0; j < kPiece; j += 2) {  // two runs at once, paired FP32 arithmetic
      float2 z[4];
      const RunC<D> &cA = rc[j], &cB = rc[j + 1];
      const bool okA = w.live && run + j < w.n_runs, okB = w.live && run + j + 1 < w.n_runs;
      const uint4 wA = philox_run<D>(w.mp, cA, blk), wB = philox_run<D>(w.mp, cB, blk);
      if constexpr (D <= 2) {
        // the 4/D spins with the same p / (4/D) share one block; spin p takes its
        // normals (p % (4/D)) D .. + D - 1, one Box-Muller pair
        constexpr uint32_t per = 4u / D;
        const uint32_t j0 = ((uint32_t)w.p % per) * D;
        const bool hi2 = j0 >= 2u;
        float2 cz, sz;
        box_muller2(hi2 ? wA.z : wA.x, hi2 ? wA.w : wA.y, hi2 ? wB.z : wB.x, hi2 ? wB.w : wB.y, w.nl2, cz, sz);
        z[0] = (j0 & 1u) ? sz : cz;
        z[1] = sz;
      } else {
        box_muller2(wA.x, wA.y, wB.x, wB.y, w.nl2, z[0], z[1]);
        if constexpr (M > 2) box_muller2(wA.z, wA.w, wB.z, wB.w, w.nl2, z[2], z[3]);
      }
      const float2 t2 = make_float2(tl[j], tl[j + 1]), nk2 = make_float2(-w.kdt, -w.kdt);
      const float2 e0 = make_float2(w.edt, w.edt), e1 = make_float2(cA.erp, cB.erp);
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const int mu = 4 * blk + m;
        const float2 xv = make_float2(x[mu][j], x[mu][j + 1]);
        const float2 sf = __ffma2_rn(__fmul2_rn(nk2, xv), xv, t2);
        const float2 inner = __ffma2_rn(mu == 0 ? e0 : e1, make_float2(y[m][j], y[m][j + 1]), z[m]);
        const float2 v = __ffma2_rn(xv, sf, inner);
        x[mu][j] = okA ? v.x : 0.f;
        x[mu][j + 1] = okB ? v.y : 0.f;
        if (okA) st_stream(xrow + (j * D + mu) * w.KP, v.x);
        if (okB) st_stream(xrow + ((j + 1) * D + mu) * w.KP, v.y);
      }
    }
  };
  block(std::integral_constant<int, 0>());
  if constexpr (D > 4) block(std::integral_constant<int, 1>());
}

// What a launch does: steps from `step0`, on P CTAs.
struct K2Span {
  int64_t step0;
  int steps, stops, P;
};

// A CTA's list of tiles: entry i is table entry base + i stride.  The list falls into phases,
// each advanced by all steps before the next begins.
struct TileWalk {
  int base, stride, count, phases;
  const K2Span* span;
  const int* phase_end;  // ends of the phases in the list (one phase: count)
  const K2Launch* L;
  const K2Desc* cache;   // descriptors of the first kTileCache tiles
  __device__ __forceinline__ int index(int i) const { return base + i * stride; }
  __device__ __forceinline__ K2Tile tile(int i) const { return L->tiles[index(i)]; }
  __device__ __forceinline__ const K2Desc& desc(int i, const K2Tile& t) const {
    return i < kTileCache ? cache[i] : L->descs[t.desc];
  }
  __device__ __forceinline__ int end_of(int ph) const { return phases > 1 ? phase_end[ph] : count; }
};

// A launch that found SMs busy goes on past step s (a multiple of kCheckSteps) unless CTAs have
// come late since, a quarter as many as it has or more: then it stops there, and the next
// launch counts anew (kept to the first SMs for the whole launch, a call of 1000 steps of N = 1000,
// D = 4, 2048 runs took 334 ms where a run of 2.3 ms held 140 SMs at its start; 34 now, 32 alone).
// Whoever gets there first decides, so nobody waits: every CTA passes its steps in order, so a
// check is open only while all before it are passed.
__device__ __forceinline__ bool go_on(const K2Launch& L, const K2Span& span, int s) {
  const unsigned e = (unsigned)(s / kCheckSteps);
  for (;;) {
    const unsigned v = ld_acquire(L.sync + 2);
    if (v >> 1 >= e) return true;
    if (v & 1u) return false;
    const unsigned late = (ld_acquire(L.sync) & ~kFrozen) - (unsigned)span.P;
    const bool stop = span.stops < L.max_stops && 4u * late >= (unsigned)span.P;
    if (atomicCAS(L.sync + 2, v, stop ? v | 1u : 2u * e) != v) continue;  // decided by another
    if (!stop) return true;
    L.progress[L.launch ^ 1] = K2Progress{span.step0 + s, span.stops + 1, 0};
    return false;
  }
}

// A place in that walk, in the order in which all roles go: phase, step of the launch, tile.
struct WalkPos {
  int i, s, i0, i1, ph;
  __device__ __forceinline__ explicit WalkPos(const TileWalk& W) : i(0), s(0), i0(0), i1(W.end_of(0)), ph(0) {
    skip_empty(W);
  }
  __device__ __forceinline__ bool done(const TileWalk& W) const { return ph >= W.phases; }
  __device__ __forceinline__ void next(const TileWalk& W) {
    if (++i < i1) return;
    i = i0;
    if (++s < W.span->steps && (W.span->P == (int)gridDim.x || s % kCheckSteps != 0 || go_on(*W.L, *W.span, s))) return;
    s = 0;
    enter(W, i1);
    skip_empty(W);
  }

 private:
  __device__ __forceinline__ void enter(const TileWalk& W, int from) {
    i = i0 = from;
    if (++ph < W.phases) i1 = W.end_of(ph);
  }
  __device__ __forceinline__ void skip_empty(const TileWalk& W) {
    while (ph < W.phases && i0 == i1) enter(W, i1);
  }
};

// The epilogue warps' loop over the CTA's tiles (see step_k2_kernel); e: share of the warp
// among the kWQ of its lane quarter.
template <int D, typename Done>
__device__ __forceinline__ bool epilogue(const TileWalk& W, const K2Launch& L, RunC<D>* rc, const uint64_t* acc_full,
                                         volatile int* abort, uint32_t lane_base, int e, Done done) {
  constexpr int kSlots = RunC<D>::kSlots;
  // The loads of x run one piece ahead, into the next tile's first piece at the end of a tile
  // (with its first run constants).  The split of a unit's first piece waits for the second,
  // so that both go out as one 16-byte row: 8-byte stores to half rows cost 9 % of a step at
  // N = 1000, D = 4.
  const int lane = threadIdx.x & 31, q = (threadIdx.x >> 5) & 3;
  float xn[D][kPiece];
  uint64_t key_n = 0;
  int64_t koff_n = 0;
  float ar_n = 0.f;
  bool ahead = false;  // xn and key_n.. hold the coming tile's first pieces and runs
  // the units of the warp in tile i of the list: e' + kWQ ui, ui < nu; the shares go round
  // with the tile, so that uneven ones (RT = 24: 3 units) even out over a list
  auto first_unit = [&](int i) { return (e + W.index(i)) % kWQ; };
  auto n_units = [&](const K2Desc& d, int e0) { return max(0, (d.RT / kUnit - e0 + kWQ - 1) / kWQ); };
  // global loads of the run constants of slot `lane` from unit ui on
  auto fetch_run = [&](const K2Desc& d, int ct, int e0, int nu, int ui) {
    const int u = ui + lane / kUnit;
    if (lane < kSlots && u < nu) {
      const int r = min(ct * d.RT + kUnit * (e0 + kWQ * u) + lane % kUnit, d.n_runs - 1);
      key_n = __ldg(d.seeds + r);
      koff_n = __ldg(d.koff + r);
      ar_n = __ldg(d.ar + r);
    }
  };
  uint32_t it = 0;
  for (WalkPos at(W); !at.done(W); ++it) {
    const int i = at.i;
    const int64_t step = W.span->step0 + at.s;
    at.next(W);  // the tile after this one
    const K2Tile tile = W.tile(i);
    const K2Desc& d = W.desc(i, tile);
    const int e0 = first_unit(i), nu = n_units(d, e0);
    EpiTile w;
    w.Xm = d.Xm;
    w.KP = d.KP;
    w.n_runs = d.n_runs;
    w.RT = d.RT;
    w.run0 = tile.ct * d.RT;
    w.p = tile.mt * 128 + q * 32 + lane;
    w.live = w.p < d.N;
    w.gdt = d.gdt;
    w.kdt = d.kdt;
    w.edt = d.edt;
    w.nl2 = d.neg2ln2s2;
    w.acc = lane_base + (it & 1u) * (uint32_t)kAccCols;
    w.mp = (uint64_t)kPhiloxM0 * (D <= 2 ? (uint32_t)w.p / (4u / (D <= 2 ? D : 4)) : (uint32_t)w.p);
    const uint32_t BB = b_block_bytes(d.n), BL = b_lo_bytes(d.n, d.lo8);
    const bool lo8 = d.lo8 != 0;
    // this thread's spin (row k = p of the next step's B) in its hi and lo blocks
    uint8_t* hi_row = d.Xt + (size_t)((step + 1) & 1) * d.buf_bytes;
    uint8_t* lo_row = hi_row + (size_t)d.CT * d.KC * BB;
    const size_t blk = (size_t)tile.ct * d.KC + (w.p / kKc);
    const size_t row_in = (size_t)((w.p % kKc) >> 3) * kCoreK + (size_t)(w.p & 7) * 16u;
    hi_row += blk * BB + row_in;
    lo_row += blk * BL + row_in;
    const int64_t k = d.k0 + step;
    // run constants of the warp's units ui .. into its slots, from key_n, koff_n and ar_n
    auto stage = [&](int ui) {
      __syncwarp();
      if (lane < kSlots && ui + lane / kUnit < nu) {
        const int64_t kl = k - koff_n;
        float ramp = 1.f;
        if (d.sched_kind == 1 && kl >= d.k_anneal)
          ramp = kl >= d.k_total ? 0.f : fmaxf(0.f, 1.f - (float)(kl - d.k_anneal) * d.inv_ramp);
        const uint32_t k0 = (uint32_t)key_n, k1 = (uint32_t)(key_n >> 32);
        RunC<D>& o = rc[lane];
#pragma unroll
        for (int b = 0; b < (D + 3) / 4; ++b)
          o.r12[b] = run_rounds12((uint32_t)b, (uint32_t)kl, (uint32_t)((uint64_t)kl >> 32), k0, k1);
#pragma unroll
        for (int r = 0; r < 4; ++r) {  // Weyl key schedule: round j (0-based) uses key + j (W0, W1)
          const uint32_t j = 2u * r + 2u;
          o.rk[r] = make_uint4(k0 + j * kPhiloxW0, k1 + j * kPhiloxW1, k0 + (j + 1u) * kPhiloxW0,
                               k1 + (j + 1u) * kPhiloxW1);
        }
        o.ar = ar_n;
        o.erp = w.edt * ramp;
      }
      __syncwarp();
    };
    auto x_of = [&](int run) { return w.Xm + (size_t)run * D * w.KP + w.p; };
    if (nu > 0) {
      const int run = w.run0 + kUnit * e0;
      if (!ahead) load_piece<D>(x_of(run), w.KP, w.n_runs - run, w.live, xn);
      if (!ahead) fetch_run(d, tile.ct, e0, nu, 0);
      stage(0);
    }
    ahead = false;
    const uint32_t bar = smem_addr(acc_full + (it & 1u));
    if (!__all_sync(0xffffffffu, mbar_wait(bar, (it >> 1) & 1u, L.wait_ns) && !*abort)) return false;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
    for (int ui = 0; ui < nu; ++ui) {
      if (ui > 0 && ui % (kSlots / kUnit) == 0) {
        fetch_run(d, tile.ct, e0, nu, ui);
        stage(ui);
      }
      const int u = e0 + kWQ * ui;
      uint32_t hs[D][kPiece / 2], ls[D][kPiece / 2];  // the split that waits
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int run = w.run0 + kUnit * u + kPiece * h;
        float x[D][kPiece];
#pragma unroll
        for (int mu = 0; mu < D; ++mu)
#pragma unroll
          for (int j = 0; j < kPiece; ++j) x[mu][j] = xn[mu][j];
        if (h == 0 || ui + 1 < nu) {
          const int nx = h == 0 ? run + kPiece : w.run0 + kUnit * (u + kWQ);
          load_piece<D>(x_of(nx), w.KP, w.n_runs - nx, w.live, xn);
        } else if (!at.done(W)) {  // the next tile's first piece and run constants
          const int i2 = at.i;
          const K2Tile t2 = W.tile(i2);
          const K2Desc& d2 = W.desc(i2, t2);
          const int f2 = first_unit(i2), nu2 = n_units(d2, f2);
          if (nu2 > 0) {
            const int nx = t2.ct * d2.RT + kUnit * f2, p2 = t2.mt * 128 + q * 32 + lane;
            load_piece<D>(d2.Xm + (size_t)nx * D * d2.KP + p2, d2.KP, d2.n_runs - nx, p2 < d2.N, xn);
            fetch_run(d2, t2.ct, f2, nu2, 0);
            ahead = true;
          }
        }
        advance_piece<D>(w, rc + kUnit * (ui % (kSlots / kUnit)) + kPiece * h, run,
                         (uint32_t)(kUnit * u + kPiece * h), x);
#pragma unroll
        for (int mu = 0; mu < D; ++mu) {
          uint32_t hv[kPiece / 2], lv[kPiece / 2];
          if (lo8) split_piece8<kPiece>(x[mu], hv, lv);
          else split_piece<kPiece>(x[mu], hv, lv);
          const int col = mu * w.RT + kUnit * u;
          uint8_t* hd = hi_row + (size_t)(col >> 3) * kCoreMN;  // a row of the unit's 8 columns
          uint8_t* ld = lo8 ? lo_row + (size_t)(col >> 4) * kCoreMN + (size_t)(col & 15)
                            : lo_row + (size_t)(col >> 3) * kCoreMN;
          if (h == 0) {
#pragma unroll
            for (int j = 0; j < kPiece / 2; ++j) {
              hs[mu][j] = hv[j];
              ls[mu][j] = lv[j];
            }
          } else {
            *reinterpret_cast<uint4*>(hd) = make_uint4(hs[mu][0], hs[mu][1], hv[0], hv[1]);
            if (lo8) *reinterpret_cast<uint2*>(ld) = make_uint2(ls[mu][0], lv[0]);
            else *reinterpret_cast<uint4*>(ld) = make_uint4(ls[mu][0], ls[mu][1], lv[0], lv[1]);
          }
        }
      }
    }
    done(it);
  }
  return true;
}

template <int D>
__global__ void __launch_bounds__(kThreads, 1) step_k2_kernel(K2Launch L) {
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ __align__(8) uint64_t full_bar[kMaxStages], empty_bar[kMaxStages];
  __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2], stored[2], drain_bar;
  __shared__ uint32_t s_tmem, s_cleared;
  __shared__ int s_rank;
  __shared__ K2Span s_span;
  __shared__ volatile int s_abort;
  __shared__ RunC<D> s_runc[kEpiWarps][RunC<D>::kSlots];
  __shared__ K2Desc s_desc[kTileCache];

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int S = L.stages;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_addr(&s_tmem)), "r"(2 * kAccCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 32) {
    s_abort = 0;
    s_cleared = 0;
    for (int s = 0; s < S; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&full_bar[s])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&empty_bar[s])));
    }
    for (int b = 0; b < 2; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&acc_full[b])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(&acc_empty[b])),
                   "r"(kEpiWarps + 1));  // and the publisher
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(&stored[b])), "r"(kEpiWarps));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&drain_bar)));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid == 64) {  // count this CTA in; the first one closes the count
    const K2Progress begin = L.progress[L.launch];
    const unsigned old = atomicAdd(L.sync, 1u);
    int P = 0;
    if (begin.step >= L.total) {  // earlier launches have taken all steps
      if (old == 0) L.progress[L.launch ^ 1] = begin;
    } else if (!(old & kFrozen)) {
      if (old == 0) {
        counter_wait(L.sync, gridDim.x, kJoinNs);
        P = (int)(atomicOr(L.sync, kFrozen) & ~kFrozen);
        L.progress[L.launch ^ 1] =
            K2Progress{begin.step + min((int64_t)kLaunchSteps, L.total - begin.step), begin.stops, 0};
        __threadfence();
        atomicExch(L.sync + 1, (unsigned)P);
      } else if (counter_wait(L.sync + 1, 1u, L.wait_ns)) {
        P = (int)ld_acquire(L.sync + 1);
      } else {
        atomicOr(L.status, STATUS_TIMEOUT);
      }
    }
    s_rank = (int)old;
    // P = 0: too late (or timed out), nothing to do
    s_span = K2Span{begin.step, (int)min((int64_t)kLaunchSteps, L.total - begin.step), begin.stops, P};
  }
  __syncthreads();
  const int P = s_span.P, rank = s_rank;
  // all present: this CTA's own list; else the table is dealt out round the present ones
  TileWalk W{0, 1, 0, 1, &s_span, nullptr, &L, s_desc};
  if (P == (int)gridDim.x) {
    W.base = L.cta_begin[rank];
    W.count = L.cta_begin[rank + 1] - W.base;
    W.phases = L.phases;
    W.phase_end = L.phase_end + (size_t)rank * L.phases;
  } else if (P > 0) {
    W.base = rank;
    W.stride = P;
    W.count = (L.n_tiles - rank + P - 1) / P;
  }
  {  // descriptors of the first tiles, word by word
    constexpr int kWords = sizeof(K2Desc) / 4;
    static_assert(sizeof(K2Desc) % 4 == 0, "copied by words");
    for (int i = tid; i < min(W.count, kTileCache) * kWords; i += kThreads)
      reinterpret_cast<uint32_t*>(s_desc)[i] =
          reinterpret_cast<const uint32_t*>(L.descs + L.tiles[W.index(i / kWords)].desc)[i % kWords];
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = s_tmem;
  auto give_up = [&]() {
    atomicOr(L.status, STATUS_TIMEOUT);
    s_abort = 1;
  };

  if (W.count == 0) {
    // too late: the CTAs present do this one's tiles
  } else if (warp < kEpiWarp0) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kHelperRegs));
    if (warp == 0) {
      // ---------------- producer ----------------
      if (lane == 0) {
        uint32_t s = 0, ph = 1, g = 0, it = 0;  // stage, parity of its empty barrier, uses, tiles
        bool ok = true;
        for (WalkPos at(W); ok && !at.done(W); at.next(W), ++it) {
          const int i = at.i, st = at.s;
          const K2Tile tile = W.tile(i);
          const K2Desc& d = W.desc(i, tile);
          // the tile's constants in registers (the loop's asm statements clobber memory)
          const int KC = d.KC, terms = d.a_terms, lo8 = d.lo8;
          const uint32_t BB = b_block_bytes(d.n), BL = b_lo_bytes(d.n, lo8);
          const uint32_t bytes = stage_bytes(d.n, terms, lo8);
          const uint32_t a2 = terms > 1 ? kABlock : lo8 ? kA8Block : 0u;  // second A term
          const uint8_t* a_src = d.Aimg + (size_t)tile.mt * KC * kABlock;       // term 0, K chunk 0
          const size_t a_term = (size_t)d.MT * KC * kABlock;                    // to the second term
          const uint8_t* a2_src = d.Aimg + a_term + (size_t)tile.mt * KC * a2;
          const uint8_t* bx = d.Xt + (size_t)((W.span->step0 + st) & 1) * d.buf_bytes;
          const uint8_t* b_src = bx + (size_t)tile.ct * KC * BB;
          const uint8_t* bl_src = bx + (size_t)d.CT * KC * BB + (size_t)tile.ct * KC * BL;
          // the scout has cleared this tile
          uint64_t t0 = 0;
          for (uint32_t n = 0; (int32_t)(ld_acquire_cta(smem_addr(&s_cleared)) - it) <= 0; ++n) {
            const uint64_t t = global_timer();
            if (n == 0) t0 = t;
            if (s_abort || t - t0 > L.wait_ns) {
              ok = false;
              break;
            }
          }
          for (int kc = 0; kc < KC && ok; ++kc, ++g, a_src += kABlock, a2_src += a2, b_src += BB, bl_src += BL) {
            if (g >= (uint32_t)S && !mbar_wait(smem_addr(&empty_bar[s]), ph, L.wait_ns)) {
              ok = false;
              break;
            }
            const uint32_t base = smem_addr(smem) + s * L.stage_stride;
            const uint32_t fb = smem_addr(&full_bar[s]);
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "r"(bytes)
                         : "memory");
            bulk_g2s(base, a_src, kABlock, fb);
            if (a2) bulk_g2s(base + kABlock, a2_src, a2, fb);
            const uint32_t bb = base + kABlock + a2;
            bulk_g2s(bb, b_src, BB, fb);
            bulk_g2s(bb + BB, bl_src, BL, fb);
            if (++s == (uint32_t)S) {
              s = 0;
              ph ^= 1u;
            }
          }
          if (s_abort) break;
        }
        if (!ok) give_up();
        // drain: every copy issued must have landed before the CTA may exit
        const uint32_t first = g > (uint32_t)S ? g - (uint32_t)S : 0u;
        for (uint32_t u = first; u < g; ++u)
          if (!mbar_wait(smem_addr(&full_bar[u % S]), (u / S) & 1u, L.wait_ns)) atomicOr(L.status, STATUS_TIMEOUT);
      }
    } else if (warp == 1) {
      // ---------------- MMA issuer (the whole warp, see mma_bf16) ----------------
      uint32_t s = 0, ph = 0, it = 0;  // ring stage and its phase, tiles
      bool ok = true;
      for (WalkPos at(W); ok && !at.done(W); at.next(W), ++it) {
        const int i = at.i;
        const K2Tile tile = W.tile(i);
        const K2Desc& d = W.desc(i, tile);
        const uint32_t n = (uint32_t)d.n, BB = b_block_bytes(d.n);
        const uint32_t b = it & 1u, use = it >> 1;
        // kind::f16, FP32 accumulator, BF16 A (K-major) and B (MN-major), N = n, M = 128
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((n >> 3) << 17) |
                               ((uint32_t)(128 >> 4) << 24);
        // FP8 mode: e4m3 J (K-major, 8 x 16-byte cores, 256 bytes between row groups) and
        // e4m3 lo (MN-major, 16 columns a core row, 512 bytes between column groups)
        const uint32_t idesc8 = (1u << 4) | (1u << 16) | ((n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        const uint32_t acc = tmem + b * (uint32_t)kAccCols;
        const bool real_j = d.a_terms > 1, lo8 = d.lo8 != 0;
        const bool stall = d.stall != 0;
        const uint32_t a2 = real_j ? kABlock : lo8 ? kA8Block : 0u;
        // a stage and a K step move only the start-address field (shared addresses stay below
        // 256 KB, so the field never carries)
        const uint64_t d0 = smem_desc(smem_addr(smem), kCoreK, kCoreMN), d80 = smem_desc(smem_addr(smem), kCoreK, 256u);
        const uint64_t o_bhi = (kABlock + a2) >> 4, o_blo = o_bhi + (BB >> 4), o_alo = kABlock >> 4;
        constexpr uint64_t kStep = 2u * kCoreK >> 4;
        const int KC = d.KC;
        // (voted on, like every wait of a warp that goes on together)
        if (use > 0 && !__all_sync(0xffffffffu, mbar_wait(smem_addr(&acc_empty[b]), (use - 1u) & 1u, L.wait_ns) && !s_abort)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        for (int kc = 0; kc < KC; ++kc) {
          if (!__all_sync(0xffffffffu, mbar_wait(smem_addr(&full_bar[s]), ph, L.wait_ns) && !s_abort)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t off = (uint64_t)(s * (L.stage_stride >> 4));
          const uint64_t a = d0 + off;
          const uint32_t acc0 = kc > 0 ? 1u : 0u;
          static_assert(kKc == 32, "two BF16 K steps per chunk");
          mma_bf16(acc, a, a + o_bhi, idesc, acc0);
          if (lo8) {
            mma_bf16(acc, a + kStep, a + o_bhi + kStep, idesc, 1u);
            mma_f8(acc, d80 + off + o_alo, a + o_blo, idesc8);
          } else {
            mma_bf16(acc, a, a + o_blo, idesc, 1u);
            if (real_j) mma_bf16(acc, a + o_alo, a + o_bhi, idesc, 1u);
            mma_bf16(acc, a + kStep, a + o_bhi + kStep, idesc, 1u);
            mma_bf16(acc, a + kStep, a + o_blo + kStep, idesc, 1u);
            if (real_j) mma_bf16(acc, a + o_alo + kStep, a + o_bhi + kStep, idesc, 1u);
          }
          mma_commit(smem_addr(&empty_bar[s]));
          if (++s == (uint32_t)S) {
            s = 0;
            ph ^= 1u;
          }
        }
        // (test of the timeout path: the signal is withheld, so the epilogue's wait runs
        // out; the drain below still waits for every product issued)
        if (ok && !stall) mma_commit(smem_addr(&acc_full[b]));
      }
      if (!ok && lane == 0) give_up();
      // every product issued must be complete before TMEM is freed
      mma_commit(smem_addr(&drain_bar));
      if (!mbar_wait(smem_addr(&drain_bar), 0u, L.wait_ns) && lane == 0) atomicOr(L.status, STATUS_TIMEOUT);
    } else if (warp == kPubWarp) {
      // ---------------- publisher ----------------
      if (lane == 0) {
        uint32_t it = 0;
        bool ok = true;
        for (WalkPos at(W); ok && !at.done(W); at.next(W), ++it) {
          const int i = at.i;
          const K2Tile tile = W.tile(i);
          unsigned* done = L.flags + W.desc(i, tile).flag0 + tile.ct;
          ok = mbar_wait(smem_addr(&stored[it & 1u]), (it >> 1) & 1u, L.wait_ns) && !s_abort;
          if (!ok) break;
          // seen: only now may the tile after next take this accumulator and complete its
          // `stored` once more (a parity tells the last phase from the one under way, no more;
          // a publisher two tiles late would wait for a phase that never comes).  Behind the
          // publication, 2 us later, it costs 1 % where a CTA has few short tiles
          asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&acc_empty[it & 1u])) : "memory");
          fence_proxy_async();  // the epilogue's stores (generic proxy) before other SMs' TMA reads
          asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(done), "r"(1u) : "memory");
        }
        if (!ok) give_up();
      }
    } else {
      // ---------------- scout ----------------
      if (lane == 0) {
        uint32_t it = 0;
        bool ok = true;
        for (WalkPos at(W); ok && !at.done(W); at.next(W)) {
          const int i = at.i, st = at.s;
          const K2Tile tile = W.tile(i);
          const K2Desc& d = W.desc(i, tile);
          // every M tile of the column tile has finished the steps before this one
          ok = counter_wait(L.flags + d.flag0 + tile.ct, (unsigned)d.MT * (unsigned)st, L.wait_ns) && !s_abort;
          if (!ok) break;
          fence_proxy_async();  // their stores before this CTA's TMA reads
          st_release_cta(smem_addr(&s_cleared), ++it);
        }
        if (!ok) give_up();
      }
    }
  } else {
    // ---------------- epilogue: 4 kWQ warps ----------------
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kEpiRegs));
    const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const bool ok = epilogue<D>(W, L, s_runc[warp - kEpiWarp0], acc_full, &s_abort, lane_base, (warp - kEpiWarp0) >> 2, [&](uint32_t it) {
      // The tile's stores may be published and its accumulator overwritten.  A warp may be a
      // tile ahead of another, so each accumulator has its own `stored`; it arrives there first,
      // so that two tiles ahead, behind acc_empty, every warp has.
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) {
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&stored[it & 1u])) : "memory");
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&acc_empty[it & 1u])) : "memory");
      }
    });
    if (!ok && lane == 0) give_up();
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * kAccCols));
  }
}

// X[run][p][mu] (float) -> Xm[c][p] and the hi/lo blocks of buffer 0, padding spins and runs
// (up to the column tiles' last) included; buffer 1 is written whole by the first step.
// Thread = (spin, component) of one unit of 8 runs, unit0 + blockIdx.y: coalesced reads, one
// 16-byte row of each block.  (Per element, with 2-byte stores after a memset of both
// buffers: 201 us for 8192 runs of N = 1000, D = 4.)
template <int D>
__global__ void __launch_bounds__(256) k2_pack_kernel(const float* __restrict__ X, float* __restrict__ Xm,
                                                      uint8_t* __restrict__ Xt, int N, int KP, int KC, int CT, int RT,
                                                      int n_runs, int lo8, int unit0) {
  const int e = blockIdx.x * 256 + threadIdx.x;
  if (e >= KP * D) return;
  const int p = e / D, mu = e % D, run0 = (unit0 + blockIdx.y) * kUnit;
  const int n = D * RT, ct = run0 / RT, col = mu * RT + run0 % RT;
  const size_t BB = b_block_bytes(n), BL = b_lo_bytes(n, lo8);
  float v[kUnit];
#pragma unroll
  for (int j = 0; j < kUnit; ++j) {
    v[j] = p < N && run0 + j < n_runs ? X[((size_t)(run0 + j) * N) * D + e] : 0.f;
    if (run0 + j < n_runs) Xm[((size_t)(run0 + j) * D + mu) * KP + p] = v[j];
  }
  const size_t row_in = (size_t)((p % kKc) >> 3) * kCoreK + (size_t)(p & 7) * 16, blk = (size_t)ct * KC + p / kKc;
  uint8_t* hi = Xt + blk * BB + (size_t)(col >> 3) * kCoreMN + row_in;
  uint8_t* lo = Xt + (size_t)CT * KC * BB + blk * BL + row_in;
  const float (&v0)[kPiece] = *reinterpret_cast<const float (*)[kPiece]>(v);
  const float (&v1)[kPiece] = *reinterpret_cast<const float (*)[kPiece]>(v + kPiece);
  uint32_t h0[2], l0[2], h1[2], l1[2];
  if (lo8) {  // both halves scaled by 2^kLoScaleLog2, lo in e4m3
    split_piece8<kPiece>(v0, h0, l0);
    split_piece8<kPiece>(v1, h1, l1);
    *reinterpret_cast<uint2*>(lo + (size_t)(col >> 4) * kCoreMN + (size_t)(col & 15)) = make_uint2(l0[0], l1[0]);
  } else {
    split_piece<kPiece>(v0, h0, l0);
    split_piece<kPiece>(v1, h1, l1);
    *reinterpret_cast<uint4*>(lo + (size_t)(col >> 3) * kCoreMN) = make_uint4(l0[0], l0[1], l1[0], l1[1]);
  }
  *reinterpret_cast<uint4*>(hi) = make_uint4(h0[0], h0[1], h1[0], h1[1]);
}

// Xm[c][p] -> X[run][p][mu]; blockIdx.y = run.
template <int D>
__global__ void __launch_bounds__(256) k2_unpack_kernel(const float* __restrict__ Xm, float* __restrict__ X, int N,
                                                        int KP) {
  const size_t run = blockIdx.y;
  const int e = blockIdx.x * 256 + threadIdx.x;
  if (e < N * D) X[run * N * D + e] = Xm[(run * D + e % D) * KP + e / D];
}

// per-run constant 1 + dt (h - 1)
__global__ void k2_runconst_kernel(const double* __restrict__ h, const int32_t* __restrict__ hidx,
                                   int n_runs, double dt, float* ar) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n_runs; r += gridDim.x * blockDim.x)
    ar[r] = (float)(1.0 + dt * (h[hidx[r]] - 1.0));
}

// A-operand blocks of J: hi = bf16(J) and, for real couplings, lo = bf16(J - hi).
__global__ void k2_aimg_kernel(const double* __restrict__ J, int N, int MT, int KC, int terms,
                               __nv_bfloat16* __restrict__ img) {
  const int KP = MT * 128;
  const size_t total = (size_t)KP * KP;
  const size_t per_term = (size_t)MT * KC * 128 * kKc;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x) {
    const int m = (int)(e / KP), k = (int)(e % KP);
    const double v = (m < N && k < N) ? J[(size_t)m * N + k] : 0.0;
    const __nv_bfloat16 hi = __float2bfloat16_rn((float)v);
    const int mt = m / 128, r = m % 128, kc = k / kKc, kk = k % kKc;
    const size_t off = ((size_t)mt * KC + kc) * (128 * kKc) + (size_t)(r / 8) * (kCoreMN / 2) +
                       (size_t)(kk / 8) * (kCoreK / 2) + (r % 8) * 8 + (kk % 8);  // in elements
    img[off] = hi;
    if (terms > 1) {
      img[per_term + off] = __float2bfloat16_rn((float)(v - (double)__bfloat162float(hi)));
    } else {  // +-1 couplings: J in e4m3 (exact) after the BF16 blocks, K-major 8 x 16-byte cores
      uint8_t* img8 = reinterpret_cast<uint8_t*>(img + per_term);
      const size_t off8 = ((size_t)mt * KC + kc) * kA8Block + (size_t)(r / 8) * 256 + (size_t)(kk / 16) * 128 +
                          (r % 8) * 16 + (kk % 16);
      img8[off8] = (uint8_t)__nv_cvt_float_to_fp8((float)v, __NV_SATFINITE, __NV_E4M3);
    }
  }
}

// Runs per column tile of a context: the most for its D (or the autotuner's choice
// `want`), shrunk (in multiples of 32) for contexts with fewer runs so that small
// instances waste no columns.
int k2_rt(int D, int n_runs, int want = 0) {
  const int r32 = (n_runs + 31) / 32 * 32;
  const int top = want > 0 && k2_rt_valid(D, want) ? want : k2_rt_max(D);
  return std::min(top, std::max(32, r32));
}

// Time of a tile in the planner's units (ns): the ring's feed against the epilogue, which
// overlap.  95 bytes a ns of feed were measured with the epilogue emptied, and per run and D
// the epilogue's share of full steps (N = 1000; D = 2 costs as much noise as D = 4, its blocks
// serving two spins); the constant is the hand-over between them.
double k2_tile_ns(int N, int D, int RT, int a_terms, int lo8) {
  constexpr double run_ns[9] = {0, 150, 160, 240, 250, 400, 450, 560, 620};
  const int KC = (N + 127) / 128 * 128 / kKc;
  const double feed = KC * (double)stage_bytes(D * RT, a_terms, lo8) / 95.0, epi = run_ns[D] * RT;
  return std::max(feed, epi) + 0.3 * std::min(feed, epi) + 1000.0;
}

}  // namespace

// Runs per column tile of every context of a call on `ctas` CTAs.  While the tiles do not
// fill the CTAs, the costliest tile's context takes column tiles of half the runs: with
// fewer tiles than SMs a step lasts as long as its costliest tile (N = 250, D = 3, 1024
// runs: 32 tiles of 64 runs, 128 of 16).  Below 16 runs a tile's J blocks outweigh its
// columns.  A context whose tile width was chosen (want) keeps it.
std::vector<int> k2_pick_rt(const std::vector<K2Shape>& shapes, int ctas) {
  std::vector<int> rt;
  long long tiles = 0;
  auto count = [&](const K2Shape& s, int r) {
    return (long long)((s.N + 127) / 128) * ((s.n_runs + r - 1) / r);
  };
  for (const K2Shape& s : shapes) {
    rt.push_back(k2_rt(s.D, s.n_runs, s.want));
    tiles += count(s, rt.back());
  }
  for (;;) {
    int best = -1;
    double cost = 0.0;
    for (size_t i = 0; i < shapes.size(); ++i) {
      const K2Shape& s = shapes[i];
      // whole 4-run blocks for the two warps of a lane quarter, n = D RT a multiple of 16
      const int half = rt[i] / 2;
      if (s.want > 0 || half < 16 || rt[i] % 16 || s.D * half % 16) continue;
      const double c = k2_tile_ns(s.N, s.D, rt[i], s.a_terms, s.lo8);
      if (c > cost) {
        cost = c;
        best = (int)i;
      }
    }
    if (best < 0) return rt;
    const int half = rt[best] / 2;
    const long long more = count(shapes[best], half) - count(shapes[best], rt[best]);
    if (tiles + more > ctas) return rt;
    rt[best] = half;
    tiles += more;
  }
}

int k2_max_stages(int D, int rt, int n_runs, int a_terms, int lo8) {
  const int n = D * k2_rt(D, n_runs, rt);
  const uint32_t stride = (stage_bytes(n, a_terms, lo8) + 1023u) / 1024u * 1024u;
  return (int)std::min<size_t>(kMaxStages, std::max<size_t>(2, kRingBudget / stride));
}

long long k2_work_units(int N, int D, int n_runs, int rt) {
  if (D < 1 || D > 8) return 0;
  const long long MT = (N + 127) / 128, K64 = 2 * MT;  // K in units of 64 spins
  const int RT = k2_rt(D, n_runs, rt);
  const long long CT = (n_runs + RT - 1) / RT;
  return MT * CT * K64 * (long long)(D * RT) / 128;  // in 128-column tile units
}

// A-operand blocks of J (and of its BF16 residual for real couplings), built on
// the device from the FP64 copy of J.
cudaError_t prepare_k2_operand(chym_ctx* c) {
  if (c->d_Ak2) return cudaSuccess;
  const int N = c->N, MT = (N + 127) / 128, KP = MT * 128, KC = KP / kKc;
  const int terms = c->kind == CHYM_J_PM1 ? 1 : 2;
  // real J: J and its BF16 residual; +-1 J: J in BF16 and in e4m3 (FP8 mode)
  const size_t bytes = (size_t)MT * KC * (kABlock + (terms > 1 ? kABlock : kA8Block));
  cudaError_t e = cudaMalloc(&c->d_Ak2, bytes);
  if (e != cudaSuccess) return e;
  k2_aimg_kernel<<<152 * 8, 256>>>(c->d_J64, N, MT, KC, terms, (__nv_bfloat16*)c->d_Ak2);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return cudaDeviceSynchronize();
}

// ---------------------------------------------------------------------------
// Runner: a set of large-N contexts integrated together for `steps` steps.
// ---------------------------------------------------------------------------
// f(std::integral_constant<int, D>()) for the D of a context.
template <typename F>
void with_dim(int D, F f) {
  switch (D) {
    case 1: f(std::integral_constant<int, 1>()); break;
    case 2: f(std::integral_constant<int, 2>()); break;
    case 3: f(std::integral_constant<int, 3>()); break;
    case 4: f(std::integral_constant<int, 4>()); break;
    case 5: f(std::integral_constant<int, 5>()); break;
    case 6: f(std::integral_constant<int, 6>()); break;
    case 7: f(std::integral_constant<int, 7>()); break;
    case 8: f(std::integral_constant<int, 8>()); break;
  }
}

// Workspace, per-run constants and buffer 0 of one context; fills its descriptor.
cudaError_t k2_prepare(chym_ctx* c, const StepConsts& sc, cudaStream_t st, void* desc_out, int RT) {
  cudaError_t e = prepare_k2_operand(c);
  if (e != cudaSuccess) return e;
  K2Desc& d = *reinterpret_cast<K2Desc*>(desc_out);
  const int N = c->N, D = c->D, MT = (N + 127) / 128, KP = MT * 128, KC = KP / kKc;
  const int n = D * RT;
  const int CT = (sc.n_runs + RT - 1) / RT;
  const int lo8 = sc.fp8 && c->kind == CHYM_J_PM1 ? 1 : 0;
  const size_t BB = b_block_bytes(n), BL = b_lo_bytes(n, lo8);
  const size_t xm_bytes = ((size_t)sc.n_runs * D * KP * 4 + 255) / 256 * 256;
  const size_t buf_bytes = ((size_t)CT * KC * (BB + BL) + 255) / 256 * 256;
  const size_t xt_bytes = 2 * buf_bytes;
  const size_t ar_bytes = ((size_t)sc.n_runs * 4 + 255) / 256 * 256;
  const size_t need = xm_bytes + xt_bytes + ar_bytes;
  if (need > c->k2_ws_bytes) {
    if (c->d_k2_ws) cudaFree(c->d_k2_ws);
    c->d_k2_ws = nullptr;
    c->k2_ws_bytes = 0;
    e = cudaMalloc(&c->d_k2_ws, need);
    if (e != cudaSuccess) return e;
    c->k2_ws_bytes = need;
  }
  uint8_t* ws = (uint8_t*)c->d_k2_ws;
  float* Xm = (float*)ws;
  uint8_t* Xt = ws + xm_bytes;
  float* ar = (float*)(Xt + xt_bytes);
  k2_runconst_kernel<<<(sc.n_runs + 255) / 256, 256, 0, st>>>(c->d_h, c->d_hidx, sc.n_runs, sc.dt, ar);
  with_dim(D, [&](auto dim) {
    constexpr int kD = decltype(dim)::value;
    const int units = CT * RT / kUnit;
    for (int u0 = 0; u0 < units; u0 += kMaxGridY) {
      const dim3 grid((unsigned)((KP * kD + 255) / 256), (unsigned)std::min(kMaxGridY, units - u0));
      k2_pack_kernel<kD><<<grid, 256, 0, st>>>((const float*)c->d_X, Xm, Xt, N, KP, KC, CT, RT, sc.n_runs, lo8, u0);
    }
  });
  d.D = D;
  d.flag0 = 0;  // set by k2_integrate
  d.Aimg = (const uint8_t*)c->d_Ak2;
  d.Xm = Xm;
  d.Xt = Xt;
  d.ar = ar;
  d.seeds = c->d_seeds;
  d.koff = c->d_koff;
  d.buf_bytes = (unsigned long long)buf_bytes;
  d.N = N;
  d.KP = KP;
  d.MT = MT;
  d.KC = KC;
  d.CT = CT;
  d.RT = RT;
  d.n = n;
  d.n_runs = sc.n_runs;
  d.a_terms = c->kind == CHYM_J_PM1 ? 1 : 2;
  d.lo8 = lo8;
  d.stall = sc.test_stall;
  d.sched_kind = sc.sched_kind;
  d.k0 = sc.k0;
  d.k_anneal = sc.k_anneal;
  d.k_total = sc.k_total;
  d.gdt = (float)(sc.dt * sc.gamma);
  d.kdt = (float)(sc.dt * sc.kappa);
  // FP8 mode: the accumulator holds 2^kLoScaleLog2 y (both operand halves carry it)
  d.edt = (float)(sc.dt * sc.eps / (lo8 ? (double)(1u << kLoScaleLog2) : 1.0));
  d.neg2ln2s2 = (float)(-2.0 * 0.69314718055994531 * sc.noise_scale * sc.noise_scale);
  d.inv_ramp = sc.sched_kind == 1 ? (float)(1.0 / (double)(sc.k_total - sc.k_anneal)) : 0.f;
  return cudaGetLastError();
}

size_t k2_desc_bytes() { return sizeof(K2Desc); }

cudaError_t k2_finish(chym_ctx* c, const void* desc, cudaStream_t st) {
  const K2Desc& d = *reinterpret_cast<const K2Desc*>(desc);
  with_dim(c->D, [&](auto dim) {
    constexpr int kD = decltype(dim)::value;
    for (int r0 = 0; r0 < d.n_runs; r0 += kMaxGridY) {
      const dim3 grid((unsigned)((c->N * kD + 255) / 256), (unsigned)std::min(kMaxGridY, d.n_runs - r0));
      k2_unpack_kernel<kD><<<grid, 256, 0, st>>>(d.Xm + (size_t)r0 * kD * d.KP,
                                                 (float*)c->d_X + (size_t)r0 * c->N * kD, c->N, d.KP);
    }
  });
  return cudaGetLastError();
}

namespace {

cudaError_t k2_launch(int D, const K2Launch& L, int grid, size_t smem, cudaStream_t st) {
  auto go = [&](auto kern) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<grid, kThreads, smem, st>>>(L);
    return cudaGetLastError();
  };
  switch (D) {
    case 1: return go(step_k2_kernel<1>);
    case 2: return go(step_k2_kernel<2>);
    case 3: return go(step_k2_kernel<3>);
    case 4: return go(step_k2_kernel<4>);
    case 5: return go(step_k2_kernel<5>);
    case 6: return go(step_k2_kernel<6>);
    case 7: return go(step_k2_kernel<7>);
    case 8: return go(step_k2_kernel<8>);
  }
  return cudaErrorInvalidValue;
}

// Column tiles [ct, ct + n) of a context.
struct K2Cols {
  int desc, ct, n;
};
using K2Phase = std::vector<K2Cols>;

// The contexts of one D: their tiles in lists per CTA, and where these sit in the device block.
struct K2Group {
  int D = 0, grid = 0, phases = 1;
  double cost = 0.0;
  size_t n_tiles = 0, o_sync = 0, n_sync = 0, o_progress = 0, o_tile = 0, o_cta = 0;
  int max_stops = 0;
  std::vector<int> descs;  // the costliest tiles first
  std::vector<std::vector<K2Tile>> lists;
  std::vector<std::vector<int>> phase_end;  // per CTA
};

// The column tiles of a group in phases of at most `rounds` tiles a CTA, each column tile in
// the first phase with room for it; the last takes up to a round more rather than leave it to
// one of its own.
template <typename Desc>
std::vector<K2Phase> k2_phases(const K2Group& g, Desc desc, int grid, size_t rounds) {
  std::vector<K2Phase> out;
  std::vector<size_t> room;
  size_t left = g.n_tiles;
  for (int i : g.descs) {
    const size_t MT = (size_t)desc(i).MT;
    size_t f = 0;
    for (int ct = 0; ct < desc(i).CT;) {
      while (f < room.size() && room[f] < MT) ++f;
      if (f == room.size()) {
        out.emplace_back();
        room.push_back(left <= (rounds + 1) * grid ? left : std::max(rounds * grid, MT));
      }
      const int n = (int)std::min<size_t>(desc(i).CT - ct, room[f] / MT);
      out[f].push_back(K2Cols{i, ct, n});
      room[f] -= n * MT;
      left -= n * MT;
      ct += n;
    }
  }
  return out;
}

// Deals a phase's tiles out to `grid` CTAs, each next one to the CTA with the least work so
// far (the lowest of equals, mt fastest); lists may be null.  Returns the longest load.
template <typename Desc>
double k2_deal(const K2Phase& phase, Desc desc, const std::vector<double>& tile_ns, int grid,
               std::vector<std::vector<K2Tile>>* lists) {
  std::vector<std::pair<double, int>> load(grid), merged(grid);
  for (int b = 0; b < grid; ++b) load[b] = {0.0, b};
  for (const K2Cols& c : phase) {
    const double ns = tile_ns[c.desc];
    const int MT = desc(c.desc).MT;
    for (long long t = 0, n = (long long)c.n * MT; t < n;) {
      // one tile each to the CTAs that stay below the least loaded one's next tile
      int m = 1;
      while (m < grid && load[m].first < load[0].first + ns) ++m;
      const long long rounds = !lists && m == grid ? std::max(1LL, (n - t) / grid) : 1;
      m = (int)std::min<long long>(m, n - t);
      for (int j = 0; j < m; ++j, ++t) {
        if (lists) (*lists)[load[j].second].push_back(K2Tile{c.desc, (int)(t % MT), c.ct + (int)(t / MT), 0});
        load[j].first += ns * rounds;
      }
      t += m * (rounds - 1);
      std::merge(load.begin(), load.begin() + m, load.begin() + m, load.end(), merged.begin());  // both sorted
      load.swap(merged);
    }
  }
  return load.back().first;
}

}  // namespace

// Integrate the contexts whose descriptors are in `descs` (host copies, dims[i] =
// their D) for `steps` steps on stream st: one persistent launch per D and kLaunchSteps
// steps.  Several D take all CTAs one after the other, or shares of them in proportion to
// their work, side by side on the runner's streams (see kBesideLoss).
cudaError_t k2_integrate(K2Runner& R, std::vector<unsigned char>& descs, const std::vector<int>& dims,
                         int64_t steps, unsigned* status, cudaStream_t st, int ctas, const int* stage_choice) {
  const size_t db = sizeof(K2Desc);
  const int n_desc = (int)dims.size();
  cudaError_t e = cudaSuccess;
  auto desc = [&](int i) -> K2Desc& { return *reinterpret_cast<K2Desc*>(descs.data() + i * db); };
  bool stall = false;  // CHYM_FLAG_TEST_STALL on any context: the short wait limit
  std::vector<double> tile_ns(n_desc);
  std::vector<K2Group> groups;
  double total = 0.0;
  for (int D = 1; D <= 8; ++D) {
    K2Group g;
    g.D = D;
    for (int i = 0; i < n_desc; ++i) {
      if (dims[i] != D) continue;
      K2Desc& d = desc(i);
      stall = stall || d.stall;
      d.flag0 = (int)g.n_sync;  // column-tile counters of the group so far
      g.n_sync += d.CT;
      tile_ns[i] = k2_tile_ns(d.N, D, d.RT, d.a_terms, d.lo8);
      g.n_tiles += (size_t)d.CT * d.MT;
      g.cost += tile_ns[i] * d.CT * d.MT;
      g.descs.push_back(i);
    }
    if (g.descs.empty()) continue;
    g.n_sync += 4;  // join words
    total += g.cost;
    groups.push_back(g);
  }
  for (K2Group& g : groups)
    std::stable_sort(g.descs.begin(), g.descs.end(), [&](int x, int y) { return tile_ns[x] > tile_ns[y]; });
  // The phases of a group on n CTAs, and the time of a step over all of them.  Each is dealt out
  // by itself: what counts is the longest load of every phase, not of the lists (dealt over the
  // lists, CTAs had 1 to 3 tiles of a phase: N = 800 above 877, N = 600 130, the uneven workload 1275).
  auto plan = [&](const K2Group& g, int n, double* ns) {
    const int grid = (int)std::min<size_t>(g.n_tiles, (size_t)n);
    const size_t rounds = (g.n_tiles + grid - 1) / grid;
    auto step = [&](const std::vector<K2Phase>& p) {
      double t = rounds == 1 ? kHandOverNs : 0.0;
      for (const K2Phase& c : p) t += k2_deal(c, desc, tile_ns, grid, nullptr);
      return t;
    };
    std::vector<K2Phase> p = k2_phases(g, desc, grid, rounds);
    *ns = step(p);
    if (steps >= kPhaseSteps && g.n_tiles >= kPhaseMin * (size_t)grid) {
      std::vector<K2Phase> q = k2_phases(g, desc, grid, kPhaseTiles);
      const double t = step(q);
      if (t < *ns * kDriftLoss) {
        p.swap(q);
        *ns = t;
      }
    }
    return p;
  };
  std::vector<int> share(groups.size(), ctas);
  std::vector<std::vector<K2Phase>> phases(groups.size());
  std::vector<double> step_ns(groups.size());
  double in_turn = 0.0;
  for (size_t gi = 0; gi < groups.size(); ++gi) {
    phases[gi] = plan(groups[gi], ctas, &step_ns[gi]);
    in_turn += step_ns[gi] + kLaunchNs / (double)std::min<int64_t>(steps, kLaunchSteps);
  }
  bool beside = false;
  if (groups.size() > 1 && ctas >= 2 * (int)groups.size()) {
    std::vector<int> part(groups.size());
    std::vector<std::vector<K2Phase>> p(groups.size());
    std::vector<double> part_ns(groups.size());
    int left = ctas;
    double longest = 0.0;
    for (size_t gi = 0; gi < groups.size(); ++gi) {
      const int others = (int)(groups.size() - gi) - 1;
      part[gi] = std::min(left - others, std::max(1, (int)(left * groups[gi].cost / total + 0.5)));
      left -= part[gi];
      total -= groups[gi].cost;
      p[gi] = plan(groups[gi], part[gi], &part_ns[gi]);
      longest = std::max(longest, part_ns[gi]);
    }
    if (longest * kBesideLoss < in_turn) {
      beside = true;
      share.swap(part);
      phases.swap(p);
      step_ns.swap(part_ns);
    }
  }
  for (size_t gi = 0; gi < groups.size(); ++gi) {
    K2Group& g = groups[gi];
    g.grid = (int)std::min<size_t>(g.n_tiles, (size_t)share[gi]);
    // a launch for each stop; one that finds nothing left to do takes 3 us
    const double call_ms = 1e-6 * step_ns[gi] * (double)steps;
    g.max_stops = (call_ms > 1.0) + (call_ms > 2.0) + (call_ms > 6.0) + (call_ms > 20.0);
    g.phases = (int)phases[gi].size();
    g.lists.resize(g.grid);
    g.phase_end.resize(g.grid);
    for (const K2Phase& p : phases[gi]) {
      k2_deal(p, desc, tile_ns, g.grid, &g.lists);
      for (int b = 0; b < g.grid; ++b) g.phase_end[b].push_back((int)g.lists[b].size());
    }
  }
  // device block: [join words | column-tile counters] of every group (zeroed per launch), then
  // descriptors, tiles and lists
  auto up16 = [](size_t x) { return (x + 15) / 16 * 16; };
  size_t at = 0;
  for (K2Group& g : groups) {
    g.o_sync = at;
    at = up16(at + sizeof(unsigned) * g.n_sync);
  }
  for (K2Group& g : groups) {  // zero: the first launch begins at step 0
    g.o_progress = at;
    at = up16(at + 2 * sizeof(K2Progress));
  }
  const size_t o_desc = at;
  at = up16(at + descs.size());
  for (K2Group& g : groups) {
    g.o_tile = at;
    g.o_cta = at + g.n_tiles * sizeof(K2Tile);
    at = up16(g.o_cta + sizeof(int) * (size_t)(g.grid + 1 + g.grid * g.phases));
  }
  if (at > R.bytes) {
    if (R.d_buf) cudaFree(R.d_buf);
    R.d_buf = nullptr;
    R.bytes = 0;
    e = cudaMalloc(&R.d_buf, at);
    if (e != cudaSuccess) return e;
    R.bytes = at;
  }
  std::vector<unsigned char> blob(at, 0);
  memcpy(blob.data() + o_desc, descs.data(), descs.size());
  for (const K2Group& g : groups) {
    K2Tile* bt = reinterpret_cast<K2Tile*>(blob.data() + g.o_tile);
    int* bc = reinterpret_cast<int*>(blob.data() + g.o_cta);
    int n = 0;
    for (int b = 0; b < g.grid; ++b) {
      bc[b] = n;
      for (const K2Tile& t : g.lists[b]) bt[n++] = t;
    }
    bc[g.grid] = n;
    for (int b = 0; b < g.grid; ++b)
      for (int ph = 0; ph < g.phases; ++ph) bc[g.grid + 1 + b * g.phases + ph] = g.phase_end[b][ph];
  }
  unsigned char* base = (unsigned char*)R.d_buf;
  e = cudaMemcpyAsync(base, blob.data(), at, cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return e;
  if (beside) {
    if (!R.fork) e = cudaEventCreateWithFlags(&R.fork, cudaEventDisableTiming);
    for (size_t gi = 1; gi < groups.size() && e == cudaSuccess; ++gi) {
      if (!R.streams[gi]) e = cudaStreamCreateWithFlags(&R.streams[gi], cudaStreamNonBlocking);
      if (e == cudaSuccess && !R.joins[gi]) e = cudaEventCreateWithFlags(&R.joins[gi], cudaEventDisableTiming);
    }
    if (e == cudaSuccess) e = cudaEventRecord(R.fork, st);
    if (e != cudaSuccess) return e;
  }
  for (size_t gi = 0; gi < groups.size(); ++gi) {
    const K2Group& g = groups[gi];
    uint32_t stride = 0;
    for (int i : g.descs) {
      const K2Desc& d = desc(i);
      stride = std::max(stride, (stage_bytes(d.n, d.a_terms, d.lo8) + 1023u) / 1024u * 1024u);
    }
    // ring depth: as many stages as the ring budget holds, or fewer when the autotuner chose so
    int stages = (int)std::min<size_t>(kMaxStages, std::max<size_t>(2, kRingBudget / stride));
    if (stage_choice && stage_choice[g.D] >= 2) stages = std::min(stages, stage_choice[g.D]);
    // at least 120 KB: one CTA (which owns 512 TMEM columns) per SM
    const size_t smem = std::max<size_t>((size_t)stages * stride, 120 * 1024);
    const bool side = beside && gi > 0;
    cudaStream_t s = side ? R.streams[gi] : st;
    if (side && (e = cudaStreamWaitEvent(s, R.fork, 0)) != cudaSuccess) return e;
    const int64_t launches = (steps + kLaunchSteps - 1) / kLaunchSteps + g.max_stops;
    for (int64_t i = 0; i < launches; ++i) {
      if (i > 0 && (e = cudaMemsetAsync(base + g.o_sync, 0, sizeof(unsigned) * g.n_sync, s)) != cudaSuccess) return e;
      K2Launch L;
      L.descs = (const K2Desc*)(base + o_desc);
      L.tiles = (const K2Tile*)(base + g.o_tile);
      L.n_tiles = (int)g.n_tiles;
      L.cta_begin = (const int*)(base + g.o_cta);
      L.phase_end = L.cta_begin + g.grid + 1;
      L.phases = g.phases;
      L.sync = (unsigned*)(base + g.o_sync);
      L.flags = L.sync + 4;
      L.progress = (K2Progress*)(base + g.o_progress);
      L.launch = (int)(i & 1);
      L.max_stops = g.max_stops;
      L.total = steps;
      L.stages = stages;
      L.stage_stride = stride;
      L.status = status;
      L.wait_ns = stall ? kTestWaitLimitNs : kWaitLimitNs;
      e = k2_launch(g.D, L, g.grid, smem, s);
      if (e != cudaSuccess) return e;
    }
    if (side) {
      e = cudaEventRecord(R.joins[gi], s);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(st, R.joins[gi], 0);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

void k2_runner_release(K2Runner& R) {
  if (R.d_buf) cudaFree(R.d_buf);
  if (R.fork) cudaEventDestroy(R.fork);
  for (int i = 0; i < 8; ++i) {
    if (R.streams[i]) cudaStreamDestroy(R.streams[i]);
    if (R.joins[i]) cudaEventDestroy(R.joins[i]);
  }
  R = K2Runner();
}

cudaError_t launch_step_k2(chym_ctx* c, const StepConsts& sc, cudaStream_t st) {
  int sms = 0;
  cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  if (e != cudaSuccess) return e;
  const int rt = k2_pick_rt({k2_shape(c, sc.fp8, sc.n_runs, 0)}, sms)[0];
  std::vector<unsigned char> desc(sizeof(K2Desc));
  e = k2_prepare(c, sc, st, desc.data(), rt);
  if (e != cudaSuccess) return e;
  e = k2_integrate(c->k2_runner, desc, std::vector<int>{c->D}, sc.steps, c->d_status, st, sms, nullptr);
  if (e != cudaSuccess) return e;
  return k2_finish(c, desc.data(), st);
}

}  // namespace chym
