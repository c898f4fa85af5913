// Batched complex FP64 products on the bf16 tensor cores, by an exact digit split.
//
// Why.  The FP64 pipe of this part gives 1.06 TFLOP/s, its bf16 tensor cores 1940 TFLOP/s
// (cuBLAS, 8192^3).  Each operand row (terms k along it) is scaled by a power of two and cut
// into seven signed digits of eight bits (Ozaki's error-free splitting, here with fixed-point
// digits and one exponent per row): x = 2^(e - 7) sum_s d_s 2^(-8 s), s = 0 .. 6, |d_s| <= 128,
// exact to 2^(e - 56).  Digits are exact in bf16, and pairs (i, j) of equal weight i + j share an
// FP32 accumulator, which is exact while the sums in it stay within 2^24.  SG_FULL keeps the 34 pairs
// with i + j <= 7 in seven accumulators, the two lowest weights sharing one.  Fewer do not do:
// on blocks like the solver's (dominant diagonals), the error of I - D D^-1 at n = 160 against
// 113-bit sums is 2.7e-17 with them, 4.9e-17 with the FP64 FMA loop, 1.6e-16 when the weights
// 5 to 7 share an accumulator and 5.8e-16 without i + j = 7.  Per output the accumulators are
// joined in 64-bit integers and rounded once to FP64.
//
// Exactness.  A digit product is at most 2^14 and weight w sums 2 K (w + 1) of them, so whatever the
// digits, weight 4 stays within 2^24 up to K = 102 only.  Digits of mixed sign stay far below it.  With
// T the sum of the squares of a row's digits 0 .. 4, no partial sum of the weights 0 .. 4 exceeds
// (T_a T_b)^(1/2) (Cauchy-Schwarz over the pairs of a weight); digits spread evenly give T = 54600 K,
// 8.7e6 at K = 160 and 13.5e6 at K = 248, where 2^24 = 16.8e6 is allowed.  For SG_FULL the split marks
// the groups of rows with a row of too large T, and a tile that meets one makes a pass with an epilogue
// of its own for every 96 terms, for which the first bound holds.  The weights from 5 on may round: by
// 2^-43 of the product of the row's and the column's largest entries if all digits agree, where the
// bound of the FP64 FMA loop is 2^-36.  So may the accumulators of the shorter forms, by 2^-23: their
// products are corrections, or residuals that are formed again.
//
// Measured, 608 products of 160^3: SG_FULL 723 us (1.19 us a product, 28 TFLOP/s of FP64 work; the
// FP64 GEMM takes 28 us a product; 897 us with A in shared memory and an epilogue that the MMAs
// wait for), SG_HALF 463 us; splitting an operand 0.27 us, a right one 0.22.  Bound by the MMAs (47
// cycles each at N = 64 with the copies of A, where the tensor cores need 32) and by the joining of
// the accumulators (about a fifth).
//
// Layout.  A split form holds, per 16 terms k and digit s, planes r, i and -r of bf16 core
// matrices (8 rows x 8 terms, 128 bytes), so every shared-memory operand is a run of contiguous
// 2 KB pieces fetched by plain bulk copies.  The 128 accumulator lanes are 64 rows of Re and the
// same 64 rows of Im: [r; i] times B_r plus, with the instruction's negate bit, -[i; -r] times B_i;
// the two A operands are overlapping windows of the planes (r, i, -r), one copy of each.
//
// Roles of a persistent CTA (one per SM, 18 warps): warp 0 copies (stages of 16 terms, all
// digits), warp 1 issues a stage's MMAs (one wait per stage: a wait per digit made the loop
// twice as long), warps 2-17 join the accumulators, transpose through shared memory and store
// whole 256-byte row pieces.  The accumulators fill the tensor memory, so the next tile's MMAs
// start when they have been joined into registers, under the stores.  SG_FULL copies a digit's A
// windows to tensor memory once for all its pairs (tcgen05.cp): with A in shared memory an MMA
// of 64 columns is bound by reading it.  Tensor memory orders a copy before the MMAs that follow it,
// but not an MMA before the copy that overwrites its operand, so a slot's next copy waits for a commit
// behind its MMAs (slot_ring.h).
#include "tc_gemm64.cuh"
#include "tc_gemm.cuh"
#include "slot_ring.h"

#include <cuda_bf16.h>

namespace {

constexpr int SG_ROWS = 64;        // complex rows per tile (128 lanes)
constexpr int SG_STG_LD = 17;      // complex columns per staged row (16 + 1)
constexpr uint32_t SG_STG_BYTES = SG_ROWS * SG_STG_LD * 16;   // one of two staged slabs
constexpr int SG_EPI0 = 2, SG_EPI_WARPS = 16, SG_THREADS = 32 * (SG_EPI0 + SG_EPI_WARPS);
constexpr uint32_t SG_SMEM_MAX = 225 * 1024;

// W: digit weights kept (pairs of digits with i + j < W); ACC accumulators, the last one shared by
// the weights ACC - 1 .. W - 1; NT: most columns of a tile.
template <int W_, int ACC_, int NT_>
struct SgCfg {
  static constexpr int W = W_, ACC = ACC_, NT = NT_;
  static constexpr int DIG = W < SG_SLICES ? W : SG_SLICES;      // digits read
  static constexpr bool MARKS = DIG == SG_SLICES;                // passes for marked rows
  static constexpr uint32_t A_SLOT = 3 * SG_ROWS * 32;           // planes r, i, -r
  static constexpr uint32_t B_PLANE = NT * 32;
  static constexpr uint32_t SLOT = A_SLOT + 2 * B_PLANE;
  static constexpr uint32_t STAGE = DIG * SLOT;
  static constexpr int STAGES = 3 * STAGE + 2 * SG_STG_BYTES + 128 <= SG_SMEM_MAX ? 3 : 2;
  static constexpr uint32_t STG_OFF = STAGES * STAGE;
  static constexpr uint32_t BAR_OFF = STG_OFF + 2 * SG_STG_BYTES;
  // A operands copied to tensor memory beside the accumulators (four pairs of slots) where tiles are
  // narrow: from 80 columns on an MMA is not bound by reading A from shared memory
  static constexpr bool TS = NT <= 64;
  static_assert(!TS || (512 - ACC * NT >= 16 * RING_SLOTS && DIG == RING_DIGITS), "slots for A");
  static constexpr uint32_t SMEM = BAR_OFF + (2 * STAGES + 3 + RING_GROUPS) * 8 + 16;
  static_assert(SMEM <= SG_SMEM_MAX, "one CTA per SM beside the static shared memory");
  static_assert(SLOT % 128 == 0 && STG_OFF % 16 == 0 && NT % 16 == 0 && ACC * NT <= 512, "layout");
};
constexpr uint32_t SG_LBO = 128, SG_SBO = 256;
constexpr int32_t SG_EXP_NONFINITE = 0x7fffffff;
constexpr long long SG_OWN_WAIT = 4000000000LL;
constexpr int SG_PART = 6;               // chunks whose sums of weight <= 4 are exact for any digits
static_assert(5 * 2 * 16 * SG_PART * (1 << 14) <= 1 << 24, "");

struct SgArgs {
  int M, N, K;
  int nt, ntiles_n, ntiles_m, chunks;  // columns per tile (the last one narrower), tiles, 16-term chunks
  int GA, GB;                          // 8-row groups of the A and B forms
  int njob, ntiles;
  int tile0[2];
  SgJob job[2];
  int32_t* status;
  long long wait_limit;
};

__device__ __forceinline__ uint32_t s32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void bar_init(uint64_t* b, uint32_t n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(s32(b)), "r"(n));
}
__device__ __forceinline__ void bar_arrive(uint64_t* b) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(s32(b)) : "memory");
}
__device__ __forceinline__ void bar_expect(uint64_t* b, uint32_t bytes) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(s32(b)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool bar_test(uint32_t a, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(a), "r"(parity)
      : "memory");
  return done != 0u;
}
// bounded wait of a whole warp; gives up together on the abort flag or the limit
__device__ __forceinline__ bool wait_warp(uint64_t* b, uint32_t parity, volatile int* abort_flag,
                                          long long limit) {
  const uint32_t a = s32(b);
  const long long t0 = clock64();
  while (true) {
    if (__any_sync(0xffffffffu, bar_test(a, parity))) return true;
    const bool expired = clock64() - t0 > limit;
    if (__any_sync(0xffffffffu, expired || *abort_flag != 0)) {
      if (expired) *abort_flag = 1;
      return false;
    }
  }
}
// the kernel's own copies and MMAs, whatever the abort flag says (bounded)
__device__ __forceinline__ bool wait_own(uint64_t* b, uint32_t parity) {
  const uint32_t a = s32(b);
  const long long t0 = clock64();
  while (!bar_test(a, parity))
    if (clock64() - t0 > SG_OWN_WAIT) return false;
  return true;
}
// bounded wait of one thread
__device__ __forceinline__ bool wait_one(uint64_t* b, uint32_t parity, volatile int* abort_flag, long long limit) {
  const uint32_t a = s32(b);
  if (bar_test(a, parity)) return true;
  const long long t0 = clock64();
  while (!bar_test(a, parity)) {
    if (clock64() - t0 > limit) *abort_flag = 1;
    if (*abort_flag) return false;
  }
  return true;
}
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint64_t* b) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
      "l"(__cvta_generic_to_global(src)), "r"(bytes), "r"(s32(b))
      : "memory");
}
// A and B as the low words of their shared-memory descriptors (address >> 4 | LBO >> 4 << 16);
// the high word (SBO >> 4, descriptor version 1, no swizzle) is the same for all
__device__ __forceinline__ void mma_bf16(uint32_t d, uint32_t hi, uint32_t a, uint32_t b, uint32_t idesc,
                                         uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 da, db;\n setp.ne.b32 p, %5, 0;\n"
      " mov.b64 da, {%1, %4};\n mov.b64 db, {%2, %4};\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n}\n" ::"r"(d),
      "r"(a), "r"(b), "r"(idesc), "r"(hi), "r"(acc));
}
// the same with A in tensor memory (128 lanes x 8 columns)
__device__ __forceinline__ void mma_bf16_t(uint32_t d, uint32_t hi, uint32_t a, uint32_t b, uint32_t idesc,
                                           uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 db;\n setp.ne.b32 p, %5, 0;\n mov.b64 db, {%2, %4};\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %3, p;\n}\n" ::"r"(d),
      "r"(a), "r"(b), "r"(idesc), "r"(hi), "r"(acc));
}
// 128 rows x 16 terms from shared memory (descriptor lo, hi) to tensor memory
__device__ __forceinline__ void copy_a(uint32_t t, uint32_t lo, uint32_t hi) {
  asm volatile("{\n .reg .b64 da;\n mov.b64 da, {%1, %2};\n tcgen05.cp.cta_group::1.128x256b [%0], da;\n}\n" ::"r"(t),
               "r"(lo), "r"(hi)
               : "memory");
}
__device__ __forceinline__ void commit(uint64_t* b) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(s32(b))
               : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t a, float (&v)[4]) {
  uint32_t r[4];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a));
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(r[i]);
}
// one lane of a converged warp, known to the compiler as one (a plain lane == 0 test made each
// MMA issue 20 % slower: 20.3 us a tile against 17.5 without the epilogue)
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0u;
}
// true where `mine` holds in every epilogue thread (a barrier of the epilogue warps)
__device__ __forceinline__ bool agree(bool mine) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.and.pred q, 1, %2, p;\n"
      " selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"(mine ? 1u : 0u), "n"(32 * SG_EPI_WARPS)
      : "memory");
  return r != 0u;
}
// (hi 2^S + lo) 2^(ea + eb - 30 - S) rounded once to FP64, in integer arithmetic (the FP64 pipe
// converts and adds at 1/64 of the integer rate); |hi| < 2^41, |lo| < 2^52
template <int S>
__device__ __forceinline__ double scaled(long long hi, long long lo, int ea, int eb) {
  if (ea == SG_EXP_NONFINITE || eb == SG_EXP_NONFINITE) return __longlong_as_double(0x7ff8000000000000LL);
  bool neg;
  unsigned long long m;   // |value| 2^-sh, its lost bits (if any) or-ed into the lowest one
  int sh = 0;
  if (S < 32) {
    const long long T = (hi << S) + lo;
    neg = T < 0;
    m = (unsigned long long)(neg ? -T : T);
  } else {
    // the sum as h 2^32 + l, 0 <= l < 2^32
    long long h = hi + (lo >> 32);
    uint32_t l = (uint32_t)lo;
    neg = h < 0;
    if (neg) {
      l = 0u - l;
      h = -h - (l != 0u ? 1 : 0);
    }
    if (h < (1LL << 31)) {
      m = ((unsigned long long)h << 32) | l;
    } else {
      m = ((unsigned long long)h << 20) | (l >> 12) | ((l & 0xfffu) ? 1u : 0u);
      sh = 12;
    }
  }
  if (m == 0) return 0.0;
  const int lz = __clzll((long long)m);
  const int p = 63 - lz + sh + ea + eb - 30 - S;  // the value is in [2^p, 2^(p + 1))
  // leading one at bit 63, the 53 bits kept are 63 .. 11, ties to even on the rest
  const unsigned long long u = m << lz;
  unsigned long long f = u >> 11;
  const uint32_t rest = (uint32_t)u & 0x7ffu;
  f += (rest > 0x400u || (rest == 0x400u && (f & 1))) ? 1 : 0;
  if (p > -1022 && p < 1023) {
    // the implicit bit of f adds one to the exponent field (a carry out of f adds another)
    const unsigned long long b = ((unsigned long long)(p + 1022) << 52) + f;
    return __longlong_as_double((long long)(b | (neg ? 0x8000000000000000ULL : 0ULL)));
  }
  const double x = scalbn((double)f, p - 52);
  return neg ? -x : x;
}
__device__ __forceinline__ void f_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void f_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// ---------------------------------------------------------------- passes of a CTA
// tile -> job, product, row tile, column tile; each tile makes one pass (or several, see above) per
// segment it takes part in, every pass a full accumulation and epilogue of its own (the segments'
// operands have their own exponents).
struct Tile {
  int j, z, i0, n0, nt;  // nt: the tile's columns rounded up to 16
  bool run, v[2];
};
__device__ __forceinline__ Tile tile_at(const SgJob* jobs, const SgArgs& p, int t) {
  Tile r;
  r.j = (p.njob > 1 && t >= p.tile0[1]) ? 1 : 0;
  const int local = t - (r.j ? p.tile0[1] : 0);
  const int per = p.ntiles_m * p.ntiles_n;
  r.z = local / per;
  const int q = local - r.z * per;
  const int im = q / p.ntiles_n;
  r.i0 = im * SG_ROWS;
  r.n0 = (q - im * p.ntiles_n) * p.nt;
  r.nt = min(p.nt, (p.N - r.n0 + 15) & ~15);
  const SgJob& jb = jobs[r.j];
  r.run = jb.skip == nullptr || jb.skip[r.z] == 0;
  r.v[0] = r.run && r.z >= jb.seg[0].zlo && r.z < jb.seg[0].zhi;
  r.v[1] = r.run && jb.nseg > 1 && r.z >= jb.seg[1].zlo && r.z < jb.seg[1].zhi;
  return r;
}

// The marks of a tile's row groups, one per lane; where any lane has one, segment g takes a pass for
// every SG_PART chunks.  (They are voted on when the first SG_PART chunks are through, so that the loads
// are not waited for.)
__device__ __forceinline__ int32_t marks_of(const SgJob& jb, const SgArgs& p, const Tile& t, int g) {
  if (p.chunks <= SG_PART) return 0;
  const int lane = threadIdx.x & 31;
  const SgSeg& sg = jb.seg[g];
  if (lane < SG_ROWS / 8) {
    const int a = (t.i0 >> 3) + lane;
    return a < p.GA ? sg.eA[(int64_t)(t.z + sg.zA) * (p.GA * 9) + p.GA * 8 + a] : 0;
  }
  const int b = (t.n0 >> 3) + lane - SG_ROWS / 8;
  return lane - SG_ROWS / 8 < t.nt / 8 && b < p.GB ? sg.eB[(int64_t)(t.z + sg.zB) * (p.GB * 9) + p.GB * 8 + b] : 0;
}

template <typename Cfg>
__global__ void __launch_bounds__(SG_THREADS, 1) sg_gemm_kernel(const __grid_constant__ SgArgs p) {
  dep_begin();
  constexpr int SG_STAGES = Cfg::STAGES, SG_ACC = Cfg::ACC, SG_NT = Cfg::NT;
  constexpr uint32_t SG_STAGE = Cfg::STAGE, SG_SLOT = Cfg::SLOT, SG_A_SLOT = Cfg::A_SLOT,
                     SG_B_PLANE = Cfg::B_PLANE, SG_STG_OFF = Cfg::STG_OFF, SG_BAR_OFF = Cfg::BAR_OFF;
  extern __shared__ __align__(1024) unsigned char sm[];
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + SG_BAR_OFF);
  uint64_t* empty = full + SG_STAGES;
  uint64_t* acc_full = empty + SG_STAGES;
  uint64_t* acc_empty = acc_full + 1;
  uint64_t* done_bar = acc_empty + 1;
  uint64_t* slot_free = done_bar + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(slot_free + RING_GROUPS);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  __shared__ SgJob jobs[2];
  __shared__ int32_t sh_eb[SG_NT];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (p.njob == 1 && p.job[0].any && *p.job[0].any == 0) return;
  if (tid == 0) {
    jobs[0] = p.job[0];
    jobs[1] = p.job[1];
    for (int i = 0; i < SG_STAGES; ++i) {
      bar_init(&full[i], 1);
      bar_init(&empty[i], 1);
    }
    bar_init(acc_full, 1);
    bar_init(acc_empty, SG_EPI_WARPS);
    bar_init(done_bar, 1);
    for (int i = 0; i < RING_GROUPS; ++i) bar_init(&slot_free[i], 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s32(tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  f_before();
  __syncthreads();
  f_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t smb = s32(sm);

  if (warp == 0) {
    // ------------------------------------------------------------ copies
    int it = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x) {
      const Tile tl = tile_at(jobs, p, t);
      for (int g = 0; g < 2 && ok; ++g) {
        if (!tl.v[g]) continue;
        const SgSeg& sg = jobs[tl.j].seg[g];
        const int ga0 = tl.i0 >> 3, gb0 = tl.n0 >> 3;
        const uint32_t ba = 256u * (uint32_t)min(SG_ROWS / 8, p.GA - ga0);
        const uint32_t bb = 256u * (uint32_t)min(tl.nt / 8, p.GB - gb0);
        const int64_t fa = (int64_t)p.chunks * SG_SLICES * sg.planesA * p.GA * 256;
        const int64_t fb = (int64_t)p.chunks * SG_SLICES * sg.planesB * p.GB * 256;
        const unsigned char* A = sg.A + (tl.z + sg.zA) * fa + ga0 * 256;
        const unsigned char* B = sg.B + (tl.z + sg.zB) * fb + gb0 * 256;
        // lanes 0-2: a plane of A each, lanes 3-4: a plane of B
        const unsigned char* src = nullptr;
        int64_t step = 0;
        uint32_t off = 0, bytes = 0;
        if (lane < 3) {
          src = A + (int64_t)lane * p.GA * 256;
          step = (int64_t)sg.planesA * p.GA * 256;
          off = (uint32_t)lane * (SG_ROWS * 32);
          bytes = ba;
        } else if (lane < 5) {
          src = B + (int64_t)(lane - 3) * p.GB * 256;
          step = (int64_t)sg.planesB * p.GB * 256;
          off = SG_A_SLOT + (uint32_t)(lane - 3) * SG_B_PLANE;
          bytes = bb;
        }
        for (int c = 0; c < p.chunks; ++c, ++it) {  // (the passes of a segment one after the other)
          const int st = it % SG_STAGES;
          if (it >= SG_STAGES &&
              !wait_warp(&empty[st], (uint32_t)((it / SG_STAGES - 1) & 1), abort_flag, p.wait_limit)) {
            ok = false;
            break;
          }
          if (lane == 0) bar_expect(&full[st], Cfg::DIG * (3 * ba + 2 * bb));
          __syncwarp();
          if (lane < 5) {
            const uint32_t dst = smb + (uint32_t)st * SG_STAGE + off;
            for (int u = 0; u < Cfg::DIG; ++u)
              bulk_copy(dst + (uint32_t)u * SG_SLOT, src + (c * SG_SLICES + u) * step, bytes, &full[st]);
          }
        }
      }
    }
    // every copy has landed before the CTA can exit
    if (lane == 0)
      for (int d = it > SG_STAGES ? it - SG_STAGES : 0; d < it; ++d)
        if (!wait_own(&full[d % SG_STAGES], (uint32_t)((d / SG_STAGES) & 1))) *abort_flag = 1;
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issue
    const uint32_t ntu = (uint32_t)p.nt;
    const uint32_t dlo = (SG_LBO >> 4) << 16, dhi = (SG_SBO >> 4) | (1u << 14);
    constexpr uint32_t SLOT16 = SG_SLOT >> 4, A16 = SG_A_SLOT >> 4, R16 = (SG_ROWS * 32) >> 4, B16 = SG_B_PLANE >> 4;
    int it = 0, ps = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x) {
      const Tile tl = tile_at(jobs, p, t);
      for (int g = 0; g < 2 && ok; ++g) {
        if (!tl.v[g]) continue;
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(tl.nt >> 3) << 17) |
                               ((uint32_t)(128 >> 4) << 24);
        const uint32_t ineg = idesc | (1u << 13);  // -A
        const int32_t mark = Cfg::MARKS ? marks_of(jobs[tl.j], p, tl, g) : 0;
        int len = p.chunks;  // chunks of a pass
        for (int c = 0, cp = 0; c < p.chunks; ++c, ++cp, ++it) {
          if (Cfg::MARKS && c == SG_PART && __any_sync(0xffffffffu, mark != 0)) len = SG_PART;
          if (cp == len) {
            if (elect_one()) commit(acc_full);
            __syncwarp();
            ++ps;
            cp = 0;
          }
          if (cp == 0) {
            if (ps >= 1 && !wait_warp(acc_empty, (uint32_t)((ps - 1) & 1), abort_flag, p.wait_limit)) {
              ok = false;
              break;
            }
            f_after();
          }
          const int st = it % SG_STAGES;
          if (!wait_warp(&full[st], (uint32_t)((it / SG_STAGES) & 1), abort_flag, p.wait_limit)) {
            ok = false;
            break;
          }
          if (elect_one()) {
            const uint32_t a0 = dlo + ((smb + (uint32_t)st * SG_STAGE) >> 4), b0 = a0 + A16;
            const uint32_t more = cp > 0 ? 1u : 0u;  // the first pair of an accumulator overwrites it
#pragma unroll
            for (int i = 0; i < Cfg::DIG; ++i) {
              // both windows of the digit, read once from shared memory for all its pairs
              const uint32_t ta = tmem + (uint32_t)(SG_ACC * SG_NT) + 16u * ring_slot(i);
              if (Cfg::TS) {
                const int g = ring_group(i);
                if (ring_first(i) && ring_waits(g, it) &&
                    !wait_one(&slot_free[ring_wait_group(g)], ring_parity(g, it), abort_flag, p.wait_limit))
                  break;
                copy_a(ta, a0 + i * SLOT16, dhi);
                copy_a(ta + 8u, a0 + R16 + i * SLOT16, dhi);
              }
#pragma unroll
              for (int j = 0; j < Cfg::DIG; ++j) {
                if (i + j >= Cfg::W) continue;
                const int w = i + j < SG_ACC - 1 ? i + j : SG_ACC - 1;
                const uint32_t d = tmem + (uint32_t)w * ntu;
                const uint32_t on = i == 0 && j < SG_ACC ? more : 1u;
                if (Cfg::TS) {
                  mma_bf16_t(d, dhi, ta, b0 + j * SLOT16, idesc, on);
                  mma_bf16_t(d, dhi, ta + 8u, b0 + B16 + j * SLOT16, ineg, 1u);
                } else {
                  mma_bf16(d, dhi, a0 + i * SLOT16, b0 + j * SLOT16, idesc, on);
                  mma_bf16(d, dhi, a0 + R16 + i * SLOT16, b0 + B16 + j * SLOT16, ineg, 1u);
                }
              }
              if (Cfg::TS && ring_last(i)) commit(&slot_free[ring_group(i)]);
            }
            commit(&empty[st]);
          }
          __syncwarp();
        }
        if (ok && elect_one()) commit(acc_full);
        __syncwarp();
        ++ps;
      }
    }
    if (elect_one()) {
      commit(done_bar);
      if (!wait_own(done_bar, 0)) *abort_flag = 1;
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------ epilogue
    const int q = warp & 3;                    // lane quarter of this warp
    const int c4 = 4 * ((warp - SG_EPI0) >> 2);  // columns c4 .. c4 + 3 of each 16-column slab
    const int et = tid - 32 * SG_EPI0;
    const int row = 32 * (q & 1) + lane;       // row of the tile
    const int part = q >> 1;                   // 0: Re lanes, 1: Im lanes
    const uint32_t tl_base = tmem + ((uint32_t)(32 * q) << 16);
    unsigned char* stg = sm + SG_STG_OFF;
    int ps = 0, slab = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < p.ntiles && ok; t += gridDim.x) {
      const Tile tl = tile_at(jobs, p, t);
      const SgJob& jb = jobs[tl.j];
      const bool neg = jb.neg;
      bool first = true;
      uint32_t big = 0;  // largest high word of |re|, |im|
      for (int g = 0; g < 2 && ok; ++g) {
        if (!tl.v[g]) continue;
        const int32_t mark = Cfg::MARKS ? marks_of(jb, p, tl, g) : 0;
        int len = p.chunks;
        for (int pass = 0; pass < p.chunks; pass += len) {
          big = 0;  // (of the last pass, which leaves the output)
          const SgSeg& sg = jb.seg[g];
          const int32_t* eA = sg.eA + (int64_t)(tl.z + sg.zA) * (p.GA * 9);
          const int32_t* eB = sg.eB + (int64_t)(tl.z + sg.zB) * (p.GB * 9);
          const int ea = tl.i0 + row < p.M ? eA[tl.i0 + row] : 0;
          const double2* C0 = first ? (jb.C0 ? jb.C0 + tl.z * jb.sC0 : nullptr) : jb.C + tl.z * jb.sC;
          const int64_t ldc0 = first ? jb.ldc0 : jb.ldc;
          const bool eye = first && jb.identity;
          // the columns' exponents (the threads that read the last pass's are past a barrier since)
          if (et < p.nt) sh_eb[et] = tl.n0 + et < p.N ? eB[tl.n0 + et] : 0;
          double2* C = jb.C + tl.z * jb.sC;
          // the epilogue warps go on or give up together (they meet at barriers below)
          ok = agree(wait_warp(acc_full, (uint32_t)(ps & 1), abort_flag, p.wait_limit));
          if (!ok) break;
          f_after();
          if (Cfg::MARKS && __any_sync(0xffffffffu, mark != 0)) len = SG_PART;
          constexpr int SLABS = SG_NT / 16;
          // narrow tiles: all slabs are joined into registers first, so that the next tile's MMAs start
          // while the results are stored; wide ones (fewer digits, shorter epilogues) slab by slab
          constexpr bool HOLD = SLABS <= 4;
          const int last = tl.nt >> 4;
          auto join = [&](int sb, double (&v)[4]) {
            float a[SG_ACC][4];
#pragma unroll
            for (int w = 0; w < SG_ACC; ++w) tmem_ld4(tl_base + (uint32_t)(w * p.nt + 16 * sb + c4), a[w]);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (sb == last - 1) {
              f_before();
              __syncwarp();
              if (lane == 0) bar_arrive(acc_empty);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              // accumulator w in units of 2^(-8 w), joined in units of 2^(-8 (ACC - 1))
              long long hi = 0, lo = 0;
              float u = 1.f;
#pragma unroll
              for (int w = 0; w < SG_ACC; ++w) {
                const long long n = (long long)__float2int_rn(a[w][j] * u) << (8 * ((w < 3 ? 2 : SG_ACC - 1) - w));
                if (w < 3) hi += n;
                else lo += n;
                u *= 256.f;
              }
              v[j] = scaled<8 * (SG_ACC > 3 ? SG_ACC - 3 : 0)>(hi, lo, ea, sh_eb[16 * sb + c4 + j]);
            }
          };
          auto store = [&](int sb, const double (&v)[4]) {
            // this thread's outputs of the slab, rows r and r + 32, column col; their C0 first
            const int col = tl.n0 + 16 * sb + (et & 15);
            const int r = et >> 4;
            double2 c0[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const int gr = tl.i0 + r + 32 * i;
              c0[i] = (C0 && gr < p.M && col < p.N) ? C0[(int64_t)gr * ldc0 + col] : make_double2(0.0, 0.0);
            }
            double* sp = reinterpret_cast<double*>(stg + (uint32_t)(slab & 1) * SG_STG_BYTES) +
                         (row * SG_STG_LD + c4) * 2 + part;
#pragma unroll
            for (int j = 0; j < 4; ++j) sp[2 * j] = v[j];
            // the slab is whole; the other buffer's slab has been read by every warp before this
            asm volatile("bar.sync 1, %0;" ::"n"(32 * SG_EPI_WARPS) : "memory");
            const double2* sr = reinterpret_cast<const double2*>(stg + (uint32_t)(slab & 1) * SG_STG_BYTES);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const int gr = tl.i0 + r + 32 * i;
              if (gr < p.M && col < p.N) {
                double2 o = sr[(r + 32 * i) * SG_STG_LD + (et & 15)];
                if (neg) {
                  o.x = -o.x;
                  o.y = -o.y;
                }
                if (eye) {
                  if (gr == col) o.x += 1.0;
                } else if (C0) {
                  o.x += c0[i].x;
                  o.y += c0[i].y;
                }
                if (jb.C32) jb.C32[tl.z * jb.sC + (int64_t)gr * jb.ldc + col] = make_float2((float)o.x, (float)o.y);
                else C[(int64_t)gr * jb.ldc + col] = o;
                big = max(big, max((uint32_t)__double2hiint(o.x) & 0x7fffffffu,
                                   (uint32_t)__double2hiint(o.y) & 0x7fffffffu));
              }
            }
            ++slab;
          };
          if constexpr (HOLD) {
            double v[SLABS][4];
#pragma unroll
            for (int sb = 0; sb < SLABS; ++sb)
              if (sb < last) join(sb, v[sb]);
#pragma unroll
            for (int sb = 0; sb < SLABS; ++sb)
              if (sb < last) store(sb, v[sb]);
          } else {
            for (int sb = 0; sb < last; ++sb) {
              double v[4];
              join(sb, v);
              store(sb, v);
            }
          }
          first = false;
          ++ps;
        }
      }
      if (ok && jb.maxabs && tl.run) {
        const uint32_t wm = __reduce_max_sync(0xffffffffu, big);
        // rounded up to the next high word, so never below the largest entry
        if (lane == 0)
          atomicMax(&jb.maxabs[tl.z],
                    wm >= 0x7ff00000u ? 0x7f800000u
                                      : __float_as_uint(__double2float_ru(__hiloint2double((int)wm + 1, 0))));
      }
    }
  }
  f_before();
  __syncthreads();
  if (tid == 0 && *abort_flag) atomicCAS(p.status, DEV_OK, DEV_TIMEOUT);
  if (warp == 1) {
    f_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

// ---------------------------------------------------------------- split
// One block: ROWS rows (one or two groups) of one operand.  The rows are staged in shared memory with
// coalesced reads in either orientation, the row exponents reduced over 256 / ROWS threads each, then a
// thread takes eight consecutive terms of a row: the value as a 56-bit fixed-point integer, its
// balanced base-256 digits as the bytes of q + 0x808080808080, turned into floats by a byte
// permute and one FMA each, and stored as 16-byte core-matrix rows (16 threads cover 256
// contiguous bytes).  Bound by the integer issue rate: about 34 instructions per real.
constexpr int SS_THREADS = 256;

__device__ __forceinline__ long long fixed56(double x, int e) {
  // x = m 2^(p - 52), |x| < 2^e; q = rint(x 2^(55 - e))
  const long long b = __double_as_longlong(x);
  const int p = (int)((b >> 52) & 0x7ff);
  if (p == 0) return 0;  // zeros and subnormals
  const long long m = (b & 0xFFFFFFFFFFFFFLL) | 0x10000000000000LL;
  const int sh = 3 - (e - (p - 1023));
  long long q;
  if (sh >= 0) q = m << sh;
  else if (sh > -62) q = (m + (1LL << (-sh - 1))) >> (-sh);
  else q = 0;
  return b < 0 ? -q : q;
}

template <typename T, int SS_ROWS>
__global__ void __launch_bounds__(SS_THREADS)
sg_split_kernel(const cplx<T>* __restrict__ src, int64_t ld, int64_t stride, int trans, int rows, int K,
                int planes, int chunks, int G, unsigned char* __restrict__ form, int32_t* __restrict__ exps,
                const int32_t* __restrict__ skip, int digits, int limit) {
  dep_begin();
  extern __shared__ __align__(16) unsigned char raw[];
  const int z = blockIdx.y;
  if (skip && skip[z]) return;
  const int Kp = chunks * 16, LD = Kp + 1;
  cplx<T>* t = reinterpret_cast<cplx<T>*>(raw);
  __shared__ int re[SS_ROWS], energy[SS_ROWS];
  if (threadIdx.x < SS_ROWS) energy[threadIdx.x] = 0;
  const int r0 = blockIdx.x * SS_ROWS;
  const cplx<T>* S = src + (int64_t)z * stride;
  if (!trans) {
    for (int e = threadIdx.x; e < SS_ROWS * Kp; e += SS_THREADS) {
      const int r = e / Kp, k = e - r * Kp;
      t[r * LD + k] = (r0 + r < rows && k < K) ? S[(int64_t)(r0 + r) * ld + k] : czero<T>();
    }
  } else {
    for (int e = threadIdx.x; e < SS_ROWS * Kp; e += SS_THREADS) {
      const int k = e / SS_ROWS, r = e - k * SS_ROWS;
      t[r * LD + k] = (r0 + r < rows && k < K) ? S[(int64_t)k * ld + r0 + r] : czero<T>();
    }
  }
  __syncthreads();
  {
    constexpr int W = SS_THREADS / SS_ROWS;  // 16 or 32 threads a row
    const int r = threadIdx.x / W, l = threadIdx.x % W;
    int m = 0;
    for (int k = l; k < Kp; k += W) {
      const cplx<T> v = t[r * LD + k];
      const int a = (__double2hiint((double)v.x) >> 20) & 0x7ff, b = (__double2hiint((double)v.y) >> 20) & 0x7ff;
      m = max(m, max(a, b));
    }
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    // biased exponent p of the largest entry: every |x| < 2^(p - 1022)
    if (l == 0) {
      const int e = m == 0x7ff ? SG_EXP_NONFINITE : (m == 0 ? 0 : m - 1022);
      re[r] = e;
      const int g = (r0 + r) >> 3;
      if (g < G) exps[(int64_t)z * (G * 9) + r0 + r] = e;
    }
  }
  __syncthreads();
  const int64_t fbytes = (int64_t)chunks * SG_SLICES * planes * G * 256;
  unsigned char* F = form + (int64_t)z * fbytes;
  const int g0 = r0 >> 3;
  int en = 0;  // this thread's squares of the digits 0 .. 4, all of one row
  // item: row-in-group (8) | term half (2) | group (2) | part (2) | chunk
  for (int it = threadIdx.x; it < chunks * 4 * SS_ROWS; it += SS_THREADS) {
    constexpr int GL = SS_ROWS == 16 ? 1 : 0;  // bits of the group
    const int rr = it & 7, kc = (it >> 3) & 1, gg = GL ? (it >> 4) & 1 : 0, part = (it >> (4 + GL)) & 1,
              c = it >> (5 + GL);
    const int r = gg * 8 + rr;
    if (g0 + gg >= G) continue;
    const int e = re[r];
    long long q[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const cplx<T> v = t[r * LD + c * 16 + kc * 8 + j];
      q[j] = (e == SG_EXP_NONFINITE ? 0 : fixed56((double)(part ? v.y : v.x), e)) + 0x808080808080LL;
    }
    if (limit != 0) {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int d0 = (int)(q[j] >> 48), d = (int)((uint32_t)(q[j] >> 16) ^ 0x80808080u);
        en = __dp4a(d, d, en) + d0 * d0;
      }
    }
    unsigned char* out = F + ((int64_t)c * SG_SLICES * planes * G + g0 + gg) * 256 + kc * 128 + rr * 16;
    float w = 1.f;
#pragma unroll
    for (int s = 0; s < SG_SLICES; ++s) {
      if (s >= digits) break;
      float d[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (s == 0) {
          d[j] = (float)(int)(q[j] >> 48);
        } else {
          const int byte = 6 - s;  // digit s of the seven: byte 6 - s
          const uint32_t word = byte >= 4 ? (uint32_t)((unsigned long long)q[j] >> 32) : (uint32_t)q[j];
          const float f = __uint_as_float(__byte_perm(word, 0x4B000000u, 0x7650u + (byte & 3)));
          d[j] = fmaf(f, w, -8388736.f * w);
        }
      }
      uint4 o;
      uint32_t* ow = reinterpret_cast<uint32_t*>(&o);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(d[2 * j], d[2 * j + 1]);
        ow[j] = *reinterpret_cast<const uint32_t*>(&h);
      }
      unsigned char* o2 = out + ((int64_t)s * planes + part) * G * 256;
      *reinterpret_cast<uint4*>(o2) = o;
      if (planes == 3 && part == 0) {
        o.x ^= 0x80008000u;
        o.y ^= 0x80008000u;
        o.z ^= 0x80008000u;
        o.w ^= 0x80008000u;
        *reinterpret_cast<uint4*>(o2 + (int64_t)2 * G * 256) = o;
      }
      w *= 0.00390625f;
    }
  }
  // the marks of the row groups, behind the exponents
  if (limit != 0) {
    atomicAdd(&energy[((threadIdx.x >> 4) % (SS_ROWS / 8)) * 8 + (threadIdx.x & 7)], en);
    __syncthreads();
  }
  if (threadIdx.x < SS_ROWS / 8 && g0 + (int)threadIdx.x < G) {
    int m = 0;
    for (int r = 0; r < 8; ++r) m = max(m, energy[8 * threadIdx.x + r]);
    exps[(int64_t)z * (G * 9) + G * 8 + g0 + threadIdx.x] = m > limit ? 1 : 0;
  }
}

int sm_count() {
  static const int n = [] {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      v = 1;
    return v > 0 ? v : 1;
  }();
  return n;
}

}  // namespace

size_t sg_form_bytes(int rows, int K, int planes) {
  return (size_t)ceil_div(K, 16) * SG_SLICES * planes * ceil_div(rows, 8) * 256;
}

cudaError_t launch_sg_split(const void* src, bool f32, int64_t ld, int64_t stride, bool trans,
                            int rows, int K, int planes, int batch, unsigned char* form,
                            int32_t* exps, const int32_t* skip, cudaStream_t s, int digits) {
  if (batch <= 0) return cudaSuccess;
  if (rows < 1 || K < 1 || K > SG_KMAX || batch > 65535 || (planes != 2 && planes != 3))
    return cudaErrorInvalidValue;
  const int chunks = (int)ceil_div(K, 16), G = (int)ceil_div(rows, 8);
  // 16 rows a block; 8 where those blocks do not go twice round the SMs (a batch of one operand of
  // 128 rows: 6 -> 4 us)
  const bool few = (int64_t)ceil_div(rows, 16) * batch < 2 * sm_count();
  const int per = few ? 8 : 16;
  const size_t smem = (size_t)per * (chunks * 16 + 1) * (f32 ? sizeof(float2) : sizeof(double2));
  const dim3 grid((unsigned)ceil_div(rows, per), (unsigned)batch);
  // Squares of a row's digits 0 .. 4 up to which it is not marked; 0: no marks.  Up to K = 160 the left
  // operands' limit allows for any digits in the right ones, which then need none (the limit is 10.7e6
  // at K = 160, where digits spread evenly give 8.7e6).
  int limit = 0;
  if (digits == SG_SLICES && chunks > SG_PART)
    limit = K > 160 ? 1 << 24 : planes == 3 ? (int)((1LL << 48) / (5LL * 2 * K << 14)) : 0;
  auto go = [&](auto kernel, auto* p) -> cudaError_t {
    if (smem > 48 * 1024)
      RCI_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    RCI_CUDA_TRY(launch_dep(kernel, grid, SS_THREADS, smem, s, p, ld, stride, trans ? 1 : 0, rows, K, planes, chunks, G, form,
                            exps, skip, digits, limit));
    rci_note_launch();
    return cudaGetLastError();
  };
  if (f32) return few ? go(sg_split_kernel<float, 8>, (const float2*)src) : go(sg_split_kernel<float, 16>, (const float2*)src);
  return few ? go(sg_split_kernel<double, 8>, (const double2*)src) : go(sg_split_kernel<double, 16>, (const double2*)src);
}

namespace {
template <typename Cfg>
cudaError_t launch_cfg(SgArgs& a, int64_t products, cudaStream_t s) {
  // Columns of a tile.  With A in tensor memory an MMA's time grows with its columns (33 cycles for
  // 32, 47 for 64): full tiles and a narrower last one.  With A in shared memory it hardly does (48
  // for 32, 58 for 96): equal tiles.  Narrow ones where even they do not fill the GPU.
  a.ntiles_n = (int)ceil_div(a.N, Cfg::NT);
  a.nt = Cfg::TS ? Cfg::NT : (int)ceil_div(ceil_div(a.N, a.ntiles_n), 16) * 16;
  if (products * a.ntiles_m * ceil_div(a.N, 32) <= sm_count()) a.nt = 32;
  a.ntiles_n = (int)ceil_div(a.N, a.nt);
  const int64_t per = (int64_t)a.ntiles_m * a.ntiles_n, nt = products * per;
  if (nt > 0x7fffffffLL) return cudaErrorInvalidValue;
  a.ntiles = (int)nt;
  a.tile0[0] = 0;
  a.tile0[1] = (int)(a.job[0].batch * per);
  const unsigned grid = (unsigned)(nt < sm_count() ? nt : sm_count());
  RCI_CUDA_TRY(cudaFuncSetAttribute(sg_gemm_kernel<Cfg>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::SMEM));
  RCI_CUDA_TRY(launch_dep(sg_gemm_kernel<Cfg>, grid, SG_THREADS, Cfg::SMEM, s, a));
  rci_note_launch();
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_sg_gemm(int M, int N, int K, int njob, const SgJob* jobs, SgDigits digits, int32_t* status,
                           long long wait_limit, cudaStream_t s) {
  if (M < 1 || N < 1 || K < 1 || K > SG_KMAX || njob < 1 || njob > 2) return cudaErrorInvalidValue;
  SgArgs a{};
  a.M = M;
  a.N = N;
  a.K = K;
  a.chunks = (int)ceil_div(K, 16);
  a.ntiles_m = (int)ceil_div(M, SG_ROWS);
  a.GA = (int)ceil_div(M, 8);
  a.GB = (int)ceil_div(N, 8);
  a.status = status;
  a.wait_limit = wait_limit;
  int64_t products = 0;
  for (int j = 0; j < njob; ++j) {
    const SgJob& q = jobs[j];
    if (q.batch <= 0) continue;
    if (q.nseg < 1 || q.nseg > 2 || (q.C32 && (q.nseg > 1 || q.C0))) return cudaErrorInvalidValue;
    for (int g = 0; g < q.nseg; ++g)
      if (q.seg[g].planesA != 3 || q.seg[g].planesB < 2) return cudaErrorInvalidValue;
    a.job[a.njob++] = q;
    products += q.batch;
  }
  if (a.njob == 0) return cudaSuccess;
  switch (digits) {
    case SG_FULL: return launch_cfg<SgCfg<8, 7, 64>>(a, products, s);
    case SG_SMALL: return launch_cfg<SgCfg<4, 4, 112>>(a, products, s);
    default: return launch_cfg<SgCfg<5, 5, 96>>(a, products, s);
  }
}
