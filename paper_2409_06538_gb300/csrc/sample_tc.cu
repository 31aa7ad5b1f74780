// Tensor-core sampling sweep for the mixed-precision path (sm_103a tcgen05).
//
// The same autoregressive sweep as sample.cu (Sec. II.B: right-to-left contraction of the
// cached process tensors with the previous row's spins as fields, then left-to-right
// conditionals and draws), with the per-site contractions of a tile of 128 proposals done
// as (128 x CHI)(CHI x CHI) products on the tensor cores:
//   right sweep: v_y[m][al] = sum_be R_{c+1}(y)[m][be] B^y[al][be]     (A = R(y), B = B^y)
//   left sweep : u_y[m][be] = sum_al l[m][al]        B^y[al][be]       (A = l,    B = B^y^T)
// Thread m of the CTA owns proposal m, which is also TMEM lane m of the accumulator, so
// every per-proposal step (fields, normalisation, conditionals, the Philox draw, log q,
// the energy) runs in that thread's registers.
//
// Precision: operands are split x = hi + lo with hi = tf32(x) and lo = tf32(x - hi), and
// each product is hi.hi + hi.lo + lo.hi (three kind::tf32 MMAs with FP32 accumulation),
// which keeps the conditionals at FP32 accuracy; single TF32 operands would not meet the
// 1e-3 conditional tolerance because the contraction of a sign-indefinite MPS amplifies
// operand rounding.
//
// Roles (256 threads): warps 0-3 own the proposals, warp 4 issues the MMAs, warps 5-7 load the
// environment tiles ahead of time, split them and lay them out.  The A operand lives in tensor
// memory: a proposal's thread writes its row there with tcgen05.st, next to the accumulator it
// reads back, so it never passes through shared memory.  B operands use the K-major, no-swizzle
// canonical layout: 8-row x 16-byte core matrices, 128 B apart along K (LBO) and 32*CHI B apart
// along N (SBO); the two y of a site are adjacent, so the left sweep, whose A is the same for both,
// takes them in one MMA of N = 2 CHI.
//
// What bounds it: at CHI = 32 the right vectors R_{c+1}, 32 KB per site and tile written in the right
// sweep and read back in the left one (5.1 TB/s of them at L = 64 with two tiles on every SM, of 6.8
// measured for a copy); at CHI = 16 the instructions of the proposal warps.  They are kept
// [site][y][j/4][proposal][4], so every access is 512 contiguous bytes a warp (one row per proposal
// kept the load/store unit busy 32 lines an instruction), and the left sweep copies the next site's
// into shared memory while it finishes this one.  The loops over the columns are not unrolled: with
// straight-line bodies the warps waited for instructions three cycles an issue.
// One GB300, propose() before and now: CHI = 32, L = 64, 64 realizations x 1000 proposals 92 -> 38 ms;
// L = 48, 448 x 500 158 -> 65 ms; CHI = 16, L = 32, 1024 x 2000 246 -> 140 ms.
#include "common.cuh"
#include "kernels.h"
#include "rounding.cuh"

namespace tnmc {
namespace tc {

constexpr int M = 128;            // proposals per tile (MMA M)

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t kmajor_desc(uint32_t saddr, uint32_t sbo_bytes) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((128u & 0x3FFFFu) >> 4) << 16;       // LBO: next core matrix along K
  d |= (uint64_t)((sbo_bytes & 0x3FFFFu) >> 4) << 32;  // SBO: next 8-row group along M/N
  d |= (uint64_t)1 << 46;                               // descriptor version of this architecture
  return d;                                             // base offset 0, no swizzle
}

template <int N>
__host__ __device__ constexpr uint32_t idesc_tf32() {
  // FP32 accumulator, A and B TF32, both K-major, N/8 and M/16 fields
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// D (tensor memory) = A (tensor memory, K columns from a_tmem) B (shared memory) [+ D]
__device__ __forceinline__ void mma_tf32(uint32_t d_tmem, uint32_t a_tmem, uint64_t bd, uint32_t idesc, uint32_t acc) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n}\n"
               ::"r"(d_tmem), "r"(a_tmem), "l"(bd), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void mma_commit(uint64_t* mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(mbar)));
}
__device__ __forceinline__ bool try_parity(uint64_t* mbar, uint32_t parity) {
  uint32_t done = 0;
  asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(done) : "r"(su32(mbar)), "r"(parity) : "memory");
  return done != 0;
}
// Bounded wait for the given phase parity; false when the limit ran out.
__device__ __forceinline__ bool wait_parity(uint64_t* mbar, uint32_t parity, long long limit = 1ll << 20) {
  for (long long it = 0; it < limit; ++it)
    if (try_parity(mbar, parity)) return true;
  return false;
}
// One lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}
// Barrier id over NTHR threads that tells each whether any of them passed true.
template <int NTHR> __device__ __forceinline__ bool any_of(int id, bool v) {
  uint32_t r;
  asm volatile("{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbarrier.cta.red.or.pred q, %2, %3, p;\nselp.u32 %0, 1, 0, q;\n}\n"
               : "=r"(r) : "r"((uint32_t)v), "r"(id), "n"(NTHR) : "memory");
  return r != 0;
}
__device__ __forceinline__ void mbar_init(uint64_t* mbar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(mbar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* mbar) {
  asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(su32(mbar)) : "memory");
}
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// 8 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld8(uint32_t ta, float* v) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(ta));
#pragma unroll
  for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(r[j]);
}
__device__ __forceinline__ void tmem_st8(uint32_t ta, const float* v) {
  uint32_t r[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) r[j] = __float_as_uint(v[j]);
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%8], {%0,%1,%2,%3,%4,%5,%6,%7};"
               ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(ta)
               : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ float max_nan(float a, float b) {       // NaN if either is
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
// Float offset of element (row r, k) in a (rows x KD) K-major canonical operand.
template <int KD> __device__ __forceinline__ int koff(int r, int k) {
  return (r >> 3) * (8 * KD) + (k >> 2) * 32 + (r & 7) * 4 + (k & 3);
}

// Write eight values of this thread's row of an A operand: hi parts at ta, lo parts CHI columns on.
// fin (warp-uniform): all of them are finite.
template <int CHI> __device__ __forceinline__ void put8_split(uint32_t ta, const float* x, bool fin) {
  float h[8], l[8];
  if (fin) {
#pragma unroll
    for (int t = 0; t < 8; ++t) { h[t] = tf32_rna_finite(x[t]); l[t] = tf32_rna_finite(x[t] - h[t]); }
  } else {
#pragma unroll
    for (int t = 0; t < 8; ++t) { h[t] = tf32_rna(x[t]); l[t] = tf32_rna(x[t] - h[t]); }
  }
  tmem_st8(ta, h);
  tmem_st8(ta + CHI, l);
}
// The row (1, 0, ..., 0) that a sweep starts from.
template <int CHI> __device__ __forceinline__ void put_e0(uint32_t ta) {
#pragma unroll 1
  for (int j = 0; j < 2 * CHI; j += 8) {
    const float x[8] = {j == 0 ? 1.0f : 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    tmem_st8(ta + j, x);
  }
}

// Draw s = +1 iff u < q(+), u = m53 2^-53: m < ceil(q 2^53) exactly, in integers.
__device__ __forceinline__ bool draw_below(uint64_t m53, float q) {
  if (q >= 1.0f) return true;
  if (!(q > 0.0f)) return false;
  const uint32_t bits = __float_as_uint(q);
  const int ex = (int)((bits >> 23) & 0xffu);
  const uint64_t mant = (ex == 0) ? (uint64_t)(bits & 0x7fffffu) : (uint64_t)((bits & 0x7fffffu) | 0x800000u);
  const int sh = (ex == 0 ? 1 : ex) - 150 + 53;
  uint64_t C;
  if (sh >= 0) C = mant << sh;
  else { const int k = -sh; C = (k >= 64) ? 1ull : ((mant + ((1ull << k) - 1ull)) >> k); }
  return m53 < C;
}

template <int CHI> struct Cfg {
  static constexpr int NT = 256;                    // 4 proposal warps, 1 MMA warp, 3 tile warps
  static constexpr int NPROD = 96;
  static constexpr int BOP = CHI * CHI;             // floats of one B operand
  static constexpr int TILE = 2 * BOP;              // floats of one cached site tile [y][al][be]
  static constexpr int STAGE = 4 * BOP;             // [hi y0, hi y1, lo y0, lo y1]
  static constexpr int NST = CHI <= 16 ? 4 : 3;     // stages
  // tiles as they are in global memory: one being split, one on its way (a third was no faster at any size)
  static constexpr int RAWTILE = 2 * CHI * (CHI + 4), NRAW = 2;
  // tensor memory: accumulators of y = 0, 1, then the A rows R0 (or l) hi, lo, R1 hi, lo
  static constexpr int TCOLS = 6 * CHI <= 128 ? 128 : 256;
  // CTAs per SM: tensor memory and registers allow two at CHI = 32, three at 16
  static constexpr int PER_SM = CHI <= 16 ? 3 : 2;
};

}  // namespace tc

template <int CHI, int PER_SM>
__global__ void __launch_bounds__(tc::Cfg<CHI>::NT, PER_SM) sample_tc_kernel(SampleArgs a) {
  using namespace tc;
  using C = Cfg<CHI>;
  constexpr int BOP = C::BOP, TILE = C::TILE, NST = C::NST;
  constexpr uint32_t SBO = 32 * CHI;      // bytes between 8-row groups (K = CHI)
  const int L = a.L, N = L * L;
  const int tid = threadIdx.x, warp = tid >> 5;

  extern __shared__ __align__(1024) float smf[];
  float* Bbuf = smf;                                  // [stage][hi y0, hi y1, lo y0, lo y1]
  const int LP = (L + 15) & ~15;                      // keeps the uint32 arrays 16-byte aligned
  float* Rawbuf = Bbuf + NST * C::STAGE;              // [buffer][y, al][be], rows padded
  float* Rws = Rawbuf + C::NRAW * C::RAWTILE;         // [y][j / 4][proposal][4]
  int8_t* jrow = reinterpret_cast<int8_t*>(Rws + 2 * CHI * M);      // [proposal warp][Jh row, Jv row above]
  uint32_t* prow = reinterpret_cast<uint32_t*>(jrow + 8 * LP);          // [words_row][M]
  __shared__ __align__(8) uint64_t bar_a, bar_d, bar_full[NST], bar_free[NST];
  __shared__ uint32_t tslot;
  __shared__ volatile int abort_flag;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&tslot)), "r"(C::TCOLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    mbar_init(&bar_a, 4);                 // A rows written, one arrival per warp
    mbar_init(&bar_d, 1);                 // products complete
    for (int i = 0; i < NST; ++i) { mbar_init(&bar_full[i], C::NPROD / 32); mbar_init(&bar_free[i], 1); }
    asm volatile("fence.mbarrier_init.release.cluster;");
    abort_flag = 0;
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tbase = tslot;

  // Bounded wait; on a timeout, or when another thread met one, every role leaves its loops and
  // meets the others at the end.
  auto wait_or_abort = [&](uint64_t* bar, uint32_t parity) -> bool {
    for (int it = 0; it < (1 << 20); ++it) {
      if (try_parity(bar, parity)) return true;
      if (abort_flag) return false;
    }
    set_status(a.status, ST_TIMEOUT);
    abort_flag = 1;
    return false;
  };

  const int tiles_per_real = (a.n_items + M - 1) / M;
  const int64_t total = (int64_t)tiles_per_real * a.n_real;
  // Products per row: the right sweep's sites L-1 .. 1 (site 0's has no reader), then the left
  // sweep's 0 .. L-1.

  if (warp >= 5) {
    // ---------------- tile warps ----------------
    constexpr int UNITS = TILE / 4;                   // 16-byte chunks of a tile
    constexpr int RS = CHI + 4;                       // row stride of a raw tile: the reads are conflict-free
    const int ptid = tid - 160;
    int64_t lt = blockIdx.x;                          // next tile to copy
    int lr = 0, li = 0, lb = 0;
    auto copy_next = [&]() {
      if (lt < total) {
        const int c = li < L - 1 ? L - 1 - li : li - (L - 1);
        const float* tile = reinterpret_cast<const float*>(a.env) + (((size_t)(lt / tiles_per_real) * L + lr) * L + c) * TILE;
        float* dst = Rawbuf + lb * C::RAWTILE;
#pragma unroll 1
        for (int u = ptid; u < UNITS; u += C::NPROD) {
          const uint32_t d = su32(dst + (u / (CHI / 4)) * RS + 4 * (u % (CHI / 4)));
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(tile + 4 * u) : "memory");
        }
        lb ^= 1;
        if (++li == 2 * L - 1) { li = 0; if (++lr == L) { lr = 0; lt += gridDim.x; } }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    copy_next();
    const int64_t mine = blockIdx.x < total ? (total - 1 - blockIdx.x) / gridDim.x + 1 : 0;
    const int64_t operands = mine * L * (2 * L - 1);
    int i = 0, rb = 0, st = 0;
    uint32_t round = 0;                               // times the stages have been filled
    for (int64_t n = 0; n < operands; ++n) {
      // this tile's copy has arrived and the stage is free, for every tile warp; all are done with
      // the raw tile before this one, whose buffer takes the next copy
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      const bool ok = round == 0 || wait_or_abort(&bar_free[st], (round - 1) & 1u);
      if (any_of<C::NPROD>(1, !ok)) break;            // all of them leave, or none
      copy_next();
      const bool left = i >= L - 1;
      const float* src = Rawbuf + rb * C::RAWTILE;
      float* stage = Bbuf + st * C::STAGE;
#pragma unroll 1
      for (int u = ptid; u < UNITS; u += C::NPROD) {
        // right: four be of row al; left: four al of row be
        const int y = u / (UNITS / 2), e = u % (UNITS / 2);
        const float* p = src + y * CHI * RS;
        int row, kg;
        float x[4];
        if (left) {
          row = e % CHI; kg = e / CHI;
#pragma unroll
          for (int t = 0; t < 4; ++t) x[t] = p[(4 * kg + t) * RS + row];
        } else {
          row = (e / (2 * CHI)) * 8 + (e & 7); kg = (e >> 3) % (CHI / 4);
          const float4 v = *reinterpret_cast<const float4*>(p + row * RS + 4 * kg);
          x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
        }
        float h[4], l[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) { h[t] = tf32_rna(x[t]); l[t] = tf32_rna(x[t] - h[t]); }
        float* d = stage + y * BOP + koff<CHI>(row, 4 * kg);
        *reinterpret_cast<float4*>(d) = make_float4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<float4*>(d + 2 * BOP) = make_float4(l[0], l[1], l[2], l[3]);
      }
      fence_async_smem();
      __syncwarp();
      if ((tid & 31) == 0) mbar_arrive(&bar_full[st]);
      if (++i == 2 * L - 1) i = 0;
      rb ^= 1;
      if (++st == NST) { st = 0; ++round; }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  } else if (warp == 4) {
    // ---------------- MMA warp ----------------
    // the whole warp runs the loop, one lane is elected at each issue: descriptors and addresses
    // stay in uniform registers
    uint32_t n = 0, round = 0;
    int st = 0;
    bool run = true;
    const uint32_t ta = tbase + 2 * CHI;
    constexpr uint64_t LO = (uint64_t)(2 * BOP * 4) >> 4, Y1 = (uint64_t)(BOP * 4) >> 4, KK = 256u >> 4;
    const uint64_t b0 = kmajor_desc(su32(Bbuf), SBO);
    for (int64_t tileid = blockIdx.x; run && tileid < total; tileid += gridDim.x)
      for (int r = 0; run && r < L; ++r)
        for (int i = 0; i < 2 * L - 1; ++i) {
          const bool ok = wait_or_abort(&bar_full[st], round & 1u) && wait_or_abort(&bar_a, n & 1u);
          if (!__all_sync(0xffffffffu, ok)) { run = false; break; }
          fence_after();
          const uint64_t bh = b0 + (uint64_t)st * ((C::STAGE * 4) >> 4);
          if (elect_one()) {
            // hi.hi + hi.lo + lo.hi, each over K in steps of 8
            if (i < L - 1) {
#pragma unroll
              for (int y = 0; y < 2; ++y)
#pragma unroll
                for (int term = 0; term < 3; ++term)
#pragma unroll
                  for (int kk = 0; kk < CHI / 8; ++kk)
                    mma_tf32(tbase + y * CHI, ta + (2 * y + (term == 2 ? 1 : 0)) * CHI + 8 * kk,
                             bh + (term == 1 ? LO : 0) + y * Y1 + kk * KK, idesc_tf32<CHI>(), (term | kk) ? 1u : 0u);
            } else {
#pragma unroll
              for (int term = 0; term < 3; ++term)
#pragma unroll
                for (int kk = 0; kk < CHI / 8; ++kk)
                  mma_tf32(tbase, ta + (term == 2 ? CHI : 0) + 8 * kk, bh + (term == 1 ? LO : 0) + kk * KK,
                           idesc_tf32<2 * CHI>(), (term | kk) ? 1u : 0u);
            }
            mma_commit(&bar_d);
            mma_commit(&bar_free[st]);
          }
          __syncwarp();
          ++n;
          if (++st == NST) { st = 0; ++round; }
        }
    if (!run && n > 0) wait_parity(&bar_d, (n - 1) & 1);       // products in flight end before the memory is freed
    __syncwarp();
  } else {
    // ---------------- proposal warps ----------------
    const uint32_t tlane = (uint32_t)(warp * 32) << 16;
    const uint32_t td = tbase + tlane, ta = td + 2 * CHI;
    const int lane = tid & 31;
    int8_t* jh_s = jrow + warp * 2 * LP;
    int8_t* jv_s = jh_s + LP;
    uint32_t n = 0;                                   // products waited for
    bool run = true;
    // the products are complete (warp-uniform: the TMEM accesses need the whole warp)
    auto products = [&]() -> bool {
      const bool ok = __all_sync(0xffffffffu, wait_or_abort(&bar_d, n & 1));
      ++n;
      fence_after();
      return ok;
    };
    auto a_ready = [&]() {                            // this warp's A rows are written
      tmem_wait_st();
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar_a);
    };
    // R_{c+1}(y) per site and proposal, [site][y][j / 4][proposal][4]: 16-byte accesses that are
    // contiguous over the lanes
    const bool own = (int)blockIdx.x < a.work_slots;
    float* work = reinterpret_cast<float*>(own ? a.work : a.more) +
                  (size_t)(own ? (int)blockIdx.x : (int)blockIdx.x - a.work_slots) * L * 2 * M * CHI + 4 * tid;
    float* rws = Rws + 4 * tid;                       // one site's, in shared memory

    for (int64_t tileid = blockIdx.x; run && tileid < total; tileid += gridDim.x) {
      const int real = (int)(tileid / tiles_per_real);
      const int k = (int)(tileid % tiles_per_real) * M + tid;
      const bool valid = k < a.n_items;
      const int64_t item = (int64_t)real * a.n_items + k;
      const int chain = a.forced ? 0 : (a.chain_of ? a.chain_of[real] : k / a.n);
      const uint32_t step = (uint32_t)(a.step0 + (uint64_t)(a.forced ? 0 : k % a.n));
      const uint64_t seed = a.seeds[real];
      const double betad = a.beta[real];
      const float eb = (float)exp(betad), ebm = (float)exp(-betad);
      const int8_t* J = a.J + (size_t)real * 2 * L * (L - 1);
      const int8_t* forced = (a.forced && valid) ? a.forced + (size_t)item * N : nullptr;
      const int8_t* hf = a.hfield ? a.hfield + (size_t)real * N : nullptr;
      double logq = 0.0;
      int energy = 0, magnet = 0;
      long long nclamp = 0;
      uint32_t gword = 0;

      for (int r = 0; r < L; ++r) {
        // the couplings of this row, a copy per warp: no barrier between the warps
        __syncwarp();
        for (int c = lane; c < L - 1; c += 32) jh_s[c] = J[(size_t)r * (L - 1) + c];
        if (r > 0)
          for (int c = lane; c < L; c += 32) jv_s[c] = J[(size_t)L * (L - 1) + (size_t)(r - 1) * L + c];
        __syncwarp();

        // ---------------- right sweep ----------------
        put_e0<CHI>(ta);
        put_e0<CHI>(ta + 2 * CHI);
        a_ready();
        for (int c = L - 1; c > 0; --c) {
          // R_c(y') = sum_y exp(beta Jh s_y' s_y) exp(h_c s_y) v_y
          const int jh = jh_s[c - 1];
          float f0 = 1.0f, f1 = 1.0f;
          if (r > 0) {
            const int sp = ((prow[(c >> 5) * M + tid] >> (c & 31)) & 1u) ? -1 : 1;
            const int sg = jv_s[c] * sp;
            f0 = sg > 0 ? eb : ebm; f1 = sg > 0 ? ebm : eb;
          }
          if (hf) { const int kh = hf[(size_t)r * L + c]; if (kh) { f0 *= expf((float)(betad * kh)); f1 *= expf((float)(-betad * kh)); } }
          const float same = jh > 0 ? eb : ebm, diff = jh > 0 ? ebm : eb;
          const float s0 = same * f0, s1 = same * f1, d0 = diff * f0, d1 = diff * f1;
          if (!products()) { run = false; break; }
          // eight columns at a time, in loops that are not unrolled: a straight-line body is
          // fetched anew for every site (see the head of the kernel)
          auto combine = [&](int j, float* n0, float* n1) {
            float v0[8], v1[8];
            tmem_ld8(td + j, v0);
            tmem_ld8(td + CHI + j, v1);
            tmem_wait_ld();
#pragma unroll
            for (int t = 0; t < 8; ++t) {
              n0[t] = fmaf(s0, v0[t], __fmul_rn(d1, v1[t]));
              n1[t] = fmaf(d0, v0[t], __fmul_rn(s1, v1[t]));
            }
          };
          float mx0 = 0.0f, mx1 = 0.0f;
#pragma unroll 1
          for (int j = 0; j < CHI; j += 8) {
            float n0[8], n1[8];
            combine(j, n0, n1);
#pragma unroll
            for (int t = 0; t < 8; ++t) { mx0 = max_nan(mx0, fabsf(n0[t])); mx1 = max_nan(mx1, fabsf(n1[t])); }
          }
          float mx = max_nan(mx0, mx1);
          if (__any_sync(0xffffffffu, isnan(mx))) {      // a NaN takes no part in the maximum
            mx = 0.0f;
#pragma unroll 1
            for (int j = 0; j < CHI; j += 8) {
              float n0[8], n1[8];
              combine(j, n0, n1);
#pragma unroll
              for (int t = 0; t < 8; ++t) mx = fmaxf(mx, fmaxf(fabsf(n0[t]), fabsf(n1[t])));
            }
          }
          const float inv = mx > 0.0f ? 1.0f / mx : 1.0f;
          const bool fin = __all_sync(0xffffffffu, !isnan(max_nan(mx0, mx1)) && isfinite(mx) && isfinite(inv));
          // read back by the left sweep at c - 1 (the last one at once, so it stays on the chip)
          float* wsl = c > 1 ? work + (size_t)((c - 1) * 2) * M * CHI : rws;
#pragma unroll 1
          for (int j = 0; j < CHI; j += 8) {
            float n0[8], n1[8];
            combine(j, n0, n1);
#pragma unroll
            for (int t = 0; t < 8; ++t) { n0[t] *= inv; n1[t] *= inv; }
#pragma unroll
            for (int t = 0; t < 8; t += 4) {
              *reinterpret_cast<float4*>(wsl + (j + t) * M) = make_float4(n0[t], n0[t + 1], n0[t + 2], n0[t + 3]);
              *reinterpret_cast<float4*>(wsl + (CHI + j + t) * M) = make_float4(n1[t], n1[t + 1], n1[t + 2], n1[t + 3]);
            }
            put8_split<CHI>(ta + j, n0, fin);
            put8_split<CHI>(ta + 2 * CHI + j, n1, fin);
          }
          if (c > 1) a_ready();
        }
        if (!run) break;

        __threadfence();              // the copies below read what this thread has stored
        // ---------------- left sweep ----------------
        tmem_wait_st();               // stores are in no order of their own: R_1's before those of l
        put_e0<CHI>(ta);
        a_ready();
        int sprev = 0;
        float rsum = 0.0f, rcomp = 0.0f;
        uint32_t rword = 0;
        for (int c = 0; c < L; ++c) {
          // what does not depend on the products: the fields, the random number
          float f0 = 1.0f, f1 = 1.0f;
          int sp = 0;
          if (r > 0) {
            sp = ((prow[(c >> 5) * M + tid] >> (c & 31)) & 1u) ? -1 : 1;
            const int sg = jv_s[c] * sp;
            f0 = sg > 0 ? eb : ebm; f1 = sg > 0 ? ebm : eb;
          }
          if (c > 0) { const int sg = jh_s[c - 1] * sprev; f0 *= sg > 0 ? eb : ebm; f1 *= sg > 0 ? ebm : eb; }
          if (hf) { const int kh = hf[(size_t)r * L + c]; if (kh) { f0 *= expf((float)(betad * kh)); f1 *= expf((float)(-betad * kh)); } }
          uint64_t m53 = 0;
          int sforced = 0;
          if (forced) {
            sforced = forced[(size_t)r * L + c];
          } else {
            const Philox4 o = philox4x32_10((uint32_t)(r * L + c), step, (uint32_t)chain, PURPOSE_SPIN,
                                            (uint32_t)seed, (uint32_t)(seed >> 32));
            m53 = ((uint64_t)(o.x0 >> 5) << 26) | (uint64_t)(o.x1 >> 6);
          }
          if (!products()) { run = false; break; }
          asm volatile("cp.async.wait_group 0;" ::: "memory");
          float d0 = 0.0f, d1 = 0.0f;
#pragma unroll 1
          for (int j = 0; j < CHI; j += 8) {
            float u0[8], u1[8], r0[8], r1[8];
            tmem_ld8(td + j, u0);
            tmem_ld8(td + CHI + j, u1);
#pragma unroll
            for (int t = 0; t < 8; t += 4) {
              *reinterpret_cast<float4*>(r0 + t) = *reinterpret_cast<const float4*>(rws + (j + t) * M);
              *reinterpret_cast<float4*>(r1 + t) = *reinterpret_cast<const float4*>(rws + (CHI + j + t) * M);
            }
            tmem_wait_ld();
#pragma unroll
            for (int t = 0; t < 8; ++t) { d0 = fmaf(u0[t], r0[t], d0); d1 = fmaf(u1[t], r1[t], d1); }
          }
          // the next site's right vectors: a copy in flight while this site is finished
          if (c + 2 < L) {
            const float* wsl = work + (size_t)((c + 1) * 2) * M * CHI;
#pragma unroll 4
            for (int j = 0; j < 2 * CHI; j += 4)
              asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(su32(rws + j * M)), "l"(wsl + j * M) : "memory");
            asm volatile("cp.async.commit_group;" ::: "memory");
          } else if (c + 1 < L) {
#pragma unroll 4
            for (int j = 0; j < 2 * CHI; j += 4)
              *reinterpret_cast<float4*>(rws + j * M) = make_float4(j % CHI == 0 ? 1.0f : 0.0f, 0.0f, 0.0f, 0.0f);
          }
          float w0 = f0 * d0, w1 = f1 * d1;
          if (w0 < 0.0f) { w0 = 0.0f; ++nclamp; }
          if (w1 < 0.0f) { w1 = 0.0f; ++nclamp; }
          const float tot = w0 + w1;
          const bool bad = !(tot > 0.0f) || !isfinite(tot);
          // A doubly clamped or non-finite site flags the realization; the spin is still drawn from
          // the q = 1/2 that is logged, so that log q stays the probability of the proposal.
          const float qp = bad ? 0.5f : w0 / tot;
          const int s = forced ? sforced : (bad ? ((m53 < (1ull << 52)) ? 1 : -1) : (draw_below(m53, qp) ? 1 : -1));
          // l <- u_s, normalised
          if (c < L - 1) {
            auto chosen = [&](int j, float* x) {
              float u1[8];
              tmem_ld8(td + j, x);
              tmem_ld8(td + CHI + j, u1);
              tmem_wait_ld();
#pragma unroll
              for (int t = 0; t < 8; ++t) x[t] = s == 1 ? x[t] : u1[t];
            };
            __syncwarp();
            float mx0 = 0.0f, mx1 = 0.0f;
#pragma unroll 1
            for (int j = 0; j < CHI; j += 8) {
              float x[8];
              chosen(j, x);
#pragma unroll
              for (int t = 0; t < 8; t += 2) { mx0 = max_nan(mx0, fabsf(x[t])); mx1 = max_nan(mx1, fabsf(x[t + 1])); }
            }
            float mx = max_nan(mx0, mx1);
            if (__any_sync(0xffffffffu, isnan(mx))) {
              mx = 0.0f;
#pragma unroll 1
              for (int j = 0; j < CHI; j += 8) {
                float x[8];
                chosen(j, x);
#pragma unroll
                for (int t = 0; t < 8; ++t) mx = fmaxf(mx, fabsf(x[t]));
              }
            }
            const float inv = mx > 0.0f ? 1.0f / mx : 1.0f;
            const bool fin = __all_sync(0xffffffffu, !isnan(max_nan(mx0, mx1)) && isfinite(mx) && isfinite(inv));
#pragma unroll 1
            for (int j = 0; j < CHI; j += 8) {
              float x[8];
              chosen(j, x);
#pragma unroll
              for (int t = 0; t < 8; ++t) x[t] *= inv;
              put8_split<CHI>(ta + j, x, fin);
            }
            a_ready();
          }
          // what the next product does not wait for: log q, the output, the energy
          float lqs = -0.6931471805599453f;
          if (!bad) {
            const float qm = w1 / tot;
            const float qs = s == 1 ? qp : qm, qo = s == 1 ? qm : qp;
            lqs = qs > 0.5f ? log1pf(-qo) : logf(qs);
          } else if (valid) {
            set_status(a.status, ST_NUMERIC);
            if (a.real_status) set_status(a.real_status + real, ST_NUMERIC);
          }
          { const float yk = lqs - rcomp; const float tk = rsum + yk; rcomp = (tk - rsum) - yk; rsum = tk; }
          if (a.qplus && valid) a.qplus[(size_t)item * N + (size_t)r * L + c] = (double)qp;
          if (c > 0) energy -= jh_s[c - 1] * sprev * s;
          if (r > 0) energy -= jv_s[c] * sp * s;
          magnet += s;
          sprev = s;
          if (s < 0) rword |= 1u << (c & 31);
          // the previous row's word has been read to its end
          if ((c & 31) == 31 || c == L - 1) { prow[(c >> 5) * M + tid] = rword; rword = 0; }
          const int site = r * L + c;
          if (s < 0) gword |= 1u << (site & 31);
          if ((site & 31) == 31 || site == N - 1) {
            if (valid && a.spins_packed) a.spins_packed[(size_t)item * a.words + (site >> 5)] = gword;
            gword = 0;
          }
        }
        if (!run) break;
        logq += (double)rsum;
      }
      if (valid && run) {
        if (a.logq) a.logq[item] = logq;
        if (a.energy) a.energy[item] = energy;
        if (a.magnet) a.magnet[item] = magnet;
        if (a.clamps && nclamp) atomicAdd(reinterpret_cast<unsigned long long*>(a.clamps + real), (unsigned long long)nclamp);
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(C::TCOLS));
}

template <int CHI>
static size_t sample_tc_smem(int L) {
  using C = tc::Cfg<CHI>;
  const int words_row = (L + 31) / 32;
  return (size_t)(C::NST * C::STAGE + C::NRAW * C::RAWTILE + 2 * CHI * tc::M) * sizeof(float) +
         (size_t)8 * ((L + 15) & ~15) + (size_t)words_row * tc::M * sizeof(uint32_t) + 64;
}

static int64_t sample_tc_tiles(int n_items, int n_real) { return (int64_t)((n_items + tc::M - 1) / tc::M) * n_real; }

// Every context has the slots of two CTAs per SM; those of the third at CHI = 16 are allocated at the first call
// whose tiles two do not hold at once.
constexpr int kOwnSlots = 2;

SampleWork sample_tc_work(int L, int CHI, int num_sms, int n_items, int n_real) {
  const size_t slot = (size_t)L * 2 * tc::M * CHI * sizeof(float);
  const int per_sm = CHI <= 16 ? tc::Cfg<16>::PER_SM : tc::Cfg<32>::PER_SM;
  const bool more = per_sm > kOwnSlots && sample_tc_tiles(n_items, n_real) > (int64_t)kOwnSlots * num_sms;
  return SampleWork{kOwnSlots * num_sms * slot, (per_sm - kOwnSlots) * num_sms * slot, more, more};
}

template <int CHI, int PER_SM>
static cudaError_t launch_tc_t(SampleArgs a, int num_sms, cudaStream_t st) {
  const int64_t tiles = sample_tc_tiles(a.n_items, a.n_real);
  // Where two CTAs per SM hold every tile anyway, or there is no workspace for a third, the build with their
  // registers (CHI = 16: 48 tiles 2.8 -> 2.6 ms, while 16384 tiles take 158 ms with two CTAs per SM against
  // 140 with three).
  if constexpr (PER_SM > kOwnSlots)
    if (tiles <= (int64_t)kOwnSlots * num_sms || !a.more) return launch_tc_t<CHI, kOwnSlots>(a, num_sms, st);
  const cudaError_t e = allow_shared_memory<sample_tc_kernel<CHI, PER_SM>>();
  if (e != cudaSuccess) return e;
  a.work_slots = kOwnSlots * num_sms;
  const int64_t most = (int64_t)num_sms * PER_SM, grid = tiles < most ? tiles : most;
  sample_tc_kernel<CHI, PER_SM><<<(unsigned)grid, tc::Cfg<CHI>::NT, sample_tc_smem<CHI>(a.L), st>>>(a);
  return cudaGetLastError();
}

bool sample_tc_supported(int CHI) { return CHI == 16 || CHI == 32; }

// Self-test of the bounded wait the sampler uses on its MMA completions: one CTA waits on an
// mbarrier of arrival count 1; with arrive != 0 one thread arrives first, otherwise nothing
// does and every wait must give up after `limit` polls and record ST_TIMEOUT.  The kernel
// returns normally either way.
__global__ void wait_probe_kernel(int arrive, long long limit, unsigned* status) {
  __shared__ __align__(8) uint64_t mbar;
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tc::su32(&mbar)), "r"(1));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (arrive && threadIdx.x == 0) {
    asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(tc::su32(&mbar)) : "memory");
  }
  __syncthreads();
  if (!tc::wait_parity(&mbar, 0u, limit)) set_status(status, ST_TIMEOUT);
}

cudaError_t launch_wait_probe(int arrive, long long limit, unsigned* status_dev, cudaStream_t st) {
  wait_probe_kernel<<<1, 32, 0, st>>>(arrive, limit, status_dev);
  return cudaGetLastError();
}

cudaError_t launch_sample_tc(const SampleArgs& a, int CHI, int num_sms, cudaStream_t st) {
  if (CHI == 32) return launch_tc_t<32, tc::Cfg<32>::PER_SM>(a, num_sms, st);
  if (CHI == 16) return launch_tc_t<16, tc::Cfg<16>::PER_SM>(a, num_sms, st);
  return cudaErrorInvalidValue;
}

}  // namespace tnmc
