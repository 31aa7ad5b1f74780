// Autoregressive proposals from the cached row environments (Sec. II.A Eq. approximate_bayes,
// Sec. II.B reverse-order sampling, Figs. fig:Z4 / fig:ZS4), and the same sweep with given
// spins (teacher forcing) for q(s) of arbitrary configurations.
//
// Two mappings with the same arithmetic, operation by operation (which product of a sum is rounded before
// it enters a fused multiply-add is written out in both), so that the choice between them changes no
// result.  sample_thread_kernel (CHI <= 16): one thread per proposal, the whole bond index in its
// registers, a warp's 32 proposals sharing the environment tile in shared memory.
// sample_kernel: one warp per proposal, lanes over the bond index; the CTA's warps are NW proposals of
// the same realization and share every environment tile, staged once per site into shared memory
// with cp.async double buffering.  For row r (fields h_c = beta Jv[r-1][c] s_{r-1,c}):
//   right sweep  c = L-1..0 : v_y = B[c]^y R_{c+1}(y), stored to the warp's workspace;
//                 R_c(y') = sum_y exp(beta Jh[r][c-1] s_y' s_y + h_c s_y) v_y (jointly normalised)
//   left sweep   c = 0..L-1 : w(y) = exp(h_c s_y + beta Jh[r][c-1] s_{c-1} s_y) (l . v_y),
//                 clamp w >= 0, q(+) = w+/(w+ + w-), s = +1 iff u < q(+) with u the Philox
//                 uniform of counter (r*L+c, step, chain, 1); log q accumulates in FP64;
//                 l <- l B[c]^s (normalised).
#include "common.cuh"
#include "kernels.h"

namespace tnmc {

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

template <typename T> __device__ __forceinline__ T tabs(T x) { return x < T(0) ? -x : x; }

// The draw s = +1 iff u < q(+), u = m 2^-53 with m the 53-bit Philox integer.
// FP64 path: compared in double.  FP32 paths: the same comparison done exactly in integers,
// m < ceil(q 2^53), so that no FP64 instruction runs per lane.
__device__ __forceinline__ uint64_t philox_m53(uint64_t seed, uint32_t c0, uint32_t c1, uint32_t c2) {
  const Philox4 o = philox4x32_10(c0, c1, c2, PURPOSE_SPIN, (uint32_t)seed, (uint32_t)(seed >> 32));
  return ((uint64_t)(o.x0 >> 5) << 26) | (uint64_t)(o.x1 >> 6);
}
__device__ __forceinline__ bool below(uint64_t m, double q) { return (double)m * (1.0 / 9007199254740992.0) < q; }
__device__ __forceinline__ bool below(uint64_t m, float q) {
  if (!(q > 0.0f)) return false;
  if (q >= 1.0f) return true;
  const uint32_t bits = __float_as_uint(q);
  const int e = (int)((bits >> 23) & 0xffu);
  const uint64_t mant = (e == 0) ? (uint64_t)(bits & 0x7fffffu) : (uint64_t)((bits & 0x7fffffu) | 0x800000u);
  const int sh = (e == 0 ? 1 : e) - 150 + 53;          // q 2^53 = mant 2^sh, sh <= 29 for q < 1
  uint64_t C;
  if (sh >= 0) C = mant << sh;
  else { const int k = -sh; C = (k >= 64) ? 1ull : ((mant + ((1ull << k) - 1ull)) >> k); }
  return m < C;
}
// log of the chosen conditional, accurate for q near 1 (log1p of the other branch)
__device__ __forceinline__ double log_q(double qs, double qo) { return qs > 0.5 ? log1p(-qo) : log(qs); }
__device__ __forceinline__ float log_q(float qs, float qo) { return qs > 0.5f ? log1pf(-qo) : logf(qs); }

// Rows of a staged tile as the compute type, four elements at a time.
__device__ __forceinline__ void row4(const float* p, float* v) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void row4(const double* p, double* v) {
  const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void row4(const __nv_bfloat16* p, float* v) {
  const uint2 t = *reinterpret_cast<const uint2*>(p);
  v[0] = __uint_as_float(t.x << 16); v[1] = __uint_as_float(t.x & 0xffff0000u);
  v[2] = __uint_as_float(t.y << 16); v[3] = __uint_as_float(t.y & 0xffff0000u);
}
__device__ __forceinline__ float tfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double tfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float tmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double tmul(double a, double b) { return __dmul_rn(a, b); }
// Larger of m >= 0 and |x|.  Doubles as integers, whose order is the same: the FP64 pipe is what the
// FP64 sweep waits for.
__device__ __forceinline__ float abs_max(float m, float x) { return fabsf(x) > m ? fabsf(x) : m; }
__device__ __forceinline__ double abs_max(double m, double x) {
  const long long a = __double_as_longlong(m), b = __double_as_longlong(x) & 0x7fffffffffffffffll;
  return __longlong_as_double(b > a && b <= 0x7ff0000000000000ll ? b : a);
}

constexpr int kThreadWarps = 8;       // warps of sample_thread_kernel in flight on an SM
constexpr int kThreadStages = 4;      // environment tiles in flight per warp

// One thread per proposal.  The warps are independent: each stages its own tiles (cp.async, four in
// flight) and takes its own 32 proposals.  Bond indices beyond the row's bond dimensions hold zeros and
// are left out, which at L = 8, chi = 16 is five sixths of the products.
// What bounds it: in FP64 the FP64 pipe (a warp's multiply-add takes 64 of a scheduler's cycles), which a
// lane per bond index left half empty at chi = 16 and busy with every proposal's logarithm and divisions
// 32 times over; in FP32 the chain of one site after the other (few proposals, up to four CTAs of
// sample_kernel per SM, are sample_kernel's).  One GB300, propose(): L = 8, chi = 16,
// 100 x 1000 proposals in FP64 62 -> 9.7 ms; L = 16, chi = 8, 64 x 400 in FP32 4.2 -> 0.77 ms.
template <typename T, typename TE, int CHI>
__global__ void __launch_bounds__(128, kThreadWarps / 4)
sample_thread_kernel(SampleArgs a, int n_slots) {
  constexpr int TILE = 2 * CHI * CHI, NS = kThreadStages;
  constexpr int CHUNKS = TILE * (int)sizeof(TE) / 16;
  const int L = a.L, N = L * L;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int words_row = (L + 31) / 32, LP = (L + 15) & ~15;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* mine = smem_raw + (size_t)warp * (NS * TILE * sizeof(TE) + 2 * LP + (size_t)words_row * 128);
  TE* stages = reinterpret_cast<TE*>(mine);
  int8_t* jh_s = reinterpret_cast<int8_t*>(stages + NS * TILE);
  int8_t* jv_s = jh_s + LP;
  uint32_t* prow = reinterpret_cast<uint32_t*>(jv_s + LP);      // [words_row][32]

  const int slot = blockIdx.x * 4 + warp;
  if (slot >= n_slots) return;
  const int tiles_per_real = (a.n_items + 31) / 32;
  const int64_t total = (int64_t)tiles_per_real * a.n_real;
  // v_y of every site of a row, [site][y][al][proposal]
  const bool own = slot < a.work_slots;
  T* work = reinterpret_cast<T*>(own ? a.work : a.more) + (size_t)(own ? slot : slot - a.work_slots) * L * 2 * CHI * 32 + lane;

  for (int64_t tile = slot; tile < total; tile += n_slots) {
    const int real = (int)(tile / tiles_per_real);
    const int k = (int)(tile % tiles_per_real) * 32 + lane;
    const bool valid = k < a.n_items;
    const int64_t item = (int64_t)real * a.n_items + k;
    const int chain = a.forced ? 0 : (a.chain_of ? a.chain_of[real] : k / a.n);
    const uint32_t step = (uint32_t)(a.step0 + (uint64_t)(a.forced ? 0 : k % a.n));
    const uint64_t seed = a.seeds[real];
    const double betad = a.beta[real];
    const T eb = (T)exp(betad), ebm = (T)exp(-betad);
    const int8_t* J = a.J + (size_t)real * 2 * L * (L - 1);
    const TE* envr = reinterpret_cast<const TE*>(a.env) + (size_t)real * L * L * TILE;
    const int8_t* forced = (a.forced && valid) ? a.forced + (size_t)item * N : nullptr;
    const int8_t* hf = a.hfield ? a.hfield + (size_t)real * N : nullptr;

    double logq = 0.0;          // FP64 total
    int energy = 0, magnet = 0;
    int64_t nclamp = 0;
    uint32_t word = 0;

    for (int r = 0; r < L; ++r) {
      __syncwarp();
      for (int c = lane; c < L - 1; c += 32) jh_s[c] = J[(size_t)r * (L - 1) + c];
      if (r > 0)
        for (int c = lane; c < L; c += 32) jv_s[c] = J[(size_t)L * (L - 1) + (size_t)(r - 1) * L + c];
      const TE* erow = envr + (size_t)r * L * TILE;
      const int* kd = a.kdim + ((size_t)real * L + r) * (L + 1);
      // product i of the row is at site L-1-i (right sweep), then at i-L (left sweep)
      auto copy = [&](int i) {
        if (i < 2 * L) {
          const TE* src = erow + (size_t)(i < L ? L - 1 - i : i - L) * TILE;
          TE* dst = stages + (i % NS) * TILE;
          for (int u = lane; u < CHUNKS; u += 32)
            cp_async16(reinterpret_cast<char*>(dst) + 16 * u, reinterpret_cast<const char*>(src) + 16 * u);
        }
        cp_async_commit();
      };
#pragma unroll
      for (int d = 0; d < NS - 1; ++d) copy(d);
      // the tile of product i is there; the one before it is done with, so its stage is refilled
      auto tile_of = [&](int i) -> const TE* {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(kThreadStages - 2) : "memory");
        __syncwarp();
        copy(i + NS - 1);
        return stages + (i % NS) * TILE;
      };

      // ---------------- right sweep ----------------
      T R0[CHI], R1[CHI];
#pragma unroll
      for (int j = 0; j < CHI; ++j) { R0[j] = j == 0 ? T(1) : T(0); R1[j] = R0[j]; }
      int kr = kd[L];
      for (int c = L - 1; c >= 0; --c) {
        const TE* tl = tile_of(L - 1 - c);
        const int kl = kd[c];
        // R_c(y') = sum_y exp(beta Jh s_y' s_y) exp(h_c s_y) v_y
        T s0 = 0, s1 = 0, d0 = 0, d1 = 0;
        if (c > 0) {
          const int jh = jh_s[c - 1];
          T f0 = 1, f1 = 1;                     // exp(h_c s_y) for y = 0 (+1), 1 (-1)
          if (r > 0) {
            const int sg = jv_s[c] * (((prow[(c >> 5) * 32 + lane] >> (c & 31)) & 1u) ? -1 : 1);
            f0 = sg > 0 ? eb : ebm; f1 = sg > 0 ? ebm : eb;
          }
          if (hf) { const int kh = hf[(size_t)r * L + c]; if (kh) { f0 *= num<T>::exp_((T)(betad * kh)); f1 *= num<T>::exp_((T)(-betad * kh)); } }
          const T same = jh > 0 ? eb : ebm, diff = jh > 0 ? ebm : eb;
          s0 = same * f0; s1 = same * f1; d0 = diff * f0; d1 = diff * f1;
        }
        T n0[CHI], n1[CHI], mx = 0;
        T* wsl = work + (size_t)c * 2 * CHI * 32;
#pragma unroll
        for (int al = 0; al < CHI; ++al) {
          n0[al] = T(0); n1[al] = T(0);
          if (al < kl) {
            // v_y[al], summed over be = al, al + 1, ... (cyclic)
            T b0[CHI], b1[CHI], v0 = 0, v1 = 0;
#pragma unroll
            for (int j = 0; j < CHI; j += 4)
              if (j < kr) { row4(tl + al * CHI + j, b0 + j); row4(tl + CHI * CHI + al * CHI + j, b1 + j); }
#pragma unroll
            for (int t = 0; t < CHI; ++t) {
              const int be = (al + t) & (CHI - 1);
              if ((be & ~3) < kr) { v0 = tfma(b0[be], R0[be], v0); v1 = tfma(b1[be], R1[be], v1); }
            }
            wsl[al * 32] = v0;
            wsl[(CHI + al) * 32] = v1;
            n0[al] = tfma(s0, v0, tmul(d1, v1));      // y' = +1
            n1[al] = tfma(d0, v0, tmul(s1, v1));      // y' = -1
            mx = abs_max(abs_max(mx, n0[al]), n1[al]);
          }
        }
        const T inv = mx > T(0) ? T(1) / mx : T(1);
#pragma unroll
        for (int al = 0; al < CHI; ++al) {
          R0[al] = al < kl ? n0[al] * inv : T(0);
          R1[al] = al < kl ? n1[al] * inv : T(0);
        }
        kr = kl;
      }

      // ---------------- left sweep ----------------
      T ell[CHI];
#pragma unroll
      for (int j = 0; j < CHI; ++j) ell[j] = j == 0 ? T(1) : T(0);
      int sprev = 0;
      T rsum = 0, rcomp = 0;      // compensated row sum of log q terms
      uint32_t rword = 0;
      int kl = kd[0];
      for (int c = 0; c < L; ++c) {
        const TE* tl = tile_of(L + c);
        const int kn = kd[c + 1];
        const T* wsl = work + (size_t)c * 2 * CHI * 32;
        // l . v_y, the products added as a butterfly over the bond index
        T p0[CHI], p1[CHI];
#pragma unroll
        for (int j = 0; j < CHI; ++j) {
          p0[j] = T(0); p1[j] = T(0);
          if (j < kl) { p0[j] = tmul(ell[j], wsl[j * 32]); p1[j] = tmul(ell[j], wsl[(CHI + j) * 32]); }
        }
#pragma unroll
        for (int o = CHI / 2; o > 0; o >>= 1)
          if (o < kl) {                       // the upper half is all zeros otherwise
#pragma unroll
            for (int j = 0; j < o; ++j) { p0[j] += p0[j + o]; p1[j] += p1[j + o]; }
          }
        T f0 = 1, f1 = 1;
        int sp = 0;
        if (r > 0) {
          sp = ((prow[(c >> 5) * 32 + lane] >> (c & 31)) & 1u) ? -1 : 1;
          const int sg = jv_s[c] * sp;
          f0 = sg > 0 ? eb : ebm; f1 = sg > 0 ? ebm : eb;
        }
        if (c > 0) { const int sg = jh_s[c - 1] * sprev; f0 *= sg > 0 ? eb : ebm; f1 *= sg > 0 ? ebm : eb; }
        if (hf) { const int kh = hf[(size_t)r * L + c]; if (kh) { f0 *= num<T>::exp_((T)(betad * kh)); f1 *= num<T>::exp_((T)(-betad * kh)); } }
        T w0 = f0 * p0[0], w1 = f1 * p1[0];
        if (w0 < T(0)) { w0 = 0; ++nclamp; }
        if (w1 < T(0)) { w1 = 0; ++nclamp; }
        const T tot = w0 + w1;
        int s;
        T qp = T(0.5), lqs;
        if (!(tot > T(0)) || !isfinite(tot)) {
          if (valid) {
            set_status(a.status, ST_NUMERIC);
            if (a.real_status) set_status(a.real_status + real, ST_NUMERIC);
          }
          // the realization is flagged; the spin is still drawn from the q = 1/2 it logs,
          // so that log q stays the probability the proposal was drawn with
          if (forced) s = forced[(size_t)r * L + c];
          else s = (philox_m53(seed, (uint32_t)(r * L + c), step, (uint32_t)chain) < (1ull << 52)) ? 1 : -1;
          lqs = T(-0.6931471805599453);
        } else {
          qp = w0 / tot;
          const T qm = w1 / tot;
          if (forced) s = forced[(size_t)r * L + c];
          else s = below(philox_m53(seed, (uint32_t)(r * L + c), step, (uint32_t)chain), qp) ? 1 : -1;
          lqs = (s == 1) ? log_q(qp, qm) : log_q(qm, qp);
        }
        {   // Kahan: the row's log q terms summed with FP64-grade accuracy in the compute type
          const T yk = lqs - rcomp;
          const T tk = rsum + yk;
          rcomp = (tk - rsum) - yk;
          rsum = tk;
        }
        if (a.qplus && valid) a.qplus[(size_t)item * N + (size_t)r * L + c] = (double)qp;
        // l <- l B^s
        const TE* bs = tl + (s == 1 ? 0 : CHI * CHI);
        T acc[CHI];
#pragma unroll
        for (int j = 0; j < CHI; ++j) acc[j] = T(0);
#pragma unroll
        for (int t = 0; t < CHI; ++t)
          if (t < kl) {
#pragma unroll
            for (int j = 0; j < CHI; j += 4)
              if (j < kn) {
                T b[4];
                row4(bs + t * CHI + j, b);
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[j + e] = tfma(ell[t], b[e], acc[j + e]);
              }
          }
        T mx = 0;
#pragma unroll
        for (int j = 0; j < CHI; ++j) if ((j & ~3) < kn) mx = abs_max(mx, acc[j]);
#pragma unroll
        for (int j = 0; j < CHI; ++j) {
          ell[j] = acc[j];
          if (j < kn && mx > T(0)) ell[j] = acc[j] / mx;
        }
        kl = kn;
        // energy and magnetisation (Eq. E)
        if (c > 0) energy -= jh_s[c - 1] * sprev * s;
        if (r > 0) energy -= jv_s[c] * sp * s;
        magnet += s;
        sprev = s;
        if (s < 0) rword |= 1u << (c & 31);
        // the previous row's word has been read to its end
        if ((c & 31) == 31 || c == L - 1) { prow[(c >> 5) * 32 + lane] = rword; rword = 0; }
        const int site = r * L + c;
        if (s < 0) word |= 1u << (site & 31);
        if ((site & 31) == 31 || site == N - 1) {
          if (valid && a.spins_packed) a.spins_packed[(size_t)item * a.words + (site >> 5)] = word;
          word = 0;
        }
      }
      logq += (double)rsum;
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    if (valid) {
      if (a.logq) a.logq[item] = logq;
      if (a.energy) a.energy[item] = energy;
      if (a.magnet) a.magnet[item] = magnet;
      if (a.clamps && nclamp) atomicAdd(reinterpret_cast<unsigned long long*>(a.clamps + real),
                                        (unsigned long long)nclamp);
    }
  }
}

template <typename T, typename TE, int CHI, int NW>
__global__ void __launch_bounds__(32 * NW)
sample_kernel(SampleArgs a) {
  constexpr int TILE = 2 * CHI * CHI;
  constexpr int NT = 32 * NW;
  constexpr int CHUNKS = TILE * (int)sizeof(TE) / 16;
  const int L = a.L, N = L * L;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int al = lane & (CHI - 1);            // bond index handled by this lane
  const bool active_lane = lane < CHI;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  TE* stage0 = reinterpret_cast<TE*>(smem_raw);
  TE* stage1 = stage0 + TILE;
  int8_t* jh_s = reinterpret_cast<int8_t*>(stage1 + TILE);   // L
  int8_t* jv_s = jh_s + L;                                    // L
  int8_t* rows = jv_s + L;                                    // [NW][2][L]

  const int tiles_per_real = (a.n_items + NW - 1) / NW;
  const int64_t total = (int64_t)tiles_per_real * a.n_real;
  T* work = reinterpret_cast<T*>(a.work) + ((size_t)blockIdx.x * NW + warp) * (size_t)L * 2 * CHI;

  for (int64_t tile = blockIdx.x; tile < total; tile += gridDim.x) {
    const int real = (int)(tile / tiles_per_real);
    const int k = (int)(tile % tiles_per_real) * NW + warp;
    const bool valid = k < a.n_items;
    const int64_t item = (int64_t)real * a.n_items + k;
    const int chain = a.forced ? 0 : (a.chain_of ? a.chain_of[real] : k / a.n);
    const uint32_t step = (uint32_t)(a.step0 + (uint64_t)(a.forced ? 0 : k % a.n));
    const uint64_t seed = a.seeds[real];
    const double betad = a.beta[real];
    const T eb = (T)exp(betad), ebm = (T)exp(-betad);
    const int8_t* J = a.J + (size_t)real * 2 * L * (L - 1);
    const TE* envr = reinterpret_cast<const TE*>(a.env) + (size_t)real * L * L * TILE;
    int8_t* prow = rows + (size_t)warp * 2 * L;      // previous row spins
    int8_t* crow = prow + L;                          // current row spins
    const int8_t* forced = (a.forced && valid) ? a.forced + (size_t)item * N : nullptr;
    const int8_t* hf = a.hfield ? a.hfield + (size_t)real * N : nullptr;

    double logq = 0.0;          // FP64 total
    int energy = 0, magnet = 0;
    int64_t nclamp = 0;
    uint32_t word = 0;

    for (int r = 0; r < L; ++r) {
      __syncthreads();   // previous users of jh_s/jv_s/rows are done
      for (int c = tid; c < L - 1; c += NT) jh_s[c] = J[(size_t)r * (L - 1) + c];
      if (r > 0)
        for (int c = tid; c < L; c += NT) jv_s[c] = J[(size_t)L * (L - 1) + (size_t)(r - 1) * L + c];
      const TE* erow = envr + (size_t)r * L * TILE;

      // ---------------- right sweep ----------------
      T R0 = (al == 0 && active_lane) ? T(1) : T(0), R1 = R0;   // R_L(y) for y = 0, 1
      for (int i = tid; i < CHUNKS; i += NT) cp_async16(reinterpret_cast<char*>(stage0) + 16 * i,
                                                        reinterpret_cast<const char*>(erow + (size_t)(L - 1) * TILE) + 16 * i);
      cp_async_commit();
      for (int ci = 0; ci < L; ++ci) {
        const int c = L - 1 - ci;
        cp_async_wait_all();
        __syncthreads();
        const TE* tl = (ci & 1) ? stage1 : stage0;
        if (ci + 1 < L) {
          TE* nx = (ci & 1) ? stage0 : stage1;
          for (int i = tid; i < CHUNKS; i += NT) cp_async16(reinterpret_cast<char*>(nx) + 16 * i,
                                                            reinterpret_cast<const char*>(erow + (size_t)(c - 1) * TILE) + 16 * i);
          cp_async_commit();
        }
        // v_y[al] = sum_be B^y[al][be] R(y)[be]  (diagonal order: conflict-free smem reads)
        T v0 = 0, v1 = 0;
#pragma unroll 8
        for (int t = 0; t < CHI; ++t) {
          const int be = (al + t) & (CHI - 1);
          const T r0 = __shfl_sync(0xffffffffu, R0, be);
          const T r1 = __shfl_sync(0xffffffffu, R1, be);
          v0 = tfma(env_load<T, TE>(tl[al * CHI + be]), r0, v0);
          v1 = tfma(env_load<T, TE>(tl[CHI * CHI + al * CHI + be]), r1, v1);
        }
        if (!active_lane) { v0 = 0; v1 = 0; }
        if (active_lane) { work[(size_t)c * 2 * CHI + al] = v0; work[(size_t)c * 2 * CHI + CHI + al] = v1; }
        if (c > 0) {
          // R_c(y') = sum_y exp(beta Jh s_y' s_y) exp(h_c s_y) v_y
          const int jh = jh_s[c - 1];
          T f0 = 1, f1 = 1;                     // exp(h_c s_y) for y = 0 (+1), 1 (-1)
          if (r > 0) { const int sg = jv_s[c] * prow[c]; f0 = sg > 0 ? eb : ebm; f1 = sg > 0 ? ebm : eb; }
          if (hf) { const int kh = hf[(size_t)r * L + c]; if (kh) { f0 *= num<T>::exp_((T)(betad * kh)); f1 *= num<T>::exp_((T)(-betad * kh)); } }
          const T same = jh > 0 ? eb : ebm, diff = jh > 0 ? ebm : eb;
          const T n0 = tfma(same * f0, v0, tmul(diff * f1, v1));   // y' = +1
          const T n1 = tfma(diff * f0, v0, tmul(same * f1, v1));   // y' = -1
          T mx = tabs(n0) > tabs(n1) ? tabs(n0) : tabs(n1);
          mx = warp_max(mx);
          const T inv = mx > T(0) ? T(1) / mx : T(1);
          R0 = n0 * inv; R1 = n1 * inv;
        }
      }
      __syncwarp();

      // ---------------- left sweep ----------------
      T ell = (al == 0 && active_lane) ? T(1) : T(0);
      int sprev = 0;
      T rsum = 0, rcomp = 0;      // compensated row sum of log q terms
      for (int i = tid; i < CHUNKS; i += NT) cp_async16(reinterpret_cast<char*>(stage0) + 16 * i,
                                                        reinterpret_cast<const char*>(erow) + 16 * i);
      cp_async_commit();
      for (int c = 0; c < L; ++c) {
        cp_async_wait_all();
        __syncthreads();
        const TE* tl = (c & 1) ? stage1 : stage0;
        if (c + 1 < L) {
          TE* nx = (c & 1) ? stage0 : stage1;
          for (int i = tid; i < CHUNKS; i += NT) cp_async16(reinterpret_cast<char*>(nx) + 16 * i,
                                                            reinterpret_cast<const char*>(erow + (size_t)(c + 1) * TILE) + 16 * i);
          cp_async_commit();
        }
        const T v0 = active_lane ? work[(size_t)c * 2 * CHI + al] : T(0);
        const T v1 = active_lane ? work[(size_t)c * 2 * CHI + CHI + al] : T(0);
        T d0 = warp_sum(tmul(ell, v0)), d1 = warp_sum(tmul(ell, v1));
        T f0 = 1, f1 = 1;
        if (r > 0) { const int sg = jv_s[c] * prow[c]; f0 = sg > 0 ? eb : ebm; f1 = sg > 0 ? ebm : eb; }
        if (c > 0) { const int sg = jh_s[c - 1] * sprev; f0 *= sg > 0 ? eb : ebm; f1 *= sg > 0 ? ebm : eb; }
        if (hf) { const int kh = hf[(size_t)r * L + c]; if (kh) { f0 *= num<T>::exp_((T)(betad * kh)); f1 *= num<T>::exp_((T)(-betad * kh)); } }
        T w0 = f0 * d0, w1 = f1 * d1;
        if (w0 < T(0)) { w0 = 0; ++nclamp; }
        if (w1 < T(0)) { w1 = 0; ++nclamp; }
        const T tot = w0 + w1;
        int s;
        T qp = T(0.5), lqs;
        if (!(tot > T(0)) || !isfinite(tot)) {
          if (lane == 0 && valid) {
            set_status(a.status, ST_NUMERIC);
            if (a.real_status) set_status(a.real_status + real, ST_NUMERIC);
          }
          // the realization is flagged; the spin is still drawn from the q = 1/2 it logs,
          // so that log q stays the probability the proposal was drawn with
          if (forced) s = forced[(size_t)r * L + c];
          else s = (philox_m53(seed, (uint32_t)(r * L + c), step, (uint32_t)chain) < (1ull << 52)) ? 1 : -1;
          lqs = T(-0.6931471805599453);
        } else {
          qp = w0 / tot;
          const T qm = w1 / tot;
          if (forced) {
            s = forced[(size_t)r * L + c];
          } else {
            s = below(philox_m53(seed, (uint32_t)(r * L + c), step, (uint32_t)chain), qp) ? 1 : -1;
          }
          lqs = (s == 1) ? log_q(qp, qm) : log_q(qm, qp);
        }
        {   // Kahan: the row's log q terms summed with FP64-grade accuracy in the compute type
          const T yk = lqs - rcomp;
          const T tk = rsum + yk;
          rcomp = (tk - rsum) - yk;
          rsum = tk;
        }
        if (a.qplus && valid && lane == 0) a.qplus[(size_t)item * N + (size_t)r * L + c] = (double)qp;
        // l <- l B^s
        const TE* bs = tl + (s == 1 ? 0 : CHI * CHI);
        T acc = 0;
#pragma unroll 8
        for (int t = 0; t < CHI; ++t) {
          const T lt = __shfl_sync(0xffffffffu, ell, t);
          acc = tfma(lt, env_load<T, TE>(bs[t * CHI + al]), acc);
        }
        if (!active_lane) acc = 0;
        T mx = warp_max(tabs(acc));
        ell = mx > T(0) ? acc / mx : acc;
        // energy and magnetisation (Eq. E)
        if (c > 0) energy -= jh_s[c - 1] * sprev * s;
        if (r > 0) energy -= jv_s[c] * prow[c] * s;
        magnet += s;
        if (lane == 0) crow[c] = (int8_t)s;
        sprev = s;
        const int site = r * L + c;
        if (s < 0) word |= 1u << (site & 31);
        if ((site & 31) == 31 || site == N - 1) {
          if (lane == 0 && valid && a.spins_packed) a.spins_packed[(size_t)item * a.words + (site >> 5)] = word;
          word = 0;
        }
      }
      logq += (double)rsum;
      __syncwarp();
      for (int c = lane; c < L; c += 32) prow[c] = crow[c];
      __syncwarp();
    }
    if (lane == 0 && valid) {
      if (a.logq) a.logq[item] = logq;
      if (a.energy) a.energy[item] = energy;
      if (a.magnet) a.magnet[item] = magnet;
      if (a.clamps && nclamp) atomicAdd(reinterpret_cast<unsigned long long*>(a.clamps + real),
                                        (unsigned long long)nclamp);
    }
  }
}

// The same sweep for CHI = 64 (bond indices lane and lane + 32 on each lane).
template <typename T, typename TE, int CHI, int NW>
__global__ void __launch_bounds__(32 * NW)
sample_kernel_wide(SampleArgs a) {
  constexpr int E = CHI / 32;                 // bond indices per lane: lane + 32 e
  constexpr int TILE = 2 * CHI * CHI;
  constexpr int NT = 32 * NW;
  constexpr int CHUNKS = TILE * (int)sizeof(TE) / 16;
  const int L = a.L, N = L * L;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  TE* stage0 = reinterpret_cast<TE*>(smem_raw);
  TE* stage1 = stage0 + TILE;
  int8_t* jh_s = reinterpret_cast<int8_t*>(stage1 + TILE);   // L
  int8_t* jv_s = jh_s + L;                                    // L
  int8_t* rows = jv_s + L;                                    // [NW][2][L]

  const int tiles_per_real = (a.n_items + NW - 1) / NW;
  const int64_t total = (int64_t)tiles_per_real * a.n_real;
  T* work = reinterpret_cast<T*>(a.work) + ((size_t)blockIdx.x * NW + warp) * (size_t)L * 2 * CHI;

  for (int64_t tile = blockIdx.x; tile < total; tile += gridDim.x) {
    const int real = (int)(tile / tiles_per_real);
    const int k = (int)(tile % tiles_per_real) * NW + warp;
    const bool valid = k < a.n_items;
    const int64_t item = (int64_t)real * a.n_items + k;
    const int chain = a.forced ? 0 : (a.chain_of ? a.chain_of[real] : k / a.n);
    const uint32_t step = (uint32_t)(a.step0 + (uint64_t)(a.forced ? 0 : k % a.n));
    const uint64_t seed = a.seeds[real];
    const double betad = a.beta[real];
    const T eb = (T)exp(betad), ebm = (T)exp(-betad);
    const int8_t* J = a.J + (size_t)real * 2 * L * (L - 1);
    const TE* envr = reinterpret_cast<const TE*>(a.env) + (size_t)real * L * L * TILE;
    int8_t* prow = rows + (size_t)warp * 2 * L;      // previous row spins
    int8_t* crow = prow + L;                          // current row spins
    const int8_t* forced = (a.forced && valid) ? a.forced + (size_t)item * N : nullptr;
    const int8_t* hf = a.hfield ? a.hfield + (size_t)real * N : nullptr;

    double logq = 0.0;          // FP64 total
    int energy = 0, magnet = 0;
    int64_t nclamp = 0;
    uint32_t word = 0;

    for (int r = 0; r < L; ++r) {
      __syncthreads();   // previous users of jh_s/jv_s/rows are done
      for (int c = tid; c < L - 1; c += NT) jh_s[c] = J[(size_t)r * (L - 1) + c];
      if (r > 0)
        for (int c = tid; c < L; c += NT) jv_s[c] = J[(size_t)L * (L - 1) + (size_t)(r - 1) * L + c];
      const TE* erow = envr + (size_t)r * L * TILE;

      // ---------------- right sweep ----------------
      T R0[E], R1[E];                                   // R_L(y) for y = 0, 1
#pragma unroll
      for (int e = 0; e < E; ++e) { R0[e] = (lane == 0 && e == 0) ? T(1) : T(0); R1[e] = R0[e]; }
      for (int i = tid; i < CHUNKS; i += NT) cp_async16(reinterpret_cast<char*>(stage0) + 16 * i,
                                                        reinterpret_cast<const char*>(erow + (size_t)(L - 1) * TILE) + 16 * i);
      cp_async_commit();
      for (int ci = 0; ci < L; ++ci) {
        const int c = L - 1 - ci;
        cp_async_wait_all();
        __syncthreads();
        const TE* tl = (ci & 1) ? stage1 : stage0;
        if (ci + 1 < L) {
          TE* nx = (ci & 1) ? stage0 : stage1;
          for (int i = tid; i < CHUNKS; i += NT) cp_async16(reinterpret_cast<char*>(nx) + 16 * i,
                                                            reinterpret_cast<const char*>(erow + (size_t)(c - 1) * TILE) + 16 * i);
          cp_async_commit();
        }
        // v_y[al] = sum_be B^y[al][be] R(y)[be] for al = lane + 32 e (diagonal order within
        // each half of be: conflict-free smem reads)
        T v0[E], v1[E];
#pragma unroll
        for (int e = 0; e < E; ++e) { v0[e] = 0; v1[e] = 0; }
#pragma unroll
        for (int h = 0; h < E; ++h) {
#pragma unroll 8
          for (int t = 0; t < 32; ++t) {
            const int j = (lane + t) & 31, be = 32 * h + j;
            const T r0 = __shfl_sync(0xffffffffu, R0[h], j);
            const T r1 = __shfl_sync(0xffffffffu, R1[h], j);
#pragma unroll
            for (int e = 0; e < E; ++e) {
              const int al = lane + 32 * e;
              v0[e] += env_load<T, TE>(tl[al * CHI + be]) * r0;
              v1[e] += env_load<T, TE>(tl[CHI * CHI + al * CHI + be]) * r1;
            }
          }
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
          work[(size_t)c * 2 * CHI + lane + 32 * e] = v0[e];
          work[(size_t)c * 2 * CHI + CHI + lane + 32 * e] = v1[e];
        }
        if (c > 0) {
          // R_c(y') = sum_y exp(beta Jh s_y' s_y) exp(h_c s_y) v_y
          const int jh = jh_s[c - 1];
          T f0 = 1, f1 = 1;                     // exp(h_c s_y) for y = 0 (+1), 1 (-1)
          if (r > 0) { const int sg = jv_s[c] * prow[c]; f0 = sg > 0 ? eb : ebm; f1 = sg > 0 ? ebm : eb; }
          if (hf) { const int kh = hf[(size_t)r * L + c]; if (kh) { f0 *= num<T>::exp_((T)(betad * kh)); f1 *= num<T>::exp_((T)(-betad * kh)); } }
          const T same = jh > 0 ? eb : ebm, diff = jh > 0 ? ebm : eb;
          T n0[E], n1[E], mx = 0;
#pragma unroll
          for (int e = 0; e < E; ++e) {
            n0[e] = same * f0 * v0[e] + diff * f1 * v1[e];   // y' = +1
            n1[e] = diff * f0 * v0[e] + same * f1 * v1[e];   // y' = -1
            mx = tabs(n0[e]) > mx ? tabs(n0[e]) : mx;
            mx = tabs(n1[e]) > mx ? tabs(n1[e]) : mx;
          }
          mx = warp_max(mx);
          const T inv = mx > T(0) ? T(1) / mx : T(1);
#pragma unroll
          for (int e = 0; e < E; ++e) { R0[e] = n0[e] * inv; R1[e] = n1[e] * inv; }
        }
      }
      __syncwarp();

      // ---------------- left sweep ----------------
      T ell[E];
#pragma unroll
      for (int e = 0; e < E; ++e) ell[e] = (lane == 0 && e == 0) ? T(1) : T(0);
      int sprev = 0;
      T rsum = 0, rcomp = 0;      // compensated row sum of log q terms
      for (int i = tid; i < CHUNKS; i += NT) cp_async16(reinterpret_cast<char*>(stage0) + 16 * i,
                                                        reinterpret_cast<const char*>(erow) + 16 * i);
      cp_async_commit();
      for (int c = 0; c < L; ++c) {
        cp_async_wait_all();
        __syncthreads();
        const TE* tl = (c & 1) ? stage1 : stage0;
        if (c + 1 < L) {
          TE* nx = (c & 1) ? stage0 : stage1;
          for (int i = tid; i < CHUNKS; i += NT) cp_async16(reinterpret_cast<char*>(nx) + 16 * i,
                                                            reinterpret_cast<const char*>(erow + (size_t)(c + 1) * TILE) + 16 * i);
          cp_async_commit();
        }
        T p0 = 0, p1 = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          p0 += ell[e] * work[(size_t)c * 2 * CHI + lane + 32 * e];
          p1 += ell[e] * work[(size_t)c * 2 * CHI + CHI + lane + 32 * e];
        }
        T d0 = warp_sum(p0), d1 = warp_sum(p1);
        T f0 = 1, f1 = 1;
        if (r > 0) { const int sg = jv_s[c] * prow[c]; f0 = sg > 0 ? eb : ebm; f1 = sg > 0 ? ebm : eb; }
        if (c > 0) { const int sg = jh_s[c - 1] * sprev; f0 *= sg > 0 ? eb : ebm; f1 *= sg > 0 ? ebm : eb; }
        if (hf) { const int kh = hf[(size_t)r * L + c]; if (kh) { f0 *= num<T>::exp_((T)(betad * kh)); f1 *= num<T>::exp_((T)(-betad * kh)); } }
        T w0 = f0 * d0, w1 = f1 * d1;
        if (w0 < T(0)) { w0 = 0; ++nclamp; }
        if (w1 < T(0)) { w1 = 0; ++nclamp; }
        const T tot = w0 + w1;
        int s;
        T qp = T(0.5), lqs;
        if (!(tot > T(0)) || !isfinite(tot)) {
          if (lane == 0 && valid) {
            set_status(a.status, ST_NUMERIC);
            if (a.real_status) set_status(a.real_status + real, ST_NUMERIC);
          }
          // the realization is flagged; the spin is still drawn from the q = 1/2 it logs,
          // so that log q stays the probability the proposal was drawn with
          if (forced) s = forced[(size_t)r * L + c];
          else s = (philox_m53(seed, (uint32_t)(r * L + c), step, (uint32_t)chain) < (1ull << 52)) ? 1 : -1;
          lqs = T(-0.6931471805599453);
        } else {
          qp = w0 / tot;
          const T qm = w1 / tot;
          if (forced) {
            s = forced[(size_t)r * L + c];
          } else {
            s = below(philox_m53(seed, (uint32_t)(r * L + c), step, (uint32_t)chain), qp) ? 1 : -1;
          }
          lqs = (s == 1) ? log_q(qp, qm) : log_q(qm, qp);
        }
        {   // Kahan: the row's log q terms summed with FP64-grade accuracy in the compute type
          const T yk = lqs - rcomp;
          const T tk = rsum + yk;
          rcomp = (tk - rsum) - yk;
          rsum = tk;
        }
        if (a.qplus && valid && lane == 0) a.qplus[(size_t)item * N + (size_t)r * L + c] = (double)qp;
        // l <- l B^s
        const TE* bs = tl + (s == 1 ? 0 : CHI * CHI);
        T acc[E];
#pragma unroll
        for (int e = 0; e < E; ++e) acc[e] = 0;
#pragma unroll
        for (int h = 0; h < E; ++h) {
#pragma unroll 8
          for (int j = 0; j < 32; ++j) {
            const T lt = __shfl_sync(0xffffffffu, ell[h], j);
            const int t = 32 * h + j;
#pragma unroll
            for (int e = 0; e < E; ++e) acc[e] += lt * env_load<T, TE>(bs[t * CHI + lane + 32 * e]);
          }
        }
        T mx = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) mx = tabs(acc[e]) > mx ? tabs(acc[e]) : mx;
        mx = warp_max(mx);
#pragma unroll
        for (int e = 0; e < E; ++e) ell[e] = mx > T(0) ? acc[e] / mx : acc[e];
        // energy and magnetisation (Eq. E)
        if (c > 0) energy -= jh_s[c - 1] * sprev * s;
        if (r > 0) energy -= jv_s[c] * prow[c] * s;
        magnet += s;
        if (lane == 0) crow[c] = (int8_t)s;
        sprev = s;
        const int site = r * L + c;
        if (s < 0) word |= 1u << (site & 31);
        if ((site & 31) == 31 || site == N - 1) {
          if (lane == 0 && valid && a.spins_packed) a.spins_packed[(size_t)item * a.words + (site >> 5)] = word;
          word = 0;
        }
      }
      logq += (double)rsum;
      __syncwarp();
      for (int c = lane; c < L; c += 32) prow[c] = crow[c];
      __syncwarp();
    }
    if (lane == 0 && valid) {
      if (a.logq) a.logq[item] = logq;
      if (a.energy) a.energy[item] = energy;
      if (a.magnet) a.magnet[item] = magnet;
      if (a.clamps && nclamp) atomicAdd(reinterpret_cast<unsigned long long*>(a.clamps + real),
                                        (unsigned long long)nclamp);
    }
  }
}

template <int CHI, int NW>
static size_t sample_smem(int L, size_t te) {
  return 2 * (size_t)(2 * CHI * CHI) * te + 2 * (size_t)L + (size_t)NW * 2 * L + 16;
}

constexpr int kSampleWarps = 8;

// Warps of sample_thread_kernel with a workspace of their own: kThreadWarps per SM, fewer where that
// would take more than 256 MB, but never less than one per SM (32 proposals, as many as sample_kernel
// has in flight).  One per SM is what every context has (a.work); the others are allocated at the first call
// that this kernel serves with more, so that contexts of few proposals do not hold them.
template <typename T>
static int thread_slots(int L, int CHI, int num_sms) {
  const size_t per_warp = (size_t)L * 2 * CHI * 32 * sizeof(T), cap = (size_t)256 << 20;
  size_t slots = (size_t)num_sms * kThreadWarps;
  if (slots * per_warp > cap) slots = cap / per_warp;
  return (int)(slots < (size_t)num_sms ? (size_t)num_sms : slots);
}

// Whether one thread per proposal serves a call, with this many slots: from a number of proposals on; below
// it, too few warps are in flight and one thread's chain over the bond index is what the call waits for.
// Its time is the same for any number that the slots hold at once, that of the other kernel goes by the CTAs
// (eight proposals of a realization each) that an SM gets.  propose() at L = 16, one GB300, ms of this kernel
// (first) and of the other one at 1, 2 and 4 CTAs per SM:
//   FP32 chi = 4  0.39 | 0.40 0.49 0.75     FP64 chi = 4   2.7 | 2.5 4.8  9.6
//   FP32 chi = 8  0.67 | 0.42 0.49 0.79     FP64 chi = 8   4.9 | 2.7 5.2 13.0
//   FP32 chi = 16 1.40 | 0.47 0.59 1.00     FP64 chi = 16 10.8 | 3.1 6.0 15.1
// (BF16 as FP32; beyond 4 the other kernel's grow in proportion).  The line is drawn where this kernel is the
// faster one in propose() and in eval_conditionals().  With more tiles than slots (large L, or without the
// further slots) each further pass over the slots costs as much again.
template <typename T>
static bool takes_threads(int CHI, int num_sms, int n_items, int n_real, int64_t slots) {
  if (CHI > 16) return false;
  const int limit = sizeof(T) == 4 ? (CHI == 4 ? 1 : 4) : (CHI == 16 ? 3 : 1);
  const int64_t ctas = (int64_t)((n_items + kSampleWarps - 1) / kSampleWarps) * n_real;
  const int64_t tiles = (int64_t)((n_items + 31) / 32) * n_real, passes = (tiles + slots - 1) / slots;
  return ctas > (passes > 1 ? 4 * passes : limit) * num_sms;
}

template <typename T, typename TE, int CHI>
static cudaError_t launch_sample_thread(SampleArgs a, int64_t slots, int num_sms, cudaStream_t st) {
  const size_t smem = 4 * ((size_t)kThreadStages * 2 * CHI * CHI * sizeof(TE) + 2 * (size_t)((a.L + 15) & ~15) +
                           (size_t)((a.L + 31) / 32) * 128);
  cudaError_t e = allow_shared_memory<sample_thread_kernel<T, TE, CHI>>();
  if (e != cudaSuccess) return e;
  const int64_t tiles = (int64_t)((a.n_items + 31) / 32) * a.n_real;
  if (slots > tiles) slots = tiles;
  a.work_slots = num_sms;
  sample_thread_kernel<T, TE, CHI><<<(unsigned)((slots + 3) / 4), 128, smem, st>>>(a, (int)slots);
  return cudaGetLastError();
}

template <typename T, typename TE, int CHI>
static cudaError_t launch_sample_t(const SampleArgs& a, int num_sms, cudaStream_t st) {
  constexpr int NW = kSampleWarps;
  if constexpr (CHI <= 16) {
    const int64_t slots = a.more ? thread_slots<T>(a.L, CHI, num_sms) : num_sms;
    if (takes_threads<T>(CHI, num_sms, a.n_items, a.n_real, slots)) return launch_sample_thread<T, TE, CHI>(a, slots, num_sms, st);
  }
  const size_t smem = sample_smem<CHI, NW>(a.L, sizeof(TE));
  constexpr auto kern = [] {
    if constexpr (CHI > 32) return &sample_kernel_wide<T, TE, CHI, NW>;
    else return &sample_kernel<T, TE, CHI, NW>;
  }();
  cudaError_t e = allow_shared_memory<kern>();
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * NW, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  if (per_sm > 4) per_sm = 4;
  const int64_t tiles = (int64_t)((a.n_items + NW - 1) / NW) * a.n_real;
  int64_t grid = (int64_t)num_sms * per_sm;
  if (grid > tiles) grid = tiles;
  if (grid < 1) grid = 1;
  kern<<<(unsigned)grid, 32 * NW, smem, st>>>(a);
  return cudaGetLastError();
}

SampleWork sample_work(int L, int CHI, int precision, int num_sms, int n_items, int n_real) {
  const size_t slot = (size_t)L * 2 * CHI * 32 * (precision == 0 ? 8 : 4);
  static_assert(4 * kSampleWarps == 32, "sample_kernel has one slot of 32 proposals per SM");
  SampleWork w{(size_t)num_sms * slot, 0, false, false};
  if (CHI <= 16) {
    const int slots = precision == 0 ? thread_slots<double>(L, CHI, num_sms) : thread_slots<float>(L, CHI, num_sms);
    const int64_t tiles = (int64_t)((n_items + 31) / 32) * n_real;
    w.more = (size_t)(slots - num_sms) * slot;
    auto takes = [&](int64_t n_slots) {
      return w.more > 0 && tiles > num_sms &&
             (precision == 0 ? takes_threads<double>(CHI, num_sms, n_items, n_real, n_slots)
                             : takes_threads<float>(CHI, num_sms, n_items, n_real, n_slots));
    };
    w.takes_more = takes(slots);
    w.up_to = takes(tiles);               // as if one pass held them, which it does for some smaller call
  }
  return w;
}

cudaError_t launch_sample(const SampleArgs& a, int precision, int CHI, int num_sms, cudaStream_t st) {
#define TNMC_SAMPLE_CASE(T, TE)                                        \
  switch (CHI) {                                                       \
    case 4: return launch_sample_t<T, TE, 4>(a, num_sms, st);          \
    case 8: return launch_sample_t<T, TE, 8>(a, num_sms, st);          \
    case 16: return launch_sample_t<T, TE, 16>(a, num_sms, st);        \
    case 32: return launch_sample_t<T, TE, 32>(a, num_sms, st);        \
    case 64: return launch_sample_t<T, TE, 64>(a, num_sms, st);        \
    default: return cudaErrorInvalidValue;                             \
  }
  if (precision == 0) {
    if (CHI > 32) return cudaErrorInvalidValue;     // the FP64 build stops at CHI = 32
    TNMC_SAMPLE_CASE(double, double)
  }
  if (precision == 2) { TNMC_SAMPLE_CASE(float, __nv_bfloat16) }
  TNMC_SAMPLE_CASE(float, float)
#undef TNMC_SAMPLE_CASE
}

}  // namespace tnmc
