// Boundary-MPS row environments (Sec. II.B of arXiv 2409.06538) on sm_103a.
//
// For every realization (one CTA each) and every row r = L-2 .. 0:
//   A[c] = O_r[c] . Gt_{r+1}[c]  -- the row-transfer MPO (bond 2: the T tensors, copy tensor
//          with the right and bottom Boltzmann matrices absorbed) applied to the cached MPS;
//          A[c]^x_{(a,al),(b,be)} = W(x,a,b) B[c]^b_{al,be},
//          W(x,a,b) = exp(beta Jv[r][c] s_x s_b) * exp(beta Jh[r+1][c-1] s_a s_b)   (c > 0),
//          the right MPO bond b of the last site summed.
//   forward sweep  c = 0..L-2 : R_{c+1} = R-factor of [R_c A[c]^{x=0}; R_c A[c]^{x=1}]
//          (Householder; R_c^T R_c is the Gram matrix of the left part, so the left part is
//          represented without squaring its condition number);
//   backward sweep c = L-1..1 : M = A[c] contracted with the already-truncated right part,
//          Y = R_c M has the singular values and right singular vectors of the state cut
//          before site c (the left part is Q_{<c} R_c with Q an isometry).  Its SVD: two
//          Householder QRs (Y = Q1 R1, R1^T = Q2 R2) and a one-sided (Hestenes) Jacobi on R2^T,
//          V = Q2 Z (the QR-preconditioned one-sided Jacobi of Drmac and Veselic); the top
//          k = min(chi, d_c, 2 k_{c+1}) right singular vectors V give B_r[c] = V^T
//          (right-canonical), P = M V carries the rest of the state to site c-1.  Site 0 keeps
//          the normalised remainder; lam_r = log of the removed scale.
// This is the QR-sweep + truncating-SVD-sweep compression of the oracle, computed without
// forming Q: the truncated MPS is the same up to gauge (and rounding).
// Zip-up mode (args.zipup, a compression variant): no forward sweep and Y = M, the Jacobi on M
// itself (graded by columns); the rows alternate their sweep direction, a left-to-right row
// running as this backward sweep over the mirrored row (frame site f = lattice site L-1-f,
// bonds swapped, horizontal bond factors at the bond's right site).
#include "common.cuh"
#include "kernels.h"
#include "rounding.cuh"

namespace tnmc {

// Convergence: a pair counts as orthogonal when |y_p . y_q| <= tol |y_p| |y_q|, with tol =
// sqrt(D) eps, the rounding floor of a D-long dot product.  The residual non-orthogonality
// tilts the kept singular subspace where sigma_chi and sigma_{chi+1} are close; in FP32 at
// L = 256, chi = 32 a four times looser tolerance left environments whose conditionals drifted
// by up to 5e-3 from FP64 and produced doubly clamped sites (measured), for about 1 % more
// sweeps it does not.
template <typename T> struct JacobiTol;
template <> struct JacobiTol<float> { static constexpr int maxsw = 30; };
template <> struct JacobiTol<double> { static constexpr int maxsw = 40; };
template <typename T, int D> __device__ __forceinline__ T jacobi_tol() {
  return num<T>::sqrt_(T(D)) * num<T>::eps;
}

template <typename T> struct Vec16;
template <> struct Vec16<float> { using type = float4; };
template <> struct Vec16<double> { using type = double2; };
// Which product of a sum is rounded before it enters a fused multiply-add is written out, so that
// the results do not hang on how the compiler contracts each place.
__device__ __forceinline__ float dot16(const float4& a, const float4& b) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.x, b.x, __fmul_rn(a.y, b.y))));
}
__device__ __forceinline__ double dot16(const double2& a, const double2& b) {
  return fma(a.x, b.x, __dmul_rn(a.y, b.y));
}
// the square of a vector with the other product rounded first
__device__ __forceinline__ float sq16(const float4& a) {
  return fmaf(a.w, a.w, fmaf(a.z, a.z, fmaf(a.y, a.y, __fmul_rn(a.x, a.x))));
}
__device__ __forceinline__ double sq16(const double2& a) { return fma(a.y, a.y, __dmul_rn(a.x, a.x)); }
__device__ __forceinline__ float rot_u(float a, float b, float c, float s) {
  return fmaf(c, a, -__fmul_rn(s, b));
}
__device__ __forceinline__ float rot_v(float a, float b, float c, float s) {
  return fmaf(s, a, __fmul_rn(c, b));
}
__device__ __forceinline__ double rot_u(double a, double b, double c, double s) {
  return fma(c, a, -__dmul_rn(s, b));
}
__device__ __forceinline__ double rot_v(double a, double b, double c, double s) {
  return fma(s, a, __dmul_rn(c, b));
}
__device__ __forceinline__ void rot16(float4& u, float4& v, float c, float s) {
  const float4 a = u, b = v;
  u = make_float4(rot_u(a.x, b.x, c, s), rot_u(a.y, b.y, c, s), rot_u(a.z, b.z, c, s), rot_u(a.w, b.w, c, s));
  v = make_float4(rot_v(a.x, b.x, c, s), rot_v(a.y, b.y, c, s), rot_v(a.z, b.z, c, s), rot_v(a.w, b.w, c, s));
}
__device__ __forceinline__ void rot16(double2& u, double2& v, double c, double s) {
  const double2 a = u, b = v;
  u = make_double2(rot_u(a.x, b.x, c, s), rot_u(a.y, b.y, c, s));
  v = make_double2(rot_v(a.x, b.x, c, s), rot_v(a.y, b.y, c, s));
}
template <int ID> __device__ __forceinline__ void named_barrier(int nthreads) {
  asm volatile("bar.sync %0, %1;\n" ::"n"(ID), "r"(nthreads) : "memory");
}

// 4-element shared-memory vectors (16 B for float, 2 x 16 B for double); callers keep the
// index a multiple of 4 so the accesses are aligned.
__device__ __forceinline__ void ld4(const float* p, float v[4]) {
  const float4 t = *reinterpret_cast<const float4*>(p); v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void ld4(const double* p, double v[4]) {
  const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void st4(float* p, const float v[4]) { *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ void st4(double* p, const double v[4]) {
  reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
  reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
}
__device__ __forceinline__ void cp_async16_env(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit_env() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait_env() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }
// Copy `bytes` (a multiple of 16) from global to shared memory with cp.async (no wait).
__device__ __forceinline__ void prefetch_async(void* smem, const void* gmem, int bytes, int tid, int nt) {
  for (int i = tid; i < bytes / 16; i += nt)
    cp_async16_env(static_cast<char*>(smem) + 16 * i, static_cast<const char*>(gmem) + 16 * i);
  cp_async_commit_env();
}

template <int CHI, bool kCrowd = false> struct EnvCfg {
  static constexpr int D = 2 * CHI;                 // MPO bond x MPS bond
  // 8 CHI threads: 8 lanes per Jacobi pair, at least one thread per register tile of the products,
  // and no more, since all but the pivots' warp wait through the factorisations: with 256 threads at
  // CHI = 16 three realizations fit on an SM and issued 1.1 instructions a cycle between them.
  static constexpr int NT = 8 * CHI;
  static constexpr int NWARP = NT / 32;
  // Realizations per SM that the FP32 registers are cut to (shared memory allows three at CHI = 32),
  // and the runs of the factorisations.  CHI = 16 has two builds: five per SM with short runs for a
  // few realizations, seven with long ones (72 registers, a fifth less code: with more blocks in
  // different phases the instruction cache is what they wait for) for a crowd.  16 x 16 lattices, ms
  // by realizations: 100 9.5 / 10.8, 760 13.3 / 14.3, 1064 24.4 / 17.7, 1520 27.5 / 30.8.
  static constexpr int PER_SM = CHI > 32 ? 1 : (CHI == 32 ? 3 : (CHI == 16 ? (kCrowd ? 7 : 5) : (CHI == 8 ? 8 : 16)));
  static constexpr int RUN = kCrowd ? 8 : 4;
  // The sum of Y's squares is associated as VT threads' partial sums, whatever NT: it is the scale
  // that Jacobi's threshold hangs on.
  static constexpr int VT = CHI > 32 ? 512 : (CHI > 4 ? 256 : 128);
  static constexpr int TILE = 2 * CHI * CHI;        // [y][alpha][beta]
};

// Column stride of Y and V: at least 8 lanes x 16 bytes, so that the 8 lanes of a Jacobi
// pair read one contiguous 128-byte segment per vector load (no bank conflicts).
template <typename T, int CHI> struct JStride {
  static constexpr int D = 2 * CHI;
  static constexpr int VEC = 16 / (int)sizeof(T);
  static constexpr int DP = D > 8 * VEC ? D : 8 * VEC;
};

template <typename T, int CHI>
__host__ __device__ constexpr size_t env_smem_elems() {
  // CHI = 64: Y, V (D*DP each) and R (D*D) stay in shared memory (192 KB); M lives in
  // per-realization global scratch and the tile is read from global memory
  if (CHI > 32) return (size_t)2 * (2 * CHI) * JStride<T, CHI>::DP + (size_t)(2 * CHI) * (2 * CHI);
  // backward: M, R (D*D each), Y, V (D*DP each) + tile (2*CHI*CHI); P (D*CHI) lives in the Y
  //           region and Q (2*CHI*CHI) in the V region between their uses
  // forward : X (2D*D, aliases M and Y) + R (D*D) + tile; the reflectors take X's place
  // (FP32, CHI = 32: 72 KB, so three CTAs fit on one SM)
  return (size_t)2 * (2 * CHI) * (2 * CHI) + (size_t)2 * (2 * CHI) * JStride<T, CHI>::DP +
         (size_t)2 * CHI * CHI;
}

// Householder QR with the matrix in registers.  A group of G lanes owns CPT columns of the MR x NC
// matrix, lane g of a group the rows g + G u (u < RPT); warp w owns the CW consecutive columns from
// w CW on.  Reflector j is formed by the group that owns column j, published in shared memory, and
// applied by every group to its later columns.
//
// Every sum over the rows has one fixed association, whatever G: 32 partial sums, partial l over the
// rows l, l + 32, ... in this order, then the butterfly l ^ 16, 8, 4, 2, 1.  A lane holds the partials
// l = g mod G, so the levels down to G are register adds and only log2(G) shuffles remain.
//
// What bounds it: the chain dot product -> shuffles -> update -> norm -> square root -> publish of
// consecutive pivots (about 690 cycles each at 64 x 64, 400 in one warp), not the arithmetic.  With the
// columns in shared memory a reflector cost 1440 cycles: every step read and wrote the whole matrix
// there and reduced each dot product over 32 lanes, 870 cycles of the shared-memory pipe alone.
// 16 rows a lane and log2(MR/16) shuffle levels balance the serial adds of a lane against the
// shuffles (30 cycles a level).  Environment build at chi = 32, FP32 (one GB300): 203 -> 150 us a site
// step with one realization per SM (L = 64), 331 -> 214 us with three (L = 48).
template <typename T, int MR, int NC, int KR> struct QrCfg {
  // Lanes of a column: 16 rows each from MR = 32 on.  FP64 to MR = 32: four rows each, as an operation
  // of a warp keeps a scheduler's FP64 pipe for 64 cycles, so that a chain of few rows is the shorter
  // one (at MR = 64 the threads that this takes make it the longer one).  FP64 build with the roots of
  // norm_of and rotation_from_gram, before and after: chi = 16, L = 24, 256 realizations 404 -> 363 ms;
  // chi = 8, L = 12, 608 of them 28.5 -> 23.9 ms; chi = 32, L = 12, 8 of them 82.1 -> 78.4 ms (at 16
  // rows a lane as here; 89.8 ms with four).
  static constexpr bool FEW = sizeof(T) == 8 && MR <= 32;
  static constexpr int G = FEW ? (MR >= 8 ? MR / 4 : 2) : (MR >= 32 ? MR / 16 : 2);
  static constexpr int RPT = MR / G;
  static constexpr int NVL = 32 / G < RPT ? 32 / G : RPT;   // partial sums a lane holds (not if FEW)
  // The factorisation has one body for each run of KR rows of a lane (the pivots whose rows are in
  // it; the rows of earlier runs are left out): short runs save products of zeros and cost code.
  static constexpr int RUN = RPT < KR ? RPT : KR;
  static constexpr int CPT = NC * G > 512 ? (NC * G) / 512 : (NC * G > 256 || G > 4 ? 2 : 1);
  static constexpr int NTQ = NC * G / CPT < 32 ? 32 : NC * G / CPT;   // threads taking part
  static constexpr int GPW = 32 / G;                        // groups of a warp
  static constexpr int CW = GPW * CPT;                      // columns of a warp
};
// Place of row i in a column stored for QrCfg: each lane's rows in 16-byte runs of four, the runs of
// the G lanes side by side, so that a group reads its column in conflict-free vector loads.
template <int G> __device__ __forceinline__ int qr_pos(int i) {
  const int g = i % G, u = i / G;
  return (u >> 2) * (4 * G) + g * 4 + (u & 3);
}

// Two FP32 operations in one instruction (fma.rn.f32x2, add.rn.f32x2): the same roundings, half the
// issue slots.
__device__ __forceinline__ unsigned long long pack2(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(unsigned long long r, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
// c += a * b, p += q on pairs of adjacent array elements
__device__ __forceinline__ void fma_pair(const float* a, const float* b, float* c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pack2(a[0], a[1])), "l"(pack2(b[0], b[1])), "l"(pack2(c[0], c[1])));
  unpack2(r, c[0], c[1]);
}
__device__ __forceinline__ void add_pair(float* p, const float* q) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(p[0], p[1])), "l"(pack2(q[0], q[1])));
  unpack2(r, p[0], p[1]);
}
__device__ __forceinline__ void fma_pair(const double* a, const double* b, double* c) {
  c[0] = fma(a[0], b[0], c[0]);
  c[1] = fma(a[1], b[1], c[1]);
}
__device__ __forceinline__ void add_pair(double* p, const double* q) { p[0] += q[0]; p[1] += q[1]; }

// Sum of v * x over the rows of the runs C0 and later (the earlier ones hold zeros) in the fixed
// association; every lane of the group gets it.
template <typename Q, int C0, typename T>
__device__ __forceinline__ T qr_dot(const T (&v)[Q::RPT], const T (&x)[Q::RPT], int j) {
  T d;
  if constexpr (Q::FEW) {
    // one chain; rows above the pivot j hold zeros in v
    d = T(0);
#pragma unroll
    for (int u = 0; u < Q::RPT; ++u)
      if (Q::G * (u + 1) > j) d = fma(v[u], x[u], d);
  } else {
    T p[Q::NVL];
#pragma unroll
    for (int a = 0; a < Q::NVL; ++a) p[a] = T(0);
#pragma unroll
    for (int u = Q::RUN * C0; u < Q::RPT; u += 2) fma_pair(v + u, x + u, p + u % Q::NVL);
#pragma unroll
    for (int lv = Q::NVL / 2; lv > 1; lv >>= 1)
#pragma unroll
      for (int a = 0; a < lv; a += 2) add_pair(p + a, p + a + lv);
    d = p[0] + p[1];
  }
#pragma unroll
  for (int o = Q::G / 2; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
  return d;
}
template <typename Q, int C0, typename T>
__device__ __forceinline__ void qr_update(T md, const T (&v)[Q::RPT], T (&x)[Q::RPT], int j) {
  if constexpr (Q::FEW) {
#pragma unroll
    for (int u = 0; u < Q::RPT; ++u)
      if (Q::G * (u + 1) > j) x[u] = fma(md, v[u], x[u]);
  } else {
    const T m2[2] = {md, md};
#pragma unroll
    for (int u = Q::RUN * C0; u < Q::RPT; u += 2) fma_pair(m2, v + u, x + u);
  }
}
template <typename Q, int C0, typename T>
__device__ __forceinline__ void qr_load_v(const T* vs, int g, T (&v)[Q::RPT]) {
#pragma unroll
  for (int u = Q::RUN * C0; u < Q::RPT; u += 4) ld4(vs + u * Q::G + g * 4, v + u);
}
// Named barrier 3 + k (k < 4), waited for or only arrived at.  The number is spelled out in the
// instruction: with one in a register the compiler reserves all 16 barriers for the block, and an SM's
// 64 then hold four blocks.
__device__ __forceinline__ void turn_sync(int k, int n) {
  if (k & 2) {
    if (k & 1) asm volatile("bar.sync 6, %0;\n" ::"r"(n) : "memory");
    else asm volatile("bar.sync 5, %0;\n" ::"r"(n) : "memory");
  } else {
    if (k & 1) asm volatile("bar.sync 4, %0;\n" ::"r"(n) : "memory");
    else asm volatile("bar.sync 3, %0;\n" ::"r"(n) : "memory");
  }
}
__device__ __forceinline__ void turn_arrive(int k, int n) {        // k = 0, 1, 2
  if (k & 2) asm volatile("bar.arrive 5, %0;\n" ::"r"(n) : "memory");
  else if (k & 1) asm volatile("bar.arrive 4, %0;\n" ::"r"(n) : "memory");
  else asm volatile("bar.arrive 3, %0;\n" ::"r"(n) : "memory");
}

// State of one factorisation: where the reflectors go and how they are handed on.
// The warp that owns the pivot columns runs ahead: it publishes reflector after reflector, each in a
// slot of its own, and only arrives at that reflector's barrier while the others wait.  The published
// reflectors use four barriers in turn, and with every fourth the pivot's warp waits too, so that no
// barrier is used again before all have passed it.  (Flags in shared memory that the others poll
// took their issue slots: 459 instead of 388 ms at three CTAs per SM.)
template <typename T> struct QrOut {
  T* v;              // slot j (MR elements): reflector j
  T* cden;           // [j]: reflector j's coefficient 2/|v|^2 (0: no reflector), with kLate its reciprocal
  T* diag;           // [j]: R_jj
};
// In FP32 every warp inverts the coefficient beside its dot products, off the pivots' chain; in FP64,
// where a division occupies the FP64 pipe, only the pivot's warp does.
template <typename T> constexpr bool kLate = sizeof(T) == 4;

// Ranges of the FP32 build.  inverse() ends at a coefficient of 8e37, at most twice a column's squared norm;
// the Jacobi multiplies two squared norms.  A matrix with an entry beyond the limits below (weights of exp(16)
// and more: strong fields, low temperatures) is factored times a power of two that brings its largest entry
// just below the limit, so nothing is rounded by it; nothing has to be scaled back either, as R is normalised,
// the right singular vectors have no scale and the singular values are only compared.  One that has overflowed
// becomes NaN, which the sampler flags.  Whoever forms a matrix looks at its entries, and the scaling is out of
// line: that costs 1 % of the builds for chi <= 8, 4 % of the crowd's, whose code is the tightest (90.5 -> 93.9
// ms, 1024 realizations of 32 x 32), and nothing beyond.  A test of each coefficient in the warps that use it
// cost 2 to 4 % of all, in the pivot's warp 3 to 8 %, a second body that divides 1 to 3 %.
constexpr float kLargeX = 1125899906842624.0f;       // 2^50: 2 * 256 entries * kLargeX^2 = 6.5e32
constexpr float kLargeY = 8388608.0f;                // 2^23: (128 * 128 entries * kLargeY^2)^2 = 1.3e36
__device__ __forceinline__ float entry_max(float m, float x) { return fmaxf(m, fabsf(x)); }
__device__ __forceinline__ double entry_max(double m, double) { return m; }
// Leaves the bits of the largest entry beyond the limit in flag (0: none).
template <typename T> __device__ __forceinline__ void note_large(T entry, float limit, int* flag) {
  if (kLate<T> && entry > T(limit)) atomicMax(flag, __float_as_int((float)entry));
}
// The power of two that takes such an entry into [limit / 2, limit), NaN for an infinity.
__device__ __forceinline__ float down_scale(float limit, int bits) {
  const int e = bits >> 23, to = (__float_as_int(limit) >> 23) - 1;
  return e == 255 ? NAN : __int_as_float((127 + to - e) << 23);
}

// Reflector of column j, by the warp that owns it; j lies in the rows of run C0.
template <typename T, int MR, int NC, int KR, int C0>
__device__ __forceinline__ void qr_pivot(T (&x)[QrCfg<T, MR, NC, KR>::CPT][QrCfg<T, MR, NC, KR>::RPT], int j, T* vs,
                                         const QrOut<T>& o, int g, int gi, int warp) {
  using Q = QrCfg<T, MR, NC, KR>;
  constexpr int G = Q::G;
  const T tiny = (sizeof(T) == 4) ? T(1e-36) : T(1e-300);
  const int jl = j - warp * Q::CW, jq = jl / Q::GPW, jr = j - Q::RUN * G * C0;   // row of the pivot within the run
#pragma unroll
  for (int q = 0; q < Q::CPT; ++q) {
    if (Q::CPT > 1 && q != jq) continue;     // warp-uniform
    T xr[Q::RPT], x0 = T(0);
#pragma unroll
    for (int u = Q::RUN * C0; u < Q::RPT; ++u) xr[u] = x[q][u];
#pragma unroll
    for (int u = 0; u < Q::RUN; ++u) {
      const int i = g + G * u;               // rows above the pivot belong to R
      if (i < jr) xr[Q::RUN * C0 + u] = T(0);
      if (i == jr) x0 = xr[Q::RUN * C0 + u];
    }
    const T ss = qr_dot<Q, C0, T>(xr, xr, j);
    const bool null = ss <= tiny;
    const T nrm = norm_of(ss);
    if (gi == jl - jq * Q::GPW) {            // the pivot's group
      const T alpha = x0 >= T(0) ? -nrm : nrm;
      const T v0 = x0 - alpha;
#pragma unroll
      for (int u = 0; u < Q::RUN; ++u)
        if (g + G * u == jr) { xr[Q::RUN * C0 + u] = v0; if (!null) x[q][Q::RUN * C0 + u] = alpha; }
#pragma unroll
      for (int u = Q::RUN * C0; u < Q::RPT; u += 4) {
        st4(vs + u * G + g * 4, xr + u);
      }
      if (g == jr % G) {
        const T den = nrm * (nrm + (x0 >= T(0) ? x0 : -x0));
        o.cden[j] = null ? T(0) : (kLate<T> ? den : T(1) / den);
        o.diag[j] = null ? x0 : alpha;
      }
    }
  }
}

// The pivots whose rows lie in run C0, then those of the later runs.
template <typename T, int MR, int NC, int KR, int C0, typename Skip>
__device__ __forceinline__ void qr_runs(T (&x)[QrCfg<T, MR, NC, KR>::CPT][QrCfg<T, MR, NC, KR>::RPT], int nc, int& pub,
                                        const QrOut<T>& o, int g, int gi, int warp, Skip skip) {
  using Q = QrCfg<T, MR, NC, KR>;
  constexpr int J0 = Q::RUN * Q::G * C0, J1 = J0 + Q::RUN * Q::G < NC ? J0 + Q::RUN * Q::G : NC;
  const int first = warp * Q::CW, last = first + Q::CW - 1;
  const int je = nc < J1 ? nc : J1;
  for (int j = J0; j < je; ++j) {
    if (!skip(j)) {
      if (j >= first && j <= last) qr_pivot<T, MR, NC, KR, C0>(x, j, o.v + (size_t)j * MR, o, g, gi, warp);
      if constexpr (Q::NTQ == 32) {
        __syncwarp();
      } else if (j >= first && j <= last && (pub & 3) != 3) {
        __syncwarp();
        turn_arrive(pub & 3, Q::NTQ);
      } else {
        turn_sync(pub & 3, Q::NTQ);
      }
      ++pub;
      if (last > j) {
        T v[Q::RPT];
        qr_load_v<Q, C0, T>(o.v + (size_t)j * MR, g, v);
        const T den = o.cden[j];
        const T coef = !kLate<T> || den == T(0) ? den : inverse(den);
#pragma unroll
        for (int q = 0; q < Q::CPT; ++q) {
          T d = qr_dot<Q, C0, T>(v, x[q], j) * coef;
          if (first + q * Q::GPW + gi <= j) d = T(0);
          qr_update<Q, C0>(-d, v, x[q], j);
        }
      }
    }
  }
  if constexpr (J1 < NC) qr_runs<T, MR, NC, KR, C0 + 1>(x, nc, pub, o, g, gi, warp, skip);
}

// Factor the columns j < nc for which skip(j) is false (skip(j): the column is known to be zero, so
// its reflector is the identity; it must be the same for every thread).  On return x holds R on and
// above the diagonal (below it, what is left of the reflectors).
template <typename T, int MR, int NC, int KR, typename Skip>
__device__ __forceinline__ void qr_factor(T (&x)[QrCfg<T, MR, NC, KR>::CPT][QrCfg<T, MR, NC, KR>::RPT], int nc,
                                          const QrOut<T>& o, int lane, int warp, Skip skip) {
  using Q = QrCfg<T, MR, NC, KR>;
  int pub = 0;                              // reflectors published
  qr_runs<T, MR, NC, KR, 0>(x, nc, pub, o, lane % Q::G, lane / Q::G, warp, skip);
}

// x <- H_0 H_1 ... H_{n-1} x for one column per group, the reflectors as qr_factor kept them.
template <typename T, int MR, int NC, int KR, int C0 = (NC - 1) / (QrCfg<T, MR, NC, KR>::RUN * QrCfg<T, MR, NC, KR>::G)>
__device__ __forceinline__ void qr_apply_q(T (&x)[QrCfg<T, MR, NC, KR>::RPT], int n, const T* vs, const T* coefs, int g) {
  using Q = QrCfg<T, MR, NC, KR>;
  constexpr int J0 = Q::RUN * Q::G * C0, J1 = J0 + Q::RUN * Q::G < NC ? J0 + Q::RUN * Q::G : NC;
  for (int j = (n < J1 ? n : J1) - 1; j >= J0; --j) {
    const T coef = coefs[j];
    if (coef == T(0)) continue;
    T v[Q::RPT];
    qr_load_v<Q, C0, T>(vs + (size_t)j * MR, g, v);
    const T d = qr_dot<Q, C0, T>(v, x, j) * coef;
    qr_update<Q, C0>(-d, v, x, j);
  }
  if constexpr (C0 > 0) qr_apply_q<T, MR, NC, KR, C0 - 1>(x, n, vs, coefs, g);
}

// a[c][i] (i < rows, columns ld apart) times s; returns the sum of squares of the thread's own entries.
template <typename T> __device__ __noinline__ T scale_matrix(T* a, int rows, int cols, int ld, T s, int tid, int nt) {
  T f = 0;
#pragma unroll 1
  for (int e = tid; e < rows * cols; e += nt) {
    T& y = a[(size_t)(e / rows) * ld + e % rows];
    y *= s;
    f += y * y;
  }
  return f;
}

template <typename T, typename TE, int CHI, bool kCrowd>
__global__ void __launch_bounds__(EnvCfg<CHI>::NT, sizeof(T) == 8 ? 1 : EnvCfg<CHI, kCrowd>::PER_SM)
env_build_kernel(EnvBuildArgs<T, TE> args) {
  using C = EnvCfg<CHI, kCrowd>;
  constexpr int D = C::D, NWARP = C::NWARP, NT = C::NT, TILE = C::TILE;
  const int L = args.L;
  const int real = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int chi = args.chi;
  const double beta = args.beta[real];

  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sm = reinterpret_cast<T*>(smem_raw);
  // CHI = 64 (kBig): M in global scratch, the previous-row tile read where it is stored (the pointer
  // moves with the site), shared memory for Y, V and R_c
  constexpr bool kBig = CHI > 32;
  // backward-phase layout
  constexpr int DP = JStride<T, CHI>::DP;
  T* Mc = kBig ? args.Mscratch + (size_t)real * D * D : sm;   // D x D col-major, columns j = x*kn + g
  T* Yc = kBig ? sm : Mc + D * D;  // n columns of stride DP (rows >= D zero)
  T* Vc = Yc + D * DP;        // n columns of stride DP (rows >= n zero)
  T* const Rc = Vc + D * DP;  // D x D col-major R_c
  T* Bt = kBig ? nullptr : Rc + D * D;     // previous-row tile [y][al][be]
  // P is written after the SVD (Y is dead by then) and read by the next site's Q = B P before
  // that site's Y is formed; Q is written after this site's V is dead and read before the next
  // V is initialised: so P takes the Y region and Q the V region
  T* Ps = Yc;                 // D x CHI col-major: P[(b,be)][g] at g*D + b*CHI + be
  T* Qs = Vc;                 // 2 x CHI x CHI: Q[b][g][al]
  // forward-phase layout (aliases M/Y/V; R stays at Rc)
  T* Xs = sm;                 // 2D x D col-major

  __shared__ T Wc[8];               // W[x][a][b] at x*4 + a*2 + b
  int8_t* jv_s = reinterpret_cast<int8_t*>(kBig ? Rc + D * D : Bt + TILE);   // Jv[r][c], L entries
  int8_t* jh_s = jv_s + args.L;                                // Jh[r+1][c], L-1 entries
  const T eb = (T)exp(beta), ebm = (T)exp(-beta);             // exp(+-beta): every Boltzmann weight
  using QF = QrCfg<T, 2 * D, D, C::RUN>;     // the forward sweep's QR
  using QB = QrCfg<T, D, D, C::RUN>;         // the backward sweep's
  __shared__ T csave[D];            // the reflectors' coefficients (as qr_factor leaves them, then inverted)
  __shared__ T diag[D];
  __shared__ T red[32];
  __shared__ T sig[D];
  __shared__ int sel[CHI];
  __shared__ int rot[3];            // per-sweep 'any rotation' flags, a ring of three
  __shared__ int knext_s;
  __shared__ int large_s;           // of the matrix to be factored, as note_large leaves it

  const int8_t* J = args.J + (size_t)real * 2 * L * (L - 1);
  // external fields (units of beta) of this realization: the row MPO carries those of the row
  // below as a site weight exp(beta k s_b), the top-row closure of log Z those of row 0
  const int8_t* hf = args.hfield ? args.hfield + (size_t)real * L * L : nullptr;
  const int8_t* Jh = J;                          // [r][c], c < L-1
  const int8_t* Jv = J + (size_t)L * (L - 1);    // [r][c], r < L-1
  int* kd = args.kdim + (size_t)real * L * (L + 1);
  int* dqr = args.dqr + (size_t)real * (L + 1);
  T* rowbuf = args.rowbuf + (size_t)real * 2 * L * TILE;
  T* Rstore = args.Rstore + (size_t)real * L * D * D;
  TE* env = args.env + (size_t)real * L * L * TILE;
  double* lam = args.lam + (size_t)real * L;

  // ---- row L-1: the exact all-ones environment G_{L-1}(x) = 1
  {
    T* prev = rowbuf + (size_t)((L - 1) & 1) * L * TILE;
    TE* erow = env + (size_t)(L - 1) * L * TILE;
    for (int e = tid; e < L * TILE; e += NT) {
      const int t = e % TILE;
      const T v = (t == 0 || t == CHI * CHI) ? T(1) : T(0);
      prev[e] = v;
      erow[e] = env_store<TE, T>(v);
    }
    for (int c = tid; c <= L; c += NT) kd[(size_t)(L - 1) * (L + 1) + c] = 1;
    if (tid == 0) lam[L - 1] = 0.0;
  }
  __syncthreads();

  int max_sweeps_seen = 0, unconverged = 0;
  long long total_sweeps = 0, n_svd = 0;

  for (int r = L - 2; r >= 0; --r) {
    const T* prev = rowbuf + (size_t)((r + 1) & 1) * L * TILE;
    T* cur = rowbuf + (size_t)(r & 1) * L * TILE;
    TE* erow = env + (size_t)r * L * TILE;
    const int* kold = kd + (size_t)(r + 1) * (L + 1);
    int* knew = kd + (size_t)r * (L + 1);

    // Zip-up rows alternate their sweep direction; a left-to-right row runs as the right-to-left
    // sweep of the mirrored row.  The backward sweep below works in the sweep's frame: frame site
    // f is site osite(f) of the lattice, whose bonds are swapped when the row is mirrored.
    const bool zip = args.zipup != 0;
    const bool mir = zip && ((L - 2 - r) % 2 == 0);
    auto osite = [&](int f) { return mir ? L - 1 - f : f; };
    // canonical: QR bond dimensions d_c of the MPO x MPS (left-canonical form); zip-up: the
    // rows of frame site f's matrix M, (MPO bond) x (previous row's bond into f)
    if (tid == 0) {
      if (zip) {
        for (int f = 0; f < L; ++f) dqr[f] = (f == 0 ? 1 : 2) * (mir ? kold[L - f] : kold[f]);
      } else {
        dqr[0] = 1;
        for (int c = 0; c < L - 1; ++c) dqr[c + 1] = min(2 * dqr[c], 2 * kold[c + 1]);
      }
    }
    for (int c = tid; c < L; c += NT) jv_s[c] = Jv[(size_t)r * L + c];
    for (int c = tid; c < L - 1; c += NT) jh_s[c] = Jh[(size_t)(r + 1) * (L - 1) + c];
    // W(x,a,b) of (frame) site c from exp(+-beta): the vertical bond to the row below and the
    // horizontal bond of the row below to the previous frame site (absent at c = 0, where only
    // a = 0 exists) -- in a mirrored row that is the bond to the lattice site on the right
    auto set_w = [&](int c) {
      if (tid < 8) {
        const int x = tid >> 2, a = (tid >> 1) & 1, b = tid & 1;
        const int co = osite(c);
        T w = (jv_s[co] * spin_of(x) * spin_of(b) > 0) ? eb : ebm;
        if (c > 0) w *= (jh_s[mir ? co : c - 1] * spin_of(a) * spin_of(b) > 0) ? eb : ebm;
        else if (a == 1) w = T(0);
        if (hf) { const int k = hf[(size_t)(r + 1) * L + co]; if (k) w *= (T)exp(beta * (double)(k * spin_of(b))); }
        Wc[tid] = w;
      }
    };
    // R_0 = [1]
    for (int e = tid; e < D * D; e += NT) Rc[e] = (e == 0) ? T(1) : T(0);
    for (int e = tid; e < D * D; e += NT) Rstore[e] = (e == 0) ? T(1) : T(0);
    // the tile the first sweep starts on: site 0 (forward sweep), frame site L-1 (zip-up)
    if constexpr (!kBig) prefetch_async(Bt, prev + (size_t)(zip ? osite(L - 1) : 0) * TILE, TILE * (int)sizeof(T), tid, NT);
    __syncthreads();

    // ---------------- forward sweep: R factors of the left parts (canonical only) ----------------
    for (int c = 0; !zip && c < L - 1; ++c) {
      set_w(c);
      if (tid == 0) large_s = 0;
      if constexpr (kBig) Bt = const_cast<T*>(prev + (size_t)c * TILE);
      cp_async_wait_env();
      __syncthreads();
      // X[(x,i),(b,be)] = sum_al (W(x,0,b) R[i][al] + W(x,1,b) R[i][CHI+al]) B[b][al][be]:
      // four (D x CHI) = (D x CHI)(CHI x CHI) products in 4 x BW register tiles (BW = 8 where that
      // still leaves a tile per thread: the combination of R's rows is formed once per tile)
      constexpr int BW = CHI >= 32 ? 8 : 4, TI = D / 4, TB = CHI / BW;
      T xmax = 0;
      for (int u = tid; u < 4 * TI * TB; u += NT) {
        const int xb = u / (TI * TB), rem = u % (TI * TB);
        const int x = xb >> 1, b = xb & 1, i0 = (rem % TI) * 4, b0 = (rem / TI) * BW;
        const T w0 = Wc[x * 4 + 0 * 2 + b], w1 = Wc[x * 4 + 1 * 2 + b];
        T acc[4][BW] = {};
#pragma unroll 2
        for (int al = 0; al < CHI; ++al) {
          T r0[4], r1[4], bv[BW];
          ld4(Rc + al * D + i0, r0);
          ld4(Rc + (CHI + al) * D + i0, r1);
#pragma unroll
          for (int jj = 0; jj < BW; jj += 4) ld4(Bt + b * CHI * CHI + al * CHI + b0 + jj, bv + jj);
#pragma unroll
          for (int ii = 0; ii < 4; ++ii) {
            const T rw = w0 * r0[ii] + w1 * r1[ii];
#pragma unroll
            for (int jj = 0; jj < BW; ++jj) acc[ii][jj] += rw * bv[jj];
          }
        }
        // row (x, i) of X is stored at 2 i + x: the two blocks R_c A^0 and R_c A^1 share
        // R_c's row scale, which falls with i, so interleaving them lets the reflectors meet
        // the rows in order of scale (measured at L = 256 in FP32: two orders of magnitude
        // fewer clamped weights than the two blocks one after the other)
#pragma unroll
        for (int jj = 0; jj < BW; ++jj) {
          T* xc = Xs + (size_t)(b * CHI + b0 + jj) * (2 * D);
#pragma unroll
          for (int ii = 0; ii < 4; ++ii) {
            xc[qr_pos<QF::G>(2 * (i0 + ii) + x)] = acc[ii][jj];
            xmax = entry_max(xmax, acc[ii][jj]);
          }
        }
      }
      note_large(xmax, kLargeX, &large_s);
      __syncthreads();
      if (kLate<T> && large_s) {
        scale_matrix<T>(Xs, 2 * D, D, 2 * D, T(down_scale(kLargeX, large_s)), tid, NT);
        __syncthreads();
      }
      // the next site's tile streams in while the QR runs
      if constexpr (!kBig) prefetch_async(Bt, prev + (size_t)(c + 1) * TILE, TILE * (int)sizeof(T), tid, NT);
      // R factor of X in registers; R_{c+1} = R / max |R_jj| (col-major, zeros below the diagonal)
      if (warp < QF::NTQ / 32) {
        const int g = lane % QF::G, gi = lane / QF::G;
        T x[QF::CPT][QF::RPT];
#pragma unroll
        for (int q = 0; q < QF::CPT; ++q) {
          const int col = warp * QF::CW + q * QF::GPW + gi;
#pragma unroll
          for (int u = 0; u < QF::RPT; ++u) x[q][u] = T(0);
          if (col < D) qr_load_v<QF, 0, T>(Xs + (size_t)col * (2 * D), g, x[q]);
        }
        // columns (b, be) beyond the right bond of the previous row's tile are zero
        const int kr = kold[c + 1];
        auto zero_col = [&](int j) { return (j & (CHI - 1)) >= kr; };
        // the reflectors take X's place, column by column of it read by now
        if constexpr (QF::NTQ == 32) __syncwarp();
        else named_barrier<2>(QF::NTQ);
        const QrOut<T> out{Xs, csave, diag};
        qr_factor<T, 2 * D, D, C::RUN>(x, D, out, lane, warp, zero_col);
        T mx = 0;
        for (int j = lane; j < D; j += 32)
          if (!zero_col(j)) { const T v = diag[j] < 0 ? -diag[j] : diag[j]; mx = v > mx ? v : mx; }
        mx = warp_max(mx);
        const T inv = mx > T(0) ? T(1) / mx : T(1);
        T* Rout = Rstore + (size_t)(c + 1) * D * D;
#pragma unroll
        for (int q = 0; q < QF::CPT; ++q) {
          const int col = warp * QF::CW + q * QF::GPW + gi;
          if (col < D) {
#pragma unroll
            for (int u = 0; u < QF::RPT / 2; ++u) {          // rows below D are zero
              const int i = g + QF::G * u;
              const T v = i <= col ? x[q][u] * inv : T(0);
              Rc[col * D + i] = v;
              Rout[col * D + i] = v;
            }
          }
        }
      }
      __syncthreads();
    }

    // ---------------- backward sweep: truncating SVDs ----------------
    // P_L[(b,be)][g] = delta(be,0) delta(g,0) for both b (closes the right MPO bond)
    for (int e = tid; e < D * CHI; e += NT) {
      const int row = e % D, g = e / D;
      Ps[e] = (g == 0 && (row % CHI) == 0) ? T(1) : T(0);
    }
    int kn = 1;             // k_{c+1}
    // The removed scales' logarithms, added in site order.  One lane of warp 0 keeps each scale and the
    // logarithms are taken 32 at a time: one thread's FP64 logarithm held the site up for 2400 cycles.
    double logs = 0.0;
    T scale = T(1);
    int n_scales = 0;
    auto flush_scales = [&]() {
      const double l = lane < n_scales && scale > T(0) ? log((double)scale) : 0.0;
      for (int i = 0; i < n_scales; ++i) {
        const double li = __shfl_sync(0xffffffffu, l, i);
        if (__shfl_sync(0xffffffffu, scale, i) > T(0)) logs += li;
      }
      n_scales = 0;
    };
    auto keep_scale = [&](T v) {               // by the whole of warp 0
      if (lane == n_scales) scale = v;
      if (++n_scales == 32) flush_scales();
    };
    if (tid == 0) knew[L] = 1;
    __syncthreads();
    for (int c = L - 1; c >= 0; --c) {
      // Bt (tile c) and Rc (R_c) were prefetched during the previous site
      set_w(c);
      if (tid == 0) large_s = 0;
      if constexpr (kBig) Bt = const_cast<T*>(prev + (size_t)osite(c) * TILE);
      cp_async_wait_env();
      __syncthreads();
      // Q[b][al][g] = sum_be B[b][al][be] P[(b,be)][g]: 4 x 4 register tiles (a mirrored row
      // reads the previous row's tile with its bonds swapped)
      {
        constexpr int TA = CHI / 4;
        for (int u = tid; u < 2 * TA * TA; u += NT) {
          const int b = u / (TA * TA), a0 = ((u % (TA * TA)) % TA) * 4, g0 = ((u % (TA * TA)) / TA) * 4;
          T acc[4][4] = {};
          if (g0 < kn) {
            // four be at a time: vector loads of the rows of B (of its columns in a mirrored row) and
            // of the columns of P
            for (int be0 = 0; be0 < CHI; be0 += 4) {
              T bv[4][4], pv[4][4];        // [ii][be], [jj][be]
#pragma unroll
              for (int t = 0; t < 4; ++t) {
                T v[4];
                ld4(Bt + b * CHI * CHI + (mir ? (be0 + t) * CHI + a0 : (a0 + t) * CHI + be0), v);
#pragma unroll
                for (int q = 0; q < 4; ++q) { if (mir) bv[q][t] = v[q]; else bv[t][q] = v[q]; }
                ld4(Ps + (size_t)(g0 + t) * D + b * CHI + be0, pv[t]);
              }
#pragma unroll
              for (int be = 0; be < 4; ++be)
#pragma unroll
                for (int ii = 0; ii < 4; ++ii)
#pragma unroll
                  for (int jj = 0; jj < 4; ++jj) acc[ii][jj] += bv[ii][be] * pv[jj][be];
            }
          }
          // Q is kept [b][g][al]: M's rows run over al
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            T col4[4];
#pragma unroll
            for (int ii = 0; ii < 4; ++ii) col4[ii] = (g0 + jj < kn) ? acc[ii][jj] : T(0);
            st4(Qs + b * CHI * CHI + (g0 + jj) * CHI + a0, col4);
          }
        }
      }
      __syncthreads();
      if (!kBig && c > 0) prefetch_async(Bt, prev + (size_t)osite(c - 1) * TILE, TILE * (int)sizeof(T), tid, NT);
      const int n = 2 * kn;    // compact columns j = x*kn + g
      // M[(a,al)][j] = sum_b W(x,a,b) Q[b][al][g]
      for (int e = tid; e < D * n; e += NT) {
        const int row = e % D, j = e / D;
        const int a = row / CHI, al = row % CHI, x = j >= kn, g = j - x * kn;
        Mc[e] = Wc[x * 4 + a * 2 + 0] * Qs[0 * CHI * CHI + g * CHI + al] +
                Wc[x * 4 + a * 2 + 1] * Qs[1 * CHI * CHI + g * CHI + al];
      }
      __syncthreads();
      if (c == 0) {
        // site 0: the whole remaining state, row (a=0, al=0) of M
        if (warp == 0) {
          T ss = 0;
          for (int j = lane; j < n; j += 32) ss += Mc[(size_t)j * D] * Mc[(size_t)j * D];
          ss = warp_sum(ss);
          if (lane == 0) red[0] = num<T>::sqrt_(ss);
        }
        __syncthreads();
        const T nrm = red[0];
        const T inv = nrm > T(0) ? T(1) / nrm : T(0);
        T* ctile0 = cur + (size_t)osite(0) * TILE;
        TE* etile0 = erow + (size_t)osite(0) * TILE;
        for (int e = tid; e < TILE; e += NT) {
          const int y = e / (CHI * CHI), i = (e / CHI) % CHI, j = e % CHI;
          const int al = mir ? j : i, be = mir ? i : j;     // frame bonds of lattice entry (i, j)
          const T v = (al == 0 && be < kn) ? Mc[(size_t)(y * kn + be) * D] * inv : T(0);
          ctile0[e] = v;
          etile0[e] = env_store<TE, T>(v);
        }
        if (warp == 0) { flush_scales(); logs += log((double)nrm); }
        if (tid == 0) { knew[0] = 1; knew[L] = 1; }
        __syncthreads();
        break;
      }
      // Y = R_c M  (D x n; R_c, the R factor of the left part up to site c-1, was
      // prefetched): 4 x 4 register tiles over (rows, compact columns).  Zip-up: Y = M (the
      // previous row is canonical on the side not yet swept, so no R factor)
      constexpr int VK = C::VT / NT;
      T fro[VK] = {}, ymax = 0;
      if (zip) {
        for (int e = tid; e < DP * n; e += NT) {
          const int i = e % DP, j = e / DP;
          const T v = i < D ? Mc[(size_t)j * D + i] : T(0);
          Yc[e] = v;
          ymax = entry_max(ymax, v);
#pragma unroll
          for (int q = 0; q < VK; ++q) if ((e / NT) % VK == q) fro[q] += v * v;
        }
      } else {
        constexpr int TI = D / 4;
        const int TJ = (n + 3) / 4;
        for (int u = tid; u < TI * TJ; u += NT) {
          const int i0 = (u % TI) * 4, j0 = (u / TI) * 4;
          T acc[4][4] = {};
          for (int l = 0; l < D; l += 4) {
            T mv[4][4];
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
              mv[jj][0] = mv[jj][1] = mv[jj][2] = mv[jj][3] = T(0);
              if (j0 + jj < n) ld4(Mc + (size_t)(j0 + jj) * D + l, mv[jj]);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              T rv[4];
              ld4(Rc + (l + q) * D + i0, rv);
#pragma unroll
              for (int ii = 0; ii < 4; ++ii)
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) acc[ii][jj] += rv[ii] * mv[jj][q];
            }
          }
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            if (j0 + jj < n) {
#pragma unroll
              for (int ii = 0; ii < 4; ++ii) {
                Yc[(size_t)(j0 + jj) * DP + qr_pos<QB::G>(i0 + ii)] = acc[ii][jj];
                ymax = entry_max(ymax, acc[ii][jj]);
#pragma unroll
                for (int q = 0; q < VK; ++q) if ((u / NT) % VK == q) fro[q] += acc[ii][jj] * acc[ii][jj];
              }
            }
          }
        }
      }
      note_large(ymax, kLargeY, &large_s);
      // the Jacobi runs on npad = n rounded up to 8 columns (blocks of 4, an even number of
      // blocks); columns n..npad-1 of Y are zero and never rotate
      const int npad = (n + 7) & ~7;
#pragma unroll
      for (int q = 0; q < VK; ++q) {
        const T f = warp_sum(fro[q]);
        if (lane == 0) red[q * NWARP + warp] = f;
      }
      if (tid == 0) { rot[0] = 0; rot[1] = 0; rot[2] = 0; }
      __syncthreads();
      T sumY = warp_sum(lane < C::VT / 32 ? red[lane] : T(0));
      if (kLate<T> && large_s) {
        T f = scale_matrix<T>(Yc, D, n, DP, T(down_scale(kLargeY, large_s)), tid, NT);
        f = warp_sum(f);
        __syncthreads();
        if (lane == 0) red[warp] = f;
        __syncthreads();
        sumY = warp_sum(lane < NWARP ? red[lane] : T(0));
      }
      const T tinyY = sumY * num<T>::eps * num<T>::eps;
      if (zip) {
        // the zip-up's Y = M is graded by columns (P = U S), where the one-sided Jacobi is
        // accurate without preconditioning; it is not near to orthogonal, though: in the first four
        // sweeps nearly all pairs above the threshold rotate (8 to 10 sweeps a site at chi = 32,
        // 3.4 to 4 on the preconditioned matrix)
        for (int e = tid; e < DP * npad; e += NT) { const int i = e % DP, j = e / DP; Vc[e] = (i == j) ? T(1) : T(0); }
        for (int e = tid; e < DP * (npad - n); e += NT) Yc[(size_t)n * DP + e] = T(0);
        __syncthreads();
      } else {
        // Preconditioning: Y = Q1 R1 (Householder, R1 n x n), R1^T = Q2 R2, so that
        // R1 = R2^T Q2^T and the right singular vectors of Y are V = Q2 Z with Z those of R2^T.
        // The Jacobi then runs on R2^T, whose columns are already close to orthogonal and
        // graded, so it needs fewer sweeps and leaves a smaller tilt in the kept subspace than
        // on Y itself (at L = 256, chi = 32 in FP32: about half the sweeps and a five-fold
        // smaller 99.9th percentile of the conditional error).  Q1 is not kept; Q2's reflectors
        // overwrite R_c, which is not read again in this row, their coefficients go to csave.
        auto none = [](int) { return false; };
        const int g = lane % QB::G, gi = lane / QB::G;
        T x[QB::CPT][QB::RPT];
        auto load = [&](const T* A) {
#pragma unroll
          for (int q = 0; q < QB::CPT; ++q) {
            const int col = warp * QB::CW + q * QB::GPW + gi;
#pragma unroll
            for (int u = 0; u < QB::RPT; ++u) x[q][u] = T(0);
            if (col < n) qr_load_v<QB, 0, T>(A + (size_t)col * DP, g, x[q]);
          }
        };
        if (warp < QB::NTQ / 32) {
          // one body for both; pass 0: Y, its reflectors in Y's place, R1^T to V (stored for the next
          // pass); pass 1: R1^T, the reflectors in R_c's place, R2^T
          // to Y, zero outside n x n
#pragma unroll 1
          for (int pass = 0; pass < 2; ++pass) {
            load(pass ? Vc : Yc);
            if (pass == 0) {                                 // the reflectors take the place of what is read
              if constexpr (QB::NTQ == 32) __syncwarp();
              else named_barrier<2>(QB::NTQ);
            }
            const QrOut<T> out{pass ? Rc : Yc, csave, diag};
            qr_factor<T, D, D, C::RUN>(x, n, out, lane, warp, none);
            T* const to = pass ? Yc : Vc;
#pragma unroll
            for (int q = 0; q < QB::CPT; ++q) {
              const int col = warp * QB::CW + q * QB::GPW + gi;
              const int at = pass ? col : qr_pos<QB::G>(col);
              if (col < D) {
#pragma unroll
                for (int u = 0; u < QB::RPT; ++u) {
                  const int i = g + QB::G * u;
                  to[(size_t)i * DP + at] = (i <= col && col < n) ? x[q][u] : T(0);
                }
              }
            }
            if constexpr (QB::NTQ == 32) __syncwarp();
            else named_barrier<2>(QB::NTQ);
          }
          if constexpr (DP > D)
            for (int e = tid; e < (DP - D) * D; e += QB::NTQ) Yc[(size_t)(e / (DP - D)) * DP + D + e % (DP - D)] = T(0);
        }
        __syncthreads();
        if (sizeof(T) == 4 && tid < n) { const T den = csave[tid]; csave[tid] = den == T(0) ? den : T(1) / den; }
        for (int e = tid; e < DP * npad; e += NT) { const int i = e % DP, j = e / DP; Vc[e] = (i == j) ? T(1) : T(0); }
        __syncthreads();
      }
      const T tol = jacobi_tol<T, D>();
      // One-sided Jacobi in a block-cyclic order.  The npad columns form NB = npad/4 blocks of
      // four; in each block-round (a round-robin over blocks) warp wj owns one block pair and
      // its four 8-lane groups orthogonalise the 16 cross pairs in four sub-rounds (group i:
      // column i of block A against column (i+t) mod 4 of block B), and in the first
      // block-round also the six pairs inside each of its two blocks (three sub-rounds).  Every
      // pair of columns meets once per sweep; the columns a warp touches in a block-round are
      // its own, so sub-rounds are ordered by __syncwarp and only block-rounds need the
      // CTA-wide barrier (NB-1 per sweep instead of npad-1).  8 lanes per pair, each lane
      // holding DP/8 rows of both columns in 16-byte vectors.
      // Few pairs rotate: columns below tinyY never do (nor grow, so a block without a column
      // above it is left out for good), and of the others on the preconditioned matrix in FP32
      // about 70, 40, 6 and 0 of 2016 in the sweeps of a chi = 32 site, in 7.5, 6.2, 1.6 and 0.2 of
      // 91 block pairs (measured).  So a warp first tests its 16 pairs side by side, which is the
      // whole work of a block pair without rotations, and enters the sub-rounds at the first pair
      // that rotates; block-rounds without a live block pair are skipped, barrier and all.
      // 65 -> 27 thousand cycles a site at chi = 32 (L = 32); the build 150 -> 130 us a site step
      // with one realization per SM, 214 -> 172 with three.
      constexpr int NJ = 8 * CHI;
      constexpr int VEC = JStride<T, CHI>::VEC;
      constexpr int NV = DP / (8 * VEC);
      using V16 = typename Vec16<T>::type;
      int sweep = 0;
      if (tid < NJ) {
        const int wj = tid >> 5, grp = (tid >> 3) & 3, li = tid & 7;
        const int NB = npad / 4, mb = NB - 1;
        auto dot = [&](const V16* u, const V16* w) {
          T g = 0;
#pragma unroll
          for (int k = 0; k < NV; ++k) g += dot16(u[k], w[k]);
          return g;
        };
        // squared norm of a block-A column: with one vector per lane the other product of the
        // first two is the one rounded
        auto norm_a = [&](const V16* u) { return NV == 1 ? sq16(u[0]) : dot(u, u); };
        auto col = [&](T* base, int p) { return reinterpret_cast<V16*>(base + (size_t)p * DP) + li; };
        auto get = [&](V16* c, V16* u) {
#pragma unroll
          for (int k = 0; k < NV; ++k) u[k] = c[8 * k];
        };
        auto put = [&](V16* c, const V16* u) {
#pragma unroll
          for (int k = 0; k < NV; ++k) c[8 * k] = u[k];
        };
        // sums over the 8 lanes of a group, all values in step
        auto sum8 = [&](T* v, int n) {
#pragma unroll
          for (int o = 1; o <= 4; o <<= 1)
#pragma unroll
            for (int t = 0; t < n; ++t) v[t] += __shfl_xor_sync(0xffffffffu, v[t], o);
        };
        auto rotates = [&](T a, T b, T g) { return a > tinyY && b > tinyY && g * g > tol * tol * a * b; };
        // blocks with a column above tinyY (n2: the columns' squared norms; warp-uniform loops: the
        // shuffles need the whole warp)
        T* const n2 = sig;
        for (int p0 = wj * 4; p0 < npad; p0 += NJ / 8) {
          V16 u[NV];
          get(col(Yc, p0 + grp), u);
          T a[2] = {dot(u, u), norm_a(u)};
          sum8(a, 2);
          if (li == 0) n2[p0 + grp] = a[0] > a[1] ? a[0] : a[1];
        }
        named_barrier<1>(NJ);
        bool live = false;
        if (lane < NB) {
#pragma unroll
          for (int i = 0; i < 4; ++i) live |= n2[4 * lane + i] > tinyY;
        }
        const unsigned blocks = __ballot_sync(0xffffffffu, live);
        // block pair of slot w in block-round br (circle method: slot 0 keeps block NB-1)
        auto slot_pair = [&](int br, int w, int& bA, int& bB) {
          bA = w == 0 ? NB - 1 : (br + w >= mb ? br + w - mb : br + w);
          bB = w == 0 ? br : (br >= w ? br - w : br - w + mb);
        };
        // one pair from shared memory (inside a block)
        auto jpair = [&](int p, int q) {
          V16 up[NV], uq[NV];
          get(col(Yc, p), up);
          get(col(Yc, q), uq);
          T v[3] = {dot(up, uq), dot(up, up), dot(uq, uq)};
          sum8(v, 3);
          if (rotates(v[1], v[2], v[0])) {
            T cs, sn;
            rotation_from_gram(v[1], v[2], v[0], cs, sn);
            V16 wp[NV], wq[NV];
            get(col(Vc, p), wp);
            get(col(Vc, q), wq);
#pragma unroll
            for (int k = 0; k < NV; ++k) { rot16(up[k], uq[k], cs, sn); rot16(wp[k], wq[k], cs, sn); }
            put(col(Yc, p), up); put(col(Yc, q), uq);
            put(col(Vc, p), wp); put(col(Vc, q), wq);
            if (li == 0) rot[sweep % 3] = 1;
          }
        };
        for (; sweep < JacobiTol<T>::maxsw; ++sweep) {
          // clear the flag of sweep+1; the slot was last read at the end of sweep-2, and every
          // thread has passed a barrier of sweep-1 since (a two-slot ring would let a slow
          // thread read a flag that was already cleared and leave the loop alone)
          if (tid == 0) rot[(sweep + 1) % 3] = 0;
          for (int br = 0; br < mb; ++br) {
            int bA = 0, bB = 0;
            slot_pair(br, lane < NB / 2 ? lane : 0, bA, bB);
            const unsigned busy = __ballot_sync(0xffffffffu, lane < NB / 2 && ((blocks >> bA) & (blocks >> bB) & 1u));
            if (br > 0 && busy == 0) continue;         // no live block pair: the same in every warp
            if (wj < NB / 2) {
              slot_pair(br, wj, bA, bB);
              if (br == 0 && (((blocks >> bA) | (blocks >> bB)) & 1u)) {
                // pairs inside blocks A (groups 0, 1) and B (groups 2, 3):
                // {(0,1),(2,3)}, {(0,2),(1,3)}, {(0,3),(1,2)}
                const int blk = 4 * ((grp < 2) ? bA : bB), gi = grp & 1;
#pragma unroll 1
                for (int t = 0; t < 3; ++t) {
                  const int i = (t == 0) ? 2 * gi : gi;
                  const int j = (t == 0) ? 2 * gi + 1 : (t == 1 ? gi + 2 : 3 - gi);
                  jpair(blk + i, blk + j);
                  __syncwarp();
                }
              }
              if ((busy >> wj) & 1u) {
                // cross pairs: group grp holds column A = 4 bA + grp and meets the four columns
                // of block B in turn (B column (grp + t) mod 4 in sub-round t)
                const int pa = 4 * bA + grp;
                V16 ya[NV], va[NV];
                get(col(Yc, pa), ya);
                int t0 = 0;
                // The test pays where few block pairs rotate: on the preconditioned matrix in FP32
                // at once, on the zip-up's M (of the live block pairs 74, 54, 48, 42, 34, 24, 15 and
                // 9 % rotate in the sweeps of a chi = 32 site at L = 48; 66 to 24 % in the first five
                // at L = 24, 77 to 38 % at L = 64, 48 to 14 % at chi = 64) from the sixth sweep on
                // (L = 48, chi = 32: 277 ms, from the third 288, never 288), in FP64, whose tolerance
                // asks for more rotations, from the third on.
                if (sizeof(T) == 8 ? sweep >= 2 : (!zip || sweep >= 5)) {
                  T v[9];               // A's norm, four products, the four norms of block B
                  v[0] = norm_a(ya);
#pragma unroll
                  for (int t = 0; t < 4; ++t) {
                    V16 uq[NV];
                    get(col(Yc, 4 * bB + ((grp + t) & 3)), uq);
                    v[1 + t] = dot(ya, uq);
                    v[5 + t] = dot(uq, uq);
                  }
                  sum8(v, 9);
                  unsigned hit = 0;
#pragma unroll
                  for (int t = 0; t < 4; ++t) hit |= rotates(v[0], v[5 + t], v[1 + t]) ? 1u << t : 0u;
                  hit = __reduce_or_sync(0xffffffffu, hit);
                  t0 = hit ? __ffs(hit) - 1 : 4;
                }
                bool va_held = false;   // group-uniform: every lane of a group sees the same sums
#pragma unroll 1
                for (int t = t0; t < 4; ++t) {
                  const int q = 4 * bB + ((grp + t) & 3);
                  V16 uq[NV];
                  get(col(Yc, q), uq);
                  T v[3] = {dot(ya, uq), norm_a(ya), dot(uq, uq)};
                  sum8(v, 3);
                  if (rotates(v[1], v[2], v[0])) {
                    T cs, sn;
                    rotation_from_gram(v[1], v[2], v[0], cs, sn);
                    V16 wq[NV];
                    if (!va_held) { get(col(Vc, pa), va); va_held = true; }
                    get(col(Vc, q), wq);
#pragma unroll
                    for (int k = 0; k < NV; ++k) { rot16(ya[k], uq[k], cs, sn); rot16(va[k], wq[k], cs, sn); }
                    put(col(Yc, q), uq);
                    put(col(Vc, q), wq);
                    if (li == 0) rot[sweep % 3] = 1;
                  }
                  __syncwarp();
                }
                if (va_held) {          // column A changed: back to shared memory
                  put(col(Yc, pa), ya);
                  put(col(Vc, pa), va);
                }
              }
            }
            named_barrier<1>(NJ);
          }
          if (rot[sweep % 3] == 0) break;
        }
      }
      __syncthreads();
      if (sweep + 1 > max_sweeps_seen) max_sweeps_seen = sweep + 1;
      if (sweep >= JacobiTol<T>::maxsw) ++unconverged;
      total_sweeps += (long long)min(sweep + 1, JacobiTol<T>::maxsw);
      ++n_svd;
      // singular values = column norms of the rotated Y
      for (int j = warp; j < n; j += NWARP) {
        T ss = 0;
        for (int i = lane; i < D; i += 32) ss += Yc[(size_t)j * DP + i] * Yc[(size_t)j * DP + i];
        ss = warp_sum(ss);
        if (lane == 0) sig[j] = ss;
      }
      __syncthreads();
      const int k = min(chi, min(dqr[c], n));
      if (tid < n) {
        // a NaN ranks below every norm, so that the ranks are a permutation and all of sel is set
        // whatever the columns hold (an overflowed realization is flagged when it is sampled)
        const T sn = sig[tid], sj = sn >= T(0) ? sn : T(-1);
        int rank = 0;
        for (int i = 0; i < n; ++i) {
          const T st = sig[i], si = st >= T(0) ? st : T(-1);
          rank += (si > sj) || (si == sj && i < tid);
        }
        if (rank < k) sel[rank] = tid;
      }
      if (tid == 0) { knew[mir ? L - c : c] = k; knext_s = k; }
      __syncthreads();
      if (!zip) {
        // V_k = Q2 Z_sel = H_0 H_1 ... H_{n-1} Z_sel: each warp takes its selected columns into
        // registers, applies the reflectors from the last to the first, and writes the result to
        // column g of V (the selection becomes the identity)
        const int g = lane % QB::G, col = warp * QB::GPW + lane / QB::G;
        const bool mine = col < k;
        T xz[QB::RPT];
#pragma unroll
        for (int u = 0; u < QB::RPT; ++u) {
          const int i = g + QB::G * u;
          xz[u] = (mine && i < n) ? Vc[(size_t)sel[col] * DP + i] : T(0);
        }
        __syncthreads();
        if (warp * QB::GPW < k) {
          qr_apply_q<T, D, D, C::RUN>(xz, n, Rc, csave, g);
#pragma unroll
          for (int u = 0; u < QB::RPT; ++u) {
            const int i = g + QB::G * u;
            if (mine && i < n) Vc[(size_t)col * DP + i] = xz[u];
          }
        }
        __syncthreads();
        // R_{c-1} streams in while the tile and P are formed (the reflectors are consumed)
        if (c > 1) prefetch_async(Rc, Rstore + (size_t)(c - 1) * D * D, D * D * (int)sizeof(T), tid, NT);
      }
      // column of the g-th singular vector (already gathered unless zip-up)
      auto vcol = [&](int g) { return zip ? sel[g] : g; };
      // B_r[c][y][al][be] = V[(y,be)][sel[al]]
      T* ctile = cur + (size_t)osite(c) * TILE;
      TE* etile = erow + (size_t)osite(c) * TILE;
      for (int e = tid; e < TILE; e += NT) {
        const int y = e / (CHI * CHI), i = (e / CHI) % CHI, j = e % CHI;
        const int al = mir ? j : i, be = mir ? i : j;       // frame bonds of lattice entry (i, j)
        T v = T(0);
        if (al < k && be < kn) v = Vc[(size_t)vcol(al) * DP + y * kn + be];
        ctile[e] = v;
        etile[e] = env_store<TE, T>(v);
      }
      // P[(a,al)][g] = sum_j M[(a,al)][j] V[j][sel[g]]: 4 x 4 register tiles, at most one a thread,
      // kept until the largest entry is known
      {
        constexpr int TI = D / 4, TG = CHI / 4;
        static_assert(TI * TG <= NT, "one tile of P per thread");
        const int i0 = (tid % TI) * 4, g0 = (tid / TI) * 4;
        const bool mine = tid < TI * TG;
        T acc[4][4] = {}, pmax = 0;
        if (mine && g0 < k) {
          const T* vc[4];
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) vc[jj] = Vc + (size_t)vcol((g0 + jj < k) ? g0 + jj : g0) * DP;
#pragma unroll 4
          for (int j = 0; j < n; ++j) {
            T mv[4], vv[4];
            ld4(Mc + (size_t)j * D + i0, mv);
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) vv[jj] = (g0 + jj < k) ? vc[jj][j] : T(0);
#pragma unroll
            for (int ii = 0; ii < 4; ++ii)
#pragma unroll
              for (int jj = 0; jj < 4; ++jj) acc[ii][jj] += mv[ii] * vv[jj];
          }
#pragma unroll
          for (int ii = 0; ii < 4; ++ii)
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) { const T aa = acc[ii][jj] < T(0) ? -acc[ii][jj] : acc[ii][jj]; pmax = aa > pmax ? aa : pmax; }
        }
        pmax = warp_max(pmax);
        if (lane == 0) red[warp] = pmax;
        __syncthreads();
        const T pm = warp_max(lane < NWARP ? red[lane] : T(0));
        const T pinv = pm > T(0) ? T(1) / pm : T(1);
        if (mine) {
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            const T col4[4] = {acc[0][jj] * pinv, acc[1][jj] * pinv, acc[2][jj] * pinv, acc[3][jj] * pinv};
            st4(Ps + (size_t)(g0 + jj) * D + i0, col4);
          }
        }
        if (warp == 0) keep_scale(pm);
      }
      kn = knext_s;
      __syncthreads();
    }
    if (tid == 0) lam[r] = logs;
    __syncthreads();
  }

  // log Z = sum_r lam_r + log sum_x prod_c exp(beta Jh[0][c] s_c s_{c+1}) Gt_0(x)
  if constexpr (kBig) {
    // as below, each lane holding the bond indices lane + 32 e of the running vector
    constexpr int E = CHI / 32;
    if (warp == 0) {
      const T* row0 = rowbuf;
      double ell[2][E];
      double lsum = 0.0;
      for (int x = 0; x < 2; ++x) {
        const double h0 = hf ? exp(beta * (double)(hf[0] * spin_of(x))) : 1.0;
        for (int e = 0; e < E; ++e) ell[x][e] = h0 * (double)row0[x * CHI * CHI + 0 * CHI + lane + 32 * e];
      }
      for (int c = 1; c < L; ++c) {
        const T* t = row0 + (size_t)c * TILE;
        const double jb = beta * (double)Jh[c - 1];
        double nx[2][E];
        for (int x = 0; x < 2; ++x)
          for (int e = 0; e < E; ++e) nx[x][e] = 0.0;
        double f0[2], f1[2];
        for (int x = 0; x < 2; ++x) { f0[x] = exp(jb * spin_of(0) * spin_of(x)); f1[x] = exp(jb * spin_of(1) * spin_of(x)); }
        for (int h = 0; h < E; ++h)
          for (int j = 0; j < 32; ++j) {
            const int al = 32 * h + j;
            const double l0 = __shfl_sync(0xffffffffu, ell[0][h], j);
            const double l1 = __shfl_sync(0xffffffffu, ell[1][h], j);
            for (int x = 0; x < 2; ++x) {
              const double cf = f0[x] * l0 + f1[x] * l1;
              for (int e = 0; e < E; ++e) nx[x][e] += cf * (double)t[x * CHI * CHI + al * CHI + lane + 32 * e];
            }
          }
        if (hf)
          for (int x = 0; x < 2; ++x) {
            const double hc = exp(beta * (double)(hf[c] * spin_of(x)));
            for (int e = 0; e < E; ++e) nx[x][e] *= hc;
          }
        double mx = 0.0;
        for (int x = 0; x < 2; ++x)
          for (int e = 0; e < E; ++e) mx = fmax(mx, fabs(nx[x][e]));
        mx = warp_max(mx);
        for (int x = 0; x < 2; ++x)
          for (int e = 0; e < E; ++e) ell[x][e] = mx > 0.0 ? nx[x][e] / mx : nx[x][e];
        if (mx > 0.0) lsum += log(mx);
      }
      const double tot = __shfl_sync(0xffffffffu, ell[0][0] + ell[1][0], 0);
      if (lane == 0) {
        double s = 0.0;
        for (int rr = 0; rr < L; ++rr) s += lam[rr];
        args.logz[real] = s + lsum + log(tot);
        if (args.stats) {
          args.stats[real * 4 + 0] = max_sweeps_seen;
          args.stats[real * 4 + 1] = unconverged;
          args.stats[real * 4 + 2] = total_sweeps;
          args.stats[real * 4 + 3] = n_svd;
        }
      }
    }
  } else {
  if (warp == 0) {
    const T* row0 = rowbuf;   // row 0 lives in buffer (0 & 1) = 0
    double ell[2];            // lane holds ell[x][lane] for lane < CHI
    double lsum = 0.0;
    for (int x = 0; x < 2; ++x)
      ell[x] = (lane < CHI) ? (hf ? exp(beta * (double)(hf[0] * spin_of(x))) : 1.0) * (double)row0[x * CHI * CHI + 0 * CHI + lane] : 0.0;
    for (int c = 1; c < L; ++c) {
      const T* t = row0 + (size_t)c * TILE;
      const double jb = beta * (double)Jh[c - 1];
      double nx[2] = {0.0, 0.0};
      for (int al = 0; al < CHI; ++al) {
        const double l0 = __shfl_sync(0xffffffffu, ell[0], al);
        const double l1 = __shfl_sync(0xffffffffu, ell[1], al);
        for (int x = 0; x < 2; ++x) {
          const double f0 = exp(jb * spin_of(0) * spin_of(x)), f1 = exp(jb * spin_of(1) * spin_of(x));
          const double b = (lane < CHI) ? (double)t[x * CHI * CHI + al * CHI + lane] : 0.0;
          nx[x] += (f0 * l0 + f1 * l1) * b;
        }
      }
      if (hf) { nx[0] *= exp(beta * (double)hf[c]); nx[1] *= exp(-beta * (double)hf[c]); }
      double mx = fmax(fabs(nx[0]), fabs(nx[1]));
      mx = warp_max(mx);
      if (mx > 0.0) { nx[0] /= mx; nx[1] /= mx; lsum += log(mx); }
      ell[0] = nx[0]; ell[1] = nx[1];
    }
    const double tot = __shfl_sync(0xffffffffu, ell[0] + ell[1], 0);
    if (lane == 0) {
      double s = 0.0;
      for (int rr = 0; rr < L; ++rr) s += lam[rr];
      args.logz[real] = s + lsum + log(tot);
      if (args.stats) {
        args.stats[real * 4 + 0] = max_sweeps_seen;
        args.stats[real * 4 + 1] = unconverged;
        args.stats[real * 4 + 2] = total_sweeps;
        args.stats[real * 4 + 3] = n_svd;
      }
    }
  }
  }
}

template <typename T, typename TE, int CHI, bool kCrowd>
static cudaError_t env_build_setup(int L, size_t* smem) {
  // + the two rows' couplings (int8) staged behind the tile
  *smem = env_smem_elems<T, CHI>() * sizeof(T) + (size_t)2 * L + 16;
  return allow_shared_memory<env_build_kernel<T, TE, CHI, kCrowd>>();
}

template <typename T, typename TE, int CHI, bool kCrowd = false>
static cudaError_t launch_env_build_t(const EnvBuildArgs<T, TE>& a, cudaStream_t st) {
  if constexpr (CHI == 16 && sizeof(T) == 4 && !kCrowd) {
    // The crowd's build takes 4/3 of the time a full wave and holds 7/5 of the realizations: it is
    // the shorter one where it saves waves.
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int few = sms * EnvCfg<CHI, false>::PER_SM, many = sms * EnvCfg<CHI, true>::PER_SM;
    if (4 * ((a.n_real + many - 1) / many) < 3 * ((a.n_real + few - 1) / few)) return launch_env_build_t<T, TE, CHI, true>(a, st);
  }
  size_t smem = 0;
  const cudaError_t e = env_build_setup<T, TE, CHI, kCrowd>(a.L, &smem);
  if (e != cudaSuccess) return e;
  env_build_kernel<T, TE, CHI, kCrowd><<<a.n_real, EnvCfg<CHI>::NT, smem, st>>>(a);
  return cudaGetLastError();
}

template <typename T, typename TE>
cudaError_t launch_env_build(const EnvBuildArgs<T, TE>& a, int CHI, cudaStream_t st) {
  switch (CHI) {
    case 4: return launch_env_build_t<T, TE, 4>(a, st);
    case 8: return launch_env_build_t<T, TE, 8>(a, st);
    case 16: return launch_env_build_t<T, TE, 16>(a, st);
    case 32: return launch_env_build_t<T, TE, 32>(a, st);
    case 64:
      if constexpr (sizeof(T) == 4) return launch_env_build_t<T, TE, 64>(a, st);  // FP64 does not fit
      return cudaErrorInvalidValue;
    default: return cudaErrorInvalidValue;
  }
}

template cudaError_t launch_env_build<double, double>(const EnvBuildArgs<double, double>&, int, cudaStream_t);
template cudaError_t launch_env_build<float, float>(const EnvBuildArgs<float, float>&, int, cudaStream_t);
template cudaError_t launch_env_build<float, __nv_bfloat16>(const EnvBuildArgs<float, __nv_bfloat16>&, int, cudaStream_t);

template <typename T, typename TE, int CHI>
static cudaError_t occupancy_t(int L, int* per_sm) {
  size_t smem = 0;
  const cudaError_t e = env_build_setup<T, TE, CHI, false>(L, &smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, env_build_kernel<T, TE, CHI, false>, EnvCfg<CHI>::NT, smem);
}

cudaError_t env_build_occupancy(int L, int CHI, int precision, int* per_sm) {
#define TNMC_OCC(T, TE)                                           \
  switch (CHI) {                                                  \
    case 4: return occupancy_t<T, TE, 4>(L, per_sm);              \
    case 8: return occupancy_t<T, TE, 8>(L, per_sm);              \
    case 16: return occupancy_t<T, TE, 16>(L, per_sm);            \
    case 32: return occupancy_t<T, TE, 32>(L, per_sm);            \
    case 64:                                                      \
      if constexpr (sizeof(T) == 4) return occupancy_t<T, TE, 64>(L, per_sm); \
      return cudaErrorInvalidValue;                               \
    default: return cudaErrorInvalidValue;                        \
  }
  if (precision == 0) { TNMC_OCC(double, double) }
  if (precision == 2) { TNMC_OCC(float, __nv_bfloat16) }
  TNMC_OCC(float, float)
#undef TNMC_OCC
}

size_t env_build_smem_bytes(int CHI, bool fp64) {
  const size_t el = fp64 ? 8 : 4;
  switch (CHI) {
    case 4: return env_smem_elems<float, 4>() * el;
    case 8: return env_smem_elems<float, 8>() * el;
    case 16: return env_smem_elems<float, 16>() * el;
    case 32: return env_smem_elems<float, 32>() * el;
    case 64: return fp64 ? 0 : env_smem_elems<float, 64>() * el;
    default: return 0;
  }
}

}  // namespace tnmc
