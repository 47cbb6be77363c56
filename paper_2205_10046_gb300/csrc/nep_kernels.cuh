// NEP3 per-atom kernels for GB300 (sm_103a), templated on the model shape.
//
// Two kernels replace the four of the paper's Appendix B:
//   atom_kernel   two lanes per atom: radial descriptor (Eq. qin), angular sums S_nk
//                 (Eq. S_nk) and the explicit 3/4/5-body components (Sec. II D), the
//                 network U_i and dU_i/dq (Eq. Ui), then the per-type radial force
//                 coefficients and the angular partial forces dU_i/dr_ij (the angular terms
//                 of Eq. partial_force), stored per angular pair (Algorithms 1 and 3 fused).
//   gather_kernel two lanes per atom: F_i = sum_j [dU_i/dr_ij - dU_j/dr_ji] (Eqs. F_ij,
//                 F_i) and W_i = sum_j r_ij (x) dU_j/dr_ji (Eq. virial) for the radial
//                 part from both atoms' force coefficients and for the angular part from
//                 the stored partial forces of both atoms, with no atomics (Algorithms 2, 4).
//
// Differences from the paper's GPU design, for GB300:
//   * the radial descriptor accumulates the Chebyshev sums per neighbour type,
//     F^t_k = sum_{j of type t} f_k(r_ij), and contracts with c^{t_i t}_{nk} once per atom
//     (the radial list is grouped by neighbour type), so a pair costs O(K) instead of
//     O(n K); the radial partial forces likewise use e^t_k = sum_n dU/dq_n c^{t_i t}_{nk};
//   * S_nk are evaluated from the polynomials b_k of the unit vector, factored into powers of
//     (x + i y) and polynomials of z that the 24 of them share, and the angular gradient uses
//     the tangential projection of grad b_k, folded factor by factor;
//   * pair vectors come from cell-local FP32 coordinates plus an image shift table, so no
//     FP64 arithmetic (slow on GB300) runs in the pair loops;
//   * two lanes work on one atom and share a row of shared memory (S_nk, dU/dS_nk, q, dU/dq),
//     so an atom's sums fit 128 registers a thread and every phase has work for both lanes;
//     in small systems up to four groups of such lanes share an atom (kSplitAtoms).
#pragma once
#include <cuda_bf16.h>

#include "nep_internal.cuh"

namespace nep {

template <int NR_, int KR_, int NA_, int KA_, int H_, int L3_, int L4_, int L5_>
struct Shape {
  static constexpr int NR = NR_, KR = KR_, NA = NA_, KA = KA_, H = H_, L3 = L3_, L4 = L4_, L5 = L5_;
  static constexpr int NB = L3 + (L4 >= 2 ? 1 : 0) + (L5 >= 1 ? 1 : 0);
  static constexpr int NDES = (NR + 1) + (NA + 1) * NB;
  static constexpr int KEND3 = L3 == 1 ? 3 : L3 == 2 ? 8 : L3 == 3 ? 15 : 24;
  static constexpr int NK = KEND3 > 8 ? KEND3 : (L4 >= 2 ? 8 : KEND3);
  // radial force coefficients e_k of an atom and type and their sum (KR + 2 values): EF4 planes of
  // float4 over the atoms
  static constexpr int EF4 = (KR + 2 + 3) / 4;
  static constexpr int OFF4 = (NR + 1) + (NA + 1) * L3;
  static constexpr int OFF5 = OFF4 + (L4 >= 2 ? NA + 1 : 0);
  static constexpr int NDP = (NDES + 3) / 4 * 4;  // padded w0 row in shared memory
  // model table rows padded to whole float4s: c^A of a type pair (CAP), c^R rows over k (KRP)
  static constexpr int CAP = ((NA + 1) * (KA + 1) + 3) / 4 * 4;  // c^A of one type pair, [n][k] packed
  static constexpr int KRP = (KR + 1 + 3) / 4 * 4;  // c^R rows over k, padded likewise
  // float offsets of the shared regions after the shift table, each a whole number of float4s
  static constexpr int r4(int x) { return (x + 3) / 4 * 4; }
  // (the model table of TableLayout; without w0 where the network does not read it from there)
  static constexpr int off_b0(int prec) { return prec == 0 ? H * NDP : 0; }
  static constexpr int off_cR(int prec) { return off_b0(prec) + r4(2 * H + 1); }
  static constexpr int off_cA(int prec, int T) { return off_cR(prec) + T * T * (NR + 1) * KRP; }
  static constexpr int off_S(int prec, int T) { return off_cA(prec, T) + T * T * CAP; }
  // tensor-core network (BF16 operands, FP32 accumulation in TMEM), one 128-row tile (64 atoms and 64
  // unused rows):
  //   GEMM1 z[128 x NP1] = q[128 x KP1] . W0[NP1 x KP1]^T,  GEMM2 dq[128 x NP2] = beta[128 x KP2] . W0^T
  static constexpr int KP1 = (NDES + 15) / 16 * 16;
  static constexpr int NP1 = (H + 15) / 16 * 16;
  static constexpr int KP2 = NP1, NP2 = KP1;
  static constexpr int TILE_B = NP1 * KP1 * 2;           // bytes of a W0 tile
  static constexpr int ACOL = NP1 > NP2 ? NP1 : NP2;     // TMEM columns of the GEMM results; A after them
  static_assert(NP1 <= 256 && NP2 <= 256, "UMMA N limit");
};

// l of polynomial k (blocks 0-2, 3-7, 8-14, 15-23)
__host__ __device__ constexpr int l_of_k(int k) { return k < 3 ? 1 : k < 8 ? 2 : k < 15 ? 3 : 4; }

// b_k(d) of Sec. II D as homogeneous polynomials of the pair vector (s = |d|^2).
template <int k>
__device__ __forceinline__ float poly_b(float x, float y, float z, float s) {
  if constexpr (k == 0) return z;
  else if constexpr (k == 1) return x;
  else if constexpr (k == 2) return y;
  else if constexpr (k == 3) return 3.f * z * z - s;
  else if constexpr (k == 4) return x * z;
  else if constexpr (k == 5) return y * z;
  else if constexpr (k == 6) return x * x - y * y;
  else if constexpr (k == 7) return 2.f * x * y;
  else if constexpr (k == 8) return (5.f * z * z - 3.f * s) * z;
  else if constexpr (k == 9) return (5.f * z * z - s) * x;
  else if constexpr (k == 10) return (5.f * z * z - s) * y;
  else if constexpr (k == 11) return (x * x - y * y) * z;
  else if constexpr (k == 12) return 2.f * x * y * z;
  else if constexpr (k == 13) return (x * x - 3.f * y * y) * x;
  else if constexpr (k == 14) return (3.f * x * x - y * y) * y;
  else if constexpr (k == 15) return (35.f * z * z - 30.f * s) * z * z + 3.f * s * s;
  else if constexpr (k == 16) return (7.f * z * z - 3.f * s) * x * z;
  else if constexpr (k == 17) return (7.f * z * z - 3.f * s) * y * z;
  else if constexpr (k == 18) return (7.f * z * z - s) * (x * x - y * y);
  else if constexpr (k == 19) return (7.f * z * z - s) * 2.f * x * y;
  else if constexpr (k == 20) return (x * x - 3.f * y * y) * x * z;
  else if constexpr (k == 21) return (3.f * x * x - y * y) * y * z;
  else if constexpr (k == 22) return (x * x - y * y) * (x * x - y * y) - 4.f * x * x * y * y;
  else return 4.f * (x * x - y * y) * x * y;
}

// Gradient of b_k(d) with s = |d|^2 held fixed. Only its component tangential to d is
// used: grad |d|^2 = 2d is radial, so the tangential part equals that of the full gradient.
template <int k>
__device__ __forceinline__ float3 poly_grad(float x, float y, float z, float s) {
  if constexpr (k == 0) return make_float3(0.f, 0.f, 1.f);
  else if constexpr (k == 1) return make_float3(1.f, 0.f, 0.f);
  else if constexpr (k == 2) return make_float3(0.f, 1.f, 0.f);
  else if constexpr (k == 3) return make_float3(0.f, 0.f, 6.f * z);
  else if constexpr (k == 4) return make_float3(z, 0.f, x);
  else if constexpr (k == 5) return make_float3(0.f, z, y);
  else if constexpr (k == 6) return make_float3(2.f * x, -2.f * y, 0.f);
  else if constexpr (k == 7) return make_float3(2.f * y, 2.f * x, 0.f);
  else if constexpr (k == 8) return make_float3(0.f, 0.f, 15.f * z * z - 3.f * s);
  else if constexpr (k == 9) return make_float3(5.f * z * z - s, 0.f, 10.f * x * z);
  else if constexpr (k == 10) return make_float3(0.f, 5.f * z * z - s, 10.f * y * z);
  else if constexpr (k == 11) return make_float3(2.f * x * z, -2.f * y * z, x * x - y * y);
  else if constexpr (k == 12) return make_float3(2.f * y * z, 2.f * x * z, 2.f * x * y);
  else if constexpr (k == 13) return make_float3(3.f * (x * x - y * y), -6.f * x * y, 0.f);
  else if constexpr (k == 14) return make_float3(6.f * x * y, 3.f * (x * x - y * y), 0.f);
  else if constexpr (k == 15) return make_float3(0.f, 0.f, (140.f * z * z - 60.f * s) * z);
  else if constexpr (k == 16) return make_float3((7.f * z * z - 3.f * s) * z, 0.f, (21.f * z * z - 3.f * s) * x);
  else if constexpr (k == 17) return make_float3(0.f, (7.f * z * z - 3.f * s) * z, (21.f * z * z - 3.f * s) * y);
  else if constexpr (k == 18)
    return make_float3(2.f * x * (7.f * z * z - s), -2.f * y * (7.f * z * z - s), 14.f * z * (x * x - y * y));
  else if constexpr (k == 19)
    return make_float3(2.f * y * (7.f * z * z - s), 2.f * x * (7.f * z * z - s), 28.f * x * y * z);
  else if constexpr (k == 20)
    return make_float3(3.f * (x * x - y * y) * z, -6.f * x * y * z, (x * x - 3.f * y * y) * x);
  else if constexpr (k == 21)
    return make_float3(6.f * x * y * z, 3.f * (x * x - y * y) * z, (3.f * x * x - y * y) * y);
  else if constexpr (k == 22)
    return make_float3(4.f * x * (x * x - 3.f * y * y), 4.f * y * (y * y - 3.f * x * x), 0.f);
  else return make_float3(4.f * y * (3.f * x * x - y * y), 4.f * x * (x * x - 3.f * y * y), 0.f);
}

// b_k of the unit vector (x, y, z) = d / r: b_k(d) r^-l of Sec. II D. Every b_k is a polynomial
// Z(z) of degree l - m times Re or Im of (x + i y)^m, so a pair evaluates the few Z and the
// powers once (about 45 operations for all 24, where each b_k(d) by itself and its r^-l took
// about 100). UnitB holds the shared factors, ylm<k> combines them.
struct UnitB {
  float x, y, z, z2, z51, z71, z73, c2, s2, c3, s3;
};

__device__ __forceinline__ UnitB unit_b(float x, float y, float z) {
  UnitB u;
  u.x = x, u.y = y, u.z = z;
  u.z2 = __fmul_rn(z, z);
  u.z51 = __fmaf_rn(5.f, u.z2, -1.f);                  // 5 z^2 - 1
  u.z71 = __fmaf_rn(7.f, u.z2, -1.f);                  // 7 z^2 - 1
  u.z73 = __fmul_rn(__fmaf_rn(7.f, u.z2, -3.f), z);    // (7 z^2 - 3) z
  u.c2 = __fmaf_rn(x, x, -__fmul_rn(y, y));            // Re, Im (x + i y)^2
  u.s2 = __fmul_rn(__fadd_rn(x, x), y);
  u.c3 = __fmaf_rn(x, u.c2, -__fmul_rn(y, u.s2));      // Re, Im (x + i y)^3
  u.s3 = __fmaf_rn(x, u.s2, __fmul_rn(y, u.c2));
  return u;
}

template <int k>
__device__ __forceinline__ float ylm(const UnitB &u) {
  if constexpr (k == 0) return u.z;
  else if constexpr (k == 1) return u.x;
  else if constexpr (k == 2) return u.y;
  else if constexpr (k == 3) return __fmaf_rn(3.f, u.z2, -1.f);
  else if constexpr (k == 4) return __fmul_rn(u.x, u.z);
  else if constexpr (k == 5) return __fmul_rn(u.y, u.z);
  else if constexpr (k == 6) return u.c2;
  else if constexpr (k == 7) return u.s2;
  else if constexpr (k == 8) return __fmul_rn(__fmaf_rn(5.f, u.z2, -3.f), u.z);
  else if constexpr (k == 9) return __fmul_rn(u.z51, u.x);
  else if constexpr (k == 10) return __fmul_rn(u.z51, u.y);
  else if constexpr (k == 11) return __fmul_rn(u.c2, u.z);
  else if constexpr (k == 12) return __fmul_rn(u.s2, u.z);
  else if constexpr (k == 13) return u.c3;
  else if constexpr (k == 14) return u.s3;
  else if constexpr (k == 15) return __fmaf_rn(__fmaf_rn(35.f, u.z2, -30.f), u.z2, 3.f);
  else if constexpr (k == 16) return __fmul_rn(u.z73, u.x);
  else if constexpr (k == 17) return __fmul_rn(u.z73, u.y);
  else if constexpr (k == 18) return __fmul_rn(u.z71, u.c2);
  else if constexpr (k == 19) return __fmul_rn(u.z71, u.s2);
  else if constexpr (k == 20) return __fmul_rn(u.c3, u.z);
  else if constexpr (k == 21) return __fmul_rn(u.s3, u.z);
  else if constexpr (k == 22) return __fmaf_rn(u.c2, u.c2, -__fmul_rn(u.s2, u.s2));
  else return __fmul_rn(__fadd_rn(u.c2, u.c2), u.s2);
}

// Order in which the force loop takes the 24 polynomials, four at a time: the ones that share
// Re or Im (x + i y)^m together. dU/dS_nk rows are kept in this order.
__host__ __device__ constexpr int harm_k(int j) {
  constexpr int o[24] = {0, 3, 8, 15, 1, 4, 9, 16, 2, 5, 10, 17, 6, 11, 18, 13, 7, 12, 19, 14, 20, 22, 21, 23};
  return o[j];
}

// One group of four (harm_k(4 Q) ...) of one pair: with a_k = sum_n dU/dS_nk g_n and c_k =
// sum_n dU/dS_nk g_n', adds sum_k a_k grad b_k (b_k as polynomials of the unit vector, |u|
// held at 1: only the tangential part is used) to (gx, gy, gz) and sum_k c_k b_k to Y. The four
// share their Re / Im factor, so their Z and Z' sums are formed first.
template <int Q>
__device__ __forceinline__ void harm_fold(const UnitB &u, const float *a, const float *c, float &gx, float &gy, float &gz,
                                          float &Y) {
  if constexpr (Q == 0) {  // m = 0
    gz = __fadd_rn(gz, __fmaf_rn(a[3], __fmul_rn(__fmaf_rn(140.f, u.z2, -60.f), u.z),
                                 __fmaf_rn(a[2], __fmaf_rn(15.f, u.z2, -3.f), __fmaf_rn(a[1], __fmul_rn(6.f, u.z), a[0]))));
    Y = __fmaf_rn(c[0], u.z, Y);
    Y = __fmaf_rn(c[1], __fmaf_rn(3.f, u.z2, -1.f), Y);
    Y = __fmaf_rn(c[2], __fmul_rn(__fmaf_rn(5.f, u.z2, -3.f), u.z), Y);
    Y = __fmaf_rn(c[3], __fmaf_rn(__fmaf_rn(35.f, u.z2, -30.f), u.z2, 3.f), Y);
  } else if constexpr (Q == 1 || Q == 2) {  // m = 1: x, y
    const float A = __fmaf_rn(a[3], u.z73, __fmaf_rn(a[2], u.z51, __fmaf_rn(a[1], u.z, a[0])));
    const float C = __fmaf_rn(c[3], u.z73, __fmaf_rn(c[2], u.z51, __fmaf_rn(c[1], u.z, c[0])));
    const float D = __fmaf_rn(a[3], __fmaf_rn(21.f, u.z2, -3.f), __fmaf_rn(a[2], __fmul_rn(10.f, u.z), a[1]));
    const float w = Q == 1 ? u.x : u.y;
    if constexpr (Q == 1) gx = __fadd_rn(gx, A);
    else gy = __fadd_rn(gy, A);
    gz = __fmaf_rn(D, w, gz);
    Y = __fmaf_rn(C, w, Y);
  } else if constexpr (Q == 3 || Q == 4) {  // m = 2 (three), and the first of m = 3
    const float A = __fmaf_rn(a[2], u.z71, __fmaf_rn(a[1], u.z, a[0]));
    const float C = __fmaf_rn(c[2], u.z71, __fmaf_rn(c[1], u.z, c[0]));
    const float D = __fmaf_rn(a[2], __fmul_rn(14.f, u.z), a[1]);
    const float A2 = __fadd_rn(A, A), A3 = __fmul_rn(3.f, a[3]);
    if constexpr (Q == 3) {  // c2, c3: d/dx = 2x, 3 c2; d/dy = -2y, -3 s2
      gx = __fmaf_rn(A3, u.c2, __fmaf_rn(A2, u.x, gx));
      gy = __fmaf_rn(-A3, u.s2, __fmaf_rn(-A2, u.y, gy));
      gz = __fmaf_rn(D, u.c2, gz);
      Y = __fmaf_rn(c[3], u.c3, __fmaf_rn(C, u.c2, Y));
    } else {  // s2, s3: d/dx = 2y, 3 s2; d/dy = 2x, 3 c2
      gx = __fmaf_rn(A3, u.s2, __fmaf_rn(A2, u.y, gx));
      gy = __fmaf_rn(A3, u.c2, __fmaf_rn(A2, u.x, gy));
      gz = __fmaf_rn(D, u.s2, gz);
      Y = __fmaf_rn(c[3], u.s3, __fmaf_rn(C, u.s2, Y));
    }
  } else {  // c3 z, c4, s3 z, s4
    const float z3 = __fmul_rn(3.f, u.z);
    const float A0 = __fmul_rn(a[0], z3), A1 = __fmul_rn(a[2], z3);
    gx = __fmaf_rn(A1, u.s2, __fmaf_rn(A0, u.c2, gx));
    gy = __fmaf_rn(A1, u.c2, __fmaf_rn(-A0, u.s2, gy));
    gz = __fmaf_rn(a[2], u.s3, __fmaf_rn(a[0], u.c3, gz));
    const float B0 = __fmul_rn(4.f, a[1]), B1 = __fmul_rn(4.f, a[3]);
    gx = __fmaf_rn(B1, u.s3, __fmaf_rn(B0, u.c3, gx));
    gy = __fmaf_rn(B1, u.c3, __fmaf_rn(-B0, u.s3, gy));
    Y = __fmaf_rn(u.z, __fmaf_rn(c[2], u.s3, __fmul_rn(c[0], u.c3)), Y);
    Y = __fmaf_rn(c[1], ylm<22>(u), Y);
    Y = __fmaf_rn(c[3], ylm<23>(u), Y);
  }
}

// Unrolled compile-time loop helper.
template <int I, int N, class F>
__device__ __forceinline__ void static_for(F &&f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    static_for<I + 1, N>(f);
  }
}

// ------------------------------------------------------------------ tcgen05 / mbarrier
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor, no swizzle: start address, LBO (next 8x16-byte core matrix
// along K), SBO (next core matrix along M/N), version bit.
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}

// Instruction descriptor: BF16 x BF16 -> FP32, both operands K-major, M x N.
template <int M, int N>
__host__ __device__ constexpr uint32_t umma_idesc_bf16() {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// The same with B read MN-major (transpose-B bit): core matrices of 8 K-rows x 16 bytes of
// consecutive N, SBO the step along N and LBO the step along K. A K-major tile of W0 for
// D = A.W0^T read this way is W0 itself as the K x N operand of D = A.W0.
template <int M, int N>
__host__ __device__ constexpr uint32_t umma_idesc_bf16_bmn() {
  return umma_idesc_bf16<M, N>() | (1u << 16);
}

__device__ __forceinline__ void umma_commit(uint64_t *mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(mbar))
               : "memory");
}

// Wait for an mbarrier phase with an iteration limit; returns false if the limit ran out.
__device__ __forceinline__ bool mbar_wait(uint64_t *mbar, uint32_t parity) {
  uint32_t done = 0;
  for (int it = 0; it < (1 << 24) && !done; ++it) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(smem_addr(mbar)), "r"(parity)
        : "memory");
  }
  return done != 0;
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float *v) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(r[j]);
}

// D (+)= A.B with the A operand read from tensor memory (lane m = row m, K packed along the
// columns: two BF16 values per 32-bit column, the lower K index in the low half).
__device__ __forceinline__ void umma_bf16_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t db, uint32_t idesc,
                                             uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(tmem_d),
      "r"(tmem_a), "l"(db), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void tmem_st4u(uint32_t taddr, const uint32_t *v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(taddr), "r"(v[0]), "r"(v[1]),
               "r"(v[2]), "r"(v[3])
               : "memory");
}

// f_k(r) = (T_k(x) + 1) fc/2 with fc = (1 + cos(pi r/rc))/2 and x = 2(r/rc - 1)^2 - 1
// (Eq. f_n and the cosine cutoff); fills f[0..K].
template <int K>
__device__ __forceinline__ void cheb_basis(float r, float inv_rc, float *f) {
  const float u = r * inv_rc;
  const float hfc = 0.25f * (1.f + __cosf(3.14159265358979f * u));
  const float t1 = u - 1.f;
  const float x = 2.f * t1 * t1 - 1.f;
  const float x2 = 2.f * x;
  float tkm1 = 1.f, tk = x;
  f[0] = 2.f * hfc;
  if constexpr (K >= 1) f[1] = __fmaf_rn(x, hfc, hfc);
#pragma unroll
  for (int k = 2; k <= K; ++k) {
    const float tn = __fmaf_rn(x2, tk, -tkm1);
    tkm1 = tk;
    tk = tn;
    f[k] = __fmaf_rn(tn, hfc, hfc);
  }
}

// f_k(r) and f_k'(r) for k = 0..K.
template <int K>
__device__ __forceinline__ void cheb_basis_d(float r, float inv_rc, float *f, float *fp) {
  const float u = r * inv_rc;
  float sn, cs;
  __sincosf(3.14159265358979f * u, &sn, &cs);
  const float hfc = 0.25f * (1.f + cs);                       // fc/2
  const float hfcp = -0.25f * 3.14159265358979f * inv_rc * sn; // fc'/2
  const float t1 = u - 1.f;
  const float x = 2.f * t1 * t1 - 1.f;
  const float xp = 4.f * t1 * inv_rc;  // dx/dr
  const float x2 = 2.f * x;
  const float a = xp * hfc;            // T_k' coefficient
  float tkm1 = 1.f, tk = x, dkm1 = 0.f, dk = 1.f;
  f[0] = 2.f * hfc;
  fp[0] = 2.f * hfcp;
  if constexpr (K >= 1) {
    f[1] = __fmaf_rn(x, hfc, hfc);
    fp[1] = __fmaf_rn(a, 1.f, (x + 1.f) * hfcp);
  }
#pragma unroll
  for (int k = 2; k <= K; ++k) {
    const float tn = __fmaf_rn(x2, tk, -tkm1);
    const float dn = __fmaf_rn(x2, dk, __fmaf_rn(2.f, tk, -dkm1));
    tkm1 = tk;
    tk = tn;
    dkm1 = dk;
    dk = dn;
    f[k] = __fmaf_rn(tn, hfc, hfc);
    fp[k] = __fmaf_rn(a, dn, (tn + 1.f) * hfcp);
  }
}

// Request the line holding *p into L2 (no register, no wait). Callers keep p inside the
// list allocation: slot rows below the list capacity.
__device__ __forceinline__ void l2_prefetch(const void *p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// The shift table of one structure in shared memory, component by component: the lanes of a
// warp hold different image codes, and 4-byte reads of up to 64 codes meet few bank conflicts
// (16-byte entries took 8 passes of the shared memory per read).
__device__ __forceinline__ void stage_shifts(const AtomArgs &a, float *tab) {
  for (int v = threadIdx.x; v < a.ncode; v += blockDim.x) {
    const float4 d = a.dtab[v];
    tab[v] = d.x, tab[a.ncode + v] = d.y, tab[2 * a.ncode + v] = d.z;
  }
}
__device__ __forceinline__ float4 shift_at(const float *tab, int ncode, unsigned code) {
  return make_float4(tab[code], tab[ncode + code], tab[2 * ncode + code], 0.f);
}

// The block's copy of the model table into shared memory, from float `from` on (whole float4s).
template <class S>
__device__ __forceinline__ void stage_table(const float *tab, int from, int T, float *dst) {
  const float4 *src = reinterpret_cast<const float4 *>(tab + from);
  const int n4 = (S::off_S(0, T) - from) / 4;
  for (int v = threadIdx.x; v < n4; v += blockDim.x) reinterpret_cast<float4 *>(dst)[v] = __ldg(src + v);
}

// Load of a list entry: read-only cached, or streaming (evict-first) for a list that the
// kernel reads only once, so that it does not push the neighbours' data out of L1.
template <bool STREAM, class T>
__device__ __forceinline__ T ld_list(const T *p) {
  if constexpr (STREAM) return __ldcs(p);
  else return __ldg(p);
}

// Batched variant for short pair bodies: the positions of D pairs are requested together and
// the list entries AHEAD (1 or 2) batches ahead (the lists stream from DRAM).
template <int D, bool STREAM = false, int AHEAD = 2, class Body>
__device__ __forceinline__ void for_pairs_batch(const unsigned *__restrict__ nl, int slot0, int cnt, int N, int i,
                                                const float4 *__restrict__ pos4, unsigned jmask, Body &&body) {
  if (cnt <= 0) return;
  const unsigned *col = nl + (size_t)slot0 * N + i;
  unsigned e[D], en[D];
#pragma unroll
  for (int d = 0; d < D; ++d) e[d] = d < cnt ? ld_list<STREAM>(col + (size_t)d * N) : 0u;
  if constexpr (AHEAD == 2) {
#pragma unroll
    for (int d = 0; d < D; ++d) en[d] = D + d < cnt ? ld_list<STREAM>(col + (size_t)(D + d) * N) : 0u;
  }
  for (int m0 = 0; m0 < cnt; m0 += D) {
    float4 p[D];
#pragma unroll
    for (int d = 0; d < D; ++d) p[d] = __ldg(pos4 + (e[d] & jmask));
    unsigned enn[D];
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const int m = m0 + AHEAD * D + d;
      enn[d] = m < cnt ? ld_list<STREAM>(col + (size_t)m * N) : 0u;
    }
#pragma unroll
    for (int d = 0; d < D; ++d)
      if (m0 + d < cnt) body(m0 + d, e[d], p[d]);
#pragma unroll
    for (int d = 0; d < D; ++d) {
      if constexpr (AHEAD == 2) {
        e[d] = en[d];
        en[d] = enn[d];
      } else {
        e[d] = enn[d];
      }
    }
  }
}

// ------------------------------------------------------------------------ per-atom kernel
// Two lanes per atom (h = 0, 1), AB atoms per block of 2 AB threads. The pair of lanes shares
// one row of shared memory per atom: S_nk (later dU/dS_nk) and q (later dU/dq).
//   radial sums      each lane takes every second neighbour of a type; the sums are added
//                    across the pair, each lane contracts every second n with c_nk;
//   S_nk             each lane prepares every second pair and hands it across; lane 0 sums the
//                    polynomials with Re (x + i y)^m (and two of m = 0), lane 1 those with Im (and
//                    the other two): the same instructions on swapped factors, 12 (n_max^A + 1)
//                    sums a lane;
//   components       each lane takes every second n; the row passes S_nk and q across;
//   network          each lane holds every second float4 of q and dU/dq; see there;
//   dU/dS_nk         every second n, in place of S_nk;
//   partial forces   pairs 4 t + 2 h and 4 t + 2 h + 1: two pairs share every read of dU/dS_nk.
//
// What bounds it: instruction issue (70% of the slots busy with 16 warps per SM; FP32 arithmetic
// is 72% of the instructions), then shared-memory bandwidth (59%). One thread per atom, with
// all (n_max^A + 1) 24 sums in its registers or in two passes, ran 8 to 12 warps per SM and left
// small systems to one long serial chain per atom. One thread / two lanes per atom, us: 216 Si
// atoms 46 / 26, 13,824 Si atoms 41 / 28, 262,144 PbTe atoms 248 / 233, 8,000,000 Si atoms
// 7787 / 7181, 4096 structures (1.05 million atoms) 1528 / 1173, 32 candidates on 256 structures
// 3010 / 2318. Of that, reading the model table from global memory instead of copying it from
// the kernel parameters (lane-varying constant addresses, served one by one) took 0.8 ms of the
// 8,000,000-atom step, and the factored polynomials 0.6 ms.
// Small systems: up to kSplitAtoms atoms of one structure, four groups of lanes work on an atom (16
// atoms per block of 128 threads), up to kSplitAtoms2 two (32 atoms per block). The sums over
// neighbours stay with the first group, whose lanes add in the same order as ever (the same bits);
// the network, the components, dU/dS_nk and the partial forces, which are independent term by term,
// are shared. The limits are three such blocks on each of the 152 SMs (one wave of the shapes that hold
// three, less of those that hold four): beyond it the groups that wait cost more than the shorter
// chain gives. A dynamics step without / with, us (the gather kernel
// split in both): 216 Si atoms 40 / 36, 5,832 46 / 43, 8,000 46.4 / 45.8, 13,824 57.4 / 55.4, past the
// limits with four groups 13,824 Si atoms 63 / 71, 8,000 PbTe atoms 41 / 50.
template <class S>
struct PairRow {
  static constexpr int Q4 = S::NDP / 4;                  // float4s of q
  static constexpr int S4 = (S::NA + 1) * 6;             // float4s of S_nk
  static constexpr int R4 = (Q4 + S4) | 1;               // odd: 8 consecutive rows on 8 bank groups
  static constexpr int OCC = S::NA <= 4 ? 4 : 3;         // blocks of 128 threads per SM (shared memory)
  // tensor-core network (prec: BF16 terms per operand value): TMEM columns of the block
  static constexpr int AC = (S::KP1 > S::KP2 ? S::KP1 : S::KP2) / 2;  // columns of one A term
  static constexpr int COLS = 128;
  static_assert(S::ACOL + 2 * AC <= COLS, "results and both A terms within the block's TMEM columns");
  static constexpr bool tc(int prec) { return prec > 0; }
  // float offset of the rows in shared memory, after the table and the W0 tiles
  static constexpr int from(int prec) { return tc(prec) ? S::off_b0(0) : 0; }
  static constexpr int off_tiles(int prec, int T) { return S::off_S(0, T) - from(prec); }
  static constexpr int off_rows(int prec, int T) {
    return off_tiles(prec, T) + (tc(prec) ? prec * S::TILE_B / 4 : 0);
  }
};

template <class S, int PREC, bool DESC, bool BATCH, int AB, int SUB>
__global__ void __launch_bounds__(2 * AB *SUB, PairRow<S>::OCC * 64 / (AB * SUB))
    atom_kernel(const AtomArgs a, const __grid_constant__ ModelF mf) {
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int NR = S::NR, KR = S::KR, NA = S::NA, KA = S::KA, NDES = S::NDES, NDP = S::NDP;
  constexpr int CAP = S::CAP, KRP = S::KRP, NJ = (NA + 2) / 2;
  static_assert(S::NK == 24, "harm_k lists the 24 polynomials of l <= 4");
  extern __shared__ float4 smem4[];
  const int T = a.T, N = a.N;
  static_assert(SUB == 1 || (PREC == 0 && !DESC && AB % 16 == 0), "forces with the FP32 network");
  // SUB > 1: SUB groups of 2 AB threads, lanes of the same atoms
  const int sub = SUB > 1 ? threadIdx.x / (2 * AB) : 0, tl = SUB > 1 ? threadIdx.x % (2 * AB) : threadIdx.x;
  const int h = tl & 1, ia = tl >> 1;
  // rows written by an atom's lanes, read by its other lanes
  auto sync_rows = [&]() {
    if constexpr (SUB > 1) __syncthreads();
    else __syncwarp();
  };
  const int i = blockIdx.x * AB + ia;
  // Lanes past the last atom, and (serving engine) those of a finished job frozen in the batch,
  // run along with no neighbours (the pair exchanges are warp-collective); they write nothing.
  const float4 pi = i < N ? __ldg(a.pos4 + i) : make_float4(0.f, 0.f, 0.f, __int_as_float(0));
  const bool failed = build_failed(a.guard);  // tested once the block's setup is under way
  const bool active = i < N && !(BATCH && a.slots && (failed || a.slots[struct_of(pi)].phase == 2));
  const int na = active ? __ldg(a.nn_a + i) : 0;
  int cnt_r = active ? __ldg(a.nn_r + i) : 0;
  if (active) {  // the first list slots into L2 before the block's setup
#pragma unroll
    for (int m = 0; m < 16; m += 2)
      if (m + h < a.cap_r) l2_prefetch(a.nl_r + (size_t)(m + h) * N + i);
    if (h < a.cap_a) l2_prefetch(a.nl_a + (size_t)h * N + i);
  }
  const int mem = BATCH ? (int)blockIdx.y : 0;
  using PR = PairRow<S>;
  constexpr bool TC = PR::tc(PREC);
  static_assert(!DESC || PREC == 0, "the descriptors need no network");
  constexpr int NT = TC ? PREC : 1;  // BF16 terms per operand value of the tensor-core network
  // W0 tiles first (16-byte core matrices), then the shift table, the model table and the rows
  float *tiles = reinterpret_cast<float *>(smem4);
  float4 *dtab_s = smem4 + (TC ? NT * S::TILE_B / 16 : 0);  // [ncode] (one structure)
  float *w0_s = reinterpret_cast<float *>(dtab_s + (BATCH ? 0 : a.ncode)) - PR::from(PREC);  // [H][NDP] (FMA network)
  float *b0_s = w0_s + S::off_b0(0), *w1_s = b0_s + S::H;                  // [H]; [H], then b1
  float *cR_s = w0_s + S::off_cR(0);      // [T][T][NR+1][KRP]
  float *cA_s = w0_s + S::off_cA(0, T);   // [T][T][CAP]
  float4 *const rows = reinterpret_cast<float4 *>(w0_s + S::off_S(0, T));
  float4 *const row = rows + ia * PR::R4;  // [n][6], then q
  float *const qrow = reinterpret_cast<float *>(row + PairRow<S>::S4);
  if constexpr (!BATCH)
    stage_shifts(a, reinterpret_cast<float *>(dtab_s));
  stage_table<S>(a.tab + mem * a.s_tab, PR::from(PREC), T, w0_s + PR::from(PREC));
  if (failed) return;
  __shared__ __align__(8) uint64_t tc_mbar;
  __shared__ uint32_t tc_tmem;
  __shared__ float u_s[TC ? AB : 1];  // U of the rows
  if constexpr (TC) {
    const float4 *src = reinterpret_cast<const float4 *>(a.tab + mem * a.s_tab + S::off_S(0, T));
    for (int v = threadIdx.x; v < NT * S::TILE_B / 16; v += blockDim.x) reinterpret_cast<float4 *>(tiles)[v] = __ldg(src + v);
    if (threadIdx.x == 0) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&tc_mbar)));
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the tiles, before the MMAs read them
    if (threadIdx.x < 32) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tc_tmem)),
                   "r"((uint32_t)PR::COLS));
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  const int ti = type_of(pi);
  const float inv_rcR = 1.f / a.rcR, inv_rcA = 1.f / a.rcA;
  const float rcR2 = a.rcR * a.rcR, rcA2 = a.rcA * a.rcA;
  // shift vector of a list entry: from shared memory, or from the structure's own table
  const float4 *dtab_b = BATCH ? a.dtab + (size_t)struct_of(pi) * a.ncode : dtab_s;
  auto shift = [&](unsigned e) -> float4 {
    if constexpr (BATCH) return __ldg(dtab_b + (e >> a.jbits));
    else return shift_at(reinterpret_cast<const float *>(dtab_s), a.ncode, e >> a.jbits);
  };

  // ---- radial descriptor, Eq. qin: per neighbour type, sum_j T_k(x_j) fc_j/2 (k >= 1) and
  // sum_j fc_j/2, then F_0 = 2H, F_k = sum_j T_k fc_j/2 + H, contracted with c_nk
  if (sub == 0) {
    float qr[(NR + 2) / 2];
#pragma unroll
    for (int j = 0; j < (NR + 2) / 2; ++j) qr[j] = 0.f;
    int base = 0;
    for (int t = 0; t < T; ++t) {
      const int cnt = cnt_r;
      if (t + 1 < T) {  // the next type's count, and its first slots into L2
        cnt_r = active ? __ldg(a.nn_r + (size_t)(t + 1) * N + i) : 0;
        if (active)
#pragma unroll
          for (int m = 0; m < 16; m += 2)
            if (base + cnt + m + h < a.cap_r) l2_prefetch(a.nl_r + (size_t)(base + cnt + m + h) * N + i);
      }
      float Fk[KR + 1];
#pragma unroll
      for (int k = 0; k <= KR; ++k) Fk[k] = 0.f;
      // entries h, h + 2, ... of the type's group
      for_pairs_batch<4, true>(a.nl_r + (size_t)(base + h) * N, 0, (cnt + 1 - h) >> 1, 2 * N, i, a.pos4, a.jmask,
                               [&](int, unsigned e, const float4 &pj) {
        const float3 d = pair_vector(pi, pj, shift(e));
        const float r2 = norm2(d);
        if (r2 < rcR2) {
          const float u = r2 * rsqrtf(r2) * inv_rcR;
          const float hfc = 0.25f * (1.f + __cosf(3.14159265358979f * u));
          const float t1 = u - 1.f;
          const float x = 2.f * t1 * t1 - 1.f;
          const float x2 = 2.f * x;
          Fk[0] += hfc;
          if constexpr (KR >= 1) Fk[1] = __fmaf_rn(x, hfc, Fk[1]);
          float tkm1 = 1.f, tk = x;
#pragma unroll
          for (int k = 2; k <= KR; ++k) {
            const float tn = __fmaf_rn(x2, tk, -tkm1);
            tkm1 = tk;
            tk = tn;
            Fk[k] = __fmaf_rn(tn, hfc, Fk[k]);
          }
        }
      });
#pragma unroll
      for (int k = 0; k <= KR; ++k) Fk[k] = __fadd_rn(Fk[k], __shfl_xor_sync(kAll, Fk[k], 1));
#pragma unroll
      for (int k = 1; k <= KR; ++k) Fk[k] = __fadd_rn(Fk[k], Fk[0]);
      Fk[0] = __fadd_rn(Fk[0], Fk[0]);
      const float4 *c = reinterpret_cast<const float4 *>(cR_s + (ti * T + t) * (NR + 1) * KRP);
#pragma unroll
      for (int j = 0; j < (NR + 2) / 2; ++j) {
        const int n = min(2 * j + h, NR);
        float acc = qr[j];
#pragma unroll
        for (int k4 = 0; k4 < KRP / 4; ++k4) {
          const float4 cv = c[n * (KRP / 4) + k4];
          const float cw[4] = {cv.x, cv.y, cv.z, cv.w};
#pragma unroll
          for (int jj = 0; jj < 4; ++jj)
            if (4 * k4 + jj <= KR) acc = __fmaf_rn(cw[jj], Fk[4 * k4 + jj], acc);
        }
        qr[j] = acc;
      }
      base += cnt;
    }
#pragma unroll
    for (int j = 0; j < (NR + 2) / 2; ++j)
      if (2 * j + h <= NR) qrow[2 * j + h] = qr[j];
    if (h == 0)
#pragma unroll
      for (int v = NDES; v < NDP; ++v) qrow[v] = 0.f;
  }

  // ---- angular sums S_nk (Eq. S_nk, b_k of the unit vector): this lane's 12 polynomials
  if (sub == 0) {
    float Sv[NA + 1][12];
#pragma unroll
    for (int n = 0; n <= NA; ++n)
#pragma unroll
      for (int j = 0; j < 12; ++j) Sv[n][j] = 0.f;
    // Lane h takes entries h, h + 2, ...: distance, basis and g_n of its own pair, which the other
    // lane gets by shuffles (both lanes computing every pair took 40 instructions per atom and
    // pair more); each lane then adds both pairs to its own sums. Entries are fetched two steps
    // ahead, positions one.
    const unsigned *col = a.nl_a + i;
    unsigned e0 = h < na ? __ldg(col + (size_t)h * N) : 0u;
    unsigned e1 = h + 2 < na ? __ldg(col + (size_t)(h + 2) * N) : 0u;
    float4 p0 = __ldg(a.pos4 + (e0 & a.jmask));
    const int steps = __reduce_max_sync(kAll, na);
#pragma unroll 1
    for (int m = h; m < steps + h; m += 2) {
      const float3 d = pair_vector(pi, p0, shift(e0));
      const int tj = type_of(p0);
      const float r2 = norm2(d);
      const bool in = m < na && r2 < rcA2;
      e0 = e1;
      if (m + 2 < na) p0 = __ldg(a.pos4 + (e0 & a.jmask));
      e1 = m + 4 < na ? __ldg(col + (size_t)(m + 4) * N) : 0u;
      float g[NA + 1], x = 0.f, y = 0.f, z = 0.f;
#pragma unroll
      for (int n = 0; n <= NA; ++n) g[n] = 0.f;
      if (in) {
        const float rinv = rsqrtf(r2);
        float f[KA + 1];
        cheb_basis<KA>(r2 * rinv, inv_rcA, f);
        const float4 *c4 = reinterpret_cast<const float4 *>(cA_s + (ti * T + tj) * CAP);
#pragma unroll
        for (int v = 0; v < CAP / 4; ++v) {
          const float4 cv = c4[v];
          const float cw[4] = {cv.x, cv.y, cv.z, cv.w};
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (4 * v + j < (NA + 1) * (KA + 1)) {
              const int n = (4 * v + j) / (KA + 1), k = (4 * v + j) % (KA + 1);
              g[n] = __fmaf_rn(cw[j], f[k], g[n]);
            }
        }
        x = __fmul_rn(d.x, rinv), y = __fmul_rn(d.y, rinv), z = __fmul_rn(d.z, rinv);
      }
      // a pair outside the cutoff is passed on with g = 0 (and a finite vector)
      auto add_pair = [&](const UnitB &u, const float *gn) {
        // lane 0: 0, 3 | 1, 4, 9, 16 | 6, 11, 18, 13 | 20, 22; lane 1: 8, 15 | 2, 5, 10, 17 |
        // 7, 12, 19, 14 | 21, 23 (the order of harm_k, split in two)
        const float w1 = h ? u.y : u.x, w2 = h ? u.s2 : u.c2, w3 = h ? u.s3 : u.c3;
        const float bb[12] = {h ? ylm<8>(u) : u.z, h ? ylm<15>(u) : ylm<3>(u),
                              w1, __fmul_rn(w1, u.z), __fmul_rn(w1, u.z51), __fmul_rn(w1, u.z73),
                              w2, __fmul_rn(w2, u.z), __fmul_rn(w2, u.z71), w3,
                              __fmul_rn(w3, u.z), h ? ylm<23>(u) : ylm<22>(u)};
#pragma unroll
        for (int j = 0; j < 12; ++j)
#pragma unroll
          for (int n = 0; n <= NA; ++n) Sv[n][j] = __fmaf_rn(gn[n], bb[j], Sv[n][j]);
      };
      float go[NA + 1];
#pragma unroll
      for (int n = 0; n <= NA; ++n) go[n] = __shfl_xor_sync(kAll, g[n], 1);
      const UnitB uo = unit_b(__shfl_xor_sync(kAll, x, 1), __shfl_xor_sync(kAll, y, 1), __shfl_xor_sync(kAll, z, 1));
      add_pair(unit_b(x, y, z), g);
      add_pair(uo, go);
    }
#pragma unroll
    for (int n = 0; n <= NA; ++n) {
      float4 *r = row + n * 6;
      reinterpret_cast<float2 *>(r)[h] = make_float2(Sv[n][0], Sv[n][1]);
      r[1 + h] = make_float4(Sv[n][2], Sv[n][3], Sv[n][4], Sv[n][5]);
      r[3 + h] = make_float4(Sv[n][6], Sv[n][7], Sv[n][8], Sv[n][9]);
      reinterpret_cast<float2 *>(r + 5)[h] = make_float2(Sv[n][10], Sv[n][11]);
    }
  }
  sync_rows();
  // S_n of one n from the row, by polynomial index
  auto load_S = [&](int n, float *s) {
    static_for<0, 6>([&](auto qc) {
      constexpr int Q = decltype(qc)::value;
      const float4 v = row[n * 6 + Q];
      s[harm_k(4 * Q)] = v.x, s[harm_k(4 * Q + 1)] = v.y, s[harm_k(4 * Q + 2)] = v.z, s[harm_k(4 * Q + 3)] = v.w;
    });
  };

  // ---- angular descriptor components (Sec. II D) of n = h, h + 2, ...
#pragma unroll 1
  for (int n = h + 2 * sub; n <= NA; n += 2 * SUB) {
    float s[24];
    load_S(n, s);
    static_for<0, S::L3>([&](auto lc) {
      constexpr int l = decltype(lc)::value + 1;
      constexpr int k0 = l == 1 ? 0 : l == 2 ? 3 : l == 3 ? 8 : 15;
      constexpr int k1 = l == 1 ? 3 : l == 2 ? 8 : l == 3 ? 15 : 24;
      float acc = 0.f;
#pragma unroll
      for (int k = k0; k < k1; ++k) acc = __fmaf_rn(__fmul_rn(mf.c3b[k], s[k]), s[k], acc);
      qrow[(NR + 1) + (l - 1) * (NA + 1) + n] = acc;
    });
    if constexpr (S::L4 >= 2) {
      const float s3 = s[3], s4 = s[4], s5 = s[5], s6 = s[6], s7 = s[7];
      qrow[S::OFF4 + n] = mf.c4b[0] * s3 * s3 * s3 + mf.c4b[1] * s3 * (s4 * s4 + s5 * s5) +
                          mf.c4b[2] * s3 * (s6 * s6 + s7 * s7) + mf.c4b[3] * s6 * (s5 * s5 - s4 * s4) +
                          mf.c4b[4] * s4 * s5 * s7;
    }
    if constexpr (S::L5 >= 1) {
      const float s0 = s[0], s12 = s[1] * s[1] + s[2] * s[2];
      qrow[S::OFF5 + n] = mf.c5b[0] * s0 * s0 * s0 * s0 + mf.c5b[1] * s0 * s0 * s12 + mf.c5b[2] * s12 * s12;
    }
  }
  sync_rows();

  if constexpr (DESC) {
    if (active) {
      double *out = a.q_out + (a.perm ? (size_t)a.perm[i] : (size_t)i) * NDES;
      for (int v = h; v < NDES; v += 2) out[v] = (double)qrow[v];
    }
    return;
  }

  // ---- network, Eq. Ui, and dU/dq
  float U = 0.f;
  float dq[NR + 1];  // the radial part (the angular part is read from the row)
  if constexpr (TC) {
    // On the tensor cores (tcgen05, M = 128; the block's 64 atoms are rows 0 .. 63): GEMM1
    // z = q . W0^T, GEMM2 dq = beta . W0, every operand value as NT BF16 terms (hi, or hi + lo
    // with the products lo.hi + hi.lo + hi.hi in the same FP32 accumulator). A in TMEM (two K
    // values per column), W0 in shared memory (one tile per term for both GEMMs: GEMM2 reads it
    // MN-major). Every completion wait is bounded; if one runs out (all threads agree through
    // the barrier), the block flags the error, waits once more (again bounded) so that the MMAs
    // in flight finish before the TMEM is read or freed, and skips the rest of the network: its
    // results are then invalid and the host reports NEP_ERR_TIMEOUT.
    constexpr int KC1 = S::KP1 / 8, AC = PR::AC;
    static_assert(AB == 64, "rows 0 .. 63 of the 128-row MMA: two warps of 32 TMEM lanes each");
    const int warp = threadIdx.x >> 5;
    const bool mine = warp < 2;  // these two warps hold one row (atom) per thread
    const int r = mine ? threadIdx.x : 0;
    const uint32_t tm = tc_tmem + ((uint32_t)(warp * 32) << 16);
    float *const qr = reinterpret_cast<float *>(rows + r * PR::R4 + PR::S4);
    // NT BF16 terms of 8 values -> 4 columns each at A column c4
    auto put8 = [&](int c4, const float *x) {
      uint32_t u[NT][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float x0 = x[2 * j], x1 = x[2 * j + 1];
#pragma unroll
        for (int t = 0; t < NT; ++t) {
          const __nv_bfloat162 bh = __floats2bfloat162_rn(x0, x1);
          u[t][j] = *reinterpret_cast<const uint32_t *>(&bh);
          x0 -= __low2float(bh);
          x1 -= __high2float(bh);
        }
      }
#pragma unroll
      for (int t = 0; t < NT; ++t) tmem_st4u(tm + S::ACOL + t * AC + c4, u[t]);
    };
    // operands written by every thread -> visible to the MMA issued by thread 0
    auto to_mma = [&]() {
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    };
    auto gemm = [&](int ksteps, uint32_t bstep, uint32_t lbo, uint32_t sbo, uint32_t idesc) {
      uint32_t acc = 0u;
      auto terms = [&](int ta, int tb) {
        for (int st = 0; st < ksteps; ++st) {
          umma_bf16_ts(tc_tmem, tc_tmem + S::ACOL + ta * AC + 8 * st,
                       umma_desc(smem_addr(tiles) + tb * S::TILE_B + bstep * st, lbo, sbo), idesc, acc);
          acc = 1u;
        }
      };
      if constexpr (NT >= 2) {
        terms(1, 0);
        terms(0, 1);
      }
      terms(0, 0);
      umma_commit(&tc_mbar);
    };
    // wait for the commit of phase `parity`; false (block-uniform) if the wait ran out
    auto tc_wait = [&](uint32_t parity) -> bool {
      const bool ok = mbar_wait(&tc_mbar, parity);
      if (__syncthreads_or(!ok)) {
        if (threadIdx.x == 0) atomicOr(a.tc_err, 1);
        mbar_wait(&tc_mbar, parity);
        return false;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      return true;
    };
    __syncthreads();  // the rows of q are complete
    if (mine) {
#pragma unroll
      for (int c8 = 0; c8 < S::KP1 / 8; ++c8) {  // q row -> A
        float x[8];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const float4 v = 8 * c8 + 4 * j < NDP ? reinterpret_cast<const float4 *>(qr)[2 * c8 + j]
                                                : make_float4(0.f, 0.f, 0.f, 0.f);
          x[4 * j] = v.x, x[4 * j + 1] = v.y, x[4 * j + 2] = v.z, x[4 * j + 3] = v.w;
        }
        put8(4 * c8, x);
      }
    }
    to_mma();
    if (threadIdx.x == 0)  // GEMM1: z = q . W0^T into columns 0 .. NP1 - 1
      gemm(S::KP1 / 16, 256, 128, KC1 * 128, umma_idesc_bf16<128, S::NP1>());
    __syncwarp();
    if (tc_wait(0)) {
      // tanh layer from this row of z; beta = w1 (1 - h^2) -> A (the GEMM that read q has completed)
      if (mine) {
        float us = 0.f;
#pragma unroll
        for (int c8 = 0; c8 < S::NP1 / 8; ++c8) {
            float z[8], bt[8];
          tmem_ld8(tm + 8 * c8, z);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int mu = 8 * c8 + j;
            bt[j] = 0.f;
            if (mu < S::H) {
              const float t = tanhf(z[j] - b0_s[mu]);
              us = __fmaf_rn(w1_s[mu], t, us);
              bt[j] = w1_s[mu] * (1.f - t * t);
            }
          }
          put8(4 * c8, bt);
        }
        u_s[r] = us;
      }
      // every lane has read its z (tcgen05.ld waited) before GEMM2 overwrites the columns
      to_mma();
      if (threadIdx.x == 0)  // GEMM2: dq = beta . W0 into columns 0 .. NP2 - 1 (W0 MN-major)
        gemm(S::KP2 / 16, 2 * KC1 * 128, KC1 * 128, 128, umma_idesc_bf16_bmn<128, S::NP2>());
      __syncwarp();
      if (tc_wait(1) && mine) {
#pragma unroll
        for (int c8 = 0; c8 < (NDES + 7) / 8; ++c8) {
            float v[8];
          tmem_ld8(tm + 8 * c8, v);
          reinterpret_cast<float4 *>(qr)[2 * c8] = make_float4(v[0], v[1], v[2], v[3]);
          if (8 * c8 + 4 < NDP) reinterpret_cast<float4 *>(qr)[2 * c8 + 1] = make_float4(v[4], v[5], v[6], v[7]);
        }
      }
    }
    __syncthreads();
    U = u_s[ia] - w1_s[S::H];
#pragma unroll
    for (int v = 0; v <= NR; ++v) dq[v] = qrow[v];
  } else if constexpr (SUB > 1) {
    // As below, term by term: the groups share the neuron pairs of the forward sums, pass t = tanh
    // and beta on, and share the float4s of dU/dq, each adding all neurons in order.
    constexpr int V4 = NDP / 4, VJ = (V4 + 1) / 2;
    float2 *const tb = reinterpret_cast<float2 *>(rows + AB * PR::R4);  // [H][AB] (w1 t's t, beta)
    float4 q[VJ];
#pragma unroll
    for (int j = 0; j < VJ; ++j)
      q[j] = 2 * j + h < V4 ? reinterpret_cast<const float4 *>(qrow)[2 * j + h] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (int mu = 2 * sub; mu < S::H; mu += 2 * SUB) {
      const bool two = S::H % 2 == 0 || mu + 1 < S::H;
      const float4 *wr = reinterpret_cast<const float4 *>(w0_s + mu * NDP) + h;
      float za[2] = {0.f, 0.f}, zb[2] = {0.f, 0.f};
#pragma unroll
      for (int j = 0; j < VJ; ++j) {
        const bool in = V4 % 2 == 0 || 2 * j + h < V4;
        const float4 wa = in ? wr[2 * j] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 wb = in && two ? wr[V4 + 2 * j] : make_float4(0.f, 0.f, 0.f, 0.f);
        za[0] = __fmaf_rn(wa.x, q[j].x, za[0]);
        zb[0] = __fmaf_rn(wb.x, q[j].x, zb[0]);
        za[1] = __fmaf_rn(wa.y, q[j].y, za[1]);
        zb[1] = __fmaf_rn(wb.y, q[j].y, zb[1]);
        za[0] = __fmaf_rn(wa.z, q[j].z, za[0]);
        zb[0] = __fmaf_rn(wb.z, q[j].z, zb[0]);
        za[1] = __fmaf_rn(wa.w, q[j].w, za[1]);
        zb[1] = __fmaf_rn(wb.w, q[j].w, zb[1]);
      }
      const float pa = __fadd_rn(za[0], za[1]), pb = __fadd_rn(zb[0], zb[1]);
      const float zo = __shfl_xor_sync(kAll, h ? pa : pb, 1);
      const int my = two ? mu + h : mu;
      const float w1m = h == 0 || two ? w1_s[my] : 0.f;
      const float t = tanhf(__fadd_rn(h ? pb : pa, zo) - b0_s[my]);
      if (h == 0 || two) tb[my * AB + ia] = make_float2(t, w1m * (1.f - t * t));
    }
    __syncthreads();  // t and beta; every q is read
    if (sub == 0) {
#pragma unroll 2
      for (int mu = 0; mu < S::H; mu += 2) {
        const bool mine = h == 0 || S::H % 2 == 0 || mu + 1 < S::H;
        if (mine) U = __fmaf_rn(w1_s[mu + h], tb[(mu + h) * AB + ia].x, U);
      }
      U = __fadd_rn(U, __shfl_xor_sync(kAll, U, 1)) - w1_s[S::H];
    }
    constexpr int WJ = (VJ + SUB - 1) / SUB;  // this group's float4s: sub, sub + SUB, ...
    float4 dv[WJ];
#pragma unroll
    for (int w = 0; w < WJ; ++w) dv[w] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
    for (int mu = 0; mu < S::H; mu += 2) {
      const bool two = S::H % 2 == 0 || mu + 1 < S::H;
      const float ba = tb[mu * AB + ia].y, bb = two ? tb[(mu + 1) * AB + ia].y : 0.f;
      const float4 *wr = reinterpret_cast<const float4 *>(w0_s + mu * NDP) + h;
#pragma unroll
      for (int w = 0; w < WJ; ++w) {
        const int j = sub + w * SUB;
        const bool in = 2 * j + h < V4;
        const float4 wa = in ? wr[2 * j] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 wb = in && two ? wr[V4 + 2 * j] : make_float4(0.f, 0.f, 0.f, 0.f);
        dv[w].x = __fmaf_rn(bb, wb.x, __fmaf_rn(ba, wa.x, dv[w].x));
        dv[w].y = __fmaf_rn(bb, wb.y, __fmaf_rn(ba, wa.y, dv[w].y));
        dv[w].z = __fmaf_rn(bb, wb.z, __fmaf_rn(ba, wa.z, dv[w].z));
        dv[w].w = __fmaf_rn(bb, wb.w, __fmaf_rn(ba, wa.w, dv[w].w));
      }
    }
#pragma unroll
    for (int w = 0; w < WJ; ++w) {
      const int j = sub + w * SUB;
      if (2 * j + h < V4) reinterpret_cast<float4 *>(qrow)[2 * j + h] = dv[w];
    }
    __syncthreads();
#pragma unroll
    for (int v = 0; v <= NR; ++v) dq[v] = qrow[v];
  } else {
    // On the FMA pipes: each lane holds every second float4 of q and of dU/dq; two neurons at a
    // time, the lanes exchange their parts of z (lane h completes neuron mu + h), take one tanh
    // each and exchange beta.
    constexpr int V4 = NDP / 4, VJ = (V4 + 1) / 2;
    float4 q[VJ], dv[VJ];
#pragma unroll
    for (int j = 0; j < VJ; ++j) {
      q[j] = 2 * j + h < V4 ? reinterpret_cast<const float4 *>(qrow)[2 * j + h] : make_float4(0.f, 0.f, 0.f, 0.f);
      dv[j] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll 1
    for (int mu = 0; mu < S::H; mu += 2) {
      const bool two = S::H % 2 == 0 || mu + 1 < S::H;
      const float4 *wr = reinterpret_cast<const float4 *>(w0_s + mu * NDP) + h;
      float4 wa[VJ], wb[VJ];  // the rows serve both the forward and the backward sums
      float za[2] = {0.f, 0.f}, zb[2] = {0.f, 0.f};
#pragma unroll
      for (int j = 0; j < VJ; ++j) {
        const bool in = V4 % 2 == 0 || 2 * j + h < V4;
        wa[j] = in ? wr[2 * j] : make_float4(0.f, 0.f, 0.f, 0.f);
        wb[j] = in && two ? wr[V4 + 2 * j] : make_float4(0.f, 0.f, 0.f, 0.f);
        za[0] = __fmaf_rn(wa[j].x, q[j].x, za[0]);
        zb[0] = __fmaf_rn(wb[j].x, q[j].x, zb[0]);
        za[1] = __fmaf_rn(wa[j].y, q[j].y, za[1]);
        zb[1] = __fmaf_rn(wb[j].y, q[j].y, zb[1]);
        za[0] = __fmaf_rn(wa[j].z, q[j].z, za[0]);
        zb[0] = __fmaf_rn(wb[j].z, q[j].z, zb[0]);
        za[1] = __fmaf_rn(wa[j].w, q[j].w, za[1]);
        zb[1] = __fmaf_rn(wb[j].w, q[j].w, zb[1]);
      }
      const float pa = __fadd_rn(za[0], za[1]), pb = __fadd_rn(zb[0], zb[1]);
      const float zo = __shfl_xor_sync(kAll, h ? pa : pb, 1);  // the other lane's part of this lane's neuron
      const int my = two ? mu + h : mu;
      const float w1m = h == 0 || two ? w1_s[my] : 0.f;
      const float t = tanhf(__fadd_rn(h ? pb : pa, zo) - b0_s[my]);
      U = __fmaf_rn(w1m, t, U);
      const float beta = w1m * (1.f - t * t);
      const float bo = __shfl_xor_sync(kAll, beta, 1);
      const float ba = h ? bo : beta, bb = h ? beta : bo;
#pragma unroll
      for (int j = 0; j < VJ; ++j) {
        dv[j].x = __fmaf_rn(bb, wb[j].x, __fmaf_rn(ba, wa[j].x, dv[j].x));
        dv[j].y = __fmaf_rn(bb, wb[j].y, __fmaf_rn(ba, wa[j].y, dv[j].y));
        dv[j].z = __fmaf_rn(bb, wb[j].z, __fmaf_rn(ba, wa[j].z, dv[j].z));
        dv[j].w = __fmaf_rn(bb, wb[j].w, __fmaf_rn(ba, wa[j].w, dv[j].w));
      }
    }
    U = __fadd_rn(U, __shfl_xor_sync(kAll, U, 1)) - w1_s[S::H];
#pragma unroll
    for (int j = 0; j < VJ; ++j)
      if (2 * j + h < V4) reinterpret_cast<float4 *>(qrow)[2 * j + h] = dv[j];
    __syncwarp();
#pragma unroll
    for (int v = 0; v <= NR; ++v) dq[v] = qrow[v];
  }
  if (active && h == 0 && sub == 0 && a.energy) a.energy[mem * a.s_out + (a.perm ? a.perm[i] : i)] = (double)U;

  // ---- radial force coefficients e^t_k = sum_n dU/dq_n c^{t_i t}_{nk} and their sum: every second
  // group of four k
  for (int t = SUB - 1 - sub; t < T; t += SUB) {  // (the last group first: it has the fewest n below)
    const float4 *c = reinterpret_cast<const float4 *>(cR_s + (ti * T + t) * (NR + 1) * KRP);
    constexpr int E4 = S::EF4, EJ = (E4 + 1) / 2;
    float ev[EJ][4], tot = 0.f;
#pragma unroll
    for (int j = 0; j < EJ; ++j) {
      const int k4 = 2 * j + h;
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
      if (k4 < KRP / 4) {
#pragma unroll
        for (int n = 0; n <= NR; ++n) {
          const float4 cv = c[n * (KRP / 4) + k4];
          acc[0] = __fmaf_rn(dq[n], cv.x, acc[0]);
          acc[1] = __fmaf_rn(dq[n], cv.y, acc[1]);
          acc[2] = __fmaf_rn(dq[n], cv.z, acc[2]);
          acc[3] = __fmaf_rn(dq[n], cv.w, acc[3]);
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        ev[j][k] = acc[k];
        tot = __fadd_rn(tot, acc[k]);  // c^R rows are zero past KR
      }
    }
    tot = __fadd_rn(tot, __shfl_xor_sync(kAll, tot, 1));
    if (active) {
      float4 *er = reinterpret_cast<float4 *>(a.e_rad + mem * a.s_erad);
#pragma unroll
      for (int j = 0; j < EJ; ++j) {
        const int k4 = 2 * j + h;
        if (k4 >= E4) continue;
        if (k4 == (KR + 1) / 4) ev[j][(KR + 1) % 4] = tot;
        er[((size_t)t * E4 + k4) * N + i] = make_float4(ev[j][0], ev[j][1], ev[j][2], ev[j][3]);
      }
    }
  }
  __syncwarp();

  // ---- dU/dS_nk from the explicit 3/4/5-body forms, in place of S_nk: n = h, h + 2, ...
#pragma unroll 1
  for (int n = h + 2 * sub; n <= NA; n += 2 * SUB) {
    float s[24], dS[24];
    load_S(n, s);
    static_for<0, 24>([&](auto kc) {
      constexpr int k = decltype(kc)::value;
      if constexpr (k < S::KEND3) dS[k] = 2.f * mf.c3b[k] * s[k] * qrow[(NR + 1) + (l_of_k(k) - 1) * (NA + 1) + n];
      else dS[k] = 0.f;
    });
    if constexpr (S::L4 >= 2) {
      const float d4 = qrow[S::OFF4 + n];
      const float *C = mf.c4b;
      dS[3] += d4 * (3.f * C[0] * s[3] * s[3] + C[1] * (s[4] * s[4] + s[5] * s[5]) + C[2] * (s[6] * s[6] + s[7] * s[7]));
      dS[4] += d4 * (2.f * C[1] * s[3] * s[4] - 2.f * C[3] * s[6] * s[4] + C[4] * s[5] * s[7]);
      dS[5] += d4 * (2.f * C[1] * s[3] * s[5] + 2.f * C[3] * s[6] * s[5] + C[4] * s[4] * s[7]);
      dS[6] += d4 * (2.f * C[2] * s[3] * s[6] + C[3] * (s[5] * s[5] - s[4] * s[4]));
      dS[7] += d4 * (2.f * C[2] * s[3] * s[7] + C[4] * s[4] * s[5]);
    }
    if constexpr (S::L5 >= 1) {
      const float d5 = qrow[S::OFF5 + n];
      const float *C = mf.c5b;
      const float s12 = s[1] * s[1] + s[2] * s[2];
      dS[0] += d5 * (4.f * C[0] * s[0] * s[0] * s[0] + 2.f * C[1] * s[0] * s12);
      const float common = 2.f * C[1] * s[0] * s[0] + 4.f * C[2] * s12;
      dS[1] += d5 * common * s[1];
      dS[2] += d5 * common * s[2];
    }
    static_for<0, 6>([&](auto qc) {
      constexpr int Q = decltype(qc)::value;
      row[n * 6 + Q] = make_float4(dS[harm_k(4 * Q)], dS[harm_k(4 * Q + 1)], dS[harm_k(4 * Q + 2)], dS[harm_k(4 * Q + 3)]);
    });
  }
  sync_rows();

  // ---- angular partial forces dU_i/dr_ij (angular terms of Eq. partial_force): with
  // a_k = sum_n dU/dS_nk g_n and c_k = sum_n dU/dS_nk g_n',
  //   dU_i/dr_ij = (G - (G.u) u) / r + Y u,  G = sum_k a_k grad b_k(u),  Y = sum_k c_k b_k(u)
  if (4 * sub + 2 * h < na) {
    constexpr int PP = 2, STEP = 4 * SUB;
    const int first = 4 * sub + 2 * h;
    const unsigned *col = a.nl_a + i;
    unsigned ec[PP], en[PP];
    float4 pc[PP];
#pragma unroll
    for (int p = 0; p < PP; ++p) {
      const int m = first + p;
      ec[p] = m < na ? __ldg(col + (size_t)m * N) : 0u;
      en[p] = m + STEP < na ? __ldg(col + (size_t)(m + STEP) * N) : 0u;
    }
#pragma unroll
    for (int p = 0; p < PP; ++p) pc[p] = __ldg(a.pos4 + (ec[p] & a.jmask));
#pragma unroll 1
    for (int m0 = first; m0 < na; m0 += STEP) {
      float3 d[PP];
      float r2[PP];
      bool in[PP], any = false;
      int tj[PP];
#pragma unroll
      for (int p = 0; p < PP; ++p) {
        d[p] = pair_vector(pi, pc[p], shift(ec[p]));
        tj[p] = type_of(pc[p]);
        r2[p] = norm2(d[p]);
        in[p] = m0 + p < na && r2[p] < rcA2;
        any = any || in[p];
        ec[p] = en[p];
        if (m0 + STEP < na) pc[p] = __ldg(a.pos4 + (en[p] & a.jmask));
        en[p] = m0 + 2 * STEP + p < na ? __ldg(col + (size_t)(m0 + 2 * STEP + p) * N) : 0u;
      }
      if (!any) continue;
      float rinv[PP], g[PP][NA + 1], gp[PP][NA + 1];
      float gx[PP], gy[PP], gz[PP], Y[PP];
      UnitB u[PP];
#pragma unroll
      for (int p = 0; p < PP; ++p) {
        rinv[p] = rsqrtf(r2[p]);
        float f[KA + 1], fp[KA + 1];
        cheb_basis_d<KA>(r2[p] * rinv[p], inv_rcA, f, fp);
        const float4 *c4 = reinterpret_cast<const float4 *>(cA_s + (ti * T + tj[p]) * CAP);
#pragma unroll
        for (int n = 0; n <= NA; ++n) g[p][n] = gp[p][n] = 0.f;
#pragma unroll
        for (int v = 0; v < CAP / 4; ++v) {
          const float4 cv = c4[v];
          const float cw[4] = {cv.x, cv.y, cv.z, cv.w};
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (4 * v + j < (NA + 1) * (KA + 1)) {
              const int n = (4 * v + j) / (KA + 1), k = (4 * v + j) % (KA + 1);
              g[p][n] = __fmaf_rn(cw[j], f[k], g[p][n]);
              gp[p][n] = __fmaf_rn(cw[j], fp[k], gp[p][n]);
            }
        }
        u[p] = unit_b(__fmul_rn(d[p].x, rinv[p]), __fmul_rn(d[p].y, rinv[p]), __fmul_rn(d[p].z, rinv[p]));
        gx[p] = gy[p] = gz[p] = Y[p] = 0.f;
      }
      static_for<0, 6>([&](auto qc) {
        constexpr int Q = decltype(qc)::value;
        float ak[PP][4], ck[PP][4];
#pragma unroll
        for (int n = 0; n <= NA; ++n) {
          const float4 v = row[n * 6 + Q];
          const float dv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int p = 0; p < PP; ++p)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              ak[p][j] = n == 0 ? __fmul_rn(dv[j], g[p][n]) : __fmaf_rn(dv[j], g[p][n], ak[p][j]);
              ck[p][j] = n == 0 ? __fmul_rn(dv[j], gp[p][n]) : __fmaf_rn(dv[j], gp[p][n], ck[p][j]);
            }
        }
#pragma unroll
        for (int p = 0; p < PP; ++p) harm_fold<Q>(u[p], ak[p], ck[p], gx[p], gy[p], gz[p], Y[p]);
      });
#pragma unroll
      for (int p = 0; p < PP; ++p) {
        const float gu = __fmaf_rn(gz[p], u[p].z, __fmaf_rn(gy[p], u[p].y, __fmul_rn(gx[p], u[p].x)));
        const float t = __fmaf_rn(-gu, rinv[p], Y[p]);  // P = G / r + (Y - (G.u) / r) u
        if (in[p])
          a.p_ang[mem * a.s_pang + (size_t)(m0 + p) * N + i] =
              make_float4(__fmaf_rn(gx[p], rinv[p], __fmul_rn(t, u[p].x)), __fmaf_rn(gy[p], rinv[p], __fmul_rn(t, u[p].y)),
                          __fmaf_rn(gz[p], rinv[p], __fmul_rn(t, u[p].z)), 0.f);
      }
    }
  }
  if constexpr (!BATCH) {
    // deterministic block sum of U where it is read (a batch sums its structures from the
    // per-atom energies)
    // (up to kSplitAtoms2 atoms a slot per warp's 16 atoms, so that all forms agree on atom_blocks)
    static_assert(AB == 64 || SUB > 1, "slots of 64 or of 16 atoms");
    if (sums_needed(a) & kSumU) {
      __shared__ double red[2 * AB / 32];
      const int warp = threadIdx.x >> 5;
      if (sub == 0) {
        double su = active && h == 0 ? (double)U : 0.0;
#pragma unroll
        for (int o = 16; o > 1; o >>= 1) su += __shfl_xor_sync(kAll, su, o);  // lanes of one parity
        if ((threadIdx.x & 31) == 0) {
          if (N > kSplitAtoms2) red[warp] = su;
          else if (blockIdx.x * (AB / 16) + warp < (N + 15) / 16)
            a.partial_atom[blockIdx.x * (AB / 16) + warp] = su;
        }
      }
      if (N > kSplitAtoms2) {
        __syncthreads();
        if (threadIdx.x == 0) {
          double t = 0.0;
          for (int wv = 0; wv < 2 * AB / 32; ++wv) t += red[wv];
          a.partial_atom[blockIdx.x] = t;
        }
      }
    }
  }
  if constexpr (TC) {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x < 32) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tc_tmem), "r"((uint32_t)PR::COLS));
    }
  }
}

template <class S>
size_t atom_pair_smem(int T, int ncode, int prec, int ab) {
  return sizeof(float4) * ncode + sizeof(float) * (size_t)PairRow<S>::off_rows(prec, T) +
         sizeof(float4) * PairRow<S>::R4 * ab;
}

// Epilogue of the gather kernels for atom i: outputs in the caller's order, the squared force
// error of Eq. loss, the second velocity-Verlet half-kick with the kinetic energy, and the
// heat current J_i = W_i . v_i (Eq. Ji); part[] collects KE, the force error and J for the block
// sums (need: the sums formed; the others are skipped).
__device__ __forceinline__ void gather_epilogue(const AtomArgs &a, int i, const float4 &pi, int mem, const float *fw,
                                                int need, double *part) {
  const double Fx = fw[0], Fy = fw[1], Fz = fw[2];
  const float *w = fw + 3;
  const int ti = type_of(pi);
  const size_t iu = a.perm ? (size_t)a.perm[i] : (size_t)i, io = mem * a.s_out + iu;
  if (a.force) {
    a.force[3 * io] = Fx;
    a.force[3 * io + 1] = Fy;
    a.force[3 * io + 2] = Fz;
  }
  if (a.virial) {
#pragma unroll
    for (int c = 0; c < 9; ++c) a.virial[9 * io + c] = (double)w[c];
  }
  if (need & kSumFerr) {  // squared force error against target forces (the force term of Eq. loss)
    const double *ft = a.f_tar + 3 * iu;
    const double ex = Fx - ft[0], ey = Fy - ft[1], ez = Fz - ft[2];
    part[1] = ex * ex + ey * ey + ez * ez;
  }
  bool kick = a.md_kick && !(a.fire && a.fire->converged);
  double hdt = a.fire ? 0.5 * a.fire->dt : a.half_dt;
  if (a.slots) {  // batched engine: the structure's own phase and time step
    const EngineSlot &sl = a.slots[struct_of(pi)];
    kick = sl.phase == 1 && !(sl.kind == kJobFire && sl.fire.converged);
    hdt = 0.5 * (sl.kind == kJobFire ? sl.fire.dt : sl.dt);
  }
  const bool moments = (need & (kSumKE | kSumJ)) || a.heat;
  // velocity of the kinetic energy and the heat current: after the kick (MD), or given by the caller
  double vh[3] = {0.0, 0.0, 0.0};
  if (kick) {  // second half-kick of velocity Verlet
    double *v = a.vel + 3 * (size_t)i;
    const double s = hdt * a.inv_mass_kappa[ti];
    vh[0] = v[0] + s * Fx, vh[1] = v[1] + s * Fy, vh[2] = v[2] + s * Fz;
    v[0] = vh[0], v[1] = vh[1], v[2] = vh[2];
  } else if (moments && (a.md_kick || a.slots || a.vel_in)) {  // converged FIRE or no step: velocities unchanged
    const double *v = a.vel_in ? a.vel_in + 3 * iu : a.vel + 3 * (size_t)i;
    vh[0] = v[0], vh[1] = v[1], vh[2] = v[2];
  }
  if (!moments) return;
  if (need & kSumKE) part[0] = a.mass_kappa_half[ti] * (vh[0] * vh[0] + vh[1] * vh[1] + vh[2] * vh[2]);
  if ((need & kSumJ) || a.heat) {
    // J_i = W_i . v_i, W_i[a][b] in the order xx, yy, zz, xy, xz, yz, yx, zx, zy (Eq. Ji)
    part[2] = (double)w[0] * vh[0] + (double)w[3] * vh[1] + (double)w[4] * vh[2];
    part[3] = (double)w[6] * vh[0] + (double)w[1] * vh[1] + (double)w[5] * vh[2];
    part[4] = (double)w[7] * vh[0] + (double)w[8] * vh[1] + (double)w[2] * vh[2];
    if (a.heat) {
      a.heat[3 * io] = part[2];
      a.heat[3 * io + 1] = part[3];
      a.heat[3 * io + 2] = part[4];
    }
  }
}

// End of a gather kernel: fw[GA][13] holds F_i and W_i (12 floats) of the block's GA atoms, zeros
// for the inactive ones (`on` marks the others). One thread per atom runs the epilogue, then
// the block forms the sums that are read, in FP64 and a fixed order. Without the test every MD step
// of every atom paid 15 FP64 block sums for totals that only thermo rows show (half of the
// gather's time). A row shows the virial's diagonal alone: 20 steps of 100,000 PbTe atoms with a row
// each 4181 us with all nine components, 4083 with three.
template <int GA, int NT>
__device__ __forceinline__ void gather_finish(const AtomArgs &a, int mem, float (*fw)[13], const unsigned char *on) {
  static_assert(GA % 32 == 0 && NT >= GA && NT >= 96, "whole warps of atoms; 72 threads for the virial sums");
  __shared__ double red[GA / 32][5];
  const int need = sums_needed(a);
  double part[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  __syncthreads();
  if (threadIdx.x < GA && on[threadIdx.x]) {
    const int i = blockIdx.x * GA + threadIdx.x;
    gather_epilogue(a, i, a.pos4[i], mem, fw[threadIdx.x], need, part);
  }
  if (!(need & (kSumKE | kSumW | kSumP | kSumFerr | kSumJ))) return;
  double *out = a.partial_gather + ((size_t)mem * gridDim.x + blockIdx.x) * kReduceSlots;
  // eight threads per component: nine in 96 threads (whole warps), the diagonal in 32
  const int nw = (need & kSumW) ? 9 : (need & kSumP) ? 3 : 0;
  if (threadIdx.x < 32 * ((nw + 3) / 4)) {
    const int c = threadIdx.x >> 3, p = threadIdx.x & 7;
    double s = 0.0;
    if (c < nw)
      for (int r = p; r < GA; r += 8) s += (double)fw[r][3 + c];
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (c < nw && p == 0) out[2 + c] = s;
  }
  if (!(need & (kSumKE | kSumFerr | kSumJ))) return;
  if (threadIdx.x < GA) {
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      if (!(need & (k == 0 ? kSumKE : k == 1 ? kSumFerr : kSumJ))) continue;
      double v = part[k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
      if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][k] = v;
    }
  }
  __syncthreads();
  if (threadIdx.x < 5 && (need & (threadIdx.x == 0 ? kSumKE : threadIdx.x == 1 ? kSumFerr : kSumJ))) {
    double s = 0.0;
    for (int wv = 0; wv < GA / 32; ++wv) s += red[wv][threadIdx.x];
    out[threadIdx.x == 0 ? 1 : 10 + threadIdx.x] = s;  // KE 1, force error 11, J 12 .. 14
  }
}

// ------------------------------------------------------------------------ gather kernel
// kGatherLanes lanes per atom take every kGatherLanes-th entry of its lists; their sums are
// added across, and one thread per atom finishes (gather_finish).
//
// What bounds it: the L1 data stage (84% busy): the neighbours' e_k, positions and partial
// forces are 16-byte reads at 32 scattered addresses, about 10 passes each. The e_k lie in
// planes of float4 over the atoms and the image shifts component by component in shared memory,
// which took a fifth of the passes out. For one structure the kernel is held to 64 registers
// for N_bas^R <= 8 (1024 threads per SM hide more of the latency than 896: 8,000,000 Si atoms
// 2.47 against 2.73 ms) and to 72 above. Two lanes halve the serial chain of small systems; four
// shorten it further (216 atoms: 13.8 us) but cost large ones more than they give
// (8,000,000 atoms: 2.98 ms). Before / after (one thread per atom, all block sums in every
// launch), us: 216 Si atoms 32 / 18, 262,144 PbTe atoms 121 / 100, 8,000,000 Si atoms 2846 /
// 2472, 4096 structures 681 / 550. Up to kSplitGather2 atoms SUB groups of lanes work out an atom's
// pairs side by side, and the pair sums are added in the order of the plain form (the same bits).
constexpr int kGatherLanes = 2;
constexpr int gather_min_blocks(int KR, int threads) {
  return (KR <= 8 ? 1024 : 896) / threads > 0 ? (KR <= 8 ? 1024 : 896) / threads : 1;
}

template <class S, bool BATCH, int GA, int SUB>
__global__ void __launch_bounds__(GA *kGatherLanes *SUB, SUB > 1 ? 2 : gather_min_blocks(S::KR, GA *kGatherLanes))
    gather_kernel(const AtomArgs a) {
  const bool failed = build_failed(a.guard);  // tested once the first loads are under way
  constexpr int L = kGatherLanes;
  __shared__ float fw[GA][13];
  __shared__ unsigned char on[GA];
  constexpr int KR = S::KR;
  extern __shared__ float4 smem4[];
  float4 *dtab_s = smem4;
  const int mem = BATCH ? (int)blockIdx.y : 0;
  if constexpr (!BATCH) {
    stage_shifts(a, reinterpret_cast<float *>(dtab_s));
    __syncthreads();
  }
  const float *e_rad = a.e_rad + mem * a.s_erad;
  const float4 *p_ang = a.p_ang + mem * a.s_pang;
  const int N = a.N, T = a.T;
  const int ia = threadIdx.x / (L * SUB), l = threadIdx.x % L, sub = threadIdx.x % (L * SUB) / L;
  const int i = blockIdx.x * GA + ia;
  float fx = 0.f, fy = 0.f, fz = 0.f;
  float w[9];
#pragma unroll
  for (int c = 0; c < 9; ++c) w[c] = 0.f;
  // (serving engine) atoms of a finished job frozen in the batch are skipped
  const bool active = i < N && !(BATCH && a.slots && (failed || a.slots[struct_of(a.pos4[i])].phase == 2));
  if (active || SUB > 1) {  // (the lanes of a split atom exchange their pairs: whole warps)
    const float4 pi = a.pos4[active ? i : 0];
    const int ti = type_of(pi);
    const float4 *dtab_b = BATCH ? a.dtab + (size_t)struct_of(pi) * a.ncode : dtab_s;
    auto shift = [&](unsigned e) -> float4 {
      if constexpr (BATCH) return __ldg(dtab_b + (e >> a.jbits));
      else return shift_at(reinterpret_cast<const float *>(dtab_s), a.ncode, e >> a.jbits);
    };
    const float inv_rcR = 1.f / a.rcR;
    const float rcR2 = a.rcR * a.rcR, rcA2 = a.rcA * a.rcA;
    // e_k of atom j and type t and (entry KR + 1) their sum
    auto load_e = [&](float *e, int t, int j) {
#pragma unroll
      for (int k4 = 0; k4 < S::EF4; ++k4) {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(e_rad) + ((size_t)t * S::EF4 + k4) * N + j);
        e[4 * k4] = v.x, e[4 * k4 + 1] = v.y, e[4 * k4 + 2] = v.z, e[4 * k4 + 3] = v.w;
      }
    };
    // s_i and s_j of a pair at distance r from the atom's own and the neighbour's coefficients
    auto radial_terms = [&](const float *eo, const float *ej, float r, float &si, float &sj) {
      // sum_k e_k f_k'(r) = (x' fc/2) sum_k e_k T_k'(x) + (fc'/2) (sum_k e_k T_k(x) + sum_k e_k)
      const float u = r * inv_rcR;
      float sn, cs;
      __sincosf(3.14159265358979f * u, &sn, &cs);
      const float hfc = 0.25f * (1.f + cs);
      const float hfcp = -0.25f * 3.14159265358979f * inv_rcR * sn;
      const float t1 = u - 1.f;
      const float x = 2.f * t1 * t1 - 1.f;
      const float xp = 4.f * t1 * inv_rcR;
      const float x2 = 2.f * x;
      float tkm1 = 1.f, tk = x, dkm1 = 0.f, dk = 1.f;
      float oT = eo[0], oD = 0.f, jT = ej[0], jD = 0.f;
      if (KR >= 1) {
        oT = __fmaf_rn(eo[1], x, oT);
        jT = __fmaf_rn(ej[1], x, jT);
        oD = eo[1];
        jD = ej[1];
      }
#pragma unroll
      for (int k = 2; k <= KR; ++k) {
        const float tn = __fmaf_rn(x2, tk, -tkm1);
        const float dn = __fmaf_rn(x2, dk, __fmaf_rn(2.f, tk, -dkm1));
        tkm1 = tk; tk = tn; dkm1 = dk; dk = dn;
        oT = __fmaf_rn(eo[k], tn, oT);
        jT = __fmaf_rn(ej[k], tn, jT);
        oD = __fmaf_rn(eo[k], dn, oD);
        jD = __fmaf_rn(ej[k], dn, jD);
      }
      const float a1 = xp * hfc;
      si = __fmaf_rn(a1, oD, hfcp * (oT + eo[KR + 1]));
      sj = __fmaf_rn(a1, jD, hfcp * (jT + ej[KR + 1]));
    };
    auto add_radial = [&](const float3 &d, float fs, float ws) {
      fx = __fmaf_rn(fs, d.x, fx);
      fy = __fmaf_rn(fs, d.y, fy);
      fz = __fmaf_rn(fs, d.z, fz);
      // W_i += r_ij (x) dU_j/dr_ji with dU_j/dr_ji = -s_j d / r
      const float px = ws * d.x, py = ws * d.y, pz = ws * d.z;
      w[0] = __fmaf_rn(d.x, px, w[0]);
      w[1] = __fmaf_rn(d.y, py, w[1]);
      w[2] = __fmaf_rn(d.z, pz, w[2]);
      w[3] = __fmaf_rn(d.x, py, w[3]);
      w[4] = __fmaf_rn(d.x, pz, w[4]);
      w[5] = __fmaf_rn(d.y, pz, w[5]);
      w[6] = __fmaf_rn(d.y, px, w[6]);
      w[7] = __fmaf_rn(d.z, px, w[7]);
      w[8] = __fmaf_rn(d.z, py, w[8]);
    };
    auto add_angular = [&](const float3 &d, const float3 &df, const float3 &p) {
      fx += df.x;
      fy += df.y;
      fz += df.z;
      w[0] = __fmaf_rn(d.x, p.x, w[0]);
      w[1] = __fmaf_rn(d.y, p.y, w[1]);
      w[2] = __fmaf_rn(d.z, p.z, w[2]);
      w[3] = __fmaf_rn(d.x, p.y, w[3]);
      w[4] = __fmaf_rn(d.x, p.z, w[4]);
      w[5] = __fmaf_rn(d.y, p.z, w[5]);
      w[6] = __fmaf_rn(d.y, p.x, w[6]);
      w[7] = __fmaf_rn(d.z, p.x, w[7]);
      w[8] = __fmaf_rn(d.z, p.y, w[8]);
    };
    if constexpr (SUB > 1) {
      // Lane (l, sub) works out the pairs l + 2 (sub + SUB r) of its list; then every lane of parity l
      // adds the SUB pairs of the round in list order, as the one lane of the form below does.
      constexpr unsigned kAll = 0xffffffffu;
      const int lane = threadIdx.x & 31, first = (lane & ~(L * SUB - 1)) | l;
      int base = 0;
      for (int t = 0; t < T; ++t) {
        const int cnt = active ? a.nn_r[(size_t)t * N + i] : 0;
        const int nl = (cnt + L - 1 - l) / L;
        float eo[4 * S::EF4];
        load_e(eo, t, active ? i : 0);
        if (failed) return;
        const unsigned *col = a.nl_r + (size_t)(base + l) * N + i;
        const int rounds = __reduce_max_sync(kAll, (nl + SUB - 1) / SUB);
        unsigned e1 = sub < nl ? __ldg(col + (size_t)L * sub * N) : 0u;
#pragma unroll 1
        for (int r = 0; r < rounds; ++r) {
          const int q = SUB * r + sub;
          const unsigned e = e1;
          e1 = q + SUB < nl ? __ldg(col + (size_t)L * (q + SUB) * N) : 0u;
          const int j = e & a.jmask;
          const float3 d = pair_vector(pi, __ldg(a.pos4 + j), shift(e));
          const float r2 = norm2(d);
          const bool in = q < nl && r2 < rcR2;
          float fs = 0.f, ws = 0.f;
          if (in) {
            const float rinv = rsqrtf(r2);
            float ej[4 * S::EF4], si, sj;
            load_e(ej, ti, j);
            radial_terms(eo, ej, r2 * rinv, si, sj);
            fs = (si + sj) * rinv;
            ws = -sj * rinv;
          }
          const unsigned mask = __ballot_sync(kAll, in);
#pragma unroll
          for (int s = 0; s < SUB; ++s) {
            const int src = first + L * s;
            const float3 ds = make_float3(__shfl_sync(kAll, d.x, src), __shfl_sync(kAll, d.y, src),
                                          __shfl_sync(kAll, d.z, src));
            const float f1 = __shfl_sync(kAll, fs, src), w1 = __shfl_sync(kAll, ws, src);
            if ((mask >> src) & 1u) add_radial(ds, f1, w1);
          }
        }
        base += cnt;
      }
      const int na = active ? a.nn_a[i] : 0, nl = (na + L - 1 - l) / L;
      const int rounds = __reduce_max_sync(kAll, (nl + SUB - 1) / SUB);
#pragma unroll 1
      for (int r = 0; r < rounds; ++r) {
        const int q = SUB * r + sub;
        float3 d = make_float3(0.f, 0.f, 0.f), df = d, p = d;
        bool in = false;
        if (q < nl) {
          const size_t slot = (size_t)(L * q + l) * N + i;
          const unsigned e = __ldg(a.nl_a + slot);
          const float4 pij = p_ang[slot], pji = __ldg(p_ang + __ldg(a.rev_a + slot));
          d = pair_vector(pi, __ldg(a.pos4 + (e & a.jmask)), shift(e));
          in = norm2(d) < rcA2;
          df = make_float3(pij.x - pji.x, pij.y - pji.y, pij.z - pji.z);
          p = make_float3(pji.x, pji.y, pji.z);
        }
        const unsigned mask = __ballot_sync(kAll, in);
#pragma unroll
        for (int s = 0; s < SUB; ++s) {
          const int src = first + L * s;
          float v[9] = {d.x, d.y, d.z, df.x, df.y, df.z, p.x, p.y, p.z};
#pragma unroll
          for (int c = 0; c < 9; ++c) v[c] = __shfl_sync(kAll, v[c], src);
          if ((mask >> src) & 1u)
            add_angular(make_float3(v[0], v[1], v[2]), make_float3(v[3], v[4], v[5]), make_float3(v[6], v[7], v[8]));
        }
      }
    } else {
    // ---- radial part (Algorithm 2): s_i from own e^{t_j}, s_j from neighbour's e^{t_i}
    int base = 0;
    for (int t = 0; t < T; ++t) {
      const int cnt = a.nn_r[t * N + i];
      float eo[4 * S::EF4];
      load_e(eo, t, i);
      if (failed) return;
      for_pairs_batch<2, true, 1>(a.nl_r + (size_t)(base + l) * N, 0, (cnt + L - 1 - l) / L, L * N, i, a.pos4, a.jmask, [&](int, unsigned e, const float4 &pj) {
        const int j = e & a.jmask;
        const float3 d = pair_vector(pi, pj, shift(e));
        const float r2 = norm2(d);
        if (r2 < rcR2) {
          const float rinv = rsqrtf(r2);
          const float r = r2 * rinv;
          float ej[4 * S::EF4];
          load_e(ej, ti, j);
          float si, sj;
          radial_terms(eo, ej, r, si, sj);
          add_radial(d, (si + sj) * rinv, -sj * rinv);
        }
      });
      base += cnt;
    }
    // ---- angular part (Algorithm 4): F_i += P_ij - P_ji, W_i += r_ij (x) P_ji
    // Software-pipelined: list entry and reverse slot two entries ahead, the neighbour's
    // position and both partial forces one entry ahead (every reverse slot is a valid slot,
    // and a slot's partial force is used only when the pair is inside the cutoff, which is
    // exactly when the per-atom kernel wrote it).
    const int na = a.nn_a[i];
    if (l < na) {
      const unsigned *col = a.nl_a + i;
      const int *rcol = a.rev_a + i;
      auto at = [&](int m) { return (size_t)m * N; };
      unsigned e0 = __ldcs(col + at(l)), e1 = l + L < na ? __ldcs(col + at(l + L)) : 0u;
      int r1 = l + L < na ? __ldcs(rcol + at(l + L)) : 0;
      float4 p0 = __ldg(a.pos4 + (e0 & a.jmask));
      float4 pij0 = __ldcs(p_ang + at(l) + i), pji0 = __ldg(p_ang + __ldcs(rcol + at(l)));
      for (int m = l; m < na; m += L) {
        const unsigned e = e0;
        const float4 pj = p0, pij = pij0, pji = pji0;
        if (m + L < na) {
          p0 = __ldg(a.pos4 + (e1 & a.jmask));
          pij0 = __ldcs(p_ang + at(m + L) + i);
          pji0 = __ldg(p_ang + r1);
        }
        e0 = e1;
        if (m + 2 * L < na) {
          e1 = __ldcs(col + at(m + 2 * L));
          r1 = __ldcs(rcol + at(m + 2 * L));
        }
        const float3 d = pair_vector(pi, pj, shift(e));
        const float r2 = norm2(d);
        if (r2 < rcA2) {
          add_angular(d, make_float3(pij.x - pji.x, pij.y - pji.y, pij.z - pji.z), make_float3(pji.x, pji.y, pji.z));
        }
      }
    }
    }
  }
  if (failed) return;  // the threads without an atom too
  // the sums of the atom's lanes; one row per atom for the epilogue
  float v[12] = {fx, fy, fz, w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7], w[8]};
#pragma unroll
  for (int c = 0; c < 12; ++c) {
#pragma unroll
    for (int o = 1; o < L; o <<= 1) v[c] = __fadd_rn(v[c], __shfl_xor_sync(0xffffffffu, v[c], o));
    if (l == 0 && sub == 0) fw[ia][c] = v[c];
  }
  if (l == 0 && sub == 0) on[ia] = active ? 1 : 0;
  gather_finish<GA, GA * L * SUB>(a, mem, fw, on);
}

// ------------------------------------------------------------------------ launchers
// block sums of U of one structure: a slot per 16 atoms up to kSplitAtoms2, above a slot per 64 atoms, an even
// number of them
template <class S> int atom_blocks(int N) { return N <= kSplitAtoms2 ? (N + 15) / 16 : 2 * ((N + 127) / 128); }

template <class S, int PREC, bool DESC, bool BATCH, int AB, int SUB = 1>
cudaError_t launch_atom_as(const AtomArgs &a, const ModelF &mf, int members, cudaStream_t st) {
  auto kern = atom_kernel<S, PREC, DESC, BATCH, AB, SUB>;
  constexpr size_t tb = SUB > 1 ? sizeof(float2) * S::H * AB : 0;
  const cudaError_t e = smem_limit_once(kern, tb + atom_pair_smem<S>(kMaxTypes, BATCH ? 0 : 1 << 9, PREC, AB));
  if (e != cudaSuccess) return e;
  const int blocks = (!BATCH && AB == 64) ? 2 * ((a.N + 127) / 128) : (a.N + AB - 1) / AB;
  kern<<<dim3(blocks, members), 2 * AB * SUB, tb + atom_pair_smem<S>(a.T, BATCH ? 0 : a.ncode, PREC, AB), st>>>(a, mf);
  return cudaGetLastError();
}

template <class S>
cudaError_t launch_atom(const AtomArgs &a, const ModelF &mf, int descriptor_only, cudaStream_t st) {
  if (a.N <= 0) return cudaSuccess;
  if (descriptor_only) return launch_atom_as<S, 0, true, false, 64>(a, mf, 1, st);
  if (a.precision == 1) return launch_atom_as<S, 1, false, false, 64>(a, mf, 1, st);
  if (a.precision == 2) return launch_atom_as<S, 2, false, false, 64>(a, mf, 1, st);
  if (a.N <= kSplitAtoms) return launch_atom_as<S, 0, false, false, 16, 4>(a, mf, 1, st);
  if (a.N <= kSplitAtoms2) return launch_atom_as<S, 0, false, false, 32, 2>(a, mf, 1, st);
  return launch_atom_as<S, 0, false, false, 64>(a, mf, 1, st);
}

constexpr int kGatherAtoms = 64;  // atoms per CTA of the gather of one structure
// Small systems: four groups of lanes per atom (half as many atoms per CTA), then two, up to one wave
// of two CTAs per SM. A dynamics step with one / four / two groups, us: 1,000 Si atoms 43 / 36 / -,
// 8,000 53 / 46 / -, 13,824 60.4 / 62.8 / 57.4, 13,824 PbTe atoms 54.0 / 53.7 / 48.8, 21,952 Si atoms
// 71 / 79 / -.
template <class S>
cudaError_t launch_gather(const AtomArgs &a, cudaStream_t st) {
  if (a.N <= 0) return cudaSuccess;
  auto go = [&](auto ga, auto sub) {
    constexpr int GA = decltype(ga)::value, SUB = decltype(sub)::value;
    gather_kernel<S, false, GA, SUB><<<(a.N + GA - 1) / GA, GA * kGatherLanes * SUB, sizeof(float4) * a.ncode, st>>>(a);
    return cudaGetLastError();
  };
  using std::integral_constant;
  if (a.N <= kSplitGather) return go(integral_constant<int, kGatherAtoms / 2>{}, integral_constant<int, 4>{});
  if (a.N <= kSplitGather2) return go(integral_constant<int, kGatherAtoms>{}, integral_constant<int, 2>{});
  return go(integral_constant<int, kGatherAtoms>{}, integral_constant<int, 1>{});
}

// Batched launches (grid.y = population members); instantiated in the nep_batch_*.cu units.
template <class S>
cudaError_t launch_atom_batch(const AtomArgs &a, const ModelF &mf, int members, int block, cudaStream_t st);
template <class S>
cudaError_t launch_gather_batch(const AtomArgs &a, int members, int block, cudaStream_t st);

#ifdef NEP_BATCH_KERNELS
template <class S>
cudaError_t launch_atom_batch(const AtomArgs &a, const ModelF &mf, int members, int block, cudaStream_t st) {
  if (a.N <= 0 || members <= 0) return cudaSuccess;
  if (block != 64 && block != 128) return cudaErrorInvalidValue;
  if (a.precision >= 1 && block != 128) return cudaErrorInvalidValue;
  if (a.precision == 1) return launch_atom_as<S, 1, false, true, 64>(a, mf, members, st);
  if (a.precision == 2) return launch_atom_as<S, 2, false, true, 64>(a, mf, members, st);
  if (members == 1 && a.N <= kSplitAtoms) return launch_atom_as<S, 0, false, true, 16, 4>(a, mf, 1, st);
  if (members == 1 && a.N <= kSplitAtoms2) return launch_atom_as<S, 0, false, true, 32, 2>(a, mf, 1, st);
  return block == 64 ? launch_atom_as<S, 0, false, true, 64>(a, mf, members, st)
                     : launch_atom_as<S, 0, false, true, 128>(a, mf, members, st);
}

template <class S>
cudaError_t launch_gather_batch(const AtomArgs &a, int members, int block, cudaStream_t st) {
  if (a.N <= 0 || members <= 0) return cudaSuccess;
  constexpr int L = kGatherLanes;
  auto go = [&](auto ga, auto sub) {
    constexpr int GA = decltype(ga)::value, SUB = decltype(sub)::value;
    gather_kernel<S, true, GA, SUB><<<dim3((a.N + GA - 1) / GA, members), GA * L * SUB, 0, st>>>(a);
    return cudaGetLastError();
  };
  using std::integral_constant;
  if (block != 64 && block != 128 && block != 256) return cudaErrorInvalidValue;
  if (members == 1 && !a.sums && !a.sums_always) {  // no block sums, whose reader counts on `block`
    if (a.N <= kSplitGather) return go(integral_constant<int, kGatherAtoms / 2>{}, integral_constant<int, 4>{});
    if (a.N <= kSplitGather2) return go(integral_constant<int, kGatherAtoms>{}, integral_constant<int, 2>{});
  }
  const integral_constant<int, 1> one;
  if (block == 64) return go(integral_constant<int, 64>{}, one);
  if (block == 128) return go(integral_constant<int, 128>{}, one);
  return go(integral_constant<int, 256>{}, one);
}

template <class S>
void attach_batch(ShapeOps &o) {
  o.atom_batch = &launch_atom_batch<S>;
  o.gather_batch = &launch_gather_batch<S>;
}
#else
template <class S>
void attach_batch(ShapeOps &o);  // explicitly instantiated in the batch translation unit
#endif

template <class S> int gather_blocks(int N) {
  const int ga = N <= kSplitGather ? kGatherAtoms / 2 : kGatherAtoms;
  return (N + ga - 1) / ga;
}

template <class S>
ShapeOps make_ops() {
  ShapeOps o;
  o.nR = S::NR; o.KR = S::KR; o.nA = S::NA; o.KA = S::KA; o.H = S::H;
  o.L3 = S::L3; o.L4 = S::L4; o.L5 = S::L5; o.n_des = S::NDES;
  o.kp1 = S::KP1; o.np1 = S::NP1;
  o.ndp = S::NDP; o.krp = S::KRP; o.cap = S::CAP;
  o.atom = &launch_atom<S>;
  o.gather = &launch_gather<S>;
  o.atom_blocks = &atom_blocks<S>;
  o.gather_blocks = &gather_blocks<S>;
  o.lowreg = (S::NA + 1) * S::NK <= 128 ? 1 : 0;
  attach_batch<S>(o);
  return o;
}

}  // namespace nep
