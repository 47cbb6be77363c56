// NEP3 per-atom and gather kernels for any model shape, taken at run time.
//
// The compiled instantiations (nep_shape_*.cu) cover the workload shapes with every loop
// bound known to the compiler; this unit serves every other shape the parameters allow
// (n_max and N_bas up to 19, up to 256 neurons, l_max^3b 1..4, l_max^4b 0/2, l_max^5b 0/1),
// including the models the paper trains (Sec. III: MgAlCu n_max 12/8, carbon 10/8 with 100
// neurons). The arithmetic is the same (Eqs. qin, S_nk, the C3b/C4b/C5b forms, Ui, the
// partial forces and the gather of Eqs. F_ij, F_i, virial; Algorithms 1-4 fused into two
// kernels as in the compiled form), with run-time loops. FP32 network only.
#include <cuda_runtime.h>

#include "nep_kernels.cuh"

namespace nep {
namespace {

constexpr int kGenK = kGenMaxN + 1;  // most basis functions of a pair, most n of a descriptor
constexpr int kGenAtoms = 16;        // atoms per block of the per-atom kernel: two per warp
constexpr int kGenWarps = kGenAtoms / 2;
constexpr int kGenPairs = 16;  // angular pairs of an atom in shared memory at a time
constexpr int kPS = kGenPairs + 1;
constexpr int kSRow = 25;   // S_nk row of one n (24 used)
constexpr int kNeu = 32;    // neurons of the network at a time: one per lane
constexpr int kGenGatherLanes = 8;
constexpr int kBRow = 20;   // row of dU/dz of one neuron (16 atoms used)
// limits of the thread-per-atom kernel
constexpr int kThinSums = 72;            // S_nk of an atom
constexpr int kThinDes = kGenK + 40;     // descriptor components: l_max^3b = 1 with n_max^A = 19 has the most
constexpr int kThinWeights = 4096;       // N_neu x N_des
constexpr long long kThinEvals = 49152;  // least atoms x members of a call
constexpr long long kThinEvals4 = 131072;  // with l > 2 and more than 30 sums

// f_k(r), k = 0..K (Eq. f_n with the cosine cutoff), and f_k'(r) (0 without FP), given to out(k, f, fp)
// one after the other. Every multiply-add is spelled out, so that all kernels round alike.
template <bool FP, class Out>
__device__ __forceinline__ void basis_rt(float r, float inv_rc, int K, Out out) {
  const float u = r * inv_rc;
  float sn, cs;
  __sincosf(3.14159265358979f * u, &sn, &cs);
  const float hfc = 0.25f * (1.f + cs), hfcp = FP ? -0.25f * 3.14159265358979f * inv_rc * sn : 0.f;
  const float t1 = fmaf(r, inv_rc, -1.f);
  const float x = fmaf(2.f * t1, t1, -1.f), x2 = 2.f * x, xp = 4.f * t1 * inv_rc;
  float tkm1 = 1.f, tk = x, dkm1 = 0.f, dk = 1.f;
  out(0, 2.f * hfc, 2.f * hfcp);
  // unrolled in full: a caller that collects the values keeps them in registers
#pragma unroll
  for (int k = 1; k < kGenK; ++k) {
    if (k > K) break;
    if (k > 1) {
      const float tn = fmaf(x2, tk, -tkm1);
      tkm1 = tk;
      if (FP) {
        const float dn = fmaf(x2, dk, fmaf(2.f, tkm1, -dkm1));
        dkm1 = dk;
        dk = dn;
      }
      tk = tn;
    }
    out(k, (tk + 1.f) * hfc, FP ? fmaf(xp * dk, hfc, (tk + 1.f) * hfcp) : 0.f);
  }
}

// Sums over the warp of v[0..n): lane l < n returns the sum of v[l]. Each exchange halves the
// values a lane carries: 16 shuffles for up to 16 values, 6 more for up to 20.
__device__ __forceinline__ float lane_sums(float (&v)[kGenK], int n, int lane) {
  constexpr unsigned all = 0xffffffffu;
#pragma unroll
  for (int o = 8; o > 0; o >>= 1)
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const float lo = v[i], hi = v[i + o];
      v[i] = ((lane & o) ? hi : lo) + __shfl_xor_sync(all, (lane & o) ? lo : hi, o);
    }
  float r = v[0] + __shfl_xor_sync(all, v[0], 16);
  if (n > 16) {
#pragma unroll
    for (int o = 2; o > 0; o >>= 1)
#pragma unroll
      for (int i = 16; i < 16 + o; ++i) {
        const float lo = v[i], hi = v[i + o];
        v[i] = ((lane & o) ? hi : lo) + __shfl_xor_sync(all, (lane & o) ? lo : hi, o);
      }
    float h = v[16];
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) h += __shfl_xor_sync(all, h, o);
    if (lane >= 16) r = h;
  }
  return r;
}

// Shared memory of the per-atom kernel, in floats.
struct GenSmem {
  int sr, q, w, wr, x, beta, total;  // offsets; sr, wr: size of one atom's S and one warp's pair rows
};
__host__ __device__ inline GenSmem gen_smem(int nA, int KA, int D) {
  GenSmem m;
  m.sr = (nA + 1) * kSRow;
  m.q = kGenAtoms * m.sr;
  m.q = (m.q + 3) / 4 * 4;
  m.beta = m.q + D * kGenAtoms;
  m.w = m.beta + kNeu * kBRow;
  const int k1 = KA + 1;
  const int xr = k1 + 24 > 48 ? (k1 + 24 > 2 * k1 ? k1 + 24 : 2 * k1) : 48;  // rows f, b; f, f'; or A_k, C_k
  m.x = xr * kPS;
  m.wr = (xr + 2 * (nA + 1)) * kPS + kGenPairs;
  const int pairs = kGenWarps * m.wr, net = kNeu * (D | 1);
  m.total = m.w + ((pairs > net ? pairs : net) + 1) / 2 * 2 + 24 + 2 * kGenAtoms;  // even: doubles at its end
  return m;
}

// last polynomial index + 1 used by the 3-body terms and the 4-body term
__host__ __device__ inline int n_poly(int L3, int L4) {
  const int k3 = L3 == 1 ? 3 : L3 == 2 ? 8 : L3 == 3 ? 15 : 24;
  return (L4 >= 2 && k3 < 8) ? 8 : k3;
}

// Thin shapes (few S_nk and weights) in large calls: a thread per atom, S_nk, descriptor and dU/dq in
// local memory. What bounds it: latency of the scattered reads and of the L1 lines behind the local
// arrays. A warp per atom has little to spread over its lanes there and pays for its reductions and the
// block's phases; a small call of threads is one long serial chain instead. Whole calls, warp / thread
// per atom, us, of n_max 2/1, N_bas 3/2, l 2, 5 neurons: 1,000 atoms 103 / 123, 32,000 252 / 191, 64,000
// 454 / 262, 8 candidates on 67,259 atoms 2607 / 1208; of n_max 8/4, N_bas 8/4, l 2, 30 neurons: 1,000
// atoms 111 / 228, 32,000 321 / 330, 64,000 585 / 530, 8 candidates 3701 / 2387; of n_max 4/2, N_bas 4/4, l 4
// with 30 neurons (72 sums): 131,072 atoms 1142 / 1009, 200,000 1617 / 1619, 8 candidates 3802 / 3445. Past the
// limits the warp wins: l 4 with 48 sums, 67,259 atoms (this kernel alone) 372 / 440, 104 sums 849 / 1008,
// 256 neurons with 28 components 788 / 931.
// (The two forms round alike only up to the order of their sums.)
template <bool DESC_ONLY>
__global__ void __launch_bounds__(128) thin_atom_kernel(const AtomArgs a, const ModelF mf) {
  if (build_failed(a.guard)) return;
  const int N = a.N, T = a.T;
  const int nR = a.gR, KR = a.gKR, nA = a.gA, KA = a.gKA, H = a.gH, L3 = a.gL3, L4 = a.gL4, L5 = a.gL5, D = a.gD;
  const int NK = n_poly(L3, L4);
  const int off4 = (nR + 1) + (nA + 1) * L3, off5 = off4 + (L4 >= 2 ? nA + 1 : 0);
  const int mem = blockIdx.y;  // 0 for one structure, whose atoms carry structure 0
  const float *w0 = a.tab + mem * a.s_tab, *b0 = w0 + H * D, *w1 = b0 + H;
  const float *c_r = a.c_r + mem * a.s_tab, *c_a = a.c_a + mem * a.s_tab;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double U = 0.0;
  // (serving engine) atoms of a finished job frozen in the batch are skipped
  if (i < N && !(a.slots && a.slots[struct_of(a.pos4[i])].phase == 2)) {
    const float4 pi = a.pos4[i];
    const int ti = type_of(pi);
    const float4 *tab = a.dtab + (size_t)struct_of(pi) * a.ncode;
    const float inv_rcR = 1.f / a.rcR, inv_rcA = 1.f / a.rcA;
    const float rcR2 = a.rcR * a.rcR, rcA2 = a.rcA * a.rcA;
    float q[kThinDes], dq[kThinDes];  // descriptor, dU/dq
    float S[kThinSums];               // S_nk, then dU/dS_nk, row n at n * NK
    float f[kGenK], fp[kGenK], g[kGenK], gp[kGenK];
    for (int v = 0; v < D; ++v) q[v] = dq[v] = 0.f;
    for (int v = 0; v < (nA + 1) * NK; ++v) S[v] = 0.f;
    // radial descriptor (Eq. qin): the f_k summed over each neighbour type, then contracted with c_nk
    int base = 0;
    for (int t = 0; t < T; ++t) {
      const int cnt = a.nn_r[(size_t)t * N + i];
      for (int k = 0; k <= KR; ++k) f[k] = 0.f;
      for (int m = base; m < base + cnt; ++m) {
        const unsigned e = a.nl_r[(size_t)m * N + i];
        const float3 d = pair_vector(pi, a.pos4[e & a.jmask], tab[e >> a.jbits]);
        const float r2 = norm2(d);
        if (r2 < rcR2) basis_rt<false>(sqrtf(r2), inv_rcR, KR, [&](int k, float fk, float) { f[k] += fk; });
      }
      base += cnt;
      const float *c = c_r + (size_t)(ti * T + t) * (nR + 1) * (KR + 1);
      for (int n = 0; n <= nR; ++n)
        for (int k = 0; k <= KR; ++k) q[n] = fmaf(__ldg(c + n * (KR + 1) + k), f[k], q[n]);
    }
    // angular pairs inside the cutoff: body(m, d, r2, 1 / r) with g_n, and g_n' with FP
    const int na = a.nn_a[i];
    auto angular = [&](auto fpc, auto body) {
      constexpr bool FP = decltype(fpc)::value;
      for (int m = 0; m < na; ++m) {
        const unsigned e = a.nl_a[(size_t)m * N + i];
        const float4 pj = a.pos4[e & a.jmask];
        const float3 d = pair_vector(pi, pj, tab[e >> a.jbits]);
        const float r2 = norm2(d);
        if (!(r2 < rcA2)) continue;
        const float rinv = rsqrtf(r2);
        basis_rt<FP>(r2 * rinv, inv_rcA, KA, [&](int k, float fk, float fpk) {
          f[k] = fk;
          fp[k] = fpk;
        });
        const float *c = c_a + (size_t)(ti * T + type_of(pj)) * (nA + 1) * (KA + 1);
        for (int n = 0; n <= nA; ++n) {
          float x = 0.f, xp = 0.f;
          for (int k = 0; k <= KA; ++k) {
            const float ck = __ldg(c + n * (KA + 1) + k);
            x = fmaf(ck, f[k], x);
            if (FP) xp = fmaf(ck, fp[k], xp);
          }
          g[n] = x;
          gp[n] = xp;
        }
        body(m, d, r2, rinv);
      }
    };
    // angular sums S_nk (Eq. S_nk, b_k(d) r^-l)
    angular(std::false_type{}, [&](int, const float3 &d, float r2, float rinv) {
      const float rl[5] = {1.f, rinv, rinv * rinv, rinv * rinv * rinv, (rinv * rinv) * (rinv * rinv)};
      static_for<0, 24>([&](auto kc) {
        constexpr int k = decltype(kc)::value;
        if (k < NK) {
          const float b = poly_b<k>(d.x, d.y, d.z, r2) * rl[l_of_k(k)];
          for (int n = 0; n <= nA; ++n) S[n * NK + k] = fmaf(g[n], b, S[n * NK + k]);
        }
      });
    });
    // angular descriptor components (Sec. II D)
    for (int n = 0; n <= nA; ++n) {
      const float *s = S + n * NK;
      for (int l = 1; l <= L3; ++l) {
        float x = 0.f;
        for (int k = l * l - 1; k < l * (l + 2); ++k) x = fmaf(mf.c3b[k] * s[k], s[k], x);
        q[(nR + 1) + (l - 1) * (nA + 1) + n] = x;
      }
      if (L4 >= 2)
        q[off4 + n] = mf.c4b[0] * s[3] * s[3] * s[3] + mf.c4b[1] * s[3] * (s[4] * s[4] + s[5] * s[5]) +
                      mf.c4b[2] * s[3] * (s[6] * s[6] + s[7] * s[7]) + mf.c4b[3] * s[6] * (s[5] * s[5] - s[4] * s[4]) +
                      mf.c4b[4] * s[4] * s[5] * s[7];
      if (L5 >= 1) {
        const float s12 = s[1] * s[1] + s[2] * s[2];
        q[off5 + n] = mf.c5b[0] * s[0] * s[0] * s[0] * s[0] + mf.c5b[1] * s[0] * s[0] * s12 + mf.c5b[2] * s12 * s12;
      }
    }
    if constexpr (DESC_ONLY) {
      const size_t io = a.perm ? (size_t)a.perm[i] : (size_t)i;
      for (int v = 0; v < D; ++v) a.q_out[io * D + v] = (double)q[v];
      return;
    }
    // network (Eq. Ui) and dU/dq
    float u = 0.f;
    for (int mu = 0; mu < H; ++mu) {
      const float *w = w0 + mu * D;
      float z = -__ldg(b0 + mu);
      for (int v = 0; v < D; ++v) z = fmaf(__ldg(w + v), q[v], z);
      const float wo = __ldg(w1 + mu), h = tanhf(z), beta = wo * (1.f - h * h);
      u = fmaf(wo, h, u);
      for (int v = 0; v < D; ++v) dq[v] = fmaf(beta, __ldg(w + v), dq[v]);
    }
    u -= __ldg(w1 + H);
    U = (double)u;
    if (a.energy) a.energy[mem * a.s_out + (a.perm ? a.perm[i] : i)] = U;
    // radial force coefficients e^t_k = sum_n dU/dq_n c^{t_i t}_nk, rows padded with zeros
    float *const erow = a.e_rad + mem * a.s_erad + (size_t)i * T * a.est;
    for (int t = 0; t < T; ++t) {
      const float *c = c_r + (size_t)(ti * T + t) * (nR + 1) * (KR + 1);
      for (int k = 0; k < a.est; ++k) {
        float e = 0.f;
        if (k <= KR)
          for (int n = 0; n <= nR; ++n) e = fmaf(dq[n], __ldg(c + n * (KR + 1) + k), e);
        erow[t * a.est + k] = e;
      }
    }
    // dU/dS_nk from the explicit 3/4/5-body forms, in place
    for (int n = 0; n <= nA; ++n) {
      float s[8];
      float *const dS = S + n * NK;
      for (int k = 0; k < 8; ++k) s[k] = k < NK ? dS[k] : 0.f;
      for (int k = 0; k < NK; ++k) {
        const int l = k < 3 ? 1 : k < 8 ? 2 : k < 15 ? 3 : 4;
        dS[k] = l <= L3 ? 2.f * mf.c3b[k] * dS[k] * dq[(nR + 1) + (l - 1) * (nA + 1) + n] : 0.f;
      }
      if (L4 >= 2) {
        const float d4 = dq[off4 + n];
        const float *C = mf.c4b;
        dS[3] += d4 * (3.f * C[0] * s[3] * s[3] + C[1] * (s[4] * s[4] + s[5] * s[5]) + C[2] * (s[6] * s[6] + s[7] * s[7]));
        dS[4] += d4 * (2.f * C[1] * s[3] * s[4] - 2.f * C[3] * s[6] * s[4] + C[4] * s[5] * s[7]);
        dS[5] += d4 * (2.f * C[1] * s[3] * s[5] + 2.f * C[3] * s[6] * s[5] + C[4] * s[4] * s[7]);
        dS[6] += d4 * (2.f * C[2] * s[3] * s[6] + C[3] * (s[5] * s[5] - s[4] * s[4]));
        dS[7] += d4 * (2.f * C[2] * s[3] * s[7] + C[4] * s[4] * s[5]);
      }
      if (L5 >= 1) {
        const float d5 = dq[off5 + n];
        const float *C = mf.c5b;
        const float s12 = s[1] * s[1] + s[2] * s[2];
        dS[0] += d5 * (4.f * C[0] * s[0] * s[0] * s[0] + 2.f * C[1] * s[0] * s12);
        const float common = 2.f * C[1] * s[0] * s[0] + 4.f * C[2] * s12;
        dS[1] += d5 * common * s[1];
        dS[2] += d5 * common * s[2];
      }
    }
    // angular partial forces dU_i/dr_ij (angular terms of Eq. partial_force)
    float4 *const pang = a.p_ang + mem * a.s_pang;
    angular(std::true_type{}, [&](int m, const float3 &d, float r2, float rinv) {
      const float rl[5] = {1.f, rinv, rinv * rinv, rinv * rinv * rinv, (rinv * rinv) * (rinv * rinv)};
      float gx = 0.f, gy = 0.f, gz = 0.f, yy = 0.f;
      static_for<0, 24>([&](auto kc) {
        constexpr int k = decltype(kc)::value;
        if (k < NK) {
          float ak = 0.f, ck = 0.f;
          for (int n = 0; n <= nA; ++n) {
            ak = fmaf(S[n * NK + k], g[n], ak);
            ck = fmaf(S[n * NK + k], gp[n], ck);
          }
          ak *= rl[l_of_k(k)];
          ck *= rl[l_of_k(k)];
          const float3 gb = poly_grad<k>(d.x, d.y, d.z, r2);
          gx = fmaf(ak, gb.x, gx);
          gy = fmaf(ak, gb.y, gy);
          gz = fmaf(ak, gb.z, gz);
          yy = fmaf(ck, poly_b<k>(d.x, d.y, d.z, r2), yy);
        }
      });
      const float ux = d.x * rinv, uy = d.y * rinv, uz = d.z * rinv;
      const float gu = gx * ux + gy * uy + gz * uz;
      pang[(size_t)m * N + i] =
          make_float4((gx - gu * ux) + yy * ux, (gy - gu * uy) + yy * uy, (gz - gu * uz) + yy * uz, 0.f);
    });
  }
  if constexpr (!DESC_ONLY) {
    if (sums_needed(a) & kSumU) {  // a slot per kGenAtoms atoms, as the other form
#pragma unroll
      for (int o = kGenAtoms / 2; o > 0; o >>= 1) U += __shfl_xor_sync(0xffffffffu, U, o);
      if (i % kGenAtoms == 0 && i < N) a.partial_atom[i / kGenAtoms] = U;
    }
  }
}

// The other shapes and calls: one kernel for one structure and for batches (grid.y: members of a
// population), so that both give the same bits. 16 atoms per block. Descriptor and forces: a warp per atom (two atoms in turn). Radial pairs:
// a lane per pair, the f_k summed over each neighbour type before the contraction with c_nk.
// Angular pairs: those inside the cutoff go through shared memory in groups of 16, so that the
// contractions over n and k spread over all lanes however few pairs there are. Network: the block
// takes all its atoms through 32 neurons at a time, weights and activations in shared memory.
//
// What bounds it: instruction issue (59% busy; 21 of 32 lanes at work on average). The form before
// (a thread per atom, S_nk and the descriptor in local memory, every weight read per atom) was
// bound by local-memory traffic, 4 KB per thread: 20,000 MgAlCu atoms 511 us, now 162. Three
// blocks of 256 threads per SM (80 registers, a few spilled) are best: two and four take a sixth longer.
template <bool DESC_ONLY>
__global__ void __launch_bounds__(32 * kGenWarps, 3) generic_atom_kernel(const AtomArgs a, const ModelF mf) {
  if (build_failed(a.guard)) return;
  constexpr unsigned all = 0xffffffffu;
  const int N = a.N, T = a.T;
  const int nR = a.gR, KR = a.gKR, nA = a.gA, KA = a.gKA, H = a.gH, L3 = a.gL3, L4 = a.gL4, L5 = a.gL5, D = a.gD;
  const int NK = n_poly(L3, L4);
  const int off4 = (nR + 1) + (nA + 1) * L3, off5 = off4 + (L4 >= 2 ? nA + 1 : 0);
  const int mem = blockIdx.y;  // 0 for one structure, whose atoms carry structure 0
  const float *ann = a.tab + mem * a.s_tab;
  const float *w0 = ann, *b0 = ann + H * D, *w1 = b0 + H;
  const float *c_r = a.c_r + mem * a.s_tab, *c_a = a.c_a + mem * a.s_tab;
  extern __shared__ float4 gsm4[];
  float *const sm = reinterpret_cast<float *>(gsm4);
  const GenSmem lay = gen_smem(nA, KA, D);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float *const Q = sm + lay.q;            // [D][16] descriptor, then dU/dq
  float *const beta = sm + lay.beta;      // [32][kBRow]
  float *const W = sm + lay.w;            // [32][D | 1] weights of 32 neurons
  float *const X = W + warp * lay.wr;     // this warp's pair rows [..][kPS] (not while W is in use)
  float *const G = X + lay.x;             // g_n, g_n' [2 (nA + 1)][kPS]
  int *const tj_s = reinterpret_cast<int *>(G + 2 * (nA + 1) * kPS);
  float *const c3b = sm + lay.total - 24 - 2 * kGenAtoms;
  double *const Us = reinterpret_cast<double *>(sm + lay.total - 2 * kGenAtoms);
  if (tid < 24) c3b[tid] = mf.c3b[tid];
  __syncthreads();
  const float inv_rcR = 1.f / a.rcR, inv_rcA = 1.f / a.rcA;
  const float rcR2 = a.rcR * a.rcR, rcA2 = a.rcA * a.rcA;
  const int cA = (nA + 1) * (KA + 1), cR = (nR + 1) * (KR + 1);
  // (serving engine) atoms of a finished job frozen in the batch are skipped
  auto active = [&](int i) { return i < N && !(a.slots && a.slots[struct_of(a.pos4[i])].phase == 2); };
  // Angular pairs of atom i inside the cutoff, up to 16 at a time: mine(rank, ...) on the lane that
  // holds a pair, then all(count) on the whole warp, then done(rank, ...) on the pair's lane again.
  auto angular = [&](int i, const float4 &pi, const float4 *tab, auto mine, auto whole, auto done) {
    const int na = a.nn_a[i];
    for (int m0 = 0; m0 < na; m0 += 32) {
      const int m = m0 + lane;
      float3 d = make_float3(0.f, 0.f, 0.f);
      float r2 = 0.f;
      int tj = 0;
      bool in = false;
      if (m < na) {
        const unsigned e = a.nl_a[(size_t)m * N + i];
        const float4 pj = a.pos4[e & a.jmask];
        d = pair_vector(pi, pj, tab[e >> a.jbits]);
        r2 = norm2(d);
        tj = type_of(pj);
        in = r2 < rcA2;
      }
      const unsigned mask = __ballot_sync(all, in);
      const int cnt = __popc(mask), rank = __popc(mask & ((1u << lane) - 1u));
      for (int b = 0; b < cnt; b += kGenPairs) {
        const bool my = in && rank >= b && rank < b + kGenPairs;
        if (my) {
          tj_s[rank - b] = tj;
          mine(rank - b, d, r2);
        }
        __syncwarp();
        whole(cnt - b < kGenPairs ? cnt - b : kGenPairs);
        if (my) done(rank - b, m, d, r2);
        __syncwarp();
      }
    }
  };

  // ---- descriptor
  for (int u = 0; u < 2; ++u) {
    const int ia = 2 * warp + u, i = blockIdx.x * kGenAtoms + ia;
    float *const S = sm + ia * lay.sr;
    if (!active(i)) {
      for (int v = lane; v < D; v += 32) Q[v * kGenAtoms + ia] = 0.f;
      continue;
    }
    const float4 pi = a.pos4[i];
    const int ti = type_of(pi);
    const float4 *tab = a.dtab + (size_t)struct_of(pi) * a.ncode;
    // radial (Eq. qin)
    float qr[kGenK];
#pragma unroll
    for (int n = 0; n < kGenK; ++n) qr[n] = 0.f;
    int base = 0;
    for (int t = 0; t < T; ++t) {
      const int cnt = a.nn_r[(size_t)t * N + i];
      if (cnt == 0) continue;
      float f[kGenK];
#pragma unroll
      for (int k = 0; k < kGenK; ++k) f[k] = 0.f;
      for (int m = base + lane; m < base + cnt; m += 32) {
        const unsigned e = a.nl_r[(size_t)m * N + i];
        const float3 d = pair_vector(pi, a.pos4[e & a.jmask], tab[e >> a.jbits]);
        const float r2 = norm2(d);
        if (r2 < rcR2) basis_rt<false>(sqrtf(r2), inv_rcR, KR, [&](int k, float fk, float) { f[k] += fk; });
      }
      __syncwarp();
      base += cnt;
      const float F = lane_sums(f, KR + 1, lane);
      const float *c = c_r + (size_t)(ti * T + t) * cR + lane;
      if (lane <= KR) {
#pragma unroll
        for (int n = 0; n < kGenK; ++n)
          if (n <= nR) qr[n] = fmaf(__ldg(c + n * (KR + 1)), F, qr[n]);
      }
      __syncwarp();
    }
    const float qn = lane_sums(qr, nR + 1, lane);
    if (lane <= nR) Q[lane * kGenAtoms + ia] = qn;
    // angular sums S_nk (Eq. S_nk, b_k(d) r^-l): lane l holds the sums l, l + 32, ... of [n][24]
    constexpr int NS = (kGenK * 24 + 31) / 32;
    float acc[NS];
#pragma unroll
    for (int r = 0; r < NS; ++r) acc[r] = 0.f;
    float *const bk = X + (KA + 1) * kPS;
    angular(
        i, pi, tab,
        [&](int p, const float3 &d, float r2) {
          const float rinv = rsqrtf(r2);
          basis_rt<false>(r2 * rinv, inv_rcA, KA, [&](int k, float fk, float) { X[k * kPS + p] = fk; });
          const float rl[5] = {1.f, rinv, rinv * rinv, rinv * rinv * rinv, (rinv * rinv) * (rinv * rinv)};
          static_for<0, 24>([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            if (k < NK) bk[k * kPS + p] = poly_b<k>(d.x, d.y, d.z, r2) * rl[l_of_k(k)];
          });
        },
        [&](int cnt) {
          const int sh = cnt > 1 ? 32 - __clz(cnt - 1) : 0;
          for (int it = lane; it < ((nA + 1) << sh); it += 32) {
            const int p = it & ((1 << sh) - 1), n = it >> sh;
            if (p >= cnt) continue;
            const float *c = c_a + (size_t)(ti * T + tj_s[p]) * cA + n * (KA + 1);
            float g = 0.f;
            for (int k = 0; k <= KA; ++k) g = fmaf(__ldg(c + k), X[k * kPS + p], g);
            G[n * kPS + p] = g;
          }
          __syncwarp();
#pragma unroll
          for (int r = 0; r < NS; ++r) {
            if (32 * r >= (nA + 1) * 24) break;
            const int o = lane + 32 * r, n = o / 24, k = o % 24;
            if (n > nA || k >= NK) continue;
            for (int p = 0; p < cnt; ++p) acc[r] = fmaf(G[n * kPS + p], bk[k * kPS + p], acc[r]);
          }
          __syncwarp();
        },
        [](int, int, const float3 &, float) {});
#pragma unroll
    for (int r = 0; r < NS; ++r) {
      const int o = lane + 32 * r;
      if (o < (nA + 1) * 24) S[o / 24 * kSRow + o % 24] = acc[r];
    }
    __syncwarp();
    // angular descriptor components (Sec. II D)
    for (int it = lane; it < L3 * (nA + 1); it += 32) {
      const int l = it / (nA + 1) + 1, n = it - (l - 1) * (nA + 1);
      const float *s = S + n * kSRow;
      float q = 0.f;
      for (int k = l * l - 1; k < l * (l + 2); ++k) q = fmaf(c3b[k] * s[k], s[k], q);
      Q[((nR + 1) + it) * kGenAtoms + ia] = q;
    }
    if (lane <= nA) {
      const float *s = S + lane * kSRow;
      if (L4 >= 2)
        Q[(off4 + lane) * kGenAtoms + ia] =
            mf.c4b[0] * s[3] * s[3] * s[3] + mf.c4b[1] * s[3] * (s[4] * s[4] + s[5] * s[5]) +
            mf.c4b[2] * s[3] * (s[6] * s[6] + s[7] * s[7]) + mf.c4b[3] * s[6] * (s[5] * s[5] - s[4] * s[4]) +
            mf.c4b[4] * s[4] * s[5] * s[7];
      if (L5 >= 1) {
        const float s12 = s[1] * s[1] + s[2] * s[2];
        Q[(off5 + lane) * kGenAtoms + ia] =
            mf.c5b[0] * s[0] * s[0] * s[0] * s[0] + mf.c5b[1] * s[0] * s[0] * s12 + mf.c5b[2] * s12 * s12;
      }
    }
    __syncwarp();
    if constexpr (DESC_ONLY) {
      const size_t io = a.perm ? (size_t)a.perm[i] : (size_t)i;
      for (int v = lane; v < D; v += 32) a.q_out[io * D + v] = (double)Q[v * kGenAtoms + ia];
    }
  }
  if constexpr (!DESC_ONLY) {
    // ---- network (Eq. Ui) and dU/dq: forward a lane per neuron and a warp per two atoms, backward a
    // thread per descriptor component and eight atoms
    const int DP = D | 1;
    constexpr int NB = (2 * kGenMaxDes + 32 * kGenWarps - 1) / (32 * kGenWarps);
    float dq[NB][8];
#pragma unroll
    for (int r = 0; r < NB; ++r)
#pragma unroll
      for (int j = 0; j < 8; ++j) dq[r][j] = 0.f;
    float U[2] = {0.f, 0.f};
    for (int c0 = 0; c0 < H; c0 += kNeu) {
      const int nm = H - c0 < kNeu ? H - c0 : kNeu;
      __syncthreads();  // pair rows and weights of the chunk before are read
      for (int mu = warp; mu < nm; mu += kGenWarps)
        for (int v = lane; v < D; v += 32) W[mu * DP + v] = __ldg(w0 + (size_t)(c0 + mu) * D + v);
      __syncthreads();
      if (lane < nm) {
        const int mu = c0 + lane;
        float z[2];
        z[0] = z[1] = -__ldg(b0 + mu);
        for (int v = 0; v < D; ++v) {
          const float w = W[lane * DP + v];
          const float2 q = *reinterpret_cast<const float2 *>(Q + v * kGenAtoms + 2 * warp);
          z[0] = fmaf(w, q.x, z[0]);
          z[1] = fmaf(w, q.y, z[1]);
        }
        const float wo = __ldg(w1 + mu);
        float be[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const float h = tanhf(z[u]);
          U[u] = fmaf(wo, h, U[u]);
          be[u] = wo * (1.f - h * h);
        }
        *reinterpret_cast<float2 *>(beta + lane * kBRow + 2 * warp) = make_float2(be[0], be[1]);
      }
      __syncthreads();
#pragma unroll
      for (int r = 0; r < NB; ++r) {
        const int idx = tid + r * 32 * kGenWarps, v = idx >> 1, o = (idx & 1) * 8;
        if (v >= D) continue;
        for (int mu = 0; mu < nm; ++mu) {
          const float w = W[mu * DP + v];
          const float4 p = *reinterpret_cast<const float4 *>(beta + mu * kBRow + o);
          const float4 s = *reinterpret_cast<const float4 *>(beta + mu * kBRow + o + 4);
          dq[r][0] = fmaf(p.x, w, dq[r][0]);
          dq[r][1] = fmaf(p.y, w, dq[r][1]);
          dq[r][2] = fmaf(p.z, w, dq[r][2]);
          dq[r][3] = fmaf(p.w, w, dq[r][3]);
          dq[r][4] = fmaf(s.x, w, dq[r][4]);
          dq[r][5] = fmaf(s.y, w, dq[r][5]);
          dq[r][6] = fmaf(s.z, w, dq[r][6]);
          dq[r][7] = fmaf(s.w, w, dq[r][7]);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) U[u] += __shfl_xor_sync(all, U[u], o);
    __syncthreads();  // descriptor and weights are read
#pragma unroll
    for (int r = 0; r < NB; ++r) {
      const int idx = tid + r * 32 * kGenWarps, v = idx >> 1, o = (idx & 1) * 8;
      if (v >= D) continue;
#pragma unroll
      for (int j = 0; j < 8; ++j) Q[v * kGenAtoms + o + j] = dq[r][j];
    }
    __syncthreads();

    // ---- forces
    const float b1 = w1[H];
    for (int u = 0; u < 2; ++u) {
      const int ia = 2 * warp + u, i = blockIdx.x * kGenAtoms + ia;
      float *const S = sm + ia * lay.sr;
      const bool on = active(i);
      const float Ui = (u ? U[1] : U[0]) - b1;
      if (lane == 0) Us[ia] = on ? (double)Ui : 0.0;
      if (!on) continue;
      const float4 pi = a.pos4[i];
      const int ti = type_of(pi);
      const float4 *tab = a.dtab + (size_t)struct_of(pi) * a.ncode;
      if (a.energy && lane == 0) a.energy[mem * a.s_out + (a.perm ? a.perm[i] : i)] = (double)Ui;
      // radial force coefficients e^t_k = sum_n dU/dq_n c^{t_i t}_nk, rows padded with zeros
      float *const erow = a.e_rad + mem * a.s_erad + (size_t)i * T * a.est;
      for (int it = lane; it < T * a.est; it += 32) {
        const int t = it / a.est, k = it - t * a.est;
        float e = 0.f;
        if (k <= KR) {
          const float *c = c_r + (size_t)(ti * T + t) * cR + k;
          for (int n = 0; n <= nR; ++n) e = fmaf(Q[n * kGenAtoms + ia], __ldg(c + n * (KR + 1)), e);
        }
        erow[it] = e;
      }
      // dU/dS_nk from the explicit 3/4/5-body forms, in place: the 3-body part spread over the lanes,
      // the others a lane per n
      float s[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) s[k] = lane <= nA ? S[lane * kSRow + k] : 0.f;
      __syncwarp();
      for (int o = lane; o < (nA + 1) * 24; o += 32) {
        const int n = o / 24, k = o % 24, l = k < 3 ? 1 : k < 8 ? 2 : k < 15 ? 3 : 4;
        float *const x = S + n * kSRow + k;
        *x = l <= L3 ? 2.f * c3b[k] * *x * Q[((nR + 1) + (l - 1) * (nA + 1) + n) * kGenAtoms + ia] : 0.f;
      }
      __syncwarp();
      if (lane <= nA) {
        float *const dS = S + lane * kSRow;
        if (L4 >= 2) {
          const float d4 = Q[(off4 + lane) * kGenAtoms + ia];
          const float *C = mf.c4b;
          dS[3] += d4 * (3.f * C[0] * s[3] * s[3] + C[1] * (s[4] * s[4] + s[5] * s[5]) + C[2] * (s[6] * s[6] + s[7] * s[7]));
          dS[4] += d4 * (2.f * C[1] * s[3] * s[4] - 2.f * C[3] * s[6] * s[4] + C[4] * s[5] * s[7]);
          dS[5] += d4 * (2.f * C[1] * s[3] * s[5] + 2.f * C[3] * s[6] * s[5] + C[4] * s[4] * s[7]);
          dS[6] += d4 * (2.f * C[2] * s[3] * s[6] + C[3] * (s[5] * s[5] - s[4] * s[4]));
          dS[7] += d4 * (2.f * C[2] * s[3] * s[7] + C[4] * s[4] * s[5]);
        }
        if (L5 >= 1) {
          const float d5 = Q[(off5 + lane) * kGenAtoms + ia];
          const float *C = mf.c5b;
          const float s12 = s[1] * s[1] + s[2] * s[2];
          dS[0] += d5 * (4.f * C[0] * s[0] * s[0] * s[0] + 2.f * C[1] * s[0] * s12);
          const float common = 2.f * C[1] * s[0] * s[0] + 4.f * C[2] * s12;
          dS[1] += d5 * common * s[1];
          dS[2] += d5 * common * s[2];
        }
      }
      __syncwarp();
      // angular partial forces dU_i/dr_ij (angular terms of Eq. partial_force)
      float4 *const pang = a.p_ang + mem * a.s_pang;
      float *const Xp = X + (KA + 1) * kPS, *const Gp = G + (nA + 1) * kPS;
      float *const A = X, *const C = X + 24 * kPS;
      angular(
          i, pi, tab,
          [&](int p, const float3 &, float r2) {
            basis_rt<true>(r2 * rsqrtf(r2), inv_rcA, KA, [&](int k, float fk, float fpk) {
              X[k * kPS + p] = fk;
              Xp[k * kPS + p] = fpk;
            });
          },
          [&](int cnt) {
            const int sh = cnt > 1 ? 32 - __clz(cnt - 1) : 0;
            for (int it = lane; it < ((nA + 1) << sh); it += 32) {
              const int p = it & ((1 << sh) - 1), n = it >> sh;
              if (p >= cnt) continue;
              const float *c = c_a + (size_t)(ti * T + tj_s[p]) * cA + n * (KA + 1);
              float g = 0.f, gp = 0.f;
              for (int k = 0; k <= KA; ++k) {
                const float ck = __ldg(c + k);
                g = fmaf(ck, X[k * kPS + p], g);
                gp = fmaf(ck, Xp[k * kPS + p], gp);
              }
              G[n * kPS + p] = g;
              Gp[n * kPS + p] = gp;
            }
            __syncwarp();
            for (int it = lane; it < (NK << sh); it += 32) {
              const int p = it & ((1 << sh) - 1), k = it >> sh;
              if (p >= cnt) continue;
              float ak = 0.f, ck = 0.f;
              for (int n = 0; n <= nA; ++n) {
                const float x = S[n * kSRow + k];
                ak = fmaf(x, G[n * kPS + p], ak);
                ck = fmaf(x, Gp[n * kPS + p], ck);
              }
              A[k * kPS + p] = ak;
              C[k * kPS + p] = ck;
            }
            __syncwarp();
          },
          [&](int p, int m, const float3 &d, float r2) {
            const float rinv = rsqrtf(r2);
            const float rl[5] = {1.f, rinv, rinv * rinv, rinv * rinv * rinv, (rinv * rinv) * (rinv * rinv)};
            float gx = 0.f, gy = 0.f, gz = 0.f, yy = 0.f;
            static_for<0, 24>([&](auto kc) {
              constexpr int k = decltype(kc)::value;
              if (k < NK) {
                const float ak = A[k * kPS + p] * rl[l_of_k(k)], ck = C[k * kPS + p] * rl[l_of_k(k)];
                const float3 gb = poly_grad<k>(d.x, d.y, d.z, r2);
                gx = fmaf(ak, gb.x, gx);
                gy = fmaf(ak, gb.y, gy);
                gz = fmaf(ak, gb.z, gz);
                yy = fmaf(ck, poly_b<k>(d.x, d.y, d.z, r2), yy);
              }
            });
            const float ux = d.x * rinv, uy = d.y * rinv, uz = d.z * rinv;
            const float gu = gx * ux + gy * uy + gz * uz;
            pang[(size_t)m * N + i] =
                make_float4((gx - gu * ux) + yy * ux, (gy - gu * uy) + yy * uy, (gz - gu * uz) + yy * uz, 0.f);
          });
    }
    if (sums_needed(a) & kSumU) {
      __syncthreads();
      if (tid == 0) {
        double e = 0.0;
        for (int k = 0; k < kGenAtoms; ++k) e += Us[k];
        a.partial_atom[blockIdx.x] = e;
      }
    }
  }
}

// F_i and W_i (Algorithms 2 and 4, Eqs. F_ij, F_i, virial) with the run-time basis size of the
// radial coefficients; the epilogue (kick, kinetic energy, heat current, block sums) is the
// compiled gather kernel's.
//
// Eight lanes per atom take every eighth entry of its lists. What bounds it: latency of the
// scattered reads (positions, the neighbour's coefficients in 16-byte pieces, partial forces).
// 20,000 MgAlCu atoms: 34 us, 120 with a thread per atom and the f_k' in local memory.
template <bool BATCH, int GA, int NT>
__global__ void __launch_bounds__(NT) generic_gather_kernel(const AtomArgs a) {
  if (build_failed(a.guard)) return;
  constexpr int L = kGenGatherLanes;
  const int mem = BATCH ? (int)blockIdx.y : 0;
  const float *e_rad = a.e_rad + mem * a.s_erad;
  const float4 *p_ang = a.p_ang + mem * a.s_pang;
  const int N = a.N, T = a.T, KR = a.gKR, est4 = a.est / 4;
  __shared__ float fw[GA][13];
  __shared__ unsigned char on[GA];
  const float inv_rcR = 1.f / a.rcR;
  const float rcR2 = a.rcR * a.rcR, rcA2 = a.rcA * a.rcA;
  const int l = threadIdx.x % L;
  for (int ia = threadIdx.x / L; ia < GA; ia += NT / L) {
    const int i = blockIdx.x * GA + ia;
    float fx = 0.f, fy = 0.f, fz = 0.f;
    float w[9];
#pragma unroll
    for (int c = 0; c < 9; ++c) w[c] = 0.f;
    const bool active = i < N && !(BATCH && a.slots && a.slots[struct_of(a.pos4[i])].phase == 2);
    if (active) {
      const float4 pi = a.pos4[i];
      const int ti = type_of(pi);
      const float4 *tab = a.dtab + (BATCH ? (size_t)struct_of(pi) * a.ncode : 0);
      int cnt = 0;
      for (int t = 0; t < T; ++t) cnt += a.nn_r[(size_t)t * N + i];
      for (int m = l; m < cnt; m += L) {
        const unsigned e = a.nl_r[(size_t)m * N + i];
        const int j = e & a.jmask;
        const float4 pj = a.pos4[j];
        const float3 d = pair_vector(pi, pj, tab[e >> a.jbits]);
        const float r2 = norm2(d);
        if (!(r2 < rcR2)) continue;
        const float rinv = rsqrtf(r2);
        const float4 *eo = reinterpret_cast<const float4 *>(e_rad) + ((size_t)i * T + type_of(pj)) * est4;
        const float4 *ej = reinterpret_cast<const float4 *>(e_rad) + ((size_t)j * T + ti) * est4;
        float si = 0.f, sj = 0.f;
        float4 o4, j4;
        basis_rt<true>(r2 * rinv, inv_rcR, KR, [&](int k, float, float fp) {
          if (k % 4 == 0) o4 = __ldg(eo + k / 4), j4 = __ldg(ej + k / 4);
          si = fmaf(k % 4 == 0 ? o4.x : k % 4 == 1 ? o4.y : k % 4 == 2 ? o4.z : o4.w, fp, si);
          sj = fmaf(k % 4 == 0 ? j4.x : k % 4 == 1 ? j4.y : k % 4 == 2 ? j4.z : j4.w, fp, sj);
        });
        const float fs = (si + sj) * rinv;
        fx = fmaf(fs, d.x, fx);
        fy = fmaf(fs, d.y, fy);
        fz = fmaf(fs, d.z, fz);
        const float ws = -sj * rinv;
        const float px = ws * d.x, py = ws * d.y, pz = ws * d.z;
        w[0] = fmaf(d.x, px, w[0]); w[1] = fmaf(d.y, py, w[1]); w[2] = fmaf(d.z, pz, w[2]);
        w[3] = fmaf(d.x, py, w[3]); w[4] = fmaf(d.x, pz, w[4]); w[5] = fmaf(d.y, pz, w[5]);
        w[6] = fmaf(d.y, px, w[6]); w[7] = fmaf(d.z, px, w[7]); w[8] = fmaf(d.z, py, w[8]);
      }
      const int na = a.nn_a[i];
      for (int m = l; m < na; m += L) {
        const unsigned e = a.nl_a[(size_t)m * N + i];
        const float3 d = pair_vector(pi, a.pos4[e & a.jmask], tab[e >> a.jbits]);
        if (!(norm2(d) < rcA2)) continue;
        const float4 pij = p_ang[(size_t)m * N + i], pji = p_ang[a.rev_a[(size_t)m * N + i]];
        fx += pij.x - pji.x;
        fy += pij.y - pji.y;
        fz += pij.z - pji.z;
        w[0] = fmaf(d.x, pji.x, w[0]); w[1] = fmaf(d.y, pji.y, w[1]); w[2] = fmaf(d.z, pji.z, w[2]);
        w[3] = fmaf(d.x, pji.y, w[3]); w[4] = fmaf(d.x, pji.z, w[4]); w[5] = fmaf(d.y, pji.z, w[5]);
        w[6] = fmaf(d.y, pji.x, w[6]); w[7] = fmaf(d.z, pji.x, w[7]); w[8] = fmaf(d.z, pji.y, w[8]);
      }
    }
    __syncwarp();
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) {
      fx += __shfl_xor_sync(0xffffffffu, fx, o);
      fy += __shfl_xor_sync(0xffffffffu, fy, o);
      fz += __shfl_xor_sync(0xffffffffu, fz, o);
#pragma unroll
      for (int c = 0; c < 9; ++c) w[c] += __shfl_xor_sync(0xffffffffu, w[c], o);
    }
    if (l == 0) {
      float *row = fw[ia];
      row[0] = fx, row[1] = fy, row[2] = fz;
#pragma unroll
      for (int c = 0; c < 9; ++c) row[3 + c] = w[c];
      on[ia] = active ? 1 : 0;
    }
  }
  gather_finish<GA, NT>(a, mem, fw, on);
}

// ------------------------------------------------------------------------ launchers
constexpr int kGenGatherAtoms = 32;  // one structure; batches: 128 (the caller's block)

template <bool DESC_ONLY>
cudaError_t launch_generic_atom(const AtomArgs &a, const ModelF &mf, int members, cudaStream_t s) {
  const int nk = n_poly(a.gL3, a.gL4);
  const int sums = (a.gA + 1) * nk;
  if (sums <= kThinSums && a.gH * a.gD <= kThinWeights &&
      (long long)a.N * a.pop >= (nk <= 8 || sums <= 30 ? kThinEvals : kThinEvals4)) {
    thin_atom_kernel<DESC_ONLY><<<dim3((a.N + 127) / 128, members), 128, 0, s>>>(a, mf);
    return cudaGetLastError();
  }
  auto *kern = &generic_atom_kernel<DESC_ONLY>;
  const cudaError_t e = smem_limit_once(kern, sizeof(float) * gen_smem(kGenMaxN, kGenMaxN, kGenMaxDes).total);
  if (e != cudaSuccess) return e;
  kern<<<dim3((a.N + kGenAtoms - 1) / kGenAtoms, members), 32 * kGenWarps,
         sizeof(float) * gen_smem(a.gA, a.gKA, a.gD).total, s>>>(a, mf);
  return cudaGetLastError();
}

cudaError_t generic_atom(const AtomArgs &a, const ModelF &mf, int descriptor_only, cudaStream_t s) {
  if (a.N <= 0) return cudaSuccess;
  return descriptor_only ? launch_generic_atom<true>(a, mf, 1, s) : launch_generic_atom<false>(a, mf, 1, s);
}

cudaError_t generic_gather(const AtomArgs &a, cudaStream_t s) {
  if (a.N <= 0) return cudaSuccess;
  constexpr int GA = kGenGatherAtoms, NT = GA * kGenGatherLanes;
  generic_gather_kernel<false, GA, NT><<<(a.N + GA - 1) / GA, NT, 0, s>>>(a);
  return cudaGetLastError();
}

// batches: one block size (128 atoms per CTA of the gather kernel, whose block sums the population
// loss reads), population members along grid.y
cudaError_t generic_atom_batch(const AtomArgs &a, const ModelF &mf, int members, int block, cudaStream_t s) {
  if (a.N <= 0 || members <= 0) return cudaSuccess;
  if (block != 128 || a.precision != 0) return cudaErrorInvalidValue;
  return launch_generic_atom<false>(a, mf, members, s);
}

cudaError_t generic_gather_batch(const AtomArgs &a, int members, int block, cudaStream_t s) {
  if (a.N <= 0 || members <= 0) return cudaSuccess;
  if (block != 128) return cudaErrorInvalidValue;
  generic_gather_kernel<true, 128, 512><<<dim3((a.N + 127) / 128, members), 512, 0, s>>>(a);
  return cudaGetLastError();
}

int generic_atom_blocks(int N) { return (N + kGenAtoms - 1) / kGenAtoms; }
int generic_gather_blocks(int N) { return (N + kGenGatherAtoms - 1) / kGenGatherAtoms; }

}  // namespace

const ShapeOps *shape_generic() {
  static const ShapeOps ops = [] {
    ShapeOps o{};
    o.nR = o.KR = o.nA = o.KA = o.H = o.L3 = o.L4 = o.L5 = -1;  // any shape: taken from the handle
    o.n_des = 0;
    o.kp1 = o.np1 = 0;  // no tensor-core form
    o.atom = &generic_atom;
    o.gather = &generic_gather;
    o.atom_batch = &generic_atom_batch;
    o.gather_batch = &generic_gather_batch;
    o.atom_blocks = &generic_atom_blocks;
    o.gather_blocks = &generic_gather_blocks;
    o.lowreg = 0;
    return o;
  }();
  return &ops;
}

}  // namespace nep
