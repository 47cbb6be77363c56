// Internal declarations of libnep (GB300 / sm_103a). Not part of the public ABI.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <unordered_map>
#include <vector>

namespace nep {

constexpr int kMaxTypes = 8;
constexpr int kWideBuildAtoms = 131072;  // most atoms of the one-kernel neighbour build
constexpr int kListBuf = 512;   // largest neighbour-list capacity per atom
constexpr int kMaxImage = 3;    // largest cell/image offset searched per axis
// Distance (A) added to r_c^R + skin before a cell is left out of the neighbour search: far
// above the FP32 rounding of a pair distance, so no candidate that the distance test would
// accept is left out.
constexpr double kReachMargin = 2e-3;
// most atoms of the per-atom and gather kernels with four and with two groups of lanes per atom; the
// reasons stand at the kernels
constexpr int kSplitAtoms = 152 * 3 * 16, kSplitAtoms2 = 152 * 3 * 32;
constexpr int kSplitGather = 152 * 2 * 32, kSplitGather2 = 152 * 2 * 64;
constexpr int kReduceSlots = 16; // per-block partial sums: U, KE, W[9], force error, J[3], spare
// sums over all atoms that a call or an MD step reads (AtomArgs::sums)
enum { kSumU = 1, kSumKE = 2, kSumW = 4, kSumFerr = 8, kSumJ = 16, kSumP = 32 };  // kSumP: W's diagonal alone

// Geometry of one neighbour build: the cell grid, the packing of list entries and the
// table of pair shift vectors indexed by the packed image code.
struct Grid {
  int nc[3];          // cells per axis
  int R[3];           // cell offsets searched per axis (1 for large cells)
  int ncell;
  int jbits;          // bits of the atom index in a list entry
  unsigned jmask;
  int obits;          // bits of one offset component in the code (2 or 3)
  int ncode;          // entries of the shift table (2^(3 obits))
  double H[3][3];     // cell rows
  double Hinv[3][3];  // s = r . Hinv
  double Hc[3][3];    // rows of one grid cell: H[a] / nc[a]
  float Hf[3][3], Hinvf[3][3];  // H and Hinv rounded to FP32 (candidate search: the FP64 to FP32
                                // conversions run on the slow FP64 pipe)
  float reach[3];     // (r_c^R + skin + kReachMargin) / cell thickness per axis: a cell whose
                      // gap to an atom's cell position exceeds it along any axis holds no pair
  int cell_off;       // first global cell of this structure (batches; 0 for one structure)
  int dtab_off;       // first shift-table entry of this structure (batches; 0 for one structure)
};

// Structures of a batch: grid of every structure and the structure of every atom (internal
// order). A single structure uses grids == nullptr and the grid passed by value.
struct Batch {
  const Grid *grids;
  const int *sid;
  int n;
  // serving engine: per-structure build requests of the drift kernel. A build that is not
  // forced (BuildStatus::full == 0) then re-sorts and re-lists only the flagged structures;
  // every other structure keeps its atom order, cells, lists and reference positions.
  int *sflag = nullptr;
};

// Per-atom device arrays. Internally atoms are kept in cell order (re-sorted at every
// neighbour rebuild); perm[i] is the caller's index of internal atom i.
struct AtomState {
  double *x, *v, *F, *x_ref, *origin;  // [N][3]
  int *types, *perm, *cell_of;         // [N]
  float4 *pos4;                        // [N] cell-local FP32 coordinates + type bits
  float4 *posA;                        // [N] FP32 coordinates in the structure's cell frame at the
                                       // last build (neighbour search only) + type bits
  double *x2, *v2, *F2;                // reorder scratch [N][3]
  int *types2, *perm2, *cell2;         // reorder scratch [N]
};

// A structure as the caller holds it (device arrays), taken over at the start of a build; pos ==
// nullptr: the build uses the atoms in place. dtab: shift table to fill (one structure), or null.
struct LoadSrc {
  const double *pos = nullptr;
  const int *types = nullptr;
  float4 *dtab = nullptr;
};

// Cell list and neighbour lists.
struct ListBufs {
  int *cell_count, *cell_cursor, *cell_start, *cell_atoms;
  unsigned *nl_r;  // [cap_r][N]
  int *nn_r;       // [T][N]
  unsigned *nl_a;  // [cap_a][N]
  int *nn_a;       // [N]
  int *rev_a;      // [cap_a][N]
  int cap_r, cap_a;
  unsigned *stage_e;        // [cap_r][N] accepted candidates of one build, or null (second scan)
  unsigned char *stage_g;   // [cap_r][N] their groups
  unsigned long long *part;  // [kStatSlots][4] partial sums of a build's list statistics
  unsigned *bar;             // [1 + kBuildSums] barrier of the one-kernel build (zero between launches), block sums
  unsigned polls;            // most polls of a wait at the barrier (kBarrierPolls, or fewer for tests)
};
constexpr int kStatSlots = 64;
constexpr int kBuildSums = 1023;  // blocks of the one-kernel build at most
constexpr unsigned kBarrierPolls = 1u << 22;  // seconds

// Device-visible status written by the builders.
struct BuildStatus {
  int overflow;        // any atom exceeded a list capacity
  int max_r, max_a;    // largest radial/angular list length
  int rev_missing;     // angular pairs without their reverse pair (must stay 0)
  unsigned long long sum_r, sum_a;  // total list entries
  unsigned long long in_r, in_a;    // entries with r < r_c (at build time)
  int rebuild;         // a rebuild is pending (set by the drift kernel or the host)
  int full;            // the pending build covers every structure (forced); else, with
                       // per-structure flags, only the flagged ones
  int bad_input;       // bit 0: type out of range, bit 1: non-finite position, bit 2: the build's
                       // grid barrier ran out
  int tc_timeout;      // a tensor-core completion wait or a grid barrier ran out (results invalid)
  long long n_rebuilds;
  long long md_steps;
};

// FIRE minimisation state (Bitzek et al., Phys. Rev. Lett. 97, 170201 (2006)), kept on the
// device so that a relaxation step needs no host round trip.
struct FireState {
  double dt;         // current time step (fs)
  double alpha;      // current mixing factor
  double dt_max;     // largest time step
  double fmax2;      // convergence threshold on max_i |F_i|^2
  int n_pos;         // consecutive steps with P = F . v > 0
  int converged;     // set once max_i |F_i| < fmax: later steps change nothing
  int steps;         // steps taken before convergence
  int pad;
};

// One job of the batched serving engine (a structure of the batch), device resident.
enum { kJobSingle = 0, kJobFire = 1, kJobNve = 2 };
struct EngineSlot {
  int kind;          // kJob*
  int phase;         // 0: initial evaluation this iteration, 1: stepping, 2: finished (frozen)
  int steps_done;    // velocity-Verlet steps taken
  int n_steps;       // NVE: steps to take; FIRE: most steps
  double dt;         // NVE time step (fs)
  FireState fire;    // FIRE state (kind == kJobFire)
};

// A job entering the batched serving engine (host arrays stay valid during engine_relayout).
struct EngineJob {
  int kind, n, n_steps;
  double box[9];
  double dt, fmax;
  const double *pos, *vel;
  const int *types;
};

// Bussi-Donadio-Parrinello velocity rescaling (J. Chem. Phys. 126, 014101 (2007)), device
// resident: the caller's random numbers for every step (R1 ~ N(0,1), S ~ chi^2 with N_f - 1
// degrees of freedom) and the factor of the current step.
struct ThermoState {
  double c;              // exp(-dt / tau)
  double kbar;           // target kinetic energy N_f k_B T0 / 2 (eV)
  double nf;             // degrees of freedom N_f = 3N - 3
  double alpha;          // velocity factor of the last step
  const double *rand;    // [n_steps][2] (R1, S)
  long long step;        // steps thermostatted in this run
};

// Pair vector d = r_j - r_i from cell-local FP32 coordinates and the shift of the image
// code. The explicitly rounded operations make d_ji the exact negation of d_ij, so both
// atoms of a pair take the same inclusion decision in every kernel.
__device__ __forceinline__ float3 pair_vector(const float4 &pi, const float4 &pj, const float4 &D) {
  return make_float3(__fadd_rn(__fsub_rn(pj.x, pi.x), D.x), __fadd_rn(__fsub_rn(pj.y, pi.y), D.y),
                     __fadd_rn(__fsub_rn(pj.z, pi.z), D.z));
}
__device__ __forceinline__ float norm2(const float3 &d) {
  return __fmaf_rn(d.z, d.z, __fmaf_rn(d.y, d.y, __fmul_rn(d.x, d.x)));
}
// pos4.w holds the atom type in bits 0-7 and its structure (batches) in bits 8-31.
__device__ __forceinline__ int type_of(const float4 &p) { return __float_as_int(p.w) & 0xFF; }
__device__ __forceinline__ int struct_of(const float4 &p) { return __float_as_int(p.w) >> 8; }

// Raise a kernel's dynamic shared memory limit once, to a bound that covers every launch
// (any type count up to kMaxTypes, the largest shift table). The attribute is per function
// and process-wide: setting it per launch to that launch's size would race between threads
// launching the same kernel with different sizes.
template <class K>
cudaError_t smem_limit_once(K kern, size_t bound) {
  static std::mutex mu;
  static std::unordered_map<const void *, size_t> done;
  std::lock_guard<std::mutex> lk(mu);
  const void *key = reinterpret_cast<const void *>(kern);
  auto it = done.find(key);
  if (it != done.end() && it->second >= bound) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bound);
  if (e == cudaSuccess) done[key] = bound;
  return e;
}

// Arguments of the per-atom and gather kernels (everything except the model weights).
struct AtomArgs {
  int N, T;
  int jbits;
  unsigned jmask;
  int ncode;
  float rcR, rcA;
  const float4 *pos4;      // [N] cell-local xyz + type bits
  const float4 *dtab;      // [ncode] pair shift vectors
  const unsigned *nl_r;    // [cap_r][N] packed entries, grouped by neighbour type
  const int *nn_r;         // [T][N] radial entries per neighbour type
  const unsigned *nl_a;    // [cap_a][N]
  const int *nn_a;         // [N]
  const int *rev_a;        // [cap_a][N] flat index of the reverse angular pair
  int cap_r, cap_a;        // list capacities (slots per atom), bounds of the list prefetches
  // model table(s) in FP32 (TableLayout): network and descriptor coefficients, one per member
  const float *tab;        // [members][s_tab]
  long long s_tab;         // member stride in floats (0: one model)
  const float *c_r;        // its c^R [T][T][nR+1][krp]
  const float *c_a;        // its c^A [T][T][cap]
  float *e_rad;            // [N][T][est] radial force coefficients
  int est;
  float4 *p_ang;           // [cap_a][N] angular partial forces
  const int *perm;         // [N] caller index of each internal atom (outputs are scattered)
  double *energy;          // [N] or null
  double *q_out;           // [N][N_des] descriptor output (descriptor mode) or null
  double *partial_atom;    // [gridDim] block sums of U
  // gather outputs
  double *force;           // [N][3] or null (md keeps FP64 forces here)
  double *virial;          // [N][9] or null
  double *partial_gather;  // [gridDim][kReduceSlots]
  // block sums to form (kSum*): every launch the `sums_always`, and the `sums` on every launch or,
  // with step_ctl (MD), on steps that write a thermo row: step_ctl[0] is the step's number in
  // the call (counted by the drift kernel), step_ctl[2] the interval of the rows
  int sums, sums_always;
  const int *step_ctl;
  // md kick in the gather epilogue
  int md_kick;
  double half_dt;          // dt/2 in fs
  const double *inv_mass_kappa;  // [T] 1 / (m * 103.64...) for a = F * that
  const double *mass_kappa_half; // [T] m * 103.64... / 2 for kinetic energy
  double *vel;             // [N][3]
  int precision;           // network: 0 FP32 on the FMA pipes; 1 BF16, 2 split BF16 on the tensor cores
  int *tc_err;             // set when a tensor-core wait ran out
  const BuildStatus *guard;  // of the build queued before this launch (build_failed), or null
  // Batched kernels only. dtab then holds ncode shift vectors per structure (the structure
  // index sits in pos4.w above the type bits), and blockIdx.y selects the member of a
  // population whose coefficients and network the block uses; every per-member array is
  // offset by member x its stride (in elements).
  long long s_erad, s_pang;           // strides of e_rad, p_ang
  long long s_out;                    // atoms per member in energy (x1), force (x3), virial (x9)
  const double *f_tar;     // [N][3] caller order, or null: sum of (F_i - F_tar,i)^2 per block
  const FireState *fire;   // FIRE relaxation: kick with its dt, none once converged (or null)
  // heat current J_i = W_i . v_i (Eq. Ji) with the velocities after the kick (MD) or these
  // caller-order velocities; per-atom values in caller order, or null
  const double *vel_in;    // [N][3] caller order, or null
  double *heat;            // [N][3] caller order, or null
  // batched serving engine: per-structure kick (phase, time step, FIRE state), or null
  const EngineSlot *slots;
  // model shape at run time: read only by the kernels that take the shape at run time (shapes
  // without a compiled instantiation)
  int gR, gKR, gA, gKA, gH, gL3, gL4, gL5, gD;
  int pop;  // members of the whole call (however many a launch holds): 1, or the population's
};

// The build before this launch failed (the host, which has not looked yet, reports it or builds
// again): kernels queued behind it write nothing, and follow no list entry or reverse slot, which a
// build whose barrier ran out may not have written.
__device__ __forceinline__ bool build_failed(const BuildStatus *st) {
  return st && (st->overflow | st->bad_input | st->rev_missing);
}

// The block sums that this launch forms.
__device__ __forceinline__ int sums_needed(const AtomArgs &a) {
  const bool row = !a.step_ctl || a.step_ctl[0] % a.step_ctl[2] == 0;
  return a.sums_always | (row ? a.sums : 0);
}

// Model constants of one handle, FP32.
struct ModelF {
  float c3b[24];
  float c4b[5];
  float c5b[3];
};

// Per-shape launchers (one instantiation per compiled hyper-parameter shape).
struct ShapeOps {
  int nR, KR, nA, KA, H, L3, L4, L5;
  int n_des;
  int kp1, np1;  // tensor-core network tile shapes (K of GEMM1, N of GEMM1)
  int ndp, krp, cap;  // padded rows of the model table (TableLayout); 0: unpadded
  cudaError_t (*atom)(const AtomArgs &, const ModelF &, int descriptor_only, cudaStream_t s);
  cudaError_t (*gather)(const AtomArgs &, cudaStream_t s);
  // batched kernels (per-structure shift tables; `members` population members along y;
  // `block` atoms per CTA: 64 or 128 for the atom kernel (128 names the 64 of the tensor-core network),
  // 64, 128 or 256 for the gather kernel)
  cudaError_t (*atom_batch)(const AtomArgs &, const ModelF &, int members, int block, cudaStream_t s);
  cudaError_t (*gather_batch)(const AtomArgs &, int members, int block, cudaStream_t s);
  int (*atom_blocks)(int N);
  int (*gather_blocks)(int N);
  int lowreg;  // nep_tuning.atom_form 3 exists ((n_max^A + 1) x 24 <= 128)
};

int shape_count();
const ShapeOps *shape_at(int i);
// kernels that take the model shape at run time (any shape within these limits)
constexpr int kGenMaxN = 19;     // n_max^R, n_max^A, N_bas^R, N_bas^A
constexpr int kGenMaxNeu = 256;  // N_neu
constexpr int kGenMaxDes = (kGenMaxN + 1) * 7;
const ShapeOps *shape_generic();

// FP32 table of one model on the device: w0 [H][ndp], b0 [H], w1 [H], b1, c^R [T][T][n_R+1][krp],
// c^A [T][T][cap] ([n][k] packed), and w0 as the BF16 operand tiles of the tensor-core network
// (two terms hi + lo of every value, K-major core matrices of 8 rows x 16 bytes, zero padded
// to [np1][kp1]); the parts at multiples of 4 floats. The compiled shapes pad
// the rows to whole float4s, so that a block copies the table into shared memory as it stands.
struct TableLayout {
  int T, nR, KR, nA, KA, H, D;  // model shape
  int ndp, krp, cap;
  int np1, kp1;                 // W0 tile of the tensor-core network (0: none)
  int cr, ca, tc, total;        // offsets of c^R, c^A and the two tiles, size (floats)
};
inline TableLayout table_layout(const ShapeOps *o, int T, int nR, int KR, int nA, int KA, int H, int D) {
  TableLayout t{T, nR, KR, nA, KA, H, D, o->ndp ? o->ndp : D, o->krp ? o->krp : KR + 1,
                o->cap ? o->cap : (nA + 1) * (KA + 1), o->np1, o->kp1, 0, 0, 0, 0};
  auto r4 = [](int x) { return (x + 3) / 4 * 4; };
  t.cr = r4(H * t.ndp + 2 * H + 1);
  t.ca = t.cr + r4(T * T * (nR + 1) * t.krp);
  t.tc = t.ca + r4(T * T * t.cap);
  t.total = t.tc + t.np1 * t.kp1;  // two tiles of 2-byte values
  return t;
}
// Place in the table of entry v of the parameter vector (order c^R, c^A, w0, b0, w1, b1).
__host__ __device__ inline int table_place(const TableLayout &t, int v) {
  const int ncr = t.T * t.T * (t.nR + 1) * (t.KR + 1);
  if (v < ncr) return t.cr + v / (t.KR + 1) * t.krp + v % (t.KR + 1);
  v -= ncr;
  const int c = (t.nA + 1) * (t.KA + 1), nca = t.T * t.T * c;
  if (v < nca) return t.ca + v / c * t.cap + v % c;
  v -= nca;
  return v < t.H * t.D ? v / t.D * t.ndp + v % t.D : t.H * t.ndp + (v - t.H * t.D);
}

// Element (mu, nu) of a W0 tile.
__host__ __device__ inline int tile_place(const TableLayout &t, int mu, int nu) {
  return ((mu / 8) * (t.kp1 / 8) + nu / 8) * 64 + (mu % 8) * 8 + (nu % 8);
}

// Host helpers shared by the handle-based and the static-scratch entry points.
struct Grid;
void model_constants(ModelF &m);
int build_grid(const double *box, double rl, int N, Grid &g, double *volume, const char **err);
cudaError_t load_source(int N, const double *pos, const int *types, float4 *dtab, const AtomState &a, int device,
                        cudaStream_t s, LoadSrc *out);
cudaError_t launch_rebuild(int N, int T, const Grid &g, const Batch &B, float rlR2, float rlA2, float rcR2, float rcA2,
                           const AtomState &a, const ListBufs &L, int count_only,
                           int move, const LoadSrc &src, BuildStatus *st, cudaStream_t s);
void launch_export(int N, const AtomState &a, const Grid &g, const Batch &B, double *pos, double *vel, double *force,
                   cudaStream_t s);
void launch_export_lists(int N, int T, const float4 *pos4, const int *perm, const ListBufs &L, const float4 *dtab,
                         int ncode, int jbits, unsigned jmask, int cap, int *nn_r, int *j_r, float *d_r,
                         int *nn_a, int *j_a, float *d_a, cudaStream_t s);
// batches: structure index of every atom, the shift tables of all structures, and the
// per-structure sums of per-atom energies and virials (caller order, per member)
void launch_struct_ids(int n_struct, const int *offsets, int *sid, cudaStream_t s);
void launch_shift_tables(int n_struct, const Grid *grids, int ncode, float4 *dtab, cudaStream_t s);
// max_atoms: the largest structure (structures above kWideSum atoms are summed by a block)
void launch_struct_sums(int n_struct, int members, const int *offsets, int N, const double *e_atom,
                        const double *w_atom, double *e_struct, double *w_struct, int max_atoms,
                        const BuildStatus *guard, cudaStream_t s);
void launch_arm_rebuild(BuildStatus *st, unsigned *bar, cudaStream_t s);
void launch_fire_mix(int N, const AtomState &a, FireState *fire, int check_only, cudaStream_t s);
// batched serving engine
void launch_engine_drift(int N, const AtomState &a, const int *sid, const EngineSlot *slots,
                         const double *inv_mass_kappa, double half_skin2, int *sflag, BuildStatus *st,
                         cudaStream_t s);
void launch_clear_flags(BuildStatus *st, unsigned *bar, cudaStream_t s);
void launch_engine_advance(int n_struct, const int *offsets, const AtomState &a, EngineSlot *slots, cudaStream_t s);
void launch_engine_export(int o, int n, const AtomState &a, const Grid &g, double *out, int *bad, cudaStream_t s);
void launch_engine_relayout(int n_keep, const int4 *table, const AtomState &src, AtomState dst, cudaStream_t s);
void launch_thermostat(int N, const AtomState &a, int nb_gather, const double *partial_gather, ThermoState *ts,
                       cudaStream_t s);
// population evaluation: parameter vectors into kernel arrays, BF16 tiles, Eq. loss
void launch_unpack_population(int n_pop, const double *z, int n_par, const TableLayout &t, float *tab, double *reg,
                              cudaStream_t s);
void launch_population_tiles(int n_pop, float *tab, const TableLayout &t, cudaStream_t s);
void launch_population_loss(int members, int n_struct, const int *offsets, const double *e_struct,
                            const double *w_struct, const double *e_tar, const double *w_tar,
                            const double *partial_gather, int nb_gather, int N, const double *reg, int n_par,
                            const double *lambda, double *loss, cudaStream_t s);

}  // namespace nep

// Batched serving engine on a library handle (implemented with the C ABI, used by the server).
struct nep_handle;
namespace nep {
int engine_relayout(nep_handle *h, const std::vector<int> &keep, const std::vector<EngineJob> &add, cudaStream_t s,
                    size_t target_bytes = 0);
int engine_step(nep_handle *h, cudaStream_t s, int n_iter, bool force_rebuild);
// neighbour builds of the engine's batch so far (read with the status after every chunk)
long long engine_builds(const nep_handle *h);
int engine_fetch(nep_handle *h, const std::vector<int> &jobs, size_t first, size_t *end, cudaStream_t s);
const double *engine_arrays(nep_handle *h, size_t q);
int engine_jobs(const nep_handle *h);
int engine_atoms(const nep_handle *h);
const EngineSlot &engine_slot(const nep_handle *h, int k);
double engine_energy(const nep_handle *h, int k);
const double *engine_virial(const nep_handle *h, int k);
void set_thread_alloc_stream(cudaStream_t s);
void release_workspace(nep_handle *h);
size_t workspace_bytes(nep_handle *h);
cudaError_t stream_sync(cudaStream_t s);
}  // namespace nep
