// Internal declarations shared by the kernel translation units and api.cu.
#pragma once

#include <cuda_runtime.h>

#include <utility>
#include <vector>

#include "common.cuh"
#include "hpic.h"

namespace hpic {

// Kernels of a step follow one another in a stream.  A chained launch lets the
// next one's blocks take their places while the last one's are finishing
// (programmatic dependent launch) instead of after its end has been reported;
// every kernel of the chain begins with after_previous(), which waits for the
// kernels before it to end and their stores to be visible, so only the launch
// itself overlaps.  No kernel releases the next one early: its blocks would
// take the SMs that happen to be free first and crowd there (FP64, 1e5
// electrons: a step 226 instead of 198 us).  Small runs are made of such gaps:
// with one clearing for two, the step closed by the heating kernel and chained
// launches, a step of 1e5 electrons (FP32) went from 50 to 37 us, of 2e3
// electrons from 33 to 25 us.  Only a launch that directly follows another
// kernel of the same call is chained.
__device__ __forceinline__ void after_previous() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <typename... P, typename... A>
inline void launch_chained(void (*kernel)(P...), int grid, int threads, size_t smem,
                           cudaStream_t st, A &&...args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

// particle storage: structure of arrays, positions in cells, momenta u = p/(m_e c)
template <typename R>
struct PView {
  R *x, *y, *z, *ux, *uy, *uz, *tau;
  R *w;  // per-electron weight (read only when Consts::weighted)
  uint32_t *id;
};

// grid storage: vector components as (nx+1)(ny+1)(nz+1) arrays (x fastest)
template <typename R>
struct GView {
  R *E[3], *B[3], *J[3];
  double *T, *eta, *H;  // cell-centred, double
  R *eta_r;             // eta in the field precision (its own FP32 copy, or eta itself)
  double *Ti;           // ion temperature (K)
  R *Fsig;              // F_sigma of each cell, from T_i
};

struct TallyView {
  double *tal;      // T_COUNT scalars
  double *hist;     // 2 x (n_E+2) x n_th: energy-weighted, then number-weighted
  double *history;  // max_history
};

// the per-electron constants in the kernel's own precision (folded on the
// host so that no double->float conversion runs per electron)
//
// Everything the per-electron code needs that differs between the targets
// of a batch is here (with the grid and tally views); from Consts it reads
// only run-wide values, so the batched kernel can take Consts as a kernel
// parameter and keep just these per target.
template <typename R>
struct HotK {
  R w, cdt, E_cut, K_tau, k_min, inv_boost;
  R K_ion[4], L_I[4], K_sc[4], K_lg[4];  // per element (n_solids used)
  R eps_esc, du_reflux, sigma_dtheta, tE_min, tE_max, inv_dlogE, th_scale, t_inv_dlog;
  double w_d;                // the weight in FP64 (photon weights)
  int nx, ny, nz, n_solids;  // the target's cells and elements
  uint32_t target_index;     // fourth Philox counter word
};

// the hot constants in precision R
template <typename R>
inline HotK<R> make_hot(const Consts &K) {
  HotK<R> h;
  h.w = R(K.w);
  h.cdt = R(K.cdt_dx);
  h.E_cut = R(K.E_cut);
  for (int s = 0; s < 4; ++s) {
    h.K_ion[s] = R(K.K_ion[s]);
    h.L_I[s] = R(K.L_I[s]);
    h.K_sc[s] = R(K.K_sc[s]);
    h.K_lg[s] = R(K.K_lg[s]);
  }
  h.K_tau = R(K.K_tau);
  h.k_min = R(K.k_min);
  h.inv_boost = R(K.inv_boost);
  h.eps_esc = R(K.eps_esc);
  h.du_reflux = R(K.du_reflux);
  h.sigma_dtheta = R(K.sigma_dtheta);
  h.tE_min = R(K.tE_min);
  h.tE_max = R(K.tE_max);
  h.inv_dlogE = R(K.inv_dlogE);
  h.th_scale = R(K.n_th / 3.14159265358979323846);
  h.t_inv_dlog = R(K.t_inv_dlog);
  h.w_d = K.w;
  h.nx = K.nx;
  h.ny = K.ny;
  h.nz = K.nz;
  h.n_solids = K.n_solids;
  h.target_index = K.target_index;
  return h;
}

// n / d of n < 2^31 as a multiplication (see node_of)
struct Quotient {
  uint32_t m;  // floor(2^(31 + s) / d) + 1, s = ceil(log2 d)
  int sh;      // s - 1
  __device__ __forceinline__ unsigned quotient(unsigned n) const { return __umulhi(n, m) >> sh; }
};
inline Quotient make_quotient(uint32_t d) {  // d >= 2
  int s = 1;
  while ((1ull << s) < d) ++s;
  return Quotient{(uint32_t)((1ull << (31 + s)) / d + 1), s - 1};
}

// what the field and heating kernels need of one target: the sizes, and the
// constants in the precision each is used in, so that no conversion runs per
// node (an FP64 conversion costs as much as an FP64 operation there)
struct FieldCommon {
  int nx, ny, nz, sy, sz;  // sy, sz: nodes per row and plane
  int physics, n_solids;
  int cold;                // lambda1 > 0: eta_cold limits eta
  Quotient by_sy, by_sz;
  unsigned nvec;
  double F_H, dx3;
  double eta_hot, eta_cold, eta_max;  // eta = min(eta_hot T^-1.5, eta_cold T^0.5, eta_max), T in K
  float eta_Tlo, eta_Thi;             // eta(T) is at its cap in this band
  double ei_a, ei_mi, ei_me, Zstar, fs_q, fs_c;
};
template <typename R>
struct FieldK : FieldCommon {
  R F_curl, F_j, cdt, F_ohm, heat_den;
  R Tp_fac[4], ne_frac[4];  // per element
};
template <typename R>
inline FieldK<R> make_field(const Consts &K) {
  FieldK<R> f{};
  f.nx = K.nx;
  f.ny = K.ny;
  f.nz = K.nz;
  f.sy = K.nx + 1;
  f.sz = (K.nx + 1) * (K.ny + 1);
  f.physics = K.physics;
  f.n_solids = K.n_solids;
  f.by_sy = make_quotient((uint32_t)f.sy);
  f.by_sz = make_quotient((uint32_t)f.sz);
  f.nvec = (unsigned)K.nvec;
  f.F_H = K.F_H;
  f.dx3 = K.dx3;
  f.eta_hot = K.eta_hot_T;
  f.eta_cold = K.eta_cold_T;
  f.cold = K.eta_cold_T > 0.0;
  f.eta_max = K.eta_max;
  // the exact band's ends moved inwards by more than a float's rounding
  f.eta_Tlo = (float)(K.eta_Tlo * (1.0 + 5e-7));
  f.eta_Thi = (float)(K.eta_Thi * (1.0 - 5e-7));
  f.ei_a = K.ei_a;
  f.ei_mi = K.ei_mi;
  f.ei_me = K.ei_me;
  f.Zstar = K.Zstar;
  f.fs_q = K.fs_q;
  f.fs_c = K.fs_c;
  f.F_curl = R(K.F_curl);
  f.F_j = R(K.F_j);
  f.cdt = R(K.cdt_dx);
  f.F_ohm = R(K.F_ohm);
  f.heat_den = R(K.heat_den);
  for (int s = 0; s < 4; ++s) {
    f.Tp_fac[s] = R(K.Tp_fac_s[s]);
    f.ne_frac[s] = R(K.ne_frac[s]);
  }
  return f;
}

// message returned by hpic_last_error(NULL) (entry points without a context)
void set_global_error(const char *msg);

// fold one target's SI parameters into normalised kernel constants (laser may
// be NULL: a0 = 0, weight 1), and the resistivity eta(T) of Eqs. (A4)-(A6)
void fold(const hpic_target_desc &t, const hpic_run_params &r, const hpic_laser_desc *laser,
          Consts &K);
double eta_of(const Consts &K, double T);
// F_sigma of App. B at ion temperature Ti (K)
double fsigma_of(const Consts &K, double Ti);
// the injecting face cells of a Gaussian-envelope laser (empty otherwise)
std::vector<InjCell> injection_cells(const hpic_target_desc &t, const hpic_laser_desc &l);

// Launch shape of the single-target particle kernel: resident blocks per SM
// (it is launched as one persistent wave of sm_count times this many blocks)
// and threads per block (one deposit stage per warp).  FP32: three blocks of
// 384 threads, 36 warps at 56 registers with few spills; a block's twelve
// warps take consecutive slots, so their gathers share L1 lines.  (Against
// it: five blocks of 256 at 48 registers, 84 B of spills, 3.5 % slower; six
// of 192 at 56 registers 3.2 %; four of 288 1.2 %; two of 576 level.)  FP64:
// two blocks of 256.
enum PushMode {
  kPushPlain = 0,  // a plain step
  kPushKeys = 1,   // one that also computes the next sort's keys (KeyOut)
  kPushSort = 2    // one that also sorts (SortOut)
};
template <typename R>
constexpr int push_blocks_per_sm() { return sizeof(R) == 4 ? 3 : 2; }
template <typename R>
constexpr int push_threads() { return sizeof(R) == 4 ? 384 : 256; }
// Slots that fill less than kPushFewWaves such waves are pushed by as many
// warps in blocks of kPushFewThreads instead: the scheduler deals them out over
// all SMs, where the large blocks of a partial wave fill some SMs and leave the
// others idle.  k_push in us, large blocks -> 64 threads (32), gold 64^3, FP32:
// 1e5 electrons 24.1 -> 19.0 (19.4), 3e5 38.8 -> 33.9 (35.9), 8e5 68.5 -> 62.0
// (74.6), 1.5e6 107.7 -> 105.9; FP64: 2e4 66.7 -> 52.8 (49.8), 1e5 157 -> 147
// (145), 2e5 278 -> 252, 5e5 592 -> 562.  Beyond about eight waves the twelve
// warps of a large block gain more from the L1 lines that they share: 1e7 655
// (64 threads: 661), FP64 1e6 level.
constexpr int kPushFewThreads = 64, kPushFewWaves = 8;
// resident 256-thread blocks per SM of the field and heating kernels (their
// launch bounds); they are launched as one wave of sm_count times this many
// blocks (grid-stride over the nodes), so no partial second wave trails.  Four
// (64 registers) hold a node's loads all at once: against six (40 registers)
// the heating of 128^3 cells took 63 for 69 us, the field solve 23 for 25 us;
// three were level.
constexpr int kFieldBlocksPerSm = 4;
constexpr int kBatchFieldBlocksPerSm = 4;

// host transfers of the electron state (the C-ABI's read and load calls):
// live-slot compaction in storage order and FP64 <-> R conversion on the
// device; the arrays on the far side are x .. tau and ids (null: skipped)
struct ParticleOut {
  double *a[7];
  uint32_t *id;
};
struct ParticleIn {
  const double *a[7];
  const uint32_t *id;
};
long long xfer_chunks(long long n);  // chunk counts needed: xfer_chunks(n) + 1
void launch_live_scan(const uint32_t *id, long long n, uint32_t *cc, cudaStream_t st);
template <typename R>
void launch_read_out(PView<R> p, long long n, const uint32_t *cc, double dx, const ParticleOut &out,
                     cudaStream_t st);
template <typename R>
void launch_load_in(const ParticleIn &in, long long n, double dx, const int (&cells)[3],
                    int unbounded, PView<R> dst, int weighted, R w, unsigned *bad, int grid,
                    cudaStream_t st);
template <typename T>
void launch_scale_out(const T *src, long long n, double scale, double *out, int grid,
                      cudaStream_t st);

// allow the push kernels their shared-memory deposit stages (above the
// default 48 KB for FP64 and the batch); once per device, before any launch
cudaError_t prepare_push();
cudaError_t prepare_batch_push();
// Where a step that also sorts writes its electrons: an electron live at
// the start of the step goes to slot offsets[key] + rank (+ a shift: 0 for
// one target; a batch target's first slot minus its first offset) of dst,
// where the counting sort's key pass ran on that start-of-step state (key
// and rank of each slot) and its scan turned the counts into offsets; one
// that is absorbed or escapes leaves its slot there marked dead.
// dst.x == nullptr: the electrons stay in their slots.
template <typename R>
struct SortOut {
  PView<R> dst;
  const uint32_t *keys, *ranks, *offsets;
};

// The sort key pass folded into the step before a sort: each electron that
// survives the step gets, from its new state, the key of the cell it reaches
// `lead` cells per unit of u/gamma ahead (as the key pass computes it from
// the start of the sorting step) and its rank among its key's electrons
// (counts must be cleared before).  keys == nullptr: no keys.
template <typename R>
struct KeyOut {
  uint32_t *keys, *ranks, *counts;
  R lead;
};

template <typename R>
void launch_push(const Consts &K, PView<R> p, GView<R> g, const R *table, Counters *cnt,
                 TallyView tv, long long cap, int sm_count, cudaStream_t st,
                 const SortOut<R> &so, const KeyOut<R> &ko);
// What closes a step: the slots kept by a sort (kept: their count on the
// device, or NULL), the injected electrons and the clock.  The heating kernel
// does it where nothing comes after it, else launch_advance.
struct StepEnd {
  Counters *cnt;  // NULL: not here
  const uint32_t *kept;
  long long cap;
};
__device__ __forceinline__ void close_step(const StepEnd &end) {
  Counters *cnt = end.cnt;
  const long long c = cnt->inj_cnt;
  const long long n = (end.kept ? (long long)*end.kept : cnt->n) + c;
  cnt->n = n < end.cap ? n : end.cap;
  cnt->next_id += c;
  cnt->step += 1;
  cnt->inj_cnt = 0;
}
template <typename R>
void launch_inject(const Consts &K, PView<R> p, const StepEnd &end, TallyView tv, int grid,
                   cudaStream_t st);
void launch_advance(const StepEnd &end, cudaStream_t st);
// bulk seeding (two launches); mean kinetic energy in m_e c^2
template <typename R>
void launch_seed(const Consts &K, PView<R> p, Counters *cnt, long long cap, long long count,
                 double mean, TallyView tv, int grid, cudaStream_t st);

template <typename R>
void launch_efield(const Consts &K, GView<R> g, int grid, cudaStream_t st);
template <typename R>
void launch_bheat(const Consts &K, GView<R> g, TallyView tv, const StepEnd &end, int grid,
                  cudaStream_t st);

// counting sort by cell: keys/counts/offsets are scratch; electrons are keyed
// by the cell they reach `lead` steps ahead at their current velocity (0: the
// cell they are in); returns launches made
template <typename R>
int launch_sort(const Consts &K, PView<R> src, PView<R> dst, Counters *cnt, uint32_t *keys,
                uint32_t *counts, uint32_t *partials, int grid, cudaStream_t st, double lead);

// Lead (steps) of the sort that runs every `interval` steps: the cell each
// electron reaches halfway through the coming interval, so that the gathers
// at x^n and the deposits at x^{n+1} of the steps until the next sort find
// a warp's electrons in as few cells as the drift allows
inline double sort_lead(int interval) { return interval > 0 ? 0.5 * (interval + 1) : 0.0; }

// The counting sort folded into a step: keys, ranks (each slot's place among
// the slots of its key) and the scanned offsets of the electrons in p, keyed
// `lead` steps ahead; the step's push then writes each electron to its
// sorted slot (SortOut) and the end of the step sets the slot count to the
// electrons kept (StepEnd).  Return launches made.
template <typename R>
int launch_sort_keys(const Consts &K, PView<R> p, Counters *cnt, uint32_t *keys, uint32_t *ranks,
                     uint32_t *counts, uint32_t *partials, int grid, cudaStream_t st, double lead);

void launch_table(const Consts &K, double k_min, double E_max, double *t64, float *t32,
                  cudaStream_t st);

template <typename R>
void launch_live_energy(const Consts &K, PView<R> p, Counters *cnt, double *dst, int grid,
                        cudaStream_t st);
template <typename R>
void launch_field_energy(const Consts &K, GView<R> g, double *dst, int grid, cudaStream_t st);

// ---------------------------------------------------------------- batches
// One target of a batch as the batched kernels see it (a device array of
// these, one per target).
template <typename R>
struct BatchItem {
  Consts K;
  HotK<R> h;
  FieldK<R> f;
  GView<R> g;
  TallyView tv;
  Counters *cnt;
  long long off, cap;  // particle slots [off, off + cap) of the shared arrays
};

// device arrays shared by the batched kernels (n + 1 prefix sums over targets)
struct BatchDev {
  int n;                  // targets
  long long *wpref;       // warp-sized particle tasks, from the live counts
  long long *ipref;       // electrons injected in this step
  const long long *npref; // warp-sized (32-node) pieces of the vector grids
  const long long *kpref; // sort keys (each target's tile keys, then its dead bin)
  long long *sstart;      // sort: first sorted offset of each target (n entries)
  long long *snew;        // sort: slots kept per target (n entries)
};

// counts per step and per target: warp tasks and injections (one block)
template <typename R>
void launch_batch_plan(const BatchItem<R> *items, BatchDev d, cudaStream_t st);
// persistent particle kernel, sm_count * blocks_per_sm blocks; Krun: the
// run-wide constants (any target's Consts: those fields are common);
// single: every target is a single-element solid
template <typename R>
void launch_batch_push(const Consts &Krun, const BatchItem<R> *items, BatchDev d, PView<R> p,
                       const R *table, int sm_count, int blocks_per_sm, bool single,
                       cudaStream_t st, const SortOut<R> &so);
template <typename R>
void launch_batch_inject(const BatchItem<R> *items, BatchDev d, PView<R> p, bool sorted, int grid,
                         cudaStream_t st);
template <typename R>
void launch_batch_advance(const BatchItem<R> *items, BatchDev d, bool sorted, cudaStream_t st);
template <typename R>
void launch_batch_efield(const BatchItem<R> *items, BatchDev d, int grid, cudaStream_t st);
template <typename R>
void launch_batch_bheat(const BatchItem<R> *items, BatchDev d, int grid, cudaStream_t st);
// the cell sort of every target inside its own slots, folded into a step as
// for one target: keys, ranks and scan over the targets' concatenated key
// ranges, each target's first offset and kept slots (the step's plan must
// have run), then the push writes each electron to its sorted slot and the
// finish sets each target's slot count; return launches made
template <typename R>
int launch_batch_sort_keys(const BatchItem<R> *items, BatchDev d, PView<R> p, uint32_t *keys,
                           uint32_t *ranks, uint32_t *counts, uint32_t *partials,
                           long long nkeys_total, int grid, cudaStream_t st, double lead);
// counts summed per block of the scan; the partials scratch of a scan of m
// counts holds scan_partials(m) words
constexpr long long kScanTile = 4096;
constexpr long long scan_partials(long long m) { return (m + kScanTile - 1) / kScanTile + 1; }
// exclusive scan of counts[0, m) in place (partials: scratch of
// scan_partials(m) words); chained: it follows a kernel of the same call;
// returns launches made
int launch_scan(uint32_t *counts, long long m, uint32_t *partials, cudaStream_t st,
                bool chained = false);

}  // namespace hpic
