// Grid-side kernels of the hybrid-PIC step (arXiv 2107.01723):
//   k_efield : E = eta (curl B / mu0 - j_h) on edges, Eq. (A2), tangential E
//              zero on the walls (conducting boundary)
//   k_bheat  : B -= dt curl E on faces, Eq. (A3), fused with the background
//              heating dT = rho/(Z n_i C k_B), Eqs. (A7)-(A8), rho = Ohmic
//              eta j_h.j_h dt + ionisation heat, and eta(T), Eqs. (A4)-(A6)
//   sort     : counting sort of electrons by cell (GPU data layout)
//   k_table  : inverse-CDF bremsstrahlung table from the closed-form CDF
#include "fields.cuh"

namespace hpic {

template <typename R>
__global__ void __launch_bounds__(256, kFieldBlocksPerSm) k_efield(const FieldK<R> K, GView<R> g) {
  after_previous();
  for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < K.nvec; q += gridDim.x * blockDim.x)
    efield_node(K, g, q);
}

template <typename R>
__global__ void __launch_bounds__(256, kFieldBlocksPerSm)
k_bheat(const FieldK<R> K, GView<R> g, TallyView tv, const StepEnd end) {
  __shared__ WideSum<R> part[8];  // the warps' Ohmic sums
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  after_previous();
  // nothing in this kernel or after it in the step reads the counters
  if (end.cnt && blockIdx.x == 0 && threadIdx.x == 0) close_step(end);
  WideSum<R> ohm{};
  for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < K.nvec; q += gridDim.x * blockDim.x)
    ohm.add(bheat_node(K, g, q));
  ohm.over_warp();
  if (lane == 0) part[warp] = ohm;
  __syncthreads();
  if (warp == 0) {
    const double sum = warp_sum(lane < 8 ? part[lane].value() : 0.0);
    if (lane == 0 && sum != 0.0) atomicAdd(tv.tal + T_E_OHMIC, sum * K.dx3);
  }
}

// ---------------------------------------------------------------- batched field kernels
// The targets' nodes go in pieces of 32, a warp to a piece (prefix d.npref),
// so a warp's nodes are of one target; a warp walks its pieces in increasing
// order and keeps its target's constants and views in shared memory.
template <typename R>
struct FieldHot {
  FieldK<R> K;
  GView<R> g;
};

template <typename R>
__device__ __forceinline__ int enter_target(FieldHot<R> &w, const BatchItem<R> *items,
                                            const long long *pref, int t, long long piece) {
  int tn = t < 0 ? 0 : t;
  while (pref[tn + 1] <= piece) ++tn;
  if (tn != t) {  // warp-uniform
    static_assert(sizeof(FieldK<R>) % 4 == 0 && sizeof(GView<R>) % 4 == 0, "copied by words");
    __syncwarp();
    auto copy = [&](void *dst, const void *from, int bytes) {
      const uint32_t *a = static_cast<const uint32_t *>(from);
      uint32_t *b = static_cast<uint32_t *>(dst);
      for (int k = threadIdx.x & 31; k < bytes / 4; k += 32) b[k] = __ldg(a + k);
    };
    copy(&w.K, &items[tn].f, (int)sizeof(FieldK<R>));
    copy(&w.g, &items[tn].g, (int)sizeof(GView<R>));
    __syncwarp();
  }
  return tn;
}

template <typename R>
__global__ void __launch_bounds__(256, kBatchFieldBlocksPerSm)
k_batch_efield(const BatchItem<R> *items, BatchDev d) {
  extern __shared__ long long npref_s[];
  __shared__ FieldHot<R> hot[8];
  after_previous();
  for (int t = threadIdx.x; t <= d.n; t += blockDim.x) npref_s[t] = d.npref[t];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long N = npref_s[d.n];
  int t = -1;
  for (long long w = blockIdx.x * 8ll + warp; w < N; w += gridDim.x * 8ll) {
    t = enter_target(hot[warp], items, npref_s, t, w);
    const unsigned q = (unsigned)(w - npref_s[t]) * 32u + lane;
    if (q < hot[warp].K.nvec) efield_node(hot[warp].K, hot[warp].g, q);
  }
}

// A warp meets each target for a few pieces only (three of 7.9e6 cells in 16
// targets), so its sums over the lanes are many: they stay in FP32 parts, one of
// each warp and target, and become FP64 at the kernel's end, 8 lanes to a target.
// (16 targets: 133 us; with the sums made FP64 each time 171.  Each thread used to add
// its FP64 sum to its target's shared double, a compare-and-swap loop of up to 256
// threads on one address.)
template <typename R>
__global__ void __launch_bounds__(256, kBatchFieldBlocksPerSm)
k_batch_bheat(const BatchItem<R> *items, BatchDev d) {
  extern __shared__ long long npref_s[];
  __shared__ FieldHot<R> hot[8];
  WideSum<R> *part = reinterpret_cast<WideSum<R> *>(npref_s + d.n + 1);  // [n][8]
  after_previous();
  for (int t = threadIdx.x; t <= d.n; t += blockDim.x) npref_s[t] = d.npref[t];
  for (int t = threadIdx.x; t < 8 * d.n; t += blockDim.x) part[t] = WideSum<R>{};
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long N = npref_s[d.n];
  int t = -1;
  WideSum<R> ohm{};
  auto flush = [&]() {
    ohm.over_warp();
    if (lane == 0) part[t * 8 + warp] = ohm;
    ohm = WideSum<R>{};
  };
  for (long long w = blockIdx.x * 8ll + warp; w < N; w += gridDim.x * 8ll) {
    if (t >= 0 && npref_s[t + 1] <= w) flush();
    t = enter_target(hot[warp], items, npref_s, t, w);
    const unsigned q = (unsigned)(w - npref_s[t]) * 32u + lane;
    if (q < hot[warp].K.nvec) ohm.add(bheat_node(hot[warp].K, hot[warp].g, q));
  }
  if (t >= 0) flush();
  __syncthreads();
  for (int u = threadIdx.x; u < (8 * d.n + 31) / 32 * 32; u += blockDim.x) {  // whole warps
    double sum = u < 8 * d.n ? part[u].value() : 0.0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (u % 8 == 0 && sum != 0.0)
      atomicAdd(items[u / 8].tv.tal + T_E_OHMIC, sum * items[u / 8].f.dx3);
  }
}

// ---------------------------------------------------------------- counting sort
// Key of each slot: the tile key of the cell at x + lead (u/gamma), lead in
// cells per unit of u/gamma (0: the current cell), clamped to the grid.
template <typename R>
__global__ void __launch_bounds__(256)
k_sort_keys(const Consts K, PView<R> p, const Counters *cnt, uint32_t *keys, uint32_t *counts,
            R lead, uint32_t *ranks) {
  after_previous();
  const long long n = cnt->n;
  for (long long ip = blockIdx.x * (long long)blockDim.x + threadIdx.x; ip < n;
       ip += (long long)gridDim.x * blockDim.x) {
    uint32_t key = (uint32_t)K.nkeys;
    if (p.id[ip] != kDead) {
      R X = p.x[ip], Y = p.y[ip], Z = p.z[ip];
      if (lead != R(0)) {  // uniform over the launch
        const R ux = p.ux[ip], uy = p.uy[ip], uz = p.uz[ip];
        const R a = lead / m_sqrt(R(1) + ux * ux + uy * uy + uz * uz);
        X += a * ux;
        Y += a * uy;
        Z += a * uz;
      }
      int i = (int)m_floor(X), j = (int)m_floor(Y), k = (int)m_floor(Z);
      i = min(max(i, 0), K.nx - 1);
      j = min(max(j, 0), K.ny - 1);
      k = min(max(k, 0), K.nz - 1);
      key = tile_key(i, j, k, K.nti, K.ntj);
    }
    keys[ip] = key;
    if (ranks)  // uniform over the launch
      ranks[ip] = agg_inc(counts, key);
    else
      agg_inc(counts, key);
  }
}


// per-tile sums of counts[0, m)
__global__ void __launch_bounds__(1024) k_scan_tiles(const uint32_t *counts, long long m,
                                                     uint32_t *partials) {
  __shared__ uint32_t ws[32];
  after_previous();
  const long long base = (long long)blockIdx.x * kScanTile;
  uint32_t s = 0;
  for (int t = threadIdx.x; t < kScanTile; t += blockDim.x) {
    const long long q = base + t;
    if (q < m) s += counts[q];
  }
  s = __reduce_add_sync(0xffffffffu, s);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    uint32_t v = ws[threadIdx.x];
    v = __reduce_add_sync(0xffffffffu, v);
    if (threadIdx.x == 0) partials[blockIdx.x] = v;
  }
}

// exclusive scan of the tile sums in one block; total to partials[ntiles]
__global__ void __launch_bounds__(1024) k_scan_top(uint32_t *partials, int ntiles) {
  __shared__ uint32_t ws[32];
  __shared__ uint32_t carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  after_previous();
  for (int base = 0; base < ntiles; base += blockDim.x) {
    const int t = base + threadIdx.x;
    const uint32_t v = t < ntiles ? partials[t] : 0u;
    // inclusive warp scan
    uint32_t x = v;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    if (warp == 0) {
      uint32_t z = ws[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, z, o);
        if (lane >= o) z += y;
      }
      ws[lane] = z;
    }
    __syncthreads();
    const uint32_t incl = x + (warp > 0 ? ws[warp - 1] : 0u) + carry;
    if (t < ntiles) partials[t] = incl - v;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = incl;
    __syncthreads();
  }
  if (threadIdx.x == 0) partials[ntiles] = carry;
}

// exclusive scan within each tile plus its tile offset, in place
__global__ void __launch_bounds__(1024) k_scan_apply(uint32_t *counts, long long m,
                                                     const uint32_t *partials) {
  __shared__ uint32_t ws[32];
  __shared__ uint32_t carry;
  const long long base = (long long)blockIdx.x * kScanTile;
  after_previous();
  if (threadIdx.x == 0) carry = partials[blockIdx.x];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int off = 0; off < kScanTile; off += blockDim.x) {
    const long long q = base + off + threadIdx.x;
    const uint32_t v = q < m ? counts[q] : 0u;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    if (warp == 0) {
      uint32_t z = ws[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, z, o);
        if (lane >= o) z += y;
      }
      ws[lane] = z;
    }
    __syncthreads();
    const uint32_t incl = x + (warp > 0 ? ws[warp - 1] : 0u) + carry;
    if (q < m) counts[q] = incl - v;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = incl;
    __syncthreads();
  }
}

// The same of a short range (up to kScanShort) by one block: a thread takes
// `per` consecutive counts, all loaded before the block's one scan.
constexpr int kScanPer = 16;  // counts per thread at most, a multiple of 4
constexpr long long kScanShort = 1024 * kScanPer;

__global__ void __launch_bounds__(1024) k_scan_short(uint32_t *counts, int m) {
  __shared__ uint32_t ws[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = ((m + 1023) / 1024 + 3) & ~3, first = (int)threadIdx.x * per;
  after_previous();
  uint4 v[kScanPer / 4];
  uint32_t s = 0;
#pragma unroll
  for (int q = 0; q < kScanPer / 4; ++q) {
    const int at = first + 4 * q;
    v[q] = make_uint4(0u, 0u, 0u, 0u);
    if (4 * q < per) {
      if (at + 3 < m) {
        v[q] = *reinterpret_cast<const uint4 *>(counts + at);
      } else {
        if (at < m) v[q].x = counts[at];
        if (at + 1 < m) v[q].y = counts[at + 1];
        if (at + 2 < m) v[q].z = counts[at + 2];
      }
    }
    s += v[q].x + v[q].y + v[q].z + v[q].w;
  }
  uint32_t x = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) ws[warp] = x;
  __syncthreads();
  uint32_t z = ws[lane];  // every warp scans the warps' sums for itself
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, z, o);
    if (lane >= o) z += y;
  }
  const uint32_t before = __shfl_sync(0xffffffffu, z, warp ? warp - 1 : 0);
  uint32_t run = (warp ? before : 0u) + x - s;
#pragma unroll
  for (int q = 0; q < kScanPer / 4; ++q) {
    const int at = first + 4 * q;
    if (4 * q >= per) break;
    const uint4 o = make_uint4(run, run + v[q].x, run + v[q].x + v[q].y, run + v[q].x + v[q].y + v[q].z);
    run = o.w + v[q].w;
    if (at + 3 < m) {
      *reinterpret_cast<uint4 *>(counts + at) = o;
    } else {
      if (at < m) counts[at] = o.x;
      if (at + 1 < m) counts[at + 1] = o.y;
      if (at + 2 < m) counts[at + 2] = o.z;
    }
  }
}

template <typename R>
__global__ void __launch_bounds__(256)
k_sort_scatter(const Consts K, PView<R> src, PView<R> dst, const Counters *cnt,
               const uint32_t *keys, uint32_t *offsets) {
  const long long n = cnt->n;
  for (long long ip = blockIdx.x * (long long)blockDim.x + threadIdx.x; ip < n;
       ip += (long long)gridDim.x * blockDim.x) {
    const uint32_t key = keys[ip];
    if (key >= (uint32_t)K.nkeys) continue;
    const uint32_t q = agg_inc(offsets, key);
    dst.x[q] = src.x[ip];
    dst.y[q] = src.y[ip];
    dst.z[q] = src.z[ip];
    dst.ux[q] = src.ux[ip];
    dst.uy[q] = src.uy[ip];
    dst.uz[q] = src.uz[ip];
    dst.tau[q] = src.tau[ip];
    if (K.weighted) dst.w[q] = src.w[ip];
    dst.id[q] = src.id[ip];
  }
}

// live count = exclusive offset of the dead bin (the scatter never touches it)
__global__ void k_sort_finish(Counters *cnt, const uint32_t *offsets, long long ncell) {
  if (threadIdx.x == 0 && blockIdx.x == 0) cnt->n = offsets[ncell];
}

// ---------------------------------------------------------------- photon table
// Row i: eps_i = k_min (E_max/k_min)^(i/(rows-1)); column j: the photon
// energy k with CDF(k/eps_i) = j/(cols-1), where CDF is the normalised
// integral of s(u)/u, s(u) = (4/3)(1-u) + u^2, from u0 = k_min/eps to u,
// stored as the log-ratio w = ln(eps_i/k) / ln(eps_i/k_min) (the sampler
// subtracts k from eps through it without cancellation).  Solved by
// Newton's method on y = ln u (dG/dy = s(e^y)) inside a bracket.
__global__ void k_table(int rows, int cols, double k_min, double E_max, double *t64, float *t32) {
  const long long nt = (long long)rows * cols;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < nt;
       q += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(q / cols), j = (int)(q - (long long)i * cols);
    const double r = (double)j / (double)(cols - 1);
    // w = ln(eps/k) / ln(eps/k_min): 1 at k = k_min, 0 at k = eps
    double w;
    if (i == 0 || j == 0 || j == cols - 1) {
      w = (i == 0) ? 1.0 - r : (j == 0 ? 1.0 : 0.0);
    } else {
      const double lu0 = ((double)i / (double)(rows - 1)) * -log(E_max / k_min);  // ln u0 < 0
      const double u0 = exp(lu0);
      // G(y) = (4/3)(y - lu0 - (e^y - u0)) + (e^{2y} - u0^2)/2, target r G(0)
      const double G1 = (4.0 / 3.0) * (-lu0 - (1.0 - u0)) + 0.5 * (1.0 - u0 * u0);
      const double target = r * G1;
      double lo = lu0, hi = 0.0, y = lu0 + r * (-lu0);
      for (int it = 0; it < 100; ++it) {
        const double e = exp(y);
        const double Gy = (4.0 / 3.0) * (y - lu0 - (e - u0)) + 0.5 * (e * e - u0 * u0) - target;
        if (Gy < 0.0) lo = y; else hi = y;
        const double dG = (4.0 / 3.0) * (1.0 - e) + e * e;
        double yn = y - Gy / dG;
        if (!(yn > lo && yn < hi)) yn = 0.5 * (lo + hi);
        if (fabs(yn - y) < 1e-16 * fabs(lu0)) { y = yn; break; }
        y = yn;
      }
      w = y / lu0;  // y = ln(k/eps)
    }
    t64[q] = w;
    t32[q] = (float)w;
  }
}

// ---------------------------------------------------------------- read-time sums
template <typename R>
__global__ void __launch_bounds__(256)
k_live_energy(const Consts K, PView<R> p, const Counters *cnt, double *dst) {
  __shared__ double smem[32];
  const long long n = cnt->n;
  double e = 0.0;
  for (long long ip = blockIdx.x * (long long)blockDim.x + threadIdx.x; ip < n;
       ip += (long long)gridDim.x * blockDim.x) {
    if (p.id[ip] == kDead) continue;
    // (the shared weight comes in at the end)
    const double ux = p.ux[ip], uy = p.uy[ip], uz = p.uz[ip];
    double gam;
    const double k = kinetic_near(ux * ux + uy * uy + uz * uz, gam);
    e = K.weighted ? fma((double)p.w[ip], k, e) : e + k;
  }
  const double v[1] = {K.weighted ? e : e * K.w};
  const int slot[1] = {0};
  block_flush<1>(v, slot, dst, smem);
}

template <typename R>
__global__ void __launch_bounds__(256) k_field_energy(const Consts K, GView<R> g, double *dst) {
  __shared__ double smem[32];
  double e = 0.0;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < K.nvec;
       q += (long long)gridDim.x * blockDim.x) {
    for (int c = 0; c < 3; ++c) {
      const double b = g.B[c][q];
      e += b * b;
    }
  }
  const double v[1] = {e};
  const int slot[1] = {0};
  block_flush<1>(v, slot, dst, smem);
}

// ---------------------------------------------------------------- launchers
template <typename R>
void launch_efield(const Consts &K, GView<R> g, int grid, cudaStream_t st) {
  launch_chained(k_efield<R>, grid, 256, 0, st, make_field<R>(K), g);
}

template <typename R>
void launch_bheat(const Consts &K, GView<R> g, TallyView tv, const StepEnd &end, int grid,
                  cudaStream_t st) {
  launch_chained(k_bheat<R>, grid, 256, 0, st, make_field<R>(K), g, tv, end);
}

// Up to kScanShort counts one block scans: one launch for three.  (8e3 counts
// of five small targets: 3.1 us, for three kernels of 7.4 us and their gaps;
// 32769 counts of 32^3 cells in 36 per thread: 8.3 us, no gain.)
int launch_scan(uint32_t *counts, long long m, uint32_t *partials, cudaStream_t st, bool chained) {
  if (m <= kScanShort) {
    if (chained) launch_chained(k_scan_short, 1, 1024, 0, st, counts, (int)m);
    else k_scan_short<<<1, 1024, 0, st>>>(counts, (int)m);
    return 1;
  }
  const int ntiles = (int)((m + kScanTile - 1) / kScanTile);
  if (chained) launch_chained(k_scan_tiles, ntiles, 1024, 0, st, counts, m, partials);
  else k_scan_tiles<<<ntiles, 1024, 0, st>>>(counts, m, partials);
  launch_chained(k_scan_top, 1, 1024, 0, st, partials, ntiles);
  launch_chained(k_scan_apply, ntiles, 1024, 0, st, counts, m, partials);
  return 3;
}

template <typename R>
int launch_sort(const Consts &K, PView<R> src, PView<R> dst, Counters *cnt, uint32_t *keys,
                uint32_t *counts, uint32_t *partials, int grid, cudaStream_t st, double lead) {
  const long long m = K.nkeys + 1;
  cudaMemsetAsync(counts, 0, m * sizeof(uint32_t), st);
  k_sort_keys<R><<<grid, 256, 0, st>>>(K, src, cnt, keys, counts, R(lead * K.cdt_dx), nullptr);
  const int launches = launch_scan(counts, m, partials, st);
  k_sort_scatter<R><<<grid, 256, 0, st>>>(K, src, dst, cnt, keys, counts);
  k_sort_finish<<<1, 32, 0, st>>>(cnt, counts, K.nkeys);
  return 3 + launches;
}

template <typename R>
int launch_sort_keys(const Consts &K, PView<R> p, Counters *cnt, uint32_t *keys, uint32_t *ranks,
                     uint32_t *counts, uint32_t *partials, int grid, cudaStream_t st, double lead) {
  const long long m = K.nkeys + 1;
  cudaMemsetAsync(counts, 0, m * sizeof(uint32_t), st);
  k_sort_keys<R><<<grid, 256, 0, st>>>(K, p, cnt, keys, counts, R(lead * K.cdt_dx), ranks);
  return 1 + launch_scan(counts, m, partials, st, true);
}

void launch_table(const Consts &K, double k_min, double E_max, double *t64, float *t32,
                  cudaStream_t st) {
  const long long nt = (long long)K.t_rows * K.t_cols;
  const int grid = (int)((nt + 255) / 256);
  k_table<<<grid, 256, 0, st>>>(K.t_rows, K.t_cols, k_min, E_max, t64, t32);
}

template <typename R>
void launch_batch_efield(const BatchItem<R> *items, BatchDev d, int grid, cudaStream_t st) {
  launch_chained(k_batch_efield<R>, grid, 256, (d.n + 1) * sizeof(long long), st, items, d);
}

template <typename R>
void launch_batch_bheat(const BatchItem<R> *items, BatchDev d, int grid, cudaStream_t st) {
  const size_t sm = (d.n + 1) * sizeof(long long) + 8 * d.n * sizeof(WideSum<R>);
  launch_chained(k_batch_bheat<R>, grid, 256, sm, st, items, d);
}

template <typename R>
void launch_live_energy(const Consts &K, PView<R> p, Counters *cnt, double *dst, int grid,
                        cudaStream_t st) {
  k_live_energy<R><<<grid, 256, 0, st>>>(K, p, cnt, dst);
}

template <typename R>
void launch_field_energy(const Consts &K, GView<R> g, double *dst, int grid, cudaStream_t st) {
  k_field_energy<R><<<grid, 256, 0, st>>>(K, g, dst);
}

// ---------------------------------------------------------------- host transfers
// Reading the electrons out: the live slots in storage order, converted to
// double with a scale.  Slots go in chunks of kXferChunk: the live count of
// each chunk, an exclusive scan of the chunk counts, then the arrays written
// at the compacted positions.
constexpr int kXferChunk = 2048;

__global__ void __launch_bounds__(256) k_live_counts(const uint32_t *id, long long n,
                                                     uint32_t *cc) {
  __shared__ uint32_t ws[8];
  const long long base = (long long)blockIdx.x * kXferChunk + threadIdx.x * 8;
  uint32_t c = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) c += (base + k < n && id[base + k] != kDead) ? 1u : 0u;
  c = __reduce_add_sync(0xffffffffu, c);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t t = 0;
    for (int w = 0; w < 8; ++w) t += ws[w];
    cc[blockIdx.x] = t;
  }
}

// exclusive scan of cc[0, nb) in one block; the total goes to cc[nb]
__global__ void __launch_bounds__(1024) k_scan_chunks(uint32_t *cc, long long nb) {
  __shared__ uint32_t part[1024];
  const long long per = (nb + 1023) / 1024;
  const long long b0 = threadIdx.x * per, b1 = b0 + per < nb ? b0 + per : nb;
  uint32_t s = 0;
  for (long long b = b0; b < b1; ++b) s += cc[b];
  part[threadIdx.x] = s;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {  // inclusive scan of the slice sums
    const uint32_t v = threadIdx.x >= o ? part[threadIdx.x - o] : 0u;
    __syncthreads();
    part[threadIdx.x] += v;
    __syncthreads();
  }
  uint32_t run = threadIdx.x ? part[threadIdx.x - 1] : 0u;
  for (long long b = b0; b < b1; ++b) {
    const uint32_t c = cc[b];
    cc[b] = run;
    run += c;
  }
  if (threadIdx.x == 1023) cc[nb] = part[1023];
}

// out[q][rank] = array q of slot i, converted to double, for the live slots i
// of this block's chunk, rank = the slot's place among the live slots (a
// warp's 32 slots at a time, so that loads and stores run along the arrays);
// null outputs are skipped.  The outputs may be page-locked host memory: the
// stores then cross to the host at once, all arrays in one launch.  (Bound by
// the link: 1e7 electrons, 600 MB, 3.6 ms through one copy per array before.)
template <typename R>
__global__ void __launch_bounds__(256) k_read_out(const PView<R> p, long long n, const uint32_t *cc,
                                                  double dx, const ParticleOut out) {
  __shared__ uint32_t ws[8];
  constexpr int kRounds = kXferChunk / 256;  // of 32 slots per warp
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long base = (long long)blockIdx.x * kXferChunk + warp * (32 * kRounds) + lane;
  uint32_t id[kRounds], live = 0, total = 0;
#pragma unroll
  for (int k = 0; k < kRounds; ++k) {
    const long long i = base + 32 * k;
    id[k] = i < n ? p.id[i] : kDead;
    if (id[k] != kDead) live |= 1u << k;
    total += __popc(__ballot_sync(0xffffffffu, id[k] != kDead));
  }
  if (lane == 0) ws[warp] = total;
  __syncthreads();
  long long first = cc[blockIdx.x];
  for (int w = 0; w < warp; ++w) first += ws[w];
  const R *src[7] = {p.x, p.y, p.z, p.ux, p.uy, p.uz, p.tau};
#pragma unroll
  for (int k = 0; k < kRounds; ++k) {
    const bool on = (live >> k) & 1u;
    const uint32_t mask = __ballot_sync(0xffffffffu, on);
    const long long i = base + 32 * k, q = first + __popc(mask & ((1u << lane) - 1u));
    if (on) {
#pragma unroll
      for (int a = 0; a < 7; ++a)
        if (out.a[a]) out.a[a][q] = (double)src[a][i] * (a < 3 ? dx : 1.0);
      if (out.id) out.id[q] = id[k];
    }
    first += __popc(mask);
  }
}

// Loading electrons in: the arrays (device memory, or page-locked host memory
// read across the link) checked and converted in one pass, where a pass to
// check and one to convert took positions and ids across twice: 1e7 electrons
// 5.3 -> 3.0 ms (600 MB, 200 GB/s; the link's bandwidth).  Counts positions
// outside [0, hi] after division by dx (any non-finite value with unbounded)
// and reserved ids.  The division is made only where the product with 1/dx
// does not decide: within 1e-12 of a wall, or below zero.
template <typename R>
__global__ void __launch_bounds__(256) k_load_in(const ParticleIn in, long long n, double dx,
                                                 double inv_dx, int nx, int ny, int nz,
                                                 int unbounded, PView<R> dst, int weighted, R w,
                                                 unsigned *bad) {
  unsigned b = 0;
  R *to[7] = {dst.x, dst.y, dst.z, dst.ux, dst.uy, dst.uz, dst.tau};
  const double hi[3] = {(double)nx, (double)ny, (double)nz};
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    double v[7];
    uint32_t id = 0;
#pragma unroll
    for (int a = 0; a < 7; ++a)
      if (in.a[a]) v[a] = in.a[a][i];
    if (in.id) id = in.id[i];
#pragma unroll
    for (int a = 0; a < 7; ++a) {
      if (!in.a[a]) continue;
      if (a < 3) {
        const double q = v[a] * inv_dx;
        if (!(q > 0.0 && q < hi[a] * (1.0 - 1e-12))) {
          const double X = v[a] / dx;
          b += (unbounded ? !isfinite(X) : !(X >= 0.0 && X <= hi[a])) ? 1u : 0u;
        }
        to[a][i] = (R)q;
      } else {
        to[a][i] = (R)v[a];
      }
    }
    if (in.id) {
      b += id == kDead ? 1u : 0u;
      dst.id[i] = id;
      if (weighted) dst.w[i] = w;
    }
  }
  if (b) atomicAdd(bad, b);
}

// a grid out: scaled to SI in double (in host loops before: four grids of 128^3
// read in 3.7-5.4 ms, now 0.5 ms)
template <typename T>
__global__ void __launch_bounds__(256) k_scale_out(const T *src, long long n, double scale,
                                                   double *out) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    out[i] = (double)src[i] * scale;
}

long long xfer_chunks(long long n) { return (n + kXferChunk - 1) / kXferChunk; }

void launch_live_scan(const uint32_t *id, long long n, uint32_t *cc, cudaStream_t st) {
  const long long nb = xfer_chunks(n);
  if (nb > 0) k_live_counts<<<(unsigned)nb, 256, 0, st>>>(id, n, cc);
  k_scan_chunks<<<1, 1024, 0, st>>>(cc, nb);
}

template <typename R>
void launch_read_out(PView<R> p, long long n, const uint32_t *cc, double dx, const ParticleOut &out,
                     cudaStream_t st) {
  const long long nb = xfer_chunks(n);
  if (nb > 0) k_read_out<R><<<(unsigned)nb, 256, 0, st>>>(p, n, cc, dx, out);
}

template <typename R>
void launch_load_in(const ParticleIn &in, long long n, double dx, const int (&cells)[3],
                    int unbounded, PView<R> dst, int weighted, R w, unsigned *bad, int grid,
                    cudaStream_t st) {
  k_load_in<R><<<grid, 256, 0, st>>>(in, n, dx, 1.0 / dx, cells[0], cells[1], cells[2], unbounded,
                                     dst, weighted, w, bad);
}

template <typename T>
void launch_scale_out(const T *src, long long n, double scale, double *out, int grid,
                      cudaStream_t st) {
  k_scale_out<T><<<grid, 256, 0, st>>>(src, n, scale, out);
}

#define HPIC_INST(R)                                                                          \
  template void launch_efield<R>(const Consts &, GView<R>, int, cudaStream_t);                \
  template void launch_bheat<R>(const Consts &, GView<R>, TallyView, const StepEnd &, int,    \
                                cudaStream_t);                                                \
  template int launch_sort<R>(const Consts &, PView<R>, PView<R>, Counters *, uint32_t *,     \
                              uint32_t *, uint32_t *, int, cudaStream_t, double);             \
  template int launch_sort_keys<R>(const Consts &, PView<R>, Counters *, uint32_t *, uint32_t *, \
                                   uint32_t *, uint32_t *, int, cudaStream_t, double);        \
  template void launch_live_energy<R>(const Consts &, PView<R>, Counters *, double *, int,    \
                                      cudaStream_t);                                          \
  template void launch_field_energy<R>(const Consts &, GView<R>, double *, int, cudaStream_t); \
  template void launch_batch_efield<R>(const BatchItem<R> *, BatchDev, int, cudaStream_t);     \
  template void launch_batch_bheat<R>(const BatchItem<R> *, BatchDev, int, cudaStream_t);     \
  template void launch_read_out<R>(PView<R>, long long, const uint32_t *, double,             \
                                   const ParticleOut &, cudaStream_t);                        \
  template void launch_load_in<R>(const ParticleIn &, long long, double, const int (&)[3],    \
                                  int, PView<R>, int, R, unsigned *, int, cudaStream_t);      \
  template void launch_scale_out<R>(const R *, long long, double, double *, int, cudaStream_t);
HPIC_INST(float)
HPIC_INST(double)
#undef HPIC_INST

}  // namespace hpic
