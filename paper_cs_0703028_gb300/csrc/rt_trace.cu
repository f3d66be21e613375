// Monte-Carlo ray tracing through finite volumes (Section 3, Fig. ray) and the
// final tally reduction.
//   k_walk_setup: per cell, the binary32 temperature bracket (k, frac) of the kappa table,
//                 the density scale (p x)/(p_ref x_ref) and T, and an 8-byte step record; the
//                 walk's copy of the table, {kappa_k, kappa_k+1} per (wavenumber, node), so a
//                 step's interpolation is one 8-byte load, or wavenumber-major.
//   k_walk      : per ray, Philox draws -> emission cell, wavenumber, position,
//                 isotropic direction -> cell-by-cell walk with Beer-Lambert
//                 attenuation (Eq. I, first term), binary64 atomic deposits;
//                 persistent warps refilled by ballot.
//   k_reduce / k_final : deterministic two-pass binary64 sum of the absorbed
//                 power and the energy balance.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "rt_common.cuh"
#include "rt_walk.cuh"

namespace rt {

rt_status validate_spec(const rt_spectral *s);

namespace {

constexpr int kWalkThreads = 256, kWalkBlocks = 4;  // resident blocks per SM
constexpr int kReduceBlocks = 256;

// Persistent walk: each warp owns a contiguous range of rays.  Lanes step their
// own rays; when half of the warp's lanes are idle (ballot), the idle lanes take
// the warp's next rays together, so ray set-up and stepping stay converged.
constexpr int kRefillIdleDefault = 16;
constexpr int kWalkUnroll = 8;  // steps per pass of the walk loop
constexpr int kPassLanes = 14;  // lanes for which a pass with newly loaded rays goes on

// ---------------------------------------------------------------- grouping rays by wavenumber band
constexpr int kBandHist = 8192;  // bands counted in a shared-memory histogram (else global atomics)

// rays per band (counts zeroed before the launch)
__global__ void k_band_count(WalkParams W, int band_pts, long long n_bands, unsigned long long *__restrict__ counts) {
  __shared__ unsigned int hist[kBandHist];
  const bool local = n_bands <= kBandHist;
  if (local)
    for (int b = threadIdx.x; b < (int)n_bands; b += blockDim.x) hist[b] = 0u;
  __syncthreads();
  for (unsigned long long rr = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; rr < W.n_rays;
       rr += (unsigned long long)gridDim.x * blockDim.x) {
    const int b = ray_nu_index(W, rr) / band_pts;
    if (local) atomicAdd(&hist[b], 1u);
    else atomicAdd(&counts[b], 1ull);
  }
  __syncthreads();
  if (local)
    for (int b = threadIdx.x; b < (int)n_bands; b += blockDim.x)
      if (hist[b]) atomicAdd(&counts[b], (unsigned long long)hist[b]);
}

// band_start and item_start (exclusive prefix sums over the bands; one block), the
// scatter cursors; counts == nullptr: one band holding all n_rays rays
__global__ void k_band_plan(const unsigned long long *__restrict__ counts, long long n_bands,
                            unsigned long long n_rays, long long chunk, long long *__restrict__ band_start,
                            long long *__restrict__ item_start, int *__restrict__ item_band,
                            unsigned long long *__restrict__ cursor) {
  __shared__ long long sc[1024], si[1024];
  const int t = threadIdx.x, nt = blockDim.x;
  // each thread sums a contiguous run of bands, then the runs are scanned
  const long long per = (n_bands + nt - 1) / nt;
  const long long b0 = min(n_bands, (long long)t * per), b1 = min(n_bands, b0 + per);
  long long c = 0, it = 0;
  for (long long b = b0; b < b1; ++b) {
    const long long k = counts ? (long long)counts[b] : (long long)n_rays;
    c += k;
    it += (k + chunk - 1) / chunk;
  }
  sc[t] = c;
  si[t] = it;
  __syncthreads();
  for (int o = 1; o < nt; o <<= 1) {  // inclusive scan of the runs (Hillis-Steele)
    const long long a = t >= o ? sc[t - o] : 0, bi = t >= o ? si[t - o] : 0;
    __syncthreads();
    sc[t] += a;
    si[t] += bi;
    __syncthreads();
  }
  long long pc = sc[t] - c, pi = si[t] - it;
  for (long long b = b0; b < b1; ++b) {
    const long long k = counts ? (long long)counts[b] : (long long)n_rays;
    band_start[b] = pc;
    item_start[b] = pi;
    if (cursor) cursor[b] = (unsigned long long)pc;
    pc += k;
    for (const long long end = pi + (k + chunk - 1) / chunk; pi < end; ++pi)
      if (item_band) item_band[pi] = (int)b;
  }
  if (t == nt - 1) {
    band_start[n_bands] = sc[t];
    item_start[n_bands] = si[t];
  }
}

// ray offsets into their band's run of order (order within a band: arrival order)
__global__ void k_band_scatter(WalkParams W, int band_pts, unsigned long long *__restrict__ cursor,
                               uint32_t *__restrict__ order) {
  for (unsigned long long rr = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; rr < W.n_rays;
       rr += (unsigned long long)gridDim.x * blockDim.x) {
    const int b = ray_nu_index(W, rr) / band_pts;
    order[atomicAdd(&cursor[b], 1ull)] = (uint32_t)rr;
  }
}

}  // namespace

int g_walk_blocks = 5;   // kept for rt_get_tuning only: no launch reads it
int g_walk_refill = 16;  // idle lanes that trigger a refill (12 or 16)
// Rays grouped by wavenumber only when asked for (2; 0 and 1 never): the counting passes
// cost more than the shared table rows save.  Off / on: 1e7 rays of the opaque 32^3 box
// 0.39 / 0.87 ms; 4e8 of the opaque 128^3 box 15.9 / 30.0 ms; 2e7 rays of a thin gas there
// 6.7 / 10.1 ms; thin gas with a 410 MB table and 1e8 rays (62 a wavenumber) 32.5 / 48.8 ms.
int g_walk_group = 0;

namespace {

constexpr int kSetupThreads = 256;
constexpr int kPairRows = 64;
// Blocks of the walk's copy of a T-major table: bx over 32-wavenumber slices, by over nodes.
// Layout 1, [nT][n_nu] -> [n_nu][nT]: tiles of kPairRows nodes x 32 wavenumbers, eight loads a
// thread in flight (64 nodes x 300k wavenumbers 28.6 us; 32 x 32 tiles, four loads, 56 here and 42 in
// a kernel of their own).  Layout 2, node pairs out[j (nT - 1) + k] =
// {in[k][j], in[k + 1][j]}: each block stages kPairRows + 1 rows of 32 wavenumbers and writes
// the pairs wavenumber by wavenumber.
template <int LAYOUT>
__device__ __forceinline__ void table_block(const float *__restrict__ in, int nT, long long n_nu,
                                            float *__restrict__ out, long long bx, int by) {
  __shared__ float t[kPairRows + 1][33];
  const long long j0 = bx * 32;
  if (LAYOUT == 2) {
    const int k0 = by * kPairRows;
    const int rows = min(kPairRows + 1, nT - k0);
    for (int idx = threadIdx.x; idx < rows * 32; idx += kSetupThreads) {
      const int r = idx >> 5, c = idx & 31;
      if (j0 + c < n_nu) t[r][c] = in[(long long)(k0 + r) * n_nu + j0 + c];
    }
    __syncthreads();
    const int np = rows - 1;
    for (int idx = threadIdx.x; idx < np * 32; idx += kSetupThreads) {
      const int c = idx / np, r = idx - c * np;
      if (j0 + c < n_nu)
        reinterpret_cast<float2 *>(out)[(j0 + c) * (long long)(nT - 1) + k0 + r] = make_float2(t[r][c], t[r + 1][c]);
    }
  } else {
    const int r0 = by * kPairRows, x = threadIdx.x & 31;
    if (nT == 1) {  // the table itself
      if (threadIdx.x < 32 && j0 + x < n_nu) out[j0 + x] = in[j0 + x];
      return;
    }
#pragma unroll
    for (int q = 0; q < kPairRows; q += kSetupThreads / 32) {
      const int i = q + (threadIdx.x >> 5);
      if (r0 + i < nT && j0 + x < n_nu) t[i][x] = in[(long long)(r0 + i) * n_nu + j0 + x];
    }
    __syncthreads();
    const int r = threadIdx.x % kPairRows;
#pragma unroll
    for (int q = 0; q < 32; q += kSetupThreads / kPairRows) {
      const int c = q + threadIdx.x / kPairRows;
      if (r0 + r < nT && j0 + c < n_nu) out[(j0 + c) * nT + r0 + r] = t[r][c];
    }
  }
}

template <int LAYOUT>
__global__ void __launch_bounds__(kSetupThreads)
k_walk_table(const float *__restrict__ in, int nT, long long n_nu, float *__restrict__ out) {
  table_block<LAYOUT>(in, nT, n_nu, out, blockIdx.x, blockIdx.y);
}

// What a step of the table walk needs of a cell, in 8 bytes: its position in the node grid
// (bracket + fraction, their sum exact: the fraction is u - floor u, or 0 or 1 at the ends)
// and its density scale.  The walk of a thin gas is bound by the L1 misses it sends to L2 (one
// request per missed 32-byte sector or deposit, 79 % of their peak rate), and four cells
// share a sector instead of two: 8e6 rays of a thin gas in a 75 x 52 x 61 box 2.29 -> 2.24 ms,
// 4e8 of the opaque 128^3 box 14.2 -> 14.0.
__device__ __forceinline__ float2 step_cell(const float4 cd) {
  return make_float2(__fadd_rn((float)__float_as_int(cd.w), cd.x), cd.y);
}
// back to {fraction, scale, -, bracket}; ktop = max(nT - 2, 0)
__device__ __forceinline__ float4 step_bracket(const float2 c, float ktop) {
  const float fl = fminf(floorf(c.x), ktop);
  return make_float4(__fsub_rn(c.x, fl), c.y, 0.0f, __int_as_float((int)fl));
}

// The set-up of a table walk in one launch: the first cell_blocks blocks prepare the cells
// (whole records for the emission, then step records), the others copy the table.
template <int LAYOUT>
__global__ void __launch_bounds__(kSetupThreads)
k_walk_setup(const float *__restrict__ T, const float *__restrict__ p, const float *__restrict__ x, CellParams C,
             float4 *__restrict__ cells, float2 *__restrict__ step_cells, uint32_t *status, unsigned cell_blocks,
             const float *__restrict__ in, int nT, long long n_nu, unsigned slices, float *__restrict__ out) {
  const unsigned b = blockIdx.x;
  if (b < cell_blocks) {
    const long long c = (long long)b * kSetupThreads + threadIdx.x;
    if (c < C.ncells) {
      const float4 cd = cell_prep_one(T, p, x, c, C, status);
      cells[c] = cd;
      step_cells[c] = step_cell(cd);
    }
    return;
  }
  const unsigned q = b - cell_blocks, y = q / slices;
  table_block<LAYOUT>(in, nT, n_nu, out, q - y * slices, (int)y);
}

// Four blocks of 64 registers: at five of 48 the walk spills, and more resident rays share
// one L1 (8e6 rays of a thin gas in a 75 x 52 x 61 box: 2.29 ms against 2.61 ms; 4e8 rays of
// the opaque 128^3 box, where it matters least: 15.9 ms against 16.9 ms).
// FEW: a tally of at most kFewCells cells is kept per block in shared memory and added to the
// caller's at the end; otherwise the rays' deposits queue on few addresses of L2.  Whole trace,
// global / shared tally: 1e5 rays of a 64-cell slab 64 / 42 us; 3e6 rays of a thin gas in 8^3
// cells 1049 / 260 us, 12^3 603 / 296, 16^3 561 / 343; 1e5 rays of an opaque gas in 16^3 49 / 54
// (zeroing and adding 4096 cells a block), so the line lies between 12^3 and 16^3.
constexpr int kFewCells = 2048;
template <bool REC, int TAB, int REFILL, bool FEW = false>
__global__ void __launch_bounds__(kWalkThreads, kWalkBlocks)
k_walk(const float4 *__restrict__ cells, const float2 *__restrict__ step_cells, const float *__restrict__ tab,
       const uint32_t *__restrict__ order, WalkParams W, double *__restrict__ absorbed, double *__restrict__ scalars,
       unsigned long long *__restrict__ steps_out, uint32_t *status, RecordPtrs rec) {
  const int lane = threadIdx.x & 31;
  const unsigned long long nwarps = (unsigned long long)gridDim.x * (blockDim.x >> 5);
  const unsigned long long wid = (unsigned long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  unsigned long long next = W.n_rays * wid / nwarps;
  const unsigned long long last = W.n_rays * (wid + 1) / nwarps;
  const bool record = REC;
  __shared__ double s_tally[FEW ? kFewCells : 1];
  if (FEW)
    for (int c = threadIdx.x; c < (int)W.ncells; c += kWalkThreads) s_tally[c] = 0.0;
  double *const tally = FEW ? s_tally : absorbed;
  __shared__ int4 s_axes[3];  // per axis {n, cell stride, h bits}
  if (threadIdx.x < 3) {
    const int a = threadIdx.x;
    s_axes[a] = make_int4(W.n[a], a == 0 ? 1 : (a == 1 ? W.n[0] : W.n[0] * W.n[1]), __float_as_int(W.h[a]), 0);
  }
  __syncthreads();
  double em = 0.0, esc = 0.0;
  unsigned long long nsteps = 0;
  Ray R;
  float2 sc = make_float2(0.0f, 0.0f);  // step record of the ray's current cell
  const float ktop = (float)max(W.nT - 2, 0);
  const float2 *krow = nullptr;  // node-pair table: the ray's wavenumber row
  const float *krow1 = nullptr;  // wavenumber-major table: the ray's row
  bool active = false;
  for (;;) {
    const unsigned idle = __ballot_sync(0xffffffffu, !active);
    bool fresh = false;  // rays loaded for this pass
    if (next < last && (idle == 0xffffffffu || __popc(idle) >= REFILL)) {
      const unsigned rank = __popc(idle & ((1u << lane) - 1u));
      if (!active && next + rank < last) {
        float4 cd = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        // order: the rays grouped by wavenumber, so that a warp's lanes share a table row
        ray_init<TAB>(W, cells, tab, order ? (unsigned long long)__ldg(order + next + rank) : next + rank, record, R,
                 &cd);
        sc = step_cell(cd);
        if (TAB == 2) krow = reinterpret_cast<const float2 *>(tab) + (long long)R.j * (W.nT - 1);
        if (TAB == 1) krow1 = tab + (long long)R.j * W.nT;
        active = true;
      }
      next += __popc(idle);
      fresh = true;
    }
    const unsigned am = __ballot_sync(0xffffffffu, active);
    if (!am) break;
    if (!active) continue;
    bool done = false, dark = false;
    // kWalkUnroll steps per pass of the loop; each step loads the table value of
    // its cell and the next cell's data, both in flight while its arithmetic runs
#pragma unroll
    for (int u = 0; u < kWalkUnroll; ++u) {
      // rays of an opaque gas are over after a step or two: with few lanes left the pass ends
      // and new rays are loaded (4e8 rays of the 128^3 box 15.8 -> 14.4 ms, a thin gas even)
      if ((u == 1 || u == 2) && fresh && __popc(__ballot_sync(am, !done)) < kPassLanes) break;
      if (!done) {
        const float4 cd = step_bracket(sc, ktop);
        const float kap = TAB == 2 ? cell_kappa_row(cd, krow) : cell_kappa_row1(cd, krow1, W.nT);
        float2 scn = sc;
        done = ray_step<REC, true, true>(W, kap, tally, status, rec, R, true,
                                         [&](int c) { scn = __ldg(step_cells + c); }, s_axes);
        sc = scn;
        // a dark ray (transmission zero, no optical-depth cut) deposits nothing more:
        // only its visits are still to be counted
        dark = !done && R.trans == 0.0f && !W.tau_cut;
        done = done || dark;
      }
    }
    if (dark) {
      if (REC && R.row >= 0)  // a recorded ray lists its cells
        while (!ray_step<REC, true, true, true>(W, 0.0f, tally, status, rec, R, true, NoPrefetch(), s_axes)) {
        }
      else
        R.nv += dark_visits(W, R, status);
    }
    if (done) {
      const float out = R.w * R.trans;
      em += (double)R.w;
      esc += (double)out;
      nsteps += (unsigned long long)R.nv;
      if (REC && R.row >= 0) {
        rec.nvis[R.row] = R.nv;
        if (rec.weight) rec.weight[R.row] = R.w;
        if (rec.escaped) rec.escaped[R.row] = out;
      }
      active = false;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    em += __shfl_down_sync(0xffffffffu, em, o);
    esc += __shfl_down_sync(0xffffffffu, esc, o);
    nsteps += __shfl_down_sync(0xffffffffu, nsteps, o);
  }
  if (lane == 0) {
    if (em != 0.0) atomicAdd(scalars + 0, em);
    if (esc != 0.0) atomicAdd(scalars + 2, esc);
    if (nsteps) atomicAdd(steps_out, nsteps);
  }
  if (FEW) {
    __syncthreads();
    for (int c = threadIdx.x; c < (int)W.ncells; c += kWalkThreads)
      if (s_tally[c] != 0.0) atomicAdd(absorbed + c, s_tally[c]);
  }
}

// sum over the block of each thread's s, in thread 0 (a fixed tree)
__device__ __forceinline__ double block_sum(double s) {
  __shared__ double sh[32];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  }
  return s;
}

__global__ void k_reduce(const double *__restrict__ a, long long n, double *__restrict__ partial) {
  double s = 0.0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    s += a[i];
  s = block_sum(s);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// One block: the sum of a[0 .. n) (the partials of k_reduce, or a small tally itself), the
// energy balance into scalars, and what the host reads in one copy: out = {scalars[0..3],
// status bits, then copy_n values of a}.  (One thread adding 256 partials took 17 us.)
__global__ void __launch_bounds__(1024) k_final(const double *__restrict__ a, long long n, double *__restrict__ scalars,
                                                const uint32_t *__restrict__ status, double *__restrict__ out,
                                                int copy_n) {
  double s = 0.0;
  for (long long i = threadIdx.x; i < n; i += blockDim.x) {
    const double v = a[i];
    s += v;
    if (i < copy_n) out[5 + i] = v;
  }
  s = block_sum(s);
  if (threadIdx.x != 0) return;
  const double e = scalars[0], w = scalars[2], r = e != 0.0 ? fabs(e - s - w) / e : 0.0;
  scalars[1] = s;
  scalars[3] = r;
  out[0] = e;
  out[1] = s;
  out[2] = w;
  out[3] = r;
  out[4] = (double)*status;
}

__global__ void k_tally_zero(double *__restrict__ absorbed, long long n, double *__restrict__ scalars,
                             unsigned long long *__restrict__ steps, uint32_t *__restrict__ status) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (long long c = i; c < n; c += (long long)gridDim.x * blockDim.x) absorbed[c] = 0.0;
  if (i < 4) scalars[i] = 0.0;
  if (i == 0) {
    steps[0] = 0;
    *status = 0;
  }
}

rt_status validate_grid(const rt_grid *g) {
  if (!g) return fail(RT_E_INVAL, "grid is NULL");
  if (g->nx < 1 || g->ny < 1 || g->nz < 1) return fail(RT_E_INVAL, "grid dimensions must be >= 1");
  const long long nc = (long long)g->nx * g->ny * g->nz;
  if (nc > (1LL << 31) - 1) return fail(RT_E_INVAL, "grid has more than 2^31-1 cells");
  const double h[3] = {g->hx, g->hy, g->hz};
  for (int a = 0; a < 3; ++a)
    if (!(h[a] > 0) || std::isnan(h[a])) return fail(RT_E_INVAL, "grid cell sizes must be > 0 (or +inf)");
  if (!std::isfinite(g->hx) && !std::isfinite(g->hy) && !std::isfinite(g->hz))
    return fail(RT_E_INVAL, "grid needs at least one bounded axis");
  if (!g->T) return fail(RT_E_INVAL, "grid.T is NULL");
  return RT_OK;
}

}  // namespace

rt_status walk_setup(const rt_grid *grid, const rt_spectral *spec, uint64_t ray_begin,
                     uint64_t n_rays, uint64_t n_total, uint64_t seed, uint32_t enclosure,
                     int32_t flags, const rt_tally_buf *tally, const rt_record *record,
                     WalkParams *W, RecordPtrs *rp) {
  rt_status v = validate_grid(grid);
  if (v != RT_OK) return v;
  v = validate_spec(spec);
  if (v != RT_OK) return v;
  if (!tally || !tally->absorbed || !tally->scalars || !tally->steps || !tally->status)
    return fail(RT_E_INVAL, "tally buffer has a NULL pointer");
  const int mode = flags & 0xF;
  if (mode != RT_SRC_EMIT && mode != RT_SRC_BEAM) return fail(RT_E_INVAL, "flags: unknown source mode");
  if (flags & ~(0xF | RT_TAU_CUT)) return fail(RT_E_INVAL, "flags: unknown bits");
  if (n_total == 0 || n_rays > n_total) return fail(RT_E_INVAL, "n_rays_total must be >= n_rays and > 0");
  if (mode == RT_SRC_BEAM && !std::isfinite(grid->hx))
    return fail(RT_E_INVAL, "beam mode needs a bounded x axis");
  if (record) {
    if (record->n_rays < 0 || record->n_rays > (1LL << 31) - 1 ||
        (record->n_rays > 0 && (!record->cells || !record->ds || !record->n_visits ||
                                record->max_visits < 1)))
      return fail(RT_E_INVAL, "record: bad buffers");
  }
  const long long nc = (long long)grid->nx * grid->ny * grid->nz;
  W->n[0] = grid->nx; W->n[1] = grid->ny; W->n[2] = grid->nz;
  const double h[3] = {grid->hx, grid->hy, grid->hz};
  double V = 1.0;
  const int n3[3] = {grid->nx, grid->ny, grid->nz};
  for (int a = 0; a < 3; ++a) {
    W->fin[a] = std::isfinite(h[a]) ? 1 : 0;
    W->h[a] = (float)h[a];
    W->inv_h[a] = W->fin[a] ? 1.0f / W->h[a] : 0.0f;
    W->len[a] = W->fin[a] ? (float)n3[a] * W->h[a] : 0.0f;
    if (W->fin[a]) V *= h[a];
  }
  // dark_visits' closed form: its error bound holds for up to 65536 cells an axis and cell
  // sizes whose face distances neither overflow nor underflow (a direction cosine is 0 or
  // at least 5e-11)
  W->jump = 1;
  for (int a = 0; a < 3; ++a)
    if (W->fin[a] && (n3[a] > 65536 || !(W->h[a] >= 1e-15f && W->h[a] <= 1e15f))) W->jump = 0;
  for (int a = 0; a < 2; ++a) {
    uint32_t s = 0;
    while ((1ull << s) < (unsigned long long)n3[a]) ++s;
    W->div_s[a] = s;
    W->div_m[a] = (uint32_t)(((1ull << (31 + s)) + (unsigned long long)n3[a] - 1) / (unsigned long long)n3[a]);
  }
  W->ncells = nc;
  W->n_nu = spec->n_nu;
  W->nT = spec->nT;
  W->mode = mode;
  W->tau_cut = (flags & RT_TAU_CUT) ? 1 : 0;
  W->step_cap = grid->nx + grid->ny + grid->nz + 4;
  W->ray_begin = ray_begin;
  W->n_rays = n_rays;
  W->seed_lo = (uint32_t)seed;
  W->seed_hi = (uint32_t)(seed >> 32);
  W->enclosure = enclosure;
  W->nu_min = (float)spec->nu_min;
  W->dnu = (float)spec->dnu;
  const double pi = 3.14159265358979323846;
  W->w_scale = (float)(4.0 * pi * V * 100.0 * (100.0 * spec->dnu) * (double)nc *
                       (double)spec->n_nu / (double)n_total);
  const double hP = 6.62607015e-34, cL = 299792458.0, kB = 1.380649e-23;
  W->two_hc2 = (float)(2.0 * hP * cL * cL);
  W->c2_m = (float)(hP * cL / kB);
  *rp = RecordPtrs{nullptr, nullptr, nullptr, nullptr, nullptr};
  W->rec_n = 0;
  W->rec_max = 0;
  if (record && record->n_rays > 0) {
    *rp = RecordPtrs{record->cells, record->ds, record->n_visits, record->weight, record->escaped};
    W->rec_n = record->n_rays;
    W->rec_max = record->max_visits;
  }
  return RT_OK;
}

int walk_table_layout(int nT, long long n_nu) {
  return (nT >= 2 && (size_t)n_nu * (size_t)(nT - 1) * 8 <= kPairTableBytes) ? 2 : 1;
}

size_t walk_table_bytes(int layout, int nT, long long n_nu) {
  return layout == 2 ? (size_t)n_nu * (size_t)(nT - 1) * 8 : (size_t)n_nu * (size_t)nT * 4;
}

// blocks along the nodes (see table_block)
static int walk_table_rows(int layout, int nT) { return ((layout == 2 ? nT - 1 : nT) + kPairRows - 1) / kPairRows; }

rt_status launch_walk_table(int layout, const float *tab, int nT, long long n_nu, float *out, cudaStream_t st) {
  const int ny = walk_table_rows(layout, nT);
  const dim3 g((unsigned)((n_nu + 31) / 32), (unsigned)ny);
  if (layout == 2) k_walk_table<2><<<g, kSetupThreads, 0, st>>>(tab, nT, n_nu, out);
  else k_walk_table<1><<<g, kSetupThreads, 0, st>>>(tab, nT, n_nu, out);
  RT_CUDA_TRY(cudaGetLastError());
  return RT_OK;
}

CellParams cell_params(const rt_spectral *spec, long long ncells, int has_px) {
  CellParams C;
  C.ncells = ncells;
  C.Tmin = (float)spec->T_min;
  C.dT = spec->nT >= 2 ? (float)((spec->T_max - spec->T_min) / (double)(spec->nT - 1)) : 1.0f;
  C.den = (float)(spec->p_ref_atm * spec->x_ref);
  C.pref = (float)spec->p_ref_atm;
  C.xref = (float)spec->x_ref;
  C.nT = spec->nT;
  C.has_px = has_px;
  return C;
}

rt_status band_plan(const WalkParams &W, int band_pts, long long n_bands, long long chunk,
                    unsigned long long *counts, long long *band_start, long long *item_start, int *item_band,
                    uint32_t *order, int sms, cudaStream_t st) {
  if (n_bands > 1) {
    RT_CUDA_TRY(cudaMemsetAsync(counts, 0, (size_t)n_bands * sizeof(unsigned long long), st));
    const unsigned gb = (unsigned)std::min<unsigned long long>((W.n_rays + 255) / 256, 8ull * (unsigned)sms);
    k_band_count<<<gb, 256, 0, st>>>(W, band_pts, n_bands, counts);
    RT_CUDA_TRY(cudaGetLastError());
    // the counts are read by the plan, then the same words serve as the scatter cursors
    k_band_plan<<<1, 1024, 0, st>>>(counts, n_bands, W.n_rays, chunk, band_start, item_start, item_band, counts);
    RT_CUDA_TRY(cudaGetLastError());
    if (order) {
      k_band_scatter<<<gb, 256, 0, st>>>(W, band_pts, counts, order);
      RT_CUDA_TRY(cudaGetLastError());
    }
  } else {
    k_band_plan<<<1, 1024, 0, st>>>(nullptr, 1, W.n_rays, chunk, band_start, item_start, item_band, nullptr);
    RT_CUDA_TRY(cudaGetLastError());
  }
  return RT_OK;
}

rt_status trace_impl(const rt_grid *grid, const float *kappa, const rt_spectral *spec,
                     uint64_t ray_begin, uint64_t n_rays, uint64_t n_total, uint64_t seed,
                     uint32_t enclosure, int32_t flags, const rt_tally_buf *tally,
                     const rt_record *record, cudaStream_t st) {
  if (!kappa) return fail(RT_E_INVAL, "kappa is NULL");
  WalkParams W;
  RecordPtrs rp;
  rt_status v = walk_setup(grid, spec, ray_begin, n_rays, n_total, seed, enclosure, flags, tally,
                           record, &W, &rp);
  if (v != RT_OK) return v;
  if (n_rays == 0) return RT_OK;
  Scratch scr;
  const int layout = walk_table_layout(spec->nT, spec->n_nu);
  const size_t cbytes = ((size_t)W.ncells * (sizeof(float4) + sizeof(float2)) + 255) & ~size_t(255);
  const size_t tbytes = (walk_table_bytes(layout, spec->nT, spec->n_nu) + 255) & ~size_t(255);
  // rays grouped by wavenumber (one band per wavenumber): counts, band and item starts, order
  const bool group = n_rays <= 0xFFFFFFFFull && g_walk_group == 2;
  const long long nb = spec->n_nu;
  const size_t pbytes = group ? (((size_t)nb * 8 * 3 + 64 + 255) & ~size_t(255)) : 0;
  const size_t obytes = group ? (size_t)n_rays * sizeof(uint32_t) : 0;
  v = scr.alloc(cbytes + tbytes + pbytes + obytes, st);
  if (v != RT_OK) return v;
  float4 *cells = scr.as<float4>();
  float2 *step_cells = reinterpret_cast<float2 *>(cells + W.ncells);
  float *tabw = reinterpret_cast<float *>(scr.as<char>() + cbytes);
  {
    const CellParams C = cell_params(spec, W.ncells, (grid->p_atm || grid->x) ? 1 : 0);
    const long long cb = (W.ncells + kSetupThreads - 1) / kSetupThreads, slices = (spec->n_nu + 31) / 32;
    const long long ny = walk_table_rows(layout, spec->nT);
    // (a table of 2^31 blocks would take 17 TB: the scratch was refused before)
    auto setup = layout == 2 ? k_walk_setup<2> : k_walk_setup<1>;
    setup<<<(unsigned)(cb + slices * ny), kSetupThreads, 0, st>>>(grid->T, grid->p_atm, grid->x, C, cells, step_cells,
                                                                    tally->status, (unsigned)cb, kappa, spec->nT,
                                                                    spec->n_nu, (unsigned)slices, tabw);
    RT_CUDA_TRY(cudaGetLastError());
  }
  int dev = 0, sms = 0;
  RT_CUDA_TRY(cudaGetDevice(&dev));
  RT_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  uint32_t *order = nullptr;
  if (group) {
    char *pb = scr.as<char>() + cbytes + tbytes;
    unsigned long long *counts = reinterpret_cast<unsigned long long *>(pb);
    long long *band_start = reinterpret_cast<long long *>(counts + nb);
    long long *item_start = band_start + (nb + 1);
    order = reinterpret_cast<uint32_t *>(pb + pbytes);
    v = band_plan(W, 1, nb, 1LL << 40, counts, band_start, item_start, nullptr, order, sms, st);
    if (v != RT_OK) return v;
  }
  const bool rec = rp.cells != nullptr;
  // visit recording (a test path) uses one configuration; the tuned shape otherwise
  auto pick = [&](auto tab) {
    constexpr int L = decltype(tab)::value;
    if (rec) return k_walk<true, L, kRefillIdleDefault>;
    if (W.ncells <= kFewCells) return k_walk<false, L, 16, true>;
    return g_walk_refill == 12 ? k_walk<false, L, 12> : k_walk<false, L, 16>;
  };
  auto kern = layout == 2 ? pick(std::integral_constant<int, 2>()) : pick(std::integral_constant<int, 1>());
  // persistent warps, each with a contiguous ray range, at least one ray a lane (a call of 1e5
  // rays is over sooner with a ray on every lane than with two on half of them)
  const unsigned long long want = (n_rays + kWalkThreads - 1) / kWalkThreads;
  const unsigned long long cap = (unsigned long long)sms * kWalkBlocks;
  const unsigned blocks = (unsigned)(want < cap ? want : cap);
  kern<<<blocks, kWalkThreads, 0, st>>>(cells, step_cells, tabw, order, W, tally->absorbed, tally->scalars, tally->steps,
                                        tally->status, rp);
  RT_CUDA_TRY(cudaGetLastError());
  return RT_OK;
}

rt_status tally_impl(const rt_tally_buf *t, int64_t ncells, double *host_absorbed,
                     double *host_scalars, cudaStream_t st) {
  if (!t || !t->absorbed || !t->scalars || !t->steps || !t->status)
    return fail(RT_E_INVAL, "rt_tally: bad tally buffer");
  if (ncells < 1) return fail(RT_E_INVAL, "rt_tally: ncells must be >= 1");
  if (!host_scalars) return fail(RT_E_INVAL, "rt_tally: host_scalars is NULL");
  // a small tally is summed by one block and comes back with the scalars in one copy
  constexpr int kSmall = 4096;
  const bool small = ncells <= kSmall;
  const int back = small && host_absorbed ? (int)ncells : 0;
  Scratch scr;
  rt_status v = scr.alloc(sizeof(double) * (size_t)(kReduceBlocks + 5 + back), st);
  if (v != RT_OK) return v;
  double *partial = scr.as<double>(), *out = partial + kReduceBlocks;
  if (!small) {
    k_reduce<<<kReduceBlocks, 256, 0, st>>>(t->absorbed, ncells, partial);
    RT_CUDA_TRY(cudaGetLastError());
  }
  k_final<<<1, small && ncells > 256 ? 1024 : 256, 0, st>>>(small ? t->absorbed : partial, small ? ncells : kReduceBlocks,
                                                            t->scalars, t->status, out, back);
  RT_CUDA_TRY(cudaGetLastError());
  double buf[5 + kSmall];
  if (host_absorbed && !back)
    RT_CUDA_TRY(cudaMemcpyAsync(host_absorbed, t->absorbed, (size_t)ncells * sizeof(double),
                                cudaMemcpyDeviceToHost, st));
  RT_CUDA_TRY(cudaMemcpyAsync(buf, out, (size_t)(5 + back) * sizeof(double), cudaMemcpyDeviceToHost, st));
  RT_CUDA_TRY(cudaStreamSynchronize(st));
  for (int i = 0; i < 4; ++i) host_scalars[i] = buf[i];
  for (int i = 0; i < back; ++i) host_absorbed[i] = buf[5 + i];
  return status_from_bits((uint32_t)buf[4]);
}

rt_status tally_zero_impl(const rt_tally_buf *t, int64_t ncells, cudaStream_t st) {
  if (!t || !t->absorbed || !t->scalars || !t->steps || !t->status || ncells < 1)
    return fail(RT_E_INVAL, "rt_tally_zero: bad tally buffer");
  const unsigned blocks = (unsigned)std::min<int64_t>((ncells + 255) / 256, 1 << 16);
  k_tally_zero<<<blocks, 256, 0, st>>>(t->absorbed, ncells, t->scalars, t->steps, t->status);
  RT_CUDA_TRY(cudaGetLastError());
  return RT_OK;
}

}  // namespace rt

extern "C" {

rt_status rt_trace(const rt_grid *grid, const float *kappa, const rt_spectral *spec,
                   uint64_t ray_begin, uint64_t n_rays, uint64_t n_rays_total, uint64_t seed,
                   uint32_t enclosure, int32_t flags, const rt_tally_buf *tally,
                   const rt_record *record, void *stream) {
  return rt::trace_impl(grid, kappa, spec, ray_begin, n_rays, n_rays_total, seed, enclosure, flags,
                        tally, record, (cudaStream_t)stream);
}

rt_status rt_tally_zero(const rt_tally_buf *tally, int64_t ncells, void *stream) {
  return rt::tally_zero_impl(tally, ncells, (cudaStream_t)stream);
}

rt_status rt_tally(const rt_tally_buf *tally, int64_t ncells, double *host_absorbed,
                   double host_scalars[4], void *stream) {
  return rt::tally_impl(tally, ncells, host_absorbed, host_scalars, (cudaStream_t)stream);
}

}  // extern "C"
