// Absorption-coefficient table on a temperature grid: Eqs. (S) and (tau) of
// Section 3, for one absorbing gas, with Lorentz or Voigt line shapes and a
// wing cutoff.  Kernels:
//   k_line_geometry : per line, the binary64 grid decisions (cutoff window
//                     [j_lo, j_hi], nearest grid index j_c and offset) and the
//                     profile-evaluation count; validates device-resident lists.
//   k_line_setup    : that, and per (T node, line), Eq. (S) times the number density
//                     and the width parameters, in binary32 with double-float
//                     arithmetic for the Boltzmann exponent; for Voigt lines
//                     also the far-wing polynomial coefficients.
//   k_line_list     : a short host list, its kernel parameters, into device memory.
//   k_adaptive_windows : with adaptive points, per (T node, line) its own window.
//   k_tile_lines    : per 256-point wavenumber tile, the range of lines whose
//                     windows reach it, split into segments by kind: lines far from
//                     the tile (summed at a few nodes and interpolated), lines whose
//                     window ends inside it, covering lines with the degree-4 series,
//                     and the general path (near-centre zone).
//   k_kappa         : per (tile, up to 8 T nodes), the line sum.  The tile's
//                     lines are staged in shared memory by bulk asynchronous
//                     copies (cp.async.bulk + mbarrier), double buffered; each
//                     lane owns 8 consecutive points (two float4 stores) and
//                     Kahan-sums over lines.
//   k_kappa_ppl     : with a fixed number of points per line, one thread per
//                     point and eight T nodes over the few lines whose windows hold it.
#include <cmath>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "rt_common.cuh"

namespace rt {
namespace {

constexpr int kPtsPerThread = 8;
constexpr int kTilePts = 32 * kPtsPerThread;  // 256 wavenumbers per block, one warp per T node
constexpr int kMaxTPerBlock = 8;              // warps (T nodes) per block
constexpr int kChunk = 192;                   // lines per staged chunk that need P only (half that with P2)
constexpr int kArgLines = 1000;               // host lists up to this travel as kernel parameters (32 of 32,764 B)
constexpr int kDirectPairs = 65536;           // (node, line) pairs up to which the set-up reads them there
constexpr int kGroup = 8;                     // fast-path lines summed before one compensated add
constexpr int kNodeGroup = 4;                 // interpolated lines a lane sums before one compensated add
constexpr unsigned kWaitLimit = 1u << 22;     // bounded mbarrier waits

// CODATA 2018 (SI); derived quantities are formed on the host in binary64.
constexpr double kH = 6.62607015e-34, kC = 299792458.0, kKB = 1.380649e-23;
constexpr double kAmu = 1.66053906660e-27, kAtm = 101325.0;
constexpr double kPi = 3.14159265358979323846;

struct GeomParams {
  double nu_min, dnu, inv_dnu, cutoff;
  long long n_nu, n_lines;
  int nT, check, ppl;
};

struct PrefParams {
  double T_min, T_max, T_ref;  // exact inputs, split into double-float in the kernel
  df c2;                       // second radiation constant h c / k_B, cm K
  float u_coef;                // x_ref p_ref atm / k_B * 1e-6  [cm^-3 K]
  float p_ref, n_T, q_exp;
  float doppler;               // sqrt(2 ln2 k_B / (m amu)) / c  [K^-1/2]
  float inv_dnu, dnu;
  long long n_lines;
  int nT, profile;
};

__device__ __forceinline__ double grid_nu(double nu_min, long long j, double dnu) {
  return __dadd_rn(nu_min, __dmul_rn((double)j, dnu));
}

__device__ __forceinline__ void line_geometry(const double *__restrict__ nu0, const double *__restrict__ S,
                                              const double *__restrict__ g, const double *__restrict__ E,
                                              const GeomParams &P, int4 *__restrict__ R,
                                              unsigned long long *evals, uint32_t *status, long long l) {
  unsigned long long cnt = 0;
  if (l < P.n_lines) {
    const double v = nu0[l];
    if (P.check) {
      const double s = S[l], gg = g[l], e = E[l];
      if (!isfinite(v) || !isfinite(s) || !(s > 0.0) || !isfinite(gg) || !(gg > 0.0) ||
          !isfinite(e) || !(e >= 0.0))
        status_or(status, RT_DEV_NONFINITE);
      if (l > 0 && !(nu0[l - 1] <= v)) status_or(status, RT_DEV_UNSORTED);
    }
    // nearest grid index: the origin of the line's local coordinate (any index within a
    // grid step of the centre serves, the offset below is exact for it)
    double fc = (v - P.nu_min) * P.inv_dnu;
    fc = fmin(fmax(isfinite(fc) ? fc : 0.0, -536870912.0), 536870912.0);
    const long long jc = llrint(fc);
    const double dc = __dsub_rn(grid_nu(P.nu_min, jc, P.dnu), v);  // nu_jc - nu0
    const float dg = __double2float_rn(dc * P.inv_dnu);             // grid units
    // inclusive cutoff window: -cutoff <= nu_j - nu0 <= cutoff, decided in binary64 below
    // from an estimate (a multiplication by 1 / dnu: the two divisions it replaces took half
    // of the kernel's time)
    double flo = ceil((v - P.cutoff - P.nu_min) * P.inv_dnu);
    double fhi = floor((v + P.cutoff - P.nu_min) * P.inv_dnu);
    flo = fmin(fmax(isfinite(flo) ? flo : 0.0, -1.0), (double)P.n_nu + 1.0);
    fhi = fmin(fmax(isfinite(fhi) ? fhi : 0.0, -2.0), (double)P.n_nu + 1.0);
    long long lo = (long long)flo, hi = (long long)fhi;
    if (P.ppl > 0) {  // fixed points per line around the centre
      double jf = floor((v - P.nu_min) / P.dnu);
      jf = fmin(fmax(isfinite(jf) ? jf : 0.0, -536870912.0), 536870912.0);
      lo = (long long)jf - P.ppl / 2 + 1;
      hi = (long long)jf + P.ppl / 2;
    }
    if (lo < 0) lo = 0;
    if (hi > P.n_nu - 1) hi = P.n_nu - 1;
    if (P.ppl <= 0) {
      auto below = [&](long long j) { return __dsub_rn(grid_nu(P.nu_min, j, P.dnu), v) < -P.cutoff; };
      auto above = [&](long long j) { return __dsub_rn(grid_nu(P.nu_min, j, P.dnu), v) > P.cutoff; };
      int it = 0;
#pragma unroll 1
      for (; it < 6 && lo < P.n_nu && below(lo); ++it) ++lo;
      if (it == 0) {
#pragma unroll 1
        for (; it < 6 && lo > 0 && !below(lo - 1); ++it) --lo;
      }
      it = 0;
#pragma unroll 1
      for (; it < 6 && hi >= 0 && above(hi); ++it) --hi;
      if (it == 0) {
#pragma unroll 1
        for (; it < 6 && hi < P.n_nu - 1 && !above(hi + 1); ++it) ++hi;
      }
    }
    R[l] = make_int4((int)lo, (int)hi, (int)jc, __float_as_int(dg));
    if (hi >= lo) cnt = (unsigned long long)(hi - lo + 1) * (unsigned long long)P.nT;
  }
  if (evals) {
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, o);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(evals, cnt);
  }
}

__global__ void k_line_geometry(const double *__restrict__ nu0, const double *__restrict__ S,
                                const double *__restrict__ g, const double *__restrict__ E,
                                GeomParams P, int4 *__restrict__ R,
                                unsigned long long *evals, uint32_t *status) {
  line_geometry(nu0, S, g, E, P, R, evals, status, (long long)blockIdx.x * blockDim.x + threadIdx.x);
}

// Eq. (S) times the number density, and the profile's coefficients, for line l
// at T node k.  Voigt: P = {c0, s dnu, y^2, c2}, P2 = {c3, c4, y, half-width of |z| < 8}
// with the far-wing series c0 t + c1 t^2 + c2 t^3 + c3 t^4 + c4 t^5 (c1 = 1.5 c0).
// Returns the line's far-zone distance in grid units (float bits): beyond it the t^3, t^4
// and t^5 terms drop at most 1.25 * 2^-24 of the value, so the degree-1 series
// c0 t (1 + 1.5 t) stands for the full one.
// The quantities of T node k that every line shares.
struct PrefNode {
  df Tk, iT, iTref;
  float tr, qratio, wratio, sqrtT;
};

__device__ __forceinline__ PrefNode pref_node(const PrefParams &Q, int k) {
  // T_k = T_min + k (T_max - T_min) / (nT - 1) and 1/T_k in double-float
  PrefNode N;
  df Tk = df_from_double(Q.T_min);
  if (Q.nT > 1) {
    const df span = df_add(df_from_double(Q.T_max), df_neg(Tk));
    const df step = df_mul(span, df_recip(df{(float)(Q.nT - 1), 0.0f}));
    Tk = df_add(Tk, df_mul(step, df{(float)k, 0.0f}));
  }
  N.Tk = Tk;
  N.iT = df_recip(Tk);
  const df Tref = df_from_double(Q.T_ref);
  N.iTref = df_recip(Tref);
  N.tr = Tref.hi * N.iT.hi;  // T_ref / T
  N.qratio = powf(N.tr, Q.q_exp);
  N.wratio = powf(N.tr, Q.n_T);
  N.sqrtT = sqrtf(Tk.hi);
  return N;
}

__device__ __forceinline__ void prefactor_one(const double *__restrict__ nu0, const double *__restrict__ S,
                                                  const double *__restrict__ g, const double *__restrict__ E,
                                                  const PrefParams &Q, const PrefNode &N,
                                                  float4 *__restrict__ Pout, float4 *__restrict__ P2out,
                                                  long long l, int k, unsigned &far) {
  const df iT = N.iT, iTref = N.iTref;
  const float iTf = iT.hi;
  // Eq. (S): Q ratio, Boltzmann ratio (exponent in double-float), stimulated emission
  const float qratio = N.qratio;
  const df arg = df_mul(df_mul(Q.c2, df_from_double(E[l])), df_add(iTref, df_neg(iT)));
  const float boltz = expf(arg.hi) * (1.0f + arg.lo);
  const float nu0f = __double2float_rn(nu0[l]);
  const float c2nu = Q.c2.hi * nu0f;
  const float stim = expm1f(-c2nu * iTf) / expm1f(-c2nu * iTref.hi);
  const float S_T = __double2float_rn(S[l]) * qratio * boltz * stim;
  const float A = (Q.u_coef * iTf) * S_T;  // u(T) S(T), cm^-1 per unit profile
  const float gam = __double2float_rn(g[l]) * Q.p_ref * N.wratio;
  float4 out;
  far = 0;
  if (Q.profile == RT_PROFILE_LORENTZ) {
    const float gg = gam * Q.inv_dnu;  // half-width in grid units
    out = make_float4(A * gg * (float)(1.0 / kPi) * Q.inv_dnu, gg * gg, 0.0f, 0.0f);
  } else {
    const float alpha = nu0f * N.sqrtT * Q.doppler;  // Doppler HWHM, cm^-1
    const float s = 0.83255461f / alpha;                  // sqrt(ln 2) / alpha
    const float y = s * gam;
    const float sd = s * Q.dnu;
    const float y2 = y * y;
    // far wing: c0 t (1 + 1.5 t + (3.75 - 2 y^2) t^2 - 15 y^2 t^3 + 12 y^4 t^4), t = 1/|z|^2
    const float c0 = A * s * (float)(1.0 / kPi) * y;
    out = make_float4(c0, sd, y2, __fmaf_rn(-2.0f, y2, 3.75f) * c0);
    // half-width (grid units) of |z| < 8, inside which the general path takes the rational form
    const float u_core = sqrtf(fmaxf(64.0f - y2, 0.0f)) / sd;
    P2out[(long long)k * Q.n_lines + l] = make_float4(-15.0f * y2 * c0, 12.0f * y2 * y2 * c0, y, u_core);
    // (27 y^2 / 2^-24)^(1/6) = 27.66 y^(1/3), beyond which 27 y^2 t^3 <= 2^-24 (t <= 1/x^2),
    // and (2^25 (3.75 + 2 y^2))^(1/4), with 5 % margin, in grid units
    const float d2 = 29.1f * cbrtf(y) / sd;
    const float d1 = fmaxf(1.05f * sqrtf(sqrtf(33554432.0f * (3.75f + 2.0f * y2))) / sd, d2);
    far = (d1 >= 0.0f && d1 < 1e9f) ? __float_as_uint(d1) : __float_as_uint(1e9f);
  }
  Pout[(long long)k * Q.n_lines + l] = out;
}

__device__ __forceinline__ void prefactors(const double *__restrict__ nu0, const double *__restrict__ S,
                                           const double *__restrict__ g, const double *__restrict__ E,
                                           const PrefParams &Q, float4 *__restrict__ Pout, float4 *__restrict__ P2out,
                                           unsigned *__restrict__ far_bits, long long l, int k) {
  __shared__ PrefNode s_node;  // T node k's shared quantities, formed once per block
  if (threadIdx.x == 0) s_node = pref_node(Q, k);
  __syncthreads();
  const PrefNode N = s_node;
  unsigned fb = 0;  // this line's far-zone distance (grid units, float bits)
  if (l < Q.n_lines) prefactor_one(nu0, S, g, E, Q, N, Pout, P2out, l, k, fb);
  // block maximum, one atomic per block (non-negative floats order like their bits)
  __shared__ unsigned s_max[32];
  const unsigned wm = __reduce_max_sync(0xffffffffu, fb);
  if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = wm;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned m = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = max(m, s_max[w]);
    if (m) atomicMax(far_bits, m);
  }
}

// The lines: arrays on the GPU, or a short host list as kernel parameters, which a launch copies
// before it returns (no allocation, no wait, nothing kept).
struct LineArrays {
  const double *nu0, *S, *g, *E;
  __device__ const double *array(int q) const { return q == 0 ? nu0 : (q == 1 ? S : (q == 2 ? g : E)); }
};
template <int N>
struct LineArgs {
  double v[4][N];
  __device__ const double *array(int q) const { return v[q]; }
};

// The lines' set-up in one launch: line_blocks blocks of k_line_geometry's work, then as many
// for each T node's prefactors (neither reads what the other writes).
template <class Lines>
__global__ void k_line_setup(const __grid_constant__ Lines L, GeomParams G, PrefParams Q,
                             unsigned line_blocks, int4 *__restrict__ R, float4 *__restrict__ Pout,
                             float4 *__restrict__ P2out, unsigned *__restrict__ far_bits,
                             unsigned long long *evals, uint32_t *status) {
  const double *nu0 = L.array(0), *S = L.array(1), *g = L.array(2), *E = L.array(3);
  const unsigned y = blockIdx.x / line_blocks;
  const long long l = (long long)(blockIdx.x - y * line_blocks) * blockDim.x + threadIdx.x;
  if (y == 0) line_geometry(nu0, S, g, E, G, R, evals, status, l);
  else prefactors(nu0, S, g, E, Q, Pout, P2out, far_bits, l, (int)y - 1);
}

// ---- bulk asynchronous copies global -> shared, completed on an mbarrier
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ long long lower_bound_hi(const int4 *R, long long n, int j) {
  long long a = 0, b = n;  // first l with R[l].y >= j
  while (a < b) {
    long long m = (a + b) >> 1;
    if (R[m].y < j) a = m + 1; else b = m;
  }
  return a;
}
__device__ __forceinline__ long long lower_bound_lo(const int4 *R, long long n, int j) {
  long long a = 0, b = n;  // first l with R[l].x >= j
  while (a < b) {
    long long m = (a + b) >> 1;
    if (R[m].x < j) a = m + 1; else b = m;
  }
  return a;
}

// ---- interpolation of far lines
// The sum of the lines far from a tile is smooth over it: it is evaluated at a few nodes
// and interpolated to the tile's points (the line-by-line interpolation technique of Fomin,
// JQSRT 53 (1995) 663, and Kuntz and Hoepfner, JQSRT 63 (1999) 97, here on Chebyshev
// nodes).  A Lorentz-like wing 1/(u^2 + g^2) whose centre is D half-widths from the middle of
// an interval has its poles on or outside the Bernstein ellipse of
// rho = D + sqrt(D^2 - 1), so M nodes leave an error of order M rho^-M of the value.
// The distances are those beyond which the interpolation changes no line's value by more than
// half a binary32 rounding, 2^-25 = 3.0e-8 of it, at any point (computed in binary64 for g = 0 ..
// 1000 grid points; the nodes are Chebyshev's rounded to 1/16 grid point, so that u is exact):
//   8 nodes on the tile (half-width 128 points), centre >= 704 points from it: 2.7e-8
//  16 nodes on the tile, centre >= 141 points from it:                        1.7e-8
//   4 nodes on a 32-point sub-block, centre >= 1080 points from it:           2.9e-8
// The tables' error is that of the values' roundings: 36 tables are 1.55e-7 from binary64 in the
// mean, 1.60e-7 with every line at every point, 1.54e-7 with 900, 160 and 1600 points, which take
// 4.82 instead of 4.72 ms for the 128^3 workload.
template <int M>
struct Nodes {
  double u[M];
};
constexpr Nodes<8> kNodes8{{1.9375, 21.0625, 56.375, 102.5, 152.5, 198.625, 233.9375, 253.0625}};
constexpr Nodes<16> kNodes16{{0.125, 5.0, 14.625, 28.5625, 46.3125, 67.1875, 90.3125, 114.9375, 140.0625, 164.6875,
                              187.8125, 208.6875, 226.4375, 240.375, 250.0, 254.875}};
constexpr Nodes<4> kNodes4{{0.6875, 9.375, 21.625, 30.3125}};
constexpr int kDist8 = 704, kDist16 = 141, kDistEdge = 1080;  // grid points from the tile's nearest point

// Lagrange weights w[m][j] of the M nodes at N positions, and the nodes in binary32
template <int M, int N>
struct NodeTable {
  float u[M];
  float w[M][N];
};
template <int M, int N, class At>
constexpr NodeTable<M, N> node_table(const Nodes<M> &nd, At at) {
  NodeTable<M, N> t{};
  for (int m = 0; m < M; ++m) t.u[m] = (float)nd.u[m];
  for (int j = 0; j < N; ++j)
    for (int m = 0; m < M; ++m) {
      double p = 1.0;
      for (int q = 0; q < M; ++q)
        if (q != m) p *= (at(j) - nd.u[q]) / (nd.u[m] - nd.u[q]);
      t.w[m][j] = (float)p;
    }
  return t;
}
struct AtPoint {
  constexpr double operator()(int j) const { return (double)j; }
};
struct AtNode16 {
  constexpr double operator()(int j) const { return kNodes16.u[j]; }
};
__device__ constexpr NodeTable<16, kTilePts> kTab16 = node_table<16, kTilePts>(kNodes16, AtPoint{});
__device__ constexpr NodeTable<8, 16> kTab8 = node_table<8, 16>(kNodes8, AtNode16{});
__device__ constexpr NodeTable<4, 32> kTab4 = node_table<4, 32>(kNodes4, AtPoint{});

// Weideman's series for the core points.  Its error falls fast with y: relative to Re w over
// |z| < 8 (against binary64), 24 terms give 1.8e-8 at y = 0.1 and 4e-10 at 0.75; 16 and 12 terms
// are used from the y on where theirs is as small, 1.5e-8 and 1.8e-8.  Fewer terms also round less
// often: the 36 tables are 1.60e-7 from binary64 with 24 terms throughout, 1.55e-7 so.
constexpr float kTerms16 = 2.3f, kTerms12 = 5.0f;
struct WeidSet {
  WeidSeries<24> n24;
  WeidSeries<16> n16;
  WeidSeries<12> n12;
};

// Kinds of line ranges within a tile (see k_tile_lines).
enum SegKind : int {
  kSegGeneral = 0,     // window masking and near-centre test per line
  kSegFast = 1,        // covering, degree-4 far-wing series at every point
  kSegNodes16 = 2,     // covering, degree-4 series at 16 nodes
  kSegNodes8 = 3,      // covering, degree-1 series at 8 nodes
  kSegEdge = 4,        // window ends inside the tile: degree-1 series at 4 nodes of each covered
                       // 32-point sub-block and at the points of the one it ends in
  kSegFar1Masked = 5,  // window ends inside the tile, degree-1 series at every point
};
__device__ __forceinline__ bool degree1_kind(int kd) { return kd >= kSegNodes8; }
constexpr int kMaxSegs = 12;
constexpr int kTileInts = 5;  // int4 per tile: {lb, ub, nseg, 0}, 12 ends, 16 kind bytes

// Per tile of kTilePts wavenumbers [jw0, jw0 + kTilePts): the lines [lb, ub)
// whose windows reach it, split into ranges by kind.  Windows and centres are
// monotone in the (sorted) line index, so every set below is an index range:
//   cover : the window holds every point of the tile that is on the grid (no masking);
//   near  : j_c within W + 4 grid points of the tile, W bounding the near-centre
//           half-width of every line (lines outside it have no point |z| < 20);
//   n16, n8, edge : j_c at least kDist16 (and W + 4), kDist8 or kDistEdge (and D1) grid
//           points from the tile, D1 bounding every line's far-zone distance (degree-1
//           series).
// Covering lines are nodes-8, nodes-16, fast or (near) general; partially covering lines
// are edge, far1-masked or general.
__device__ __forceinline__ int clamp_int(long long v) {
  return (int)min(max(v, -0x40000000LL), 0x40000000LL);  // centres lie within 2^29 grid steps
}

__global__ void k_tile_lines(const int4 *__restrict__ R, long long n, long long n_nu, int W,
                             const unsigned *__restrict__ far_bits, long long n_tiles,
                             int4 *__restrict__ out) {
  // One warp per tile.  The 14 searches run side by side, 32 lanes a search: each round reads
  // 32 lines spread over the remaining range of every search at once and keeps the gap the
  // key lies in, so that a list of 500 lines takes two dependent reads and one of 1e6 four
  // (a lane per search took 9 and 20; with the warp-parallel split below instead of one
  // lane's insertion sort the kernel's time fell from 8.4 to 5.3 us for 500 lines).
  const long long t = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (t >= n_tiles) return;  // warp-uniform
  const long long near = (long long)W + 4;
  const long long D1 = max(near, (long long)ceilf(fminf(__uint_as_float(far_bits[0]), 1e9f)) + 2);
  const long long d16 = max(near, (long long)kDist16), d8 = max(D1, (long long)kDist8), dE = max(D1, (long long)kDistEdge);
  const long long jw0 = t * kTilePts, jw1 = jw0 + kTilePts - 1;
  // search i: the first line whose field (0: window start, 1: window end, 2: centre) >= key;
  // 0, 1: the tile's lines [lb, ub); 2, 3: covering ones; 4 .. 8: centres left of the tile by
  // dE, D1, d8, d16, near; 9 .. 13: right of it by near, d16, d8, D1, dE
  constexpr int kSearches = 14;
  const int key[kSearches] = {(int)jw0, (int)min(jw0 + (long long)kTilePts, n_nu), (int)min(jw1, n_nu - 1), (int)jw0 + 1,
                              clamp_int(jw0 - dE), clamp_int(jw0 - D1), clamp_int(jw0 - d8), clamp_int(jw0 - d16),
                              clamp_int(jw0 - near), clamp_int(jw1 + near + 1), clamp_int(jw1 + d16 + 1),
                              clamp_int(jw1 + d8 + 1), clamp_int(jw1 + D1 + 1), clamp_int(jw1 + dE + 1)};
  int pos[kSearches];  // the answer lies in [pos, pos + len]
#pragma unroll
  for (int i = 0; i < kSearches; ++i) pos[i] = 0;
  for (long long len = n; len > 0;) {
    // probes at pos + (lane + 1) step - 1: those below the key are a prefix of the lanes
    const long long step = (len + 31) / 32;
    int v[kSearches];
#pragma unroll
    for (int i = 0; i < kSearches; ++i) {
      const long long q = (long long)pos[i] + (long long)(lane + 1) * step - 1;
      const int *f = reinterpret_cast<const int *>(R + min(q, n - 1)) + ((i == 1 || i == 3) ? 0 : ((i == 0 || i == 2) ? 1 : 2));
      v[i] = q < (long long)pos[i] + len && q < n ? __ldg(f) : 0x7fffffff;
    }
#pragma unroll
    for (int i = 0; i < kSearches; ++i)
      pos[i] += (int)(__popc(__ballot_sync(0xffffffffu, v[i] < key[i])) * step);
    len = step - 1;
  }
  const int lb = min(pos[0], (int)n), ub = max(lb, min(pos[1], (int)n));
  // change point `lane` (0, 1: the covering range; then the distances as searched; 12: ub)
  int mine = ub;
#pragma unroll
  for (int i = 0; i < 12; ++i)
    if (lane == i) mine = min(max(pos[i + 2], lb), ub);
  int c[12];
#pragma unroll
  for (int i = 0; i < 12; ++i) c[i] = __shfl_sync(0xffffffffu, mine, i);
  // in ascending order: lane r takes the r-th of the 13
  int rank = 0;
#pragma unroll
  for (int i = 0; i < 12; ++i) rank += (c[i] < mine || (c[i] == mine && i < lane)) ? 1 : 0;
  if (lane >= 12) rank = lane;
  int end = ub;
#pragma unroll
  for (int i = 0; i < 13; ++i) {
    const int e = __shfl_sync(0xffffffffu, mine, i), r = __shfl_sync(0xffffffffu, rank, i);
    if (r == lane) end = e;
  }
  const int prev = __shfl_up_sync(0xffffffffu, end, 1);
  const int start = lane == 0 ? lb : prev;
  auto beyond = [&](int q) { return start < c[2 + q] || start >= c[11 - q]; };
  int kd;
  if (start < c[0] || start >= c[1])
    kd = beyond(0) ? kSegEdge : (beyond(1) ? kSegFar1Masked : kSegGeneral);
  else
    kd = beyond(2) ? kSegNodes8 : (beyond(3) ? kSegNodes16 : (beyond(4) ? kSegFast : kSegGeneral));
  // one segment per maximal run of equal kind among the non-empty ranges: a range ends one
  // when the next non-empty range is of another kind
  const unsigned full = __ballot_sync(0xffffffffu, lane < 13 && end > start);
  const unsigned above = full & ~((2u << lane) - 1u);
  const int next_kd = __shfl_sync(0xffffffffu, kd, above ? __ffs(above) - 1 : 0);
  const bool last = ((full >> lane) & 1u) && (!above || next_kd != kd);
  const unsigned ends = __ballot_sync(0xffffffffu, last);
  // at most 12 of the 13: the change at d8 counts among covering lines, the one at D1 among the
  // others, and with d8 >= D1 they never both count (searches of one field end in the order of
  // their keys, sorted lines or not)
  const int nseg = __popc(ends);
  const int seg = __popc(ends & ((1u << lane) - 1u));
  int *o = reinterpret_cast<int *>(out + kTileInts * t);
  unsigned char *kinds = reinterpret_cast<unsigned char *>(o + 16);
  if (lane < 16) kinds[lane] = 0;
  if (lane >= nseg && lane < kMaxSegs) o[4 + lane] = ub;
  __syncwarp();
  if (last) {
    o[4 + seg] = end;
    kinds[seg] = (unsigned char)kd;
  }
  if (lane == 0) *reinterpret_cast<int4 *>(o) = make_int4(lb, ub, nseg, 0);
}

__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Paired binary32 arithmetic (one f32x2 instruction for two lanes' worth of
// work): each component is rounded exactly as the scalar __fmaf_rn /
// __fadd_rn, so the paired forms give the same bits as the scalar ones.
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 rcp2(float2 d) { return make_float2(rcp_approx(d.x), rcp_approx(d.y)); }

// compensated (Kahan) add of v into s with running compensation c, per component
__device__ __forceinline__ void kahan_add2(float2 &s, float2 &c, float2 v) {
  const float2 y = __fadd2_rn(v, neg2(c));
  const float2 t = __fadd2_rn(s, y);
  c = __fadd2_rn(__fadd2_rn(t, neg2(s)), neg2(y));
  s = t;
}
// the same for a v that may exceed s (Knuth's two-sum)
__device__ __forceinline__ void two_sum_add2(float2 &s, float2 &c, float2 v) {
  const float2 y = __fadd2_rn(v, neg2(c));
  const float2 t = __fadd2_rn(s, y);
  const float2 yy = __fadd2_rn(t, neg2(s));
  const float2 ss = __fadd2_rn(t, neg2(yy));
  c = __fadd2_rn(__fadd2_rn(ss, neg2(s)), __fadd2_rn(yy, neg2(y)));
  s = t;
}

// Block = 256 consecutive wavenumbers x up to 8 temperature nodes (one warp per
// node, 8 consecutive points per lane).  All warps walk the same lines: the
// block's lines are staged chunk by chunk (geometry R once, coefficients P and,
// where a kind needs them, P2 per node) with bulk asynchronous copies on an mbarrier,
// double buffered.  A point's or node's offset from a line centre, in grid units, is exact
// but for one rounding of the centre's sub-grid offset, so its rounding error is relative
// to the distance itself.
// Voigt far wing (|z| >= 20): with t = 1/|z|^2 the three-term series is the
// polynomial c0 t + c1 t^2 + c2 t^3 + c3 t^4 + c4 t^5 (coefficients from
// k_line_setup).  The binary32 arithmetic runs on pairs of points, nodes or lines (f32x2
// instructions).  By kind: far lines at 8 or 16 nodes of the tile, several lines per warp at
// a time; lines whose window ends in the tile at 4 nodes of the covered sub-blocks plus the
// points of the one it ends in; fast lines at every point, kGroup per compensated add;
// general lines by a five-term series with the points |z| < 8 replaced by the rational
// series, window ends masked, added in pairs.
// Lorentz: P = {A g / (pi dnu), g^2}.
// Of the 2560 lines a tile of the 128^3 workload sums (64 T x 400k points, 100k lines), 2000
// cost 8 evaluations, 280 16, 128 about 64 and 134 256 each instead of 256 each: 16.2 -> 4.6
// ms (32^3 workload 1.89 -> 0.91 ms).  Of the 4.6, by timing copies that leave a kind out:
// general lines 2.2 (their core points 1.2), window ends 0.8, 8 nodes 0.35, fast 0.35, 16 nodes
// 0.2, interpolation 0.07, chunks and barriers the rest; the FMA pipe (a paired FMA takes two
// of its cycles) and issue bound it, the reciprocals no longer do.  A barrier a chunk keeps the
// warps on the same code: with the buffers handed on warp by warp instead 3 % slower.
// ADAPT: every line has its own window at each node (AW, within the cutoff window), staged
// with the coefficients.  A warp sorts each range's lines by its node's windows (ballots):
// lines whose window holds the tile go the range's way, lines whose window ends in it the
// masked or window-end way, the others cost nothing more.  64 T x 100k points, 20k lines,
// kappa_min 1e-3: 0.98 ms, where a gather over each tile's kept lines took 4.24.
template <int PROFILE, bool ADAPT>
__global__ void __launch_bounds__(32 * kMaxTPerBlock, 3)
k_kappa(const float4 *__restrict__ P, const float4 *__restrict__ P2, const int4 *__restrict__ R,
        const int2 *__restrict__ AW,
        const int4 *__restrict__ tiles, long long n_lines, long long n_nu, int nT,
        const __grid_constant__ WeidSet ws,
        int vec_ok, int accumulate, float *__restrict__ kappa, uint32_t *status) {
  constexpr bool kVoigt = PROFILE == RT_PROFILE_VOIGT;
  constexpr int kCap = ADAPT ? 128 : kChunk, kCapP2 = kCap / 2;  // lines of a chunk: P only, P and P2
  constexpr int kFull = kVoigt ? kCapP2 : kCap;                  // lines of a chunk of any kind
  __shared__ __align__(16) int4 sR[2][kCap];
  __shared__ __align__(16) float4 sP[2][kMaxTPerBlock][kCap];  // P, and P2 from kCapP2 on
  // windows at the node (16-byte copies: one element of margin each side); a warp's lists of
  // chunk lines: covering; ending in the tile from the front, masked ones from the back
  __shared__ __align__(16) int2 sW[2][ADAPT ? kMaxTPerBlock : 1][ADAPT ? kCap + 2 : 2];
  __shared__ unsigned char s_list[ADAPT ? kMaxTPerBlock : 1][2][ADAPT ? kCap : 1];
  __shared__ __align__(8) uint64_t bars[2];
  __shared__ __align__(16) float s_res[kMaxTPerBlock][2 * kTilePts];  // a warp's core values or node sums

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tpb = blockDim.x >> 5;
  const int k0 = blockIdx.y * tpb;
  const int nk = min(tpb, nT - k0);          // T nodes of this block
  const int k = k0 + min(warp, nk - 1);      // surplus warps shadow the last node, store nothing
  const long long j0 = (long long)blockIdx.x * kTilePts;
  const long long jend = min(j0 + (long long)kTilePts, n_nu);
  const int jw0 = (int)j0, jw1 = jw0 + kTilePts - 1;
  const int jt = jw0 + lane * kPtsPerThread;
  // Lorentz lines with windows of their own add the sub-grid offset last at each point, a rounding
  // less (1 % of the tables' error); the other paths add the points to the lane's first offset.
  constexpr bool kExactU = ADAPT && !kVoigt;
  // offset of point j from a line centre j_c with sub-grid offset dg: the exact
  // integer difference, then one rounding
  auto point_offset = [&](int j, int jc, int dg_bits) -> float {
    return __fadd_rn((float)(j - jc), __int_as_float(dg_bits));
  };

  __shared__ int s_end[kMaxSegs];
  __shared__ unsigned char s_kind[kMaxSegs];
  const int4 *tinfo = tiles + (long long)kTileInts * blockIdx.x;
  const int4 ta = __ldg(tinfo);
  const int lb = ta.x, ub = ta.y;
  if (threadIdx.x < kMaxSegs) {
    const int q = threadIdx.x & 3;
    const int4 e = __ldg(tinfo + 1 + (threadIdx.x >> 2));
    const int4 kw = __ldg(tinfo + 4);
    const int w = (threadIdx.x >> 2) == 0 ? kw.x : ((threadIdx.x >> 2) == 1 ? kw.y : kw.z);
    s_end[threadIdx.x] = q == 0 ? e.x : (q == 1 ? e.y : (q == 2 ? e.z : e.w));
    s_kind[threadIdx.x] = (unsigned char)((w >> (8 * q)) & 255);
  }
  if (threadIdx.x == 0) {
    mbar_init(&bars[0], 1);
    mbar_init(&bars[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  // Chunks: the last kFull lines or fewer in one; else lines of one degree-1 range (P only),
  // kCap at most, or the next kFull lines.  sg: the segment of line l, carried along.
  auto chunk_at = [&](int l, int &sg, bool &with_p2) -> int {
    while (s_end[sg] <= l) ++sg;  // the last segment ends at ub > l
    with_p2 = kVoigt;
    if (ub - l <= kFull) return ub - l;
    if (!degree1_kind(s_kind[sg])) return kFull;
    with_p2 = false;
    return min(kCap, s_end[sg] - l);
  };
  // copies of the chunk at line l into buffer b, issued by the lanes of warp 0: R, then P (and
  // P2) of one node each
  auto issue = [&](int l, int cnt, bool with_p2, int b) {
    const uint32_t bytes = (uint32_t)cnt * 16u;
    // windows: from the 16-byte boundary at or below the node's first to the one past its last
    const long long w0 = (long long)(k0 + lane) * n_lines + l;
    const uint32_t wbytes = ADAPT && lane < nk ? (uint32_t)(((int)(w0 & 1) + cnt + 1) >> 1) * 16u : 0u;
    const uint32_t wall = ADAPT ? __reduce_add_sync(0xffffffffu, wbytes) : 0u;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (lane == 0) {
      mbar_arrive_expect_tx(&bars[b], bytes * (uint32_t)(nk * (with_p2 ? 2 : 1) + 1) + wall);
      bulk_g2s(&sR[b][0], R + l, bytes, &bars[b]);
    }
    __syncwarp();
    if (lane < nk) {
      bulk_g2s(&sP[b][lane][0], P + (long long)(k0 + lane) * n_lines + l, bytes, &bars[b]);
      if (ADAPT) bulk_g2s(&sW[b][lane][0], AW + (w0 & ~1LL), wbytes, &bars[b]);
      if (with_p2) bulk_g2s(&sP[b][lane][kCapP2], P2 + (long long)(k0 + lane) * n_lines + l, bytes, &bars[b]);
    }
  };

  // compensated sums for the lane's points, as pairs (2h, 2h + 1)
  constexpr int kPairs = kPtsPerThread / 2;
  float2 acc[kPairs], cmp[kPairs];
#pragma unroll
  for (int h = 0; h < kPairs; ++h) acc[h] = cmp[h] = make_float2(0.0f, 0.0f);
  // sums of the interpolated lines at the lane's two nodes: 8 nodes (lane & 3) over every
  // eighth line, 16 nodes (lane & 7) over every fourth
  float2 n8 = make_float2(0.0f, 0.0f), n8c = n8, n16 = n8, n16c = n8;
  bool nodes = false;
  // warp 0 issues chunks up to two ahead of the one being summed
  int pl = lb, pseg = 0, issued = 0;
  auto issue_next = [&]() {
    if (pl >= ub) return;
    bool with_p2;
    const int cnt = chunk_at(pl, pseg, with_p2);
    issue(pl, cnt, with_p2, issued & 1);
    pl += cnt;
    ++issued;
  };
  if (warp == 0) {
    issue_next();
    issue_next();
  }
  const int wsel = min(warp, nk - 1);
  int seg = 0;  // current segment, carried across chunks
  bool aborted = false;
  int cnt = 0;
  for (int c = 0, l0 = lb; l0 < ub; ++c, l0 += cnt) {
    const int b = c & 1;
    const uint32_t parity = (uint32_t)((c >> 1) & 1);
    unsigned spins = 0;
    int timed_out = 0;
    while (!mbar_try_wait(&bars[b], parity)) {
      if (++spins > kWaitLimit) {
        timed_out = 1;
        break;
      }
    }
    timed_out = __any_sync(0xffffffffu, timed_out);  // warp-uniform: such a warp sums nothing
    bool with_p2;
    cnt = chunk_at(l0, seg, with_p2);
    const int4 *cR = sR[b];
    const float4 *cP = sP[b][wsel], *cP2 = cP + kCapP2;
    const int2 *cW = sW[b][ADAPT ? wsel : 0] + (ADAPT ? (((long long)k * n_lines + l0) & 1) : 0);
    // line i's window: its own at this node, or the cutoff's
    auto window = [&](int i) -> int2 { return ADAPT ? cW[i] : *reinterpret_cast<const int2 *>(&cR[i].x); };

    // the line's value at a pair of offsets u (grid units) from its centre; DEG 4 or 1: the far-wing series' degree
    auto far_value = [&](auto deg, float2 u, const float4 &p, int i) -> float2 {
      constexpr int DEG = decltype(deg)::value;
      if (!kVoigt) return __fmul2_rn(dup2(p.x), rcp2(__ffma2_rn(u, u, dup2(p.y))));
      const float2 c0 = dup2(p.x), c1 = dup2(1.5f * p.x);
      const float2 x = __fmul2_rn(dup2(p.y), u);
      const float2 t = rcp2(__ffma2_rn(x, x, dup2(p.z)));
      if (DEG == 4) {
        const float4 p2 = cP2[i];
        return __fmul2_rn(t, __ffma2_rn(t, __ffma2_rn(t, __ffma2_rn(t, __ffma2_rn(t, dup2(p2.y), dup2(p2.x)), dup2(p.w)), c1), c0));
      }
      return __fmul2_rn(t, __ffma2_rn(t, c1, c0));
    };
    // Below, a range's lines are at(0) .. at(n - 1), chunk indices.
    // run_nodes: at the M tile nodes: M / 2 lanes take a line (two nodes each), the warp
    // 64 / M lines at a time; whole groups without bounds checks (with them 4.99 ms of the
    // 128^3 workload, 4.72 without)
    auto run_nodes = [&](auto deg, auto m, const float *un, auto at, int n, float2 &s, float2 &sc) {
      constexpr int kLanes = decltype(m)::value / 2, kLines = 32 / kLanes;
      const float2 u0 = *reinterpret_cast<const float2 *>(un + 2 * (lane % kLanes));
      auto value = [&](int e) -> float2 {
        const int q = at(e);
        const int2 r = *reinterpret_cast<const int2 *>(&cR[q].z);
        const float2 u = __fadd2_rn(__fadd2_rn(dup2((float)(jw0 - r.x)), u0), dup2(__int_as_float(r.y)));
        return far_value(deg, u, cP[q], q);
      };
      int i = lane / kLanes, left = n;
#pragma unroll 1
      for (; left >= kLines * kNodeGroup; left -= kLines * kNodeGroup, i += kLines * kNodeGroup) {
        float2 g = value(i);
#pragma unroll
        for (int e = 1; e < kNodeGroup; ++e) g = __fadd2_rn(g, value(i + e * kLines));
        kahan_add2(s, sc, g);
      }
      if (left > 0) {
        float2 g = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int e = 0; e < kNodeGroup; ++e) {
          const bool in = i + e * kLines < n;
          const float2 v = value(in ? i + e * kLines : n - 1);
          if (in) g = __fadd2_rn(g, v);
        }
        kahan_add2(s, sc, g);
      }
      nodes = true;
    };
    // lines whose windows end inside the tile (on one side), one after the other: lane (b, m) takes
    // node m of sub-block b where the window covers it, and point `lane` of the sub-block the
    // window ends in.  Both sums go to the points before returning.
    auto run_edge = [&](auto at, int n) {
      float *res = s_res[warp];
      const int sb = lane >> 2, nu_last = (int)(n_nu - 1);
      const float un = 32.0f * (float)sb + kTab4.u[lane & 3];
      float2 s = make_float2(0.0f, 0.0f), sc = s;
#pragma unroll
      for (int q = 0; q < (ADAPT ? 2 : 1) * kPtsPerThread; ++q) res[32 * q + lane] = 0.0f;
      int cur = -1;
      // the sum of the lines that end in sub-block cur is put away: cutoff windows end in a
      // sub-block once, windows of their own any number of times, so their sums wait with their
      // compensation (the second half of res) for the next line that ends there
      auto flush = [&]() {
        if (cur >= 0 && cur < kTilePts / 32) {
          float &r = res[32 * cur + lane];
          if (ADAPT) {
            r = s.y;
            res[kTilePts + 32 * cur + lane] = sc.y;
          } else {
            r += __fsub_rn(s.y, sc.y);
          }
        }
        s.y = sc.y = 0.0f;
      };
#pragma unroll 1
      for (int q = 0; q < n; ++q) {
        const int i = at(q);
        const int4 r = cR[i];
        const int2 win = window(i);
        // covered tile points; a window that holds the grid's last point has no end here
        const int a = max(win.x - jw0, 0), e = win.y >= nu_last ? kTilePts - 1 : min(win.y - jw0, kTilePts - 1);
        const int eb = a == 0 ? (e + 1) >> 5 : a >> 5;                      // sub-block of the end
        if (eb != cur) {  // warp-uniform; cutoff windows' ends are monotone in the line index
          flush();
          cur = eb;
          if (ADAPT && cur >= 0 && cur < kTilePts / 32) {
            s.y = res[32 * cur + lane];
            sc.y = res[kTilePts + 32 * cur + lane];
          }
        }
        const int pt = 32 * eb + lane;
        const float2 u = __fadd2_rn(__fadd2_rn(dup2((float)(jw0 - r.z)), make_float2(un, (float)pt)), dup2(__int_as_float(r.w)));
        float2 v = far_value(std::integral_constant<int, 1>(), u, cP[i], i);
        if (32 * sb < a || 32 * sb + 31 > e) v.x = 0.0f;
        if (pt < a || pt > e || (32 * eb >= a && 32 * eb + 31 <= e)) v.y = 0.0f;
        kahan_add2(s, sc, v);
      }
      flush();
      __syncwarp();
      const float f = __fsub_rn(s.x, sc.x);
      float fm[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) fm[m] = __shfl_sync(0xffffffffu, f, (lane & ~3) + m);
      const int p0 = lane * kPtsPerThread, w0 = p0 & 31;
#pragma unroll
      for (int h = 0; h < kPairs; ++h) {
        float2 v = *reinterpret_cast<const float2 *>(res + p0 + 2 * h);
        v = __fadd2_rn(v, dup2(fm[1]));  // interpolate the differences to one node's value
#pragma unroll
        for (int m = 0; m < 4; ++m)
          if (m != 1)
            v = __ffma2_rn(*reinterpret_cast<const float2 *>(&kTab4.w[m][w0 + 2 * h]), dup2(fm[m] - fm[1]), v);
        if (ADAPT) v = __fadd2_rn(v, neg2(*reinterpret_cast<const float2 *>(res + kTilePts + p0 + 2 * h)));
        two_sum_add2(acc[h], cmp[h], v);
      }
      __syncwarp();  // res is the general path's next
    };

    // fast paths: g[q] += value of line i at the lane's points (or = when first).
    // DEG 4: full far-wing series; DEG 1: far lines; MASK: zero outside the line's window.
    auto fast_line = [&](auto deg, auto mask, int i, float2 (&g)[kPairs], bool first) {
      constexpr int DEG = decltype(deg)::value;
      constexpr bool MASK = decltype(mask)::value;
      int4 r = cR[i];
      if (MASK && ADAPT) r.x = cW[i].x, r.y = cW[i].y;
      const float4 p = cP[i];
      const float ul = point_offset(jt, r.z, r.w);
      if (!kVoigt) {
        const float2 u0 = dup2(kExactU ? (float)(jt - r.z) : ul), dg = dup2(__int_as_float(r.w));
        const float2 g2 = dup2(p.y), a2 = dup2(p.x);
#pragma unroll
        for (int h = 0; h < kPairs; ++h) {
          float2 u = __fadd2_rn(u0, make_float2((float)(2 * h), (float)(2 * h + 1)));
          if (kExactU) u = __fadd2_rn(u, dg);
          float2 rr = rcp2(__ffma2_rn(u, u, g2));
          if (MASK) {
            if (jt + 2 * h < r.x || jt + 2 * h > r.y) rr.x = 0.0f;
            if (jt + 2 * h + 1 < r.x || jt + 2 * h + 1 > r.y) rr.y = 0.0f;
          }
          g[h] = first ? __fmul2_rn(a2, rr) : __ffma2_rn(a2, rr, g[h]);
        }
      } else {
        const float2 c0 = dup2(p.x), c1 = dup2(1.5f * p.x), sd = dup2(p.y), y2 = dup2(p.z);
        const float2 xt = dup2(p.y * ul);
        float4 p2 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (DEG == 4) p2 = cP2[i];
#pragma unroll
        for (int h = 0; h < kPairs; ++h) {
          const float2 x = __ffma2_rn(sd, make_float2((float)(2 * h), (float)(2 * h + 1)), xt);
          const float2 t = rcp2(__ffma2_rn(x, x, y2));
          float2 v;
          if (DEG == 4)
            v = __ffma2_rn(t, __ffma2_rn(t, __ffma2_rn(t, __ffma2_rn(t, dup2(p2.y), dup2(p2.x)), dup2(p.w)), c1), c0);
          else
            v = __ffma2_rn(t, c1, c0);
          if (MASK) {
            if (jt + 2 * h < r.x || jt + 2 * h > r.y) v.x = 0.0f;
            if (jt + 2 * h + 1 < r.x || jt + 2 * h + 1 > r.y) v.y = 0.0f;
          }
          g[h] = first ? __fmul2_rn(t, v) : __ffma2_rn(t, v, g[h]);
        }
      }
    };
    auto run_fast = [&](auto deg, auto mask, auto at, int n) {
      int i = 0;
#pragma unroll 1
      for (; i + kGroup <= n; i += kGroup) {
        float2 g[kPairs];
        fast_line(deg, mask, at(i), g, true);
#pragma unroll
        for (int e = 1; e < kGroup; ++e) fast_line(deg, mask, at(i + e), g, false);
#pragma unroll
        for (int h = 0; h < kPairs; ++h) kahan_add2(acc[h], cmp[h], g[h]);
      }
      if (i < n) {
        float2 g[kPairs];
        fast_line(deg, mask, at(i), g, true);
#pragma unroll 1
        for (int e = i + 1; e < n; ++e) fast_line(deg, mask, at(e), g, false);
#pragma unroll
        for (int h = 0; h < kPairs; ++h) kahan_add2(acc[h], cmp[h], g[h]);
      }
    };

    // general path, two lines at a time (the second may be absent).  line_series: a line's
    // five-term series at the lane's points, valid for |z| >= 8; Lorentz: its value.
    auto line_series = [&](int i, float2 (&v)[kPairs]) {
      const int4 r = cR[i];
      const float4 p = cP[i];
      const float ul = point_offset(jt, r.z, r.w);
      if (!kVoigt) {
        const float2 u0 = dup2(kExactU ? (float)(jt - r.z) : ul), dg = dup2(__int_as_float(r.w));
        const float2 g2 = dup2(p.y), a2 = dup2(p.x);
#pragma unroll
        for (int h = 0; h < kPairs; ++h) {
          float2 u = __fadd2_rn(u0, make_float2((float)(2 * h), (float)(2 * h + 1)));
          if (kExactU) u = __fadd2_rn(u, dg);
          v[h] = __fmul2_rn(a2, rcp2(__ffma2_rn(u, u, g2)));
        }
        return;
      }
      const float4 p2 = cP2[i];
      // in t: the degree-4 polynomial plus 13.125 t^3, (59.0625 - 105 q) t^4 and the powers
      // above of the fourth and fifth terms, q = y^2 (see faddeeva_series5)
      const float q1 = p.z * p.x, q2 = p.z * q1, q3 = p.z * q2;
      const float2 y22 = dup2(p.z), sd = dup2(p.y), xt = dup2(p.y * ul);
      const float2 c8 = dup2(1680.0f * p.z * q3), c7 = dup2(-3780.0f * q3);
      const float2 c6 = dup2(__fmaf_rn(2835.0f, q2, -120.0f * q3)), c5 = dup2(__fmaf_rn(-787.5f, q1, 210.0f * q2));
      const float2 c4 = dup2(__fmaf_rn(59.0625f, p.x, __fmaf_rn(-105.0f, q1, p2.y)));
      const float2 c3 = dup2(__fmaf_rn(13.125f, p.x, p2.x)), c2 = dup2(p.w), c1 = dup2(1.5f * p.x), c0 = dup2(p.x);
#pragma unroll
      for (int h = 0; h < kPairs; ++h) {
        const float2 x = __ffma2_rn(sd, make_float2((float)(2 * h), (float)(2 * h + 1)), xt);
        const float2 t = rcp2(__ffma2_rn(x, x, y22));
        float2 w = __ffma2_rn(t, c8, c7);
        w = __ffma2_rn(t, __ffma2_rn(t, __ffma2_rn(t, w, c6), c5), c4);
        w = __ffma2_rn(t, __ffma2_rn(t, __ffma2_rn(t, __ffma2_rn(t, w, c3), c2), c1), c0);
        v[h] = __fmul2_rn(t, w);
      }
    };
    // the tile points with |z| < 8 of line i: |u| <= u_core, the contiguous indices
    // [first, first + n) (warp-uniform)
    auto core_range = [&](int i, int &first) -> int {
      const int2 r = *reinterpret_cast<const int2 *>(&cR[i].z);
      const float fu = (float)(jw0 - r.x) + __int_as_float(r.y), uc = cP2[i].w;
      first = (int)fmaxf(ceilf(-uc - fu), 0.0f);
      const int last = (int)fminf(floorf(uc - fu), (float)(kTilePts - 1));
      return uc > 0.0f ? last - first + 1 : 0;
    };
    // Those points by Weideman's rational series, one lane a point, two lines in one paired
    // pass (a line has 16 to 40 such points on a 0.005 cm^-1 grid: 32 lanes take them in one
    // or two passes), into shared memory for their owners.
    auto core_values = [&](int ia, int ib, int fa, int fb, int n) {
      const float4 pa = cP[ia], pb = cP[ib];
      const int2 ra = *reinterpret_cast<const int2 *>(&cR[ia].z), rb = *reinterpret_cast<const int2 *>(&cR[ib].z);
      const float2 y = make_float2(cP2[ia].z, cP2[ib].z);
      const float2 coef = make_float2(__fdividef(pa.x, y.x), __fdividef(pb.x, y.y));
      const float2 sd = make_float2(pa.y, pb.y), dg = make_float2(__int_as_float(ra.y), __int_as_float(rb.y));
      const float2 first = make_float2((float)(jw0 + fa - ra.x), (float)(jw0 + fb - rb.x));
      float *res = s_res[warp];  // the first line's at 0, the second's at kTilePts
      auto points = [&](auto &wc) {
        constexpr int N = sizeof(wc.a) / sizeof(float);
        const float2 dr = __fadd2_rn(dup2(wc.L), y), nr = __fadd2_rn(dup2(wc.L), neg2(y));
#pragma unroll 1
        for (int e = lane; e < n; e += 32) {
          const float2 x = __fmul2_rn(sd, __fadd2_rn(__fadd2_rn(first, dup2((float)e)), dg));
          // iz = -y + ix, v = 1 / (L - iz), Z = (L + iz) v; sqrt(pi) w = v (p(Z) v + 1)
          const float2 d = __ffma2_rn(dr, dr, __fmul2_rn(x, x));
          float2 inv = rcp2(d);  // one Newton step: the tables are no further from binary64 than by division
          inv = __ffma2_rn(inv, __ffma2_rn(neg2(d), inv, dup2(1.0f)), inv);
          const float2 vr = __fmul2_rn(dr, inv), vi = __fmul2_rn(x, inv);
          const float2 zr = __ffma2_rn(nr, vr, neg2(__fmul2_rn(x, vi))), zi = __ffma2_rn(nr, vi, __fmul2_rn(x, vr));
          const float2 nzi = neg2(zi);
          float2 pr = dup2(wc.a[N - 1]), pi = make_float2(0.0f, 0.0f);
#pragma unroll
          for (int n = N - 2; n >= 0; --n) {
            const float2 t = __ffma2_rn(pr, zr, __ffma2_rn(pi, nzi, dup2(wc.a[n])));
            pi = __ffma2_rn(pr, zi, __fmul2_rn(pi, zr));
            pr = t;
          }
          const float2 nvi = neg2(vi);
          const float2 qr = __fadd2_rn(__ffma2_rn(pr, vr, __fmul2_rn(pi, nvi)), dup2(1.0f));
          const float2 qi = __ffma2_rn(pr, vi, __fmul2_rn(pi, vr));
          const float2 w = __fmul2_rn(coef, __ffma2_rn(vr, qr, __fmul2_rn(nvi, qi)));
          res[e] = w.x;
          res[kTilePts + e] = w.y;
        }
      };
      // fewer terms where the line is broad (warp-uniform; see WeidSet)
      const float ymin = fminf(y.x, y.y);
      if (ymin >= kTerms12) points(ws.n12);
      else if (ymin >= kTerms16) points(ws.n16);
      else points(ws.n24);
      __syncwarp();
    };
    // the lane's points among the n core points from tile point `first` on, from res + c
    auto take_core = [&](int c, int first, int n, float2 (&v)[kPairs]) {
      const int a = lane * kPtsPerThread - first;  // the lane's first point in res
      if (a + kPtsPerThread <= 0 || a >= n) return;
      const float *res = s_res[warp] + c + a;
#pragma unroll
      for (int h = 0; h < kPairs; ++h) {
        if ((unsigned)(a + 2 * h) < (unsigned)n) v[h].x = res[2 * h];
        if ((unsigned)(a + 2 * h + 1) < (unsigned)n) v[h].y = res[2 * h + 1];
      }
    };
    auto mask_window = [&](int i, float2 (&v)[kPairs]) {
      const int2 r = window(i);
      if (r.x > jw0 || r.y < jw1) {  // warp-uniform: the window ends inside this block's points
#pragma unroll
        for (int h = 0; h < kPairs; ++h) {
          if (jt + 2 * h < r.x || jt + 2 * h > r.y) v[h].x = 0.0f;
          if (jt + 2 * h + 1 < r.x || jt + 2 * h + 1 > r.y) v[h].y = 0.0f;
        }
      }
    };
    // lines enter the compensated sum in pairs: the sum of two positive line
    // values is rounded once (relative error <= 2^-24 of the pair)
    auto run_general = [&](auto at, int n) {
      int q0 = 0;
      if (!kVoigt) {  // four lines at a time: a grid of few tiles is bound by the latency of a pair
#pragma unroll 1
        for (; q0 + 4 <= n; q0 += 4) {
          float2 v[2][kPairs], w[kPairs];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int i = at(q0 + 2 * e), j = at(q0 + 2 * e + 1);
            line_series(i, v[e]);
            mask_window(i, v[e]);
            line_series(j, w);
            mask_window(j, w);
#pragma unroll
            for (int h = 0; h < kPairs; ++h) v[e][h] = __fadd2_rn(v[e][h], w[h]);
          }
#pragma unroll
          for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int h = 0; h < kPairs; ++h) kahan_add2(acc[h], cmp[h], v[e][h]);
        }
      }
#pragma unroll 1
      for (int q = q0; q < n; q += 2) {
        const bool two = q + 1 < n;
        const int i = at(q), j = two ? at(q + 1) : i;
        int fa = 0, fb = 0, na = 0, nb = 0;
        if (kVoigt) {
          na = core_range(i, fa);
          nb = two ? core_range(j, fb) : 0;
          if (max(na, nb) > 0) core_values(i, j, fa, fb, max(na, nb));
        }
        float2 v[kPairs], w[kPairs];
        line_series(i, v);
        if (na > 0) take_core(0, fa, na, v);
        mask_window(i, v);
        if (two) {
          line_series(j, w);
          if (nb > 0) take_core(kTilePts, fb, nb, w);
          mask_window(j, w);
#pragma unroll
          for (int h = 0; h < kPairs; ++h) v[h] = __fadd2_rn(v[h], w[h]);
        }
        __syncwarp();  // res is the next lines'
#pragma unroll
        for (int h = 0; h < kPairs; ++h) kahan_add2(acc[h], cmp[h], v[h]);
      }
    };

    // the chunk [l0, l0 + cnt) split at the tile's segment ends (block-uniform)
    int i = timed_out ? cnt : 0;
#pragma unroll 1
    while (i < cnt) {
      const int l = l0 + i;
      while (s_end[seg] <= l) ++seg;  // the last segment ends at ub > l
      const int i1 = min(cnt, s_end[seg] - l0);
      const int kd = s_kind[seg];
      const std::integral_constant<int, 1> d1;
      const std::integral_constant<int, 4> d4;
      const std::integral_constant<int, 8> m8;
      const std::integral_constant<int, 16> m16;
      const std::false_type all;
      const std::true_type masked;
      if (!ADAPT) {
        const int n = i1 - i;
        auto at = [i](int e) { return i + e; };
        if (kd == kSegNodes8) run_nodes(d1, m8, kTab8.u, at, n, n8, n8c);
        else if (kd == kSegNodes16) run_nodes(d4, m16, kTab16.u, at, n, n16, n16c);
        else if (kd == kSegEdge) run_edge(at, n);
        else if (kd == kSegFast) run_fast(d4, all, at, n);
        else if (kd == kSegFar1Masked) run_fast(d1, masked, at, n);
        else run_general(at, n);
      } else {
        // a general line goes with the covering ones (its path masks), a degree-1 line far
        // enough for the sub-blocks' nodes with the window ends, the rest are masked
        unsigned char *lc = s_list[warp][0], *lp = s_list[warp][1];
        int nc = 0, ne = 0, nm = 0;
        const int last = (int)min((long long)jw1, n_nu - 1);
        for (int q0 = i; q0 < i1; q0 += 32) {
          const int q = q0 + lane;
          int to = 0;  // 0 none, 1 covering, 2 window end, 3 masked
          if (q < i1) {
            const int2 w = cW[q];
            const int jc = cR[q].z;
            if (w.y >= w.x && w.y >= jw0 && w.x <= last) {
              if (kd == kSegGeneral || (w.x <= jw0 && w.y >= last)) to = 1;
              else to = degree1_kind(kd) && max(jw0 - jc, jc - jw1) >= kDistEdge ? 2 : 3;
            }
          }
          const unsigned lt = (1u << lane) - 1u;
          const unsigned c = __ballot_sync(0xffffffffu, to == 1), e = __ballot_sync(0xffffffffu, to == 2),
                         m = __ballot_sync(0xffffffffu, to == 3);
          if (to == 1) lc[nc + __popc(c & lt)] = (unsigned char)q;
          if (to == 2) lp[ne + __popc(e & lt)] = (unsigned char)q;
          if (to == 3) lp[kCap - 1 - nm - __popc(m & lt)] = (unsigned char)q;
          nc += __popc(c);
          ne += __popc(e);
          nm += __popc(m);
        }
        __syncwarp();
        auto cover = [lc](int e) { return (int)lc[e]; };
        auto ends = [lp](int e) { return (int)lp[e]; };
        auto rest = [lp](int e) { return (int)lp[kCap - 1 - e]; };
        if (kd == kSegGeneral) {
          run_general(cover, nc);
        } else if (degree1_kind(kd)) {
          if (nc > 0) run_nodes(d1, m8, kTab8.u, cover, nc, n8, n8c);
          if (ne > 0) run_edge(ends, ne);
          run_fast(d1, masked, rest, nm);
        } else {
          if (kd == kSegFast) run_fast(d4, all, cover, nc);
          else if (nc > 0) run_nodes(d4, m16, kTab16.u, cover, nc, n16, n16c);
          run_fast(d4, masked, rest, nm);
        }
        __syncwarp();  // the lists are the next range's
      }
      i = i1;
    }
    // every warp is done with buffer b (the waits above order each thread's own reads)
    if (__syncthreads_or(timed_out)) {  // the block leaves together
      if (threadIdx.x == 0) {
        status_or(status, RT_DEV_TIMEOUT);
        // The copies of this chunk and of the next one (issued one chunk ahead) may
        // still be writing into this block's shared memory: wait for them, again with
        // a bound, so that no copy lands after the block has released it.
        for (int d = c; d < issued; ++d) {
          unsigned n = 0;
          while (!mbar_try_wait(&bars[d & 1], (uint32_t)((d >> 1) & 1)) && ++n <= kWaitLimit) {
          }
        }
      }
      aborted = true;
      break;
    }
    if (warp == 0) issue_next();
  }
  if (aborted || warp >= nk) return;

  if (nodes) {  // warp-uniform: the interpolated lines' node sums to the lane's points
    // as hi + lo pairs throughout, so that the interpolation adds next to nothing to the
    // rounding error of the line values themselves
    float2 f8 = n8, l8 = neg2(n8c), f16 = n16, l16 = neg2(n16c);
    auto two_sum2 = [](float2 &hi, float2 &lo, float2 v) {  // hi + lo += v
      const float2 t = __fadd2_rn(hi, v), vv = __fadd2_rn(t, neg2(hi)), hh = __fadd2_rn(t, neg2(vv));
      lo = __fadd2_rn(lo, __fadd2_rn(__fadd2_rn(hi, neg2(hh)), __fadd2_rn(v, neg2(vv))));
      hi = t;
    };
    auto add_lanes = [&](float2 &hi, float2 &lo, int o) {
      lo = __fadd2_rn(lo, make_float2(__shfl_xor_sync(0xffffffffu, lo.x, o), __shfl_xor_sync(0xffffffffu, lo.y, o)));
      two_sum2(hi, lo, make_float2(__shfl_xor_sync(0xffffffffu, hi.x, o), __shfl_xor_sync(0xffffffffu, hi.y, o)));
    };
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) add_lanes(f8, l8, o);
#pragma unroll
    for (int o = 8; o < 32; o <<= 1) add_lanes(f16, l16, o);
    // the 8-node interpolant at the lane's two of the 16 nodes; only differences to one
    // node's value are weighted, so that the weights' signs cost no accuracy
    const int p16 = 2 * (lane & 7);
    const float r8 = __shfl_sync(0xffffffffu, f8.x, 2), rl8 = __shfl_sync(0xffffffffu, l8.x, 2);
    float2 d8 = dup2(rl8);
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const float f = __shfl_sync(0xffffffffu, (m & 1) ? f8.y : f8.x, m >> 1) - r8;
      const float l = __shfl_sync(0xffffffffu, (m & 1) ? l8.y : l8.x, m >> 1) - rl8;
      d8 = __ffma2_rn(*reinterpret_cast<const float2 *>(&kTab8.w[m][p16]), dup2(f + l), d8);
    }
    two_sum2(f16, l16, dup2(r8));
    two_sum2(f16, l16, d8);
    float *res = s_res[warp];
    __syncwarp();
    if (lane < 8) {
      *reinterpret_cast<float2 *>(res + p16) = f16;
      *reinterpret_cast<float2 *>(res + 16 + p16) = l16;
    }
    __syncwarp();
    const float ref = res[8], refl = res[16 + 8];
    float2 v[kPairs];
#pragma unroll
    for (int h = 0; h < kPairs; ++h) v[h] = dup2(refl);
    const int p0 = lane * kPtsPerThread;
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const float2 f = dup2((res[m] - ref) + (res[16 + m] - refl));
      const float4 wa = *reinterpret_cast<const float4 *>(&kTab16.w[m][p0]);
      const float4 wb = *reinterpret_cast<const float4 *>(&kTab16.w[m][p0 + 4]);
      v[0] = __ffma2_rn(make_float2(wa.x, wa.y), f, v[0]);
      v[1] = __ffma2_rn(make_float2(wa.z, wa.w), f, v[1]);
      v[2] = __ffma2_rn(make_float2(wb.x, wb.y), f, v[2]);
      v[3] = __ffma2_rn(make_float2(wb.z, wb.w), f, v[3]);
    }
#pragma unroll
    for (int h = 0; h < kPairs; ++h) {
      two_sum_add2(acc[h], cmp[h], dup2(ref));
      two_sum_add2(acc[h], cmp[h], v[h]);
    }
  }

  float *row = kappa + (long long)k * n_nu;
  float out[kPtsPerThread];
#pragma unroll
  for (int h = 0; h < kPairs; ++h) {
    out[2 * h] = __fsub_rn(acc[h].x, cmp[h].x);
    out[2 * h + 1] = __fsub_rn(acc[h].y, cmp[h].y);
  }
  if ((long long)jt + kPtsPerThread <= jend && vec_ok) {
#pragma unroll
    for (int q4 = 0; q4 < kPtsPerThread; q4 += 4) {
      float4 *dst = reinterpret_cast<float4 *>(row + jt + q4);
      if (accumulate) {
        const float4 o = *dst;
        out[q4] += o.x; out[q4 + 1] += o.y; out[q4 + 2] += o.z; out[q4 + 3] += o.w;
      }
      *dst = make_float4(out[q4], out[q4 + 1], out[q4 + 2], out[q4 + 3]);
    }
  } else {
#pragma unroll
    for (int q = 0; q < kPtsPerThread; ++q)
      if ((long long)jt + q < jend) row[jt + q] = accumulate ? row[jt + q] + out[q] : out[q];
  }
}

// Fixed points per line (each line on the few grid points around its centre):
// one thread per point j, looping over kPplNodes T nodes; the lines whose windows
// hold j are a contiguous index range (windows are monotone in the sorted line
// index), found once per thread by binary search within the block's range, and
// summed in ascending nu0 with compensation at each node.  Every point is near its
// lines' centres, so each value is the near-centre form (faddeeva_re_near) rather
// than a far-wing series.
constexpr int kPplNodes = 8;

template <int PROFILE>
__global__ void __launch_bounds__(kTilePts)
k_kappa_ppl(const float4 *__restrict__ P, const int4 *__restrict__ R, long long n_lines, long long n_nu,
            int nT, WeidCoef wc, int accumulate, float *__restrict__ kappa) {
  __shared__ long long s_range[2];
  const long long jw0 = (long long)blockIdx.x * kTilePts;
  const long long jend = min(jw0 + (long long)kTilePts, n_nu);
  const int k0 = blockIdx.y * kPplNodes, k1 = min(k0 + kPplNodes, nT);
  if (threadIdx.x == 0) s_range[0] = lower_bound_hi(R, n_lines, (int)jw0);
  if (threadIdx.x == 1) s_range[1] = lower_bound_lo(R, n_lines, (int)jend);
  __syncthreads();
  const long long j = jw0 + threadIdx.x;
  if (j >= n_nu) return;
  // lines [a, b) of the block's range with hi >= j and lo <= j
  long long a = s_range[0], hi_end = max(s_range[0], s_range[1]);
  while (a < hi_end) {
    const long long m = (a + hi_end) >> 1;
    if (__ldg(&R[m].y) < (int)j) a = m + 1; else hi_end = m;
  }
  long long b = a, b_end = max(s_range[0], s_range[1]);
  while (b < b_end) {
    const long long m = (b + b_end) >> 1;
    if (__ldg(&R[m].x) <= (int)j) b = m + 1; else b_end = m;
  }
#pragma unroll 1
  for (int k = k0; k < k1; ++k) {
    const float4 *Pk = P + (long long)k * n_lines;
    float acc = 0.0f, cmp = 0.0f;
    for (long long l = a; l < b; ++l) {
      const int4 r = __ldg(R + l);
      const float4 p = __ldg(Pk + l);
      const float u = __fadd_rn((float)((int)j - r.z), __int_as_float(r.w));
      float v;
      if (PROFILE == RT_PROFILE_LORENTZ) {
        v = p.x * rcp_approx(__fmaf_rn(u, u, p.y));
      } else {
        const float x = p.y * u;
        const float y = sqrtf(p.z);
        v = __fdividef(p.x, y) * faddeeva_re_near(x, y, __fmaf_rn(x, x, p.z), wc);
      }
      const float yk = __fsub_rn(v, cmp);
      const float t = __fadd_rn(acc, yk);
      cmp = __fsub_rn(__fsub_rn(t, acc), yk);
      acc = t;
    }
    float *dst = kappa + (long long)k * n_nu + j;
    const float out = __fsub_rn(acc, cmp);
    *dst = accumulate ? *dst + out : out;
  }
}

// ---- adaptive points per line
// Each line's window at each T node: |nu_j - nu0| <= w = min(cutoff, sqrt(A gamma /
// (pi kappa_min))) with A = u(T_k) S(T_k) and gamma the Lorentz half-width at T_k, in
// binary64 in the order the float64 reading states it (number density x p atm / (k_B T)
// 1e-6, Eq. (S) as S_ref (T_ref/T)^q Boltzmann ratio stimulated-emission ratio).
struct AdaptParams {
  double nu_min, dnu, cutoff, T_min, T_max, T_ref, c2, x_ref, p_ref, n_T, q_exp, kappa_min;
  long long n_nu, n_lines;
  int nT;
};

__device__ __noinline__ int2 adaptive_window64(double v, double S, double g, double E, const AdaptParams &P, int k) {
  const double T = P.nT > 1 ? P.T_min + (double)k * ((P.T_max - P.T_min) / (double)(P.nT - 1)) : P.T_min;
  const double q = pow(P.T_ref / T, P.q_exp);
  const double boltz = exp(-P.c2 * E / T) / exp(-P.c2 * E / P.T_ref);
  const double stim = (-expm1(-P.c2 * v / T)) / (-expm1(-P.c2 * v / P.T_ref));
  const double ST = S * q * boltz * stim;
  const double A = P.x_ref * P.p_ref * kAtm / (kKB * T) * 1e-6 * ST;
  const double gam = g * P.p_ref * pow(P.T_ref / T, P.n_T);
  double w = sqrt(A * gam / (kPi * P.kappa_min));
  if (!(w <= P.cutoff)) w = P.cutoff;
  double flo = floor((v - w - P.nu_min) / P.dnu) - 1.0;
  double fhi = ceil((v + w - P.nu_min) / P.dnu) + 1.0;
  flo = fmin(fmax(isfinite(flo) ? flo : 0.0, -1.0), (double)P.n_nu + 1.0);
  fhi = fmin(fmax(isfinite(fhi) ? fhi : 0.0, -2.0), (double)P.n_nu + 1.0);
  long long lo = (long long)flo, hi = (long long)fhi;
  if (lo < 0) lo = 0;
  if (hi > P.n_nu - 1) hi = P.n_nu - 1;
#pragma unroll 1
  for (int it = 0; it < 6 && lo < P.n_nu; ++it)
    if (__dsub_rn(grid_nu(P.nu_min, lo, P.dnu), v) < -w) ++lo;
#pragma unroll 1
  for (int it = 0; it < 6 && hi >= 0; ++it)
    if (__dsub_rn(grid_nu(P.nu_min, hi, P.dnu), v) > w) --hi;
  return make_int2((int)lo, (int)hi);
}

// Windows of 256 lines at kWinNodes nodes per block, after k_line_setup.  The binary32
// coefficients give the half-width in grid units, sqrt(c0 / kappa_min) / (s dnu) for Voigt and
// sqrt(P.x / kappa_min) for Lorentz lines, to a relative error below kWinTol (half that of
// A gamma: two roundings of expf, four of powf each for q and gamma, a dozen others, 2e-6 in
// all).  An end further than that from any grid point's edge, and a half-width further than
// that from the cutoff, is decided already (a window at the cutoff is the line's cutoff
// window); the others, about 2 % of the pairs, are queued and decided in binary64 as
// stated.  The binary64 form for every pair took 1060 us for 64 nodes x 20k lines, this 54 us.
constexpr int kWinNodes = 8;
constexpr float kWinTol = 4e-6f;
struct WinParams {
  float inv_kmin, cut_grid, tol;  // 1 / kappa_min, cutoff in grid units, relative tolerance
  float min_w2;                   // half-widths^2 above min_w2 gamma_ref: S(T) is above 1e-36
  double min_S;                   // intensities whose product with the partition ratio is
};
template <int PROFILE>
__global__ void __launch_bounds__(256)
k_adaptive_windows(const double *__restrict__ nu0, const double *__restrict__ S, const double *__restrict__ g,
                   const double *__restrict__ E, AdaptParams P, const float4 *__restrict__ coef,
                   const int4 *__restrict__ R, WinParams Q, int2 *__restrict__ AW,
                   unsigned long long *evals) {
  __shared__ unsigned short s_queue[256 * kWinNodes];
  __shared__ int s_n;
  const long long l = (long long)blockIdx.x * 256 + threadIdx.x;
  const int k0 = blockIdx.y * kWinNodes, k1 = min(k0 + kWinNodes, P.nT);
  if (threadIdx.x == 0) s_n = 0;
  __syncthreads();
  unsigned long long cnt = 0;
  if (l < P.n_lines) {
    const int4 r = R[l];
    const float dg = __int_as_float(r.w);
    const bool plain = S[l] > Q.min_S;  // no binary32 underflow on the way to the coefficients
    const float w2_min = Q.min_w2 * __double2float_ru(g[l]);
    for (int k = k0; k < k1; ++k) {
      const float4 c = __ldg(coef + (long long)k * P.n_lines + l);
      const float w = PROFILE == RT_PROFILE_LORENTZ ? sqrtf(c.x * Q.inv_kmin) : sqrtf(c.x * Q.inv_kmin) / c.y;
      const float tol = __fmaf_rn(Q.tol, w, 1e-6f);
      int2 win = make_int2(r.x, r.y);
      const bool known = plain && c.x > 1e-30f && w * w > w2_min && w < 1e18f;
      bool sure = known && w - tol > Q.cut_grid;
      if (known && w + tol < Q.cut_grid && w < 1e6f) {
        // points j with |j - j_c + dg| <= w
        const float a = -w - dg, b = w - dg;
        const float ca = ceilf(a), fb = floorf(b);
        sure = ca - a > tol && a - (ca - 1.0f) > tol && b - fb > tol && fb + 1.0f - b > tol;
        win.x = max(r.z + (int)ca, 0);
        win.y = (int)min((long long)r.z + (long long)fb, P.n_nu - 1);
      }
      if (sure) {
        AW[(long long)k * P.n_lines + l] = win;
        if (win.y >= win.x) cnt += (unsigned long long)(win.y - win.x + 1);
      } else {
        s_queue[atomicAdd(&s_n, 1)] = (unsigned short)((k - k0) * 256 + threadIdx.x);
      }
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < s_n; q += 256) {
    const int k = k0 + (s_queue[q] >> 8);
    const long long m = (long long)blockIdx.x * 256 + (s_queue[q] & 255);
    const int2 win = adaptive_window64(nu0[m], S[m], g[m], E[m], P, k);
    AW[(long long)k * P.n_lines + m] = win;
    if (win.y >= win.x) cnt += (unsigned long long)(win.y - win.x + 1);
  }
  if (evals) {
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, o);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(evals, cnt);
  }
}

int g_kappa_tpb = kMaxTPerBlock;

rt_status launch_kappa(const float4 *P, const float4 *P2, const int4 *R, int4 *tiles,
                       const unsigned *far_bits, const int2 *AW, long long n, const rt_spectral *spec,
                       double nu_abs_max, double mass_amu, float *kappa, uint32_t *status,
                       cudaStream_t st) {
  static const WeidSet ws{weideman_series<24>(), weideman_series<16>(), weideman_series<12>()};
  const WeidCoef &wc = ws.n24;
  // W bounds every line's near-centre half-width sqrt(400 - y^2) / (s dnu) <= 20 alpha /
  // (sqrt(ln 2) dnu), alpha the largest Doppler half-width of a line that reaches the grid
  int W = 0;
  if (spec->profile == RT_PROFILE_VOIGT) {
    const double alpha = nu_abs_max * std::sqrt(spec->T_max) *
                         std::sqrt(2.0 * std::log(2.0) * kKB / (mass_amu * kAmu)) / kC;
    const double w = 20.0 * alpha / (std::sqrt(std::log(2.0)) * spec->dnu) * 1.01 + 2.0;
    W = (!(w < (double)(1 << 28))) ? (1 << 28) : (int)std::ceil(w);
  }
  const long long n_tiles = (spec->n_nu + kTilePts - 1) / kTilePts;
  if (spec->points_per_line > 0) {  // fixed points per line: the gather kernel
    dim3 g((unsigned)n_tiles, (unsigned)((spec->nT + kPplNodes - 1) / kPplNodes));
    if (spec->profile == RT_PROFILE_LORENTZ)
      k_kappa_ppl<RT_PROFILE_LORENTZ><<<g, kTilePts, 0, st>>>(P, R, n, spec->n_nu, spec->nT, wc,
                                                              spec->accumulate ? 1 : 0, kappa);
    else
      k_kappa_ppl<RT_PROFILE_VOIGT><<<g, kTilePts, 0, st>>>(P, R, n, spec->n_nu, spec->nT, wc,
                                                            spec->accumulate ? 1 : 0, kappa);
    RT_CUDA_TRY(cudaGetLastError());
    return RT_OK;
  }
  k_tile_lines<<<(unsigned)((n_tiles + 3) / 4), 128, 0, st>>>(R, n, spec->n_nu, W, far_bits, n_tiles,
                                                                tiles);  // a warp per tile
  RT_CUDA_TRY(cudaGetLastError());
  const int vec_ok = ((reinterpret_cast<uintptr_t>(kappa) & 15u) == 0 && spec->n_nu % 4 == 0) ? 1 : 0;
  int want = g_kappa_tpb;
  if (want < 1 || want > kMaxTPerBlock) want = kMaxTPerBlock;
  const int tpb = spec->nT < want ? spec->nT : want;
  dim3 gk((unsigned)n_tiles, (unsigned)((spec->nT + tpb - 1) / tpb));
  auto kernel = spec->profile == RT_PROFILE_LORENTZ
                    ? (AW ? k_kappa<RT_PROFILE_LORENTZ, true> : k_kappa<RT_PROFILE_LORENTZ, false>)
                    : (AW ? k_kappa<RT_PROFILE_VOIGT, true> : k_kappa<RT_PROFILE_VOIGT, false>);
  kernel<<<gk, 32 * tpb, 0, st>>>(P, P2, R, AW, tiles, n, spec->n_nu, spec->nT, ws, vec_ok,
                                  spec->accumulate ? 1 : 0, kappa, status);
  RT_CUDA_TRY(cudaGetLastError());
  return RT_OK;
}

}  // namespace

rt_status validate_spec(const rt_spectral *s) {
  if (!s) return fail(RT_E_INVAL, "spec is NULL");
  if (!(s->n_nu >= 1) || s->n_nu > (1LL << 30))
    return fail(RT_E_INVAL, "spec.n_nu must be in [1, 2^30]");
  if (!std::isfinite(s->nu_min) || !std::isfinite(s->dnu) || !(s->dnu > 0))
    return fail(RT_E_INVAL, "spec.nu_min / dnu must be finite, dnu > 0");
  if (!std::isfinite(s->cutoff) || s->cutoff < 0 || s->cutoff / s->dnu > (double)(1 << 28))
    return fail(RT_E_INVAL, "spec.cutoff must be finite, >= 0 and < 2^28 dnu");
  if (s->profile != RT_PROFILE_LORENTZ && s->profile != RT_PROFILE_VOIGT)
    return fail(RT_E_INVAL, "spec.profile must be RT_PROFILE_LORENTZ or RT_PROFILE_VOIGT");
  if (s->nT < 1 || s->nT > 65535) return fail(RT_E_INVAL, "spec.nT must be in [1, 65535]");
  if (!std::isfinite(s->T_min) || !std::isfinite(s->T_max) || !(s->T_min > 0) ||
      s->T_max < s->T_min || (s->nT > 1 && !(s->T_max > s->T_min)))
    return fail(RT_E_INVAL, "spec temperatures must satisfy 0 < T_min <= T_max (< when nT > 1)");
  if (!std::isfinite(s->p_ref_atm) || !(s->p_ref_atm > 0) || !std::isfinite(s->x_ref) ||
      !(s->x_ref > 0))
    return fail(RT_E_INVAL, "spec.p_ref_atm and spec.x_ref must be finite and > 0");
  if (s->points_per_line < 0 || s->points_per_line > (1 << 20))
    return fail(RT_E_INVAL, "spec.points_per_line must be in [0, 2^20]");
  if (s->accumulate != 0 && s->accumulate != 1) return fail(RT_E_INVAL, "spec.accumulate must be 0 or 1");
  if (!std::isfinite(s->kappa_min) || s->kappa_min < 0)
    return fail(RT_E_INVAL, "spec.kappa_min must be finite and >= 0");
  if (s->kappa_min > 0 && s->points_per_line > 0)
    return fail(RT_E_INVAL, "spec.kappa_min (adaptive points) and points_per_line exclude each other");
  return RT_OK;
}

namespace {

rt_status validate_host_lines(const rt_lines *L, const rt_spectral *s) {
  const double lim = 536870912.0 * s->dnu;  // 2^29 grid steps
  for (int64_t l = 0; l < L->n; ++l) {
    const double v = L->nu0[l], S = L->S_ref[l], g = L->gamma_ref[l], E = L->E_lower[l];
    if (!std::isfinite(v) || !std::isfinite(S) || !(S > 0) || !std::isfinite(g) || !(g > 0) ||
        !std::isfinite(E) || !(E >= 0))
      return fail(RT_E_NONFINITE, "line %lld: non-finite or non-positive parameter", (long long)l);
    if (!(std::fabs(v - s->nu_min) <= lim))
      return fail(RT_E_INVAL, "line %lld: centre too far from the spectral grid", (long long)l);
    if (l > 0 && !(L->nu0[l - 1] <= v))
      return fail(RT_E_UNSORTED, "line %lld: centres not in ascending order", (long long)l);
  }
  return RT_OK;
}

}  // namespace

rt_status launch_line_geometry(const double *nu0, const double *S, const double *g, const double *E,
                               long long n, const rt_spectral *spec, int check, int4 *R,
                               unsigned long long *evals, uint32_t *status, cudaStream_t st) {
  if (n <= 0) return RT_OK;
  GeomParams G{spec->nu_min, spec->dnu, 1.0 / spec->dnu, spec->cutoff, spec->n_nu, n, spec->nT, check,
               spec->points_per_line};
  k_line_geometry<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(nu0, S, g, E, G, R, evals, status);
  RT_CUDA_TRY(cudaGetLastError());
  return RT_OK;
}

namespace {

// Scratch of one build: [line arrays if host-resident][R: n int4][P: nT n float4]
// [P2: nT n float4, Voigt][tile segments: kTileInts int4 per 256-point tile][far-zone bound]
// [adaptive windows: nT n int2]
struct KappaLayout {
  size_t off_R, off_P, off_P2, off_tiles, off_far, off_AW, total;
};

KappaLayout kappa_layout(const rt_lines *lines, const rt_spectral *spec) {
  auto up = [](size_t v) { return (v + 255) & ~size_t(255); };
  const size_t n = (size_t)lines->n;
  const size_t pn = (size_t)spec->nT * n * sizeof(float4);
  KappaLayout L;
  L.off_R = up(lines->memory == RT_MEM_HOST ? 4 * n * sizeof(double) : 0);
  L.off_P = up(L.off_R + n * sizeof(int4));
  L.off_P2 = up(L.off_P + pn);
  L.off_tiles = up(L.off_P2 + (spec->profile == RT_PROFILE_VOIGT ? pn : 0));
  const size_t n_tiles = (size_t)((spec->n_nu + kTilePts - 1) / kTilePts);
  L.off_far = up(L.off_tiles + n_tiles * kTileInts * sizeof(int4));
  L.off_AW = L.off_far + 256;  // adaptive windows: nT n int2
  L.total = L.off_AW + (spec->kappa_min > 0 ? up((size_t)spec->nT * n * sizeof(int2)) : 0);
  return L;
}

rt_status validate_build_args(const rt_lines *lines, const rt_spectral *spec, float *kappa,
                              uint32_t *status, const char *who) {
  rt_status v = validate_spec(spec);
  if (v != RT_OK) return v;
  if (!lines || !kappa) return fail(RT_E_INVAL, "%s: lines or kappa is NULL", who);
  if (lines->n < 0 || lines->n > (1LL << 31) - 1) return fail(RT_E_INVAL, "lines.n out of range");
  if (lines->memory != RT_MEM_HOST && lines->memory != RT_MEM_DEVICE)
    return fail(RT_E_INVAL, "lines.memory must be RT_MEM_HOST or RT_MEM_DEVICE");
  if (!std::isfinite(lines->T_ref) || !(lines->T_ref > 0) || !std::isfinite(lines->n_T) ||
      !std::isfinite(lines->q_exp) || !std::isfinite(lines->mass_amu) || !(lines->mass_amu > 0))
    return fail(RT_E_INVAL, "lines: T_ref, n_T, q_exp, mass_amu must be finite (T_ref, mass > 0)");
  if (lines->n > 0 && (!lines->nu0 || !lines->S_ref || !lines->gamma_ref || !lines->E_lower))
    return fail(RT_E_INVAL, "lines: NULL array");
  if (lines->memory == RT_MEM_DEVICE && !status)
    return fail(RT_E_INVAL, "device-resident lines need a device status word");
  return RT_OK;
}

template <int N>
LineArgs<N> line_args(const double *const (&src)[4], long long n) {
  LineArgs<N> A;
  for (int q = 0; q < 4; ++q) std::memcpy(A.v[q], src[q], (size_t)n * sizeof(double));
  return A;
}
template <int N>
__global__ void k_line_list(const __grid_constant__ LineArgs<N> A, int n, double *__restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, q = i / N;
  if (i - q * N < n) out[q * n + i - q * N] = A.v[q][i - q * N];
}

// Everything after validation, on scratch laid out by kappa_layout.
rt_status run_build(char *base, const KappaLayout &L, const rt_lines *lines, const rt_spectral *spec,
                    float *kappa, unsigned long long *evals_out, uint32_t *status, cudaStream_t st) {
  const long long n = lines->n;
  const double *d_nu0 = lines->nu0, *d_S = lines->S_ref, *d_g = lines->gamma_ref, *d_E = lines->E_lower;
  unsigned *far_bits = reinterpret_cast<unsigned *>(base + L.off_far);
  int4 *R = reinterpret_cast<int4 *>(base + L.off_R);
  float4 *P = reinterpret_cast<float4 *>(base + L.off_P);
  float4 *P2 = reinterpret_cast<float4 *>(base + L.off_P2);
  int4 *tiles = reinterpret_cast<int4 *>(base + L.off_tiles);

  GeomParams G{spec->nu_min, spec->dnu, 1.0 / spec->dnu, spec->cutoff, spec->n_nu, n, spec->nT,
               lines->memory == RT_MEM_DEVICE ? 1 : 0, spec->points_per_line};
  const int tb = 256;
  const bool adaptive = spec->kappa_min > 0;
  PrefParams Q;
  Q.T_min = spec->T_min;
  Q.T_max = spec->T_max;
  Q.T_ref = lines->T_ref;
  const double c2 = 100.0 * kH * kC / kKB;
  Q.c2.hi = (float)c2;
  Q.c2.lo = (float)(c2 - (double)Q.c2.hi);
  Q.u_coef = (float)(spec->x_ref * spec->p_ref_atm * kAtm / kKB * 1e-6);
  Q.p_ref = (float)spec->p_ref_atm;
  Q.n_T = (float)lines->n_T;
  Q.q_exp = (float)lines->q_exp;
  Q.doppler = (float)(std::sqrt(2.0 * std::log(2.0) * kKB / (lines->mass_amu * kAmu)) / kC);
  Q.inv_dnu = (float)(1.0 / spec->dnu);
  Q.dnu = (float)spec->dnu;
  Q.n_lines = n;
  Q.nT = spec->nT;
  Q.profile = spec->profile;
  RT_CUDA_TRY(cudaMemsetAsync(far_bits, 0, sizeof(unsigned), st));
  // A host list goes to the scratch in four copies (out of pageable memory about 2 us each) or, as
  // far as a launch's parameters reach, in a launch: 500 Lorentz lines 42 us, so 32; 1000 lines 47
  // and 35.  The set-up kernel carries the list itself, 3 us less, unless later kernels read it or
  // many pairs do (1000 lines at 8 nodes 42 us, so 38; at 64 nodes 77 and 75, the gain falling).
  // A capturing stream takes the copies: its replays read the caller's arrays again.
  int carried = 0;  // capacity of the set-up kernel's list
  if (lines->memory == RT_MEM_HOST) {
    double *d = reinterpret_cast<double *>(base);
    const double *src[4] = {d_nu0, d_S, d_g, d_E};
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (n <= kArgLines) RT_CUDA_TRY(cudaStreamIsCapturing(st, &capture));
    if (n > kArgLines || capture != cudaStreamCaptureStatusNone) {
      for (int q = 0; q < 4; ++q)
        RT_CUDA_TRY(cudaMemcpyAsync(d + q * n, src[q], (size_t)n * sizeof(double), cudaMemcpyHostToDevice, st));
    } else if (adaptive || n * spec->nT > kDirectPairs) {
      const auto list = [&](auto cap) {
        constexpr int N = decltype(cap)::value;
        k_line_list<N><<<(4 * N + 255) / 256, 256, 0, st>>>(line_args<N>(src, n), (int)n, d);
      };
      if (n <= kArgLines / 2) list(std::integral_constant<int, kArgLines / 2>());
      else list(std::integral_constant<int, kArgLines>());
      RT_CUDA_TRY(cudaGetLastError());
    } else {
      carried = n <= kArgLines / 2 ? kArgLines / 2 : kArgLines;
    }
    d_nu0 = d; d_S = d + n; d_g = d + 2 * n; d_E = d + 3 * n;
  }
  // with adaptive points the evaluations are counted per (node, line) window below
  unsigned long long *ev = adaptive ? nullptr : evals_out;
  const unsigned line_blocks = (unsigned)((n + tb - 1) / tb);
  // (the coefficients of 2^31 blocks would take 8 TB: the scratch was refused before)
  const auto setup = [&](const auto &list) {
    k_line_setup<<<line_blocks * (spec->nT + 1u), tb, 0, st>>>(list, G, Q, line_blocks, R, P, P2, far_bits, ev, status);
  };
  const double *src[4] = {lines->nu0, lines->S_ref, lines->gamma_ref, lines->E_lower};
  if (carried == kArgLines) setup(line_args<kArgLines>(src, n));
  else if (carried) setup(line_args<kArgLines / 2>(src, n));
  else setup(LineArrays{d_nu0, d_S, d_g, d_E});
  RT_CUDA_TRY(cudaGetLastError());

  int2 *AW = nullptr;
  if (adaptive) {
    AW = reinterpret_cast<int2 *>(base + L.off_AW);
    AdaptParams A{spec->nu_min, spec->dnu, spec->cutoff, spec->T_min, spec->T_max, lines->T_ref,
                  100.0 * (kH * kC / kKB), spec->x_ref, spec->p_ref_atm, lines->n_T, lines->q_exp,
                  spec->kappa_min, spec->n_nu, n, spec->nT};
    dim3 ga((unsigned)((n + tb - 1) / tb), (unsigned)((spec->nT + kWinNodes - 1) / kWinNodes));
    auto windows = spec->profile == RT_PROFILE_LORENTZ ? k_adaptive_windows<RT_PROFILE_LORENTZ>
                                                       : k_adaptive_windows<RT_PROFILE_VOIGT>;
    // gamma <= gamma_ref p G and u <= u_max over the nodes; A gamma / pi = kappa_min (w dnu)^2
    const double ra = lines->T_ref / spec->T_min, rb = lines->T_ref / spec->T_max;
    const double G = std::fmax(std::pow(ra, lines->n_T), std::pow(rb, lines->n_T)) * spec->p_ref_atm;
    const double qmin = std::fmin(std::pow(ra, lines->q_exp), std::pow(rb, lines->q_exp));
    const double u_max = spec->x_ref * spec->p_ref_atm * kAtm / (kKB * spec->T_min) * 1e-6;
    WinParams wp;
    wp.inv_kmin = (float)(1.0 / spec->kappa_min);
    wp.cut_grid = (float)(spec->cutoff / spec->dnu);
    // the ratio T_ref / T carries 2^-23 into its powers
    wp.tol = kWinTol + 2e-7f * (float)(std::fabs(lines->q_exp) + std::fabs(lines->n_T));
    wp.min_w2 = (float)(1e-36 * u_max * G / (kPi * spec->dnu * spec->dnu * spec->kappa_min));
    wp.min_S = 1e-36 / std::fmin(qmin, 1.0);
    windows<<<ga, tb, 0, st>>>(d_nu0, d_S, d_g, d_E, A, P, R, wp, AW, evals_out);
    RT_CUDA_TRY(cudaGetLastError());
  }

  // largest |nu0| of a line whose window (cutoff or fixed points) reaches the grid
  const double reach = spec->cutoff + (spec->points_per_line + 2.0) * spec->dnu;
  const double nu_abs_max =
      std::fmax(std::fabs(spec->nu_min - reach),
                std::fabs(spec->nu_min + (double)spec->n_nu * spec->dnu + reach));
  return launch_kappa(P, P2, R, tiles, far_bits, AW, n, spec, nu_abs_max, lines->mass_amu, kappa, status, st);
}

}  // namespace

rt_status build_kappa_impl(const rt_lines *lines, const rt_spectral *spec, float *kappa,
                           unsigned long long *evals_out, uint32_t *status, cudaStream_t st) {
  rt_status v = validate_build_args(lines, spec, kappa, status, "rt_build_kappa");
  if (v != RT_OK) return v;
  if (lines->memory == RT_MEM_HOST && lines->n > 0) {
    v = validate_host_lines(lines, spec);
    if (v != RT_OK) return v;
  }
  const size_t table = (size_t)spec->nT * (size_t)spec->n_nu;
  if (lines->n == 0) {
    if (!spec->accumulate) RT_CUDA_TRY(cudaMemsetAsync(kappa, 0, table * sizeof(float), st));
    return RT_OK;
  }
  const KappaLayout L = kappa_layout(lines, spec);
  Scratch scr;
  v = scr.alloc(L.total, st);
  if (v != RT_OK) return v;
  return run_build(scr.as<char>(), L, lines, spec, kappa, evals_out, status, st);
}

// ---------------------------------------------------------------------------
// Allocation-free variant.  Its scratch is this file-scope device array: every
// GPU that loads the library holds it until the process exits.  Host code must
// not hand the array's name to a kernel (in host code it is a host-side stand-in
// for the symbol); the device address is looked up once per device below.
constexpr size_t kStaticScratchBytes = size_t(32) << 20;  // 32 MiB
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

static rt_status static_scratch_address(void **out) {
  static std::mutex mu;
  static void *addr[256] = {};
  int dev = 0;
  RT_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 256) return fail(RT_E_INVAL, "rt_build_kappa_static: device index out of range");
  std::lock_guard<std::mutex> lock(mu);
  if (!addr[dev]) {
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_static_scratch)");
    addr[dev] = p;
  }
  *out = addr[dev];
  return RT_OK;
}

rt_status build_kappa_static_impl(const rt_lines *lines, const rt_spectral *spec, float *kappa,
                                  unsigned long long *evals_out, uint32_t *status, cudaStream_t st) {
  rt_status v = validate_build_args(lines, spec, kappa, status, "rt_build_kappa_static");
  if (v != RT_OK) return v;
  // same scratch layout as rt_build_kappa, checked against the fixed array
  const KappaLayout L = kappa_layout(lines, spec);
  if (L.total > kStaticScratchBytes)
    return fail(RT_E_INVAL,
                "rt_build_kappa_static: needs %zu bytes of scratch (16 B per line and T node, 32 B "
                "for Voigt lines, 16 B per line, 80 B per 256 wavenumbers, plus 32 B per line for "
                "host-resident lines), the static array holds %zu",
                L.total, kStaticScratchBytes);
  if (lines->memory == RT_MEM_HOST && lines->n > 0) {
    v = validate_host_lines(lines, spec);
    if (v != RT_OK) return v;
  }
  const size_t table = (size_t)spec->nT * (size_t)spec->n_nu;
  if (lines->n == 0) {
    if (!spec->accumulate) RT_CUDA_TRY(cudaMemsetAsync(kappa, 0, table * sizeof(float), st));
    return RT_OK;
  }
  void *scratch = nullptr;
  v = static_scratch_address(&scratch);
  if (v != RT_OK) return v;
  return run_build(reinterpret_cast<char *>(scratch), L, lines, spec, kappa, evals_out, status, st);
}

}  // namespace rt

extern "C" rt_status rt_build_kappa(const rt_lines *lines, const rt_spectral *spec, float *kappa,
                                    unsigned long long *evals_out, uint32_t *status, void *stream) {
  return rt::build_kappa_impl(lines, spec, kappa, evals_out, status, (cudaStream_t)stream);
}

extern "C" rt_status rt_build_kappa_static(const rt_lines *lines, const rt_spectral *spec, float *kappa,
                                           unsigned long long *evals_out, uint32_t *status,
                                           void *stream) {
  return rt::build_kappa_static_impl(lines, spec, kappa, evals_out, status, (cudaStream_t)stream);
}

namespace rt {
extern int g_walk_blocks, g_walk_refill, g_walk_group;  // rt_trace.cu
}

extern "C" rt_status rt_set_tuning(const rt_tuning *t) {
  if (!t) return rt::fail(RT_E_INVAL, "rt_set_tuning: NULL");
  if (t->kappa_t_per_block < 0 || t->kappa_t_per_block > 8)
    return rt::fail(RT_E_INVAL, "rt_set_tuning: kappa_t_per_block must be in [0, 8]");
  if (t->walk_blocks_per_sm != 0 && t->walk_blocks_per_sm != 4 && t->walk_blocks_per_sm != 5)
    return rt::fail(RT_E_INVAL, "rt_set_tuning: walk_blocks_per_sm must be 0, 4 or 5");
  if (t->walk_refill_idle != 0 && t->walk_refill_idle != 12 && t->walk_refill_idle != 16)
    return rt::fail(RT_E_INVAL, "rt_set_tuning: walk_refill_idle must be 0, 12 or 16");
  if (t->walk_group < 0 || t->walk_group > 2) return rt::fail(RT_E_INVAL, "rt_set_tuning: walk_group must be 0, 1 or 2");
  rt::g_kappa_tpb = t->kappa_t_per_block == 0 ? 8 : t->kappa_t_per_block;
  rt::g_walk_blocks = t->walk_blocks_per_sm == 0 ? 5 : t->walk_blocks_per_sm;
  rt::g_walk_refill = t->walk_refill_idle == 0 ? 16 : t->walk_refill_idle;
  rt::g_walk_group = t->walk_group;
  return RT_OK;
}

extern "C" rt_status rt_get_tuning(rt_tuning *t) {
  if (!t) return rt::fail(RT_E_INVAL, "rt_get_tuning: NULL");
  *t = rt_tuning{};
  t->kappa_t_per_block = rt::g_kappa_tpb;
  t->walk_blocks_per_sm = rt::g_walk_blocks;
  t->walk_refill_idle = rt::g_walk_refill;
  t->walk_group = rt::g_walk_group;
  return RT_OK;
}
