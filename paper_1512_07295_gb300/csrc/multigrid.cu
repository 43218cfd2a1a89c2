// Interlacing with more than two grids (the extension Sec. 3.1 points to): J = 1, 2, 4 or 8 mass grids,
// grid j holding the particles shifted by d_j H with d_j in {0, 1/2}^3, each transformed, multiplied by
// e^{+i k.d_j H} = e^{+2 pi i n.d_j/N} and averaged:
//   delta(n) = sum_j e^{+2 pi i n.d_j/N} G_j(n) / (J sum(w) W(n)).
// By the shift theorem, image m of grid j then carries e^{+2 pi i m.d_j}, so the average keeps image m
// with the weight theta_m = (1/J) sum_j (-1)^{m.(2 d_j)}:
//   J = 2, d = {0, (1,1,1)/2}:                                 theta = 1 for m_x+m_y+m_z even (eq:intdelta);
//   J = 4, d = {0, (1,1,0)/2, (1,0,1)/2, (0,1,1)/2}:           theta = 1 when m_x, m_y, m_z have one parity;
//   J = 8, d = {0, 1/2}^3:                                      theta = 1 when every m_i is even.
// The first images left are |m|^2 = 2 (J = 2), 3 (J = 4) and 4 (J = 8). The grids come from the
// existing assignment: J = 2 and J = 8 as interlaced pairs (d, d + (1,1,1)/2) of the shifted
// particles, J = 4 as single grids. Every mode of the full N^3 grid is binned once, the stored mode
// and, for 0 < i_z < N/2, its partner -n with its own signed index (the phases of a Nyquist slot are
// not conjugate), as in the two-grid estimate.
#include "host.cuh"

namespace pk {

namespace {

// Shift pattern of grid j in half cells (h = 2 d, components 0, 1 or 2).
struct Shifts {
  int h[8][3];
  int bases;      // particle shifts to assign
  bool pairs;     // each base gives an interlaced pair (d, d + (1,1,1)/2)
};

bool make_shifts(int J, Shifts* s) {
  static const int base4[4][3] = {{0, 0, 0}, {1, 1, 0}, {1, 0, 1}, {0, 1, 1}};
  switch (J) {
    case 1: s->bases = 1; s->pairs = false; break;
    case 2: s->bases = 1; s->pairs = true; break;
    case 4: s->bases = 4; s->pairs = false; break;
    case 8: s->bases = 4; s->pairs = true; break;
    default: return false;
  }
  int j = 0;
  for (int b = 0; b < s->bases; ++b) {
    for (int a = 0; a < 3; ++a) s->h[j][a] = base4[b][a];
    ++j;
    if (s->pairs) {
      for (int a = 0; a < 3; ++a) s->h[j][a] = base4[b][a] + 1;
      ++j;
    }
  }
  return true;
}

}  // namespace

// Copies of the positions shifted by h H/2 (h in {0, 1} per axis).
__global__ void k_shift_f64(const double* __restrict__ in, int64_t n, double hx, double hy, double hz, double* __restrict__ out) {
  for (int64_t i = gtid(); i < n; i += gstride()) {
    out[3 * i] = in[3 * i] + hx;
    out[3 * i + 1] = in[3 * i + 1] + hy;
    out[3 * i + 2] = in[3 * i + 2] + hz;
  }
}

__global__ void k_shift_cells(const pk_cellpos* __restrict__ in, int64_t n, int ng, int h, pk_cellpos* __restrict__ out) {
  for (int64_t i = gtid(); i < n; i += gstride()) out[i] = shift_rec(in[i], h, ng);
}

// Per-slot tables (n the signed index of the slot), FP64: 1/W_1d(n), then e^{i pi n h/N} for h = 1 and
// h = 2 (cosine row, sine row each).
constexpr int kMultiTabRows = 5;
__global__ void k_multi_tables(double* __restrict__ tab, int ng, int order) {
  for (int i = threadIdx.x + blockIdx.x * blockDim.x; i < ng; i += blockDim.x * gridDim.x) {
    const int n = signed_mode(i, ng);
    const double x = double(n) / double(ng);
    const double s = n == 0 ? 1.0 : sinpi(x) / (3.14159265358979323846 * x);
    double w = 1.0;
    for (int k = 0; k < order; ++k) w *= s;
    double sn, cs, sn2, cs2;
    sincospi(x, &sn, &cs);
    sincospi(2.0 * x, &sn2, &cs2);
    tab[i] = 1.0 / w;
    tab[ng + i] = cs;
    tab[2 * ng + i] = sn;
    tab[3 * ng + i] = cs2;
    tab[4 * ng + i] = sn2;
  }
}

struct MultiArgs {
  int ng, J, nbins, lo2, w2;
  int64_t grid_stride;  // complex elements between transformed grids
  double vol;
  const double* wsums;
  double* bin_sum;
  double* bin_k;
  unsigned long long* bin_cnt;
  void* delta_out;
};

template <typename R>
struct Cx {
  R x, y;
};
// Shift of grid j of J in half cells along axis d (make_shifts as constants).
template <int J>
__host__ __device__ constexpr int shift_of(int j, int d) {
  if (J == 1) return 0;
  if (J == 2) return j;
  const int base = J == 8 ? j / 2 : j, odd = J == 8 ? j % 2 : 0;
  return (base != 0 && d != 3 - base ? 1 : 0) + odd;  // bases 0, (1,1,0), (1,0,1), (0,1,1)
}

// The roundings of the combine are written out, so that the compiler's choice of fused operations cannot move with the code.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
// a b; F picks the product that each component rounds first (bit 0: x, bit 1: y).
template <int F, typename R>
__device__ __forceinline__ Cx<R> mul_as(Cx<R> a, Cx<R> b) {
  return {F & 1 ? fma(-a.y, b.y, mul_rn(a.x, b.x)) : fma(a.x, b.x, -mul_rn(a.y, b.y)),
          F & 2 ? fma(a.y, b.x, mul_rn(a.x, b.y)) : fma(a.x, b.y, mul_rn(a.y, b.x))};
}

// The sum over the grids at one mode: sum_j e^{i pi n.h_j / N} G_j, phases e[axis][h - 1].
template <int FG, typename R, int J>
__device__ __forceinline__ Cx<R> combine(const Cx<R> (&g)[J], const Cx<R> (&e)[3][2]) {
  Cx<R> sum = {R(0), R(0)};
#pragma unroll
  for (int j = 0; j < J; ++j) {
    Cx<R> ph = {R(1), R(0)};
    bool any = false;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int h = shift_of<J>(j, d);
      if (h != 0) {
        ph = any ? mul_as<0>(ph, e[d][h - 1]) : e[d][h - 1];
        any = true;
      }
    }
    const Cx<R> t = any ? mul_as<FG>(g[j], ph) : g[j];  // grid 0 alone is not shifted
    sum = {add_rn(sum.x, t.x), add_rn(sum.y, t.y)};
  }
  return sum;
}

// Shifted-grid combine of J transformed grids and k-shell sums (eq:intdelta generalised to the shift
// set h_j, Sec. 3.1). Per stored mode n (and its partner -n on the half-complex layout):
//   delta(n) = sum_j e^{i pi n.h_j / N} G_j(n) / (J sum(w) W(n)),
// the per-axis phases e^{i pi n h/N} (h = 0, 1, 2) read from tables; the arithmetic runs in the grids'
// precision (FP32 grids: FP32 combine), the shell sums in FP64.
// Consecutive lanes hold consecutive i_z, so a warp's modes fall in few shells: runs of equal shell
// are summed with a segmented warp scan and one lane per run adds them to shared memory.
// FP64 arithmetic is the scarce unit, so the sums of |n|, which depend on (|n_x|, |n_y|, n_z) and not on the order of
// n_x and n_y, are taken on the rows 0 <= i_y <= i_x <= N/2 alone, with the rows' multiplicity; the shifts are
// constants of J, the slots advance without divisions, and the next modes' loads are in flight while these are summed.
// N = 256, J = 4, FP32: 285 us with an FP64 root and scan at every mode, 100 us so (270 MB from L2 and HBM, 2.7 TB/s; issue-bound).
// SMALL: every bin edge squared fits 32 bits (as in k_estimate_rows).
template <typename V, int J, bool SMALL>
__global__ void __launch_bounds__(256) k_estimate_multi(const V* __restrict__ G, const double* __restrict__ tab_g, MultiArgs a) {
  using R = decltype(V{}.x);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int ng = a.ng, half = ng / 2, H = half + 1;
  double* s_sum = reinterpret_cast<double*>(smem_raw);
  double* s_k = s_sum + a.nbins;
  unsigned long long* s_cnt = reinterpret_cast<unsigned long long*>(s_k + a.nbins);
  R* tab = reinterpret_cast<R*>(s_cnt + a.nbins);  // [kMultiTabRows][ng], the grids' precision
  for (int i = threadIdx.x; i < kMultiTabRows * ng; i += blockDim.x) tab[i] = R(tab_g[i]);
  for (int i = threadIdx.x; i < a.nbins; i += blockDim.x) {
    s_sum[i] = 0.0;
    s_k[i] = 0.0;
    s_cnt[i] = 0ull;
  }
  __syncthreads();
  const R norm = R(1.0 / (double(J) * a.wsums[0]));
  const R vol = R(a.vol);
  const float inv_w2 = 1.0f / float(a.w2);
  const int count = ng * ng * H;  // <= 1024^2 * 513 < 2^31
  const int lane = threadIdx.x & 31;
  const int stride = int(gridDim.x) * int(blockDim.x);
  // this lane's slot, advanced by the grid's stride with carries
  const int step_row = stride / H, step_z = stride - step_row * H;
  const int step_x = step_row / ng, step_y = step_row - step_x * ng;
  int m0 = int(blockIdx.x) * int(blockDim.x) + (threadIdx.x & ~31);
  int iz, iy, ix;
  {
    const int r = (m0 + lane) / H;
    iz = m0 + lane - r * H;
    ix = r / ng;
    iy = r - ix * ng;
  }
  V next[J];
  auto load = [&](int m) {
#pragma unroll
    for (int j = 0; j < J; ++j) next[j] = m < count ? __ldg(G + j * a.grid_stride + m) : V{};
  };
  load(m0 + lane);
  // whole warps step together (the shell sums are warp-collective)
  while (m0 < count) {
    const int m = m0 + lane;
    const bool live = m < count;
    Cx<R> g[J];
#pragma unroll
    for (int j = 0; j < J; ++j) g[j] = {next[j].x, next[j].y};
    // the last round's m0 + stride stays below 2^31: count <= 538 M, stride far below 1.6 G
    load(m + stride);
    int b = -1, mult = 0;
    R pv = R(0);
    const int sx = live ? ix : 0, sy = live ? iy : 0;  // lanes past the last slot read a valid table entry
    const int n2 = [&] {
      const int nx = signed_mode(sx, ng), ny = signed_mode(sy, ng);
      return nx * nx + ny * ny + iz * iz;  // |n_z| = i_z, also on the plane i_z = N/2; < 2^20
    }();
    const bool edge = iz == 0 || iz == half;  // its partner -n is a stored mode of the plane itself
    {
      const R iw = tab[sx] * tab[sy] * tab[iz] * norm;
      Cx<R> e[3][2];
      const int slot[3] = {sx, sy, iz};
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int h = 0; h < 2; ++h) e[d][h] = {tab[(1 + 2 * h) * ng + slot[d]], tab[(2 + 2 * h) * ng + slot[d]]};
      Cx<R> dn = combine<2, R, J>(g, e);
      dn.x *= iw;
      dn.y *= iw;
      if (m == 0) dn = {R(0), R(0)};
      if (a.delta_out && live) {
        V o;
        o.x = dn.x;
        o.y = dn.y;
        static_cast<V*>(a.delta_out)[m] = o;
      }
      if (a.nbins > 0) {
        const R own = fma(dn.x, dn.x, mul_rn(dn.y, dn.y));
        // the partner: conjugate phases, but on a Nyquist slot the mode's own
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if (d == 2 || slot[d] != half) e[d][h].y = -e[d][h].y;
#pragma unroll
        for (int j = 0; j < J; ++j) g[j].y = -g[j].y;  // G(-n) = conj G(n)
        Cx<R> dp = combine<1, R, J>(g, e);
        dp.x *= iw;
        dp.y *= iw;
        const R other = fma(dp.x, dp.x, mul_rn(dp.y, dp.y));
        if (live) {
          const float rn = sqrtf(__int_as_float(0x4B000000 | n2) - 8388608.0f);  // exact conversion
          b = SMALL ? bin_of32(4 * n2, 2.0f * rn, a.lo2, a.w2, inv_w2, a.nbins)
                    : bin_of(4 * (long long)n2, a.lo2, a.w2, a.nbins);
        }
        if (b >= 0) {
          pv = mul_rn(vol, own);
          if (!edge) pv = fma(vol, other, pv);
          mult = edge ? 1 : 2;
        }
      }
    }
    const bool krow = live && iy <= ix && ix <= half;  // carries the |n| sums of (+-n_x, +-n_y) and (+-n_y, +-n_x)
    const int kmult = (ix == 0 || ix == half ? 1 : 2) * (iy == 0 || iy == half ? 1 : 2) * (iy < ix ? 2 : 1);
    m0 += stride;
    iz += step_z;
    iy += step_y;
    ix += step_x;
    if (iz >= H) {
      iz -= H;
      ++iy;
    }
    if (iy >= ng) {
      iy -= ng;
      ++ix;
    }
    if (a.nbins == 0) continue;
    // segmented inclusive scan over runs of equal b; the last lane of each run adds the run's sums
    const int bprev = __shfl_up_sync(0xffffffffu, b, 1);
    const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || bprev != b);
    const int start = 31 - __clz(heads & ((2u << lane) - 1u));
    const int bnext = __shfl_down_sync(0xffffffffu, b, 1);
    const bool end = lane == 31 || bnext != b;
    const unsigned run = ((2u << lane) - 1u) & ~((1u << start) - 1u);
    const int modes = __popc(__ballot_sync(0xffffffffu, mult >= 1) & run) + __popc(__ballot_sync(0xffffffffu, mult == 2) & run);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const R tv = __shfl_up_sync(0xffffffffu, pv, o);
      if (lane - o >= start) pv += tv;
    }
    const bool any_krow = __any_sync(0xffffffffu, krow);
    double kv = 0.0;
    if (any_krow) {
      kv = krow && b >= 0 ? double(mult * kmult) * sqrt_int(max(n2, 1)) : 0.0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const double tk = __shfl_up_sync(0xffffffffu, kv, o);
        if (lane - o >= start) kv += tk;
      }
    }
    if (end && b >= 0) {
      atomicAdd(&s_sum[b], double(pv));
      if (any_krow) atomicAdd(&s_k[b], kv);
      atomicAdd(&s_cnt[b], (unsigned long long)modes);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < a.nbins; i += blockDim.x) {
    if (s_cnt[i] == 0ull) continue;
    atomicAdd(&a.bin_sum[i], s_sum[i]);
    atomicAdd(&a.bin_k[i], s_k[i]);
    atomicAdd(&a.bin_cnt[i], s_cnt[i]);
  }
}

// Tables (1/W and the phases of h = 1, 2) in shared memory behind the bins; every block resident at once.
template <typename V>
cudaError_t launch_estimate_multi(const V* G, const double* tab, const MultiArgs& a, cudaStream_t s) {
  const size_t smem = size_t(a.nbins) * (2 * sizeof(double) + sizeof(unsigned long long)) + sizeof(V) / 2 * kMultiTabRows * size_t(a.ng);
  const bool small = int64_t(a.lo2) + int64_t(a.nbins + 1) * a.w2 <= 46340;
  using Kernel = void (*)(const V*, const double*, MultiArgs);
  Kernel k = nullptr;
  switch (a.J) {
    case 1: k = small ? k_estimate_multi<V, 1, true> : k_estimate_multi<V, 1, false>; break;
    case 2: k = small ? k_estimate_multi<V, 2, true> : k_estimate_multi<V, 2, false>; break;
    case 4: k = small ? k_estimate_multi<V, 4, true> : k_estimate_multi<V, 4, false>; break;
    case 8: k = small ? k_estimate_multi<V, 8, true> : k_estimate_multi<V, 8, false>; break;
    default: return cudaErrorInvalidValue;
  }
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(k), smem);
  if (e != cudaSuccess) return e;
  int per_sm = 1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, 256, smem) != cudaSuccess || per_sm < 1) per_sm = 1;
  const int64_t hc = half_count(a.ng);
  k<<<int(std::min<int64_t>(int64_t(num_sms()) * per_sm, (hc + 255) / 256)), 256, smem, s>>>(G, tab, a);
  count_launch();
  return cudaGetLastError();
}

namespace {

struct MultiLayout {
  void* grids = nullptr;  // [J] padded grids (real) = half-complex after the in-place R2C
  void* shifted = nullptr;
  BinStage b;
  pk_cellpos* sorted = nullptr;
  float* wsorted = nullptr;
  int64_t* offsets = nullptr;
  double* wsums = nullptr;
  double* tab = nullptr;
  double* bin_sum = nullptr;
  double* bin_k = nullptr;
  unsigned long long* bin_cnt = nullptr;
  void* fft_work = nullptr;
  PlanEntry plan;
  int kind = 0;
};

pk_status carve_multi(const pk_config* c, int J, int64_t n, Carver& cv, MultiLayout* L) {
  const bool dbl = c->prec != PK_FP32;
  L->kind = dbl ? 1 : 0;
  L->grids = cv.take<char>(size_t(J) * padded_count(c->ng) * (dbl ? 8 : 4));
  // shifted copies in the input's format (the larger of the two), where later bases are not shifted by the binning
  if (J > 2 && c->prec != PK_FP32) L->shifted = cv.take<char>(size_t(std::max<int64_t>(n, 1)) * 24);
  if (c->prec != PK_FP64) {
    carve_bin_stage(c, n, true, cv, &L->b);
    L->sorted = cv.take<pk_cellpos>(size_t(std::max<int64_t>(n, 1)));
    L->wsorted = cv.take<float>(size_t(std::max<int64_t>(n, 1)));
    const int nt = tiles_per_axis(c->ng);
    L->offsets = cv.take<int64_t>(size_t(int64_t(nt) * nt * nt + 1));
  }
  L->wsums = cv.take<double>(3);
  L->tab = cv.take<double>(size_t(kMultiTabRows) * c->ng);
  L->bin_sum = cv.take<double>(c->nbins);
  L->bin_k = cv.take<double>(c->nbins);
  L->bin_cnt = cv.take<unsigned long long>(c->nbins);
  pk_status st = get_plan(c->ng, L->kind, J, &L->plan);
  if (st != PK_OK) return st;
  L->fft_work = cv.take<char>(std::max<size_t>(L->plan.work, 256));
  return PK_OK;
}

}  // namespace

pk_status multigrid_ws(const pk_config* c, int J, int64_t n, size_t* out) {
  Shifts sh;
  if (!make_shifts(J, &sh)) return fail(PK_EINVAL, "ngrids must be 1, 2, 4 or 8 (got %d)", J);
  Carver cv(nullptr);
  MultiLayout L;
  pk_status st = carve_multi(c, J, n, cv, &L);
  if (st != PK_OK) return st;
  *out = cv.size();
  return PK_OK;
}

}  // namespace pk

using namespace pk;

extern "C" {

size_t pk_multigrid_workspace_size(const pk_config* cfg, int32_t ngrids, int64_t n) {
  clear_err();
  if (validate(cfg) != PK_OK) return 0;
  if (n < 0) {
    fail(PK_EINVAL, "n < 0");
    return 0;
  }
  size_t out = 0;
  return multigrid_ws(cfg, ngrids, n, &out) == PK_OK ? out : 0;
}

pk_status pk_power_multigrid(const pk_config* cfg, int32_t ngrids, const void* pos_dev, int32_t pos_format,
                             const float* w_dev, int64_t n, double* pk_dev, double* kmean_dev, int64_t* nmodes_dev,
                             void* delta_k_dev, void* ws, size_t ws_bytes, void* stream) {
  clear_err();
  pk_status st = validate(cfg);
  if (st != PK_OK) return st;
  Shifts sh;
  if (!make_shifts(ngrids, &sh)) return fail(PK_EINVAL, "ngrids must be 1, 2, 4 or 8 (got %d)", ngrids);
  if (pos_format != PK_POS_F64_XYZ && pos_format != PK_POS_CELL_F32OFF) return fail(PK_EINVAL, "bad pos_format");
  if (n < 1 || !pos_dev) return fail(PK_EINVAL, "need at least one particle");
  if (!pk_dev || !nmodes_dev) return fail(PK_EINVAL, "bad output pointers");
  size_t need = 0;
  if ((st = multigrid_ws(cfg, ngrids, n, &need)) != PK_OK) return st;
  if (!ws || ws_bytes < need) return fail(PK_ESIZE, "workspace %zu < %zu bytes", ws_bytes, need);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  Carver cv(ws);
  MultiLayout L;
  if ((st = carve_multi(cfg, ngrids, n, cv, &L)) != PK_OK) return st;
  const int ng = cfg->ng;
  const bool dbl = cfg->prec != PK_FP32;
  const int64_t per = padded_count(ng);
  const size_t gbytes = size_t(per) * (dbl ? 8 : 4);
  cudaError_t e;
  if ((st = run_weight_sums(w_dev, n, L.wsums, s)) != PK_OK) return st;
  pk_config sub = *cfg;
  sub.interlace = sh.pairs ? 1 : 0;
  const int blocks = int(std::min<int64_t>(int64_t(num_sms()) * 8, (n + 255) / 256));
  const double half = 0.5 * cfg->box / ng;
  // FP32 from FP64 positions: the first (unshifted) base prepares the packed records once; later bases
  // shift those records instead of preparing shifted FP64 positions again
  const bool reuse_prepared = cfg->prec == PK_FP32 && pos_format == PK_POS_F64_XYZ;
  for (int b = 0; b < sh.bases; ++b) {
    const int* hb = sh.h[sh.pairs ? 2 * b : b];
    const void* pos = pos_dev;
    int fmt = pos_format;
    const int shift = (hb[0] ? 1 : 0) | (hb[1] ? 2 : 0) | (hb[2] ? 4 : 0);
    // packed records (given, or prepared by the first, unshifted base) are shifted by the binning on its way; the FP64
    // mode, and FIXED64 from FP64 positions, take a shifted copy
    const bool shift_in_bin = cfg->prec != PK_FP64 && (reuse_prepared || pos_format == PK_POS_CELL_F32OFF);
    if (shift && shift_in_bin) {
      if (reuse_prepared) pos = L.b.cells;
      fmt = PK_POS_CELL_F32OFF;
    } else if (shift) {
      if (pos_format == PK_POS_F64_XYZ)
        k_shift_f64<<<blocks, 256, 0, s>>>(static_cast<const double*>(pos_dev), n, hb[0] * half, hb[1] * half, hb[2] * half,
                                           static_cast<double*>(L.shifted));
      else
        k_shift_cells<<<blocks, 256, 0, s>>>(static_cast<const pk_cellpos*>(pos_dev), n, ng, shift,
                                             static_cast<pk_cellpos*>(L.shifted));
      count_launch();
      if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "shift");
      pos = L.shifted;
    }
    void* grids = static_cast<char*>(L.grids) + gbytes * size_t(sh.pairs ? 2 * b : b);
    if (cfg->prec == PK_FP64) {
      st = run_assign_into(&sub, pos, fmt, nullptr, w_dev, nullptr, n, L.wsums, grids, ng + 2, s);
    } else {
      if ((st = run_bin(&sub, pos, fmt, w_dev, n, L.b, L.sorted, w_dev ? L.wsorted : nullptr, L.offsets, s, nullptr,
                        shift_in_bin ? shift : 0)) != PK_OK)
        return st;
      st = run_assign_into(&sub, nullptr, PK_POS_CELL_F32OFF, L.sorted, w_dev ? L.wsorted : nullptr, L.offsets, n, L.wsums,
                           grids, ng + 2, s);
    }
    if (st != PK_OK) return st;
  }
  if ((st = exec_plan(L.plan, L.kind, L.grids, L.fft_work, s)) != PK_OK) return st;
  k_multi_tables<<<(ng + 127) / 128, 128, 0, s>>>(L.tab, ng, cfg->order); count_launch();
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "tables");
  if ((e = clear_bins(L.bin_sum, L.bin_cnt, size_t(cfg->nbins), s)) != cudaSuccess) return cuda_fail(e, "memset");
  MultiArgs a{};
  a.ng = ng;
  a.J = ngrids;
  a.nbins = cfg->nbins;
  a.lo2 = cfg->bin_lo2;
  a.w2 = cfg->bin_w2;
  a.grid_stride = per / 2;
  a.vol = cfg->box * cfg->box * cfg->box;
  a.wsums = L.wsums;
  a.bin_sum = L.bin_sum;
  a.bin_k = L.bin_k;
  a.bin_cnt = L.bin_cnt;
  a.delta_out = delta_k_dev;
  e = dbl ? launch_estimate_multi(static_cast<const double2*>(L.grids), L.tab, a, s)
          : launch_estimate_multi(static_cast<const float2*>(L.grids), L.tab, a, s);
  if (e != cudaSuccess) return cuda_fail(e, "estimate");
  EstimateArgs f{};
  f.ng = ng;
  f.nbins = cfg->nbins;
  f.bin_lo2 = cfg->bin_lo2;
  f.bin_w2 = cfg->bin_w2;
  f.box = cfg->box;
  f.wsums = L.wsums;
  f.bin_sum = L.bin_sum;
  f.bin_k = L.bin_k;
  f.bin_cnt = L.bin_cnt;
  if ((e = launch_finalize(f, cfg->subtract_shot, pk_dev, kmean_dev, nmodes_dev, s)) != cudaSuccess)
    return cuda_fail(e, "finalize");
  return PK_OK;
}

}  // extern "C"
