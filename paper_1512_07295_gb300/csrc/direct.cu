// Direct summation of the Fourier coefficients of a particle set (eq:deltaDS, Sec. 2.2): the
// alias-free, window-free reference against which grid estimators are compared (Sec. 3.2), at cost
// N_P x (number of modes); and the binned cross power of two half-complex fields.
//
// For every stored mode of the half-complex layout [N][N][N/2+1] (signed n as in pk_fft_estimate):
//   delta(n) = (1/sum w) sum_i w_i exp(-2 pi i n.x_i/L),   delta(0) = 0.
// The sum is separable: with rows r = (i_x, i_z) and columns c = i_y,
//   delta[r][c] = sum_i a_i(r) b_i(c),  a_i(r) = w_i e^{-2 pi i (n_x x + n_z z)/L},  b_i(c) = e^{-2 pi i n_y y/L},
// a complex matrix product over the particles. Phases are exact integer products n * Phi of a
// fixed-point position fraction Phi = x/L mod 1 (32 bits in FP32, 64 in FP64) before the sine and
// cosine are taken, so no large argument is ever reduced in floating point.
//   FP32: k_ds_modes_tc, the product on the tensor cores (tcgen05, TF32 operands split in two).
//   FP64: k_ds_modes, FP64 FMAs on the CUDA cores in 256 x 32 mode tiles, each thread a 4 x 8
//         register tile, operands built in shared memory from per-particle, per-axis phase tables.
// Partial sums of particle slices meet in FP64 atomics.
#include "host.cuh"
#include "tc.cuh"

namespace pk {

PK_ERR_ACCESSOR(take_err_direct)

constexpr int kDsRows = 256;  // rows (i_x, i_z) per block
constexpr int kDsCols = 32;   // columns i_y per block
constexpr int kDsThreads = 256;

template <typename R>
struct DsT;
template <>
struct DsT<float> {
  using Phase = uint32_t;
  struct Rec {
    uint32_t px, py, pz;
    float w;
  };
  __device__ __forceinline__ static Phase from_frac(double t) { return uint32_t((unsigned long long)rint(t * 4294967296.0)); }
};
template <>
struct DsT<double> {
  using Phase = uint64_t;
  struct Rec {
    uint64_t px, py, pz;
    double w;
  };
  __device__ __forceinline__ static Phase from_frac(double t) {
    const double th = t * 4294967296.0;
    const double hi = floor(th);
    const double lo = rint((th - hi) * 4294967296.0);
    return ((unsigned long long)hi << 32) + (unsigned long long)lo;
  }
  // w e^{-2 pi i T/2^64}
  __device__ __forceinline__ static void expi(Phase t, double w, double& re, double& im) {
    double s, c;
    sincospi(double(int64_t(t)) * 1.0842021724855044340e-19, &s, &c);  // 2^-63
    re = w * c;
    im = -(w * s);
  }
};


// Positions -> fixed-point phase fractions and weights; per-block partial sums of the weights.
template <typename R>
__global__ void __launch_bounds__(256) k_ds_prep(const void* __restrict__ pos, int fmt, const float* __restrict__ w,
                                                 int64_t n, int ng, double box, typename DsT<R>::Rec* __restrict__ out,
                                                 double* __restrict__ wpart) {
  double local = 0.0;
  for (int64_t i = gtid(); i < n; i += gstride()) {
    double t[3];
    if (fmt == PK_POS_F64_XYZ) {
      const double* p = static_cast<const double*>(pos) + 3 * i;
      bool bad = false;
      for (int a = 0; a < 3; ++a) {
        double x = p[a];
        if (!isfinite(x)) bad = true;
        const double q = x / box;
        t[a] = q - floor(q);
      }
      if (bad) {
        raise_err(PK_DERR_NONFINITE);
        t[0] = t[1] = t[2] = 0.0;
      }
    } else {
      const pk_cellpos r = static_cast<const pk_cellpos*>(pos)[i];
      const int c[3] = {cell_x(r.cell), cell_y(r.cell), cell_z(r.cell)};
      const float f[3] = {r.fx, r.fy, r.fz};
      bool bad = false;
      for (int a = 0; a < 3; ++a) {
        if (c[a] >= ng || !(f[a] >= 0.0f && f[a] < 1.0f)) bad = true;
        t[a] = (double(c[a]) + double(f[a])) / double(ng);
      }
      if (bad) {
        raise_err(PK_DERR_CELLRANGE);
        t[0] = t[1] = t[2] = 0.0;
      }
    }
    const double wi = w ? double(w[i]) : 1.0;
    typename DsT<R>::Rec rec;
    rec.px = DsT<R>::from_frac(t[0]);
    rec.py = DsT<R>::from_frac(t[1]);
    rec.pz = DsT<R>::from_frac(t[2]);
    rec.w = R(wi);
    out[i] = rec;
    local += double(rec.w);
  }
  __shared__ double red[256];
  red[threadIdx.x] = local;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) wpart[blockIdx.x] = red[0];
}

// sum w from the per-block partials, in a fixed order.
__global__ void k_ds_wsum(const double* __restrict__ wpart, int nblk, double* __restrict__ wsum) {
  __shared__ double red[256];
  double v = 0.0;
  for (int i = threadIdx.x; i < nblk; i += 256) v += wpart[i];
  red[threadIdx.x] = v;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) *wsum = red[0];
}

// Mode tiles. A block owns 256 rows r = (i_x, i_z) x 32 columns i_y of the mode matrix. Rows with
// i_z < N/2 come in rectangles of 8 i_x x 32 i_z, so a row operand is the product of two per-particle
// tables, w e^{-2 pi i n_x x/L} (8 entries) and e^{-2 pi i n_z z/L} (32 entries); the rows of the
// Nyquist plane i_z = N/2 (n_z = -N/2) come 256 i_x at a time and take their operands directly.
constexpr int kDsTx = 8, kDsTz = 32;
__host__ __device__ inline int ds_main_x_tiles(int ng) { return (ng + kDsTx - 1) / kDsTx; }
__host__ __device__ inline int ds_main_z_tiles(int ng) { return (ng / 2 + kDsTz - 1) / kDsTz; }
__host__ __device__ inline int ds_row_tiles(int ng) {
  return ds_main_x_tiles(ng) * ds_main_z_tiles(ng) + (ng + kDsRows - 1) / kDsRows;
}

// Shared-memory order of the operands, chosen so that the 16-byte loads of the register tiles take one
// wavefront: in each 32-row warp block, row 4 rg + q sits at (q/2) 16 + 2 rg + q%2; column 8 cg + j
// at (j/2) 8 + 2 cg + j%2.
__device__ __forceinline__ int ds_row_slot(int l) {
  const int w = l >> 5, rg = (l >> 2) & 7, q = l & 3;
  return 32 * w + (q >> 1) * 16 + 2 * rg + (q & 1);
}
__device__ __forceinline__ int ds_col_slot(int c) {
  const int cg = c >> 3, j = c & 7;
  return (j >> 1) * 8 + 2 * cg + (j & 1);
}

// One block: a row tile x 32 columns of the mode matrix, the particles of one slice. acc_out: FP64 sums
// on the half-complex layout [N][N][N/2+1], added to with atomics. Each thread accumulates a 4 x 8
// register tile of complex sums with four scalar FMAs per product.
constexpr int kDsK = 32;  // particles per chunk
__global__ void __launch_bounds__(kDsThreads, 1) k_ds_modes(const DsT<double>::Rec* __restrict__ recs, int64_t n, int ng,
                                                             int64_t slice_len, double2* __restrict__ acc_out) {
  using Rec = DsT<double>::Rec;
  using Phase = DsT<double>::Phase;
  constexpr int K = kDsK;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* sA = reinterpret_cast<double2*>(smem_raw);  // [K][kDsRows], row slots
  double2* sB = sA + K * kDsRows;                 // [K][kDsCols], column slots
  double2* sEx = sB + K * kDsCols;                // [K][kDsTx]
  double2* sEz = sEx + K * kDsTx;                 // [K][kDsTz]

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int H = ng / 2 + 1;
  const int col0 = blockIdx.y * kDsCols;
  const int64_t k_beg = int64_t(blockIdx.z) * slice_len;
  const int64_t k_end = min(n, k_beg + slice_len);

  // this block's rows: tile origin, and for row l the mode (i_x, i_z) = (ix0 + l / tz, iz0 + l % tz)
  const int tmain = ds_main_x_tiles(ng) * ds_main_z_tiles(ng);
  const bool nyq = int(blockIdx.x) >= tmain;
  int ix0, iz0;
  if (!nyq) {
    ix0 = (int(blockIdx.x) / ds_main_z_tiles(ng)) * kDsTx;
    iz0 = (int(blockIdx.x) % ds_main_z_tiles(ng)) * kDsTz;
  } else {
    ix0 = (int(blockIdx.x) - tmain) * kDsRows;
    iz0 = ng / 2;
  }
  // operand generation: the row of thread tid is l = tid (main: i_x = ix0 + warp, i_z = iz0 + lane)
  const int my_ix = nyq ? ix0 + tid : ix0 + warp;
  const int my_iz = nyq ? iz0 : iz0 + lane;
  const bool row_ok = my_ix < ng && (nyq || my_iz < ng / 2);
  const Phase nx_row = Phase(int64_t(signed_mode(min(my_ix, ng - 1), ng)));
  const Phase nz_nyq = Phase(int64_t(-(ng / 2)));
  const int a_slot = ds_row_slot(tid);
  // table entries of thread tid: Ex[k][x] for x = tid & 7; Ez[k][lane] and B[k][lane] for k = warp + 8 j
  const int tx_ix = ix0 + (tid & 7);
  const Phase nx_tab = Phase(int64_t(signed_mode(min(tx_ix, ng - 1), ng)));
  const bool tx_ok = tx_ix < ng;
  const Phase nz_tab = Phase(int64_t(iz0 + lane));
  const bool tz_ok = iz0 + lane < ng / 2;
  const int gen_col = col0 + lane;
  const bool col_ok = gen_col < ng;
  const Phase ny = Phase(int64_t(signed_mode(min(gen_col, ng - 1), ng)));
  const int b_slot = ds_col_slot(lane);

  // register tile: rows 32 warp + 4 rg + (0..3), columns 8 cg + (0..7)
  const int rg = lane >> 2, cg = lane & 3;
  double acc[64];
#pragma unroll
  for (int i = 0; i < 64; ++i) acc[i] = 0.0;

  for (int64_t k0 = k_beg; k0 < k_end; k0 += K) {
    const int cnt = int(min(int64_t(K), k_end - k0));
    __syncthreads();  // the previous chunk's operands are consumed
    // per-particle tables (Ex carries the weight) and the column operands
    for (int e = tid; e < K * kDsTx; e += kDsThreads) {
      const int k = e >> 3;
      double re = 0.0, im = 0.0;
      if (k < cnt && tx_ok && !nyq) {
        const Rec r = recs[k0 + k];
        DsT<double>::expi(Phase(nx_tab * r.px), r.w, re, im);
      }
      sEx[e] = double2{re, im};
    }
#pragma unroll
    for (int j = 0; j < K / 8; ++j) {
      const int k = warp + 8 * j;
      double bre = 0.0, bim = 0.0, zre = 0.0, zim = 0.0;
      if (k < cnt) {
        const Rec r = recs[k0 + k];
        if (col_ok) DsT<double>::expi(Phase(ny * r.py), 1.0, bre, bim);
        if (tz_ok && !nyq) DsT<double>::expi(Phase(nz_tab * r.pz), 1.0, zre, zim);
      }
      sB[k * kDsCols + b_slot] = double2{bre, bim};
      sEz[k * kDsTz + lane] = double2{zre, zim};
    }
    __syncthreads();
    if (!nyq) {
#pragma unroll 4
      for (int k = 0; k < K; ++k) {
        const double2 x = sEx[k * kDsTx + warp], z = sEz[k * kDsTz + lane];
        double2 a;
        a.x = row_ok ? x.x * z.x - x.y * z.y : 0.0;
        a.y = row_ok ? x.x * z.y + x.y * z.x : 0.0;
        sA[k * kDsRows + a_slot] = a;
      }
    } else {
#pragma unroll 4
      for (int k = 0; k < K; ++k) {
        double re = 0.0, im = 0.0;
        if (row_ok && k < cnt) {
          const Rec r = recs[k0 + k];
          DsT<double>::expi(Phase(nx_row * r.px + nz_nyq * r.pz), r.w, re, im);
        }
        sA[k * kDsRows + a_slot] = double2{re, im};
      }
    }
    __syncthreads();
#pragma unroll 2
    for (int k = 0; k < K; ++k) {
      double2 a[4], b[8];
      const double2* pa = sA + k * kDsRows + 32 * warp + 2 * rg;
      const double2* pb = sB + k * kDsCols + 2 * cg;
      a[0] = pa[0];
      a[1] = pa[1];
      a[2] = pa[16];
      a[3] = pa[17];
#pragma unroll
      for (int j2 = 0; j2 < 4; ++j2) {
        b[2 * j2] = pb[8 * j2];
        b[2 * j2 + 1] = pb[8 * j2 + 1];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          double& re = acc[2 * (8 * i + j)];
          double& im = acc[2 * (8 * i + j) + 1];
          re = fma(a[i].x, b[j].x, re);
          re = fma(-a[i].y, b[j].y, re);
          im = fma(a[i].x, b[j].y, im);
          im = fma(a[i].y, b[j].x, im);
        }
      }
    }
  }

#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int l = 32 * warp + 4 * rg + i;
    const int ix = nyq ? ix0 + l : ix0 + (l >> 5);
    const int iz = nyq ? iz0 : iz0 + (l & 31);
    if (ix >= ng || (!nyq && iz >= ng / 2)) continue;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int c = col0 + 8 * cg + j;
      if (c >= ng) continue;
      double2* dst = acc_out + (int64_t(ix) * ng + c) * H + iz;
      const int q = 2 * (8 * i + j);
      atomicAdd(&dst->x, acc[q]);
      atomicAdd(&dst->y, acc[q + 1]);
    }
  }
}

// delta = sums / sum w in the output precision; delta(0) = 0.
template <typename V>
__global__ void k_ds_finish(const double2* __restrict__ sums, const double* __restrict__ wsum, int64_t count,
                            V* __restrict__ out) {
  const double inv = 1.0 / *wsum;
  for (int64_t m = gtid(); m < count; m += gstride()) {
    const double2 v = sums[m];
    V o;
    o.x = m == 0 ? 0.0 : v.x * inv;
    o.y = m == 0 ? 0.0 : v.y * inv;
    out[m] = o;
  }
}

// One lane's run of equal bins: bin (-2: none yet), sum of Re[a conj b] and of |n| (slots counted once on the
// planes of multiplicity 1 at half weight), modes.
struct CrossRun {
  int b;
  double v, k;
  int c;
};

// Private bins of k_cross_rows: one copy per row of a warp, updated without atomics.
struct CrossBin {
  double sum, k;
};

__device__ __forceinline__ void cross_add(CrossBin* pw, unsigned* cw, int b, double v, double k, int c, bool krow) {
  pw[b].sum += v;
  if (krow) pw[b].k += k;
  cw[b] += unsigned(c);
}

// x (halved if half) as a double, for x = 0 (+0) or a normal float: integer instructions (exponent rebased,
// significand moved up), as the conversion instruction runs on the FP64 pipe.
__device__ __forceinline__ double widen(float x, bool half) {
  const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
  const unsigned hi = (b & 0x80000000u) | ((m >> 3) + (half ? 0x37f00000u : 0x38000000u));
  return __hiloint2double(m ? int(hi) : 0, int(b << 29));
}
__device__ __forceinline__ bool widens(float x) {
  const unsigned m = __float_as_uint(x) & 0x7fffffffu;
  return m == 0u || m - 0x00800000u < 0x7f000000u;
}
// acc + Re[a conj c] (half of it if half); called by whole warps.
__device__ __forceinline__ double cross_term(float2 a, float2 c, bool half, double acc) {
  // subnormals, infinities and NaN (in any lane) take the conversion instructions
  if (__any_sync(0xffffffffu, !(widens(a.x) && widens(a.y) && widens(c.x) && widens(c.y)))) {
    const double w = half ? 0.5 : 1.0;
    return fma(w * double(a.x), double(c.x), fma(w * double(a.y), double(c.y), acc));
  }
  return fma(widen(a.x, half), widen(c.x, false), fma(widen(a.y, half), widen(c.y, false), acc));
}
__device__ __forceinline__ double cross_term(double2 a, double2 c, bool half, double acc) {
  const double w = half ? 0.5 : 1.0;
  return fma(w * a.x, c.x, fma(w * a.y, c.y, acc));
}

// Binned V Re[a(n) conj b(n)] over the stored modes, each with its multiplicity (2 for 0 < i_z < N/2, where the unstored
// partner -n adds the conjugate product; 1 on the planes i_z = 0 and N/2), by rows as k_estimate_rows: a warp takes
// RW rows (i_x, i_y) at a time, and the L = 32 / RW lanes of a row share its slots within the bins, consecutive ones to a
// lane; slots outside every bin are not read. Along a row |n| grows with i_z, so a lane's slots form runs of
// equal bins, summed in registers; runs inside a lane go to the row's private bins without atomics, and one
// segmented scan per row joins the runs that continue across lanes.
// FP64 arithmetic is the scarce unit (2 operations per clock and SM), so a mode costs two multiply-adds: the floats
// become doubles by integer instructions, V is applied to whole bins, and the sums of |n|, which depend on
// (|n_x|, |n_y|, n_z) and not on the order of n_x and n_y, are taken on the rows 0 <= i_y <= i_x <= N/2 alone,
// an eighth of them, with the rows' multiplicity.
// Whole call, FP32 fields, N = 256: 376 us with one atomic per mode and sum, 117 us with private bins and every slot read,
// 91 us now (the default bins hold half of the slots). Few bins on a large grid (8 bins up to |n| = 80, N = 512): 470 us
// with the atomics, which skipped the modes outside, 580 us with every slot read, 68 us now. One bin for all modes
// (N = 400): 14.8 ms with the atomics, 0.32 now.
template <typename V>
__global__ void __launch_bounds__(256, 3) k_cross_rows(const V* __restrict__ da, const V* __restrict__ db, int ng, double vol,
                                                       int lo2, int w2, int nbins, int RW, double* __restrict__ bin_sum,
                                                       double* __restrict__ bin_k, unsigned long long* __restrict__ bin_cnt) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int ncopy = int(blockDim.x >> 5) * RW;
  CrossBin* pbin = reinterpret_cast<CrossBin*>(smem_raw);
  unsigned* pcnt = reinterpret_cast<unsigned*>(pbin + size_t(ncopy) * nbins);
  for (int i = threadIdx.x; i < ncopy * nbins; i += blockDim.x) {
    pbin[i].sum = 0.0;
    pbin[i].k = 0.0;
    pcnt[i] = 0u;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, half = ng / 2, lz = half + 1;
  const int L = 32 / RW, grp = lane / L, sub = lane - grp * L;
  const float lo_sq = 0.25f * float(lo2) * float(lo2), hi_sq = 0.25f * float(lo2 + nbins * w2) * float(lo2 + nbins * w2);
  CrossBin* pw = pbin + size_t((threadIdx.x >> 5) * RW + grp) * nbins;
  unsigned* cw = pcnt + size_t((threadIdx.x >> 5) * RW + grp) * nbins;
  const float inv_w2 = 1.0f / float(w2);
  const int rows = ng * ng;
  const int nwarps = int((int64_t(gridDim.x) * blockDim.x) >> 5);
  for (int row0 = int((int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5) * RW; row0 < rows; row0 += nwarps * RW) {
    const int row = min(row0 + grp, rows - 1);
    const int ix = row / ng;
    int iy = row - ix * ng + ix;  // rows of one i_y lie apart in the order of the work: those within the bins are short or long by i_y
    if (iy >= ng) iy -= ng;
    const int nx = signed_mode(ix, ng), ny = signed_mode(iy, ng);
    const int nxy2 = nx * nx + ny * ny;
    // the slots within the bins, and up to two beside them (the bin test decides): the others are not read
    const int zb = max(0, int(sqrtf(fmaxf(lo_sq - float(nxy2), 0.0f))) - 1);
    int ze = hi_sq > float(nxy2) ? min(lz, int(fminf(sqrtf(hi_sq - float(nxy2)), float(lz))) + 2) : 0;
    if (row0 + grp >= rows) ze = 0;  // rows past the last
    const int per = max(0, (ze - zb + L - 1) / L);  // per lane
    const int J = int(__reduce_max_sync(0xffffffffu, unsigned(per)));
    if (J == 0) continue;
    const int z0 = min(zb + sub * per, ze), z1 = min(z0 + per, ze);
    // rows that carry the |n| sums of the rows (+-n_x, +-n_y) and (+-n_y, +-n_x)
    const bool krow = iy <= ix && ix <= half;
    const double kmult = double((ix == 0 || ix == half ? 1 : 2) * (iy == 0 || iy == half ? 1 : 2) * (iy < ix ? 2 : 1));
    const V* pa = da + (int64_t(ix) * ng + iy) * lz;
    const V* pb = db + (int64_t(ix) * ng + iy) * lz;
    CrossRun head = {-2, 0.0, 0.0, 0}, cur = {-2, 0.0, 0.0, 0};
    constexpr int PF = 2;  // the next two slots' loads are in flight while a slot is summed
    V qa[PF] = {}, qb[PF] = {};
#pragma unroll
    for (int u = 0; u < PF; ++u)
      if (z0 + u < z1) {
        qa[u] = __ldg(pa + z0 + u);
        qb[u] = __ldg(pb + z0 + u);
      }
    const bool any_krow = __any_sync(0xffffffffu, krow);
    // the lanes step together and the FP64 operations run without branches around them: an FP64 instruction
    // takes the same 16 clocks for a few lanes as for all
    for (int j = 0; j < J; ++j) {
      const int iz = z0 + j;
      const V a = qa[0], c = qb[0];
#pragma unroll
      for (int u = 0; u + 1 < PF; ++u) {
        qa[u] = qa[u + 1];
        qb[u] = qb[u + 1];
      }
      if (iz + PF < z1) {
        qa[PF - 1] = __ldg(pa + iz + PF);
        qb[PF - 1] = __ldg(pb + iz + PF);
      }
      const int n2 = nxy2 + iz * iz;  // |n_z| = i_z, also on the plane i_z = N/2
      const float rn = sqrtf(__int_as_float(0x4B000000 | n2) - 8388608.0f);  // n2 < 2^21, exact in FP32
      const bool live = iz < z1;
      const int b = live ? bin_of32(4 * n2, 2.0f * rn, lo2, w2, inv_w2, nbins) : cur.b;
      __syncwarp();
      if (b != cur.b && cur.b != -2 && head.b != -2 && cur.b >= 0)  // the run cur.b began and ended inside this lane
        cross_add(pw, cw, cur.b, cur.v, cur.k, cur.c, krow);
      __syncwarp();
      if (b != cur.b) {
        if (cur.b != -2 && head.b == -2) head = cur;
        cur = {b, 0.0, 0.0, 0};
      }
      const bool in = live && b >= 0;
      const bool edge = iz == 0 || iz == half;  // its partner -n is a stored mode of the plane itself
      const double v = cross_term(a, c, edge, cur.v);
      cur.v = in ? v : cur.v;
      cur.c += in ? (edge ? 1 : 2) : 0;
      if (any_krow) {  // warp-uniform
        const double k = fma(edge ? 0.5 * kmult : kmult, sqrt_int(max(n2, 1)), cur.k);
        cur.k = in && krow ? k : cur.k;
      }
    }
    // runs at the lane's two ends: one run only (pass) or a head and a tail (cur), joined across the row
    const bool pass = head.b == -2;
    const int first = pass ? cur.b : head.b;
    const int next_first = __shfl_down_sync(0xffffffffu, first, 1);
    const bool cont = sub < L - 1 && cur.b >= 0 && next_first == cur.b;
    const bool prev_cont = __shfl_up_sync(0xffffffffu, cont ? 1 : 0, 1) != 0 && sub > 0;
    const unsigned starts = __ballot_sync(0xffffffffu, sub == 0 || !(prev_cont && pass));
    const int start = 31 - __clz(starts & ((2u << lane) - 1u));
    double sv = cur.v, sk = cur.k;
    int sc = cur.c;
    // segments longer than two lanes are rare away from the i_z = 0 end: stop when none reaches further
    for (int o = 1; o < 32; o <<= 1) {
      if (__all_sync(0xffffffffu, lane - o < start)) break;
      const double tv = __shfl_up_sync(0xffffffffu, sv, o);
      const double tk = __shfl_up_sync(0xffffffffu, sk, o);
      const int tc = __shfl_up_sync(0xffffffffu, sc, o);
      if (lane - o >= start) {
        sv += tv;
        if (krow) sk += tk;
        sc += tc;
      }
    }
    const double iv = __shfl_up_sync(0xffffffffu, sv, 1), ik = __shfl_up_sync(0xffffffffu, sk, 1);
    const int ic = __shfl_up_sync(0xffffffffu, sc, 1);
    if (!pass && head.b >= 0) {
      if (prev_cont)
        cross_add(pw, cw, head.b, head.v + iv, krow ? head.k + ik : 0.0, head.c + ic, krow);
      else
        cross_add(pw, cw, head.b, head.v, head.k, head.c, krow);
    }
    __syncwarp();
    if (cur.b >= 0 && !cont) cross_add(pw, cw, cur.b, sv, sk, sc, krow);
    __syncwarp();
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nbins; i += blockDim.x) {
    double v = 0.0, k = 0.0;
    unsigned long long c = 0;
    for (int q = 0; q < ncopy; ++q) {
      v += pbin[q * nbins + i].sum;
      k += pbin[q * nbins + i].k;
      c += pcnt[q * nbins + i];
    }
    if (c) {
      atomicAdd(&bin_sum[i], 2.0 * vol * v);
      if (k != 0.0) atomicAdd(&bin_k[i], 2.0 * k);
      atomicAdd(&bin_cnt[i], c);
    }
  }
}

// ---- FP32 on the tensor cores (tcgen05, kind::tf32) -----------------------------------------------------
//
// Rows are the pairs p = i_x H + i_z (H = N/2 + 1) with the phase theta = 2 pi (n_x x + n_z z)/L, columns
// the numbers n_y = 0 .. N/2 with phi = 2 pi n_y y/L. The modes n_y and -n_y share four real sums:
//   D0[p][c] = sum w cos theta f_c(phi),  D1[p][c] = sum w sin theta f_c(phi),  f_c = cos or sin,
//   delta(n_y)  = (D0cos - D1sin) - i (D1cos + D0sin),
//   delta(-n_y) = (D0cos + D1sin) - i (D1cos - D0sin),
// half the products of a complex matrix product over all i_y (two real products per mode instead of
// four, K = 1 per particle instead of 2), and half the column operands.
// A block owns 128 pairs x NCOL real columns (NCOL / 2 values of n_y): two M = 128 accumulators, D0
// and D1, that share the B operand.
//  - A (cos and sin of 128 pairs) goes from the registers that computed it straight to TMEM (row =
//    lane): with A in shared memory an M = 128, N = 80 MMA would read 6.6 KB per 40 clocks, above the
//    128 B per clock of the SM; B alone is 64 B per clock.
//  - B (w cos, w sin) is K-major in shared memory without swizzle: 8-row x 16-byte core matrices,
//    K-adjacent cores 128 B apart (LBO), 8-row groups (kTcK / 4) 128 B apart (SBO).
// TF32 keeps 10 mantissa bits, so each operand x is split into big = x rounded to TF32 and small = x - big
// (exact in FP32, at most 12 bits, of which TF32 keeps 11), and D accumulates big.big + big.small + small.big:
// each product then errs by at most 2^-21 of its size, 2^-23 from each operand's small part and 2^-22 from the
// product of the two that is left out.
//
// Pipeline over chunks of 16 particles in three operand stages. 16 warps build operands and signal
// full[stage]; a warp of its own issues the chunk's MMAs and commits them to empty[stage]. (An issuing
// thread stalls while the MMA queue is full: one that also builds holds back every barrier of the block.)
// Four chunks form a run of 64 particles with accumulators of its own (two in turn); when a building warp
// finds the last chunk of a run done, on its way to reuse that chunk's stage, it adds its share of
// the accumulators to compensated pairs in registers (TwoSum, packed two by two). A
// run's records arrive by bulk copy two runs ahead in a ring of four. Every mbarrier wait is bounded in
// time.
//
// Bound: the building warps, which keep the issue slots 70 % busy and set the pace (0.80 us per chunk against 0.26 us
// of MMAs of 44.5 clocks each; tensor pipe 29 % busy). 64^3 particles on N = 64, whole call: 3.86 ms (complex
// product, one barrier-stepped pipeline) to 1.58 ms; 128^3 on N = 128: 262 ms to 88 ms.
constexpr int kTcRows = 128, kTcK = 16, kTcRun = 4, kTcRunLen = kTcRun * kTcK, kTcStages = 3, kTcRing = 4;
// 16 building warps and a warpgroup whose first warp issues. Registers: launched with 96 per thread (640
// threads), the issuing warpgroup keeps 32 and the building ones take 112: 4 x 112 + 32 = 5 x 96.
constexpr int kTcBuilders = 16, kTcThreads = 32 * (kTcBuilders + 4);
constexpr int kTcMaxCols = 80;  // real columns per block at most
// accumulators and A stages, rounded up to a power of two (TMEM is allocated so): all 512 at kTcMaxCols
__host__ __device__ constexpr uint32_t tc_tmem_cols(int ncol) { return 4 * ncol + kTcStages * 4 * kTcK <= 256 ? 256 : 512; }
static_assert(4 * kTcMaxCols + kTcStages * 4 * kTcK <= 512, "an SM has 512 TMEM columns");
constexpr uint64_t kTcWaitNs = 1000000000ull;  // bound of every mbarrier wait
constexpr uint32_t kTcSbo = (kTcK / 4) * 128;  // 8-row groups of B

inline int64_t tc_row_tiles(int ng) { return (int64_t(ng) * (ng / 2 + 1) + kTcRows - 1) / kTcRows; }
// n_y values per block: the N/2 + 1 values in as few blocks as the accumulators allow, a multiple of 8 each
inline int tc_col_tiles(int ng) { return (ng / 2 + 1 + kTcMaxCols / 2 - 1) / (kTcMaxCols / 2); }
inline int tc_cols(int ng) {
  const int t = tc_col_tiles(ng), per = (ng / 2 + 1 + t - 1) / t;
  return 2 * ((per + 7) / 8 * 8);
}

template <int NCOL>
struct TcSmem {  // byte offsets in the dynamic shared memory (base aligned to 128)
  static constexpr uint32_t b_part = NCOL * kTcK * 4;
  static constexpr uint32_t stage = 2 * b_part;  // B big, B small
  static constexpr uint32_t rec = kTcStages * stage;           // [kTcRing][kTcRunLen] records
  static constexpr uint32_t full = rec + kTcRing * kTcRunLen * 16, empty = full + 8 * kTcStages;
  static constexpr uint32_t ring = empty + 8 * kTcStages, tmem = ring + 8 * kTcRing, total = tmem + 16;
};

// e^{i 2 pi T / 2^32}: the phase T (a fraction of a turn, exact in integers) becomes an angle in
// [-pi, pi) and the hardware sine and cosine (__sincosf, absolute error about 2^-21.4 there) take it.
__device__ __forceinline__ void tc_sincos(uint32_t t, float& s, float& c) {
  __sincosf(float(int32_t(t)) * 1.46291807926715968e-9f, &s, &c);  // pi / 2^31
}

template <int NCOL>
__global__ void __launch_bounds__(kTcThreads, 1) k_ds_modes_tc(const DsT<float>::Rec* __restrict__ recs, int64_t n, int ng,
                                                               int64_t slice_len, double2* __restrict__ acc_out) {
  static_assert(NCOL % 16 == 0 && NCOL <= kTcMaxCols, "an M = 128 MMA takes N in steps of 16");
  using Rec = DsT<float>::Rec;
  using Sm = TcSmem<NCOL>;
  constexpr int CY = NCOL / 2;   // n_y values of the block: B row 2 j is w cos, 2 j + 1 is w sin of value j
  constexpr int PT = NCOL / 2;   // accumulator columns per thread
  constexpr uint32_t kIdesc = tc::idesc_tf32(NCOL, kTcRows);
  // TMEM columns: accumulators (buffer, D0 / D1) of NCOL, then the A stages (D0 / D1, big / small) of kTcK
  constexpr uint32_t kABase = 4 * NCOL;
  extern __shared__ __align__(128) unsigned char smem_tc[];
  unsigned char* sm = smem_tc;
  const uint32_t sbase = uint32_t(__cvta_generic_to_shared(sm));
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + Sm::tmem);

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int H = ng / 2 + 1;
  const int col0 = blockIdx.y * CY;
  const int64_t k_beg = int64_t(blockIdx.z) * slice_len;
  const int64_t k_end = min(n, k_beg + slice_len);
  const int nchunks = k_end > k_beg ? int((k_end - k_beg + kTcK - 1) / kTcK) : 0;
  const int nruns = (nchunks + kTcRun - 1) / kTcRun;
  volatile int* s_bad = reinterpret_cast<volatile int*>(sm + Sm::tmem + 4);  // a wait ran out

  if (warp == 0) tc::tmem_alloc(sbase + Sm::tmem, tc_tmem_cols(NCOL));
  if (tid == 0) {
    *s_bad = 0;
    for (int q = 0; q < kTcStages; ++q) {
      tc::mbar_init(sbase + Sm::full + 8 * q, kTcBuilders);
      tc::mbar_init(sbase + Sm::empty + 8 * q, 1);
    }
    for (int q = 0; q < kTcRing; ++q) tc::mbar_init(sbase + Sm::ring + 8 * q, 1);
    tc::fence_mbar_init();
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = *tmem_slot;
  bool bad = false;
  // a bounded wait; every other wait of the block gives up once one has run out
  auto wait = [&](uint32_t bar, int use) {
    bad = !tc::wait(sbase + bar, uint32_t(use) & 1u, kTcWaitNs, s_bad);
    return !bad;
  };

  if (warp >= kTcBuilders) {  // ---- records and MMAs
    tc::regs_dec<32>();
    if (warp == kTcBuilders && lane == 0) {
      auto load_run = [&](int r) {
        const int64_t k0 = k_beg + int64_t(r) * kTcRunLen;
        tc::bulk_load(sbase + Sm::rec + uint32_t((r % kTcRing) * kTcRunLen * 16), recs + k0,
                      uint32_t(min(int64_t(kTcRunLen), k_end - k0)) * 16u, sbase + Sm::ring + 8 * (r % kTcRing));
      };
      int loaded = 0;
      for (; loaded < min(2, nruns); ++loaded) load_run(loaded);
      int issued = 0;
      int st = 0, use = 0;  // chunk c's stage and the stage's use: c % kTcStages, c / kTcStages
      for (int c = 0; c < nchunks && wait(Sm::full + 8 * st, use); ++c) {
        // chunk c built by every warp: no warp reads the records of run c / kTcRun - 2 any more
        if (c % kTcRun == 0 && loaded < nruns) load_run(loaded++);
        tc::fence_after();
        const uint32_t d0 = tmem + uint32_t(2 * NCOL * ((c / kTcRun) & 1));
        const uint32_t a0 = tmem + kABase + uint32_t(st * 4 * kTcK);
        const uint64_t bb0 = tc::desc(sbase + st * Sm::stage, kTcSbo);
        const uint64_t bs0 = tc::desc(sbase + st * Sm::stage + Sm::b_part, kTcSbo);
#pragma unroll
        for (int s = 0; s < kTcK / 8; ++s) {  // a k-step: 8 TMEM columns of A, two core matrices (256 B) of B
          const uint32_t on = (s > 0 || (c % kTcRun) != 0) ? 1u : 0u;
#pragma unroll
          for (int d = 0; d < 2; ++d) {
            const uint32_t dd = d0 + uint32_t(d * NCOL), ab = a0 + uint32_t(2 * d * kTcK + 8 * s), as = ab + kTcK;
            tc::mma_tf32_ts(dd, ab, bb0 + 16u * s, kIdesc, on);
            tc::mma_tf32_ts(dd, ab, bs0 + 16u * s, kIdesc, 1u);
            tc::mma_tf32_ts(dd, as, bb0 + 16u * s, kIdesc, 1u);
          }
        }
        tc::commit(sbase + Sm::empty + 8 * st);
        issued = c + 1;
        if (++st == kTcStages) {
          st = 0;
          ++use;
        }
      }
      if (bad) {  // bounded waits for what is still in flight, before shared memory and TMEM are given up
        *s_bad = 1;
        if (issued > 0)
          tc::wait(sbase + Sm::empty + 8 * ((issued - 1) % kTcStages), uint32_t((issued - 1) / kTcStages) & 1u, kTcWaitNs, nullptr);
        for (int r = max(0, loaded - 3); r < loaded; ++r)
          tc::wait(sbase + Sm::ring + 8 * (r % kTcRing), uint32_t(r / kTcRing) & 1u, kTcWaitNs, nullptr);
      }
    }
    __syncwarp();
    __syncthreads();
  } else {  // ---- operands and sums
    tc::regs_inc<112>();
    // A: a warp reaches the 32 TMEM lanes 32 (warp % 4) .., so row 32 (warp % 4) + lane; the four warps of
    // those lanes take four particles each
    const int quad = warp & 3, part = warp >> 2;
    const uint32_t tlane = uint32_t(32 * quad) << 16;
    const int64_t pair = int64_t(blockIdx.x) * kTcRows + 32 * quad + lane;
    const bool row_ok = pair < int64_t(ng) * H;
    const int ix = row_ok ? int(pair / H) : 0, iz = row_ok ? int(pair - int64_t(ix) * H) : 0;
    uint64_t ks[PT / 2], kc[PT / 2];  // compensated sums: value and compensation, two columns per register pair
#pragma unroll
    for (int j = 0; j < PT / 2; ++j) ks[j] = kc[j] = 0ull;
    const uint32_t nx = uint32_t(signed_mode(ix, ng)), nz = uint32_t(iz == ng / 2 ? -iz : iz);
    int st = kTcStages - 1, use = -1;  // chunk c's stage and the stage's use (c % kTcStages, c / kTcStages)
    for (int c = 0; c < nchunks + kTcStages; ++c) {
      if (++st == kTcStages) {
        st = 0;
        ++use;
      }
      if (c >= kTcStages) {  // chunk p done: its stage is free, and after the last chunk of a run its sums
        const int p = c - kTcStages;
        wait(Sm::empty + 8 * st, use - 1);
        if (!__all_sync(0xffffffffu, !bad)) break;
        // the commit orders chunk p's reads of this stage's TMEM columns (and its sums) before what follows this
        // fence: the stores of the next A operand below, and the loads of the sums
        tc::fence_after();
        if (p % kTcRun == kTcRun - 1 || p == nchunks - 1) {
          tc::twosum_acc<PT>(tmem + tlane + uint32_t(2 * NCOL * ((p / kTcRun) & 1) + PT * part), ks, kc);
        }
      }
      if (c >= nchunks) continue;
      const int run = c / kTcRun;
      if (c % kTcRun == 0) {
        wait(Sm::ring + 8 * (run % kTcRing), run / kTcRing);
        if (!__all_sync(0xffffffffu, !bad)) break;
      }
      const Rec* rc = reinterpret_cast<const Rec*>(sm + Sm::rec) + (run % kTcRing) * kTcRunLen + (c % kTcRun) * kTcK;
      // A: cos and sin of this row's phase for particles 4 part .. + 3, split, to TMEM (particles past the
      // slice: any phase, their weight on the B side is zero)
      {
        float ab[2][4], as[2][4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          float sn, cs;
          tc_sincos(nx * rc[4 * part + k].px + nz * rc[4 * part + k].pz, sn, cs);
          tc::split(cs, ab[0][k], as[0][k]);
          tc::split(sn, ab[1][k], as[1][k]);
        }
        const uint32_t a0 = tmem + tlane + kABase + uint32_t(st * 4 * kTcK + 4 * part);
#pragma unroll
        for (int d = 0; d < 2; ++d) {
          tc::store4(a0 + uint32_t(2 * d * kTcK), ab[d]);
          tc::store4(a0 + uint32_t((2 * d + 1) * kTcK), as[d]);
        }
      }
      // B: two particles of one n_y per item: w cos and w sin, split, to shared memory. The items fill
      // up to ten warps, another ten each chunk (the warps run up to kTcStages chunks apart).
      unsigned char* stg = sm + st * Sm::stage;
      const int left = int(min(int64_t(kTcK), k_end - k_beg - int64_t(c) * kTcK));
      for (int it = 32 * ((warp + 6 * c) % kTcBuilders) + lane; it < CY * (kTcK / 2); it += 32 * kTcBuilders) {
        const int j = it % CY, k = 2 * (it / CY);
        const uint32_t ny = uint32_t(col0 + j);
        float v[2][2] = {};
        if (col0 + j < H) {
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const float w = k + u < left ? rc[k + u].w : 0.0f;
            float sn, cs;
            tc_sincos(ny * rc[k + u].py, sn, cs);
            v[0][u] = w * cs;
            v[1][u] = w * sn;
          }
        }
#pragma unroll
        for (int f = 0; f < 2; ++f) {
          float2 big, small;
          tc::split(v[f][0], big.x, small.x);
          tc::split(v[f][1], big.y, small.y);
          const uint32_t off = tc::off(2 * j + f, k, kTcK);
          *reinterpret_cast<float2*>(stg + off) = big;
          *reinterpret_cast<float2*>(stg + Sm::b_part + off) = small;
        }
      }
      tc::wait_st();
      tc::fence_async_smem();
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::arrive(sbase + Sm::full + 8 * st);
    }
    if (bad) *s_bad = 1;
    __syncthreads();
    if (*s_bad && tid == 0) raise_err(PK_DERR_TIMEOUT);
    if (!*s_bad && row_ok && nchunks > 0) {
      const bool sine_row = part >= 2;  // this thread's columns are of D1
#pragma unroll
      for (int q = 0; q < PT; ++q) {
        const int col = (PT * part) % NCOL + q, j = col0 + col / 2;
        const bool sine_col = (col & 1) != 0;
        if (j >= H || (sine_col && j == 0)) continue;  // sin(0) = 0
        const float2 s2 = tc::unpack(ks[q / 2]), c2 = tc::unpack(kc[q / 2]);
        const double v = (q & 1) ? double(s2.y) + double(c2.y) : double(s2.x) + double(c2.x);
        double2* plus = acc_out + (int64_t(ix) * ng + j) * H + iz;
        double2* minus = acc_out + (int64_t(ix) * ng + (ng - j)) * H + iz;
        const bool has_plus = j < ng / 2, has_minus = j > 0;  // i_y = N/2 is n_y = -N/2
        if (sine_row == sine_col) {  // real parts: D0cos -+ D1sin
          if (has_plus) atomicAdd(&plus->x, sine_row ? -v : v);
          if (has_minus) atomicAdd(&minus->x, v);
        } else {  // imaginary parts: -(D1cos +- D0sin)
          if (has_plus) atomicAdd(&plus->y, -v);
          if (has_minus) atomicAdd(&minus->y, sine_row ? -v : v);
        }
      }
    }
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 0) {
    tc::fence_after();
    tc::tmem_dealloc(tmem, tc_tmem_cols(NCOL));
  }
}

// ---- host side --------------------------------------------------------------------------------------------

namespace {

constexpr int kPrepBlocks = 1024;

struct DsLayout {
  void* recs = nullptr;
  double* wpart = nullptr;
  double* wsum = nullptr;
  double2* sums = nullptr;
};

void carve_ds(const pk_config* c, int64_t n, Carver& cv, DsLayout* L) {
  const size_t rec = c->prec == PK_FP32 ? sizeof(DsT<float>::Rec) : sizeof(DsT<double>::Rec);
  L->recs = cv.take<char>(rec * size_t(std::max<int64_t>(n, 1)));
  L->wpart = cv.take<double>(kPrepBlocks);
  L->wsum = cv.take<double>(1);
  L->sums = cv.take<double2>(size_t(half_count(c->ng)));
}

struct CrossLayout {
  double* bin_sum = nullptr;
  double* bin_k = nullptr;
  unsigned long long* bin_cnt = nullptr;
  double* wsums = nullptr;
};

void carve_cross(const pk_config* c, Carver& cv, CrossLayout* L) {
  L->bin_sum = cv.take<double>(c->nbins);
  L->bin_k = cv.take<double>(c->nbins);
  L->bin_cnt = cv.take<unsigned long long>(c->nbins);
  L->wsums = cv.take<double>(3);
}

// Particle slices per column of mode tiles: enough blocks for whole waves of one block per SM.
int ds_slices(int64_t tiles, int64_t n, int K) {
  const int64_t sms = num_sms();
  const int64_t chunks = (n + K - 1) / K;
  int best = 1;
  double best_eff = 0.0;
  for (int s = 1; s <= 64 && s <= chunks; ++s) {
    const int64_t blocks = tiles * s;
    const int64_t waves = (blocks + sms - 1) / sms;
    // particles per slice rounded up to whole chunks: the longest slice sets the time
    const double eff = double(blocks) / double(waves * sms);
    if (eff > best_eff + 0.02) {
      best_eff = eff;
      best = s;
    }
    if (blocks >= 4 * sms) break;
  }
  return best;
}

// Slices of the tensor-core kernel: whole waves of one block per SM, each as long as its runs and the block's
// start and end (TMEM, first records, FP64 additions of its sums), taken as eight runs: with four or sixteen the times
// are the same within 1 % (5000 to 400 000 particles on N = 16 to 128).
int tc_slices(int64_t tiles, int64_t runs) {
  const int64_t sms = num_sms();
  int best = 1;
  int64_t best_cost = INT64_MAX;
  for (int s = 1; s <= 64 && s <= runs; ++s) {
    const int64_t waves = (tiles * s + sms - 1) / sms, cost = waves * ((runs + s - 1) / s + 8);
    if (cost < best_cost) {
      best_cost = cost;
      best = s;
    }
  }
  return best;
}

template <int NCOL>
cudaError_t launch_tc(dim3 grid, const DsT<float>::Rec* recs, int64_t n, int ng, int64_t slice_len, double2* sums,
                      cudaStream_t s) {
  k_ds_modes_tc<NCOL><<<grid, kTcThreads, TcSmem<NCOL>::total, s>>>(recs, n, ng, slice_len, sums);
  count_launch();
  return cudaGetLastError();
}

template <typename R>
pk_status run_direct(const pk_config* c, const void* pos, int fmt, const float* w, int64_t n, void* delta_out, DsLayout& L,
                     cudaStream_t s) {
  using Rec = typename DsT<R>::Rec;
  const int ng = c->ng;
  cudaError_t e;
  const int prep_blocks = int(std::min<int64_t>(kPrepBlocks, std::max<int64_t>(1, (n + 255) / 256)));
  k_ds_prep<R><<<prep_blocks, 256, 0, s>>>(pos, fmt, w, n, ng, c->box, static_cast<Rec*>(L.recs), L.wpart); count_launch();
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "direct prep");
  k_ds_wsum<<<1, 256, 0, s>>>(L.wpart, prep_blocks, L.wsum); count_launch();
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "direct wsum");
  const int64_t hc = half_count(ng);
  if ((e = cudaMemsetAsync(L.sums, 0, sizeof(double2) * size_t(hc), s)) != cudaSuccess) return cuda_fail(e, "memset");
  if constexpr (std::is_same_v<R, float>) {  // the tensor-core kernel
    const int64_t row_tiles = tc_row_tiles(ng);
    const int col_tiles = tc_col_tiles(ng);
    const int64_t runs = (n + kTcRunLen - 1) / kTcRunLen;
    const int slices = tc_slices(row_tiles * col_tiles, runs);
    const int64_t slice_len = ((runs + slices - 1) / slices) * kTcRunLen;
    const dim3 grid{unsigned(row_tiles), unsigned(col_tiles), unsigned(slices)};
    const Rec* recs = static_cast<const Rec*>(L.recs);
    switch (tc_cols(ng)) {
      case 16: e = launch_tc<16>(grid, recs, n, ng, slice_len, L.sums, s); break;
      case 32: e = launch_tc<32>(grid, recs, n, ng, slice_len, L.sums, s); break;
      case 48: e = launch_tc<48>(grid, recs, n, ng, slice_len, L.sums, s); break;
      case 64: e = launch_tc<64>(grid, recs, n, ng, slice_len, L.sums, s); break;
      default: e = launch_tc<80>(grid, recs, n, ng, slice_len, L.sums, s); break;
    }
    if (e != cudaSuccess) return cuda_fail(e, "direct modes");
    const int fblocks = int(std::min<int64_t>(int64_t(num_sms()) * 8, (hc + 255) / 256));
    k_ds_finish<float2><<<fblocks, 256, 0, s>>>(L.sums, L.wsum, hc, static_cast<float2*>(delta_out));
    count_launch();
    e = cudaGetLastError();
    return e == cudaSuccess ? PK_OK : cuda_fail(e, "direct finish");
  } else {  // the CUDA-core kernel
    const int64_t row_tiles = ds_row_tiles(ng);
    const int col_tiles = (ng + kDsCols - 1) / kDsCols;
    const int slices = ds_slices(row_tiles * col_tiles, n, kDsK);
    const int64_t chunks = (n + kDsK - 1) / kDsK;
    const int64_t slice_len = ((chunks + slices - 1) / slices) * kDsK;
    const size_t smem = sizeof(double2) * size_t(kDsK) * (kDsRows + kDsCols + kDsTx + kDsTz);
    if ((e = ensure_dynamic_smem(reinterpret_cast<const void*>(k_ds_modes), smem)) != cudaSuccess)
      return cuda_fail(e, "direct smem");
    if (row_tiles > 2147483647) return fail(PK_EINVAL, "too many rows");
    k_ds_modes<<<dim3(unsigned(row_tiles), col_tiles, slices), kDsThreads, smem, s>>>(static_cast<const Rec*>(L.recs), n, ng,
                                                                                       slice_len, L.sums); count_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "direct modes");
    const int fblocks = int(std::min<int64_t>(int64_t(num_sms()) * 8, (hc + 255) / 256));
    k_ds_finish<double2><<<fblocks, 256, 0, s>>>(L.sums, L.wsum, hc, static_cast<double2*>(delta_out));
    count_launch();
    e = cudaGetLastError();
    return e == cudaSuccess ? PK_OK : cuda_fail(e, "direct finish");
  }
}

// Only the bins that can hold a mode (half-integer |n| up to sqrt(3) N/2) reach k_cross_rows: at most 1774, whose private
// copies for two warps fit 96 KB (two blocks per SM), and edges that fit its 32-bit test (the one bin of a wider
// w2 ends at the largest |n|). Rows share a warp until a lane has at least eight slots (a lane's FP64 additions to
// the bins and the row's scan then weigh less than its modes), but not where fewer than twelve warps per SM would
// be left: N = 100 takes 24.6 us per call with four rows per warp and 28.9 with eight, N = 16 took 37 with all
// its rows in one block, now 24. Blocks have 8 warps, else 4 or 2, as the copies' room and the rows allow.
template <typename V>
cudaError_t launch_cross(const pk_config* c, const V* a, const V* b, double vol, const CrossLayout& L, cudaStream_t s) {
  const int ng = c->ng, lz = ng / 2 + 1;
  const int top = int(std::sqrt(3.0 * ng * ng));  // the largest 2 |n|, rounded down (3 N^2 is no square)
  if (c->bin_lo2 > top) return cudaSuccess;       // no mode in the bins: the sums stay cleared
  const int nbins = std::min(c->nbins, (top - c->bin_lo2) / c->bin_w2 + 1);
  const int w2 = nbins == 1 ? std::min(c->bin_w2, top + 1 - c->bin_lo2) : c->bin_w2;
  const size_t bin_bytes = size_t(nbins) * (sizeof(CrossBin) + sizeof(unsigned));
  const int64_t rows = int64_t(ng) * ng, sms = num_sms();
  int wpb = 0, RW = 1;
  while (RW < 32 && (lz + 32 / RW - 1) / (32 / RW) < 8 && rows / (2 * RW) >= 12 * sms) RW *= 2;
  for (; RW >= 1 && !wpb; RW = wpb ? RW : RW / 2)
    for (int w = 8; w >= 2 && !wpb; w /= 2)
      if (size_t(w) * RW * bin_bytes <= 96 * 1024) wpb = w;
  const int64_t items = (rows + RW - 1) / RW;
  while (wpb > 2 && items < sms * wpb) wpb /= 2;
  const size_t smem = size_t(wpb) * RW * bin_bytes;
  cudaError_t e;
  if ((e = ensure_dynamic_smem(reinterpret_cast<const void*>(k_cross_rows<V>), smem)) != cudaSuccess) return e;
  int per_sm = 1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_cross_rows<V>, 32 * wpb, smem) != cudaSuccess || per_sm < 1)
    per_sm = 1;
  const int blocks = int(std::max<int64_t>(1, std::min<int64_t>((items + wpb - 1) / wpb, sms * per_sm)));
  k_cross_rows<V><<<blocks, 32 * wpb, smem, s>>>(a, b, ng, vol, c->bin_lo2, w2, nbins, RW, L.bin_sum, L.bin_k, L.bin_cnt);
  count_launch();
  return cudaGetLastError();
}

}  // namespace

pk_status direct_ws(const pk_config* c, int64_t n, bool cross, size_t* out) {
  Carver cv(nullptr);
  if (cross) {
    CrossLayout L;
    carve_cross(c, cv, &L);
  } else {
    DsLayout L;
    carve_ds(c, n, cv, &L);
  }
  *out = cv.size();
  return PK_OK;
}

}  // namespace pk

using namespace pk;

extern "C" {

pk_status pk_direct_modes(const pk_config* cfg, const void* pos_dev, int32_t pos_format, const float* w_dev, int64_t n,
                          void* delta_k_dev, void* ws, size_t ws_bytes, void* stream) {
  clear_err();
  pk_status st = validate(cfg);
  if (st != PK_OK) return st;
  if (pos_format != PK_POS_F64_XYZ && pos_format != PK_POS_CELL_F32OFF) return fail(PK_EINVAL, "bad pos_format");
  if (n < 1 || !pos_dev) return fail(PK_EINVAL, "need at least one particle");
  if (!delta_k_dev) return fail(PK_EINVAL, "delta_k_dev is NULL");
  const size_t need = pk_workspace_size(cfg, n, PK_WS_DIRECT);
  if (!ws || ws_bytes < need) return fail(PK_ESIZE, "workspace %zu < %zu bytes", ws_bytes, need);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  Carver cv(ws);
  DsLayout L;
  carve_ds(cfg, n, cv, &L);
  return cfg->prec == PK_FP32 ? run_direct<float>(cfg, pos_dev, pos_format, w_dev, n, delta_k_dev, L, s)
                              : run_direct<double>(cfg, pos_dev, pos_format, w_dev, n, delta_k_dev, L, s);
}

pk_status pk_cross_power(const pk_config* cfg, const void* delta_a_dev, const void* delta_b_dev, double* pk_dev,
                         double* kmean_dev, int64_t* nmodes_dev, void* ws, size_t ws_bytes, void* stream) {
  clear_err();
  pk_status st = validate(cfg);
  if (st != PK_OK) return st;
  if (!delta_a_dev || !delta_b_dev || !pk_dev || !nmodes_dev) return fail(PK_EINVAL, "bad pointers");
  const size_t need = pk_workspace_size(cfg, 0, PK_WS_CROSS);
  if (!ws || ws_bytes < need) return fail(PK_ESIZE, "workspace %zu < %zu bytes", ws_bytes, need);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  Carver cv(ws);
  CrossLayout L;
  carve_cross(cfg, cv, &L);
  cudaError_t e;
  // the accumulators are carved one after another: one clear for all
  if ((e = cudaMemsetAsync(L.bin_sum, 0, size_t(reinterpret_cast<char*>(L.wsums + 3) - reinterpret_cast<char*>(L.bin_sum)), s)) !=
      cudaSuccess)
    return cuda_fail(e, "memset");
  const double vol = cfg->box * cfg->box * cfg->box;
  e = cfg->prec == PK_FP32 ? launch_cross(cfg, static_cast<const float2*>(delta_a_dev), static_cast<const float2*>(delta_b_dev), vol, L, s)
                           : launch_cross(cfg, static_cast<const double2*>(delta_a_dev), static_cast<const double2*>(delta_b_dev), vol, L, s);
  if (e != cudaSuccess) return cuda_fail(e, "cross bins");
  EstimateArgs a{};
  a.ng = cfg->ng;
  a.nbins = cfg->nbins;
  a.bin_lo2 = cfg->bin_lo2;
  a.bin_w2 = cfg->bin_w2;
  a.box = cfg->box;
  a.wsums = L.wsums;  // zeros: no shot noise is subtracted
  a.bin_sum = L.bin_sum;
  a.bin_k = L.bin_k;
  a.bin_cnt = L.bin_cnt;
  if ((e = launch_finalize(a, 0, pk_dev, kmean_dev, nmodes_dev, s)) != cudaSuccess) return cuda_fail(e, "finalize");
  return PK_OK;
}

}  // extern "C"
