// a8 adjoint of the power spectrum with respect to particle positions (the paper has no adjoint; this
// is the chain rule through a3..a6).
//
// With P_b = (V/M_b) sum_{n in b} |delta(n)|^2, delta(n) = [G_1(n) + phi(n) G_2(n)] c(n),
// c(n) = a / (sum(w) W(n)) (a = 1/2 interlaced, 1 otherwise), phi(n) = e^{+i pi (n_x+n_y+n_z)/N}:
//   A(n)       = 2 kappa(n) c(n) conj(delta(n)),   kappa(n) = (dL/dP_b) V / M_b for n in bin b
//   dL/drho_1[j] = Re sum_n A(n) e^{-2 pi i n.j/N},   dL/drho_2[j] = Re sum_n A(n) phi(n) e^{-2 pi i n.j/N}.
// Re sum_n B(n) e^{-i theta_n} = sum_n X(n) e^{+i theta_n} with X(n) = [conj B(n) + B(-n)] / 2 Hermitian,
// i.e. one inverse real FFT per grid. B(-n) uses delta(-n) = [conj G_1(n) + phi(-n) conj G_2(n)] c(n),
// with the Nyquist-slot phase rule of the forward estimate. Finally
//   dL/dx_{i,a} = w_i (N/L) sum_g sum_{j in stencil} dL/drho_g[j] dW(j_a - u_a)/du_a prod_{b != a} W(j_b - u_b).
#include "host.cuh"
#include "position.cuh"

namespace pk {

template <typename R>
struct CC {
  R x, y;
};
template <typename R>
__device__ __forceinline__ CC<R> mul(CC<R> a, CC<R> b) {
  return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <typename R>
__device__ __forceinline__ CC<R> cj(CC<R> a) {
  return {a.x, -a.y};
}

// FP64 tables per slot (n its signed index): 1/W_1d(n), cos and sin of pi n/N.
__global__ void k_adjoint_tables(double* __restrict__ tab, int ng, int order) {
  for (int i = threadIdx.x + blockIdx.x * blockDim.x; i < ng; i += blockDim.x * gridDim.x) {
    const int n = signed_mode(i, ng);
    const double x = 3.14159265358979323846 * double(n) / double(ng);
    const double s = n == 0 ? 1.0 : sin(x) / x;
    double w = 1.0;
    for (int k = 0; k < order; ++k) w *= s;
    tab[i] = 1.0 / w;
    tab[ng + i] = cos(x);
    tab[2 * ng + i] = sin(x);
  }
}

// Mode counts of the bins on the full N^3 grid (|n|^2 does not depend on signs or on the order of n_x and n_y): the
// rows 0 <= i_y <= i_x <= N/2 with their multiplicity, an eighth of the stored modes. Integer counts in
// shared memory; a warp takes rows, its lanes the slots. (The gradient took the whole forward estimate for
// its counts before: 17 us at N = 128, 4 so.)
__global__ void __launch_bounds__(256) k_mode_counts(int ng, int lo2, int w2, int nbins, unsigned long long* __restrict__ counts) {
  extern __shared__ unsigned s_count[];
  for (int b = threadIdx.x; b < nbins; b += blockDim.x) s_count[b] = 0u;
  __syncthreads();
  const int half = ng / 2, lane = threadIdx.x & 31;
  const int nwarps = int(gridDim.x * blockDim.x) >> 5;
  for (int row = int(blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < (half + 1) * (half + 1); row += nwarps) {
    const int ix = row / (half + 1), iy = row - ix * (half + 1);
    if (iy > ix) continue;
    const int mult = (ix == 0 || ix == half ? 1 : 2) * (iy == 0 || iy == half ? 1 : 2) * (iy < ix ? 2 : 1);
    for (int iz = lane; iz <= half; iz += 32) {
      const int b = bin_of(4 * ((long long)ix * ix + (long long)iy * iy + (long long)iz * iz), lo2, w2, nbins);
      if (b >= 0) atomicAdd(&s_count[b], unsigned(iz == 0 || iz == half ? mult : 2 * mult));
    }
  }
  __syncthreads();
  for (int b = threadIdx.x; b < nbins; b += blockDim.x)
    if (s_count[b]) atomicAdd(&counts[b], (unsigned long long)s_count[b]);
}

// In place: (G_1, G_2) at every stored slot -> (X_1, X_2). A warp takes rows (i_x, i_y), lanes take slots; a mode's window
// and phase are products of the FP64 tables' entries, those of the row formed once, and are rounded to the grids'
// precision once. Off the Nyquist slots phi(-n) is the conjugate of phi(n), so A(-n) = conj A(n), and
// X_1 = 2 kappa c delta(n), X_2 = X_1 conj phi(n).
// Bound by the reads and writes of the grids and, in the FP32 mode, by the FP64 pipe: two products of phases, the window's
// and three conversions per mode: 32 us at N = 128 (417 with the window, sine and cosine of every mode in FP64). With
// FP32 factors, rounded before they are multiplied, the whole gradient takes 429 us instead of 434.
template <typename R>
__global__ void __launch_bounds__(256) k_adjoint_modes(CC<R>* __restrict__ G1, CC<R>* __restrict__ G2, int ng, int interlace,
                                                       int lo2, int w2, int nbins, double box, const double* __restrict__ tab,
                                                       const double* __restrict__ wsums, const double* __restrict__ dl_dpk,
                                                       const unsigned long long* __restrict__ counts) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int half = ng / 2, lz = half + 1;
  double* iwz = reinterpret_cast<double*>(smem_raw);  // 1/W, cos, sin of the slots i_z
  R* kap2 = reinterpret_cast<R*>(iwz + 3 * lz);       // 2 kappa per bin
  __shared__ double s_norm;  // one FP64 division per block (by every warp: 35 us instead of 32 at N = 128)
  {
    if (threadIdx.x == blockDim.x - 1) s_norm = (interlace ? 0.5 : 1.0) / wsums[0];
    const double vol = box * box * box;
    for (int b = threadIdx.x; b < nbins; b += blockDim.x)
      kap2[b] = counts[b] > 0 ? R(2.0 * dl_dpk[b] * vol / double(counts[b])) : R(0);
    for (int i = threadIdx.x; i < 3 * lz; i += blockDim.x) iwz[i] = tab[(i / lz) * ng + i % lz];
  }
  __syncthreads();
  const bool small = int64_t(lo2) + int64_t(nbins + 1) * w2 <= 46340;  // bin edges whose squares fit 32 bits
  const float inv_w2 = 1.0f / float(w2);
  const long long top = (long long)lo2 + (long long)nbins * w2;
  const double norm = s_norm;
  const int lane = threadIdx.x & 31;
  const int nwarps = int(gridDim.x * blockDim.x) >> 5;
  for (int row = int(blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < ng * ng; row += nwarps) {
    const int ix = row / ng, iy = row - ix * ng;
    const int nx = signed_mode(ix, ng), ny = signed_mode(iy, ng), nxy2 = nx * nx + ny * ny;
    const bool nyq_row = ix == half || iy == half;
    double cxy = 0.0, phx = 0.0, phy = 0.0, phx_p = 0.0, phy_p = 0.0;
    if (4 * (long long)nxy2 < top * top) {  // else the row lies beyond the last bin
      const double cx = tab[ng + ix], sx = tab[2 * ng + ix], cy = tab[ng + iy], sy = tab[2 * ng + iy];
      cxy = tab[ix] * tab[iy] * norm;
      phx = cx * cy - sx * sy;
      phy = sx * cy + cx * sy;
      phx_p = phx;  // phase of the partner's n_x, n_y: the conjugate except on the Nyquist slots, which keep n = -N/2
      phy_p = -phy;
      if (nyq_row) {
        const double sxp = ix == half ? sx : -sx, syp = iy == half ? sy : -sy;
        phx_p = cx * cy - sxp * syp;
        phy_p = sxp * cy + cx * syp;
      }
    }
    for (int iz = lane; iz < lz; iz += 32) {
      const int64_t i = int64_t(row) * lz + iz;
      const int n2 = nxy2 + iz * iz;
      const int b = small ? bin_of32(4 * n2, 2.0f * sqrtf(float(n2)), lo2, w2, inv_w2, nbins)
                          : bin_of(4 * (long long)n2, lo2, w2, nbins);
      CC<R> x1 = {R(0), R(0)}, x2 = {R(0), R(0)};
      if (b >= 0) {
        const R c = R(cxy * iwz[iz]), kap2c = kap2[b] * c;
        const CC<R> g1 = G1[i];
        if (!interlace) {
          x1 = {kap2c * (g1.x * c), kap2c * (g1.y * c)};
        } else {
          const CC<R> g2 = G2[i];
          const double cz = iwz[lz + iz], sz = iwz[2 * lz + iz];  // slot N/2: n_z = -N/2
          const CC<R> phi = {R(phx * cz - phy * sz), R(phx * sz + phy * cz)};
          const CC<R> t = mul(phi, g2);
          const CC<R> d = {(g1.x + t.x) * c, (g1.y + t.y) * c};
          if (!nyq_row && iz != half) {
            x1 = {kap2c * d.x, kap2c * d.y};
            x2 = mul(x1, cj(phi));
          } else {
            const double szp = iz == half ? sz : -sz;
            const CC<R> phip = {R(phx_p * cz - phy_p * szp), R(phx_p * szp + phy_p * cz)};
            const CC<R> tp = mul(phip, cj(g2));
            const CC<R> dm = {(g1.x + tp.x) * c, (-g1.y + tp.y) * c};
            const CC<R> A = {kap2c * d.x, -kap2c * d.y};     // 2 kappa c conj(delta(n))
            const CC<R> Am = {kap2c * dm.x, -kap2c * dm.y};  // 2 kappa c conj(delta(-n))
            // X_1 = [conj A(n) + A(-n)] / 2, X_2 the same of B = A phi
            x1 = {R(0.5) * (A.x + Am.x), R(0.5) * (-A.y + Am.y)};
            const CC<R> B = mul(A, phi), Bm = mul(Am, phip);
            x2 = {R(0.5) * (B.x + Bm.x), R(0.5) * (-B.y + Bm.y)};
          }
        }
      }
      G1[i] = x1;
      if (interlace) G2[i] = x2;
    }
  }
}

// Sum over one grid's stencil. Along z the row is contracted with the weights and with their derivatives, and the
// two row sums with the x and y weights: two multiply-adds per node and five per row instead of some
// nine operations per node.
template <int P, typename R>
__device__ __forceinline__ void gather_grid(const R* __restrict__ g, const int* c, const R* f, int ng, R* grad) {
  R w[3][P], dw[3][P];
  int st[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) st[a] = bspline_deriv<P>(f[a], w[a], dw[a]);
  const int ldz = ng + 2, z0 = c[2] + st[2];
  const bool inside = z0 >= 0 && z0 + P <= ng;  // no node of a row wraps in z
  int gz[P];
#pragma unroll
  for (int k = 0; k < P; ++k) gz[k] = inside ? z0 + k : wrap(z0 + k, ng);
#pragma unroll
  for (int i = 0; i < P; ++i) {
    const int gx = wrap(c[0] + st[0] + i, ng);
    R u0 = R(0), u1 = R(0), u2 = R(0);
#pragma unroll
    for (int j = 0; j < P; ++j) {
      const R* row = g + (int64_t(gx) * ng + wrap(c[1] + st[1] + j, ng)) * ldz;
      R v[P];
      if (inside) {
#pragma unroll
        for (int k = 0; k < P; ++k) v[k] = __ldg(row + z0 + k);
      } else {
#pragma unroll
        for (int k = 0; k < P; ++k) v[k] = __ldg(row + gz[k]);
      }
      R s = R(0), ds = R(0);
#pragma unroll
      for (int k = 0; k < P; ++k) {
        s += v[k] * w[2][k];
        ds += v[k] * dw[2][k];
      }
      u0 += w[1][j] * s;
      u1 += dw[1][j] * s;
      u2 += w[1][j] * ds;
    }
    grad[0] += dw[0][i] * u0;
    grad[1] += w[0][i] * u1;
    grad[2] += w[0][i] * u2;
  }
}

template <int P, typename R>
__global__ void __launch_bounds__(256) k_gather(const void* __restrict__ pos, int fmt, const float* __restrict__ wts, int64_t n,
                                                int ng, double box, int interlace, int f32pos, const R* __restrict__ g1,
                                                const R* __restrict__ g2, R* __restrict__ out) {
  const double scale = double(ng) / box;
  for (int64_t i = gtid(); i < n; i += gstride()) {
    int c[3];
    R f[3];
    bool ok = true;
    if (fmt == PK_POS_F64_XYZ && !f32pos) {
      const double* p = static_cast<const double*>(pos) + 3 * i;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        double x = p[a];
        if (!isfinite(x)) { ok = false; x = 0.0; }
        if (!(x >= 0.0 && x < box)) {  // another periodic image (fmod is the identity on [0, L))
          x = fmod(x, box);
          if (x < 0.0) x += box;
        }
        const double u = x * scale;
        const double fl = floor(u);
        int ci = int(fl);
        if (ci >= ng) ci -= ng;
        c[a] = ci;
        f[a] = R(u - fl);
      }
    } else {
      pk_cellpos r;
      if (fmt == PK_POS_F64_XYZ) {  // the forward's rounding (PK_FP32, PK_FIXED64)
        bool bad;
        r = prepare_one(static_cast<const double*>(pos) + 3 * i, ng, box, scale, &bad);
        ok = !bad;
      } else {
        r = static_cast<const pk_cellpos*>(pos)[i];
      }
      c[0] = cell_x(r.cell); c[1] = cell_y(r.cell); c[2] = cell_z(r.cell);
      f[0] = R(r.fx); f[1] = R(r.fy); f[2] = R(r.fz);
      ok = ok && c[0] < ng && c[1] < ng && c[2] < ng;
    }
    R grad[3] = {R(0), R(0), R(0)};
    if (ok) {
      gather_grid<P, R>(g1, c, f, ng, grad);
      if (interlace) {
        int c2[3];
        R f2[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) c2[a] = c[a] + half_shift(f[a], &f2[a]);
        gather_grid<P, R>(g2, c2, f2, ng, grad);
      }
    }
    const R s = R(scale) * (wts ? R(wts[i]) : R(1));
    out[3 * i] = grad[0] * s;
    out[3 * i + 1] = grad[1] * s;
    out[3 * i + 2] = grad[2] * s;
  }
}

template <typename R>
static cudaError_t launch_gather(int order, const void* pos, int fmt, const float* w, int64_t n, int ng, double box, int interlace,
                                 int f32pos, const R* g1, const R* g2, R* out, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int blocks = int(std::min<int64_t>((n + 255) / 256, int64_t(num_sms()) * 16));
  switch (order) {
    case 2: k_gather<2, R><<<blocks, 256, 0, s>>>(pos, fmt, w, n, ng, box, interlace, f32pos, g1, g2, out); count_launch(); break;
    case 3: k_gather<3, R><<<blocks, 256, 0, s>>>(pos, fmt, w, n, ng, box, interlace, f32pos, g1, g2, out); count_launch(); break;
    case 4: k_gather<4, R><<<blocks, 256, 0, s>>>(pos, fmt, w, n, ng, box, interlace, f32pos, g1, g2, out); count_launch(); break;
    case 5: k_gather<5, R><<<blocks, 256, 0, s>>>(pos, fmt, w, n, ng, box, interlace, f32pos, g1, g2, out); count_launch(); break;
    default: k_gather<6, R><<<blocks, 256, 0, s>>>(pos, fmt, w, n, ng, box, interlace, f32pos, g1, g2, out); count_launch(); break;
  }
  return cudaGetLastError();
}

struct BackLayout {
  ForwardStage f;
  PlanEntry inv;
  void* inv_work = nullptr;
  double* tab = nullptr;  // k_adjoint_tables
};

static pk_status carve_back(const pk_config* c, int64_t n, Carver& cv, BackLayout* L) {
  pk_status st = carve_forward(c, n, cv, &L->f);
  if (st != PK_OK) return st;
  const bool dbl = c->prec != PK_FP32;
  if ((st = get_plan(c->ng, dbl ? 3 : 2, c->interlace ? 2 : 1, &L->inv)) != PK_OK) return st;
  L->inv_work = cv.take<char>(std::max<size_t>(L->inv.work, 256));
  L->tab = cv.take<double>(size_t(3) * c->ng);
  return PK_OK;
}

pk_status backward_ws(const pk_config* c, int64_t n, size_t* out) {
  Carver cv(nullptr);
  BackLayout L;
  pk_status st = carve_back(c, n, cv, &L);
  if (st != PK_OK) return st;
  *out = cv.size();
  return PK_OK;
}

}  // namespace pk

using namespace pk;

extern "C" pk_status pk_power_backward(const pk_config* cfg, const void* pos_dev, int32_t pos_format, const float* w_dev,
                                       int64_t n, const double* dl_dpk_dev, void* dl_dx_dev, void* ws, size_t ws_bytes,
                                       void* stream) {
  clear_err();
  pk_status st = validate(cfg);
  if (st != PK_OK) return st;
  if (cfg->order < 2) return fail(PK_EINVAL, "the adjoint needs order 2..6 (NGP has no derivative)");
  if (pos_format != PK_POS_F64_XYZ && pos_format != PK_POS_CELL_F32OFF) return fail(PK_EINVAL, "bad pos_format");
  if (n < 1 || !pos_dev || !dl_dpk_dev || !dl_dx_dev) return fail(PK_EINVAL, "bad pointers");
  size_t need = 0;
  if ((st = backward_ws(cfg, n, &need)) != PK_OK) return st;
  if (!ws || ws_bytes < need) return fail(PK_ESIZE, "workspace %zu < %zu bytes", ws_bytes, need);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  Carver cv(ws);
  BackLayout L;
  if ((st = carve_back(cfg, n, cv, &L)) != PK_OK) return st;
  GridStage& g = L.f.g;
  // forward grids and their transforms (recomputed), then the exact mode counts of the bins
  if ((st = run_forward_grids(cfg, pos_dev, pos_format, w_dev, n, L.f, s)) != PK_OK) return st;
  if ((st = exec_plan(g.plan, g.kind, g.grids, g.fft_work, s)) != PK_OK) return st;
  const bool dbl = cfg->prec != PK_FP32;
  cudaError_t e;
  if ((e = cudaMemsetAsync(g.bin_cnt, 0, sizeof(unsigned long long) * cfg->nbins, s)) != cudaSuccess) return cuda_fail(e, "memset");
  const int64_t per = padded_count(cfg->ng);
  const size_t gbytes = size_t(per) * (dbl ? 8 : 4);
  void* G1 = g.grids;
  void* G2 = cfg->interlace ? static_cast<char*>(g.grids) + gbytes : nullptr;
  const int ng = cfg->ng, half = ng / 2;
  const int cblocks = std::min(num_sms() * 4, ((half + 1) * (half + 1) + 7) / 8);
  k_mode_counts<<<cblocks, 256, sizeof(unsigned) * size_t(cfg->nbins), s>>>(ng, cfg->bin_lo2, cfg->bin_w2, cfg->nbins, g.bin_cnt);
  count_launch();
  k_adjoint_tables<<<(ng + 127) / 128, 128, 0, s>>>(L.tab, ng, cfg->order); count_launch();
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "mode counts");
  const int blocks = std::min(num_sms() * 8, (ng * ng + 7) / 8);
  const size_t smem = size_t(cfg->nbins) * (dbl ? 8 : 4) + 3 * size_t(half + 1) * sizeof(double);
  if (dbl)
    k_adjoint_modes<double><<<blocks, 256, smem, s>>>(static_cast<CC<double>*>(G1), static_cast<CC<double>*>(G2), ng,
                                                      cfg->interlace, cfg->bin_lo2, cfg->bin_w2, cfg->nbins, cfg->box, L.tab,
                                                      g.wsums, dl_dpk_dev, g.bin_cnt);
  else
    k_adjoint_modes<float><<<blocks, 256, smem, s>>>(static_cast<CC<float>*>(G1), static_cast<CC<float>*>(G2), ng,
                                                     cfg->interlace, cfg->bin_lo2, cfg->bin_w2, cfg->nbins, cfg->box, L.tab,
                                                     g.wsums, dl_dpk_dev, g.bin_cnt);
  count_launch();
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "adjoint modes");
  if ((st = exec_plan(L.inv, dbl ? 3 : 2, g.grids, L.inv_work, s)) != PK_OK) return st;
  if (dbl)
    e = launch_gather<double>(cfg->order, pos_dev, pos_format, w_dev, n, cfg->ng, cfg->box, cfg->interlace,
                              cfg->prec != PK_FP64, static_cast<const double*>(G1), static_cast<const double*>(G2), static_cast<double*>(dl_dx_dev), s);
  else
    e = launch_gather<float>(cfg->order, pos_dev, pos_format, w_dev, n, cfg->ng, cfg->box, cfg->interlace, 1,
                             static_cast<const float*>(G1), static_cast<const float*>(G2), static_cast<float*>(dl_dx_dev), s);
  return e == cudaSuccess ? PK_OK : cuda_fail(e, "gather");
}
