// p-adaptation (Sec. 3.1) on the device: the spectral decay smoothness
// indicator, the degree decision, the neighbour jump limit, and the
// reordering of elements into (p, element id) buckets with prolongation /
// projection of their state.  This replaces the paper's ParMETIS
// repartition and all-gather redistribution (Sec. 3.2) on one GPU.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "fr_launch.h"

namespace frgb {

// ---------------------------------------------------------------------------
// indicator: eta = sum w|J| (s - s_{p-1})^2 / sum w|J| s^2 with s_{p-1} the
// Legendre truncation that drops every mode with an index equal to p.  One
// thread per element, fixed summation order (deterministic).
// ---------------------------------------------------------------------------
template <typename T, int ND, int P>
__global__ void k_indicator(const T* __restrict__ q, int var, const int32_t* __restrict__ slot_elem,
                            const BasisTab<double>* __restrict__ basis, GeoView<double> geo,
                            int64_t state_base, int count, int slot_begin, double* __restrict__ eta) {
  constexpr int NV = ND + 2;
  constexpr int NSP = ND == 2 ? P * P : P * P * P;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const BasisTab<double>& B = basis[P];
  const int e = slot_elem[slot_begin + i];
  const T* s = q + state_base + ((int64_t)i * NV + var) * NSP;
  double c[NSP], t[NSP];
  for (int k = 0; k < NSP; ++k) c[k] = (double)s[k];
  // modal coefficients, one direction at a time (xi, eta, zeta)
  for (int d = 0; d < ND; ++d) {
    const int stride = d == 0 ? 1 : (d == 1 ? P : P * P);
    for (int k = 0; k < NSP; ++k) {
      const int id = (k / stride) % P, base = k - id * stride;
      double acc = 0.0;
      for (int m = 0; m < P; ++m) acc += B.modal[id][m] * c[base + m * stride];
      t[k] = acc;
    }
    for (int k = 0; k < NSP; ++k) c[k] = t[k];
  }
  // keep only the modes with some index equal to p (they are s - s_{p-1})
  for (int k = 0; k < NSP; ++k) {
    const int i0 = k % P, i1 = (k / P) % P, i2 = ND == 3 ? k / (P * P) : 0;
    const bool top = i0 == P - 1 || i1 == P - 1 || (ND == 3 && i2 == P - 1);
    if (!top) c[k] = 0.0;
  }
  for (int d = 0; d < ND; ++d) {
    const int stride = d == 0 ? 1 : (d == 1 ? P : P * P);
    for (int k = 0; k < NSP; ++k) {
      const int id = (k / stride) % P, base = k - id * stride;
      double acc = 0.0;
      for (int m = 0; m < P; ++m) acc += B.nodal[id][m] * c[base + m * stride];
      t[k] = acc;
    }
    for (int k = 0; k < NSP; ++k) c[k] = t[k];
  }
  double num = 0.0, den = 0.0;
  for (int k = 0; k < NSP; ++k) {
    const int i0 = k % P, i1 = (k / P) % P, i2 = ND == 3 ? k / (P * P) : 0;
    double w = B.w[i0] * B.w[i1];
    if (ND == 3) w *= B.w[i2];
    w *= geo.vol[(int64_t)e * geo.ves + (int64_t)(ND * ND) * geo.vks + (int64_t)k * geo.vps];
    const double sv = (double)s[k];
    num += w * c[k] * c[k];
    den += w * sv * sv;
  }
  eta[e] = den > 0.0 ? num / den : 0.0;
}

__global__ void k_max_partial(const double* __restrict__ x, int n, double* __restrict__ part) {
  __shared__ double sm[256];
  double m = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) m = fmax(m, x[i]);
  sm[threadIdx.x] = m;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sm[threadIdx.x] = fmax(sm[threadIdx.x], sm[threadIdx.x + o]);
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sm[0];
}

__global__ void k_max_final(const double* __restrict__ part, int nb, double* __restrict__ out) {   // one warp
  double m = 0.0;
  for (int b = threadIdx.x; b < nb; b += 32) m = fmax(m, part[b]);
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (threadIdx.x == 0) out[0] = m;
}

template <typename T, int ND>
static void launch_indicator(fr_ctx* c, const T* q, int var, double* eta, cudaStream_t s) {
  for (const auto& b : c->buckets) {
    GeoView<double> g{};
    const int P = b.p + 1, NKV = geo_nk_vol(c->nd), NKF = geo_nk_face(c->nd);
    int NSP = 1;
    for (int d = 0; d < ND; ++d) NSP *= P;
    if (c->affine) {
      g.vol = c->d_gaff64; g.ves = NKF; g.vks = 1; g.vps = 0;
    } else {
      g.vol = c->d_gvol64[b.p]; g.ves = (int64_t)NKV * NSP; g.vks = NSP; g.vps = 1;
    }
    const unsigned grid = (unsigned)((b.count + 127) / 128);
    const double nb = (double)b.count * NSP * sizeof(T);
#define IND_CASE(PP) \
  case PP: FR_LAUNCH_B(c, "indicator", s, nb, k_indicator<T, ND, PP><<<grid, 128, 0, s>>>(q, var, c->lt.slot_elem, c->d_basis64, g, b.state_base, b.count, b.slot_begin, eta)); break;
    switch (P) {
      IND_CASE(2)
      IND_CASE(3)
      IND_CASE(4)
      IND_CASE(5)
      IND_CASE(6)
    }
#undef IND_CASE
  }
}

// Nodal polynomial filter: q <- q - alpha (q - P_{p-1} q) = (1 - alpha) q +
// alpha P_{p-1} q, one thread per (element, variable): modal coefficients
// direction by direction, the modes with some index equal to p kept (they are
// q - P_{p-1} q), back to nodal values, subtracted with weight alpha.
template <int ND, int P>
__global__ void k_filter(double* __restrict__ q, const BasisTab<double>* __restrict__ basis, int64_t state_base,
                         int count, double alpha) {
  constexpr int NV = ND + 2;
  constexpr int NSP = ND == 2 ? P * P : P * P * P;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (tid >= (int64_t)count * NV) return;
  const BasisTab<double>& B = basis[P];
  double* s = q + state_base + tid * NSP;   // element tid / NV, variable tid % NV
  double c[NSP], t[NSP];
  for (int k = 0; k < NSP; ++k) c[k] = s[k];
  for (int d = 0; d < ND; ++d) {
    const int stride = d == 0 ? 1 : (d == 1 ? P : P * P);
    for (int k = 0; k < NSP; ++k) {
      const int id = (k / stride) % P, base = k - id * stride;
      double acc = 0.0;
      for (int m = 0; m < P; ++m) acc += B.modal[id][m] * c[base + m * stride];
      t[k] = acc;
    }
    for (int k = 0; k < NSP; ++k) c[k] = t[k];
  }
  for (int k = 0; k < NSP; ++k) {
    const int i0 = k % P, i1 = (k / P) % P, i2 = ND == 3 ? k / (P * P) : 0;
    const bool top = i0 == P - 1 || i1 == P - 1 || (ND == 3 && i2 == P - 1);
    if (!top) c[k] = 0.0;
  }
  for (int d = 0; d < ND; ++d) {
    const int stride = d == 0 ? 1 : (d == 1 ? P : P * P);
    for (int k = 0; k < NSP; ++k) {
      const int id = (k / stride) % P, base = k - id * stride;
      double acc = 0.0;
      for (int m = 0; m < P; ++m) acc += B.nodal[id][m] * c[base + m * stride];
      t[k] = acc;
    }
    for (int k = 0; k < NSP; ++k) c[k] = t[k];
  }
  for (int k = 0; k < NSP; ++k) s[k] -= alpha * c[k];
}

// ---------------------------------------------------------------------------
// adaptation
// ---------------------------------------------------------------------------
__global__ void k_decide(const double* __restrict__ eta, const double* __restrict__ eta_max,
                         const int8_t* __restrict__ p_old, double nu_max, double nu_min, int p_min,
                         int p_max, int E, int8_t* __restrict__ p_new) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= E) return;
  int p = p_old[e];
  const double em = eta_max[0];
  if (em > 0.0) {
    if (eta[e] > nu_max * em) p += 1;
    if (eta[e] < nu_min * em) p -= 1;
  }
  p = p < p_min ? p_min : (p > p_max ? p_max : p);
  p_new[e] = (int8_t)p;
}

// one Jacobi sweep of p_e <- max(p_e, max_n p_n - 1)
__global__ void k_smooth(const int8_t* __restrict__ p_in, const int32_t* __restrict__ nbr, int nf, int E,
                         int8_t* __restrict__ p_out) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= E) return;
  int p = p_in[e];
  for (int f = 0; f < nf; ++f) {
    const int n = nbr[(int64_t)e * nf + f];
    if (n >= 0) p = max(p, (int)p_in[n] - 1);
  }
  p_out[e] = (int8_t)p;
}

// dst[0, *n) = src[0, *n): the transferred state back into the caller's buffer
// (its length is still on the device)
template <typename T>
__global__ void k_copy_n(const T* __restrict__ src, T* __restrict__ dst, const int64_t* __restrict__ n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < *n; i += (int64_t)gridDim.x * blockDim.x)
    dst[i] = src[i];
}

// state transfer: one block per new slot; 1D operator applied in each direction
template <typename T, int ND>
__global__ void k_transfer(const T* __restrict__ q_old, T* __restrict__ q_new,
                           const int32_t* __restrict__ new_slot_elem, const int32_t* __restrict__ old_elem_slot,
                           const int64_t* __restrict__ old_state_off, const int8_t* __restrict__ old_slot_p,
                           const int8_t* __restrict__ p_new, const int64_t* __restrict__ new_state_off,
                           const double* __restrict__ xfer, int E) {
  constexpr int NV = ND + 2;
  constexpr int MAXSP = ND == 2 ? 36 : 216;
  __shared__ double a[MAXSP], b[MAXSP];
  const int slot = blockIdx.x;
  if (slot >= E) return;
  const int e = new_slot_elem[slot];
  const int so = old_elem_slot[e];
  const int Po = old_slot_p[so] + 1, Pn = p_new[e] + 1;
  const T* src = q_old + old_state_off[so];
  T* dst = q_new + new_state_off[slot];
  const double* M = xfer + ((size_t)Po * (kPM + 1) + Pn) * kPM * kPM;   // M[i_new][k_old]
  const int nso = ND == 2 ? Po * Po : Po * Po * Po;
  const int nsn = ND == 2 ? Pn * Pn : Pn * Pn * Pn;
  for (int v = 0; v < NV; ++v) {
    for (int k = threadIdx.x; k < nso; k += blockDim.x) a[k] = (double)src[v * nso + k];
    __syncthreads();
    // apply along xi, eta, zeta; sizes change from Po to Pn one axis at a time
    int dims[3] = {Po, Po, ND == 3 ? Po : 1};
    double* in = a;
    double* out = b;
    for (int d = 0; d < ND; ++d) {
      int nd_[3] = {dims[0], dims[1], dims[2]};
      nd_[d] = Pn;
      const int nout = nd_[0] * nd_[1] * nd_[2];
      for (int k = threadIdx.x; k < nout; k += blockDim.x) {
        int i[3] = {k % nd_[0], (k / nd_[0]) % nd_[1], k / (nd_[0] * nd_[1])};
        double acc = 0.0;
        for (int m = 0; m < dims[d]; ++m) {
          int j[3] = {i[0], i[1], i[2]};
          j[d] = m;
          acc += M[i[d] * kPM + m] * in[j[0] + dims[0] * (j[1] + dims[1] * j[2])];
        }
        out[k] = acc;
      }
      __syncthreads();
      dims[d] = Pn;
      double* tmp = in;
      in = out;
      out = tmp;
    }
    for (int k = threadIdx.x; k < nsn; k += blockDim.x) dst[v * nsn + k] = (T)in[k];
    __syncthreads();
  }
}

static fr_status ensure_transfer_tables(fr_ctx* c, double** out) {
  static_assert(kPM == 6, "transfer table layout");
  if (c->d_xfer) {
    *out = c->d_xfer;
    return FR_OK;
  }
  std::vector<double> h((size_t)(kPM + 1) * (kPM + 1) * kPM * kPM, 0.0);
  for (int Po = 2; Po <= kPM; ++Po)
    for (int Pn = 2; Pn <= kPM; ++Pn) {
      double* M = h.data() + ((size_t)Po * (kPM + 1) + Pn) * kPM * kPM;
      double xo[kPM], wo[kPM], xn[kPM], wn[kPM];
      gauss_legendre(Po, xo, wo);
      gauss_legendre(Pn, xn, wn);
      if (Pn >= Po) {
        // prolongation: interpolate the degree Po-1 polynomial at the new points
        for (int i = 0; i < Pn; ++i) lagrange_eval(xo, Po, xn[i], M + i * kPM);
      } else {
        // projection: Legendre coefficients of the old field, modes < Pn kept
        for (int i = 0; i < Pn; ++i)
          for (int k = 0; k < Po; ++k) {
            double acc = 0.0;
            for (int m = 0; m < Pn; ++m) acc += legendre_p(m, xn[i]) * 0.5 * (2 * m + 1) * wo[k] * legendre_p(m, xo[k]);
            M[i * kPM + k] = acc;
          }
      }
    }
  if (cudaMalloc(&c->d_xfer, sizeof(double) * h.size()) != cudaSuccess) return FR_ERR_NOMEM;
  cudaMemcpy(c->d_xfer, h.data(), sizeof(double) * h.size(), cudaMemcpyHostToDevice);
  *out = c->d_xfer;
  return FR_OK;
}

}  // namespace frgb

using namespace frgb;

extern "C" {

fr_status spectral_decay_indicator(fr_ctx* c, const void* q_dev, fr_prec prec, int32_t var, double* eta_dev,
                                   double* eta_max_dev, void* stream) {
  if (!c || !q_dev || !eta_dev || (prec != FR_F64 && prec != FR_F32 && prec != FR_BF16OP) || var < 0 || var >= c->nv) {
    set_error("spectral_decay_indicator: bad argument");
    return FR_ERR_INVALID;
  }
  cudaStream_t s = (cudaStream_t)stream;
  if (c->nd == 2) {
    if (prec == FR_F64) launch_indicator<double, 2>(c, (const double*)q_dev, var, eta_dev, s);
    else launch_indicator<float, 2>(c, (const float*)q_dev, var, eta_dev, s);
  } else {
    if (prec == FR_F64) launch_indicator<double, 3>(c, (const double*)q_dev, var, eta_dev, s);
    else launch_indicator<float, 3>(c, (const float*)q_dev, var, eta_dev, s);
  }
  if (eta_max_dev) {
    if (!c->d_adapt_f64 && cudaMalloc(&c->d_adapt_f64, sizeof(double) * 1024) != cudaSuccess) return FR_ERR_NOMEM;
    double* part = c->d_adapt_f64;
    FR_LAUNCH(c, "indicator", s, k_max_partial<<<256, 256, 0, s>>>(eta_dev, c->E, part));
    FR_LAUNCH(c, "indicator", s, k_max_final<<<1, 32, 0, s>>>(part, 256, eta_max_dev));
  }
  return cuda_check(cudaGetLastError(), "spectral_decay_indicator");
}

fr_status p_rebucket(fr_ctx* c, const double* eta_dev, const double* eta_max_dev, const fr_adapt_opts* o,
                     void* q_dev, fr_prec prec, int32_t* perm_out_dev, void* stream) {
  if (!c || !eta_dev || !eta_max_dev || !o || !q_dev || (prec != FR_F64 && prec != FR_F32 && prec != FR_BF16OP) ||
      o->p_min < c->p_min || o->p_max > c->p_max || o->p_min > o->p_max) {
    set_error("p_rebucket: bad argument (degrees must lie within the context's limits)");
    return FR_ERR_INVALID;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const int E = c->E, nf = c->nf;
  if (!c->d_adapt_i8 && cudaMalloc(&c->d_adapt_i8, 2 * (size_t)E) != cudaSuccess) return FR_ERR_NOMEM;
  fr_status e = layout_spare(c);
  if (e != FR_OK) return e;
  double* xfer = nullptr;
  if ((e = ensure_transfer_tables(c, &xfer)) != FR_OK) return e;
  void* tmp = prec == FR_F64 ? (void*)vec64(c, 10) : (void*)vec32(c, 3);
  if (!tmp) return FR_ERR_NOMEM;
  int8_t* pa = c->d_adapt_i8;
  int8_t* pb = pa + E;
  const unsigned ge = (unsigned)((E + 255) / 256);
  FR_LAUNCH(c, "rebucket", s, k_decide<<<ge, 256, 0, s>>>(eta_dev, eta_max_dev, c->d_p, o->nu_max, o->nu_min,
                                                           o->p_min, o->p_max, E, pa));
  // jump limit: after k Jacobi sweeps an element holds max_n (p_n - d(e, n)) over
  // the elements within k faces, and one further away than p_max - p_min - 1
  // cannot raise it above p_min: the fixed point, without asking the device
  for (int k = 0; k < o->p_max - o->p_min - 1; ++k) {
    FR_LAUNCH(c, "rebucket", s, k_smooth<<<ge, 256, 0, s>>>(pa, c->d_nbr, nf, E, pb));
    std::swap(pa, pb);
  }
  // the new layout beside the current one, which the transfer reads and which
  // calls in flight on other streams of this context may still be reading
  const LayoutTables& now = c->lt;
  const LayoutTables& next = c->lt_spare;
  if ((e = layout_device(c, pa, next, s)) != FR_OK) return e;
  cudaMemcpyAsync(c->d_p, pa, E, cudaMemcpyDeviceToDevice, s);
  const unsigned gc = (unsigned)std::max<int64_t>(1, std::min<int64_t>((c->n_dof_cap + 255) / 256, (int64_t)c->sms * 16));
#define FR_TRANSFER(T, ND)                                                                                            \
  do {                                                                                                                \
    FR_LAUNCH(c, "rebucket", s,                                                                                       \
              k_transfer<T, ND><<<E, 128, 0, s>>>((const T*)q_dev, (T*)tmp, next.slot_elem, now.elem_slot,            \
                                                  now.state_off, now.slot_p, pa, next.state_off, xfer, E));           \
    FR_LAUNCH(c, "rebucket", s, k_copy_n<T><<<gc, 256, 0, s>>>((const T*)tmp, (T*)q_dev, layout_n_dof(c)));            \
  } while (0)
  if (c->nd == 2) {
    if (prec == FR_F64) FR_TRANSFER(double, 2);
    else FR_TRANSFER(float, 2);
  } else {
    if (prec == FR_F64) FR_TRANSFER(double, 3);
    else FR_TRANSFER(float, 3);
  }
#undef FR_TRANSFER
  if (perm_out_dev) cudaMemcpyAsync(perm_out_dev, next.slot_elem, sizeof(int32_t) * E, cudaMemcpyDeviceToDevice, s);
  if (cudaStreamSynchronize(s) != cudaSuccess) return cuda_check(cudaGetLastError(), "p_rebucket");
  const int8_t* pnew = layout_degrees(c);
  if (!std::equal(pnew, pnew + E, c->p.begin())) {   // unchanged degrees: the current tables stay
    // once nothing in flight reads the current tables (nor the tile table,
    // which layout_host rewrites), they become the next call's spare ones
    if (cudaDeviceSynchronize() != cudaSuccess) return cuda_check(cudaGetLastError(), "p_rebucket");
    std::swap(c->lt, c->lt_spare);
    c->p.assign(pnew, pnew + E);
    if ((e = layout_host(c, s)) != FR_OK) return e;
    if (cudaStreamSynchronize(s) != cudaSuccess) return cuda_check(cudaGetLastError(), "p_rebucket");   // its tile table
  }
  return cuda_check(cudaGetLastError(), "p_rebucket");
}

fr_status fr_filter(fr_ctx* c, double* q_dev, double alpha, int32_t p_above, void* stream) {
  if (!c || !q_dev || !(alpha >= 0.0 && alpha <= 1.0)) {
    set_error("fr_filter: bad argument");
    return FR_ERR_INVALID;
  }
  cudaStream_t s = (cudaStream_t)stream;
  for (const auto& b : c->buckets) {
    if (b.p <= p_above || b.count == 0 || alpha == 0.0) continue;
    const int P = b.p + 1, NSP = c->nd == 2 ? P * P : P * P * P;
    const int64_t nt = (int64_t)b.count * c->nv;
    const unsigned grid = (unsigned)((nt + 127) / 128);
    const double nb = 16.0 * nt * NSP;
#define FILT_CASE(ND, PP) \
  case PP: FR_LAUNCH_B(c, "filter", s, nb, k_filter<ND, PP><<<grid, 128, 0, s>>>((double*)q_dev, c->d_basis64, b.state_base, b.count, alpha)); break;
    if (c->nd == 2) {
      switch (P) { FILT_CASE(2, 2) FILT_CASE(2, 3) FILT_CASE(2, 4) FILT_CASE(2, 5) FILT_CASE(2, 6) }
    } else {
      switch (P) { FILT_CASE(3, 2) FILT_CASE(3, 3) FILT_CASE(3, 4) FILT_CASE(3, 5) FILT_CASE(3, 6) }
    }
#undef FILT_CASE
    (void)NSP;
  }
  return cuda_check(cudaGetLastError(), "fr_filter");
}

fr_status fr_esdirk_tableau(int32_t order, fr_tableau* t) {
  if (!t || (order != 2 && order != 3)) {
    set_error("fr_esdirk_tableau: order must be 2 or 3");
    return FR_ERR_INVALID;
  }
  std::memset(t, 0, sizeof(*t));
  if (order == 2) {
    // 3 stages, stiffly accurate, diagonal g = 1 - sqrt(2)/2, c = (0, 2g, 1)
    const double g = 1.0 - std::sqrt(2.0) / 2.0;
    const double b2 = (0.5 - g) / (2.0 * g), b1 = 1.0 - g - b2;
    t->s = 3;
    const double A[9] = {0, 0, 0, g, g, 0, b1, b2, g};
    std::memcpy(t->A, A, sizeof(A));
    t->b[0] = b1; t->b[1] = b2; t->b[2] = g;
    return FR_OK;
  }
  // 4 stages, order 3, stiffly accurate; g: root of 6g^3 - 18g^2 + 9g - 1 near 0.4359
  double g = 0.44;
  for (int it = 0; it < 60; ++it) g -= (6 * g * g * g - 18 * g * g + 9 * g - 1) / (18 * g * g - 36 * g + 9);
  const double c2 = 2 * g, c3 = 0.6;
  const double r1 = 0.5 - g, r2 = 1.0 / 3.0 - g;
  const double det = c2 * c3 * c3 - c3 * c2 * c2;
  const double b2 = (r1 * c3 * c3 - c3 * r2) / det, b3 = (c2 * r2 - r1 * c2 * c2) / det;
  const double b1 = 1.0 - g - b2 - b3;
  const double a32 = (1.0 / 6.0 - 0.5 * g - 2 * g * g * b2 - g * c3 * b3) / (2 * g * b3);
  const double a31 = c3 - g - a32;
  t->s = 4;
  const double A[16] = {0, 0, 0, 0, g, g, 0, 0, a31, a32, g, 0, b1, b2, b3, g};
  std::memcpy(t->A, A, sizeof(A));
  t->b[0] = b1; t->b[1] = b2; t->b[2] = b3; t->b[3] = g;
  return FR_OK;
}

}  // extern "C"
