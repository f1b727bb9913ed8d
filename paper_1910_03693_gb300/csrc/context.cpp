// Context creation: validation and metric terms; the C-ABI entry points that
// only need host logic.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <vector>

#include "fr_internal.h"

namespace frgb {

static thread_local std::string g_last_error;

void set_error(const std::string& msg) { g_last_error = msg; }

fr_status cuda_check(cudaError_t e, const char* what) {
  if (e == cudaSuccess) return FR_OK;
  set_error(std::string(what) + ": " + cudaGetErrorString(e));
  return e == cudaErrorMemoryAllocation ? FR_ERR_NOMEM : FR_ERR_CUDA;
}

#define FR_TRY(x)                      \
  do {                                 \
    fr_status _st = (x);               \
    if (_st != FR_OK) return _st;      \
  } while (0)
#define FR_CUDA(x) FR_TRY(cuda_check((x), #x))

static int ipow(int b, int e) {
  int r = 1;
  while (e-- > 0) r *= b;
  return r;
}

// ---------------------------------------------------------------------------
// Metric terms of one element at degree p (cross-product form from the
// derivatives of the degree-p interpolant of the element map).
//   vol  [(nd*nd+1)][NSP]   : S[d][j] at k = d*nd + j, |J| at k = nd*nd
//   face [nf][(nd*nd+1)][NFP]: the same extrapolated to every face
// ---------------------------------------------------------------------------
static void element_metrics(const fr_ctx* c, int e, int p, double* vol, double* face) {
  const int nd = c->nd, g = c->geom_order, nn = g + 1, P = p + 1;
  const int NSP = ipow(P, nd), NFP = ipow(P, nd - 1), NK = nd * nd + 1;
  BasisTab<double> B;
  build_basis(p, B);
  double equi[3];
  for (int a = 0; a < nn; ++a) equi[a] = -1.0 + 2.0 * a / g;
  double N1[kPM][3];
  for (int i = 0; i < P; ++i) lagrange_eval(equi, nn, B.x[i], N1[i]);
  const double* X = c->nodes.data() + (size_t)e * ipow(nn, nd) * nd;
  // coordinates at the solution points
  std::vector<double> Xs((size_t)nd * NSP, 0.0);
  for (int sp = 0; sp < NSP; ++sp) {
    int id[3] = {sp % P, (sp / P) % P, nd == 3 ? sp / (P * P) : 0};
    for (int node = 0; node < ipow(nn, nd); ++node) {
      int nid[3] = {node % nn, (node / nn) % nn, nd == 3 ? node / (nn * nn) : 0};
      double w = 1.0;
      for (int d = 0; d < nd; ++d) w *= N1[id[d]][nid[d]];
      for (int cc = 0; cc < nd; ++cc) Xs[cc * NSP + sp] += w * X[node * nd + cc];
    }
  }
  // derivatives dX[d][comp] at the solution points
  std::vector<double> dX((size_t)nd * nd * NSP, 0.0);
  for (int sp = 0; sp < NSP; ++sp) {
    int id[3] = {sp % P, (sp / P) % P, nd == 3 ? sp / (P * P) : 0};
    for (int d = 0; d < nd; ++d) {
      const int stride = ipow(P, d);
      const int base = sp - id[d] * stride;
      for (int cc = 0; cc < nd; ++cc) {
        double acc = 0.0;
        for (int k = 0; k < P; ++k) acc += B.D[id[d]][k] * Xs[cc * NSP + base + k * stride];
        dX[(d * nd + cc) * NSP + sp] = acc;
      }
    }
  }
  for (int sp = 0; sp < NSP; ++sp) {
    auto D = [&](int d, int cc) { return dX[(d * nd + cc) * NSP + sp]; };
    if (nd == 2) {
      vol[0 * NSP + sp] = D(1, 1);    // S[0][0] = y_eta
      vol[1 * NSP + sp] = -D(1, 0);   // S[0][1] = -x_eta
      vol[2 * NSP + sp] = -D(0, 1);   // S[1][0] = -y_xi
      vol[3 * NSP + sp] = D(0, 0);    // S[1][1] = x_xi
      vol[4 * NSP + sp] = D(0, 0) * D(1, 1) - D(1, 0) * D(0, 1);
    } else {
      for (int i = 0; i < 3; ++i) {
        int j = (i + 1) % 3, k = (i + 2) % 3;
        vol[(i * 3 + 0) * NSP + sp] = D(j, 1) * D(k, 2) - D(j, 2) * D(k, 1);
        vol[(i * 3 + 1) * NSP + sp] = D(j, 2) * D(k, 0) - D(j, 0) * D(k, 2);
        vol[(i * 3 + 2) * NSP + sp] = D(j, 0) * D(k, 1) - D(j, 1) * D(k, 0);
      }
      // det of a[comp][d] = dX[d][comp]
      double a00 = D(0, 0), a01 = D(1, 0), a02 = D(2, 0);
      double a10 = D(0, 1), a11 = D(1, 1), a12 = D(2, 1);
      double a20 = D(0, 2), a21 = D(1, 2), a22 = D(2, 2);
      vol[9 * NSP + sp] = a00 * (a11 * a22 - a12 * a21) - a01 * (a10 * a22 - a12 * a20) +
                          a02 * (a10 * a21 - a11 * a20);
    }
  }
  // extrapolate every component to every face
  for (int f = 0; f < 2 * nd; ++f) {
    const int d = f / 2, s = f % 2, stride = ipow(P, d);
    for (int t = 0; t < NFP; ++t) {
      int ta = t % P, tb = t / P;
      int id[3];
      if (nd == 2) {
        id[d == 0 ? 1 : 0] = ta;
      } else {
        int ax[2] = {d == 0 ? 1 : 0, d == 2 ? 1 : 2};
        id[ax[0]] = ta;
        id[ax[1]] = tb;
      }
      id[d] = 0;
      if (nd == 2) id[2] = 0;
      int base = id[0] + P * id[1] + (nd == 3 ? P * P * id[2] : 0);
      for (int kk = 0; kk < NK; ++kk) {
        double acc = 0.0;
        for (int k = 0; k < P; ++k) acc += B.ext[s][k] * vol[kk * NSP + base + k * stride];
        face[((size_t)f * NK + kk) * NFP + t] = acc;
      }
    }
  }
}

static bool element_is_affine(const fr_ctx* c, int e) {
  if (c->geom_order != 1) return false;
  const int nd = c->nd;
  const double* X = c->nodes.data() + (size_t)e * ipow(2, nd) * nd;
  auto node = [&](int i, int j, int k, int cc) { return X[(i + 2 * j + 4 * k) * nd + cc]; };
  double scale = 0.0, twist = 0.0;
  for (int cc = 0; cc < nd; ++cc) {
    scale = std::max(scale, std::fabs(node(1, 0, 0, cc) - node(0, 0, 0, cc)));
    scale = std::max(scale, std::fabs(node(0, 1, 0, cc) - node(0, 0, 0, cc)));
    if (nd == 2) {
      twist = std::max(twist, std::fabs(node(0, 0, 0, cc) - node(1, 0, 0, cc) - node(0, 1, 0, cc) +
                                        node(1, 1, 0, cc)));
    } else {
      scale = std::max(scale, std::fabs(node(0, 0, 1, cc) - node(0, 0, 0, cc)));
      // coefficients of xi*eta, xi*zeta, eta*zeta, xi*eta*zeta of the trilinear map
      double t1 = node(0, 0, 0, cc) - node(1, 0, 0, cc) - node(0, 1, 0, cc) + node(1, 1, 0, cc);
      double t2 = node(0, 0, 0, cc) - node(1, 0, 0, cc) - node(0, 0, 1, cc) + node(1, 0, 1, cc);
      double t3 = node(0, 0, 0, cc) - node(0, 1, 0, cc) - node(0, 0, 1, cc) + node(0, 1, 1, cc);
      double t4 = -node(0, 0, 0, cc) + node(1, 0, 0, cc) + node(0, 1, 0, cc) + node(0, 0, 1, cc) -
                  node(1, 1, 0, cc) - node(1, 0, 1, cc) - node(0, 1, 1, cc) + node(1, 1, 1, cc);
      twist = std::max({twist, std::fabs(t1), std::fabs(t2), std::fabs(t3), std::fabs(t4)});
    }
  }
  return twist <= 1e-13 * scale;
}

// Whether both sides of every interior face have the same axis and the same
// tangential metric (axis-aligned elements, metrics g as below).  The viscous
// diagonal-metric face kernels rely on it: they take the tangential part of the
// common gradient from q^com with the master's metric, and the slave's normal
// metric on the master's axis.  The connectivity alone does not ensure it
// (layers of different extent glued together, axes exchanged or reflected
// across a face).  Extents are compared to the rounding of the nodes they are
// differences of.
static bool faces_match(const fr_ctx* c, const std::vector<double>& g, int nk) {
  const int nd = c->nd, nf = c->nf;
  double xmax = 0.0;
  for (double x : c->nodes) xmax = std::max(xmax, std::fabs(x));
  auto extent = [&](int e, int j) {   // |J| / S_jj
    const double* m = g.data() + (size_t)e * nk;
    return m[nd * nd] / m[j * nd + j];
  };
  for (int e = 0; e < c->E; ++e)
    for (int f = 0; f < nf; ++f) {
      const int n = c->nbr[(size_t)e * nf + f], o = c->orient[(size_t)e * nf + f];
      if (n < 0) continue;
      const int d = f >> 1;
      if ((c->nbr_face[(size_t)e * nf + f] >> 1) != d || (o & 1)) return false;
      for (int j = 0, k = 0; j < nd; ++j) {
        if (j == d) continue;
        const double a = extent(e, j), b = extent(n, j), flip = (o >> ++k) & 1 ? -1.0 : 1.0;
        if (std::fabs(a - flip * b) > 1e-12 * std::fabs(a) + 64.0 * 2.2e-16 * xmax) return false;
      }
    }
  return true;
}

void collect_graph_timers(fr_ctx* c) {
  for (int k = 0; k < 2; ++k)
    if (c->graph_timers_live[k]) {
      c->timing.accumulate(c->graph_timers[k]);
      c->graph_timers_live[k] = false;
    }
}

void clear_graphs(fr_ctx* c) {
  collect_graph_timers(c);
  for (int k = 0; k < 2; ++k) {
    if (c->jvp_graph[k]) cudaGraphExecDestroy(c->jvp_graph[k]);
    c->jvp_graph[k] = nullptr;
    for (auto& r : c->graph_timers[k]) c->timing.give_back(r);
    c->graph_timers[k].clear();
    c->graph_timers_live[k] = false;
    for (auto& p : c->jvp_graph_key[k]) p = nullptr;
  }
}

void clear_work_cache(fr_ctx* c) {
  c->pc_ready = false;   // the layout or the tuning changed: blocks must be rebuilt
  clear_graphs(c);
  cudaDeviceSynchronize();   // launches still reading the tile table
  rebuild_work_table(c, nullptr);
  cudaStreamSynchronize(nullptr);
}

template <typename T>
static fr_status upload_cast(const std::vector<double>& h, T** d) {
  std::vector<T> tmp(h.begin(), h.end());
  FR_CUDA(cudaMalloc(d, sizeof(T) * std::max<size_t>(tmp.size(), 1)));
  FR_CUDA(cudaMemcpy(*d, tmp.data(), sizeof(T) * tmp.size(), cudaMemcpyHostToDevice));
  return FR_OK;
}

static fr_status create_impl(const fr_mesh_desc* m, const fr_physics* ph, const fr_limits* lim,
                             fr_ctx* c) {
  if (!m || !ph || !lim || !m->nodes || !m->nbr || !m->nbr_face || !m->orient || !m->p) {
    set_error("fr_create: null argument");
    return FR_ERR_INVALID;
  }
  if ((m->nd != 2 && m->nd != 3) || m->n_elem <= 0 || (m->geom_order != 1 && m->geom_order != 2)) {
    set_error("fr_create: nd must be 2 or 3, n_elem > 0, geom_order 1 or 2");
    return FR_ERR_INVALID;
  }
  if (lim->p_min < 1 || lim->p_max > kMaxDeg || lim->p_min > lim->p_max) {
    set_error("fr_create: need 1 <= p_min <= p_max <= 5");
    return FR_ERR_INVALID;
  }
  if (!(ph->gamma > 1.0) || ph->mu < 0.0 || (ph->mu > 0.0 && !(ph->Pr > 0.0)) ||
      (ph->flux != FR_FLUX_RUSANOV && ph->flux != FR_FLUX_ROE)) {
    set_error("fr_create: need gamma > 1, mu >= 0, Pr > 0 and a known common flux");
    return FR_ERR_INVALID;
  }
  c->nd = m->nd;
  c->nv = m->nd + 2;
  c->nf = 2 * m->nd;
  c->E = m->n_elem;
  c->geom_order = m->geom_order;
  c->p_min = lim->p_min;
  c->p_max = lim->p_max;
  c->visc = ph->mu > 0.0;
  c->phys.gamma = ph->gamma;
  c->phys.mu = ph->mu;
  c->phys.Pr = ph->Pr;
  c->phys.kappa = c->visc ? ph->mu * ph->gamma / ((ph->gamma - 1.0) * ph->Pr) : 0.0;
  for (int v = 0; v < 5; ++v) c->phys.q_inf[v] = ph->q_inf[v];
  c->phys.flux = ph->flux;
  const int nd = c->nd, nf = c->nf, E = c->E, nn = c->geom_order + 1;
  c->nodes.assign(m->nodes, m->nodes + (size_t)E * ipow(nn, nd) * nd);
  c->nbr.assign(m->nbr, m->nbr + (size_t)E * nf);
  c->nbr_face.assign(m->nbr_face, m->nbr_face + (size_t)E * nf);
  c->orient.assign(m->orient, m->orient + (size_t)E * nf);
  c->p.assign(m->p, m->p + E);
  for (int e = 0; e < E; ++e) {
    if (c->p[e] < c->p_min || c->p[e] > c->p_max) {
      set_error("fr_create: element degree outside [p_min, p_max]");
      return FR_ERR_INVALID;
    }
    for (int f = 0; f < nf; ++f) {
      const int n = c->nbr[(size_t)e * nf + f];
      if (n >= E || (n < 0 && n != FR_BC_WALL && n != FR_BC_FARFIELD)) {
        set_error("fr_create: bad neighbour index");
        return FR_ERR_INVALID;
      }
      if (n >= 0) {
        const int g = c->nbr_face[(size_t)e * nf + f];
        if (g < 0 || g >= nf || c->nbr[(size_t)n * nf + g] != e || c->nbr_face[(size_t)n * nf + g] != f) {
          set_error("fr_create: face connectivity is not symmetric");
          return FR_ERR_INVALID;
        }
        const int o = c->orient[(size_t)e * nf + f];
        if (o < 0 || o > 7 || (nd == 2 && (o & 5))) {
          set_error("fr_create: bad orientation code");
          return FR_ERR_INVALID;
        }
      }
    }
  }
  FR_CUDA(cudaGetDevice(&c->device));
  if (cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess || c->sms <= 0) {
    cudaGetLastError();
    c->sms = 152;
  }
  c->nvt = c->visc ? (1 + nd) * c->nv : c->nv;

  // basis and mortar tables
  std::vector<BasisTab<double>> b64(kPM + 1);
  std::vector<BasisTab<float>> b32(kPM + 1);
  for (int P = 2; P <= kPM; ++P) {
    build_basis(P - 1, b64[P]);
    const double* src = reinterpret_cast<const double*>(&b64[P]);
    float* dst = reinterpret_cast<float*>(&b32[P]);
    for (size_t k = 0; k < sizeof(BasisTab<double>) / sizeof(double); ++k) dst[k] = (float)src[k];
  }
  std::vector<MortarTab<double>> m64((kPM + 1) * (kPM + 1));
  std::vector<MortarTab<float>> m32((kPM + 1) * (kPM + 1));
  for (int Pm = 2; Pm <= kPM; ++Pm)
    for (int Ps = 2; Ps < Pm; ++Ps) {
      auto& t = m64[Pm * (kPM + 1) + Ps];
      build_mortar(Ps - 1, Pm - 1, t);
      const double* src = reinterpret_cast<const double*>(&t);
      float* dst = reinterpret_cast<float*>(&m32[Pm * (kPM + 1) + Ps]);
      for (size_t k = 0; k < sizeof(MortarTab<double>) / sizeof(double); ++k) dst[k] = (float)src[k];
    }
  // the same tables rounded to bfloat16 (nearest, ties to even), kept in float
  auto bf16 = [](float x) {
    uint32_t u;
    std::memcpy(&u, &x, 4);
    if ((u & 0x7f800000u) != 0x7f800000u) u = (u + 0x7fffu + ((u >> 16) & 1u)) & 0xffff0000u;
    float y;
    std::memcpy(&y, &u, 4);
    return y;
  };
  std::vector<BasisTab<float>> b16(b32);
  std::vector<MortarTab<float>> m16(m32);
  for (auto& t : b16) {
    float* f = reinterpret_cast<float*>(&t);
    for (size_t k = 0; k < sizeof(BasisTab<float>) / sizeof(float); ++k) f[k] = bf16(f[k]);
  }
  for (auto& t : m16) {
    float* f = reinterpret_cast<float*>(&t);
    for (size_t k = 0; k < sizeof(MortarTab<float>) / sizeof(float); ++k) f[k] = bf16(f[k]);
  }
  FR_CUDA(cudaMalloc(&c->d_basis16, sizeof(BasisTab<float>) * b16.size()));
  FR_CUDA(cudaMemcpy(c->d_basis16, b16.data(), sizeof(BasisTab<float>) * b16.size(), cudaMemcpyHostToDevice));
  FR_CUDA(cudaMalloc(&c->d_mortar16, sizeof(MortarTab<float>) * m16.size()));
  FR_CUDA(cudaMemcpy(c->d_mortar16, m16.data(), sizeof(MortarTab<float>) * m16.size(), cudaMemcpyHostToDevice));
  FR_CUDA(cudaMalloc(&c->d_basis64, sizeof(BasisTab<double>) * b64.size()));
  FR_CUDA(cudaMalloc(&c->d_basis32, sizeof(BasisTab<float>) * b32.size()));
  FR_CUDA(cudaMemcpy(c->d_basis64, b64.data(), sizeof(BasisTab<double>) * b64.size(), cudaMemcpyHostToDevice));
  FR_CUDA(cudaMemcpy(c->d_basis32, b32.data(), sizeof(BasisTab<float>) * b32.size(), cudaMemcpyHostToDevice));
  FR_CUDA(cudaMalloc(&c->d_mortar64, sizeof(MortarTab<double>) * m64.size()));
  FR_CUDA(cudaMalloc(&c->d_mortar32, sizeof(MortarTab<float>) * m32.size()));
  FR_CUDA(cudaMemcpy(c->d_mortar64, m64.data(), sizeof(MortarTab<double>) * m64.size(), cudaMemcpyHostToDevice));
  FR_CUDA(cudaMemcpy(c->d_mortar32, m32.data(), sizeof(MortarTab<float>) * m32.size(), cudaMemcpyHostToDevice));

  // geometry
  c->affine = true;
  for (int e = 0; e < E && c->affine; ++e) c->affine = element_is_affine(c, e);
  const int NK = nd * nd + 1, NKV = geo_nk_vol(nd), NKF = geo_nk_face(nd);
  // the derived components of one point: src holds S and |J| with stride `ss`
  auto derive = [nd, NK](const double* src, int64_t ss, double* dst, int64_t ds, bool face_terms) {
    for (int k = 0; k < NK; ++k) dst[k * ds] = src[k * ss];
    dst[NK * ds] = 1.0 / src[(NK - 1) * ss];
    if (!face_terms) return;
    for (int d = 0; d < nd; ++d) {
      double a2 = 0.0;
      for (int j = 0; j < nd; ++j) a2 += src[(d * nd + j) * ss] * src[(d * nd + j) * ss];
      const double a = std::sqrt(a2);
      dst[(NK + 1 + d) * ds] = a;
      dst[(NK + 1 + nd + d) * ds] = 1.0 / a;
    }
  };
  if (c->affine) {
    // one set of constants per element serves both views (vol uses the first NKV)
    std::vector<double> g((size_t)E * NKF);
    bool diag = nd == 3;
    for (int e = 0; e < E; ++e) {
      // constant metrics: evaluate at degree 0 would be degenerate; use p = 1, first point
      std::vector<double> v1((size_t)NK * ipow(2, nd)), f1((size_t)nf * NK * ipow(2, nd - 1));
      element_metrics(c, e, 1, v1.data(), f1.data());
      // axis-aligned box: the off-diagonal metric terms are rounding noise of
      // the metric evaluation; they are set to exact zeros
      double smax = 0.0, offmax = 0.0;
      for (int d = 0; d < nd; ++d)
        for (int j = 0; j < nd; ++j) {
          const double x = std::fabs(v1[(size_t)(d * nd + j) * ipow(2, nd)]);
          smax = std::max(smax, x);
          if (d != j) offmax = std::max(offmax, x);
        }
      if (offmax <= 1e-13 * smax) {
        for (int d = 0; d < nd; ++d)
          for (int j = 0; j < nd; ++j)
            if (d != j) v1[(size_t)(d * nd + j) * ipow(2, nd)] = 0.0;
      } else {
        diag = false;
      }
      derive(v1.data(), ipow(2, nd), g.data() + (size_t)e * NKF, 1, true);
    }
    c->diag_mesh = diag && (!c->visc || faces_match(c, g, NKF));
    c->diag = c->diag_mesh && c->use_diag;
    FR_TRY(upload_cast(g, &c->d_gaff64));
    FR_TRY(upload_cast(g, &c->d_gaff32));
  } else {
    for (int p = c->p_min; p <= c->p_max; ++p) {
      const int P = p + 1, NSP = ipow(P, nd), NFP = ipow(P, nd - 1);
      std::vector<double> vol((size_t)E * NKV * NSP), face((size_t)E * nf * NKF * NFP);
#pragma omp parallel for schedule(static)
      for (int e = 0; e < E; ++e) {
        std::vector<double> v0((size_t)NK * NSP), f0((size_t)nf * NK * NFP);
        element_metrics(c, e, p, v0.data(), f0.data());
        double* ve = vol.data() + (size_t)e * NKV * NSP;
        double* fe = face.data() + (size_t)e * nf * NKF * NFP;
        for (int sp = 0; sp < NSP; ++sp) derive(v0.data() + sp, NSP, ve + sp, NSP, false);
        for (int f = 0; f < nf; ++f)
          for (int t = 0; t < NFP; ++t)
            derive(f0.data() + (size_t)f * NK * NFP + t, NFP, fe + (size_t)f * NKF * NFP + t, NFP, true);
      }
      FR_TRY(upload_cast(vol, &c->d_gvol64[p]));
      FR_TRY(upload_cast(vol, &c->d_gvol32[p]));
      FR_TRY(upload_cast(face, &c->d_gface64[p]));
      FR_TRY(upload_cast(face, &c->d_gface32[p]));
    }
  }

  // capacities (all elements at p_max)
  {
    const int P = c->p_max + 1, NSP = ipow(P, nd), NFP = ipow(P, nd - 1);
    c->n_dof_cap = (int64_t)E * c->nv * NSP;
    c->trace_cap = (int64_t)E * nf * c->nvt * NFP;
    c->fout_cap = (int64_t)E * nf * 3 * c->nv * NFP;
  }
  FR_CUDA(cudaMalloc(&c->d_trace_q, sizeof(double) * c->trace_cap));
  FR_CUDA(cudaMalloc(&c->d_trace_v, sizeof(double) * c->trace_cap));
  FR_CUDA(cudaMalloc(&c->d_fout, sizeof(double) * c->fout_cap));
  FR_CUDA(cudaMalloc(&c->d_nbr, sizeof(int32_t) * E * nf));
  FR_CUDA(cudaMalloc(&c->d_status, sizeof(int)));
  FR_CUDA(cudaMemset(c->d_status, 0, sizeof(int)));
  FR_CUDA(cudaMemcpy(c->d_nbr, c->nbr.data(), sizeof(int32_t) * E * nf, cudaMemcpyHostToDevice));
  FR_TRY(layout_alloc(c));
  return build_layout(c);
}

static void destroy_impl(fr_ctx* c) {
  cudaFree(c->d_basis64);
  cudaFree(c->d_basis32);
  cudaFree(c->d_basis16);
  cudaFree(c->d_mortar16);
  cudaFree(c->d_mortar64);
  cudaFree(c->d_mortar32);
  cudaFree(c->d_gaff64);
  cudaFree(c->d_gaff32);
  for (int p = 0; p <= kMaxDeg; ++p) {
    cudaFree(c->d_gvol64[p]);
    cudaFree(c->d_gvol32[p]);
    cudaFree(c->d_gface64[p]);
    cudaFree(c->d_gface32[p]);
    cudaFree(c->d_gvol_df[p]);
    cudaFree(c->d_gface_df[p]);
  }
  cudaFree(c->d_basis_df);
  cudaFree(c->d_mortar_df);
  cudaFree(c->d_gaff_df);
  cudaFree(c->d_trace_q);
  cudaFree(c->d_trace_v);
  cudaFree(c->d_fout);
  cudaFree(c->d_fbar);
  cudaFree(c->d_trbar);
  layout_free(c->lt);
  layout_free(c->lt_spare);
  cudaFree(c->d_nbr);
  clear_graphs(c);
  cudaFree(c->d_p);
  cudaFree(c->d_nbr_face);
  cudaFree(c->d_orient);
  cudaFree(c->d_lay);
  cudaFree(c->d_face_hist);
  if (c->h_lay) cudaFreeHost(c->h_lay);
  cudaFree(c->d_work);
  cudaFree(c->d_status);
  cudaFree(c->d_jidx);
  if (c->cap_stream) cudaStreamDestroy(c->cap_stream);
  if (c->h_jidx) cudaFreeHost(c->h_jidx);
  cudaFree(c->d_krylov);
  cudaFree(c->d_krylov32);
  cudaFree(c->d_step);
  free_pc_lanes(c);
  cudaFree(c->d_pc);
  cudaFree(c->d_pc_off);
  cudaFree(c->d_slot_color);
  cudaFree(c->d_pc_status);
  for (auto& v : c->d_vec64) cudaFree(v);
  for (auto& v : c->d_vec32) cudaFree(v);
  cudaFree(c->d_red);
  if (c->h_red) cudaFreeHost(c->h_red);
  cudaFree(c->d_gm);
  if (c->h_gm) cudaFreeHost(c->h_gm);
  cudaFree(c->d_xfer);
  cudaFree(c->d_adapt_i8);
  cudaFree(c->d_adapt_f64);
  delete c;
}

}  // namespace frgb

using namespace frgb;

extern "C" {

const char* fr_last_error(void) { return g_last_error.c_str(); }

fr_status fr_create(const fr_mesh_desc* mesh, const fr_physics* phys, const fr_limits* lim,
                    fr_ctx** out) {
  if (!out) {
    set_error("fr_create: out is null");
    return FR_ERR_INVALID;
  }
  *out = nullptr;
  fr_ctx* c = new (std::nothrow) fr_ctx();
  if (!c) return FR_ERR_NOMEM;
  fr_status st = create_impl(mesh, phys, lim, c);
  if (st != FR_OK) {
    destroy_impl(c);
    return st;
  }
  *out = c;
  return FR_OK;
}

fr_status fr_destroy(fr_ctx* ctx) {
  if (!ctx) return FR_ERR_INVALID;
  destroy_impl(ctx);
  return FR_OK;
}

fr_status fr_layout(const fr_ctx* c, fr_layout_info* info) {
  if (!c || !info) return FR_ERR_INVALID;
  std::memset(info, 0, sizeof(*info));
  info->nd = c->nd;
  info->nv = c->nv;
  info->n_elem = c->E;
  info->n_dof = c->n_dof;
  info->n_dof_capacity = c->n_dof_cap;
  info->affine = c->affine ? 1 : 0;
  for (const auto& b : c->buckets) {
    info->bucket_count[b.p] = b.count;
    info->bucket_offset[b.p] = b.state_base;
  }
  return FR_OK;
}

fr_status fr_get_p(const fr_ctx* c, int8_t* p_host) {
  if (!c || !p_host) return FR_ERR_INVALID;
  std::memcpy(p_host, c->p.data(), c->E);
  return FR_OK;
}

}  // extern "C"
