// Element-Jacobi preconditioner of Sec. 2.3: the inverses of the diagonal
// blocks of sigma I - dR/dq, one dense block per element (all of its DOFs),
// applied from the left in GMRES.
//
// Build (once per physical time step in the paper):
//  * the blocks are read off the exact FP32 JVP with unit vectors: elements
//    of one colour of a distance-1 colouring of the face graph are probed
//    together (a face neighbour never shares the colour, so the product
//    restricted to a probed element is that element's own column), one
//    product per colour and local DOF index;
//  * each block sigma I - J_ee is inverted by Gauss-Jordan elimination with
//    partial pivoting (FP32), and stored column-major.
// Blocks of up to kPcSmem DOFs are inverted in shared memory;
// larger ones (3D p >= 3: 320, 625 and 1080 DOFs) by a blocked in-place
// Gauss-Jordan elimination on the block in global memory (below).
// Apply: z_e = M_e^-1 (a w_e + b u_e), FP32 arithmetic on FP64 vectors.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "fr_launch.h"

namespace frgb {

constexpr int kPcSmem = 144;   // largest block inverted in shared memory (2 x 144^2 floats)
constexpr int kPcMax = 1080;   // largest block stored: 3D p = 5 (5 x 216 DOFs)
constexpr int kPanel = 32;     // columns eliminated together by the blocked inversion
constexpr int kTile = 64;      // columns of one tile of the blocked update

static inline int nsp_host(int nd, int p) { return nd == 2 ? (p + 1) * (p + 1) : (p + 1) * (p + 1) * (p + 1); }

// The buckets of one launch: slots slot_begin .. + count of block size nb.
struct PcBuckets {
  int slot_begin[kMaxDeg + 1], count[kMaxDeg + 1], nb[kMaxDeg + 1];
  int64_t first[kMaxDeg + 2];   // threads (probes) or CTAs (apply) of the buckets before this one
  int n;
};

// One step of the probing of colour `col`, one thread per block row: column k of
// B_s = sigma I - J_ss (column-major, B[k nb + i]) from the product J of the
// unit vectors e_k (skipped for k < 0), and the unit vectors moved on to `next`.
__global__ void k_pc_probe(PcBuckets bk, float* __restrict__ B, const int64_t* __restrict__ pc_off,
                           const float* __restrict__ J, float* __restrict__ v, const int64_t* __restrict__ state_off,
                           const int32_t* __restrict__ slot_color, int col, int k, int next, float sigma) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= bk.first[bk.n]) return;
  int q = 0;
  while (t >= bk.first[q + 1]) ++q;
  const int nb = bk.nb[q];
  const int i = (int)((t - bk.first[q]) % nb);
  const int s = bk.slot_begin[q] + (int)((t - bk.first[q]) / nb);
  if (slot_color[s] != col || pc_off[s] < 0) return;
  const int64_t so = state_off[s];
  if (k >= 0 && k < nb) B[pc_off[s] + (int64_t)k * nb + i] = (i == k ? sigma : 0.0f) - J[so + i];
  if (i == k) v[so + i] = 0.0f;
  if (i == next) v[so + i] = 1.0f;
}

// In-place inverse of one nb x nb block per CTA (column-major in global
// memory) by Gauss-Jordan elimination in shared memory, partial pivoting by
// rows; the row swaps are undone as column swaps at the end.  A warp owns every
// eighth row, its lanes the columns, with the scaled pivot row in registers.
// A zero pivot sets *status and leaves the block as is.  In place the block
// takes nb^2 floats (three CTAs an SM at 135 DOFs; [A | I] with its 2 nb columns
// allowed one and did twice the work: 854 blocks of 40 and 853 of 135 DOFs took
// 12.2 ms, now 1.5 ms, with the same bits).
__global__ void __launch_bounds__(256) k_pc_invert(float* __restrict__ B, const int64_t* __restrict__ pc_off,
                                                   int slot_begin, int nb, int* __restrict__ status) {
  extern __shared__ __align__(16) float sm[];
  const int ld = nb | 1;              // odd: column reads without bank conflicts
  float* M = sm;                      // [nb][ld] row-major
  float* rk = M + (size_t)nb * ld;    // the scaled pivot row
  int* perm = reinterpret_cast<int*>(rk + nb);
  int* cm = perm + nb;
  __shared__ int piv;
  __shared__ float pval;
  constexpr int CW = (kPcSmem + 31) / 32;
  const int s = slot_begin + blockIdx.x;
  const int64_t off = pc_off[s];
  if (off < 0) return;
  float* A = B + off;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int t = tid; t < nb * nb; t += 256) M[(t % nb) * ld + t / nb] = A[t];
  __syncthreads();
  for (int k = 0; k < nb; ++k) {
    // pivot: the row r >= k with the largest |M[r][k]| (lowest row at a tie)
    if (warp == 0) {
      float best = -1.0f;
      int br = k;
      for (int r = k + lane; r < nb; r += 32) {
        const float a = fabsf(M[r * ld + k]);
        if (a > best) {
          best = a;
          br = r;
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const float ob = __shfl_down_sync(0xffffffffu, best, o);
        const int orr = __shfl_down_sync(0xffffffffu, br, o);
        if (ob > best || (ob == best && orr < br)) {
          best = ob;
          br = orr;
        }
      }
      if (lane == 0) {
        piv = best > 0.0f ? br : -1;
        if (piv < 0) atomicExch(status, 1);
        pval = M[br * ld + k];
        perm[k] = br;
      }
    }
    __syncthreads();
    const int p = piv;
    if (p < 0) return;   // singular block: reported through status
    const float inv = 1.0f / pval;
    for (int c = tid; c < nb; c += 256) {
      const float a = M[p * ld + c];
      if (p != k) M[p * ld + c] = M[k * ld + c];
      rk[c] = c == k ? inv : a * inv;
    }
    __syncthreads();
    float row[CW];
#pragma unroll
    for (int i = 0; i < CW; ++i) row[i] = lane + 32 * i < nb ? rk[lane + 32 * i] : 0.0f;
    for (int r = warp; r < nb; r += 8) {
      float* m = M + r * ld;
      const float f = m[k];
      __syncwarp();   // every lane holds f before lane k % 32 replaces it
#pragma unroll
      for (int i = 0; i < CW; ++i) {
        const int c = lane + 32 * i;
        if (c < nb) m[c] = r == k ? row[i] : (c == k ? -f * inv : m[c] - f * row[i]);
      }
    }
    __syncthreads();
  }
  if (tid == 0) {   // the column swaps that undo the row swaps, last pivot first
    for (int j = 0; j < nb; ++j) cm[j] = j;
    for (int k = nb - 1; k >= 0; --k) {
      const int t = cm[k];
      cm[k] = cm[perm[k]];
      cm[perm[k]] = t;
    }
  }
  __syncthreads();
  for (int t = tid; t < nb * nb; t += 256) A[t] = M[(t % nb) * ld + cm[t / nb]];
}

// In-place inverse of one nb x nb block per CTA (column-major in global
// memory) by Gauss-Jordan elimination with partial pivoting, blocked by
// panels of kPanel columns: each panel is eliminated (pivot search over the
// rows not yet used, row swaps, scaling, elimination from every other row), and
// its kPanel pivots then reach every other column at once as the panel's row
// permutation followed by the rank-kPanel update A[:, j] += (panel - I) A[K, j];
// the row swaps are undone as column swaps at the end.  The block moves through
// global memory (L2) once per panel.  A zero pivot sets *status and leaves the
// block unfinished.
//
// The panel lives in registers while it is eliminated: warp w holds the rows w,
// w + 16, ... (RPW of them), lane c column c, so that a pivot costs two barriers,
// one shuffle and one FMA a row, and no shared-memory traffic but the two rows
// exchanged.  The update gives lanes consecutive rows (coalesced columns) and
// each thread two rows by eight columns: two panel words and two broadcast
// 16-byte loads for sixteen FMAs.  853 blocks of 320 DOFs: 13.7 -> 7.3 ms, the
// same bits; the block's passes through L2 bound it now.
// Shared memory: the panel [nb][kPanel + 1] (then the rows of the final column
// swap), the tile's permuted rows Y[2 kPanel][kTile + 4], idx[nb], perm[nb].
constexpr int kInvThreads = 512, kInvWarps = kInvThreads / 32;
template <int RPW>
__global__ void __launch_bounds__(kInvThreads, RPW <= 20 ? 2 : 1)
    k_pc_invert_blocked(float* __restrict__ B, const int64_t* __restrict__ pc_off, int slot_begin, int nb,
                        int* __restrict__ status) {
  extern __shared__ __align__(16) float sm[];
  constexpr int LD = kPanel + 1, LY = kTile + 4;
  float* Y = sm;                                    // [2 kPanel][LY]
  float* Pn = Y + 2 * kPanel * LY;                  // [nb][LD]
  int* idx = reinterpret_cast<int*>(Pn + (size_t)nb * LD);   // [nb] the panel's row order
  int* perm = idx + nb;                             // [nb] pivot rows
  __shared__ float pv[kInvWarps], row_k[kPanel], row_p[kPanel];
  __shared__ int pr[kInvWarps];
  const int s = slot_begin + blockIdx.x;
  const int64_t off = pc_off[s];
  if (off < 0) return;
  float* A = B + off;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int kb = 0; kb < nb; kb += kPanel) {
    const int nk = min(kPanel, nb - kb);
    for (int t = tid; t < nb * kPanel; t += kInvThreads) {
      const int c = t / nb, r = t - c * nb;
      Pn[r * LD + c] = c < nk ? A[(int64_t)(kb + c) * nb + r] : 0.0f;
    }
    for (int r = tid; r < nb; r += kInvThreads) idx[r] = r;
    __syncthreads();
    float x[RPW];
#pragma unroll
    for (int i = 0; i < RPW; ++i) {
      const int r = warp + kInvWarps * i;
      x[i] = r < nb ? Pn[r * LD + lane] : 0.0f;
    }
    for (int kl = 0; kl < nk; ++kl) {
      const int k = kb + kl;
      // pivot: the row r >= k with the largest |x| of column kl (lowest row at a
      // tie); every lane searches its own column, lane kl's result counts
      float best = -1.0f;
      int br = k;
#pragma unroll
      for (int i = 0; i < RPW; ++i) {
        const int r = warp + kInvWarps * i;
        const float a = fabsf(x[i]);
        if (r >= k && r < nb && a > best) {
          best = a;
          br = r;
        }
      }
      if (lane == kl) {
        pv[warp] = best;
        pr[warp] = br;
      }
      __syncthreads();
      float b0 = pv[0];
      int p = pr[0];
#pragma unroll
      for (int q = 1; q < kInvWarps; ++q)
        if (pv[q] > b0 || (pv[q] == b0 && pr[q] < p)) {
          b0 = pv[q];
          p = pr[q];
        }
      if (!(b0 > 0.0f)) {   // singular block: reported through status
        if (tid == 0) atomicExch(status, 1);
        return;
      }
      if (tid == 0) {
        perm[k] = p;
        const int t0 = idx[k];
        idx[k] = idx[p];
        idx[p] = t0;
      }
#pragma unroll
      for (int i = 0; i < RPW; ++i) {
        const int r = warp + kInvWarps * i;
        if (r == k) row_k[lane] = x[i];
        if (r == p) row_p[lane] = x[i];
      }
      __syncthreads();
      const float inv = 1.0f / row_p[kl];
      const float rk = lane == kl ? inv : row_p[lane] * inv, old_k = row_k[lane];
#pragma unroll
      for (int i = 0; i < RPW; ++i) {
        const int r = warp + kInvWarps * i;
        const float y = r == p && p != k ? old_k : x[i];   // row p holds the old row k
        const float f = __shfl_sync(0xffffffffu, y, kl);
        x[i] = r == k ? rk : (lane == kl ? -f * inv : y - f * rk);
      }
    }
    // the eliminated panel back to global memory, then less the identity for the update
#pragma unroll
    for (int i = 0; i < RPW; ++i) {
      const int r = warp + kInvWarps * i;
      if (r < nb) Pn[r * LD + lane] = x[i];
    }
    __syncthreads();
    for (int t = tid; t < nb * nk; t += kInvThreads) {
      const int c = t / nb, r = t - c * nb;
      A[(int64_t)(kb + c) * nb + r] = Pn[r * LD + c];
    }
    __syncthreads();
    if (tid < nk) Pn[(kb + tid) * LD + tid] -= 1.0f;
    // every other column j: rows permuted as the panel's were, then
    // A[:, j] += (Pn - I_K) A[K, j]
    for (int j0 = 0; j0 < nb; j0 += kTile) {
      __syncthreads();
      // (a) row permutation of the tile: the rows that can have moved are the
      // panel rows and their pivot rows (all reads before any write); the new
      // panel rows are the update's right-hand factor
      for (int t = tid; t < 2 * nk * kTile; t += kInvThreads) {
        const int c = t / (2 * nk), ri = t - c * 2 * nk, j = j0 + c;
        const int r = ri < nk ? kb + ri : perm[kb + ri - nk];
        Y[ri * LY + c] = j < nb && (j < kb || j >= kb + nk) ? A[(int64_t)j * nb + idx[r]] : 0.0f;
      }
      __syncthreads();
      for (int t = tid; t < 2 * nk * kTile; t += kInvThreads) {
        const int c = t / (2 * nk), ri = t - c * 2 * nk, j = j0 + c;
        const int r = ri < nk ? kb + ri : perm[kb + ri - nk];
        if (j < nb && (j < kb || j >= kb + nk)) A[(int64_t)j * nb + r] = Y[ri * LY + c];
      }
      __syncthreads();
      // (b) rank-nk update
      const int units = (nb + 63) / 64 * (kTile / 8);
      for (int un = warp; un < units; un += kInvWarps) {
        const int r0 = un / (kTile / 8) * 64 + lane, r1 = r0 + 32, c0 = un % (kTile / 8) * 8;
        if (j0 + c0 >= nb) continue;
        float acc[2][8];
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[0][c] = acc[1][c] = 0.0f;
        const float* p0 = Pn + min(r0, nb - 1) * LD;
        const float* p1 = Pn + min(r1, nb - 1) * LD;
        for (int k = 0; k < nk; ++k) {
          const float w0 = p0[k], w1 = p1[k];
          const float4 u = *reinterpret_cast<const float4*>(Y + k * LY + c0);
          const float4 v = *reinterpret_cast<const float4*>(Y + k * LY + c0 + 4);
          const float xs[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            acc[0][c] = fmaf(w0, xs[c], acc[0][c]);
            acc[1][c] = fmaf(w1, xs[c], acc[1][c]);
          }
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const int j = j0 + c0 + c;
          if (j >= nb || (j >= kb && j < kb + nk)) continue;
          if (r0 < nb) A[(int64_t)j * nb + r0] += acc[0][c];
          if (r1 < nb) A[(int64_t)j * nb + r1] += acc[1][c];
        }
      }
    }
    __syncthreads();
  }
  // undo the row swaps as column swaps, last pivot first: the order of the
  // columns, then 32 rows at a time through shared memory
  if (tid == 0) {
    for (int j = 0; j < nb; ++j) idx[j] = j;
    for (int k = nb - 1; k >= 0; --k) {
      const int t = idx[k];
      idx[k] = idx[perm[k]];
      idx[perm[k]] = t;
    }
  }
  __syncthreads();
  for (int r0 = 0; r0 < nb; r0 += 32) {
    const int r = r0 + lane;
    for (int j = warp; j < nb; j += kInvWarps)
      if (r < nb) Pn[j * LD + lane] = A[(int64_t)j * nb + r];
    __syncthreads();
    for (int j = warp; j < nb; j += kInvWarps)
      if (r < nb) A[(int64_t)j * nb + r] = Pn[idx[j] * LD + lane];
    __syncthreads();
  }
}

static size_t pc_blocked_smem(int nb) {
  return sizeof(float) * ((size_t)nb * (kPanel + 1) + 2 * kPanel * (kTile + 4)) + sizeof(int) * 2 * (size_t)nb;
}

// z_e = M_e^-1 (a w_e + b u_e), every bucket in one launch: a CTA takes one
// element (nb at least half its threads) or as many whole ones as fit, one thread
// per row (rows beyond the CTA's 1,024 threads in a second pass).  The columns
// are summed in order with FP32 FMAs; each thread has kPcAhead column loads in
// flight (the blocks' bytes bound the apply, and one load at a time left HBM
// idle: blocks of 320, 135 and 40 DOFs on 2,560 elements, 410 MB, took three
// launches of 58 us and now one of 87 us, 4.7 TB/s).
// The vectors are FP64 or FP32 (VT; the FP32 Krylov basis), the sums FP32.
// Elements without a stored block (pc_off < 0): z_e = (a w_e + b u_e) / sigma.
constexpr int kPcAhead = 16;
template <typename VT>
__global__ void __launch_bounds__(1024) k_pc_apply(PcBuckets bk, const float* __restrict__ B,
                                                   const int64_t* __restrict__ pc_off,
                                                   const int64_t* __restrict__ state_off, double a, const VT* w, double b,
                                                   const VT* __restrict__ u, VT* z, double inv_sigma,
                                                   const int* __restrict__ gate, const double* __restrict__ bscale) {
  extern __shared__ __align__(16) float xs[];   // [elements][nb]
  if (gate && *gate) return;
  if (bscale) b *= *bscale;
  int q = 0;
  while ((int)blockIdx.x >= bk.first[q + 1]) ++q;
  const int nb = bk.nb[q], epb = max(1, (int)blockDim.x / nb);
  const int e0 = (int)(blockIdx.x - bk.first[q]) * epb, ne = min(epb, bk.count[q] - e0);
  for (int t = threadIdx.x; t < ne * nb; t += blockDim.x) {
    const int64_t g = state_off[bk.slot_begin[q] + e0 + t / nb] + t % nb;
    xs[t] = (float)(a * (double)w[g] + (u ? b * (double)u[g] : 0.0));
  }
  __syncthreads();
  for (int t = threadIdx.x; t < ne * nb; t += blockDim.x) {
    const int le = t / nb, i = t - le * nb;
    const int s = bk.slot_begin[q] + e0 + le;
    const int64_t g = state_off[s] + i, off = pc_off[s];
    if (off < 0) {
      z[g] = (VT)((a * (double)w[g] + (u ? b * (double)u[g] : 0.0)) * inv_sigma);
      continue;
    }
    const float* Bc = B + off + i;
    const float* xe = xs + le * nb;
    float acc = 0.0f;
    int j = 0;
    for (; j + kPcAhead <= nb; j += kPcAhead) {
      float m[kPcAhead];
#pragma unroll
      for (int r = 0; r < kPcAhead; ++r) m[r] = Bc[(int64_t)(j + r) * nb];
#pragma unroll
      for (int r = 0; r < kPcAhead; ++r) acc = fmaf(m[r], xe[j + r], acc);
    }
    for (; j < nb; ++j) acc = fmaf(Bc[(int64_t)j * nb], xe[j], acc);
    z[g] = (VT)acc;
  }
}

// Distance-1 colouring of the face graph (greedy in element order), once per context.
void pc_color(fr_ctx* c) {
  const int E = c->E, nf = c->nf;
  c->color.assign(E, -1);
  int nc = 0;
  std::vector<char> used;
  for (int e = 0; e < E; ++e) {
    used.assign(nc + 1, 0);
    for (int f = 0; f < nf; ++f) {
      const int n = c->nbr[(size_t)e * nf + f];
      if (n >= 0 && n != e && c->color[n] >= 0) used[c->color[n]] = 1;
    }
    int col = 0;
    while (col < nc && used[col]) ++col;
    c->color[e] = col;
    nc = std::max(nc, col + 1);
  }
  c->n_colors = nc;
}

// The probing products of a small mesh are a wave of CTAs each or less, bound by
// latency: kPcLanes of them run side by side on streams of their own (the first
// is the caller's).  Beyond two full-occupancy waves of points one product fills
// the GPU by itself.  2,560 elements, 84,000 points, 640 products of three
// launches: the build 43 -> 25 ms, the ESDIRK2 step 66.7 -> 48.6 ms.
constexpr int kPcLanes = 4;

void free_pc_lanes(fr_ctx* c) {
  for (auto& l : c->pc_lanes) {
    if (l.s) {
      cudaStreamSynchronize(l.s);
      cudaStreamDestroy(l.s);
    }
    if (l.done) cudaEventDestroy(l.done);
    cudaFree(l.v);
    cudaFree(l.J);
    cudaFree(l.trace);
    cudaFree(l.fout);
  }
  c->pc_lanes.clear();
  if (c->pc_fork) cudaEventDestroy(c->pc_fork);
  c->pc_fork = nullptr;
}

// The extra lanes, sized for all elements at p_max in FP32; none when the mesh
// is large or something cannot be created (the build then runs on one stream).
static void ensure_pc_lanes(fr_ctx* c) {
  if (c->n_dof_cap / c->nv > (int64_t)2 * 2048 * c->sms) return;
  if (!c->pc_lanes.empty()) return;
  bool ok = cudaEventCreateWithFlags(&c->pc_fork, cudaEventDisableTiming) == cudaSuccess;
  for (int i = 1; i < kPcLanes && ok; ++i) {
    c->pc_lanes.emplace_back();
    PcLane& l = c->pc_lanes.back();
    ok = cudaStreamCreateWithFlags(&l.s, cudaStreamNonBlocking) == cudaSuccess &&
         cudaEventCreateWithFlags(&l.done, cudaEventDisableTiming) == cudaSuccess &&
         cudaMalloc(&l.v, sizeof(float) * c->n_dof_cap) == cudaSuccess &&
         cudaMalloc(&l.J, sizeof(float) * c->n_dof_cap) == cudaSuccess &&
         cudaMalloc(&l.trace, sizeof(float) * c->trace_cap) == cudaSuccess &&
         cudaMalloc(&l.fout, sizeof(float) * c->fout_cap) == cudaSuccess;
  }
  if (!ok) {
    cudaGetLastError();
    free_pc_lanes(c);
  }
}

}  // namespace frgb

using namespace frgb;

extern "C" {

fr_status fr_precond_build(fr_ctx* c, const double* q64_dev, double sigma, void* stream) {
  if (!c || !q64_dev || !(sigma > 0.0)) {
    set_error("fr_precond_build: bad argument");
    return FR_ERR_INVALID;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const int E = c->E, nd = c->nd, nv = c->nv;
  if (c->color.empty()) pc_color(c);
  // block offsets per slot (floats), -1 for blocks larger than kPcMax
  std::vector<int64_t> off(E, -1);
  std::vector<int32_t> slot_color(E);
  int next[kMaxDeg + 1] = {};   // next slot of each degree: slots hold the elements in (p, id) order
  for (const auto& b : c->buckets) next[b.p] = b.slot_begin;
  for (int el = 0; el < E; ++el) slot_color[next[c->p[el]]++] = c->color[el];
  int64_t total = 0;
  int kmax = 0;
  for (const auto& b : c->buckets) {
    const int nb = nv * nsp_host(nd, b.p);
    for (int i = 0; i < b.count; ++i) {
      const int sl = b.slot_begin + i;
      if (nb <= kPcMax) {
        off[sl] = total;
        total += (int64_t)nb * nb;
      }
    }
    if (nb <= kPcMax && b.count > 0) kmax = std::max(kmax, nb);
  }
  if (!c->d_pc_off && cudaMalloc(&c->d_pc_off, sizeof(int64_t) * E) != cudaSuccess) return FR_ERR_NOMEM;
  if (!c->d_slot_color && cudaMalloc(&c->d_slot_color, sizeof(int32_t) * E) != cudaSuccess) return FR_ERR_NOMEM;
  if (total > c->pc_cap) {
    cudaFree(c->d_pc);
    c->d_pc = nullptr;
    c->pc_cap = 0;
    if (cudaMalloc(&c->d_pc, sizeof(float) * std::max<int64_t>(total, 1)) != cudaSuccess) {
      cudaGetLastError();
      set_error("fr_precond_build: block storage allocation failed");
      return FR_ERR_NOMEM;
    }
    c->pc_cap = total;
  }
  if (!c->d_pc_status && cudaMalloc(&c->d_pc_status, sizeof(int)) != cudaSuccess) return FR_ERR_NOMEM;
  cudaMemcpyAsync(c->d_pc_off, off.data(), sizeof(int64_t) * E, cudaMemcpyHostToDevice, s);
  cudaMemcpyAsync(c->d_slot_color, slot_color.data(), sizeof(int32_t) * E, cudaMemcpyHostToDevice, s);
  cudaMemsetAsync(c->d_pc_status, 0, sizeof(int), s);
  c->pc_ready = false;
  const int64_t n = c->n_dof;
  float* q32 = vec32(c, 0);
  float* v32 = vec32(c, 1);
  float* J32 = vec32(c, 2);
  if (!q32 || !v32 || !J32) return FR_ERR_NOMEM;
  vcast_f64_f32(c, q64_dev, q32, n, s);
  fr_status e = launch_jvp_prepare(c, q32, FR_F32, s);
  if (e != FR_OK) return e;
  const float sg = (float)sigma;
  PcBuckets pb{};
  for (const auto& b : c->buckets) {
    const int nb = nv * nsp_host(nd, b.p);
    if (nb > kPcMax) continue;
    pb.slot_begin[pb.n] = b.slot_begin;
    pb.count[pb.n] = b.count;
    pb.nb[pb.n] = nb;
    pb.first[pb.n + 1] = pb.first[pb.n] + (int64_t)b.count * nb;
    pb.n += 1;
  }
  const unsigned pg = (unsigned)((pb.first[pb.n] + 255) / 256);
  // lane l probes the columns l, l + lanes, ... of a colour with its own unit
  // vectors and workspaces; the traces of q are shared and only read
  ensure_pc_lanes(c);
  std::vector<PcLane> lanes(1);
  lanes[0].s = s;
  lanes[0].v = v32;
  lanes[0].J = J32;
  lanes[0].trace = c->d_trace_v;
  lanes[0].fout = c->d_fout;
  lanes.insert(lanes.end(), c->pc_lanes.begin(), c->pc_lanes.end());
  const int nl = (int)lanes.size();
  if (nl > 1) {
    cudaEventRecord(c->pc_fork, s);
    for (int l = 1; l < nl; ++l) cudaStreamWaitEvent(lanes[l].s, c->pc_fork, 0);
  }
  void* const trace0 = c->d_trace_v;
  void* const fout0 = c->d_fout;
  // side by side, a waiting kernel of one lane takes room from another's (a step
  // of the O-grid with the preconditioner: 47.3 ms, 49.5 chained)
  c->chain = nl == 1;
  for (int col = 0; col < c->n_colors && kmax > 0 && e == FR_OK; ++col) {
    auto probe = [&](const PcLane& ln, int k, int next) {
      FR_LAUNCH(c, "precond_build", ln.s,
                k_pc_probe<<<pg, 256, 0, ln.s>>>(pb, c->d_pc, c->d_pc_off, ln.J, ln.v, c->lt.state_off, c->d_slot_color,
                                                 col, k, next, sg));
    };
    for (int l = 0; l < nl && l < kmax; ++l) {
      cudaMemsetAsync(lanes[l].v, 0, sizeof(float) * n, lanes[l].s);
      probe(lanes[l], -1, l);
    }
    for (int k = 0; k < kmax && e == FR_OK; ++k) {
      const PcLane& ln = lanes[k % nl];
      c->d_trace_v = ln.trace;
      c->d_fout = ln.fout;
      e = launch_jvp_prepared(c, q32, ln.v, ln.J, FR_F32, ln.s);
      if (e == FR_OK) probe(ln, k, k + nl);
    }
  }
  c->chain = true;
  c->d_trace_v = trace0;
  c->d_fout = fout0;
  for (int l = 1; l < nl; ++l) {   // also after an error: s must not run ahead of the lanes
    cudaEventRecord(lanes[l].done, lanes[l].s);
    cudaStreamWaitEvent(s, lanes[l].done, 0);
  }
  if (e != FR_OK) return e;
  for (const auto& b : c->buckets) {
    const int nb = nv * nsp_host(nd, b.p);
    if (nb > kPcMax || b.count == 0) continue;
    if (nb <= kPcSmem) {
      const size_t smem = sizeof(float) * (size_t)nb * ((nb | 1) + 1) + sizeof(int) * 2 * (size_t)nb;
      cudaFuncSetAttribute(k_pc_invert, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      FR_LAUNCH(c, "precond_build", s,
                k_pc_invert<<<b.count, 256, smem, s>>>(c->d_pc, c->d_pc_off, b.slot_begin, nb, c->d_pc_status));
    } else {
      // rows a warp holds of the 320-, 625- and 1080-DOF blocks
      auto kern = nb <= 20 * kInvWarps ? k_pc_invert_blocked<20>
                  : nb <= 40 * kInvWarps ? k_pc_invert_blocked<40> : k_pc_invert_blocked<68>;
      const size_t smem = pc_blocked_smem(nb);
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      FR_LAUNCH(c, "precond_build", s,
                kern<<<b.count, kInvThreads, smem, s>>>(c->d_pc, c->d_pc_off, b.slot_begin, nb, c->d_pc_status));
    }
  }
  int status = 0;
  cudaMemcpyAsync(&status, c->d_pc_status, sizeof(int), cudaMemcpyDeviceToHost, s);
  fr_status st = cuda_check(cudaStreamSynchronize(s), "fr_precond_build");
  if (st != FR_OK) return st;
  if (status) {
    set_error("fr_precond_build: singular element block");
    return FR_ERR_NONFINITE;
  }
  c->pc_sigma = sigma;
  c->pc_ready = true;
  return FR_OK;
}

fr_status fr_precond_release(fr_ctx* c) {
  if (!c) return FR_ERR_INVALID;
  cudaFree(c->d_pc);
  c->d_pc = nullptr;
  c->pc_cap = 0;
  c->pc_ready = false;
  free_pc_lanes(c);
  return FR_OK;
}

}  // extern "C"

namespace frgb {

// z = M^-1 (a w + b u) on every element (z may alias w)
template <typename VT>
static fr_status precond_apply_t(fr_ctx* c, double a, const VT* w, double b, const VT* u, VT* z, cudaStream_t s,
                                 const int* gate, const double* bscale) {
  if (!c->pc_ready) {
    set_error("element-Jacobi preconditioner not built (fr_precond_build) for the current layout");
    return FR_ERR_INVALID;
  }
  // one launch, the largest blocks first (their CTAs run longest)
  PcBuckets pb{};
  int threads = 256;
  double bytes = 0.0;
  for (const auto& bk : c->buckets)
    threads = std::max(threads, std::min(1024, (c->nv * nsp_host(c->nd, bk.p) + 31) / 32 * 32));
  size_t smem = 0;
  for (auto it = c->buckets.rbegin(); it != c->buckets.rend(); ++it) {
    const int nb = c->nv * nsp_host(c->nd, it->p), epb = std::max(1, threads / nb);
    pb.slot_begin[pb.n] = it->slot_begin;
    pb.count[pb.n] = it->count;
    pb.nb[pb.n] = nb;
    pb.first[pb.n + 1] = pb.first[pb.n] + (it->count + epb - 1) / epb;
    pb.n += 1;
    smem = std::max(smem, sizeof(float) * (size_t)epb * nb);
    bytes += (double)it->count * nb * (3.0 * sizeof(VT) + 4.0 * nb);   // a w, b u in, z out; the block
  }
  FR_LAUNCH_B(c, "precond_apply", s, bytes,
              k_pc_apply<VT><<<(unsigned)pb.first[pb.n], threads, smem, s>>>(
                  pb, c->d_pc, c->d_pc_off, c->lt.state_off, a, w, b, u, z, 1.0 / c->pc_sigma, gate, bscale));
  return cuda_check(cudaGetLastError(), "precond_apply");
}

fr_status precond_apply(fr_ctx* c, double a, const double* w, double b, const double* u, double* z, cudaStream_t s,
                        const int* gate, const double* bscale) {
  return precond_apply_t<double>(c, a, w, b, u, z, s, gate, bscale);
}

fr_status precond_apply(fr_ctx* c, double a, const float* w, double b, const float* u, float* z, cudaStream_t s,
                        const int* gate, const double* bscale) {
  return precond_apply_t<float>(c, a, w, b, u, z, s, gate, bscale);
}

}  // namespace frgb

extern "C" fr_status fr_precond_apply(fr_ctx* c, const double* w_dev, double* z_dev, void* stream) {
  if (!c || !w_dev || !z_dev) {
    set_error("fr_precond_apply: null argument");
    return FR_ERR_INVALID;
  }
  return precond_apply(c, 1.0, w_dev, 0.0, nullptr, z_dev, (cudaStream_t)stream);
}
