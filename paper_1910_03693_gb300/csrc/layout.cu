// The layout of a set of element degrees, built on the device: the stable
// counting sort of the elements into (p, id) buckets (Sec. 3.2's repartition
// on one GPU), the per-slot offset tables, the face records grouped by degree
// pair and direction, the boundary records by degree and kind, the neighbour
// table of the fused JVP and the tile table of the multi-bucket launches.
//
// The degrees stay on the device; the host reads back one block of counts
// (elements per degree, faces per group) and the degrees themselves, from
// which it forms the buckets and groups.  Every buffer has its size from the
// mesh alone (each interior face has one record, whatever the degrees), so
// nothing is allocated when the degrees change.  Built on the host, with the
// records' vectors, uploads and one allocation and free a group, one adaptation
// of 8,000 hexahedra with its way back (two changes of degrees) took 2.96 ms;
// it takes 0.43 ms, 0.33 ms of it in kernels.
#include <algorithm>
#include <cstring>
#include <vector>

#include "fr_launch.h"

namespace frgb {

constexpr int kND = kMaxDeg + 1;             // entries of a per-degree table (index p)
constexpr int kSortBlock = 1024;             // elements of one block of the counting sort
constexpr int kFaceBlock = 256;              // element faces of one block of the face sort
// face keys: degree pair (pm, ps) then the master face's direction (the
// diagonal-metric face kernel branches on it), then boundary degree and kind
constexpr int kPairKeys = kMaxDeg * kMaxDeg * 3;
constexpr int kFaceKeys = kPairKeys + 2 * kMaxDeg;

// What the host reads back.
struct LayoutMeta {
  int64_t n_dof;
  int32_t count[kND];        // elements of degree p
  int32_t faces[kFaceKeys];
};

__host__ __device__ inline int pw(int b, int e) {
  int r = 1;
  while (e-- > 0) r *= b;
  return r;
}

// per-degree bases of the slots, states, traces and face outputs
struct Bases {
  int first[kND];
  int64_t state[kND], trace[kND], out[kND];
};

__host__ __device__ inline void bases_of(const int32_t* count, int nd, int nv, int nf, int nvt, Bases& b) {
  int slot = 0;
  int64_t st = 0, tr = 0, ou = 0;
  for (int p = 0; p < kND; ++p) {
    b.first[p] = slot;
    b.state[p] = st;
    b.trace[p] = tr;
    b.out[p] = ou;
    const int64_t n = count[p];
    slot += count[p];
    st += n * nv * pw(p + 1, nd);
    tr += n * nf * nvt * pw(p + 1, nd - 1);
    ou += n * nf * 3 * nv * pw(p + 1, nd - 1);
  }
}

// per-block counts of each degree
__global__ void k_sort_count(const int8_t* __restrict__ p, int E, int* __restrict__ blk_counts) {
  __shared__ int cnt[kND];
  if (threadIdx.x < kND) cnt[threadIdx.x] = 0;
  __syncthreads();
  const int e = blockIdx.x * kSortBlock + threadIdx.x;
  if (e < E) atomicAdd(&cnt[p[e]], 1);
  __syncthreads();
  if (threadIdx.x < kND) blk_counts[blockIdx.x * kND + threadIdx.x] = cnt[threadIdx.x];
}

// blk_off[b][p] = first slot of degree p + elements of degree p in earlier
// blocks; blk_canon[b] = canonical values of earlier blocks.  One warp a degree
// (and one for the canonical offsets) walks the blocks 32 at a time.
__global__ void __launch_bounds__(32 * (kND + 1)) k_sort_scan(const int* __restrict__ blk_counts, int nb, int nd, int nv,
                                                             int* __restrict__ blk_off, int64_t* __restrict__ blk_canon,
                                                             LayoutMeta* __restrict__ meta) {
  __shared__ int tot[kND];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (w < kND) {
    int n = 0;
    for (int b = lane; b < nb; b += 32) n += blk_counts[b * kND + w];
    for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
    if (lane == 0) tot[w] = n;
  }
  __syncthreads();
  int64_t run = 0;
  if (w < kND)
    for (int q = 0; q < w; ++q) run += tot[q];
  for (int b0 = 0; b0 < nb; b0 += 32) {
    const int b = b0 + lane;
    int64_t v = 0;
    if (b < nb) {
      if (w < kND) {
        v = blk_counts[b * kND + w];
      } else {
        for (int q = 0; q < kND; ++q) v += (int64_t)blk_counts[b * kND + q] * nv * pw(q + 1, nd);
      }
    }
    int64_t inc = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (b < nb) {
      if (w < kND) blk_off[b * kND + w] = (int)(run + inc - v);
      else blk_canon[b] = run + inc - v;
    }
    run += __shfl_sync(0xffffffffu, inc, 31);
  }
  if (lane == 0) {
    if (w < kND) meta->count[w] = tot[w];
    else meta->n_dof = run;
  }
}

// slots (stable: in element order within a degree) and the per-slot tables
__global__ void __launch_bounds__(kSortBlock) k_sort_scatter(const int8_t* __restrict__ p, int E, int nd, int nv,
                                                           const int* __restrict__ blk_off,
                                                           const int64_t* __restrict__ blk_canon,
                                                           const LayoutMeta* __restrict__ meta,
                                                           int32_t* __restrict__ slot_elem, int32_t* __restrict__ elem_slot,
                                                           int8_t* __restrict__ slot_p, int64_t* __restrict__ state_off,
                                                           int64_t* __restrict__ canon_off) {
  __shared__ int warp_cnt[kSortBlock / 32][kND];
  __shared__ int warp_val[kSortBlock / 32];
  __shared__ Bases bs;
  if (threadIdx.x == 0) bases_of(meta->count, nd, nv, 1, 1, bs);
  const int e = blockIdx.x * kSortBlock + threadIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int pe = e < E ? p[e] : -1;
  const int size = pe < 0 ? 0 : nv * pw(pe + 1, nd);
  int rank_in_warp = 0;
  for (int pp = 0; pp < kND; ++pp) {
    const unsigned m = __ballot_sync(0xffffffffu, pe == pp);
    if (pe == pp) rank_in_warp = __popc(m & ((1u << lane) - 1u));
    if (lane == 0) warp_cnt[warp][pp] = __popc(m);
  }
  int inc = size;   // canonical values before this element within the warp (inclusive)
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) warp_val[warp] = inc;
  __syncthreads();
  if (e >= E) return;
  int before = 0, vals = inc - size;
  for (int w = 0; w < warp; ++w) {
    before += warp_cnt[w][pe];
    vals += warp_val[w];
  }
  const int slot = blk_off[blockIdx.x * kND + pe] + before + rank_in_warp;
  slot_elem[slot] = e;
  elem_slot[e] = slot;
  slot_p[slot] = (int8_t)pe;
  state_off[slot] = bs.state[pe] + (int64_t)(slot - bs.first[pe]) * size;
  canon_off[slot] = blk_canon[blockIdx.x] + vals;
}

struct FaceMesh {
  const int32_t* nbr;        // [E][nf]
  const int8_t* nbr_face;
  const int8_t* orient;
  const int8_t* p;
  int E, nf, nd, nv, nvt;
};

// the sort key of element face id = e nf + f: the master of an interior face
// (higher degree; ties: lower element id, then lower face) and boundary faces
// have one, the slave side -1
__device__ __forceinline__ int face_key(const FaceMesh& m, int64_t id) {
  const int e = (int)(id / m.nf), f = (int)(id % m.nf);
  const int n = m.nbr[id], pe = m.p[e];
  if (n < 0) return kPairKeys + (pe - 1) * 2 + (n == FR_BC_FARFIELD ? 0 : 1);
  const int g = m.nbr_face[id], pn = m.p[n];
  if (!(pe > pn || (pe == pn && (e < n || (e == n && f < g))))) return -1;
  return ((pe - 1) * kMaxDeg + (pn - 1)) * 3 + (f >> 1);
}

// faces of every key in each block: hist[key][block]
__global__ void __launch_bounds__(kFaceBlock) k_face_count(FaceMesh m, int nfb, int* __restrict__ hist) {
  __shared__ int cnt[kFaceKeys];
  for (int k = threadIdx.x; k < kFaceKeys; k += kFaceBlock) cnt[k] = 0;
  __syncthreads();
  const int64_t id = (int64_t)blockIdx.x * kFaceBlock + threadIdx.x;
  if (id < (int64_t)m.E * m.nf) {
    const int k = face_key(m, id);
    if (k >= 0) atomicAdd(&cnt[k], 1);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < kFaceKeys; k += kFaceBlock) hist[(int64_t)k * nfb + blockIdx.x] = cnt[k];
}

// one warp a key: exclusive prefix over the blocks in place, the key's total
__global__ void __launch_bounds__(32) k_face_scan(int* __restrict__ hist, int nfb, LayoutMeta* __restrict__ meta) {
  int* h = hist + (int64_t)blockIdx.x * nfb;
  const int lane = threadIdx.x;
  int run = 0;
  for (int b0 = 0; b0 < nfb; b0 += 32) {
    const int b = b0 + lane;
    const int v = b < nfb ? h[b] : 0;
    int inc = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (b < nfb) h[b] = run + inc - v;
    run += __shfl_sync(0xffffffffu, inc, 31);
  }
  if (lane == 0) meta->faces[blockIdx.x] = run;
}

// the records in key order, stable in (element, face) within a key
__global__ void __launch_bounds__(kFaceBlock) k_face_scatter(FaceMesh m, int nfb, const int* __restrict__ hist,
                                                           const LayoutMeta* __restrict__ meta,
                                                           const int32_t* __restrict__ elem_slot,
                                                           FaceRec* __restrict__ recs, BndRec* __restrict__ brecs) {
  __shared__ int base[kFaceKeys];
  __shared__ int wc[kFaceBlock / 32][kFaceKeys];
  __shared__ Bases bs;
  if (threadIdx.x == 0) bases_of(meta->count, m.nd, m.nv, m.nf, m.nvt, bs);
  if (threadIdx.x < kFaceKeys) {   // boundary records are an array of their own
    const int k0 = threadIdx.x < kPairKeys ? 0 : kPairKeys;
    int n = 0;
    for (int k = k0; k < (int)threadIdx.x; ++k) n += meta->faces[k];
    base[threadIdx.x] = n;
  }
  for (int k = threadIdx.x; k < (kFaceBlock / 32) * kFaceKeys; k += kFaceBlock) (&wc[0][0])[k] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t id = (int64_t)blockIdx.x * kFaceBlock + threadIdx.x;
  const int key = id < (int64_t)m.E * m.nf ? face_key(m, id) : -1;
  const unsigned same = __match_any_sync(0xffffffffu, key);
  const int rank = __popc(same & ((1u << lane) - 1u));
  if (key >= 0 && rank == 0) wc[warp][key] = __popc(same);
  __syncthreads();
  if (key < 0) return;
  int pos = base[key] + hist[(int64_t)key * nfb + blockIdx.x] + rank;
  for (int w = 0; w < warp; ++w) pos += wc[w][key];
  const int e = (int)(id / m.nf), f = (int)(id % m.nf);
  const int pe = m.p[e], ie = elem_slot[e] - bs.first[pe], nfe = pw(pe + 1, m.nd - 1);
  const int64_t mt = bs.trace[pe] + ((int64_t)ie * m.nf + f) * m.nvt * nfe;
  const int64_t mo = bs.out[pe] + ((int64_t)ie * m.nf + f) * 3 * m.nv * nfe;
  const int n = m.nbr[id];
  if (n < 0) {
    brecs[pos] = BndRec{mt, mo, e, f};
    return;
  }
  const int g = m.nbr_face[id], pn = m.p[n], in = elem_slot[n] - bs.first[pn], nfn = pw(pn + 1, m.nd - 1);
  FaceRec r;
  r.mt = mt;
  r.mo = mo;
  r.st = bs.trace[pn] + ((int64_t)in * m.nf + g) * m.nvt * nfn;
  r.so = bs.out[pn] + ((int64_t)in * m.nf + g) * 3 * m.nv * nfn;
  r.me = e;
  r.se = n;
  r.mf = f;
  r.sf = g;
  r.orient = m.orient[id];
  r.pad = 0;
  recs[pos] = r;
}

// neighbour of every element face for the fused JVP (meshes without boundary
// faces; used only while every face is conforming)
__global__ void k_fused_table(FaceMesh m, const LayoutMeta* __restrict__ meta, const int32_t* __restrict__ slot_elem,
                              const int32_t* __restrict__ elem_slot, FusedNbr* __restrict__ out) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)m.E * m.nf) return;
  const int e = slot_elem[t / m.nf], f = (int)(t % m.nf);
  const int64_t id = (int64_t)e * m.nf + f;
  const int n = m.nbr[id], g = m.nbr_face[id], pn = m.p[n];
  int first = 0;
  for (int q = 0; q < pn; ++q) first += meta->count[q];
  FusedNbr r;
  r.nloc = elem_slot[n] - first;
  r.nelem = n;
  r.g = g;
  r.code = (int32_t)(uint8_t)m.orient[id] | ((e < n || (e == n && f < g)) ? 256 : 0);
  out[t] = r;
}

// Tile table of the multi-bucket launches: runs of equal-weight tiles of one
// bucket (its full tiles; its ragged last one), in the order given.
struct WorkRun {
  int bucket, first, step, start, n;
};
struct WorkRuns {
  WorkRun r[2 * kND];
  int n;
};
__global__ void k_work_fill(WorkRuns w, WorkItem* __restrict__ items) {
  for (int i = 0; i < w.n; ++i)
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < w.r[i].n; t += gridDim.x * blockDim.x)
      items[w.r[i].start + t] = WorkItem{w.r[i].bucket, w.r[i].first + t * w.r[i].step};
}

// Tiles of epb_multi elements, ordered by decreasing element weight per tile
// (higher degrees first), bucket order kept among equal weights.
fr_status rebuild_work_table(fr_ctx* c, cudaStream_t s) {
  c->n_work = 0;
  if (!c->d_work || c->buckets.size() < 2) return FR_OK;
  std::vector<std::pair<double, WorkRun>> runs;
  for (size_t bi = 0; bi < c->buckets.size(); ++bi) {
    const Bucket& b = c->buckets[bi];
    const int P = b.p + 1, e = epb_multi(c->nd, P, tile_threads(c));
    const double w = element_weight(c->epb_tab[0][0][1], pw(P, c->nd), P);
    const int full = b.count / e, rest = b.count % e;
    if (full) runs.push_back({e * w, WorkRun{(int)bi, 0, e, 0, full}});
    if (rest) runs.push_back({rest * w, WorkRun{(int)bi, full * e, e, 0, 1}});
  }
  std::stable_sort(runs.begin(), runs.end(), [](const auto& x, const auto& y) { return x.first > y.first; });
  WorkRuns h{};
  int n = 0;
  for (auto& r : runs) {
    r.second.start = n;
    n += r.second.n;
    h.r[h.n++] = r.second;
  }
  k_work_fill<<<(unsigned)std::min(256, (n + 255) / 256), 256, 0, s>>>(h, c->d_work);
  const fr_status st = cuda_check(cudaGetLastError(), "work table");
  if (st == FR_OK) c->n_work = n;
  return st;
}

template <typename T>
static bool get(T** p, size_t bytes) {
  return cudaMalloc((void**)p, std::max<size_t>(bytes, 1)) == cudaSuccess;
}

void layout_free(LayoutTables& t) {
  cudaFree(t.block);
  t = LayoutTables{};
}

// One set of tables in one allocation.
static bool tables_alloc(fr_ctx* c, LayoutTables& t, bool fnbr) {
  const size_t E = c->E;
  size_t inner = 0, bnd = 0;
  for (int32_t n : c->nbr) (n >= 0 ? inner : bnd) += 1;
  const size_t size[8] = {sizeof(int32_t) * E, sizeof(int32_t) * E, sizeof(int64_t) * E, sizeof(int64_t) * E, E,
                          sizeof(FaceRec) * (inner / 2), sizeof(BndRec) * bnd, fnbr ? sizeof(FusedNbr) * E * c->nf : 0};
  size_t at[8], end = 0;
  for (int i = 0; i < 8; ++i) {
    at[i] = end;
    end += (size[i] + 255) / 256 * 256;
  }
  if (!get(&t.block, end)) {
    cudaGetLastError();
    t.block = nullptr;
    return false;
  }
  char* p = static_cast<char*>(t.block);
  t.slot_elem = reinterpret_cast<int32_t*>(p + at[0]);
  t.elem_slot = reinterpret_cast<int32_t*>(p + at[1]);
  t.canon_off = reinterpret_cast<int64_t*>(p + at[2]);
  t.state_off = reinterpret_cast<int64_t*>(p + at[3]);
  t.slot_p = reinterpret_cast<int8_t*>(p + at[4]);
  t.recs = reinterpret_cast<FaceRec*>(p + at[5]);
  t.brecs = reinterpret_cast<BndRec*>(p + at[6]);
  t.fnbr = fnbr ? reinterpret_cast<FusedNbr*>(p + at[7]) : nullptr;
  return true;
}

// Buffers whose size the mesh decides, and the pinned mirror of what the host reads.
fr_status layout_alloc(fr_ctx* c) {
  const int64_t E = c->E, ef = E * c->nf;
  const int nb = (int)((E + kSortBlock - 1) / kSortBlock), nfb = (int)((ef + kFaceBlock - 1) / kFaceBlock);
  // a mesh without boundary faces gets the neighbour table too; without the
  // memory for it the fused JVP is not offered
  const bool closed = std::all_of(c->nbr.begin(), c->nbr.end(), [](int32_t n) { return n >= 0; });
  const bool ok = ((closed && tables_alloc(c, c->lt, true)) || tables_alloc(c, c->lt, false)) && get(&c->d_p, E) &&
                  get(&c->d_nbr_face, ef) && get(&c->d_orient, ef) &&
                  get(&c->d_lay, sizeof(LayoutMeta) + sizeof(int64_t) * nb + sizeof(int) * 2 * nb * kND) &&
                  get(&c->d_face_hist, sizeof(int) * (size_t)kFaceKeys * nfb) &&
                  cudaMallocHost(&c->h_lay, sizeof(LayoutMeta) + E) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    set_error("layout tables: allocation failed");
    return FR_ERR_NOMEM;
  }
  if (!get(&c->d_work, sizeof(WorkItem) * (E + 2 * kND))) {    // launches then go per bucket
    cudaGetLastError();
    c->d_work = nullptr;
  }
  // a context whose degrees can change gets the second set at once (60 us of the
  // first adaptation of 8,000 hexahedra), else the first rebucketing allocates it
  if (c->p_min < c->p_max) layout_spare(c);
  cudaMemcpy(c->d_nbr_face, c->nbr_face.data(), ef, cudaMemcpyHostToDevice);
  cudaMemcpy(c->d_orient, c->orient.data(), ef, cudaMemcpyHostToDevice);
  cudaMemcpy(c->d_p, c->p.data(), E, cudaMemcpyHostToDevice);
  return cuda_check(cudaGetLastError(), "layout tables");
}

// The second set of tables, once.
fr_status layout_spare(fr_ctx* c) {
  if (c->lt_spare.block || tables_alloc(c, c->lt_spare, c->lt.fnbr != nullptr)) return FR_OK;
  set_error("layout tables: allocation failed");
  return FR_ERR_NOMEM;
}

const int64_t* layout_n_dof(const fr_ctx* c) { return &static_cast<const LayoutMeta*>(c->d_lay)->n_dof; }

// Every device table of the layout of the degrees d_p (element order) into t,
// queued on s, and the copies the host needs.
fr_status layout_device(fr_ctx* c, const int8_t* d_p, const LayoutTables& t, cudaStream_t s) {
  const int E = c->E, nf = c->nf;
  const int64_t ef = (int64_t)E * nf;
  const int nb = (E + kSortBlock - 1) / kSortBlock, nfb = (int)((ef + kFaceBlock - 1) / kFaceBlock);
  LayoutMeta* meta = static_cast<LayoutMeta*>(c->d_lay);
  int64_t* blk_canon = reinterpret_cast<int64_t*>(meta + 1);
  int* blk_counts = reinterpret_cast<int*>(blk_canon + nb);
  int* blk_off = blk_counts + nb * kND;
  FaceMesh m{c->d_nbr, c->d_nbr_face, c->d_orient, d_p, E, nf, c->nd, c->nv, c->nvt};
  FR_LAUNCH(c, "rebucket", s, k_sort_count<<<nb, kSortBlock, 0, s>>>(d_p, E, blk_counts));
  FR_LAUNCH(c, "rebucket", s,
            k_sort_scan<<<1, 32 * (kND + 1), 0, s>>>(blk_counts, nb, c->nd, c->nv, blk_off, blk_canon, meta));
  FR_LAUNCH(c, "rebucket", s,
            k_sort_scatter<<<nb, kSortBlock, 0, s>>>(d_p, E, c->nd, c->nv, blk_off, blk_canon, meta, t.slot_elem,
                                                     t.elem_slot, t.slot_p, t.state_off, t.canon_off));
  FR_LAUNCH(c, "rebucket", s, k_face_count<<<nfb, kFaceBlock, 0, s>>>(m, nfb, c->d_face_hist));
  FR_LAUNCH(c, "rebucket", s, k_face_scan<<<kFaceKeys, 32, 0, s>>>(c->d_face_hist, nfb, meta));
  FR_LAUNCH(c, "rebucket", s,
            k_face_scatter<<<nfb, kFaceBlock, 0, s>>>(m, nfb, c->d_face_hist, meta, t.elem_slot, t.recs, t.brecs));
  if (t.fnbr)
    FR_LAUNCH(c, "rebucket", s,
              k_fused_table<<<(unsigned)((ef + 255) / 256), 256, 0, s>>>(m, meta, t.slot_elem, t.elem_slot, t.fnbr));
  cudaMemcpyAsync(c->h_lay, meta, sizeof(LayoutMeta), cudaMemcpyDeviceToHost, s);
  cudaMemcpyAsync(static_cast<char*>(c->h_lay) + sizeof(LayoutMeta), d_p, E, cudaMemcpyDeviceToHost, s);
  return cuda_check(cudaGetLastError(), "layout");
}

// The new degrees read back by layout_device (valid once its stream is synchronised).
const int8_t* layout_degrees(const fr_ctx* c) {
  return reinterpret_cast<const int8_t*>(static_cast<const char*>(c->h_lay) + sizeof(LayoutMeta));
}

// Buckets and face groups from the counts, once layout_device's stream is
// synchronised; drops what the old layout's pointers and offsets went into.
fr_status layout_host(fr_ctx* c, cudaStream_t s) {
  const LayoutMeta& m = *static_cast<const LayoutMeta*>(c->h_lay);
  const int nd = c->nd, nv = c->nv, nf = c->nf;
  c->pc_ready = false;
  clear_graphs(c);
  Bases bs;
  bases_of(m.count, nd, nv, nf, c->nvt, bs);
  c->buckets.clear();
  c->fgroups.clear();
  c->bgroups.clear();
  const int ct = c->visc ? 2 * nv : nv;
  int64_t cb = 0;
  for (int p = 0; p < kND; ++p) {
    if (m.count[p] == 0) continue;
    Bucket b;
    b.p = p;
    b.count = m.count[p];
    b.slot_begin = bs.first[p];
    b.state_base = bs.state[p];
    b.trace_base = bs.trace[p];
    b.out_base = bs.out[p];
    b.ctrace_base = cb;
    cb += (int64_t)b.count * nf * ct * pw(p + 1, nd - 1);
    c->buckets.push_back(b);
  }
  c->n_dof = m.n_dof;
  int at = 0;
  bool conforming = true;
  for (int k = 0; k < kPairKeys; k += 3) {
    const int n = m.faces[k] + m.faces[k + 1] + m.faces[k + 2];
    if (n == 0) continue;
    FaceGroup g;
    g.pm = k / 3 / kMaxDeg + 1;
    g.ps = k / 3 % kMaxDeg + 1;
    g.n = n;
    g.d_recs = c->lt.recs + at;
    at += n;
    conforming = conforming && g.pm == g.ps;
    c->fgroups.push_back(g);
  }
  at = 0;
  for (int k = 0; k < 2 * kMaxDeg; ++k) {
    const int n = m.faces[kPairKeys + k];
    if (n == 0) continue;
    BndGroup g;
    g.p = k / 2 + 1;
    g.kind = k % 2 == 0 ? FR_BC_FARFIELD : FR_BC_WALL;
    g.n = n;
    g.d_recs = c->lt.brecs + at;
    at += n;
    c->bgroups.push_back(g);
  }
  // the compact face kernel finds a block at the trace-gradient offset scaled
  // by ct / nvt: true when every bucket's compact base is its trace base so scaled
  c->fused_ok = c->lt.fnbr && c->bgroups.empty() && conforming && cb <= c->trace_cap;
  for (const auto& b : c->buckets)
    if (b.trace_base % c->nvt != 0 || b.trace_base / c->nvt * ct != b.ctrace_base) c->fused_ok = false;
  rebuild_work_table(c, s);   // a failure leaves no table: launches go per bucket
  return FR_OK;
}

// The layout of the degrees in d_p, complete on return (context creation).
fr_status build_layout(fr_ctx* c) {
  fr_status st = layout_device(c, c->d_p, c->lt, nullptr);
  if (st == FR_OK) st = cuda_check(cudaStreamSynchronize(nullptr), "layout");
  if (st == FR_OK) st = layout_host(c, nullptr);
  if (st == FR_OK) st = cuda_check(cudaStreamSynchronize(nullptr), "layout");
  return st;
}

}  // namespace frgb
