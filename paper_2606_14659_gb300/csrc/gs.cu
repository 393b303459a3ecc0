// gs.cu — the element dual graph from element -> vertex ids, and the Laplacian
// action without a stored graph (paper §5, gather-scatter; §2, weights).
//
// Input: ne elements, nv global vertex ids each (8 for hexes), ids in
// [0, V).  Set-up: the elements at every global vertex ("buckets": a
// counting sort by vertex id, then every bucket sorted by element id, so the
// result does not depend on the order of the atomics; a mesh of at most eight
// elements a vertex keeps them in fixed slots instead, below).  Q^T of §5 is then a
// sum over a bucket, Q a read of the vertex's sum.
//   * dual graph: element e's neighbours are the other elements in the buckets
//     of its vertices; the weight of neighbour f is how many of e's vertices f
//     shares (omega of §2): one pass counts the distinct neighbours (row
//     lengths), a scan gives row_ptr, a second pass writes them in ascending
//     order;
//   * matrix-free action y = (D_w - A_w) x with A_w = P^T Q Q^T P: per vertex
//     w_v = sum of x over its bucket (Q^T P x), per element
//     y_e = sum over e's vertices v of (c_v x_e - w_v), c_v the bucket size,
//     which is sum_v sum_{f at v} (x_e - x_f): the diagonal term of A_w and
//     D_w cancel inside every vertex term.
#include <algorithm>
#include <climits>

#include "rsb_internal.cuh"

#define GS_MAXCAND 256  // neighbour candidates of one element (with repeats)

// Bound: the read of the ids; one atomic a CTA (an atomic a warp on the one address took
// longer than the read).
__global__ void __launch_bounds__(RSB_BLOCK) k_gs_maxid(const int64_t* __restrict__ ev, int64_t cnt,
                                                      unsigned long long* vmax, int* flag) {
  __shared__ long long wm[RSB_WARPS];
  long long m = -1;
  bool bad = false;
  for (int64_t i = (int64_t)blockIdx.x * RSB_BLOCK + threadIdx.x; i < cnt;
       i += (int64_t)gridDim.x * RSB_BLOCK) {
    const long long v = ev[i];
    if (v < 0 || v >= (1ll << 31)) bad = true;
    else m = max(m, v);
  }
  if (bad) atomicOr(flag, 1);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < RSB_WARPS; ++w) m = max(m, wm[w]);
    if (m >= 0) atomicMax(vmax, (unsigned long long)m);
  }
}

// The counts of a slot table whose vertices are too full for it, widened (count[V] = 0).
__global__ void k_gs_widen(const int32_t* __restrict__ cnt, int64_t V, int64_t* count) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v <= V) count[v] = v < V ? cnt[v] : 0;
}

__global__ void k_gs_count(const int64_t* __restrict__ ev, int64_t cnt, int64_t* count) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < cnt) atomicAdd((unsigned long long*)(count + ev[i]), 1ull);
}

// bucket fill (element ids; within a bucket in arrival order) and the slot
// table ev32 (vertex ids as int32); the counts run down to zero
__global__ void k_gs_fill(const int64_t* __restrict__ ev, int64_t cnt, int nv,
                          const int64_t* __restrict__ bptr, int64_t* count, int32_t* bucket,
                          int32_t* ev32) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= cnt) return;
  const int64_t v = ev[i];
  const int64_t left = (int64_t)atomicAdd((unsigned long long*)(count + v), ~0ull);
  bucket[bptr[v + 1] - left] = (int32_t)(i / nv);  // in arrival order, nearly sorted
  ev32[i] = (int32_t)v;
}

// every bucket sorted by element id (insertion sort: buckets are small)
__global__ void k_gs_sort(const int64_t* __restrict__ bptr, int64_t V, int32_t* bucket) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= V) return;
  const int64_t b = bptr[v], e = bptr[v + 1];
  for (int64_t p = b + 1; p < e; ++p) {
    const int32_t x = bucket[p];
    int64_t q = p - 1;
    while (q >= b && bucket[q] > x) {
      bucket[q + 1] = bucket[q];
      --q;
    }
    bucket[q + 1] = x;
  }
}

// Distinct neighbours of element e with their shared-vertex counts, ascending;
// returns their number (or -1 when the candidates overflow GS_MAXCAND).
__device__ int gs_neighbours(int64_t e, int nv, const int32_t* __restrict__ ev32,
                             const int64_t* __restrict__ bptr, const int32_t* __restrict__ bucket,
                             int32_t* cand) {
  int nc = 0;
  for (int a = 0; a < nv; ++a) {
    const int32_t v = ev32[e * nv + a];
    for (int64_t p = bptr[v]; p < bptr[v + 1]; ++p) {
      const int32_t f = bucket[p];
      if (f == (int32_t)e) continue;
      if (nc >= GS_MAXCAND) return -1;
      cand[nc++] = f;
    }
  }
  for (int p = 1; p < nc; ++p) {  // insertion sort
    const int32_t x = cand[p];
    int q = p - 1;
    while (q >= 0 && cand[q] > x) {
      cand[q + 1] = cand[q];
      --q;
    }
    cand[q + 1] = x;
  }
  return nc;
}

__global__ void k_gs_rowlen(int64_t ne, int nv, const int32_t* __restrict__ ev32,
                            const int64_t* __restrict__ bptr, const int32_t* __restrict__ bucket,
                            int64_t* len, volatile int* flag) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e == ne) len[ne] = 0;  // (the scan's last entry)
  if (e >= ne) return;
  int32_t cand[GS_MAXCAND];
  const int nc = gs_neighbours(e, nv, ev32, bptr, bucket, cand);
  if (nc < 0) {
    flag[0] = 1;
    len[e] = 0;
    return;
  }
  int64_t d = 0;
  int run = 0;
  for (int p = 0; p < nc; ++p) {
    run = (p > 0 && cand[p] == cand[p - 1]) ? run + 1 : 1;
    if (p + 1 == nc || cand[p + 1] != cand[p]) {
      ++d;
      if (run > 7) flag[1] = 1;  // more than 7 shared vertices: duplicate elements
    }
  }
  len[e] = d;
}

__global__ void k_gs_dual(int64_t ne, int nv, const int32_t* __restrict__ ev32,
                          const int64_t* __restrict__ bptr, const int32_t* __restrict__ bucket,
                          const int64_t* __restrict__ row_ptr, int32_t* col, int32_t* wt) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= ne) return;
  int32_t cand[GS_MAXCAND];
  const int nc = gs_neighbours(e, nv, ev32, bptr, bucket, cand);
  if (nc < 0) return;
  int64_t out = row_ptr[e];
  int run = 0;
  for (int p = 0; p < nc; ++p) {
    run = (p > 0 && cand[p] == cand[p - 1]) ? run + 1 : 1;
    if (p + 1 == nc || cand[p + 1] != cand[p]) {
      col[out] = cand[p];
      wt[out] = run;
      ++out;
    }
  }
}

// w_v = sum of x over the elements at vertex v (Q^T P x), in bucket order
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_gs_vsum(int64_t nvert, const int64_t* __restrict__ bptr,
                                                     const int32_t* __restrict__ bucket,
                                                     const V* __restrict__ x, V* w) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= nvert) return;
  const int64_t b = bptr[v], e = bptr[v + 1];
  V s = V(0);
  for (int64_t p = b; p < e; ++p) s += __ldg(x + bucket[p]);
  w[v] = s;
}

// y_e = sum over e's vertices of (c_v x_e - w_v): (D_w - A_w) x, no stored graph
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_gs_apply(int64_t ne, int nv,
                                                      const int32_t* __restrict__ ev32,
                                                      const int64_t* __restrict__ bptr,
                                                      const V* __restrict__ w,
                                                      const V* __restrict__ x, V* y) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= ne) return;
  const V xe = x[e];
  V acc = V(0);
  for (int a = 0; a < nv; ++a) {
    const int32_t v = __ldg(ev32 + e * nv + a);
    const V c = V(__ldg(bptr + v + 1) - __ldg(bptr + v));
    acc += c * xe - __ldg(w + v);
  }
  y[e] = acc;
}

// ----------------------------------------------------------------------------
// Slot table: the elements at every vertex in GS_SLOTS fixed places, for meshes whose
// vertices have at most that many (hexes: eight in the interior) and whose ids lie
// below a bound known beforehand.  One pass over the ids takes the place of the pass
// for the largest id (and the host's wait for it), the count, the scan and the fill of
// the buckets above; a mesh that does not fit sets a word, the kernels that follow return
// almost at once, leaving the largest id, and the caller takes the general path, which
// need not look for it again, nor count when it is below the bound.  A vertex's slots hold its elements
// in arrival order; their readers sort the at most eight of them in registers, so results
// do not depend on it.
// One Laplacian application at 1.9M hexes 168 us, 717 from the buckets.
// Words behind the counts, cleared with them: [0] an id outside [0, 2^31), [1] the table
// does not hold the mesh, [2] two elements share more than 7 vertices, [3] an element has
// more than GS_ROW neighbours, [4] the largest id of a mesh that the table does not hold.
// ----------------------------------------------------------------------------
#define GS_SLOTS 8
#define GS_WORDS 8

// The ids of element e (unused places: -1).
template <bool HEX>
__device__ __forceinline__ void gs_ids(const int64_t* __restrict__ ev, int64_t e, int nv,
                                       int64_t (&id)[8]) {
  if constexpr (HEX) {  // eight ids, 16-byte aligned
    const longlong2* p = reinterpret_cast<const longlong2*>(ev + 8 * e);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const longlong2 v = __ldg(p + i);
      id[2 * i] = v.x;
      id[2 * i + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) id[i] = i < nv ? __ldg(ev + e * nv + i) : -1;
  }
}

// Word 4 takes the largest m (not negative) of the threads that are here.
__device__ __forceinline__ void gs_note_max(int32_t* cnt, int64_t cap, int m) {
  const unsigned mask = __activemask();
  m = __reduce_max_sync(mask, m);
  if ((int)(threadIdx.x & 31) == __ffs(mask) - 1 && m > *(volatile int32_t*)(cnt + cap + 4))
    atomicMax(cnt + cap + 4, m);
}

// Bound: the returned atomics (one per id, eight in flight a thread).
template <bool HEX>
__global__ void __launch_bounds__(RSB_BLOCK) k_gs_slots(const int64_t* __restrict__ ev, int64_t ne,
                                                      int nv, int64_t cap, int32_t* cnt,
                                                      int32_t* __restrict__ slot) {
  const int64_t e = (int64_t)blockIdx.x * RSB_BLOCK + threadIdx.x;
  if (e >= ne) return;
  volatile int32_t* err = cnt + cap;
  int64_t id[8];
  gs_ids<HEX>(ev, e, nv, id);
  bool out = false, full = false;
  int far = 0;
  int pos[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    pos[i] = GS_SLOTS;
    if (HEX || i < nv) {
      if (id[i] < 0 || id[i] >= (1ll << 31)) out = true;
      else if (id[i] >= cap) far = max(far, (int)id[i]);
      else pos[i] = atomicAdd(cnt + id[i], 1);
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    if (pos[i] < GS_SLOTS) slot[id[i] * GS_SLOTS + pos[i]] = (int32_t)e;
    else if ((HEX || i < nv) && id[i] >= 0 && id[i] < cap) full = true;
  }
  if (out && !err[0]) err[0] = 1;
  if ((full || far) && !err[1]) err[1] = 1;
  if (far) gs_note_max(cnt, cap, far);
}

// Not zero: the table does not hold the mesh.  (Its readers load it beside their first
// operands: as a load and a branch of its own it costs them 1 %.)
__device__ __forceinline__ int gs_unfit(const int32_t* cnt, int64_t cap) {
  return cnt[cap] | cnt[cap + 1];
}

// The elements at vertex v in ascending order, INT_MAX in the places left (a sorting
// network of 19 exchanges); returns their number (0 when the mesh does not fit: the
// largest vertex that has any is then noted).
__device__ __forceinline__ int gs_sorted_slots(int32_t* cnt, int64_t cap, const int32_t* slot,
                                               int64_t v, int32_t (&f)[GS_SLOTS]) {
  const int here = cnt[v], unfit = gs_unfit(cnt, cap);
  if (unfit && here) gs_note_max(cnt, cap, (int)v);
  const int n = unfit ? 0 : min(here, GS_SLOTS);
  const int4* p = reinterpret_cast<const int4*>(slot + v * GS_SLOTS);
  int4 lo = make_int4(0, 0, 0, 0), hi = lo;
  if (n > 0) lo = p[0];
  if (n > 4) hi = p[1];
  const int32_t r[GS_SLOTS] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
  for (int i = 0; i < GS_SLOTS; ++i) f[i] = i < n ? r[i] : INT_MAX;
  auto ex = [&](int a, int b) {
    const int32_t x = min(f[a], f[b]), y = max(f[a], f[b]);
    f[a] = x;
    f[b] = y;
  };
  ex(0, 1); ex(2, 3); ex(4, 5); ex(6, 7);
  ex(0, 2); ex(1, 3); ex(4, 6); ex(5, 7);
  ex(1, 2); ex(5, 6); ex(0, 4); ex(3, 7);
  ex(1, 5); ex(2, 6);
  ex(1, 4); ex(3, 6);
  ex(2, 4); ex(3, 5);
  ex(3, 4);
  return n;
}

// (w_v, c_v) of every vertex: the sum of x over its elements in ascending order, as
// k_gs_vsum takes it, and their number, side by side for one gather.
template <typename V>
struct alignas(2 * sizeof(V)) GsPair {
  V w, c;
};

template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_gs_vsum8(int64_t nvert, int32_t* cnt,
                                                      const int32_t* __restrict__ slot,
                                                      const V* __restrict__ x,
                                                      GsPair<V>* __restrict__ wc) {
  const int64_t v = (int64_t)blockIdx.x * RSB_BLOCK + threadIdx.x;
  if (v >= nvert) return;
  int32_t f[GS_SLOTS];
  const int n = gs_sorted_slots(cnt, nvert, slot, v, f);
  V xv[GS_SLOTS];
#pragma unroll
  for (int i = 0; i < GS_SLOTS; ++i) xv[i] = i < n ? __ldg(x + f[i]) : V(0);
  V s = V(0);
#pragma unroll
  for (int i = 0; i < GS_SLOTS; ++i)
    if (i < n) s += xv[i];
  if (n > 0) wc[v] = {s, V(n)};
}

template <typename V, bool HEX>
__global__ void __launch_bounds__(RSB_BLOCK) k_gs_apply8(int64_t ne, int nv,
                                                       const int64_t* __restrict__ ev, int64_t cap,
                                                       const GsPair<V>* __restrict__ wc,
                                                       const int32_t* __restrict__ cnt,
                                                       const V* __restrict__ x, V* __restrict__ y,
                                                       volatile int* err) {
  const int64_t e = (int64_t)blockIdx.x * RSB_BLOCK + threadIdx.x;
  if (e >= ne) return;
  const int unfit = gs_unfit(cnt, cap);
  int64_t id[8];
  gs_ids<HEX>(ev, e, nv, id);
  if (unfit) {  // told to the host, which then takes the buckets
    if (e == 0) err[0] = cnt[cap], err[1] = cnt[cap + 1], err[4] = cnt[cap + 4];
    return;
  }
  GsPair<V> p[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    p[i] = {V(0), V(0)};
    if (id[i] >= 0 && id[i] < cap) p[i] = wc[id[i]];
  }
  const V xe = x[e];
  V acc = V(0);
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (HEX || i < nv) acc += p[i].c * xe - p[i].w;
  y[e] = acc;
}

// Every vertex's slots in ascending order, INT_MAX in the places left (in place).
__global__ void __launch_bounds__(RSB_BLOCK) k_gs_sort8(int64_t nvert, int32_t* cnt, int32_t* slot) {
  const int64_t v = (int64_t)blockIdx.x * RSB_BLOCK + threadIdx.x;
  if (v >= nvert) return;
  int32_t f[GS_SLOTS];
  if (gs_sorted_slots(cnt, nvert, slot, v, f) == 0) return;
  int4* p = reinterpret_cast<int4*>(slot + v * GS_SLOTS);
  p[0] = make_int4(f[0], f[1], f[2], f[3]);
  p[1] = make_int4(f[4], f[5], f[6], f[7]);
}

// Distinct neighbours of element e with their shared-vertex counts, ascending: a merge
// of the sorted slots of its vertices, the heads in registers.  A neighbour's entry
// (packed as in the sliced form) goes to ent[(32-row group * GS_ROW + k) * 32 + lane]
// (MERGE_ROWS), their number to len[e].  An element of more than GS_ROW neighbours (of at
// most 56) sets word 3, and the rows are merged once more, straight into CSR
// (MERGE_CSR): the graph of 1M elements of 56 neighbours, counted and written by two calls,
// 2.0 ms, from the buckets 4.6.
// Bound: the loads of the heads (each slot of the element's vertices once, from L1 and
// L2).  Collecting the candidates in a local-memory array of 256 and insertion-sorting
// it, once to count and once to write, made the dual graph of 2.4M hexes take 4330 us
// (two calls); it takes 589 (one).
#define GS_ROW 32
enum { MERGE_COUNT, MERGE_ROWS, MERGE_CSR };
template <bool HEX, int MODE>
__global__ void __launch_bounds__(RSB_BLOCK) k_gs_merge(int64_t ne, int nv,
                                                      const int64_t* __restrict__ ev, int64_t cap,
                                                      const int32_t* __restrict__ slot,
                                                      uint32_t* __restrict__ ent,
                                                      int64_t* __restrict__ len, int32_t* cnt,
                                                      const int64_t* __restrict__ row_ptr,
                                                      int32_t* __restrict__ col,
                                                      int32_t* __restrict__ wt) {
  const int64_t e = (int64_t)blockIdx.x * RSB_BLOCK + threadIdx.x;
  if (MODE != MERGE_CSR && e == ne) len[ne] = 0;  // (the scan's last entry)
  if (e >= ne) return;
  const int unfit = gs_unfit(cnt, cap);
  int64_t id[8];
  gs_ids<HEX>(ev, e, nv, id);
  if (unfit) {
    if (MODE != MERGE_CSR) len[e] = 0;
    return;
  }
  const int64_t row = MODE == MERGE_CSR ? row_ptr[e] : 0;
  const int32_t* p[8];
  int32_t h[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const bool in = id[i] >= 0 && id[i] < cap;
    p[i] = slot + (in ? id[i] * GS_SLOTS : 0);
    h[i] = in ? __ldg(p[i]) : INT_MAX;
  }
  uint32_t* out = MODE == MERGE_ROWS ? ent + (e >> 5) * (GS_ROW * 32) + (e & 31) : nullptr;
  uint32_t pos = 0;  // four bits a list
  int32_t prev = -1;
  int run = 0, d = 0, most = 0;
  while (true) {
    const int32_t m = min(min(min(h[0], h[1]), min(h[2], h[3])), min(min(h[4], h[5]), min(h[6], h[7])));
    if (m != prev) {
      if (run > 0 && prev != (int32_t)e) {
        if (MODE == MERGE_ROWS && d < GS_ROW)
          out[32 * d] = ((uint32_t)min(run, 7) << RSB_COLBITS) | (uint32_t)prev;
        if (MODE == MERGE_CSR) {
          col[row + d] = prev;
          wt[row + d] = run;
        }
        most = max(most, run);
        ++d;
      }
      prev = m;
      run = 0;
    }
    if (m == INT_MAX) break;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (h[i] == m) {
        ++run;
        pos += 1u << (4 * i);
        const int k = (pos >> (4 * i)) & 15;
        h[i] = k < GS_SLOTS ? __ldg(p[i] + k) : INT_MAX;
      }
  }
  if (MODE == MERGE_CSR) return;
  len[e] = d;
  volatile int32_t* err = cnt + cap;
  if (d > GS_ROW && !err[3]) err[3] = 1;
  if (most > 7 && !err[2]) err[2] = 1;
}

// The merged rows into CSR: a warp's 32 rows are contiguous there, so they pass through
// shared memory and are written coalesced.
__global__ void __launch_bounds__(RSB_BLOCK) k_gs_write(int64_t ne, const uint32_t* __restrict__ ent,
                                                      const int64_t* __restrict__ row_ptr,
                                                      int32_t* __restrict__ col,
                                                      int32_t* __restrict__ wt) {
  __shared__ uint32_t sh[RSB_WARPS][GS_ROW * 32];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t e0 = (int64_t)blockIdx.x * RSB_BLOCK + 32 * w;
  if (e0 >= ne) return;
  const int rows = (int)min((int64_t)32, ne - e0);
  const int64_t b = row_ptr[min(e0 + lane, ne)];
  const int64_t b0 = __shfl_sync(0xffffffffu, b, 0);
  const int64_t b1 = row_ptr[e0 + rows];
  const int d = lane < rows ? (int)(row_ptr[e0 + lane + 1] - b) : 0;
  const uint32_t* in = ent + (e0 >> 5) * (GS_ROW * 32) + lane;
  uint32_t* out = sh[w] + (b - b0);
  for (int k0 = 0; k0 < GS_ROW; k0 += 8) {
    uint32_t v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = k0 + i < d ? __ldcs(in + 32 * (k0 + i)) : 0u;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (k0 + i < d) out[k0 + i] = v[i];
    if (!__any_sync(0xffffffffu, k0 + 8 < d)) break;
  }
  __syncwarp();
  const int n = (int)(b1 - b0);
  for (int i = lane; i < n; i += 32) {
    const uint32_t v = sh[w][i];
    __stcs(col + b0 + i, (int32_t)ent_col(v));
    __stcs(wt + b0 + i, (int32_t)ent_w(v));
  }
}

// ----------------------------------------------------------------------------
// launchers (workspace: the caller's; sizes from gs_sizes)
// ----------------------------------------------------------------------------
static unsigned grid_of(int64_t n, int block = RSB_BLOCK) {
  return (unsigned)((n + block - 1) / block);
}

// Largest vertex id + 1 (V) of the table, or an error for ids outside [0, 2^31).
// d_max: two device words (the largest id, a flag), h_max: two pinned host words.
int gs_vertex_count(const int64_t* ev, int64_t cnt, unsigned long long* d_max,
                    unsigned long long* h_max, int64_t* V, cudaStream_t s) {
  RSB_CK(cudaMemsetAsync(d_max, 0, 2 * sizeof(unsigned long long), s));
  if (cnt > 0) {
    int dev = 0, nsm = 0;  // CTAs of one wave, so that the atomics are few
    RSB_CK(cudaGetDevice(&dev));
    RSB_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    k_gs_maxid<<<std::min(grid_of(cnt), 8u * (unsigned)nsm), RSB_BLOCK, 0, s>>>(
        ev, cnt, d_max, (int*)(d_max + 1));
    RSB_CKL("k_gs_maxid");
  }
  RSB_CK(cudaMemcpyAsync(h_max, d_max, 2 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
  RSB_CK(cudaStreamSynchronize(s));
  if (h_max[1]) return rsb_set_error(RSB_EINVAL, "vertex ids must lie in [0, 2^31)");
  *V = cnt > 0 ? (int64_t)h_max[0] + 1 : 0;
  return RSB_OK;
}

// Buckets: bptr[V + 1], bucket[ne * nv], ev32[ne * nv]; count is int64[V + 1]
// scratch.  counted (optional): the number of elements at each of the V vertices.
int gs_buckets(const int64_t* ev, int64_t ne, int nv, int64_t V, const int32_t* counted,
               int64_t* count, int64_t* bptr, int32_t* bucket, int32_t* ev32, void* scan_tmp,
               size_t scan_bytes, cudaStream_t s) {
  const int64_t cnt = ne * nv;
  if (counted) {
    k_gs_widen<<<grid_of(V + 1), RSB_BLOCK, 0, s>>>(counted, V, count);
    RSB_CKL("k_gs_widen");
  } else {
    RSB_CK(cudaMemsetAsync(count, 0, sizeof(int64_t) * (size_t)(V + 1), s));
  }
  if (cnt > 0 && !counted) {
    k_gs_count<<<grid_of(cnt), RSB_BLOCK, 0, s>>>(ev, cnt, count);
    RSB_CKL("k_gs_count");
  }
  int rc = launch_scan_i64(count, bptr, V + 1, scan_tmp, scan_bytes, s);
  if (rc) return rc;
  if (cnt > 0) {
    k_gs_fill<<<grid_of(cnt), RSB_BLOCK, 0, s>>>(ev, cnt, nv, bptr, count, bucket, ev32);
    RSB_CKL("k_gs_fill");
    k_gs_sort<<<grid_of(V), RSB_BLOCK, 0, s>>>(bptr, V, bucket);
    RSB_CKL("k_gs_sort");
  }
  return RSB_OK;
}

// flag: two pinned host words (zero before): an element meets more than GS_MAXCAND others,
// two elements share more than 7 vertices.  len: ne + 1 entries.
int gs_row_lengths(int64_t ne, int nv, const int32_t* ev32, const int64_t* bptr,
                   const int32_t* bucket, int64_t* len, int* flag, cudaStream_t s) {
  if (ne <= 0) return RSB_OK;
  k_gs_rowlen<<<grid_of(ne + 1, 128), 128, 0, s>>>(ne, nv, ev32, bptr, bucket, len, flag);
  RSB_CKL("k_gs_rowlen");
  return RSB_OK;
}

int gs_fill_dual(int64_t ne, int nv, const int32_t* ev32, const int64_t* bptr,
                 const int32_t* bucket, const int64_t* row_ptr, int32_t* col, int32_t* wt,
                 cudaStream_t s) {
  if (ne <= 0) return RSB_OK;
  k_gs_dual<<<grid_of(ne, 128), 128, 0, s>>>(ne, nv, ev32, bptr, bucket, row_ptr, col, wt);
  RSB_CKL("k_gs_dual");
  return RSB_OK;
}

int gs_apply(int f32, int64_t ne, int nv, int64_t V, const int32_t* ev32, const int64_t* bptr,
             const int32_t* bucket, const void* x, void* w, void* y, cudaStream_t s) {
  if (ne <= 0) return RSB_OK;
  if (f32) {
    k_gs_vsum<float><<<grid_of(V), RSB_BLOCK, 0, s>>>(V, bptr, bucket, (const float*)x, (float*)w);
    RSB_CKL("k_gs_vsum<f32>");
    k_gs_apply<float><<<grid_of(ne), RSB_BLOCK, 0, s>>>(ne, nv, ev32, bptr, (const float*)w,
                                                        (const float*)x, (float*)y);
    RSB_CKL("k_gs_apply<f32>");
  } else {
    k_gs_vsum<double><<<grid_of(V), RSB_BLOCK, 0, s>>>(V, bptr, bucket, (const double*)x,
                                                       (double*)w);
    RSB_CKL("k_gs_vsum<f64>");
    k_gs_apply<double><<<grid_of(ne), RSB_BLOCK, 0, s>>>(ne, nv, ev32, bptr, (const double*)w,
                                                         (const double*)x, (double*)y);
    RSB_CKL("k_gs_apply<f64>");
  }
  return RSB_OK;
}

// ----------------------------------------------------------------------------
// slot-table path
// ----------------------------------------------------------------------------
// Ids the table is laid out for: hexes share most of their vertices (V is little more
// than ne), elements that share none have 8 ne.
int64_t gs_slot_cap(int64_t ne) { return 2 * ne + 4096; }
size_t gs_slot_bytes(int64_t cap) { return sizeof(int32_t) * GS_SLOTS * (size_t)cap; }

static bool hex_aligned(const int64_t* ev, int nv) { return nv == 8 && ((uintptr_t)ev & 15) == 0; }

size_t gs_cnt_bytes(int64_t cap) { return sizeof(int32_t) * (size_t)(cap + GS_WORDS); }

int gs_slots(const int64_t* ev, int64_t ne, int nv, int64_t cap, int32_t* cnt, int32_t* slot,
             cudaStream_t s) {
  RSB_CK(cudaMemsetAsync(cnt, 0, gs_cnt_bytes(cap), s));
  if (hex_aligned(ev, nv))
    k_gs_slots<true><<<grid_of(ne), RSB_BLOCK, 0, s>>>(ev, ne, nv, cap, cnt, slot);
  else
    k_gs_slots<false><<<grid_of(ne), RSB_BLOCK, 0, s>>>(ev, ne, nv, cap, cnt, slot);
  RSB_CKL("k_gs_slots");
  return RSB_OK;
}

template <typename V>
static int gs_slot_apply_t(const int64_t* ev, int64_t ne, int nv, int64_t cap, int32_t* cnt,
                           const int32_t* slot, const V* x, void* wc, V* y, int* err,
                           cudaStream_t s) {
  GsPair<V>* p = (GsPair<V>*)wc;
  k_gs_vsum8<V><<<grid_of(cap), RSB_BLOCK, 0, s>>>(cap, cnt, slot, x, p);
  RSB_CKL("k_gs_vsum8");
  if (hex_aligned(ev, nv))
    k_gs_apply8<V, true><<<grid_of(ne), RSB_BLOCK, 0, s>>>(ne, nv, ev, cap, p, cnt, x, y, err);
  else
    k_gs_apply8<V, false><<<grid_of(ne), RSB_BLOCK, 0, s>>>(ne, nv, ev, cap, p, cnt, x, y, err);
  RSB_CKL("k_gs_apply8");
  return RSB_OK;
}

// y = L x from the slot table (wc: 2 * cap values of the vector type); a mesh that does
// not fit leaves y as it is and sets err[0] or err[1], and err[4] (pinned host words).
int gs_slot_apply(int f32, const int64_t* ev, int64_t ne, int nv, int64_t cap, int32_t* cnt,
                  const int32_t* slot, const void* x, void* wc, void* y, int* err, cudaStream_t s) {
  return f32 ? gs_slot_apply_t<float>(ev, ne, nv, cap, cnt, slot, (const float*)x, wc, (float*)y,
                                      err, s)
             : gs_slot_apply_t<double>(ev, ne, nv, cap, cnt, slot, (const double*)x, wc, (double*)y,
                                       err, s);
}

// Row lengths of the dual graph from the slot table and, with ent, the rows
// themselves for gs_slot_write (ent: gs_rows_bytes).
size_t gs_rows_bytes(int64_t ne) { return sizeof(uint32_t) * GS_ROW * 32 * (size_t)((ne + 31) / 32); }

// err: GS_WORDS pinned host words, valid once the stream is done.  len: ne + 1 entries.
template <int MODE>
static int gs_merge(const int64_t* ev, int64_t ne, int nv, int64_t cap, int32_t* cnt,
                    const int32_t* slot, uint32_t* ent, int64_t* len, const int64_t* row_ptr,
                    int32_t* col, int32_t* wt, cudaStream_t s) {
  const unsigned nb = grid_of(ne + 1);
  if (hex_aligned(ev, nv))
    k_gs_merge<true, MODE><<<nb, RSB_BLOCK, 0, s>>>(ne, nv, ev, cap, slot, ent, len, cnt, row_ptr,
                                                   col, wt);
  else
    k_gs_merge<false, MODE><<<nb, RSB_BLOCK, 0, s>>>(ne, nv, ev, cap, slot, ent, len, cnt, row_ptr,
                                                    col, wt);
  RSB_CKL("k_gs_merge");
  return RSB_OK;
}

int gs_slot_rows(const int64_t* ev, int64_t ne, int nv, int64_t cap, int32_t* cnt, int32_t* slot,
                 uint32_t* ent, int64_t* len, int* err, cudaStream_t s) {
  k_gs_sort8<<<grid_of(cap), RSB_BLOCK, 0, s>>>(cap, cnt, slot);
  RSB_CKL("k_gs_sort8");
  int rc = ent ? gs_merge<MERGE_ROWS>(ev, ne, nv, cap, cnt, slot, ent, len, nullptr, nullptr,
                                      nullptr, s)
               : gs_merge<MERGE_COUNT>(ev, ne, nv, cap, cnt, slot, ent, len, nullptr, nullptr,
                                       nullptr, s);
  if (rc) return rc;
  RSB_CK(cudaMemcpyAsync(err, cnt + cap, GS_WORDS * sizeof(int), cudaMemcpyDeviceToHost, s));
  return RSB_OK;
}

// The rows into CSR: from ent, or where some are too long for it (ent null) merged again.
int gs_slot_write(const int64_t* ev, int64_t ne, int nv, int64_t cap, int32_t* cnt,
                  const int32_t* slot, const uint32_t* ent, const int64_t* row_ptr, int32_t* col,
                  int32_t* wt, cudaStream_t s) {
  if (!ent)
    return gs_merge<MERGE_CSR>(ev, ne, nv, cap, cnt, slot, nullptr, nullptr, row_ptr, col, wt, s);
  k_gs_write<<<grid_of(ne), RSB_BLOCK, 0, s>>>(ne, ent, row_ptr, col, wt);
  RSB_CKL("k_gs_write");
  return RSB_OK;
}
