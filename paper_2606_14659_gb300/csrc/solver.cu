// solver.cu — Fiedler solvers of librsb, batched over all units of a level.
//
// Lanczos with restarts (paper §6), the Lanczos vectors kept orthonormal by
// classical Gram-Schmidt with a second pass (CGS2).  FP64 steps:
//   A: w = L q_j, fused with the first Gram-Schmidt pass's dot products
//      against [1/sqrt(n), deflation vectors, q_0..q_j],
//   B: w -= basis * c1, fused with the second pass's dot products,
//   C: w -= basis * c2, fused with ||w||^2 -> beta_{j+1};
// q_{j+1} = w / beta_{j+1} is materialised by the next step's A, which gathers
// the unnormalised w and scales.  FP32 steps (bandwidth-bound) delay the
// second pass by one step, two passes over the basis instead of three:
//   D1: z = L v_j (v_j = w_j / nu_j, projected once),
//   D2: a = B^T v_j, g = B^T z, v.v, v.z in one pass -> q_j = (v_j - B a) / rho
//       and column j of S,
//   D3: q_j and w_{j+1} = (z - B g - (q_j.z) q_j) / rho in one pass, nu_{j+1}.
// After the cycle: the Ritz pairs of the
// projected matrix S = Q^T L Q (parallel cyclic Jacobi, one CTA per unit), the
// Ritz vector y = Q t, the true residual ||L y - theta y||, and a thick restart
// from the kept Ritz vectors and the last residual direction (an explicit
// restart from y, projected against the fixed basis, when a cycle ended on an
// invariant subspace).  Launch modes: one kernel per step phase (optionally
// replayed as a CUDA graph per cycle), one cooperative kernel per cycle (CGS2
// in both precisions), or one cooperative kernel per solve with the basis
// resident in shared memory (the steps of the per-phase kernels, bit for bit).
//
// Inverse iteration (paper §7, Algorithm 2): the right-hand side b is the
// projected, normalised previous iterate; L x = b is solved by CG from x0 = 0
// with r projected against the fixed basis every step; the Rayleigh quotient
// and residual of x decide the stop (also when CG returned after a single
// iteration, §7).
//
// Precision: V = double (plain FP64) or V = float (vectors, SpMV and updates
// in FP32; per-thread Kahan sums in FP32; CTA and cross-CTA sums, the
// Gram-Schmidt coefficients, T, and the CG alpha/beta recurrences in FP64).
#include <chrono>
#include <algorithm>
#include <cfloat>

#include "rsb_internal.cuh"
#include "rsb_probe.h"

int g_rsb_poison_barrier = 0;  // test hook, see rsb_test_poison_barrier

template <typename V>
struct LzArgs {
  const int64_t* slice_ptr;
  const uint32_t* ent;
  const int64_t* gid;
  const Tile* tiles;
  Unit* units;
  const uint64_t* ckey;
  V* Q;
  long long N;
  V* W0;
  V* W1;
  V* Y;
  V* X;
  V* R;
  V* P;
  V* AP;
  const double* D0;
  const double* D1;
  double* partials;
  long long stride;
  int* n_active;
  long long* stat_cycles;
  unsigned long long* pb_a;  // profiling byte counters (nullptr when off)
  unsigned long long* pb_a2;
  unsigned long long* pb_b;
  unsigned long long* pb_c;
  unsigned long long* pb_cg;
  double* S;                 // per unit: projected matrix S (M x M) then Ritz vectors Y
  int* jmin;                 // smallest first step of the next cycle over the units
};

// CTA-level add of per-thread byte counts to a profiling counter.
__device__ __forceinline__ void prof_add(unsigned long long* pb, unsigned long long b) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) b += __shfl_xor_sync(0xffffffffu, b, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(pb, b);
}

__device__ __forceinline__ int row_width(const int64_t* __restrict__ slice_ptr, int r) {
  return (int)((slice_ptr[(r >> 5) + 1] - slice_ptr[r >> 5]) >> 5);
}

template <typename V, bool CO = false>
__device__ __forceinline__ V spmv_row(const int64_t* __restrict__ slice_ptr,
                                      const uint32_t* __restrict__ ent, const V* x, int r, V xr) {
  const int64_t base = slice_ptr[r >> 5];
  const int width = (int)((slice_ptr[(r >> 5) + 1] - base) >> 5);
  const uint32_t* e = ent + base + (r & 31);
  V acc = V(0);
  uint32_t dsum = 0;
#pragma unroll 4
  for (int k = 0; k < width; ++k) {
    const uint32_t p = __ldg(e + 32 * k);
    if constexpr (sizeof(V) == 8) {  // FP64: d_r x_r - sum w x_c, as spmv_row_ro
      acc = fma(weight_f64(ent_w(p)), ldc<CO>(x + ent_col(p)), acc);
      dsum += ent_w(p);
    } else {
      acc += V(ent_w(p)) * (xr - ldc<CO>(x + ent_col(p)));
    }
  }
  if constexpr (sizeof(V) == 8) return fma((double)dsum, xr, -acc);
  return acc;
}

// The same for x that other CTAs of the launch wrote before a barrier: plain loads
// (L1 may serve them), eight in flight.
template <typename V>
__device__ __forceinline__ V spmv_row_batched(const int64_t* __restrict__ slice_ptr,
                                              const uint32_t* __restrict__ ent, const V* x, int r,
                                              V xr) {
  const int64_t base = slice_ptr[r >> 5];
  const int width = (int)((slice_ptr[(r >> 5) + 1] - base) >> 5);
  const uint32_t* e = ent + base + (r & 31);
  V acc = V(0);
  uint32_t dsum = 0;
  for (int k0 = 0; k0 < width; k0 += 8) {
    uint32_t p[8];
    V xv[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) p[i] = k0 + i < width ? __ldg(e + 32 * (k0 + i)) : 0u;
#pragma unroll
    for (int i = 0; i < 8; ++i) xv[i] = k0 + i < width ? x[ent_col(p[i])] : xr;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (k0 + i < width) {
        if constexpr (sizeof(V) == 8) {
          acc = fma(weight_f64(ent_w(p[i])), xv[i], acc);
          dsum += ent_w(p[i]);
        } else {
          acc += V(ent_w(p[i])) * (xr - xv[i]);
        }
      }
  }
  if constexpr (sizeof(V) == 8) return fma((double)dsum, xr, -acc);
  return acc;
}

// ----------------------------------------------------------------------------
// Gram-Schmidt building blocks.  The basis is [u0, D_0.., q_0..q_j] with
// u0 = 1/sqrt(n) on unit rows (its dot is taken as a plain sum and scaled by
// 1/sqrt(n) afterwards).  A CTA handles its tile in sub-chunks of up to
// RSB_BLOCK * RSB_SUBR rows: phase 1 computes the chunk's w (one row per
// thread and RSB_SUBR rows per thread, coefficient-outer so that every
// thread has RSB_SUBR independent loads in flight), stores it in shared
// memory; phase 2 takes the dot products warp-per-coefficient with unrolled
// coalesced loads.
// ----------------------------------------------------------------------------
#define MAXCW ((RSB_MAXC + RSB_WARPS - 1) / RSB_WARPS)
#define SUBROWS (RSB_BLOCK * RSB_SUBR)

// Warp-per-coefficient dots of basis coefficients [c0, c0 + nc) with the chunk:
// warp w owns coefficients w, w + 8, ...; each lane walks rows in groups of 4
// and issues the loads of all of its warp's coefficients for the group before
// accumulating, so up to 4 * MAXCW loads are in flight per lane.
template <typename V>
__device__ __forceinline__ void tile_dots(const LzArgs<V>& a, int nd, int c0, int nc, int base,
                                          int end, const V* ws, Acc<V> (&acc)[MAXCW]) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const V* qp[MAXCW];
  const double* dp[MAXCW];
  int kind[MAXCW];  // -1 none, 0 ones (u0), 1 FP64 deflation vector, 2 basis vector
#pragma unroll
  for (int i = 0; i < MAXCW; ++i) {
    const int c = w + RSB_WARPS * i;
    const int cc = c0 + c;
    qp[i] = nullptr;
    dp[i] = nullptr;
    if (c >= nc) kind[i] = -1;
    else if (cc == 0) kind[i] = 0;
    else if (cc <= nd) {
      kind[i] = 1;
      dp[i] = cc == 1 ? a.D0 : a.D1;
    } else {
      kind[i] = 2;
      qp[i] = a.Q + (long long)(cc - 1 - nd) * a.N;
    }
  }
  if (kind[0] < 0) return;
  constexpr int NR = sizeof(V) == 8 ? 2 : 4;  // rows a lane per round
  for (int row = base + lane; row < end; row += 32 * NR) {
    V wv[NR];
    bool ok[NR];
#pragma unroll
    for (int q = 0; q < NR; ++q) {
      ok[q] = row + 32 * q < end;
      wv[q] = ok[q] ? ws[row + 32 * q - base] : V(0);
    }
    V b[MAXCW][NR];
#pragma unroll
    for (int i = 0; i < MAXCW; ++i)
#pragma unroll
      for (int q = 0; q < NR; ++q) {
        const int r = row + 32 * q;
        b[i][q] = V(0);
        if (ok[q]) {
          if (kind[i] == 2) b[i][q] = qp[i][r];
          else if (kind[i] == 1) b[i][q] = V(dp[i][r]);
          else if (kind[i] == 0) b[i][q] = V(1);
        }
      }
#pragma unroll
    for (int i = 0; i < MAXCW; ++i)
      if (kind[i] >= 0) {
#pragma unroll
        for (int q = 0; q < NR; ++q)
          if (ok[q]) acc[i].add(b[i][q] * wv[q]);
      }
  }
}

template <typename V>
__device__ __forceinline__ void store_dots(const LzArgs<V>& a, int nc, Acc<V> (&acc)[MAXCW],
                                           int tix) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < MAXCW; ++i) {
    const int c = w + RSB_WARPS * i;
    if (c < nc) {
      const double s = warp_total(acc[i]);
      if (lane == 0) a.partials[(long long)c * a.stride + tix] = s;
    }
  }
}

// w[rr] -= sum_c cv[c] basis_c for the RSB_SUBR rows of this thread
// (rows base + rr*RSB_BLOCK + tid), coefficient-outer; cv holds the
// coefficients already in the vector type (stage_coef).
template <typename V, bool CO>
__device__ __forceinline__ void gs_update_rows(const LzArgs<V>& a, const Unit& u, const V* cv,
                                               int nd, int nq, int base, int end,
                                               V (&w)[RSB_SUBR]) {
  const V c0 = cv[0];
#pragma unroll
  for (int rr = 0; rr < RSB_SUBR; ++rr) {
    const int r = base + rr * RSB_BLOCK + threadIdx.x;
    if (r < end && unit_has(u, a.ckey, r)) w[rr] -= c0;
  }
  for (int l = 0; l < nd; ++l) {
    const double* d = l == 0 ? a.D0 : a.D1;
    const V cl = cv[1 + l];
#pragma unroll
    for (int rr = 0; rr < RSB_SUBR; ++rr) {
      const int r = base + rr * RSB_BLOCK + threadIdx.x;
      if (r < end) w[rr] -= cl * V(d[r]);
    }
  }
  const V* cq = cv + 1 + nd;
  bool ok[RSB_SUBR];
#pragma unroll
  for (int rr = 0; rr < RSB_SUBR; ++rr) ok[rr] = base + rr * RSB_BLOCK + (int)threadIdx.x < end;
  int k = 0;
  for (; k + 4 <= nq; k += 4) {  // four basis vectors per round: 4 * RSB_SUBR loads in flight
    V qv[4][RSB_SUBR];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const V* q = a.Q + (long long)(k + i) * a.N + base + threadIdx.x;
#pragma unroll
      for (int rr = 0; rr < RSB_SUBR; ++rr) qv[i][rr] = ok[rr] ? q[rr * RSB_BLOCK] : V(0);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const V ck = cq[k + i];
#pragma unroll
      for (int rr = 0; rr < RSB_SUBR; ++rr) w[rr] -= ck * qv[i][rr];
    }
  }
  for (; k < nq; ++k) {
    const V ck = cq[k];
    const V* q = a.Q + (long long)k * a.N + base + threadIdx.x;
#pragma unroll
    for (int rr = 0; rr < RSB_SUBR; ++rr)
      if (ok[rr]) w[rr] -= ck * q[rr * RSB_BLOCK];
  }
}

// ----------------------------------------------------------------------------
// Lanczos step (thick-restarted, full re-orthogonalisation): per-tile bodies
// (CO = running inside the persistent cycle kernel, where data written by
// other CTAs earlier in the launch is read through L2) and the stand-alone
// kernels that wrap them.
//   A(j): q_j = src / beta (src is the unnormalised new vector), w = L q_j,
//         first Gram-Schmidt pass coefficients c1 = [1, D, q_0..q_j]^T w;
//   B(j): w -= basis c1, second-pass coefficients c2; column j of the
//         projected matrix S = Q^T L Q is c1 + c2 on q_0..q_j;
//   C(j): w -= basis c2, beta_{j+1} = ||w|| (w stays unnormalised for A(j+1)).
// ----------------------------------------------------------------------------
__device__ __forceinline__ double* unit_S(double* S, int ui) { return S + (long long)ui * RSB_SSTRIDE; }

template <typename V, bool CO>
__device__ __forceinline__ void lz_a_t(const LzArgs<V>& a, int j, int tix, V* ws, double* out) {
  const Tile t = a.tiles[tix];
  Unit& u = a.units[t.unit];
  if (ldc<CO>(&u.status) != U_ACTIVE || j >= ldc<CO>(&u.msteps) || j < ldc<CO>(&u.j0)) return;
  const V* src = (j & 1) ? a.W1 : a.W0;
  V* dst = (j & 1) ? a.W0 : a.W1;
  V* qj = a.Q + (long long)j * a.N;
  const V s = V(ldc<CO>(&u.inu));
  const int nd = u.nd;
  const int nc = 2 + nd + j;
  Acc<V> acc[MAXCW];
  unsigned long long pbytes = 0;
  for (int base = t.row0; base < t.row1; base += SUBROWS) {
    const int end = min(t.row1, base + SUBROWS);
#pragma unroll 2
    for (int rr = 0; rr < RSB_SUBR; ++rr) {
      const int r = base + rr * RSB_BLOCK + threadIdx.x;
      V w = V(0);
      if (r < end) {
        const V xr = src[r];
        if constexpr (CO) w = s * spmv_row<V, true>(a.slice_ptr, a.ent, src, r, xr);
        else w = s * spmv_row_ro<V>(a.slice_ptr, a.ent, src, r, xr);
        qj[r] = s * xr;
        dst[r] = w;
        if (a.pb_a)
          pbytes += 4ull * row_width(a.slice_ptr, r) +
                    sizeof(V) * (unsigned long long)(4 + j) + 8ull * nd;
      }
      ws[rr * RSB_BLOCK + threadIdx.x] = w;
    }
    __syncthreads();
    tile_dots<V>(a, nd, 0, nc, base, end, ws, acc);
    __syncthreads();
  }
  store_dots<V>(a, nc, acc, tix);
  if (a.pb_a) prof_add(a.pb_a, pbytes);
  if constexpr (!CO) return;  // k_lz_close reduces
  if (last_cta(&u.cnt, u.ntile)) {
    final_reduce(a.partials, a.stride, u.tile0, u.ntile, nc, out);
    if (threadIdx.x == 0) {
      u.c1[0] = out[0] * u.isn;
      for (int c = 1; c < nc; ++c) u.c1[c] = out[c];
    }
  }
}

template <typename V, bool CO>
__device__ __forceinline__ void lz_b_t(const LzArgs<V>& a, int j, int tix, V* ws, V* cv,
                                       double* out) {
  const Tile t = a.tiles[tix];
  Unit& u = a.units[t.unit];
  if (ldc<CO>(&u.status) != U_ACTIVE || j >= ldc<CO>(&u.msteps) || j < ldc<CO>(&u.j0)) return;
  V* w_ = (j & 1) ? a.W0 : a.W1;
  const int nd = u.nd;
  const int nc = 2 + nd + j;
  stage_coef<V, CO>(u.c1, nc, u.isn, cv);
  Acc<V> acc[MAXCW];
  unsigned long long pbytes = 0;
  for (int base = t.row0; base < t.row1; base += SUBROWS) {
    const int end = min(t.row1, base + SUBROWS);
    V w[RSB_SUBR];
#pragma unroll
    for (int rr = 0; rr < RSB_SUBR; ++rr) {
      const int r = base + rr * RSB_BLOCK + threadIdx.x;
      w[rr] = r < end ? w_[r] : V(0);
    }
    gs_update_rows<V, CO>(a, u, cv, nd, j + 1, base, end, w);
#pragma unroll
    for (int rr = 0; rr < RSB_SUBR; ++rr) {
      const int r = base + rr * RSB_BLOCK + threadIdx.x;
      if (r < end) {
        w_[r] = w[rr];
        if (a.pb_b) pbytes += sizeof(V) * (unsigned long long)(3 + j) + 8ull * nd;
      }
      ws[rr * RSB_BLOCK + threadIdx.x] = r < end ? w[rr] : V(0);
    }
    __syncthreads();
    tile_dots<V>(a, nd, 0, nc, base, end, ws, acc);
    __syncthreads();
  }
  store_dots<V>(a, nc, acc, tix);
  if (a.pb_b) prof_add(a.pb_b, pbytes);
  if constexpr (!CO) return;  // k_lz_close reduces
  if (last_cta(&u.cnt, u.ntile)) {
    final_reduce(a.partials, a.stride, u.tile0, u.ntile, nc, out);
    if (threadIdx.x == 0) {
      u.c2[0] = out[0] * u.isn;
      for (int c = 1; c < nc; ++c) u.c2[c] = out[c];
    }
    __syncthreads();
    double* Sm = unit_S(a.S, t.unit);
    for (int k = threadIdx.x; k <= j; k += RSB_BLOCK) {
      const double v = ldc<CO>(&u.c1[1 + nd + k]) + out[1 + nd + k];
      Sm[k * RSB_MAXM + j] = v;
      Sm[j * RSB_MAXM + k] = v;
    }
  }
}

template <typename V, bool CO>
__device__ __forceinline__ void lz_c_t(const LzArgs<V>& a, int j, double breakdown, int tix,
                                       V* cv, double* sm, double* out, double* sp) {
  const Tile t = a.tiles[tix];
  Unit& u = a.units[t.unit];
  if (ldc<CO>(&u.status) != U_ACTIVE || j >= ldc<CO>(&u.msteps) || j < ldc<CO>(&u.j0)) return;
  V* w_ = (j & 1) ? a.W0 : a.W1;
  const int nd = u.nd;
  stage_coef<V, CO>(u.c2, 2 + nd + j, u.isn, cv);
  Acc<V> acc;
  unsigned long long pbytes = 0;
  for (int base = t.row0; base < t.row1; base += SUBROWS) {
    const int end = min(t.row1, base + SUBROWS);
    V w[RSB_SUBR];
#pragma unroll
    for (int rr = 0; rr < RSB_SUBR; ++rr) {
      const int r = base + rr * RSB_BLOCK + threadIdx.x;
      w[rr] = r < end ? w_[r] : V(0);
    }
    gs_update_rows<V, CO>(a, u, cv, nd, j + 1, base, end, w);
#pragma unroll
    for (int rr = 0; rr < RSB_SUBR; ++rr) {
      const int r = base + rr * RSB_BLOCK + threadIdx.x;
      if (r < end) {
        w_[r] = w[rr];
        acc.add(w[rr] * w[rr]);
        if (a.pb_c) pbytes += sizeof(V) * (unsigned long long)(3 + j) + 8ull * nd;
      }
    }
  }
  if (a.pb_c) prof_add(a.pb_c, pbytes);
  const double sum = block_total(acc, sm);
  if (threadIdx.x == 0) a.partials[tix] = sum;
  if (last_cta(&u.cnt, u.ntile)) {
    final_reduce_few(a.partials, a.stride, u.tile0, u.ntile, 1, out, sp);
    if (threadIdx.x == 0) {
      const double b = sqrt(out[0]);
      u.beta[j + 1] = b;
      u.inu = 1.0 / b;
      if (b <= breakdown * u.dmax) {  // invariant subspace: the cycle ends here
        u.msteps = j + 1;
        u.broke = 1;
      }
    }
  }
}

// FP64 steps A and B.  Bound: the FP64 rate (an FP64 instruction holds a sub-partition
// for 64 cycles, so one ready warp in each keeps it busy); four CTAs of 64 registers, two
// rows a lane in flight, leave some warp at its arithmetic while the others wait for
// loads.  Two CTAs of 128 registers with four rows a lane took 121 us (A) at 1M rows,
// mean over 16 steps, against 59 for the FMAs alone; this form takes about 60.
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK, 4) k_lz_a(LzArgs<V> a, int j) {
  __shared__ V ws[SUBROWS];
  __shared__ double out[RSB_MAXC];
  lz_a_t<V, false>(a, j, blockIdx.x, ws, out);
}

template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK, 4) k_lz_b(LzArgs<V> a, int j) {
  __shared__ V ws[SUBROWS];
  __shared__ V cv[RSB_MAXC];
  __shared__ double out[RSB_MAXC];
  lz_b_t<V, false>(a, j, blockIdx.x, ws, cv, out);
}

template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_lz_c(LzArgs<V> a, int j, double breakdown) {
  __shared__ double sm[RSB_WARPS];
  __shared__ V cv[RSB_MAXC];
  __shared__ double out[1];
  __shared__ double sp[RED_FEW_DOUBLES(1)];
  lz_c_t<V, false>(a, j, breakdown, blockIdx.x, cv, sm, out, sp);
}

// Step D1 of the FP32 streaming path: z = L (src / nu_j) into the work vector
// AP (src stays as it is: D2 and D3 read it).  A CTA takes A1_ROWS consecutive rows
// of a tile (CTA b: tile b / nsub, part b % nsub of it).
// Bound: the latency of entry load, then gather, at HBM's rate (the entries, 4 B
// each, are read once; 9 of 10 gathers of src hit L1).  A thread has the 13 entries
// of half an interior row of a 26-neighbour mesh in flight, then their gathers, at
// 48 registers; the entries are loaded as streams (evicted first), which keeps src
// in L1 and the basis that D2 reads next in L2.  At 3.7M rows 80 us, of which the
// bytes take 61; eight entries at a time took 94, through L1 88.  (Also measured:
// the next entries loaded before the current gathers 84 us; entries brought to
// shared memory by bulk copies, which leaves L1 too small for src, 95 us.)
#define A1_P 13
#define A1_ROWS (4 * RSB_BLOCK)
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK, 5) k_lz_a1(LzArgs<V> a, int j, int nsub) {
  const int tix = (int)(blockIdx.x / (unsigned)nsub);
  const Tile t = a.tiles[tix];
  const long long p0 =
      (long long)t.row0 + (long long)(blockIdx.x - (unsigned)tix * nsub) * A1_ROWS;
  if (p0 >= t.row1) return;
  const int p1 = (int)min((long long)t.row1, p0 + A1_ROWS);
  const Unit& u = a.units[t.unit];
  if (u.status != U_ACTIVE || j >= u.msteps || j < u.j0) return;
  const V s = V(u.inu);
  const V* __restrict__ src = (j & 1) ? a.W1 : a.W0;
  unsigned long long pbytes = 0;
  for (int r = (int)p0 + threadIdx.x; r < p1; r += RSB_BLOCK) {
    const int64_t base = a.slice_ptr[r >> 5];
    const int width = (int)((a.slice_ptr[(r >> 5) + 1] - base) >> 5);
    const uint32_t* e = a.ent + base + (r & 31);
    const V xr = src[r];
    V acc = V(0);
    int k0 = 0;
    for (; k0 + A1_P <= width; k0 += A1_P) {
      uint32_t p[A1_P];
      V xv[A1_P];
#pragma unroll
      for (int i = 0; i < A1_P; ++i) p[i] = __ldcs(e + 32 * (k0 + i));
#pragma unroll
      for (int i = 0; i < A1_P; ++i) xv[i] = __ldg(src + ent_col(p[i]));
#pragma unroll
      for (int i = 0; i < A1_P; ++i) acc += V(ent_w(p[i])) * (xr - xv[i]);
    }
    if (k0 < width) {
      uint32_t p[A1_P];
      V xv[A1_P];
#pragma unroll
      for (int i = 0; i < A1_P; ++i) p[i] = k0 + i < width ? __ldcs(e + 32 * (k0 + i)) : 0u;
#pragma unroll
      for (int i = 0; i < A1_P; ++i) xv[i] = k0 + i < width ? __ldg(src + ent_col(p[i])) : xr;
#pragma unroll
      for (int i = 0; i < A1_P; ++i)
        if (k0 + i < width) acc += V(ent_w(p[i])) * (xr - xv[i]);
    }
    a.AP[r] = s * acc;
    if (a.pb_a) pbytes += 4ull * width + 2ull * sizeof(V);
  }
  if (a.pb_a) prof_add(a.pb_a, pbytes);
}

// Closing arithmetic of step D2 for one unit (every thread of the CTA takes
// part), from the reduced totals av = [a_b (b < nb), v.v] and gz = [g_b
// (b < nb), v.z] of src, scaled here in place to v = src / nu (inu = 1 / nu)
// and u0 = 1/sqrt(n) on its entry; sc[0..1] = rho, q_j.z and sk[0..j) = S_kj come
// back in shared memory (sk to be read after a CTA barrier, sc at once).  Ss: columns < j of S (row k at
// k * RSB_MAXM; S is symmetric).  The streaming kernel and the resident kernel
// both call this, so both modes produce the same numbers.
// On GB300 an FP64 warp instruction holds its SM sub-partition for 64 cycles
// however many lanes are active, so no sum is left to one lane: a.a and a.g
// are taken by one warp in a butterfly, every S_k.a by four lanes of the other
// warps.  (These are corrections of size |a| ~ 1e-7 to v.v, v.z and g.)  With
// the sums on single threads this took 11 us at j = 39, now 2 us.
__device__ __forceinline__ void d2_finish(double* av, double* gz, int nb, int nd, int j, double inu,
                                          double isn, const double* Ss, double* sc, double* sk) {
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  if (tid <= nb) {
    double x = av[tid] * (tid < nb ? inu : inu * inu);
    if (tid == 0) x *= isn;
    av[tid] = x;
  } else if (tid >= 64 && tid - 64 <= nb) {
    const int b = tid - 64;
    if (b == 0) gz[0] *= isn;
    if (b == nb) gz[nb] *= inu;
  }
  __syncthreads();
  const double* aq = av + 1 + nd;  // a on q_0..q_{j-1}
  if (w == 7) {
    double aa = 0.0, ag = 0.0;
    for (int b = lane; b < nb; b += 32) {
      aa = fma(av[b], av[b], aa);
      ag = fma(av[b], gz[b], ag);
    }
    aa = warp_sum(aa);
    ag = warp_sum(ag);
    const double rho2 = av[nb] - aa;
    // v has unit norm and |a| is at rounding level after its first pass; a
    // non-positive rho^2 means v lies in span(B) to working precision
    const double rho = rho2 > 0.0 ? sqrt(rho2) : 1e-300;
    const double qz = (gz[nb] - ag) / rho;
    if (lane == 0) {
      sc[0] = rho;
      sc[1] = qz;  // q_j.z
    }
  } else {
    // warps 0..4 cover k < 40, four lanes per k
    const int k = 8 * w + (lane & 7), part = lane >> 3;
    double sa = 0.0;
    if (k < j)
      for (int i = part; i < j; i += 4) sa = fma(Ss[i * RSB_MAXM + k], aq[i], sa);
    sa += __shfl_xor_sync(0xffffffffu, sa, 8);
    sa += __shfl_xor_sync(0xffffffffu, sa, 16);
    if (k < j && part == 0) sk[k] = gz[1 + nd + k] - sa;
  }
  __syncthreads();
  if (tid < j) sk[tid] = sk[tid] / sc[0];
}

// alpha = S_jj after d2_finish and a CTA barrier, by one warp (valid in every lane):
// nothing of the step waits for it.
__device__ __forceinline__ double d2_alpha(const double* av, int nd, int j, const double* sc,
                                           const double* sk) {
  const double* aq = av + 1 + nd;
  double sig = 0.0;
  for (int k = threadIdx.x & 31; k < j; k += 32) sig = fma(sk[k], aq[k], sig);
  return (sc[1] - warp_sum(sig)) / sc[0];
}

// Entries k < j of column and row j of S from the finished step D2.
__device__ __forceinline__ void d2_store_S(double* Sm, int j, const double* sk) {
  for (int k = threadIdx.x; k < j; k += RSB_BLOCK) {
    Sm[k * RSB_MAXM + j] = sk[k];
    Sm[j * RSB_MAXM + k] = sk[k];
  }
}

// ----------------------------------------------------------------------------
// Step D2 of the FP32 streaming path (second Gram-Schmidt pass delayed by one
// step, DCGS2: Swirydowicz, Langou, Ananthan, Yang and Thomas, "Low
// synchronization Gram-Schmidt and GMRES algorithms", 2020).  v = src / nu_j
// has been projected once against B = [u0, D, q_0..q_{j-1}]; z = L v (D1).
// One pass over q_0..q_{j-1}, src and z takes a = B^T v, g = B^T z,
// v.v and v.z; k_lz_close then forms
//   rho = sqrt(v.v - a.a)                  q_j = (v - B a) / rho
//   L q_j = (z - L B a) / rho, where L B a lies in span(B, q_j) up to
//   rounding (L u0 = 0; D holds eigenvector approximations; L q_i for i < j
//   is in span(q_0..q_j) by the Lanczos relation), so that
//   S_kj = q_k.L q_j = (g_k - sum_i S_ki a_i) / rho           (k < j)
//   S_jj = (q_j.z - sum_k S_kj a_k) / rho, q_j.z = (v.z - a.g) / rho,
// and the coefficients of D3.  Partials: [a_b (b < nb), v.v] then
// [g_b (b < nb), v.z], nb = 1 + nd + j.
// ----------------------------------------------------------------------------
// A basis value is used by one coefficient only, so nothing is staged: a warp owns
// up to D2_CPW coefficients (c = w + W i of the W warps the launch gives a tile) and
// streams their vectors through registers, D2_RG rows a lane at a time, with no CTA
// barrier anywhere; v and z, which every warp reads, come from L1.  A lane adds the
// rows lane, lane + 32, ... of the tile in order, whatever W is.
// Bound: HBM and L2 (es (j + 2) bytes a row), with the issue slots half busy (10 FP32
// instructions per coefficient and row).  At 3.7M rows, mean over j, 74 us, of which
// the bytes take 58; with chunks of the basis staged in shared memory by bulk copies
// (four CTAs of 8 warps per SM, two barriers a chunk) 97 us; three coefficients a warp
// 75 us, four 98 us.
#define D2_CPW 2
#define D2_RG 4
#define D2_MAXTHREADS (32 * ((RSB_MAXC + D2_CPW - 1) / D2_CPW))
static inline int d2_threads(int nc) { return 32 * ((nc + D2_CPW - 1) / D2_CPW); }

// One warp's NC coefficients over the tile's rows (r0: the lane's first row).  SP:
// some are u0 (kind 1) or FP64 deflation vectors (kind 2), not vectors in V.
template <typename V, int NC, bool SP>
__device__ __forceinline__ void d2_rows(const V* const (&q)[D2_CPW], const int (&kind)[D2_CPW],
                                        const double* const (&d)[D2_CPW], const V* v, const V* z,
                                        int r, int row1, Acc<V> (&av)[D2_CPW],
                                        Acc<V> (&az)[D2_CPW]) {
  // (r + 32 (D2_RG - 1) < row1 for every lane: the bound is the warp's first row)
  const int lane = threadIdx.x & 31;
  for (; r - lane + 32 * D2_RG <= row1; r += 32 * D2_RG) {
    V vs[D2_RG], zs[D2_RG], qs[NC][D2_RG];
#pragma unroll
    for (int i = 0; i < NC; ++i) {
      if (!SP || kind[i] == 3) {
#pragma unroll
        for (int g = 0; g < D2_RG; ++g) qs[i][g] = q[i][r + 32 * g];
      } else if (kind[i] == 2) {
#pragma unroll
        for (int g = 0; g < D2_RG; ++g) qs[i][g] = V(d[i][r + 32 * g]);
      } else {
#pragma unroll
        for (int g = 0; g < D2_RG; ++g) qs[i][g] = V(1);
      }
    }
#pragma unroll
    for (int g = 0; g < D2_RG; ++g) {
      vs[g] = v[r + 32 * g];
      zs[g] = z[r + 32 * g];
    }
#pragma unroll
    for (int g = 0; g < D2_RG; ++g)
#pragma unroll
      for (int i = 0; i < NC; ++i) {
        av[i].add(qs[i][g] * vs[g]);
        az[i].add(qs[i][g] * zs[g]);
      }
  }
  for (; r < row1; r += 32) {
    const V vs = v[r], zs = z[r];
#pragma unroll
    for (int i = 0; i < NC; ++i) {
      const V qs = !SP || kind[i] == 3 ? q[i][r] : kind[i] == 2 ? V(d[i][r]) : V(1);
      av[i].add(qs * vs);
      az[i].add(qs * zs);
    }
  }
}

template <typename V>
__global__ void __launch_bounds__(D2_MAXTHREADS, 2) k_lz_d2(LzArgs<V> a, int j) {
  const Tile t = a.tiles[blockIdx.x];
  const Unit& u = a.units[t.unit];
  if (u.status != U_ACTIVE || j >= u.msteps || j < u.j0) return;
  const int nd = u.nd;
  const int nb = 1 + nd + j;  // columns of B
  const int nc = nb + 1;      // plus v itself (v.v, v.z)
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, W = blockDim.x >> 5;
  const V* v = (j & 1) ? a.W1 : a.W0;
  const V* q[D2_CPW];
  const double* d[D2_CPW];
  int kind[D2_CPW];  // 1 ones (u0), 2 FP64 deflation vector, 3 vector
  bool sp = false;
#pragma unroll
  for (int i = 0; i < D2_CPW; ++i) {
    const int c = w + W * i;
    kind[i] = c == 0 ? 1 : c <= nd ? 2 : 3;
    sp |= kind[i] != 3;
    d[i] = c == 1 ? a.D0 : a.D1;
    q[i] = c >= nb ? v : a.Q + (long long)max(c - 1 - nd, 0) * a.N;
  }
  const int ncw = (nc - 1 - w) / W + 1;  // this warp's coefficients (W <= nc)
  Acc<V> av[D2_CPW], az[D2_CPW];
  const int r0 = t.row0 + lane;
  if (ncw == 2) {
    if (sp) d2_rows<V, 2, true>(q, kind, d, v, a.AP, r0, t.row1, av, az);
    else d2_rows<V, 2, false>(q, kind, d, v, a.AP, r0, t.row1, av, az);
  } else {
    if (sp) d2_rows<V, 1, true>(q, kind, d, v, a.AP, r0, t.row1, av, az);
    else d2_rows<V, 1, false>(q, kind, d, v, a.AP, r0, t.row1, av, az);
  }
  __syncwarp();
  // the warp's sums, converted to FP64 together
  float S[4] = {av[0].s, az[0].s, av[1].s, az[1].s}, C[4] = {av[0].c, az[0].c, av[1].c, az[1].c};
  const double sum = warp_totals<4>(S, C);
  const int k = lane >> 3, c = w + W * (k >> 1);
  if ((lane & 7) == 0 && c < nc)
    a.partials[(long long)((k & 1) ? nc + c : c) * a.stride + blockIdx.x] = sum;
  if (a.pb_a2 && threadIdx.x == 0)
    atomicAdd(a.pb_a2, (t.row1 - t.row0) * (sizeof(V) * (unsigned long long)(2 + j) + 8ull * nd));
}

// ----------------------------------------------------------------------------
// Closing of a step's dots (streaming path): the sums over the unit's tiles, then
//   CLOSE_A: c1 (FP64 step A);  CLOSE_B: c2 and column j of S (FP64 step B);
//   CLOSE_D2: d2_finish and the coefficients of D3.
// The tiles' partials of one unit are nt x 2 (j + 2) FP64 values: at 973 tiles and
// j = 39 their additions alone keep one SM's FP64 pipe busy for 20 us (45 us with the
// chain of loads, if the dots' last CTA does them while the chip idles).  So a kernel of
// its own spreads the coefficients over
// close_ctas() CTAs of the unit: one for a unit of few tiles, one per 32
// coefficients (a warp sums four, as in final_reduce) up to 192 tiles, one per
// four (final_reduce_few) above.  The order of every sum stays final_reduce's.
// ----------------------------------------------------------------------------
enum { CLOSE_A = 0, CLOSE_B = 1, CLOSE_D2 = 2 };

__host__ __device__ inline int close_per_cta(int nt, int ncoef) {
  return nt <= 32 ? ncoef : nt <= 192 ? 32 : 4;
}
__host__ __device__ inline int close_ctas(int nt, int ncoef) {
  const int per = close_per_cta(nt, ncoef);
  return (ncoef + per - 1) / per;
}
template <int MODE>
__host__ __device__ inline int close_ncoef(int nd, int j) {
  return MODE == CLOSE_D2 ? 2 * (2 + nd + j) : 2 + nd + j;
}

template <typename V, int MODE>
__global__ void __launch_bounds__(RSB_BLOCK) k_lz_close(LzArgs<V> a, int j, int G) {
  __shared__ double out[2 * RSB_MAXC + 2];
  __shared__ double sp[RED_FEW_DOUBLES(4)];
  const int ui = (int)(blockIdx.x / (unsigned)G), g = (int)(blockIdx.x - (unsigned)ui * G);
  Unit& u = a.units[ui];
  if (u.status != U_ACTIVE || j >= u.msteps || j < u.j0) return;
  const int nd = u.nd, nt = u.ntile;
  const int ncoef = close_ncoef<MODE>(nd, j);
  const int per = close_per_cta(nt, ncoef), gu = close_ctas(nt, ncoef);
  if (g >= gu) return;
  const int c0 = g * per, n = min(per, ncoef - c0);
  const double* P = a.partials + (long long)c0 * a.stride;
  double* Sm = unit_S(a.S, ui);
  __shared__ double Ss[MODE == CLOSE_D2 ? RSB_MAXM * RSB_MAXM : 1];
  if constexpr (MODE == CLOSE_D2) {
    for (int idx = threadIdx.x; idx < j * RSB_MAXM; idx += RSB_BLOCK) Ss[idx] = Sm[idx];
  }
  if (per == 4) {
    final_reduce_few(P, a.stride, u.tile0, nt, n, out, sp);
  } else {
    // final_reduce takes up to RSB_MAXC + 5 coefficients at once
    for (int k = 0; k < n; k += 32)
      final_reduce(P + (long long)k * a.stride, a.stride, u.tile0, nt, min(32, n - k), out + k);
  }
  if constexpr (MODE == CLOSE_A) {
    for (int k = threadIdx.x; k < n; k += RSB_BLOCK)
      u.c1[c0 + k] = c0 + k == 0 ? out[k] * u.isn : out[k];
  } else if constexpr (MODE == CLOSE_B) {
    for (int k = threadIdx.x; k < n; k += RSB_BLOCK) {
      const int c = c0 + k;
      u.c2[c] = c == 0 ? out[k] * u.isn : out[k];
      if (c > nd) {
        const double v = u.c1[c] + out[k];
        Sm[(c - 1 - nd) * RSB_MAXM + j] = v;
        Sm[j * RSB_MAXM + c - 1 - nd] = v;
      }
    }
  } else {
    const int nb = 1 + nd + j, nc = nb + 1;
    if (gu > 1) {  // the totals meet in c2 (a, v.v) and c1 (g, v.z); the last CTA goes on
      for (int k = threadIdx.x; k < n; k += RSB_BLOCK) {
        const int c = c0 + k;
        if (c < nc) u.c2[c] = out[k];
        else u.c1[c - nc] = out[k];
      }
      if (!last_cta(&u.cnt, gu)) return;
      for (int c = threadIdx.x; c < ncoef; c += RSB_BLOCK)
        out[c] = __ldcg(c < nc ? u.c2 + c : u.c1 + (c - nc));
    }
    __shared__ double sc[2], sk[RSB_MAXM];
    __syncthreads();
    const double inu = u.inu;
    d2_finish(out, out + nc, nb, nd, j, inu, u.isn, Ss, sc, sk);
    const double rho = sc[0];
    // D3: q_j = src / (nu rho) - sum_b (a_b / rho) b,
    //     w = z / rho - sum_b (g_b / rho) b - (q_j.z / rho) q_j
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (w == 4) {
      if (lane < 3) u.dz[lane] = (float)((lane == 0 ? inu : lane == 1 ? 1.0 : sc[1]) / rho);
    } else if (w < 4) {
      const int b = threadIdx.x & 63, h = threadIdx.x >> 6;
      if (b < nb) {
        const double x = out[h * nc + b] / rho;
        u.cf[b][h] = (float)(b == 0 ? x * u.isn : x);
      }
    }
    __syncthreads();
    d2_store_S(Sm, j, sk);
    if (w == 7) {
      const double alpha = d2_alpha(out, nd, j, sc, sk);
      if (lane == 0) {
        u.alpha[j] = alpha;
        Sm[j * RSB_MAXM + j] = alpha;
      }
    }
  }
}

// Step D3 of the FP32 streaming path: per row, q_j = src / (nu rho) - B a~ and
// w_{j+1} = z / rho - B g~ - (q_j.z / rho) q_j (a~ = a / rho, g~ = g / rho;
// one pass over the basis, two updates per loaded value); q_j goes to the
// basis, w_{j+1} to the other work vector, nu_{j+1} = ||w_{j+1}||.
// Bound: HBM and L2 (es (j + 4) bytes a row).  32 registers, so that eight CTAs
// (all 64 warps of an SM) hold loads in flight and 1216 tiles run at once: 81 us at
// 3.7M rows in 973 tiles, mean over j, of which the bytes take 62; with 16 loads a
// thread, 48 registers and five CTAs the last, nearly empty wave of tiles made it 106.
// The tiles are taken in the opposite order of D2, which has just streamed the same
// vectors: what it read last is still in L2 (4 % at 1M rows, nothing at 3.7M).
// T = 256 threads, or 128 (d3_half) where the tiles are short and more than the chip holds
// CTAs of 256.  A thread of 128 keeps the sums of rows t and t + 128 of every 256 apart,
// which are merged in the order of 256 threads, so both give the same bits.
#define D3_KB 4  // basis vectors a round
#define D3_RR 2  // rows a thread
template <typename V, int T>
__global__ void __launch_bounds__(T, 2048 / T) k_lz_d3(LzArgs<V> a, int j, double breakdown) {
  __shared__ double sm[RSB_WARPS];
  __shared__ __align__(16) V cc[RSB_MAXC][2];  // a~, g~
  __shared__ double out[1];
  __shared__ double sp[RED_FEW_DOUBLES(1)];
  const int tix = gridDim.x - 1 - blockIdx.x;
  const Tile t = a.tiles[tix];
  Unit& u = a.units[t.unit];
  if (u.status != U_ACTIVE || j >= u.msteps || j < u.j0) return;
  const int nd = u.nd;
  const int nb = 1 + nd + j;
  for (int k = threadIdx.x; k < nb; k += T) {
    const float2 x = *reinterpret_cast<const float2*>(u.cf[k]);
    cc[k][0] = x.x;
    cc[k][1] = x.y;
  }
  __syncthreads();
  const V ssrc = u.dz[0], sz = u.dz[1], sqz = u.dz[2];
  const V* src = (j & 1) ? a.W1 : a.W0;
  V* dst = (j & 1) ? a.W0 : a.W1;
  Acc<V> acc[RSB_BLOCK / T];
  for (int r0 = t.row0 + threadIdx.x; r0 < t.row1; r0 += D3_RR * T) {
    V q[D3_RR], w[D3_RR];
    bool ok[D3_RR];
#pragma unroll
    for (int rr = 0; rr < D3_RR; ++rr) {
      const int r = r0 + rr * T;
      ok[rr] = r < t.row1;
      q[rr] = ok[rr] ? ssrc * src[r] : V(0);
      w[rr] = ok[rr] ? sz * a.AP[r] : V(0);
      if (ok[rr] && unit_has(u, a.ckey, r)) {
        q[rr] -= cc[0][0];
        w[rr] -= cc[0][1];
      }
    }
    for (int l = 0; l < nd; ++l) {
      const double* d = (l == 0 ? a.D0 : a.D1) + r0;
#pragma unroll
      for (int rr = 0; rr < D3_RR; ++rr)
        if (ok[rr]) {
          const V dv = V(d[rr * T]);
          q[rr] -= cc[1 + l][0] * dv;
          w[rr] -= cc[1 + l][1] * dv;
        }
    }
    const V* qk = a.Q + r0;
    const V(*ck)[2] = cc + 1 + nd;
    int k = 0;
    for (; k + D3_KB <= j; k += D3_KB, qk += D3_KB * a.N, ck += D3_KB) {
      V qv[D3_KB][D3_RR];
#pragma unroll
      for (int i = 0; i < D3_KB; ++i)
#pragma unroll
        for (int rr = 0; rr < D3_RR; ++rr)
          qv[i][rr] = ok[rr] ? qk[i * a.N + rr * T] : V(0);
#pragma unroll
      for (int i = 0; i < D3_KB; ++i)
#pragma unroll
        for (int rr = 0; rr < D3_RR; ++rr) {
          q[rr] -= ck[i][0] * qv[i][rr];
          w[rr] -= ck[i][1] * qv[i][rr];
        }
    }
    for (; k < j; ++k, qk += a.N, ++ck)
#pragma unroll
      for (int rr = 0; rr < D3_RR; ++rr)
        if (ok[rr]) {
          const V b = qk[rr * T];
          q[rr] -= ck[0][0] * b;
          w[rr] -= ck[0][1] * b;
        }
#pragma unroll
    for (int rr = 0; rr < D3_RR; ++rr)
      if (ok[rr]) {
        const int r = r0 + rr * T;
        w[rr] -= sqz * q[rr];
        a.Q[(long long)j * a.N + r] = q[rr];
        dst[r] = w[rr];
        acc[rr % (RSB_BLOCK / T)].add(w[rr] * w[rr]);
      }
  }
  if (a.pb_b && threadIdx.x == 0)
    atomicAdd(a.pb_b, (t.row1 - t.row0) * (sizeof(V) * (unsigned long long)(4 + j) + 8ull * nd));
  const double sum = block_total_n<RSB_BLOCK / T>(acc, sm);
  if (threadIdx.x == 0) a.partials[tix] = sum;
  if (last_cta(&u.cnt, u.ntile)) {
    final_reduce_few(a.partials, a.stride, u.tile0, u.ntile, 1, out, sp);
    if (threadIdx.x == 0) {
      const double b = sqrt(out[0]);
      u.beta[j + 1] = b;
      u.inu = 1.0 / b;
      if (b <= breakdown * u.dmax) {  // invariant subspace: the cycle ends here
        u.msteps = j + 1;
        u.broke = 1;
      }
    }
  }
}

// ----------------------------------------------------------------------------
// Ritz pairs of S (K x K, K <= 40): parallel cyclic Jacobi in one CTA (FP64).
// Rounds of the round-robin ("circle") ordering rotate K/2 disjoint pairs at
// once; each rotation is the symmetric 2x2 Schur rotation (Golub & Van Loan
// §8.5).  Output: theta_0..theta_kk (ascending) and their eigenvectors as the
// Y columns of the unit's storage.
// ----------------------------------------------------------------------------
template <typename T>
struct JacShared {
  T A[RSB_MAXM][RSB_MAXM + 1];
  T Z[RSB_MAXM][RSB_MAXM + 1];
  // rotations (c, s) and index pairs (p | q << 8) of a round, and of the next one
  __align__(16) T cs[2][RSB_MAXM / 2][2];
  int pq[2][RSB_MAXM / 2];
  double red[RSB_WARPS];
  int rank[RSB_MAXM];
};

// T = double for the FP64 path; T = float for the mixed path, whose Lanczos
// vectors are FP32 (so FP32-accurate Ritz vectors lose nothing) and whose
// eigenvalue comes from the FP64 Rayleigh quotient at the end.
// Rotation (c, s) of the symmetric 2x2 Schur step for (a_pp, a_qq, a_pq)
// (Golub & Van Loan 8.5): t = sign(tau) / (|tau| + sqrt(1 + tau^2)) with
// tau = (a_qq - a_pp) / (2 a_pq), c = 1 / sqrt(1 + t^2), s = t c.  The angle t
// is taken in FP32 with fast division; c is normalised by Newton steps for
// 1 / sqrt(x) (c <- c (3 - x c^2) / 2) in the working precision, so that
// c^2 + s^2 = 1 to that precision.  Any t gives an orthogonal rotation; an
// FP32-accurate t leaves a_pq at ~1e-7 of its size instead of zero, which the
// following sweeps remove.  In FP64 this replaces two divisions and two square
// roots, long dependent chains on GB300's FP64 pipe.
// (an a_pq below FP32's range gives a non-finite angle: no rotation, t = 0)
__device__ __forceinline__ float jac_tan(float app, float aqq, float apq) {
  const float tau = __fdividef(aqq - app, 2.f * apq);
  const float t = __fdividef(copysignf(1.f, tau), fabsf(tau) + sqrtf(fmaf(tau, tau, 1.f)));
  return isfinite(t) ? t : 0.f;
}
__device__ __forceinline__ void jac_rotation(float app, float aqq, float apq, float& c, float& s) {
  const float t = jac_tan(app, aqq, apq);
  const float x = fmaf(t, t, 1.f);
  float r = rsqrtf(x);
  r = r * fmaf(-0.5f * x, r * r, 1.5f);
  c = r;
  s = t * r;
}
__device__ __forceinline__ void jac_rotation(double app, double aqq, double apq, double& c,
                                             double& s) {
  const double t = (double)jac_tan(0.f, (float)(aqq - app), (float)apq);
  const double x = fma(t, t, 1.0);
  double r = (double)rsqrtf((float)x);
  r = r * fma(-0.5 * x, r * r, 1.5);
  r = r * fma(-0.5 * x, r * r, 1.5);
  c = r;
  s = t * r;
}

// The rotations of round rnd into buffer b, by lanes < n2 / 2 of one warp
// (round-robin pairing: slot 0 holds index 0, the others rotate).
template <typename T>
__device__ __forceinline__ void jac_pairs(JacShared<T>& J, int b, int rnd, int n2, int K) {
  const int i = threadIdx.x & 31;
  if (i >= n2 / 2) return;
  int ia = i + rnd - 1, ib = n2 - 2 - i + rnd;
  if (ia >= n2 - 1) ia -= n2 - 1;
  if (ib >= n2 - 1) ib -= n2 - 1;
  int pa = i == 0 ? 0 : ia + 1;
  int pb = ib + 1;
  if (pa > pb) { const int tt = pa; pa = pb; pb = tt; }
  T cc = T(1), ss = T(0);
  const T apq = J.A[pa][pb];
  if (pb < K && apq != T(0)) jac_rotation(J.A[pa][pa], J.A[pb][pb], apq, cc, ss);
  J.pq[b][i] = pa | (pb << 8);
  J.cs[b][i][0] = cc;
  J.cs[b][i][1] = ss;
}

// The 2x2 block (rows of pair 1, columns of pair 2): the column rotation, then the
// row rotation.
template <typename T>
__device__ __forceinline__ void jac_block(T& a11, T& a12, T& a21, T& a22, T c1, T s1, T c2, T s2) {
  const T b11 = c2 * a11 - s2 * a12, b12 = s2 * a11 + c2 * a12;
  const T b21 = c2 * a21 - s2 * a22, b22 = s2 * a21 + c2 * a22;
  a11 = c1 * b11 - s1 * b21;
  a21 = s1 * b11 + c1 * b21;
  a12 = c1 * b12 - s1 * b22;
  a22 = s1 * b12 + c1 * b22;
}

// Sweeps of rotations of J.A (K x K, padded to n2) with J.Z <- J.Z R, until the
// off-diagonal mass is at most thr.
// Bound: the latency of a round (some 300 of them), in FP64 its arithmetic as well.
// A round is two phases: every thread updates its 2x2 blocks of A (all of its loads
// before its stores: the blocks are disjoint); then one warp computes the next round's
// rotations from the new A while the others apply this round's to Z, which the
// rotations do not need.  In FP32 every block is updated (both triangles, each with its
// own rounding), in FP64 the upper ones, which are mirrored.  With the rotations alone
// in a phase of their own and the updates one after the other, 40 x 40 took 200 us in
// FP32 and 1240 us in FP64.
template <typename T>
__device__ void jac_sweeps(JacShared<T>& J, int K, int n2, double thr) {
  const int tid = threadIdx.x, w = tid >> 5;
  const int np = n2 / 2;
  // this thread's blocks of A (pair i1 x pair i2; FP32: two, FP64: one with i1 <= i2)
  // and (pair, row) updates of Z (warps 1..7); fixed for the whole solve
  constexpr int NB = sizeof(T) == 8 ? 1 : 2;
  constexpr int NZ = (RSB_MAXM * RSB_MAXM / 2 + RSB_BLOCK - 33) / (RSB_BLOCK - 32);
  int i1[NB], i2[NB], zi[NZ], zr[NZ];
#pragma unroll
  for (int k = 0; k < NB; ++k) {
    const int task = tid + k * RSB_BLOCK;
    i1[k] = -1;
    i2[k] = 0;
    if constexpr (sizeof(T) == 8) {
      int row = 0, left = task;  // row-major upper triangle
      while (row < np && left >= np - row) left -= np - row++;
      if (row < np) {
        i1[k] = row;
        i2[k] = row + left;
      }
    } else if (task < np * np) {
      i1[k] = task / np;
      i2[k] = task - i1[k] * np;
    }
  }
#pragma unroll
  for (int k = 0; k < NZ; ++k) {
    const int zt = tid - 32 + k * (RSB_BLOCK - 32);
    zi[k] = -1;
    zr[k] = 0;
    if (w > 0 && zt < np * n2) {
      zi[k] = zt / n2;
      zr[k] = zt - zi[k] * n2;
    }
  }
  int buf = 0;
  if (w == 0) jac_pairs(J, 0, 0, n2, K);
  for (int sweep = 0; sweep < 20; ++sweep) {
    // off-diagonal mass against thr: a quick FP32 sum decides unless it lies within
    // 0.1 % of thr (its own error is below 1e-5), then the FP64 sum does
    float q = 0.f;
    for (int i = tid >> 3; i < K; i += RSB_BLOCK / 8)
      for (int k = i + 1 + (tid & 7); k < K; k += 8) {
        const float x = (float)J.A[i][k];
        q = fmaf(x, x, q);
      }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    if ((tid & 31) == 0) J.red[w] = (double)q;
    __syncthreads();
    float qs = 0.f;
#pragma unroll
    for (int i = 0; i < RSB_WARPS; ++i) qs += (float)J.red[i];
    const float thrf = (float)thr;
    __syncthreads();
    if (!(qs > 1.001f * thrf)) {
      bool stop = qs < 0.999f * thrf;
      if (!stop || sizeof(T) == 8) {  // (FP64: thr may be below FP32's range)
        double off = 0.0;
        for (int idx = tid; idx < K * K; idx += RSB_BLOCK) {
          const int i = idx / K, k = idx % K;
          if (i < k) off += (double)J.A[i][k] * (double)J.A[i][k];
        }
        off = block_sum(off, J.red);
        if (tid == 0) J.red[0] = off;
        __syncthreads();
        off = J.red[0];
        __syncthreads();
        stop = off <= thr;
      }
      if (stop) break;
    }
    for (int rnd = 0; rnd < n2 - 1; ++rnd) {
      T a11[NB], a12[NB], a21[NB], a22[NB];
      int p1[NB], q1[NB], p2[NB], q2[NB];
#pragma unroll
      for (int k = 0; k < NB; ++k)
        if (i1[k] >= 0) {
          const int x = J.pq[buf][i1[k]], y = J.pq[buf][i2[k]];
          p1[k] = x & 255;
          q1[k] = x >> 8;
          p2[k] = y & 255;
          q2[k] = y >> 8;
          a11[k] = J.A[p1[k]][p2[k]];
          a12[k] = J.A[p1[k]][q2[k]];
          a21[k] = J.A[q1[k]][p2[k]];
          a22[k] = J.A[q1[k]][q2[k]];
        }
#pragma unroll
      for (int k = 0; k < NB; ++k)
        if (i1[k] >= 0) {
          jac_block(a11[k], a12[k], a21[k], a22[k], J.cs[buf][i1[k]][0], J.cs[buf][i1[k]][1],
                    J.cs[buf][i2[k]][0], J.cs[buf][i2[k]][1]);
          J.A[p1[k]][p2[k]] = a11[k];
          J.A[q1[k]][p2[k]] = a21[k];
          J.A[p1[k]][q2[k]] = a12[k];
          J.A[q1[k]][q2[k]] = a22[k];
          if (sizeof(T) == 8 && i1[k] != i2[k]) {
            J.A[p2[k]][p1[k]] = a11[k];
            J.A[p2[k]][q1[k]] = a21[k];
            J.A[q2[k]][p1[k]] = a12[k];
            J.A[q2[k]][q1[k]] = a22[k];
          }
        }
      __syncthreads();
      if (w == 0) {
        jac_pairs(J, buf ^ 1, rnd + 1 < n2 - 1 ? rnd + 1 : 0, n2, K);
      } else {
        T zx[NZ], zy[NZ], c[NZ], sn[NZ];
        int pa[NZ], pb[NZ];
#pragma unroll
        for (int k = 0; k < NZ; ++k)
          if (zi[k] >= 0) {
            const int x = J.pq[buf][zi[k]];
            pa[k] = x & 255;
            pb[k] = x >> 8;
            c[k] = J.cs[buf][zi[k]][0];
            sn[k] = J.cs[buf][zi[k]][1];
            zx[k] = J.Z[zr[k]][pa[k]];
            zy[k] = J.Z[zr[k]][pb[k]];
          }
#pragma unroll
        for (int k = 0; k < NZ; ++k)
          if (zi[k] >= 0) {
            J.Z[zr[k]][pa[k]] = c[k] * zx[k] - sn[k] * zy[k];
            J.Z[zr[k]][pb[k]] = sn[k] * zx[k] + c[k] * zy[k];
          }
      }
      __syncthreads();
      buf ^= 1;
    }
  }
}

// J.A <- S (columns and rows < K, else 0), J.Z <- I; returns sum S_ij^2 to every thread.
template <typename T, bool CO>
__device__ double jac_load(const double* Sm, JacShared<T>& J, int K, int n2) {
  const int tid = threadIdx.x;
  for (int idx = tid; idx < n2 * n2; idx += RSB_BLOCK) {
    const int i = idx / n2, k = idx % n2;
    J.A[i][k] = (i < K && k < K) ? T(ldc<CO>(Sm + i * RSB_MAXM + k)) : T(0);
    J.Z[i][k] = i == k ? T(1) : T(0);
  }
  __syncthreads();
  double fro = 0.0;
  for (int idx = tid; idx < K * K; idx += RSB_BLOCK) {
    const double x = (double)J.A[idx / K][idx % K];
    fro += x * x;
  }
  fro = block_sum(fro, J.red);
  if (tid == 0) J.red[0] = fro;
  __syncthreads();
  fro = J.red[0];
  __syncthreads();
  return fro;
}

// FP64 eigenpairs of S from the FP32 ones: the iteration of Ogita and Aishima
// ("Iterative refinement for symmetric eigenvalue decomposition", 2018).  With
// R = I - X^T X and B = X^T S X, lambda_i = B_ii / (1 - R_ii), the correction
// X <- X + X E, E_ij = (B_ij + lambda_j R_ij) / (lambda_j - lambda_i), E_ii = R_ii / 2,
// squares the error; it ends when |E| is small enough that the square is below FP64's
// rounding.  False (uniform) when a correction is not small (eigenvalues too close for
// their FP32 vectors): the caller then takes the FP64 rotations.  On return J.Z holds
// the vectors and the diagonal of J.A the values.
// Bound: the FP64 rate, three to four K^3 products an iteration, two iterations as a
// rule, where the rotations take five to eight sweeps (816 us for 40 x 40, 183 for 16 x
// 16): 512-row box into 8 parts (14 polish cycles of 16) 12.4 -> 10.8 ms, FP64 Fiedler
// pair of 28k rows (7 cycles of 40) 15.0 -> 13.8 ms.
template <bool CO>
__device__ bool eig_refine(const double* Sm, JacShared<double>& J, int K, int n2) {
  constexpr int NE = (RSB_MAXM * RSB_MAXM + RSB_BLOCK - 1) / RSB_BLOCK;
  const int tid = threadIdx.x;
  double* lam = &J.cs[0][0][0];  // K values
  // X from the FP32 vectors (which lie in J.Z's place)
  {
    const JacShared<float>& F = *reinterpret_cast<const JacShared<float>*>(&J.Z[0][0]);
    float z[NE];
#pragma unroll
    for (int m = 0; m < NE; ++m) {
      const int idx = tid + m * RSB_BLOCK;
      z[m] = idx < K * K ? F.Z[idx / K][idx % K] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < NE; ++m) {
      const int idx = tid + m * RSB_BLOCK;
      if (idx < K * K) J.Z[idx / K][idx % K] = (double)z[m];
    }
    __syncthreads();
  }
  for (int it = 0; it < 6; ++it) {
    // J.A <- S X (S symmetric: read by rows l, coalesced over i)
    for (int idx = tid; idx < K * K; idx += RSB_BLOCK) {
      const int k = idx / K, i = idx % K;
      double x = 0.0;
#pragma unroll 4
      for (int l = 0; l < K; ++l) x = fma(ldc<CO>(Sm + l * RSB_MAXM + i), J.Z[l][k], x);
      J.A[i][k] = x;
    }
    __syncthreads();
    // B and R, entry (i, k) with i <= k in one thread
    double bij[NE], rij[NE];
#pragma unroll
    for (int m = 0; m < NE; ++m) {
      const int idx = tid + m * RSB_BLOCK;
      const int i = idx / K, k = idx % K;
      bij[m] = rij[m] = 0.0;
      if (idx < K * K && i <= k) {
        double x = 0.0, y = i == k ? 1.0 : 0.0;
        for (int l = 0; l < K; ++l) {
          const double z = J.Z[l][i];
          x = fma(z, J.A[l][k], x);
          y = fma(-z, J.Z[l][k], y);
        }
        bij[m] = x;
        rij[m] = y;
        if (i == k) lam[i] = x / (1.0 - y);
      }
    }
    __syncthreads();
    // E into J.A
    float emax = 0.f;
#pragma unroll
    for (int m = 0; m < NE; ++m) {
      const int idx = tid + m * RSB_BLOCK;
      const int i = idx / K, k = idx % K;
      if (idx < K * K && i <= k) {
        if (i == k) {
          J.A[i][i] = 0.5 * rij[m];
          const float e = fabsf((float)rij[m]);
          emax = e <= emax ? emax : e;  // (a NaN is kept)
        } else {
          // E_ik and E_ki; FP32 is accurate enough for a correction
          const float d = (float)(lam[k] - lam[i]);
          const float nik = (float)fma(lam[k], rij[m], bij[m]);
          const float nki = (float)fma(lam[i], rij[m], bij[m]);
          const bool zero = nik == 0.f && nki == 0.f;
          const float eik = zero ? 0.f : nik / d, eki = zero ? 0.f : -nki / d;
          J.A[i][k] = (double)eik;
          J.A[k][i] = (double)eki;
          const float e = fabsf(eik) + fabsf(eki);
          emax = e <= emax ? emax : e;
        }
      }
    }
    const bool bad = !(emax <= 1e-2f);
    const bool more = !(emax <= 2e-9f);
    const int any_bad = __syncthreads_or(bad);
    const int any_more = __syncthreads_or(more);
    if (any_bad) return false;
    // X <- X + X E
    double x[NE];
#pragma unroll
    for (int m = 0; m < NE; ++m) {
      const int idx = tid + m * RSB_BLOCK;
      const int i = idx / K, k = idx % K;
      x[m] = 0.0;
      if (idx < K * K) {
        double y = J.Z[i][k];
#pragma unroll 4
        for (int l = 0; l < K; ++l) y = fma(J.Z[i][l], J.A[l][k], y);
        x[m] = y;
      }
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < NE; ++m) {
      const int idx = tid + m * RSB_BLOCK;
      if (idx < K * K) J.Z[idx / K][idx % K] = x[m];
    }
    __syncthreads();
    if (!any_more) {
      if (tid < K) J.A[tid][tid] = lam[tid];
      __syncthreads();
      return true;
    }
  }
  return false;
}

// Ritz pairs of one unit: FP32 by rotations; FP64 by FP32 rotations and their
// refinement, or by FP64 rotations where that does not converge.
template <typename T, bool CO>
__device__ __noinline__ void lz_eig_u(Unit& u, double* Sm, JacShared<T>& J) {
  if (ldc<CO>(&u.status) != U_ACTIVE) return;
  const int tid = threadIdx.x;
  const int K = ldc<CO>(&u.msteps);
  const int n2 = K + (K & 1);
  if constexpr (sizeof(T) == 4) {
    const double fro = jac_load<T, CO>(Sm, J, K, n2);
    jac_sweeps(J, K, n2, fro * 1e-14);
  } else {
    static_assert(sizeof(J) - sizeof(J.A) >= sizeof(JacShared<float>), "FP32 workspace");
    JacShared<float>& F = *reinterpret_cast<JacShared<float>*>(&J.Z[0][0]);
    const double fro = jac_load<float, CO>(Sm, F, K, n2);
    jac_sweeps(F, K, n2, fro * 1e-14);
    __syncthreads();
    if (!eig_refine<CO>(Sm, J, K, n2)) {
      const double f = jac_load<T, CO>(Sm, J, K, n2);
      jac_sweeps(J, K, n2, f * 1e-30);
    }
  }
  __syncthreads();
  // ascending order (ties by index)
  if (tid < K) {
    const T e = J.A[tid][tid];
    int rk = 0;
    for (int l = 0; l < K; ++l) {
      const T f = J.A[l][l];
      rk += (f < e) || (f == e && l < tid);
    }
    J.rank[tid] = rk;
  }
  __syncthreads();
  const int kk = ldc<CO>(&u.broke) ? 0 : min(u.keep, K - 1);
  double* Ym = Sm + RSB_MAXM * RSB_MAXM;
  for (int idx = tid; idx < K * K; idx += RSB_BLOCK) {
    const int l = idx / K, i = idx % K;  // eigenvector i (unsorted), component l
    const int rk = J.rank[i];
    if (rk <= kk) Ym[l * RSB_MAXM + rk] = (double)J.Z[l][i];
  }
  if (tid < K) {
    const int rk = J.rank[tid];
    if (rk <= kk) u.th[rk] = (double)J.A[tid][tid];
    if (rk == 0) u.theta = (double)J.A[tid][tid];
  }
  if (tid == 0) u.kk = kk;
  __syncthreads();
}

template <typename T>
__global__ void __launch_bounds__(RSB_BLOCK) k_lz_eig(Unit* units, double* S, int nunits) {
  __shared__ JacShared<T> J;
  if ((int)blockIdx.x >= nunits) return;
  lz_eig_u<T, false>(units[blockIdx.x], unit_S(S, blockIdx.x), J);
}

// The Ritz-pair launch for other solvers of the library (block Lanczos).
int launch_lz_eig(int f32, Unit* units, double* S, int nunits, cudaStream_t s) {
  if (f32) k_lz_eig<float><<<nunits, RSB_BLOCK, 0, s>>>(units, S, nunits);
  else k_lz_eig<double><<<nunits, RSB_BLOCK, 0, s>>>(units, S, nunits);
  RSB_CKL("k_lz_eig");
  return RSB_OK;
}

extern "C" int rsb_probe_ritz(int f32, int K, int keep, const double* S, double* theta, double* Y) {
  if (K < 1 || K > RSB_MAXM || keep < 0 || keep >= K || keep > RSB_MAXKEEP || !S || !theta || !Y)
    return rsb_set_error(RSB_EINVAL, "ritz arguments");
  Unit u;
  memset(&u, 0, sizeof(u));
  u.status = U_ACTIVE;
  u.msteps = K;
  u.keep = keep;
  std::vector<double> h(RSB_SSTRIDE, 0.0);
  for (int i = 0; i < K; ++i)
    for (int k = 0; k < K; ++k) h[i * RSB_MAXM + k] = S[i * K + k];
  DevBuf du, ds;
  int rc;
  if ((rc = devbuf_reserve(du, sizeof(Unit))) || (rc = devbuf_reserve(ds, sizeof(double) * h.size())))
    return rc;
  cudaError_t e = cudaMemcpy(du.p, &u, sizeof(Unit), cudaMemcpyHostToDevice);
  if (!e) e = cudaMemcpy(ds.p, h.data(), sizeof(double) * h.size(), cudaMemcpyHostToDevice);
  if (!e) {
    rc = launch_lz_eig(f32, dptr<Unit>(du), dptr<double>(ds), 1, 0);
    e = cudaDeviceSynchronize();
  }
  if (!e) e = cudaMemcpy(&u, du.p, sizeof(Unit), cudaMemcpyDeviceToHost);
  if (!e) e = cudaMemcpy(h.data(), ds.p, sizeof(double) * h.size(), cudaMemcpyDeviceToHost);
  cudaFree(du.p);
  cudaFree(ds.p);
  if (rc || e) return rc ? rc : rsb_set_cuda_error(e, "rsb_probe_ritz");
  for (int i = 0; i <= keep; ++i) {
    theta[i] = u.th[i];
    for (int l = 0; l < K; ++l)
      Y[l * (keep + 1) + i] = h[RSB_MAXM * RSB_MAXM + l * RSB_MAXM + i];
  }
  return RSB_OK;
}

// ----------------------------------------------------------------------------
// Ritz vector and thick-restart basis (per row, in place): y = Q s_0 into Y;
// q_i <- Q s_i for i < kk; the residual direction moves to W[kk & 1] so that
// the next cycle's first step reads it.  A unit whose cycle cap this cycle
// reaches is not restarted: only y is formed.
//
// Bound: HBM in FP32 (K vectors read, kk + 1 written), the FP64 rate in FP64
// ((kk + 1) K FMAs a row).  The coefficients are converted to the vector type
// once per CTA and kept in shared memory, NA at a time (a row of YSTR values per
// basis vector, read as broadcasts): a basis value is loaded once and updates NA
// accumulators, RITZ_R rows per thread.  Every output sums over the basis vectors
// in ascending order.
// 40 FP32 vectors of 3.7M rows and 9 outputs 0.17 ms, 16 FP64 vectors 0.90; with
// every row thread converting each coefficient itself (an FP64 conversion per
// coefficient and warp) 2.36 and 3.08 ms.
// ----------------------------------------------------------------------------
#define YSTR 20  // RSB_MAXKEEP + 1, rounded up to 16 bytes

// The coefficients of y and of the kk kept vectors, in the vector type.
template <typename V, bool CO>
__device__ __forceinline__ void ritz_stage(const double* Ym, int K, int kk, V* Ys) {
  for (int idx = threadIdx.x; idx < K * (kk + 1); idx += RSB_BLOCK) {
    const int l = idx / (kk + 1), i = idx % (kk + 1);
    Ys[l * YSTR + i] = V(ldc<CO>(Ym + l * RSB_MAXM + i));
  }
  __syncthreads();
}

// NA outputs of RR rows (rows r0 + rr * RSB_BLOCK; ok[rr]: inside the tile) from
// the vectors q + l * ld.
template <typename V, int NA, int RR>
__device__ __forceinline__ void ritz_rows(const V* q, long long ld, int K, const V* Ys,
                                          const bool (&ok)[RR], V (&acc)[NA][RR]) {
#pragma unroll
  for (int i = 0; i < NA; ++i)
#pragma unroll
    for (int rr = 0; rr < RR; ++rr) acc[i][rr] = V(0);
  constexpr int LU = 16 / (RR * (int)sizeof(V) / 4);  // basis vectors in flight
  for (int l0 = 0; l0 < K; l0 += LU) {
    V qv[LU][RR];
#pragma unroll
    for (int u = 0; u < LU; ++u)
#pragma unroll
      for (int rr = 0; rr < RR; ++rr)
        qv[u][rr] = (ok[rr] && l0 + u < K) ? q[(long long)(l0 + u) * ld + rr * RSB_BLOCK] : V(0);
#pragma unroll
    for (int u = 0; u < LU; ++u)
      if (l0 + u < K) {
#pragma unroll
        for (int i = 0; i < NA; ++i) {
          const V c = Ys[(l0 + u) * YSTR + i];
#pragma unroll
          for (int rr = 0; rr < RR; ++rr) acc[i][rr] += c * qv[u][rr];
        }
      }
  }
}

// rows of one tile: q points at row row0 of vector 0 (global or shared memory)
template <typename V, int NA, int RR>
__device__ __forceinline__ void ritz_tile(V* q, long long ld, int K, int kk, int nr, const V* Ys,
                                          V* y) {
  for (int b = 0; b < nr; b += RR * RSB_BLOCK) {
    const int r0 = b + threadIdx.x;
    bool ok[RR];
#pragma unroll
    for (int rr = 0; rr < RR; ++rr) ok[rr] = r0 + rr * RSB_BLOCK < nr;
    V acc[NA][RR];
    ritz_rows<V, NA, RR>(q + r0, ld, K, Ys, ok, acc);
#pragma unroll
    for (int rr = 0; rr < RR; ++rr)
      if (ok[rr]) {
        y[r0 + rr * RSB_BLOCK] = acc[0][rr];
#pragma unroll
        for (int i = 0; i < NA; ++i)
          if (i < kk) q[(long long)i * ld + r0 + rr * RSB_BLOCK] = acc[i][rr];
      }
  }
}

// The number of accumulators: y alone, up to the default 8 kept vectors, or all.
template <typename V>
__device__ __forceinline__ void ritz_dispatch(V* q, long long ld, int K, int kk, int nr,
                                              const V* Ys, V* y) {
  constexpr int RR = sizeof(V) == 4 ? 4 : 2;
  if (kk == 0) ritz_tile<V, 1, RR>(q, ld, K, kk, nr, Ys, y);
  else if (kk <= 8) ritz_tile<V, 9, RR>(q, ld, K, kk, nr, Ys, y);
  else ritz_tile<V, RSB_MAXKEEP + 1, RR / 2>(q, ld, K, kk, nr, Ys, y);
}

template <typename V, bool CO>
__device__ __forceinline__ void lz_ritz_t(const LzArgs<V>& a, int tix, V* Ys) {
  const Tile t = a.tiles[tix];
  const Unit& u = a.units[t.unit];
  if (ldc<CO>(&u.status) != U_ACTIVE) return;
  const int K = ldc<CO>(&u.msteps);
  // the last cycle under the cap ends converged or capped: nothing is kept
  const int kk = ldc<CO>(&u.cycles) + 1 >= u.maxcycles ? 0 : ldc<CO>(&u.kk);
  ritz_stage<V, CO>(unit_S(a.S, t.unit) + RSB_MAXM * RSB_MAXM, K, kk, Ys);
  ritz_dispatch<V>(a.Q + t.row0, a.N, K, kk, t.row1 - t.row0, Ys, a.Y + t.row0);
  const V* wl = (K & 1) ? a.W1 : a.W0;
  V* wn = (kk & 1) ? a.W1 : a.W0;
  if (kk > 0 && wn != wl)
    for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) wn[r] = wl[r];
  if (CO && a.pb_a && threadIdx.x == 0)
    atomicAdd(a.pb_a, (unsigned long long)(t.row1 - t.row0) * sizeof(V) * (K + kk + 1));
}

// Residual of y with theta, plus the projection dots of y against the fixed
// basis.  mode 0: Lanczos cycle end (decides convergence); mode 1: the start
// vector only (no residual).
template <typename V, bool CO>
__device__ __forceinline__ void lz_resid_t(const LzArgs<V>& a, const V* y, int mode, int tix,
                                           double* sm, double* out, double* sp) {
  const Tile t = a.tiles[tix];
  Unit& u = a.units[t.unit];
  if (ldc<CO>(&u.status) != U_ACTIVE) return;
  const int nd = u.nd;
  const V th = V(ldc<CO>(&u.theta));
  Acc<V> r2, y2, ys, d0, d1;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    const V yr = y[r];
    if (mode == 0) {
      const V res = spmv_row<V, CO>(a.slice_ptr, a.ent, y, r, yr) - th * yr;
      r2.add(res * res);
    }
    y2.add(yr * yr);
    ys.add(yr);
    if (nd > 0) d0.add(V(a.D0[r]) * yr);
    if (nd > 1) d1.add(V(a.D1[r]) * yr);
  }
  if (CO && a.pb_a && threadIdx.x == 0) {
    unsigned long long b = 0;
    for (int r = t.row0; r < t.row1; ++r) b += 4ull * row_width(a.slice_ptr, r);
    b += (unsigned long long)(t.row1 - t.row0) * (sizeof(V) + 8ull * nd);
    atomicAdd(a.pb_a, b);
  }
  double v[5] = {r2.get(), y2.get(), ys.get(), d0.get(), d1.get()};
  const int nv = 3 + nd;
  for (int c = 0; c < nv; ++c) {
    const double sum = block_sum(v[c], sm);
    if (threadIdx.x == 0) a.partials[(long long)c * a.stride + tix] = sum;
  }
  if (last_cta(&u.cnt, u.ntile)) {
    final_reduce_few(a.partials, a.stride, u.tile0, u.ntile, nv, out, sp);
    if (threadIdx.x == 0) {
      u.ynorm2 = out[1];
      u.cp[0] = out[2] * u.isn;
      for (int l = 0; l < nd; ++l) u.cp[1 + l] = out[3 + l];
      if (mode == 0) {
        u.resid = sqrt(out[0] / out[1]);
        u.cycles += 1;
        atomicAdd((unsigned long long*)a.stat_cycles, 1ull);
        int st = U_ACTIVE;
        if (u.resid <= u.tolabs) st = U_CONVERGED;
        else if (u.cycles >= u.maxcycles) st = U_CAPPED;
        if (st != U_ACTIVE) {
          u.status = st;
          atomicSub(a.n_active, 1);
        } else if (u.kk > 0) {
          // thick restart: the kept Ritz vectors occupy q_0..q_{kk-1}; the next
          // cycle starts at step kk from the residual direction
          u.beta0 = u.beta[u.msteps];
          u.inu = 1.0 / u.beta0;
          u.j0 = u.kk;
          u.msteps = u.m;
          atomicMin(a.jmin, u.kk);
        } else {
          u.j0 = 0;  // explicit restart from y (proj2/proj3 follow)
          atomicMin(a.jmin, 0);
        }
      }
    }
    if (mode == 0) {
      __syncthreads();
      // next cycle's S = diag(kept Ritz values); explicit restarts clear it all
      if (u.status == U_ACTIVE) {
        double* Sm = unit_S(a.S, t.unit);
        const int kk = u.kk;
        for (int idx = threadIdx.x; idx < RSB_MAXM * RSB_MAXM; idx += RSB_BLOCK) {
          const int i = idx / RSB_MAXM, k = idx % RSB_MAXM;
          Sm[idx] = (i == k && i < kk) ? u.th[i] : 0.0;
        }
      }
    }
  }
}

// Explicit restart only (a cycle that ended on an invariant subspace without
// converging): y -= B cp (in place); dots of the result against B -> c2.
template <typename V, bool CO>
__device__ __forceinline__ void proj2_t(const LzArgs<V>& a, V* y, int tix, double* sm,
                                        double* out, double* sp) {
  const Tile t = a.tiles[tix];
  Unit& u = a.units[t.unit];
  if (ldc<CO>(&u.status) != U_ACTIVE || ldc<CO>(&u.j0) != 0) return;
  const int nd = u.nd;
  const double cp0 = ldc<CO>(&u.cp[0]), cp1 = ldc<CO>(&u.cp[1]), cp2 = ldc<CO>(&u.cp[2]);
  Acc<V> ys, d0, d1;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    V v = y[r];
    if (unit_has(u, a.ckey, r)) v -= V(cp0 * u.isn);
    if (nd > 0) v -= V(cp1) * V(a.D0[r]);
    if (nd > 1) v -= V(cp2) * V(a.D1[r]);
    y[r] = v;
    ys.add(v);
    if (nd > 0) d0.add(V(a.D0[r]) * v);
    if (nd > 1) d1.add(V(a.D1[r]) * v);
  }
  if (CO && a.pb_a && threadIdx.x == 0)
    atomicAdd(a.pb_a, (unsigned long long)(t.row1 - t.row0) * (2 * sizeof(V) + 8ull * nd));
  double v[3] = {ys.get(), d0.get(), d1.get()};
  const int nv = 1 + nd;
  for (int c = 0; c < nv; ++c) {
    const double sum = block_sum(v[c], sm);
    if (threadIdx.x == 0) a.partials[(long long)c * a.stride + tix] = sum;
  }
  if (last_cta(&u.cnt, u.ntile)) {
    final_reduce_few(a.partials, a.stride, u.tile0, u.ntile, nv, out, sp);
    if (threadIdx.x == 0) {
      u.c2[0] = out[0] * u.isn;
      for (int l = 0; l < nd; ++l) u.c2[1 + l] = out[1 + l];
    }
  }
}

// w0 = y - B c2 (second pass), beta0 = ||w0||; a cycle starts at step 0.
template <typename V, bool CO>
__device__ __forceinline__ void proj3_t(const LzArgs<V>& a, const V* y, int tix, double* sm,
                                        double* out, double* sp) {
  const Tile t = a.tiles[tix];
  Unit& u = a.units[t.unit];
  if (ldc<CO>(&u.status) != U_ACTIVE || ldc<CO>(&u.j0) != 0) return;
  const int nd = u.nd;
  const double c20 = ldc<CO>(&u.c2[0]), c21 = ldc<CO>(&u.c2[1]), c22 = ldc<CO>(&u.c2[2]);
  Acc<V> acc;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    V v = y[r];
    if (unit_has(u, a.ckey, r)) v -= V(c20 * u.isn);
    if (nd > 0) v -= V(c21) * V(a.D0[r]);
    if (nd > 1) v -= V(c22) * V(a.D1[r]);
    a.W0[r] = v;
    acc.add(v * v);
  }
  if (CO && a.pb_a && threadIdx.x == 0)
    atomicAdd(a.pb_a, (unsigned long long)(t.row1 - t.row0) * (2 * sizeof(V) + 8ull * nd));
  const double sum = block_sum(acc.get(), sm);
  if (threadIdx.x == 0) a.partials[tix] = sum;
  if (last_cta(&u.cnt, u.ntile)) {
    final_reduce_few(a.partials, a.stride, u.tile0, u.ntile, 1, out, sp);
    if (threadIdx.x == 0) {
      u.beta0 = sqrt(out[0]);
      u.inu = 1.0 / u.beta0;
      u.msteps = u.m;
      u.broke = 0;
    }
  }
}

template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_lz_ritz(LzArgs<V> a) {
  __shared__ __align__(16) V Ys[RSB_MAXM * YSTR];
  lz_ritz_t<V, false>(a, blockIdx.x, Ys);
}
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_lz_resid(LzArgs<V> a, const V* __restrict__ y,
                                                        int mode) {
  __shared__ double sm[RSB_WARPS];
  __shared__ double out[3 + RSB_MAXD];
  __shared__ double sp[RED_FEW_DOUBLES(3 + RSB_MAXD)];
  lz_resid_t<V, false>(a, y, mode, blockIdx.x, sm, out, sp);
}
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_proj2(LzArgs<V> a, V* __restrict__ y) {
  __shared__ double sm[RSB_WARPS];
  __shared__ double out[1 + RSB_MAXD];
  __shared__ double sp[RED_FEW_DOUBLES(1 + RSB_MAXD)];
  proj2_t<V, false>(a, y, blockIdx.x, sm, out, sp);
}
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_proj3(LzArgs<V> a, const V* __restrict__ y) {
  __shared__ double sm[RSB_WARPS];
  __shared__ double out[1];
  __shared__ double sp[RED_FEW_DOUBLES(1)];
  proj3_t<V, false>(a, y, blockIdx.x, sm, out, sp);
}

// ----------------------------------------------------------------------------
// Persistent cooperative kernel: one whole Lanczos cycle (steps j0..M-1, the
// Ritz pairs of S, Ritz vector and restart basis, residual) in one launch.
// CTAs walk the tiles grid-stride (the same CTA owns the same tiles in every
// phase); phases are separated by the bounded grid barrier; reductions keep
// the last-CTA scheme, whose result the barrier publishes.
// ----------------------------------------------------------------------------
template <typename V>
union CycleShared {
  JacShared<V> J;
  double wsd[SUBROWS];
  double red[RED_FEW_DOUBLES(RED_FEW)];
};

template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK, 2)
    k_lz_cycle(LzArgs<V> a, int jstart, int M, double breakdown, int ntiles, int nunits,
               GridBar* gb) {
  __shared__ CycleShared<V> sh;
  __shared__ double out[RSB_MAXC];
  __shared__ double sm[RSB_WARPS];
  __shared__ V cv[RSB_MAXC];
  V* ws = reinterpret_cast<V*>(sh.wsd);
  double* red = sh.red;
  const unsigned G = gridDim.x;
  for (int j = jstart; j < M; ++j) {
    for (int t = blockIdx.x; t < ntiles; t += G) lz_a_t<V, true>(a, j, t, ws, out);
    if (!grid_sync(gb, G)) return;
    for (int t = blockIdx.x; t < ntiles; t += G) lz_b_t<V, true>(a, j, t, ws, cv, out);
    if (!grid_sync(gb, G)) return;
    for (int t = blockIdx.x; t < ntiles; t += G) lz_c_t<V, true>(a, j, breakdown, t, cv, sm, out, red);
    if (!grid_sync(gb, G)) return;
  }
  for (int u = blockIdx.x; u < nunits; u += G) lz_eig_u<V, true>(a.units[u], unit_S(a.S, u), sh.J);
  if (!grid_sync(gb, G)) return;
  for (int t = blockIdx.x; t < ntiles; t += G) {
    lz_ritz_t<V, true>(a, t, ws);  // RSB_MAXM * YSTR <= SUBROWS values
    __syncthreads();
  }
  if (!grid_sync(gb, G)) return;
  for (int t = blockIdx.x; t < ntiles; t += G) lz_resid_t<V, true>(a, a.Y, 0, t, sm, out, red);
  if (!grid_sync(gb, G)) return;
  for (int t = blockIdx.x; t < ntiles; t += G) proj2_t<V, true>(a, a.Y, t, sm, out, red);
  if (!grid_sync(gb, G)) return;
  for (int t = blockIdx.x; t < ntiles; t += G) proj3_t<V, true>(a, a.Y, t, sm, out, red);
}

// ----------------------------------------------------------------------------
// Resident persistent solve (launch mode 3).  When every tile of the level can
// own one co-resident CTA and the tile's rows of the basis fit in that CTA's
// shared memory (the level's basis is at most the chip's shared memory: the
// 131,072-row level with 40 FP32 vectors is 21 MB over 256 CTAs), one
// cooperative launch runs every cycle of the solve.  The Gram-Schmidt passes
// then read q_0..q_j from shared memory; global memory carries the SpMV
// operand, the reduction partials and the per-unit scalars.  Steps, their
// order, the per-thread accumulation order and the reductions are those of
// the streaming kernels above, so both modes give the same numbers.
// Shared layout: JacShared | coefficients (FP64, and in the vector type) | w
// (z) of the tile | v of the tile (FP32) | deflation vectors of the tile |
// Q[k * trs + rl].
// ----------------------------------------------------------------------------
__host__ __device__ constexpr size_t res_align(size_t b) { return (b + 15) & ~(size_t)15; }

template <typename V>
__host__ __device__ constexpr size_t res_smem_bytes(int M, int trs) {
  return res_align(sizeof(JacShared<V>)) + res_align(2 * sizeof(double) * RSB_MAXC) +
         res_align(2 * sizeof(V) * RSB_MAXC) + 2 * res_align(sizeof(V) * (size_t)trs) +
         res_align(sizeof(V) * RSB_MAXD * (size_t)trs) + sizeof(V) * (size_t)M * (size_t)trs;
}

// What bounds a step here is latency: a chain of L2 round trips (SpMV, partials, two
// or three barriers) and of FP64 operations, each of which holds an SM sub-partition
// for 64 cycles.  So units synchronise on their own barriers and run their cycles
// independently of one another; FP64 work is done by whole warps, once (the closing
// divisions of a step by every warp take 1.7 us); S_jj, which nothing waits for, is
// computed while the norms travel; a unit of one tile exchanges nothing through global
// memory but the SpMV operand.  FP32 step of the 512-row mesh about 11 us, with whole-grid
// barriers and the closing on single threads 21.5; the 131072-row box into 64 parts 113 and
// 167 ms.
//
// Dots of [1, D, q_0..] with the tile's w: the coefficient split across warps
// and the per-lane row order of tile_dots.
template <typename V>
__device__ __forceinline__ void res_dots(const Tile& t, int nd, int nc, const V* Qs,
                                         const V* Ds, int trs, const V* ws,
                                         Acc<V> (&acc)[MAXCW]) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nr = t.row1 - t.row0;
#pragma unroll
  for (int i = 0; i < MAXCW; ++i) {
    const int c = w + RSB_WARPS * i;
    if (c < nc) {
      if (c == 0) {
        for (int rl = lane; rl < nr; rl += 32) acc[i].add(V(1) * ws[rl]);
      } else if (c <= nd) {
        const V* d = Ds + (size_t)(c - 1) * trs;
        for (int rl = lane; rl < nr; rl += 32) acc[i].add(d[rl] * ws[rl]);
      } else {
        const V* q = Qs + (size_t)(c - 1 - nd) * trs;
        for (int rl = lane; rl < nr; rl += 32) acc[i].add(q[rl] * ws[rl]);
      }
    }
  }
}

// w -= [1/sqrt(n), D, q_0..q_{nq-1}] cv, in the order of gs_update_rows (cv:
// the coefficients in the vector type; in_unit: the row belongs to the unit).
template <typename V>
__device__ __forceinline__ V res_upd_row(const V* cv, int nd, int nq, const V* Qs,
                                         const V* Ds, int trs, int rl, bool in_unit, V w) {
  if (in_unit) w -= cv[0];
  for (int l = 0; l < nd; ++l) w -= cv[1 + l] * Ds[(size_t)l * trs + rl];
  const V* cq = cv + 1 + nd;
  for (int k = 0; k < nq; ++k) w -= cq[k] * Qs[(size_t)k * trs + rl];
  return w;
}

// (out: where the dots of a unit of one tile go, else null)
template <typename V>
__device__ __forceinline__ void res_store_dots(double* P, long long stride, int nc,
                                               Acc<V> (&acc)[MAXCW], int tix, double* out) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < MAXCW; ++i) {
    const int c = w + RSB_WARPS * i;
    if (c < nc) {
      const double s = warp_total(acc[i]);
      if (lane == 0) {
        if (out) out[c] = s;
        else P[(long long)c * stride + tix] = s;
      }
    }
  }
}

// The step phases write per-tile partials into P; after the unit's barrier every CTA
// of the unit holds the same totals.  Consecutive phases alternate between partial
// buffers: a buffer is rewritten only after a barrier that follows every CTA's
// reduction of its previous contents.
//
// Totals of ncoef coefficients of the unit in out (shared memory).  One tile: the
// dots are in out already.  Up to RED_SMALL tiles every CTA reduces them itself (at 96
// tiles the additions take as long as a barrier); above, coefficient c is summed by
// CTA c of the unit alone, and the totals (in tot, ncoef doubles of the unit) are
// exchanged over one more barrier (256 tiles reduced by every CTA took 14.5 us).
__device__ __forceinline__ bool res_totals(const double* P, long long stride, const Unit& u, int tix,
                                           int ncoef, double* out, double* tot, double* scratch,
                                           UnitBar& ub, int fw) {
  const int nt = u.ntile;
  if (nt == 1) return true;
  if (nt <= RED_SMALL) {
    final_reduce_small(P, stride, u.tile0, nt, ncoef, out);
    return true;
  }
  // (nt > 96 >= ncoef: every CTA has at most one)
  const int c = tix - u.tile0;
  if (c < ncoef) {
    final_reduce_few(P + (long long)c * stride, stride, u.tile0, nt, 1, out, scratch, fw);
    if (threadIdx.x == 0) tot[c] = out[0];
  }
  if (!ub.sync()) return false;
  for (int k = threadIdx.x; k < ncoef; k += RSB_BLOCK) out[k] = __ldcg(tot + k);
  __syncthreads();
  return true;
}

// A(j): q_j = src * s into shared memory, w = L q_j, dots [1, D, q_0..q_j]^T w.
template <typename V>
__device__ void res_a(const LzArgs<V>& a, int j, V s, int tix, const Tile& t, const Unit& u,
                      V* Qs, const V* Ds, int trs, V* ws, double* P, double* out) {
  const int nr = t.row1 - t.row0;
  const V* src = (j & 1) ? a.W1 : a.W0;
  const int nd = u.nd;
  const int nc = 2 + nd + j;
  unsigned long long pbytes = 0;
  for (int rl = threadIdx.x; rl < nr; rl += RSB_BLOCK) {
    const int r = t.row0 + rl;
    const V xr = src[r];
    ws[rl] = s * spmv_row_batched<V>(a.slice_ptr, a.ent, src, r, xr);
    Qs[(size_t)j * trs + rl] = s * xr;
    if (a.pb_a)
      pbytes += 4ull * row_width(a.slice_ptr, r) + sizeof(V) * (unsigned long long)(4 + j) +
                8ull * nd;
  }
  __syncthreads();
  Acc<V> acc[MAXCW];
  res_dots<V>(t, nd, nc, Qs, Ds, trs, ws, acc);
  res_store_dots<V>(P, a.stride, nc, acc, tix, out);
  if (a.pb_a) prof_add(a.pb_a, pbytes);
}

// B(j): w -= basis c1, dots of the result (second pass).
template <typename V>
__device__ void res_b(const LzArgs<V>& a, int j, int tix, const Tile& t, int nd, bool masked,
                      uint64_t key, const V* Qs, const V* Ds, int trs, V* ws, const V* cv,
                      double* P, double* out) {
  const int nr = t.row1 - t.row0;
  const int nc = 2 + nd + j;
  unsigned long long pbytes = 0;
  for (int rl = threadIdx.x; rl < nr; rl += RSB_BLOCK) {
    const bool in_unit = !masked || a.ckey[t.row0 + rl] == key;
    ws[rl] = res_upd_row<V>(cv, nd, j + 1, Qs, Ds, trs, rl, in_unit, ws[rl]);
    if (a.pb_b) pbytes += sizeof(V) * (unsigned long long)(3 + j) + 8ull * nd;
  }
  __syncthreads();
  Acc<V> acc[MAXCW];
  res_dots<V>(t, nd, nc, Qs, Ds, trs, ws, acc);
  res_store_dots<V>(P, a.stride, nc, acc, tix, out);
  if (a.pb_b) prof_add(a.pb_b, pbytes);
}

// C(j): w -= basis c2 into W[(j + 1) & 1] (the next SpMV operand), ||w||^2.
template <typename V>
__device__ double res_c(const LzArgs<V>& a, int j, const Tile& t, int nd, bool masked,
                        uint64_t key, const V* Qs, const V* Ds, int trs, const V* ws,
                        const V* cv, double* sm) {
  const int nr = t.row1 - t.row0;
  V* dst = (j & 1) ? a.W0 : a.W1;
  Acc<V> acc;
  unsigned long long pbytes = 0;
  for (int rl = threadIdx.x; rl < nr; rl += RSB_BLOCK) {
    const bool in_unit = !masked || a.ckey[t.row0 + rl] == key;
    const V w = res_upd_row<V>(cv, nd, j + 1, Qs, Ds, trs, rl, in_unit, ws[rl]);
    dst[t.row0 + rl] = w;
    acc.add(w * w);
    if (a.pb_c) pbytes += sizeof(V) * (unsigned long long)(3 + j) + 8ull * nd;
  }
  if (a.pb_c) prof_add(a.pb_c, pbytes);
  return block_total(acc, sm);
}

// FP32 steps with the delayed second pass (D1-D3 of the streaming kernels,
// in their order).  D1(j): v = src rows into vs, z = L (src / nu) into ws; two rows
// of a thread at once, eight entries of each in flight.  own: the unit is this tile,
// so every gather is served from vs.
template <typename V>
__device__ void res_d1(const LzArgs<V>& a, int j, V s, const Tile& t, V* vs, V* ws, bool own) {
  const int nr = t.row1 - t.row0;
  const V* src = (j & 1) ? a.W1 : a.W0;
  for (int rl = threadIdx.x; rl < nr; rl += RSB_BLOCK) vs[rl] = __ldcg(src + t.row0 + rl);
  if (own) __syncthreads();
  unsigned long long pbytes = 0;
  for (int rl = threadIdx.x; rl < nr; rl += 2 * RSB_BLOCK) {
    int width[2];
    const uint32_t* e[2];
    V xr[2], acc[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int r = t.row0 + rl + i * RSB_BLOCK;
      width[i] = 0;
      e[i] = a.ent;
      xr[i] = acc[i] = V(0);
      if (r < t.row1) {
        const int64_t base = a.slice_ptr[r >> 5];
        width[i] = (int)((a.slice_ptr[(r >> 5) + 1] - base) >> 5);
        e[i] = a.ent + base + (r & 31);
        xr[i] = vs[rl + i * RSB_BLOCK];
        if (a.pb_a) pbytes += 4ull * width[i] + 2ull * sizeof(V);
      }
    }
    const int wmax = max(width[0], width[1]);
    for (int k0 = 0; k0 < wmax; k0 += 8) {
      uint32_t p[2][8];
      V xv[2][8];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int k = 0; k < 8; ++k)
          p[i][k] = k0 + k < width[i] ? __ldg(e[i] + 32 * (k0 + k)) : 0u;
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          xv[i][k] = xr[i];
          if (k0 + k < width[i])
            xv[i][k] = own ? vs[(int)ent_col(p[i][k]) - t.row0] : src[ent_col(p[i][k])];
        }
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (k0 + k < width[i]) acc[i] += V(ent_w(p[i][k])) * (xr[i] - xv[i][k]);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (rl + i * RSB_BLOCK < nr) ws[rl + i * RSB_BLOCK] = s * acc[i];
  }
  if (a.pb_a) prof_add(a.pb_a, pbytes);
  __syncthreads();
}

// D2(j): dots of v (vs) and z (ws) with [1, D, q_0..q_{j-1}] and with v, in the
// per-lane order of k_lz_d2 (partials [a_b, v.v] then [g_b, v.z]; out: as in
// res_store_dots).  A warp takes its coefficients two at a time.
template <typename V>
__device__ void res_d2(const LzArgs<V>& a, int j, int tix, const Tile& t, int nd, const V* Qs,
                       const V* Ds, int trs, const V* vs, const V* ws, double* P, double* out) {
  const int nr = t.row1 - t.row0;
  const int nb = 1 + nd + j;
  const int nc = nb + 1;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float S[16], C[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) S[i] = C[i] = 0.f;
#pragma unroll
  for (int i = 0; i < MAXCW; i += 2) {
    const int c0 = w + RSB_WARPS * i, c1 = c0 + RSB_WARPS;
    if (c0 >= nc) break;
    // basis vector, FP64 deflation vector in the vector type, v itself; u0 (ones)
    // takes the place of a vector by its value
    auto vec = [&](int c) {
      return c >= nb ? vs : c > nd ? Qs + (size_t)(c - 1 - nd) * trs : Ds + (size_t)max(c - 1, 0) * trs;
    };
    const V* q0 = vec(c0);
    const V* q1 = vec(c1);
    Acc<V> a0, z0, a1, z1;
    if (c0 == 0) {
      for (int rl = lane; rl < nr; rl += 32) {
        const V x = vs[rl], z = ws[rl], y = q1[rl];
        a0.add(x);
        z0.add(z);
        a1.add(y * x);
        z1.add(y * z);
      }
    } else if (c1 < nc) {
#pragma unroll 4
      for (int rl = lane; rl < nr; rl += 32) {
        const V x = vs[rl], z = ws[rl], y0 = q0[rl], y1 = q1[rl];
        a0.add(y0 * x);
        z0.add(y0 * z);
        a1.add(y1 * x);
        z1.add(y1 * z);
      }
    } else {
#pragma unroll 4
      for (int rl = lane; rl < nr; rl += 32) {
        const V y0 = q0[rl];
        a0.add(y0 * vs[rl]);
        z0.add(y0 * ws[rl]);
      }
    }
    S[2 * i] = a0.s;
    C[2 * i] = a0.c;
    S[2 * i + 1] = z0.s;
    C[2 * i + 1] = z0.c;
    S[2 * i + 2] = a1.s;
    C[2 * i + 2] = a1.c;
    S[2 * i + 3] = z1.s;
    C[2 * i + 3] = z1.c;
  }
  const double sum = warp_totals<16>(S, C);
  const int k = lane >> 1, c = w + RSB_WARPS * (k >> 1);
  if ((lane & 1) == 0 && c < nc) {
    const int cc = (k & 1) ? nc + c : c;
    if (out) out[cc] = sum;
    else P[(long long)cc * a.stride + tix] = sum;
  }
  if (a.pb_a2 && threadIdx.x == 0)
    atomicAdd(a.pb_a2, nr * (sizeof(V) * (unsigned long long)(2 + j) + 8ull * nd));
}

// D3(j): q_j = ssrc v - B ca into Qs, w = sz z - B cg - sqz q_j into
// W[(j + 1) & 1], ||w||^2 (the per-row order of k_lz_d3; cc: the pairs ca, cg; dz:
// ssrc, sz, sqz).  Returns the tile's sum in thread 0.
template <typename V>
__device__ double res_d3(const LzArgs<V>& a, int j, const Tile& t, int nd, bool masked, uint64_t key,
                         V* Qs, const V* Ds, int trs, const V* vs, const V* ws, const V (*cc)[2],
                         const V* dz, double* sm) {
  const int nr = t.row1 - t.row0;
  V* dst = (j & 1) ? a.W0 : a.W1;
  const V ssrc = dz[0], sz = dz[1], sqz = dz[2];
  Acc<V> acc;
  for (int rl = threadIdx.x; rl < nr; rl += 2 * RSB_BLOCK) {
    const bool two = rl + RSB_BLOCK < nr;
    const int r2 = two ? rl + RSB_BLOCK : rl;  // (a lone row is computed twice, kept once)
    V q[2] = {ssrc * vs[rl], ssrc * vs[r2]};
    V w[2] = {sz * ws[rl], sz * ws[r2]};
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (!masked || a.ckey[t.row0 + (i ? r2 : rl)] == key) {
        q[i] -= cc[0][0];
        w[i] -= cc[0][1];
      }
    for (int l = 0; l < nd; ++l) {
      const V d0 = Ds[(size_t)l * trs + rl], d1 = Ds[(size_t)l * trs + r2];
      q[0] -= cc[1 + l][0] * d0;
      w[0] -= cc[1 + l][1] * d0;
      q[1] -= cc[1 + l][0] * d1;
      w[1] -= cc[1 + l][1] * d1;
    }
    const V(*ck)[2] = cc + 1 + nd;
#pragma unroll 8
    for (int k = 0; k < j; ++k) {
      const V b0 = Qs[(size_t)k * trs + rl], b1 = Qs[(size_t)k * trs + r2];
      const V ka = ck[k][0], kg = ck[k][1];
      q[0] -= ka * b0;
      w[0] -= kg * b0;
      q[1] -= ka * b1;
      w[1] -= kg * b1;
    }
    w[0] -= sqz * q[0];
    Qs[(size_t)j * trs + rl] = q[0];
    dst[t.row0 + rl] = w[0];
    acc.add(w[0] * w[0]);
    if (two) {
      w[1] -= sqz * q[1];
      Qs[(size_t)j * trs + r2] = q[1];
      dst[t.row0 + r2] = w[1];
      acc.add(w[1] * w[1]);
    }
  }
  if (a.pb_b && threadIdx.x == 0)
    atomicAdd(a.pb_b, nr * (sizeof(V) * (unsigned long long)(4 + j) + 8ull * nd));
  return block_total(acc, sm);
}

// coefficients of a finished reduction: c[0] carries the 1/sqrt(n) of u0 (as
// the streaming kernels store it); cv the same in the vector type, cv[0]
// already times 1/sqrt(n) again (the u0 component of the update)
template <typename V>
__device__ __forceinline__ void res_coef(const double* out, int nc, double isn, double* c,
                                         V* cv) {
  for (int k = threadIdx.x; k < nc; k += RSB_BLOCK) {
    const double v = k == 0 ? out[0] * isn : out[k];
    c[k] = v;
    cv[k] = k == 0 ? V(v * isn) : V(v);
  }
  __syncthreads();
}

// Ritz vector y = Q s_0 into Y and the kept vectors q_i <- Q s_i (i < kk) in
// shared memory (lz_ritz_t on the resident basis); the residual direction moves
// to W[kk & 1].
template <typename V>
__device__ void res_ritz(const LzArgs<V>& a, const Tile& t, const Unit& u, V* Qs, int trs,
                         V* Ys) {
  if (ldc<true>(&u.status) != U_ACTIVE) return;
  const int nr = t.row1 - t.row0;
  const int K = ldc<true>(&u.msteps);
  const int kk = ldc<true>(&u.cycles) + 1 >= u.maxcycles ? 0 : ldc<true>(&u.kk);
  ritz_stage<V, true>(unit_S(a.S, t.unit) + RSB_MAXM * RSB_MAXM, K, kk, Ys);
  ritz_dispatch<V>(Qs, trs, K, kk, nr, Ys, a.Y + t.row0);
  const V* wl = (K & 1) ? a.W1 : a.W0;
  V* wn = (kk & 1) ? a.W1 : a.W0;
  if (kk > 0 && wn != wl)
    for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) wn[r] = __ldcg(wl + r);
  if (a.pb_a && threadIdx.x == 0)
    atomicAdd(a.pb_a, (unsigned long long)nr * sizeof(V) * (K + kk + 1));
}

// The norm of the new vector from the tiles' sums (mine: this tile's, thread 0's):
// beta_{j+1}, 1 / beta_{j+1} and the vector-type scale in shared memory; the unit's
// first CTA records it and the end of the cycle on an invariant subspace.  Returns
// true when the cycle ends here.
template <typename V>
__device__ __forceinline__ bool res_norm(const LzArgs<V>& a, Unit& u, int j, int tix, double breakdown,
                                         double mine, const double* Pn, double* out,
                                         double* scratch, double* beta, double* inu, V* scale,
                                         int fw) {
  if (u.ntile > 1) {
    final_reduce_few(Pn, a.stride, u.tile0, u.ntile, 1, out, scratch, fw);
  } else {
    if (threadIdx.x == 0) out[0] = mine;
    __syncthreads();
  }
  if ((int)threadIdx.x == 32 * fw) {
    const double b = sqrt(out[0]);
    *beta = b;
    *inu = 1.0 / b;
    *scale = V(*inu);
    if (tix == u.tile0) {
      u.beta[j + 1] = b;
      if (b <= breakdown * u.dmax) {  // invariant subspace: the cycle ends here
        u.msteps = j + 1;
        u.broke = 1;
      }
    }
  }
  __syncthreads();
  return *beta <= breakdown * u.dmax;
}

template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK, 2)
    k_lz_res(LzArgs<V> a, int M, int trs, double breakdown, int maxcyc, GridBar* gb) {
  extern __shared__ __align__(16) unsigned char res_sh[];
  JacShared<V>& J = *reinterpret_cast<JacShared<V>*>(res_sh);
  size_t off = res_align(sizeof(JacShared<V>));
  double* c1 = reinterpret_cast<double*>(res_sh + off);
  double* c2 = c1 + RSB_MAXC;
  off += res_align(2 * sizeof(double) * RSB_MAXC);
  V* cv = reinterpret_cast<V*>(res_sh + off);  // two coefficient sets (FP32: pairs)
  V(*cc)[2] = reinterpret_cast<V(*)[2]>(cv);
  off += res_align(2 * sizeof(V) * RSB_MAXC);
  V* ws = reinterpret_cast<V*>(res_sh + off);
  off += res_align(sizeof(V) * (size_t)trs);
  V* vs = reinterpret_cast<V*>(res_sh + off);
  off += res_align(sizeof(V) * (size_t)trs);
  V* Ds = reinterpret_cast<V*>(res_sh + off);
  off += res_align(sizeof(V) * RSB_MAXD * (size_t)trs);
  V* Qs = reinterpret_cast<V*>(res_sh + off);
  __shared__ double out[2 * RSB_MAXC + 2];
  __shared__ double dsc[2], dsk[RSB_MAXM];
  __shared__ double sm[RSB_WARPS];
  __shared__ double beta_sh, inu_sh;
  __shared__ V scale_sh, dz[3];
  // the Jacobi workspace is free outside lz_eig_u: the copy of S during the steps and
  // the scratch of the reductions between them
  static_assert(sizeof(JacShared<V>) >= sizeof(double) * RSB_MAXM * RSB_MAXM, "copy of S");
  static_assert(sizeof(JacShared<V>) >= sizeof(double) * RED_FEW_DOUBLES(RED_FEW), "scratch");
  double* Ssh = reinterpret_cast<double*>(res_sh);
  double* red = Ssh;
  // (the steps' own reductions must leave Ssh alone)
  __shared__ double red1[RED_FEW_DOUBLES(1)];
  const int tix = blockIdx.x;
  const Tile t = a.tiles[tix];
  Unit& u = a.units[t.unit];
  if (__ldcg(&u.status) != U_ACTIVE) return;
  const int nr = t.row1 - t.row0;
  const int nd = u.nd;
  const bool masked = u.masked;
  const uint64_t key = u.key;
  const double isn = u.isn;
  const bool first = tix == u.tile0;
  const int fw = fp64_warp();
  UnitBar ub(&u.gbar, u.ntile, __ldcg(&gb->count), gb);
  double* const direct = u.ntile == 1 ? out : nullptr;
  // partial buffers: FP32 dots in the first two, FP64 dots in each in turn, the norms
  // apart, so that no CTA rewrites rows another CTA may still reduce
  double* const Pb[2] = {a.partials, a.partials + (long long)RSB_MAXC * a.stride};
  double* const Pn = a.partials + (long long)(2 * RSB_MAXC) * a.stride;
  // exchanged totals of a unit of more than RED_SMALL tiles (RSB_MAXC a tile)
  double* const tot = a.partials + (3 * a.stride + u.tile0) * (long long)RSB_MAXC;
  // the tile's deflation vectors in the vector type, once per solve
  for (int l = 0; l < nd; ++l) {
    const double* d = l == 0 ? a.D0 : a.D1;
    for (int rl = threadIdx.x; rl < nr; rl += RSB_BLOCK) Ds[(size_t)l * trs + rl] = V(d[t.row0 + rl]);
  }
  for (int cyc = 0; cyc < maxcyc; ++cyc) {
    // the unit's step state, tracked identically by all of its CTAs
    const int j0 = __ldcg(&u.j0);
    int msteps = min(__ldcg(&u.msteps), M);
    if (threadIdx.x == 0) {
      beta_sh = __ldcg(&u.beta0);
      inu_sh = __ldcg(&u.inu);
      scale_sh = V(inu_sh);
    }
    // every CTA of the unit keeps its own copy of S during the steps
    if constexpr (sizeof(V) == 4) {
      const double* Sm = unit_S(a.S, t.unit);
      for (int idx = threadIdx.x; idx < RSB_MAXM * RSB_MAXM; idx += RSB_BLOCK)
        Ssh[idx] = __ldcg(Sm + idx);
    }
    __syncthreads();
    for (int j = j0; j < msteps; ++j) {
      double mine;
      if constexpr (sizeof(V) == 4) {
        // FP32: the streaming kernels' steps D1-D3 (second pass delayed)
        const int nb = 1 + nd + j;
        const int nc = nb + 1;
        res_d1<V>(a, j, scale_sh, t, vs, ws, direct != nullptr);
        res_d2<V>(a, j, tix, t, nd, Qs, Ds, trs, vs, ws, a.partials, direct);
        if (!ub.sync()) return;
        if (!res_totals(a.partials, a.stride, u, tix, 2 * nc, out, tot, red1, ub, fw)) return;
        const double inu = inu_sh;
        d2_finish(out, out + nc, nb, nd, j, inu, isn, Ssh, dsc, dsk);
        const double rho = dsc[0];
        const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
        if (w < 4) {
          const int k = threadIdx.x & 63, h = threadIdx.x >> 6;
          if (k < nb) {
            const double x = out[h * nc + k] / rho;
            cc[k][h] = k == 0 ? V(x * isn) : V(x);
          }
        } else if (w == 4 && lane < 3) {
          dz[lane] = V((lane == 0 ? inu : lane == 1 ? 1.0 : dsc[1]) / rho);
        }
        __syncthreads();
        mine = res_d3<V>(a, j, t, nd, masked, key, Qs, Ds, trs, vs, ws, cc, dz, sm);
        if (threadIdx.x == 0) Pn[tix] = mine;
        ub.arrive();
        // while the norms travel: column j of S
        d2_store_S(Ssh, j, dsk);
        if (first) d2_store_S(unit_S(a.S, t.unit), j, dsk);
        if (w == 7) {
          const double alpha = d2_alpha(out, nd, j, dsc, dsk);
          if (lane == 0) {
            Ssh[j * RSB_MAXM + j] = alpha;
            if (first) {
              unit_S(a.S, t.unit)[j * RSB_MAXM + j] = alpha;
              u.alpha[j] = alpha;
            }
          }
        }
        if (!ub.wait()) return;
        if (res_norm<V>(a, u, j, tix, breakdown, mine, Pn, out, red1, &beta_sh, &inu_sh, &scale_sh, fw))
          msteps = j + 1;
      } else {
        const int nc = 2 + nd + j;
        res_a<V>(a, j, scale_sh, tix, t, u, Qs, Ds, trs, ws, Pb[0], direct);
        if (!ub.sync()) return;
        if (!res_totals(Pb[0], a.stride, u, tix, nc, out, tot, red1, ub, fw)) return;
        res_coef<V>(out, nc, isn, c1, cv);
        res_b<V>(a, j, tix, t, nd, masked, key, Qs, Ds, trs, ws, cv, Pb[1], direct);
        if (!ub.sync()) return;
        if (!res_totals(Pb[1], a.stride, u, tix, nc, out, tot + RSB_MAXC, red1, ub, fw)) return;
        res_coef<V>(out, nc, isn, c2, cv + RSB_MAXC);
        if (first) {  // column j of S = Q^T L Q
          double* Sm = unit_S(a.S, t.unit);
          for (int k = threadIdx.x; k <= j; k += RSB_BLOCK) {
            const double v = c1[1 + nd + k] + c2[1 + nd + k];
            Sm[k * RSB_MAXM + j] = v;
            Sm[j * RSB_MAXM + k] = v;
          }
        }
        mine = res_c<V>(a, j, t, nd, masked, key, Qs, Ds, trs, ws, cv + RSB_MAXC, sm);
        if (threadIdx.x == 0) Pn[tix] = mine;
        if (!ub.sync()) return;
        if (res_norm<V>(a, u, j, tix, breakdown, mine, Pn, out, red1, &beta_sh, &inu_sh, &scale_sh, fw))
          msteps = j + 1;
      }
    }
    if (first) lz_eig_u<V, true>(u, unit_S(a.S, t.unit), J);
    if (!ub.sync()) return;
    res_ritz<V>(a, t, u, Qs, trs, &J.Z[0][0]);
    if (!ub.sync()) return;
    lz_resid_t<V, true>(a, a.Y, 0, tix, sm, out, red);
    if (!ub.sync()) return;
    if (__ldcg(&u.status) != U_ACTIVE) return;
    if (__ldcg(&u.j0) == 0) {  // explicit restart from y
      proj2_t<V, true>(a, a.Y, tix, sm, out, red);
      if (!ub.sync()) return;
      proj3_t<V, true>(a, a.Y, tix, sm, out, red);
      if (!ub.sync()) return;
    }
  }
}

// Start vector into Y: hash of gid on unit rows (or a given vector), 0 elsewhere.
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_start(LzArgs<V> a, uint64_t sd, const double* from64,
                                                     const float* from32) {
  const Tile t = a.tiles[blockIdx.x];
  const Unit& u = a.units[t.unit];
  if (u.status != U_ACTIVE) return;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    V v = V(0);
    if (unit_has(u, a.ckey, r)) {
      if (from64) v = V(from64[r]);
      else if (from32) v = V(from32[r]);
      else v = V(start_value(sd, a.gid[r]));
    }
    a.Y[r] = v;
  }
}

// ----------------------------------------------------------------------------
// solve set-up per unit
// ----------------------------------------------------------------------------
// mode: number of deflation vectors nd (0, 1, 2).  A unit joins the solve when
// it is valid, its space orthogonal to 1 and the deflation vectors is not
// empty, and (nd > 0) it found a cluster of size nd so far.
// Units whose dimension dim = n - 1 - nd lies outside [dim_lo, dim_hi] are left
// as they are (another solver takes them).
__global__ void k_solve_init(Unit* units, int nunits, int nd, int krylov, int maxcycles, double tol,
                             int require_cluster, int keep, long long dim_lo, long long dim_hi,
                             int* n_active) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nunits) return;
  Unit& u = units[i];
  const long long dim = u.n - 1 - nd;
  if (u.valid && dim > 0 && (dim < dim_lo || dim > dim_hi)) return;
  u.status = U_IDLE;
  if (!u.valid) return;
  if (dim <= 0) return;
  if (require_cluster && u.ncand != nd) return;
  u.nd = nd;
  u.m = (int)min((long long)krylov, dim);
  u.msteps = u.m;
  u.j0 = 0;
  u.kk = 0;
  u.broke = 0;
  u.keep = keep;
  u.cycles = 0;
  u.maxcycles = maxcycles;
  u.tolabs = tol * u.dmax;
  u.inner = 0;
  u.inner_total = 0;
  u.cg_done = 0;
  u.gbar = 0;
  u.status = U_ACTIVE;
  atomicAdd(n_active, 1);
}

// ----------------------------------------------------------------------------
// host drivers
// ----------------------------------------------------------------------------
template <typename V>
static LzArgs<V> make_args(const LevelGraph& G, const Tile* tiles, int ntiles, Unit* units,
                           const uint64_t* ckey, SolveBufs& B) {
  LzArgs<V> a;
  a.slice_ptr = G.slice_ptr;
  a.ent = G.ent;
  a.gid = G.gid;
  a.tiles = tiles;
  a.units = units;
  a.ckey = ckey;
  a.Q = (V*)B.Q;
  a.N = B.N;
  a.W0 = (V*)B.W0;
  a.W1 = (V*)B.W1;
  a.Y = (V*)B.Y;
  a.X = (V*)B.X;
  a.R = (V*)B.R;
  a.P = (V*)B.P;
  a.AP = (V*)B.AP;
  a.D0 = B.D[0];
  a.D1 = B.D[1];
  a.partials = B.partials;
  a.stride = ntiles;
  a.n_active = B.n_active;
  a.stat_cycles = B.stat_cycles;
  a.pb_a = prof_bytes(PROF_LZ_A);
  a.pb_a2 = prof_bytes(PROF_LZ_A2);
  a.pb_b = prof_bytes(PROF_LZ_B);
  a.pb_c = prof_bytes(PROF_LZ_C);
  a.pb_cg = prof_bytes(PROF_CG_AP);
  a.S = B.S;
  a.jmin = B.jmin;
  return a;
}

int solver_setup(Unit* units, int nunits, int nd, int krylov, int maxcycles, double tol,
                 int require_cluster, int keep, SolveBufs& B, cudaStream_t s, long long dim_lo,
                 long long dim_hi) {
  B.maxcycles = maxcycles;
  RSB_CK(cudaMemsetAsync(B.n_active, 0, sizeof(int), s));
  k_solve_init<<<(nunits + 127) / 128, 128, 0, s>>>(units, nunits, nd, krylov, maxcycles, tol,
                                                    require_cluster, keep, dim_lo, dim_hi,
                                                    B.n_active);
  RSB_CKL("k_solve_init");
  return RSB_OK;
}

static int read_active(SolveBufs& B, cudaStream_t s, int* out) {
  RSB_CK(cudaMemcpyAsync(B.h_active, B.n_active, sizeof(int), cudaMemcpyDeviceToHost, s));
  if (B.jmin) RSB_CK(cudaMemcpyAsync(B.h_active + 2, B.jmin, sizeof(int), cudaMemcpyDeviceToHost, s));
  if (B.gb) RSB_CK(cudaMemcpyAsync(B.h_active + 1, &B.gb->err, sizeof(int), cudaMemcpyDeviceToHost, s));
  RSB_CK(cudaStreamSynchronize(s));
  prof_collect();
  *out = *B.h_active;
  if (B.gb && B.h_active[1]) return rsb_set_error(RSB_ETIMEOUT, "a bounded device wait gave up");
  return RSB_OK;
}

template <typename V>
static int lz_start(LzArgs<V>& a, int ntiles, uint64_t sd, const double* from64,
                    const float* from32, cudaStream_t s) {
  k_start<V><<<ntiles, RSB_BLOCK, 0, s>>>(a, sd, from64, from32);
  RSB_CKL("k_start");
  k_lz_resid<V><<<ntiles, RSB_BLOCK, 0, s>>>(a, a.Y, 1);
  RSB_CKL("k_lz_resid(start)");
  k_proj2<V><<<ntiles, RSB_BLOCK, 0, s>>>(a, a.Y);
  RSB_CKL("k_proj2");
  k_proj3<V><<<ntiles, RSB_BLOCK, 0, s>>>(a, a.Y);
  RSB_CKL("k_proj3");
  return RSB_OK;
}

// D3 in CTAs of 128 threads?  The CTA of a short tile lives for a chain of loads and a
// reduction whatever its rows, so one wave of sixteen a SM beats two of eight, and half
// the threads of 256 idle on tiles of up to 128 rows; long tiles, and full ones of more
// than two waves, are better off with 256.  Sum of D3 over three cycles in CTAs of 256 and
// 128, ms (8 x 152 = 1216 CTAs of 256 a wave): 1300 tiles of 512 rows 3.05 : 2.66, 2600
// 5.11 : 5.29, 3200 4.72 : 5.08, 6000 9.64 : 9.23; 4000 of 240 rows 3.91 : 2.69; 6000 of
// 351 on average 7.34 : 6.75; the levels of 3.7M rows (tiles of 1536 and more) 37.7 : 40.9,
// of 15.9M rows 139 : 154.
static bool d3_half(int64_t rows, int ntiles, int trmax, int nsm) {
  const int64_t wave = 8ll * nsm;
  return trmax <= 2 * RSB_BLOCK && ntiles > wave && (ntiles <= 2 * wave || rows < 384ll * ntiles);
}

template <typename V>
static int lz_cycle(LzArgs<V>& a, int ntiles, int nunits, int M, double breakdown, int trmax,
                    int ntmax, int nd, bool half, cudaStream_t s) {
  // CTAs per tile of step D1
  const int nsub = std::max(1, (trmax + A1_ROWS - 1) / A1_ROWS);
  for (int j = 0; j < M; ++j) {
    int pi = prof_before(PROF_LZ_A, s);
    if constexpr (sizeof(V) == 4) {  // FP32: bandwidth-bound; CGS2 with the second pass delayed
      k_lz_a1<V><<<ntiles * nsub, RSB_BLOCK, 0, s>>>(a, j, nsub);
      RSB_CKL("k_lz_a1");
      prof_after(pi, s);
      pi = prof_before(PROF_LZ_A2, s);
      k_lz_d2<V><<<ntiles, d2_threads(2 + nd + j), 0, s>>>(a, j);
      RSB_CKL("k_lz_d2");
      const int G = close_ctas(ntmax, close_ncoef<CLOSE_D2>(nd, j));
      k_lz_close<V, CLOSE_D2><<<nunits * G, RSB_BLOCK, 0, s>>>(a, j, G);
      RSB_CKL("k_lz_close<D2>");
      prof_after(pi, s);
      pi = prof_before(PROF_LZ_B, s);
      if (half) k_lz_d3<V, 128><<<ntiles, 128, 0, s>>>(a, j, breakdown);
      else k_lz_d3<V, 256><<<ntiles, 256, 0, s>>>(a, j, breakdown);
      RSB_CKL("k_lz_d3");
      prof_after(pi, s);
    } else {  // FP64: bound by GB300's FP64 rate; register-streaming kernels, CGS2
      const int G = close_ctas(ntmax, close_ncoef<CLOSE_A>(nd, j));
      k_lz_a<V><<<ntiles, RSB_BLOCK, 0, s>>>(a, j);
      RSB_CKL("k_lz_a");
      k_lz_close<V, CLOSE_A><<<nunits * G, RSB_BLOCK, 0, s>>>(a, j, G);
      RSB_CKL("k_lz_close<A>");
      prof_after(pi, s);
      pi = prof_before(PROF_LZ_B, s);
      k_lz_b<V><<<ntiles, RSB_BLOCK, 0, s>>>(a, j);
      RSB_CKL("k_lz_b");
      k_lz_close<V, CLOSE_B><<<nunits * G, RSB_BLOCK, 0, s>>>(a, j, G);
      RSB_CKL("k_lz_close<B>");
      prof_after(pi, s);
      pi = prof_before(PROF_LZ_C, s);
      k_lz_c<V><<<ntiles, RSB_BLOCK, 0, s>>>(a, j, breakdown);
      RSB_CKL("k_lz_c");
      prof_after(pi, s);
    }
  }
  k_lz_eig<V><<<nunits, RSB_BLOCK, 0, s>>>(a.units, a.S, nunits);
  RSB_CKL("k_lz_eig");
  k_lz_ritz<V><<<ntiles, RSB_BLOCK, 0, s>>>(a);
  RSB_CKL("k_lz_ritz");
  k_lz_resid<V><<<ntiles, RSB_BLOCK, 0, s>>>(a, a.Y, 0);
  RSB_CKL("k_lz_resid");
  k_proj2<V><<<ntiles, RSB_BLOCK, 0, s>>>(a, a.Y);
  RSB_CKL("k_proj2");
  k_proj3<V><<<ntiles, RSB_BLOCK, 0, s>>>(a, a.Y);
  RSB_CKL("k_proj3");
  return RSB_OK;
}

// Runs Lanczos cycles until every participating unit converged or hit its cap.
// The start is the gid hash with seed sd, or from64 / from32 when given.
template <typename V>
static int lanczos_run(const LevelGraph& G, const Tile* tiles, int ntiles, Unit* units, int nunits,
                       const uint64_t* ckey, SolveBufs& B, int M, uint64_t sd,
                       const double* from64, const float* from32, int use_graph,
                       cudaStream_t s) {
  LzArgs<V> a = make_args<V>(G, tiles, ntiles, units, ckey, B);
  // step D1 and the resident kernel size their launches by the largest tile
  if (B.trmax <= 0) return rsb_set_error(RSB_EINVAL, "Lanczos solve without its largest tile size");
  int active = 0;
  int rc = read_active(B, s, &active);
  if (rc || active == 0) return rc;
  rc = lz_start<V>(a, ntiles, sd, from64, from32, s);
  if (rc) return rc;
  const double breakdown = 1e-14;
  const int nd = (B.D[0] ? 1 : 0) + (B.D[1] ? 1 : 0);  // deflation vectors of every active unit
  if (B.gb) {
    // a fresh barrier (count, generation, error word) for this solve; the
    // failure-path test hook starts the count where no CTA sees the last arrival
    RSB_CK(cudaMemsetAsync(B.gb, 0, sizeof(GridBar), s));
    if (g_rsb_poison_barrier && (use_graph == 2 || use_graph == 3))
      RSB_CK(cudaMemsetAsync(&B.gb->count, 0x40, sizeof(unsigned int), s));
  }
  if (use_graph == 3 && B.gb) {
    // the whole solve in one cooperative launch when every tile gets a
    // co-resident CTA holding its rows of the basis; otherwise CUDA graphs
    int dev = 0, nsm = 0, optin = 0, occ = 0;
    RSB_CK(cudaGetDevice(&dev));
    RSB_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    RSB_CK(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    int trs = B.trmax;
    const size_t smem = res_smem_bytes<V>(M, trs);
    if (smem + 4096 <= (size_t)optin) {  // room for the kernel's static shared memory
      RSB_CK(cudaFuncSetAttribute(k_lz_res<V>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)smem));
      RSB_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_lz_res<V>, RSB_BLOCK, smem));
      if ((long long)occ * nsm >= ntiles) {
        int maxcyc = B.maxcycles + 1;
        double bd = breakdown;
        GridBar* gb = B.gb;
        LzArgs<V> ar = a;  // the persistent kernel's phases count into one family
        ar.pb_a = ar.pb_a2 = ar.pb_b = ar.pb_c = prof_bytes(PROF_CYCLE);
        void* args[] = {(void*)&ar, (void*)&M, (void*)&trs, (void*)&bd, (void*)&maxcyc, (void*)&gb};
        const int pi = prof_before(PROF_CYCLE, s);
        cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_lz_res<V>, ntiles, RSB_BLOCK,
                                                    args, smem, s);
        rsb_count_launch(1);
        if (e != cudaSuccess) return rsb_set_cuda_error(e, "cudaLaunchCooperativeKernel(k_lz_res)");
        prof_after(pi, s);
        return read_active(B, s, &active);
      }
    }
  }
  if (use_graph == 2 && B.gb) {
    // one persistent cooperative launch per cycle
    int dev = 0, nsm = 0, occ = 0;
    RSB_CK(cudaGetDevice(&dev));
    RSB_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    RSB_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_lz_cycle<V>, RSB_BLOCK, 0));
    const int grid = std::max(1, std::min(ntiles, occ * nsm));
    GridBar* gb = B.gb;
    int jstart = 0;
    LzArgs<V> ar = a;  // the persistent kernel's phases count into one family
    ar.pb_a = ar.pb_a2 = ar.pb_b = ar.pb_c = prof_bytes(PROF_CYCLE);
    for (int cyc = 0; cyc < 100000; ++cyc) {
      RSB_CK(cudaMemsetAsync(B.jmin, 0x7F, sizeof(int), s));
      void* args[] = {(void*)&ar, (void*)&jstart, (void*)&M, (void*)&breakdown, (void*)&ntiles,
                      (void*)&nunits, (void*)&gb};
      const int pi = prof_before(PROF_CYCLE, s);
      cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_lz_cycle<V>, grid, RSB_BLOCK,
                                                  args, 0, s);
      rsb_count_launch(1);
      if (e != cudaSuccess) return rsb_set_cuda_error(e, "cudaLaunchCooperativeKernel(k_lz_cycle)");
      prof_after(pi, s);
      rc = read_active(B, s, &active);
      if (rc || active == 0) break;
      jstart = std::min(std::max(B.h_active[2], 0), M);
    }
    return rc;
  }
  int dev = 0, nsm = 0;
  RSB_CK(cudaGetDevice(&dev));
  RSB_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  const bool half = d3_half(G.n, ntiles, B.trmax, nsm);
  cudaGraphExec_t exec = nullptr;
  std::vector<int> cap_pairs;
  if (use_graph) {
    cudaGraph_t graph = nullptr;
    RSB_CK(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
    prof_capture_begin();
    rc = lz_cycle<V>(a, ntiles, nunits, M, breakdown, B.trmax, B.ntmax, nd, half, s);
    cap_pairs = prof_capture_end();
    cudaGraph_t g2 = nullptr;
    cudaError_t e = cudaStreamEndCapture(s, &g2);
    graph = g2;
    if (rc) {
      if (graph) cudaGraphDestroy(graph);
      return rc;
    }
    if (e != cudaSuccess) return rsb_set_cuda_error(e, "cudaStreamEndCapture");
    e = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) return rsb_set_cuda_error(e, "cudaGraphInstantiate");
  }
  const char* tr = getenv("RSB_TRACE");
  const bool trace = tr && *tr && *tr != '0';
  auto t_prev = std::chrono::steady_clock::now();
  for (int cyc = 0; cyc < 100000; ++cyc) {
    if (exec) {
      cudaError_t e = cudaGraphLaunch(exec, s);
      rsb_count_launch((sizeof(V) == 4 ? 4 : 5) * M + 5);  // the kernels of one cycle
      if (e != cudaSuccess) {
        cudaGraphExecDestroy(exec);
        return rsb_set_cuda_error(e, "cudaGraphLaunch");
      }
      prof_replay(cap_pairs);
    } else {
      rc = lz_cycle<V>(a, ntiles, nunits, M, breakdown, B.trmax, B.ntmax, nd, half, s);
      if (rc) return rc;
    }
    rc = read_active(B, s, &active);
    if (trace) {  // per-cycle wall time and units still active (RSB_TRACE=1)
      const auto now = std::chrono::steady_clock::now();
      fprintf(stderr, "[rsb]   %9.3f ms    cycle %d: %d of %d units active\n",
              std::chrono::duration<double, std::milli>(now - t_prev).count(), cyc, active,
              nunits);
      t_prev = now;
    }
    if (rc || active == 0) break;
  }
  if (exec) cudaGraphExecDestroy(exec);
  return rc;
}

int solver_lanczos(const LevelGraph& G, const Tile* tiles, int ntiles, Unit* units, int nunits,
                   const uint64_t* ckey, SolveBufs& B, int f32, int M, uint64_t sd,
                   const double* from64, const float* from32, int use_graph, cudaStream_t s) {
  if (ntiles <= 0 || nunits <= 0) return RSB_OK;
  if (f32)
    return lanczos_run<float>(G, tiles, ntiles, units, nunits, ckey, B, M, sd, from64, from32,
                              use_graph, s);
  return lanczos_run<double>(G, tiles, ntiles, units, nunits, ckey, B, M, sd, from64, from32,
                             use_graph, s);
}

// ----------------------------------------------------------------------------
// inverse iteration with CG
// ----------------------------------------------------------------------------
// CG init from w0 / beta0: x = 0, r = p = b, rr = ||b||^2.
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_cg_init(LzArgs<V> a) {
  __shared__ double sm[RSB_WARPS];
  __shared__ double out[1];
  __shared__ double sp[RED_FEW_DOUBLES(1)];
  const Tile t = a.tiles[blockIdx.x];
  Unit& u = a.units[t.unit];
  if (u.status != U_ACTIVE) return;
  const V s = V(1.0 / u.beta0);
  Acc<V> acc;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    const V b = s * a.W0[r];
    a.X[r] = V(0);
    a.R[r] = b;
    a.P[r] = b;
    acc.add(b * b);
  }
  const double sum = block_sum(acc.get(), sm);
  if (threadIdx.x == 0) a.partials[blockIdx.x] = sum;
  if (last_cta(&u.cnt, u.ntile)) {
    final_reduce_few(a.partials, a.stride, u.tile0, u.ntile, 1, out, sp);
    if (threadIdx.x == 0) {
      u.rr = out[0];
      u.bnorm = sqrt(out[0]);
      u.inner = 0;
      u.cg_done = 0;
      u.gbar = 0;
    }
  }
}

// AP = L P, pAp -> alpha
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_cg_ap(LzArgs<V> a) {
  __shared__ double sm[RSB_WARPS];
  __shared__ double out[1];
  __shared__ double sp[RED_FEW_DOUBLES(1)];
  const Tile t = a.tiles[blockIdx.x];
  Unit& u = a.units[t.unit];
  if (u.status != U_ACTIVE || u.cg_done) return;
  Acc<V> acc;
  unsigned long long pbytes = 0;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    const V pr = a.P[r];
    const V ap = spmv_row_ro<V>(a.slice_ptr, a.ent, a.P, r, pr);
    a.AP[r] = ap;
    acc.add(pr * ap);
    if (a.pb_cg) pbytes += 4ull * row_width(a.slice_ptr, r) + 2ull * sizeof(V);
  }
  if (a.pb_cg) prof_add(a.pb_cg, pbytes);
  const double sum = block_sum(acc.get(), sm);
  if (threadIdx.x == 0) a.partials[blockIdx.x] = sum;
  if (last_cta(&u.cnt, u.ntile)) {
    final_reduce_few(a.partials, a.stride, u.tile0, u.ntile, 1, out, sp);
    if (threadIdx.x == 0) u.cg_alpha = u.rr / out[0];
  }
}

// x += alpha p, r -= alpha Ap; sums for ||r||^2 and the projection of r.
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_cg_xr(LzArgs<V> a, double cg_tol, int cg_maxit,
                                                     int* n_cg) {
  __shared__ double sm[RSB_WARPS];
  __shared__ double out[2 + RSB_MAXD];
  __shared__ double sp[RED_FEW_DOUBLES(2 + RSB_MAXD)];
  const Tile t = a.tiles[blockIdx.x];
  Unit& u = a.units[t.unit];
  if (u.status != U_ACTIVE || u.cg_done) return;
  const int nd = u.nd;
  const V al = V(u.cg_alpha);
  Acc<V> r2, rs, d0, d1;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    a.X[r] += al * a.P[r];
    const V rr = a.R[r] - al * a.AP[r];
    a.R[r] = rr;
    r2.add(rr * rr);
    rs.add(rr);
    if (nd > 0) d0.add(V(a.D0[r]) * rr);
    if (nd > 1) d1.add(V(a.D1[r]) * rr);
  }
  double v[4] = {r2.get(), rs.get(), d0.get(), d1.get()};
  const int nv = 2 + nd;
  for (int c = 0; c < nv; ++c) {
    const double sum = block_sum(v[c], sm);
    if (threadIdx.x == 0) a.partials[(long long)c * a.stride + blockIdx.x] = sum;
  }
  if (last_cta(&u.cnt, u.ntile)) {
    final_reduce_few(a.partials, a.stride, u.tile0, u.ntile, nv, out, sp);
    if (threadIdx.x == 0) {
      double cp2 = 0.0;
      u.cp[0] = out[1] * u.isn;
      cp2 += u.cp[0] * u.cp[0];
      for (int l = 0; l < nd; ++l) {
        u.cp[1 + l] = out[2 + l];
        cp2 += u.cp[1 + l] * u.cp[1 + l];
      }
      const double rrn = fmax(out[0] - cp2, 0.0);
      u.inner += 1;
      u.inner_total += 1;
      if (sqrt(rrn) <= cg_tol * u.bnorm || u.inner >= cg_maxit) {
        u.cg_done = 1;
        atomicSub(n_cg, 1);
      } else {
        u.cg_beta = rrn / u.rr;
        u.rr = rrn;
      }
    }
  }
}

// r -= B cp (projection), p = r + beta p while CG continues.
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_cg_p(LzArgs<V> a) {
  const Tile t = a.tiles[blockIdx.x];
  const Unit& u = a.units[t.unit];
  if (u.status != U_ACTIVE || u.cg_done) return;
  const int nd = u.nd;
  const V be = V(u.cg_beta);
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    V v = a.R[r];
    if (unit_has(u, a.ckey, r)) v -= V(u.cp[0] * u.isn);
    if (nd > 0) v -= V(u.cp[1]) * V(a.D0[r]);
    if (nd > 1) v -= V(u.cp[2]) * V(a.D1[r]);
    a.R[r] = v;
    a.P[r] = v + be * a.P[r];
  }
}

// ----------------------------------------------------------------------------
// Flexible CG (§7): the first direction is the residual itself, later ones the
// AMG-preconditioned residual z; beta = z.(r - r_old) / (z_old . r_old).  With
// u.rr holding z.r, k_cg_ap gives alpha = z.r / p.Ap as in plain CG.
// ----------------------------------------------------------------------------
// x += alpha p; r_old = r (in W1); r -= alpha Ap; sums for ||r||^2 and the
// projection of r; convergence as in plain CG.
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_fcg_xr(LzArgs<V> a, double cg_tol, int cg_maxit,
                                                      int* n_cg) {
  __shared__ double sm[RSB_WARPS];
  __shared__ double out[2 + RSB_MAXD];
  __shared__ double sp[RED_FEW_DOUBLES(2 + RSB_MAXD)];
  const Tile t = a.tiles[blockIdx.x];
  Unit& u = a.units[t.unit];
  if (u.status != U_ACTIVE || u.cg_done) return;
  const int nd = u.nd;
  const V al = V(u.cg_alpha);
  Acc<V> r2, rs, d0, d1;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    a.X[r] += al * a.P[r];
    const V ro = a.R[r];
    const V rr = ro - al * a.AP[r];
    a.W1[r] = ro;
    a.R[r] = rr;
    r2.add(rr * rr);
    rs.add(rr);
    if (nd > 0) d0.add(V(a.D0[r]) * rr);
    if (nd > 1) d1.add(V(a.D1[r]) * rr);
  }
  double v[4] = {r2.get(), rs.get(), d0.get(), d1.get()};
  const int nv = 2 + nd;
  for (int c = 0; c < nv; ++c) {
    const double sum = block_sum(v[c], sm);
    if (threadIdx.x == 0) a.partials[(long long)c * a.stride + blockIdx.x] = sum;
  }
  if (last_cta(&u.cnt, u.ntile)) {
    final_reduce_few(a.partials, a.stride, u.tile0, u.ntile, nv, out, sp);
    if (threadIdx.x == 0) {
      double cp2 = 0.0;
      u.cp[0] = out[1] * u.isn;
      cp2 += u.cp[0] * u.cp[0];
      for (int l = 0; l < nd; ++l) {
        u.cp[1 + l] = out[2 + l];
        cp2 += u.cp[1 + l] * u.cp[1 + l];
      }
      const double rrn = fmax(out[0] - cp2, 0.0);
      u.inner += 1;
      u.inner_total += 1;
      if (sqrt(rrn) <= cg_tol * u.bnorm || u.inner >= cg_maxit) {
        u.cg_done = 1;
        atomicSub(n_cg, 1);
      }
    }
  }
}

// r -= B cp (projection): the residual the preconditioner sees
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_fcg_proj(LzArgs<V> a) {
  const Tile t = a.tiles[blockIdx.x];
  const Unit& u = a.units[t.unit];
  if (u.status != U_ACTIVE || u.cg_done) return;
  const int nd = u.nd;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    V v = a.R[r];
    if (unit_has(u, a.ckey, r)) v -= V(u.cp[0] * u.isn);
    if (nd > 0) v -= V(u.cp[1]) * V(a.D0[r]);
    if (nd > 1) v -= V(u.cp[2]) * V(a.D1[r]);
    a.R[r] = v;
  }
}

// z (in Y) restricted to the unit's rows; z.r, z.r_old and the projection sums of z
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_fcg_z(LzArgs<V> a) {
  __shared__ double sm[RSB_WARPS];
  __shared__ double out[3 + RSB_MAXD];
  __shared__ double sp[RED_FEW_DOUBLES(3 + RSB_MAXD)];
  const Tile t = a.tiles[blockIdx.x];
  Unit& u = a.units[t.unit];
  if (u.status != U_ACTIVE || u.cg_done) return;
  const int nd = u.nd;
  Acc<V> zr, zo, zs, d0, d1;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    V z = a.Y[r];
    if (!unit_has(u, a.ckey, r)) {
      z = V(0);
      a.Y[r] = z;
    }
    zr.add(z * a.R[r]);
    zo.add(z * a.W1[r]);
    zs.add(z);
    if (nd > 0) d0.add(V(a.D0[r]) * z);
    if (nd > 1) d1.add(V(a.D1[r]) * z);
  }
  double v[5] = {zr.get(), zo.get(), zs.get(), d0.get(), d1.get()};
  const int nv = 3 + nd;
  for (int c = 0; c < nv; ++c) {
    const double sum = block_sum(v[c], sm);
    if (threadIdx.x == 0) a.partials[(long long)c * a.stride + blockIdx.x] = sum;
  }
  if (last_cta(&u.cnt, u.ntile)) {
    final_reduce_few(a.partials, a.stride, u.tile0, u.ntile, nv, out, sp);
    if (threadIdx.x == 0) {
      u.fz_rz = out[0];
      u.fz_ro = out[1];
      u.cz[0] = out[2] * u.isn;
      for (int l = 0; l < nd; ++l) u.cz[1 + l] = out[3 + l];
    }
  }
}

// z -= B cz; p = z + beta p with the flexible beta; z.r becomes the new rr
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_fcg_p(LzArgs<V> a) {
  const Tile t = a.tiles[blockIdx.x];
  Unit& u = a.units[t.unit];
  if (u.status != U_ACTIVE || u.cg_done) return;
  const int nd = u.nd;
  const double rz = u.fz_rz;
  const V be = V((rz - u.fz_ro) / u.rr);
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    V z = a.Y[r];
    if (unit_has(u, a.ckey, r)) z -= V(u.cz[0] * u.isn);
    if (nd > 0) z -= V(u.cz[1]) * V(a.D0[r]);
    if (nd > 1) z -= V(u.cz[2]) * V(a.D1[r]);
    a.P[r] = z + be * a.P[r];
  }
  // every CTA of the unit has read u.rr above; the unit's rr is rewritten by
  // the next launch that needs it (k_fcg_rr), after this kernel has finished
}

template <typename V>
__global__ void k_fcg_rr(Unit* units, int nunits) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nunits) return;
  Unit& u = units[i];
  if (u.status != U_ACTIVE || u.cg_done) return;
  u.rr = u.fz_rz;
}

// Outer step: y = x; Ly, yLy, yy -> Rayleigh quotient.
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_inv_rq(LzArgs<V> a) {
  __shared__ double sm[RSB_WARPS];
  __shared__ double out[2];
  __shared__ double sp[RED_FEW_DOUBLES(2)];
  const Tile t = a.tiles[blockIdx.x];
  Unit& u = a.units[t.unit];
  if (u.status != U_ACTIVE) return;
  Acc<V> yly, yy;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    const V yr = a.X[r];
    const V ly = spmv_row_ro<V>(a.slice_ptr, a.ent, a.X, r, yr);
    a.AP[r] = ly;
    yly.add(yr * ly);
    yy.add(yr * yr);
  }
  double v[2] = {yly.get(), yy.get()};
  for (int c = 0; c < 2; ++c) {
    const double sum = block_sum(v[c], sm);
    if (threadIdx.x == 0) a.partials[(long long)c * a.stride + blockIdx.x] = sum;
  }
  if (last_cta(&u.cnt, u.ntile)) {
    final_reduce_few(a.partials, a.stride, u.tile0, u.ntile, 2, out, sp);
    if (threadIdx.x == 0) {
      u.theta = out[0] / out[1];
      u.ynorm2 = out[1];
    }
  }
}

// Outer step: residual ||Ly - lambda y|| / ||y||, stop tests, projection dots
// of y for the next right-hand side.
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_inv_res(LzArgs<V> a, int max_outer, int refine) {
  __shared__ double sm[RSB_WARPS];
  __shared__ double out[2 + RSB_MAXD];
  __shared__ double sp[RED_FEW_DOUBLES(2 + RSB_MAXD)];
  const Tile t = a.tiles[blockIdx.x];
  Unit& u = a.units[t.unit];
  if (u.status != U_ACTIVE) return;
  const int nd = u.nd;
  const V th = V(u.theta);
  Acc<V> r2, ys, d0, d1;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    const V yr = a.X[r];
    const V res = a.AP[r] - th * yr;
    r2.add(res * res);
    ys.add(yr);
    if (nd > 0) d0.add(V(a.D0[r]) * yr);
    if (nd > 1) d1.add(V(a.D1[r]) * yr);
  }
  double v[4] = {r2.get(), ys.get(), d0.get(), d1.get()};
  const int nv = 2 + nd;
  for (int c = 0; c < nv; ++c) {
    const double sum = block_sum(v[c], sm);
    if (threadIdx.x == 0) a.partials[(long long)c * a.stride + blockIdx.x] = sum;
  }
  if (last_cta(&u.cnt, u.ntile)) {
    final_reduce_few(a.partials, a.stride, u.tile0, u.ntile, nv, out, sp);
    if (threadIdx.x == 0) {
      u.resid = sqrt(out[0] / u.ynorm2);
      u.cp[0] = out[1] * u.isn;
      for (int l = 0; l < nd; ++l) u.cp[1 + l] = out[2 + l];
      if (refine) {
        u.status = u.resid <= u.tolabs ? U_CONVERGED : U_CAPPED;
        atomicSub(a.n_active, 1);
        return;
      }
      u.cycles += 1;
      atomicAdd((unsigned long long*)a.stat_cycles, 1ull);
      int st = U_ACTIVE;
      if (u.resid <= u.tolabs || u.inner == 1) st = U_CONVERGED;
      else if (u.cycles >= max_outer) st = U_CAPPED;
      if (st != U_ACTIVE) {
        u.status = st;
        atomicSub(a.n_active, 1);
      }
    }
  }
}

// ----------------------------------------------------------------------------
// Resident CG (launch mode 3): one cooperative launch runs the CG solve of every unit
// when every tile gets a co-resident CTA.  x, r, p and L p of a tile's rows stay in
// shared memory; global memory carries p (the SpMV's operand), the partials and the
// unit's barrier.  Units iterate independently.  Rows, sums and their order are those
// of k_cg_ap, k_cg_xr and k_cg_p, so both modes give the same numbers.
// Bound: latency, three barriers and two reductions an iteration; the FP64 work of
// the up to four CTAs of an SM is dealt to its sub-partitions.  Three launches, each
// with the chain of a last CTA's reduction, took 45 us an iteration at 256k rows (500
// tiles).
// The SpMV gathers p with plain loads: the barrier orders them after the other CTAs'
// stores (their release, thread 0's acquire, the CTA barrier), so L1 may serve the
// gathers that share lines.
// ----------------------------------------------------------------------------
template <typename V>
constexpr size_t cg_res_smem(int trs) {
  return 4 * res_align(sizeof(V) * (size_t)trs);
}

template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK, 4)
    k_cg_res(LzArgs<V> a, int trs, double cg_tol, int cg_maxit, GridBar* gb) {
  extern __shared__ __align__(16) unsigned char cg_sh[];
  const size_t vb = res_align(sizeof(V) * (size_t)trs);
  V* X = reinterpret_cast<V*>(cg_sh);
  V* R = reinterpret_cast<V*>(cg_sh + vb);
  V* P = reinterpret_cast<V*>(cg_sh + 2 * vb);
  V* AP = reinterpret_cast<V*>(cg_sh + 3 * vb);
  __shared__ double sm[RSB_WARPS * (2 + RSB_MAXD)];
  __shared__ double out[2 + RSB_MAXD];
  // scratch of the reductions over the tiles and, at other times, over the threads
  __shared__ double sp[RED_FEW_DOUBLES(2 + RSB_MAXD)];
  static_assert(RED_FEW_DOUBLES(2 + RSB_MAXD) >= (2 + RSB_MAXD) * RSB_BLOCK, "scratch");
  __shared__ double rr_sh;
  __shared__ V al_sh, be_sh, cp_sh[1 + RSB_MAXD];
  __shared__ int done_sh;
  const int tix = blockIdx.x;
  const Tile t = a.tiles[tix];
  Unit& u = a.units[t.unit];
  if (__ldcg(&u.status) != U_ACTIVE) return;
  const int nr = t.row1 - t.row0;
  const int nd = u.nd, nv = 2 + nd, nt = u.ntile;
  const bool first = tix == u.tile0;
  const int fw = fp64_warp(), lane = threadIdx.x & 31;
  const bool fpw = (int)(threadIdx.x >> 5) == fw;
  const double bnorm = u.bnorm, isn = u.isn;
  UnitBar ub(&u.gbar, nt, __ldcg(&gb->count), gb);
  double* const P1 = a.partials;                       // p.Lp
  double* const P2 = a.partials + a.stride;            // ||r||^2 and the projection of r
  const V* Pg = a.P;
  for (int rl = threadIdx.x; rl < nr; rl += RSB_BLOCK) {
    X[rl] = V(0);
    R[rl] = a.R[t.row0 + rl];
    P[rl] = a.P[t.row0 + rl];
  }
  if (threadIdx.x == 0) {
    rr_sh = u.rr;
    done_sh = 0;
  }
  __syncthreads();
  unsigned long long pbytes = 0;
  int it = 0;
  while (true) {
    // AP = L P, p.Lp -> alpha
    Acc<V> acc;
    for (int rl = threadIdx.x; rl < nr; rl += RSB_BLOCK) {
      const int r = t.row0 + rl;
      const int64_t base = a.slice_ptr[r >> 5];
      const int width = (int)((a.slice_ptr[(r >> 5) + 1] - base) >> 5);
      const uint32_t* e = a.ent + base + (r & 31);
      const V pr = P[rl];
      V ap = V(0);
      uint32_t dsum = 0;
      for (int k0 = 0; k0 < width; k0 += 13) {
        uint32_t p[13];
        V xv[13];
#pragma unroll
        for (int i = 0; i < 13; ++i) p[i] = k0 + i < width ? __ldg(e + 32 * (k0 + i)) : 0u;
#pragma unroll
        for (int i = 0; i < 13; ++i) xv[i] = k0 + i < width ? Pg[ent_col(p[i])] : pr;
#pragma unroll
        for (int i = 0; i < 13; ++i)
          if (k0 + i < width) {
            if constexpr (sizeof(V) == 8) {
              ap = fma(weight_f64(ent_w(p[i])), xv[i], ap);
              dsum += ent_w(p[i]);
            } else {
              ap += V(ent_w(p[i])) * (pr - xv[i]);
            }
          }
      }
      if constexpr (sizeof(V) == 8) ap = fma((double)dsum, pr, -ap);
      AP[rl] = ap;
      acc.add(pr * ap);
      if (a.pb_cg) pbytes += 4ull * width + 2ull * sizeof(V);
    }
    const double v1[1] = {acc.get()};
    double sum = block_sums<1>(v1, 1, sp, sm, fw);
    if (nt > 1) {
      if (fpw && lane == 0) P1[tix] = sum;
      if (!ub.sync()) return;
      final_reduce_few(P1, a.stride, u.tile0, nt, 1, out, sp, fw);
      sum = out[0];
    }
    if (fpw && lane == 0) al_sh = V(rr_sh / sum);
    __syncthreads();
    // x += alpha p, r -= alpha Ap; ||r||^2 and the projection of r
    const V al = al_sh;
    Acc<V> r2, rs, d0, d1;
    for (int rl = threadIdx.x; rl < nr; rl += RSB_BLOCK) {
      X[rl] += al * P[rl];
      const V rn = R[rl] - al * AP[rl];
      R[rl] = rn;
      r2.add(rn * rn);
      rs.add(rn);
      if (nd > 0) d0.add(V(a.D0[t.row0 + rl]) * rn);
      if (nd > 1) d1.add(V(a.D1[t.row0 + rl]) * rn);
    }
    const double v[2 + RSB_MAXD] = {r2.get(), rs.get(), d0.get(), d1.get()};
    const double x = block_sums<2 + RSB_MAXD>(v, nv, sp, sm, fw);
    if (fpw && lane < nv) {
      if (nt > 1) P2[(long long)lane * a.stride + tix] = x;
      else out[lane] = x;
    }
    if (nt > 1) {
      if (!ub.sync()) return;
      final_reduce_few(P2, a.stride, u.tile0, nt, nv, out, sp, fw);
    } else {
      __syncthreads();
    }
    ++it;
    if (fpw && lane == 0) {
      double cp2 = 0.0, cp[1 + RSB_MAXD];
      cp[0] = out[1] * isn;
      cp2 += cp[0] * cp[0];
      for (int l = 0; l < nd; ++l) {
        cp[1 + l] = out[2 + l];
        cp2 += cp[1 + l] * cp[1 + l];
      }
      const double rrn = fmax(out[0] - cp2, 0.0);
      if (sqrt(rrn) <= cg_tol * bnorm || it >= cg_maxit) {
        done_sh = 1;
      } else {
        be_sh = V(rrn / rr_sh);
        rr_sh = rrn;
        cp_sh[0] = V(cp[0] * isn);
        for (int l = 0; l < nd; ++l) cp_sh[1 + l] = V(cp[1 + l]);
      }
    }
    __syncthreads();
    if (done_sh) break;
    // r -= B cp, p = r + beta p
    const V be = be_sh;
    for (int rl = threadIdx.x; rl < nr; rl += RSB_BLOCK) {
      const int r = t.row0 + rl;
      V x = R[rl];
      if (unit_has(u, a.ckey, r)) x -= cp_sh[0];
      if (nd > 0) x -= cp_sh[1] * V(a.D0[r]);
      if (nd > 1) x -= cp_sh[2] * V(a.D1[r]);
      R[rl] = x;
      const V pn = x + be * P[rl];
      P[rl] = pn;
      a.P[r] = pn;
    }
    if (!ub.sync()) return;
  }
  for (int rl = threadIdx.x; rl < nr; rl += RSB_BLOCK) a.X[t.row0 + rl] = X[rl];
  if (first && threadIdx.x == 0) {
    u.inner = it;
    u.inner_total += it;
    u.cg_done = 1;
  }
  if (a.pb_cg) prof_add(a.pb_cg, pbytes);
}

__global__ void k_count_cg(Unit* units, int nunits, int* n_cg) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nunits && units[i].status == U_ACTIVE && !units[i].cg_done) atomicAdd(n_cg, 1);
}

int amg_setup(int f32, const LevelGraph& G, const Tile* tiles, int ntiles, const Unit* units,
              const std::vector<Unit>& hunits, cudaStream_t s);
int amg_apply(int f32, const LevelGraph& G, const Tile* tiles, int ntiles, const Unit* units,
              const void* r, void* z, cudaStream_t s);

template <typename V>
static int cg_block(LzArgs<V>& a, int ntiles, int iters, double cg_tol, int cg_maxit, int* n_cg,
                    cudaStream_t s, const LevelGraph* amgG = nullptr, int nunits = 0) {
  for (int i = 0; i < iters; ++i) {
    const int pi = prof_before(PROF_CG_AP, s);
    k_cg_ap<V><<<ntiles, RSB_BLOCK, 0, s>>>(a);
    RSB_CKL("k_cg_ap");
    prof_after(pi, s);
    if (!amgG) {
      k_cg_xr<V><<<ntiles, RSB_BLOCK, 0, s>>>(a, cg_tol, cg_maxit, n_cg);
      RSB_CKL("k_cg_xr");
      k_cg_p<V><<<ntiles, RSB_BLOCK, 0, s>>>(a);
      RSB_CKL("k_cg_p");
      continue;
    }
    // flexible CG preconditioned by one AMG V-cycle (§7)
    k_fcg_xr<V><<<ntiles, RSB_BLOCK, 0, s>>>(a, cg_tol, cg_maxit, n_cg);
    RSB_CKL("k_fcg_xr");
    k_fcg_proj<V><<<ntiles, RSB_BLOCK, 0, s>>>(a);
    RSB_CKL("k_fcg_proj");
    const int pv = prof_before(PROF_AMG, s);
    int rc = amg_apply(sizeof(V) == 4, *amgG, a.tiles, ntiles, a.units, a.R, a.Y, s);
    if (rc) return rc;
    prof_after(pv, s);
    k_fcg_z<V><<<ntiles, RSB_BLOCK, 0, s>>>(a);
    RSB_CKL("k_fcg_z");
    k_fcg_p<V><<<ntiles, RSB_BLOCK, 0, s>>>(a);
    RSB_CKL("k_fcg_p");
    k_fcg_rr<V><<<(nunits + 127) / 128, 128, 0, s>>>(a.units, nunits);
    RSB_CKL("k_fcg_rr");
  }
  return RSB_OK;
}

template <typename V>
static int inverse_run(const LevelGraph& G, const Tile* tiles, int ntiles, Unit* units, int nunits,
                       const uint64_t* ckey, SolveBufs& B, uint64_t sd, const double* from64,
                       const float* from32, double cg_tol, int cg_maxit, int max_outer,
                       int use_graph, int64_t* inner_out, cudaStream_t s,
                       const std::vector<Unit>* amg_units) {
  LzArgs<V> a = make_args<V>(G, tiles, ntiles, units, ckey, B);
  // step D1 and the resident kernel size their launches by the largest tile
  if (B.trmax <= 0) return rsb_set_error(RSB_EINVAL, "Lanczos solve without its largest tile size");
  int active = 0;
  int rc = read_active(B, s, &active);
  if (rc || active == 0) return rc;
  rc = lz_start<V>(a, ntiles, sd, from64, from32, s);  // W0 = projected start, beta0
  if (rc) return rc;
  const LevelGraph* amgG = nullptr;
  if (amg_units) {  // the hierarchy of every unit of the level (§7)
    if ((rc = amg_setup(sizeof(V) == 4, G, tiles, ntiles, units, *amg_units, s))) return rc;
    amgG = &G;
  }
  // one cooperative launch per CG solve when every tile gets a co-resident CTA
  bool res = false;
  const size_t cg_smem = cg_res_smem<V>(B.trmax);
  if (use_graph == 3 && !amgG && B.gb) {
    int dev = 0, nsm = 0, optin = 0, occ = 0;
    RSB_CK(cudaGetDevice(&dev));
    RSB_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    RSB_CK(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    if (cg_smem + 12288 <= (size_t)optin) {  // room for the kernel's static shared memory
      RSB_CK(cudaFuncSetAttribute(k_cg_res<V>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)cg_smem));
      RSB_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_cg_res<V>, RSB_BLOCK, cg_smem));
      res = (long long)occ * nsm >= ntiles;
    }
    RSB_CK(cudaMemsetAsync(B.gb, 0, sizeof(GridBar), s));
    if (g_rsb_poison_barrier && res)  // test hook: the units' arrivals are out of reach
      RSB_CK(cudaMemsetAsync(&B.gb->count, 0x40, sizeof(unsigned int), s));
  }
  const int CGK = 8;
  cudaGraphExec_t exec = nullptr;
  std::vector<int> cap_pairs;
  if (use_graph && !res) {
    cudaGraph_t graph = nullptr;
    RSB_CK(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
    prof_capture_begin();
    rc = cg_block<V>(a, ntiles, CGK, cg_tol, cg_maxit, B.n_cg, s, amgG, nunits);
    cap_pairs = prof_capture_end();
    cudaError_t e = cudaStreamEndCapture(s, &graph);
    if (rc) {
      if (graph) cudaGraphDestroy(graph);
      return rc;
    }
    if (e != cudaSuccess) return rsb_set_cuda_error(e, "cudaStreamEndCapture");
    e = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) return rsb_set_cuda_error(e, "cudaGraphInstantiate");
  }
  for (int outer = 0; outer < max_outer + 1 && active > 0; ++outer) {
    k_cg_init<V><<<ntiles, RSB_BLOCK, 0, s>>>(a);
    RSB_CKL("k_cg_init");
    if (!res) {
      RSB_CK(cudaMemsetAsync(B.n_cg, 0, sizeof(int), s));
      k_count_cg<<<(nunits + 127) / 128, 128, 0, s>>>(units, nunits, B.n_cg);
      RSB_CKL("k_count_cg");
    }
    if (res) {
      int trs = B.trmax;
      GridBar* gb = B.gb;
      void* args[] = {(void*)&a, (void*)&trs, (void*)&cg_tol, (void*)&cg_maxit, (void*)&gb};
      const int pi = prof_before(PROF_CG_AP, s);
      cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_cg_res<V>, ntiles, RSB_BLOCK, args,
                                                  cg_smem, s);
      rsb_count_launch(1);
      if (e != cudaSuccess) return rsb_set_cuda_error(e, "cudaLaunchCooperativeKernel(k_cg_res)");
      prof_after(pi, s);
    }
    for (int blk = 0; !res && blk < cg_maxit / CGK + 2; ++blk) {
      if (exec) {
        cudaError_t e = cudaGraphLaunch(exec, s);
        rsb_count_launch((amgG ? 7 + 13 * 20 : 3) * CGK);
        if (e != cudaSuccess) {
          cudaGraphExecDestroy(exec);
          return rsb_set_cuda_error(e, "cudaGraphLaunch");
        }
        prof_replay(cap_pairs);
      } else {
        rc = cg_block<V>(a, ntiles, CGK, cg_tol, cg_maxit, B.n_cg, s, amgG, nunits);
        if (rc) break;
      }
      int ncg = 0;
      RSB_CK(cudaMemcpyAsync(B.h_active, B.n_cg, sizeof(int), cudaMemcpyDeviceToHost, s));
      RSB_CK(cudaStreamSynchronize(s));
      prof_collect();
      ncg = *B.h_active;
      if (ncg <= 0) break;
    }
    if (rc) break;
    k_inv_rq<V><<<ntiles, RSB_BLOCK, 0, s>>>(a);
    RSB_CKL("k_inv_rq");
    k_inv_res<V><<<ntiles, RSB_BLOCK, 0, s>>>(a, max_outer, 0);
    RSB_CKL("k_inv_res");
    rc = read_active(B, s, &active);
    if (rc || active == 0) break;
    // next right-hand side: x projected (second pass) and normalised into W0
    k_proj2<V><<<ntiles, RSB_BLOCK, 0, s>>>(a, a.X);
    RSB_CKL("k_proj2");
    k_proj3<V><<<ntiles, RSB_BLOCK, 0, s>>>(a, a.X);
    RSB_CKL("k_proj3");
  }
  if (exec) cudaGraphExecDestroy(exec);
  (void)inner_out;
  return rc;
}

int solver_inverse(const LevelGraph& G, const Tile* tiles, int ntiles, Unit* units, int nunits,
                   const uint64_t* ckey, SolveBufs& B, int f32, uint64_t sd, const double* from64,
                   const float* from32, double cg_tol, int cg_maxit, int max_outer, int use_graph,
                   cudaStream_t s, const std::vector<Unit>* amg_units) {
  if (ntiles <= 0 || nunits <= 0) return RSB_OK;
  if (f32)
    return inverse_run<float>(G, tiles, ntiles, units, nunits, ckey, B, sd, from64, from32, cg_tol,
                              cg_maxit, max_outer, use_graph, nullptr, s, amg_units);
  return inverse_run<double>(G, tiles, ntiles, units, nunits, ckey, B, sd, from64, from32, cg_tol,
                             cg_maxit, max_outer, use_graph, nullptr, s, amg_units);
}

// ----------------------------------------------------------------------------
// FP64 Rayleigh-quotient refinement of an FP32 vector (mixed precision):
// y = FP64 copy of the FP32 vector, theta = y^T L y / y^T y and the residual
// ||L y - theta y|| / ||y|| in FP64; the FP64 y lands in B.X.
// ----------------------------------------------------------------------------
int solver_rq_refine(const LevelGraph& G, const Tile* tiles, int ntiles, Unit* units, int nunits,
                     const uint64_t* ckey, SolveBufs& B, const float* from32, cudaStream_t s) {
  if (ntiles <= 0 || nunits <= 0) return RSB_OK;
  SolveBufs Bx = B;
  Bx.Y = B.X;  // k_start writes a.Y; the refinement kernels read a.X
  LzArgs<double> a = make_args<double>(G, tiles, ntiles, units, ckey, Bx);
  k_start<double><<<ntiles, RSB_BLOCK, 0, s>>>(a, 0ull, nullptr, from32);
  RSB_CKL("k_start(refine)");
  k_inv_rq<double><<<ntiles, RSB_BLOCK, 0, s>>>(a);
  RSB_CKL("k_inv_rq(refine)");
  k_inv_res<double><<<ntiles, RSB_BLOCK, 0, s>>>(a, 0, 1);
  RSB_CKL("k_inv_res(refine)");
  (void)nunits;
  return RSB_OK;
}

// ----------------------------------------------------------------------------
// result vector: out = y / ||y|| (FP64), for units that took part in the solve
// ----------------------------------------------------------------------------
// better_only: a polish result, written only where its residual is below the
// one recorded for candidate cand (the refined stage-1 vector already in out);
// k_keep_better then settles the unit's record.
template <typename V>
__global__ void __launch_bounds__(RSB_BLOCK) k_write_vec(LzArgs<V> a, const V* __restrict__ y,
                                                         double* out, int cand, int better_only) {
  const Tile t = a.tiles[blockIdx.x];
  Unit& u = a.units[t.unit];
  if (u.status != U_CONVERGED && u.status != U_CAPPED) return;
  if (better_only && !(u.resid < u.res[cand])) return;
  const double sc = 1.0 / sqrt(u.ynorm2);
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) out[r] = sc * (double)y[r];
  if (!better_only && blockIdx.x == u.tile0 && threadIdx.x == 0 && cand >= 0) {
    u.lam[cand] = u.theta;
    u.res[cand] = u.resid;
  }
}

// After a polish: the unit keeps the smaller-residual of the refined stage-1
// vector and the polished one (a capped polish can end on a Ritz vector whose
// residual exceeds its start's); it counts as converged at tol1 * dmax.
__global__ void k_keep_better(Unit* units, int nunits, int cand, double tol1) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nunits) return;
  Unit& u = units[i];
  if (u.status != U_CONVERGED && u.status != U_CAPPED) return;
  if (u.resid < u.res[cand]) {
    u.lam[cand] = u.theta;
    u.res[cand] = u.resid;
  } else {
    u.theta = u.lam[cand];
    u.resid = u.res[cand];
  }
  u.status = u.resid <= tol1 * u.dmax ? U_CONVERGED : U_CAPPED;
}

int solver_write_vector(const LevelGraph& G, const Tile* tiles, int ntiles, Unit* units,
                        const uint64_t* ckey, SolveBufs& B, int f32, int from_x, double* out,
                        int cand, int better_only, cudaStream_t s) {
  if (ntiles <= 0) return RSB_OK;
  if (f32) {
    LzArgs<float> a = make_args<float>(G, tiles, ntiles, units, ckey, B);
    k_write_vec<float><<<ntiles, RSB_BLOCK, 0, s>>>(a, from_x ? a.X : a.Y, out, cand, better_only);
  } else {
    LzArgs<double> a = make_args<double>(G, tiles, ntiles, units, ckey, B);
    k_write_vec<double><<<ntiles, RSB_BLOCK, 0, s>>>(a, from_x ? a.X : a.Y, out, cand,
                                                     better_only);
  }
  RSB_CKL("k_write_vec");
  return RSB_OK;
}

int solver_keep_better(Unit* units, int nunits, int cand, double tol1, cudaStream_t s) {
  k_keep_better<<<(nunits + 127) / 128, 128, 0, s>>>(units, nunits, cand, tol1);
  RSB_CKL("k_keep_better");
  return RSB_OK;
}

// ----------------------------------------------------------------------------
// R5: rotation of a 2- or 3-dimensional cluster basis minimising sum (U R)^4
// ----------------------------------------------------------------------------
// Moments M[a][b][c][d] = sum_r U_a U_b U_c U_d over unit rows, stored for
// a <= b <= c <= d (15 for three columns); the rotation is then found from the
// tensor alone by cyclic pairwise steps, each the closed-form optimum of a
// 2-D rotation (maximise sum (x' y')^2).
__device__ __forceinline__ int mom_index(int a, int b, int c, int d) {
  // sort a<=b<=c<=d then enumerate combinations with repetition of {0,1,2}
  int v[4] = {a, b, c, d};
  for (int i = 0; i < 4; ++i)
    for (int j = i + 1; j < 4; ++j)
      if (v[j] < v[i]) { const int t = v[i]; v[i] = v[j]; v[j] = t; }
  int idx = 0;
  for (int p = 0; p < 3; ++p)
    for (int q = p; q < 3; ++q)
      for (int r = q; r < 3; ++r)
        for (int s = r; s < 3; ++s) {
          if (p == v[0] && q == v[1] && r == v[2] && s == v[3]) return idx;
          ++idx;
        }
  return 0;
}

__global__ void __launch_bounds__(RSB_BLOCK)
    k_quartic_moments(const Tile* __restrict__ tiles, Unit* units, const uint64_t* __restrict__ ckey,
                      const double* __restrict__ v0, const double* __restrict__ v1,
                      const double* __restrict__ v2, double* partials, long long stride,
                      double* mom) {
  __shared__ double sm[RSB_WARPS];
  __shared__ double out[15];
  const Tile t = tiles[blockIdx.x];
  Unit& u = units[t.unit];
  if (!u.valid || u.ncand < 2) return;
  const int m = u.ncand;
  double acc[15];
  for (int i = 0; i < 15; ++i) acc[i] = 0.0;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    if (!unit_has(u, ckey, r)) continue;
    const double x[3] = {v0[r], v1[r], m > 2 ? v2[r] : 0.0};
    int idx = 0;
    for (int p = 0; p < 3; ++p)
      for (int q = p; q < 3; ++q)
        for (int rr = q; rr < 3; ++rr)
          for (int s = rr; s < 3; ++s) acc[idx++] += x[p] * x[q] * x[rr] * x[s];
  }
  for (int c = 0; c < 15; ++c) {
    const double sum = block_sum(acc[c], sm);
    if (threadIdx.x == 0) partials[(long long)c * stride + blockIdx.x] = sum;
  }
  if (last_cta(&u.cnt, u.ntile)) {
    final_reduce(partials, stride, u.tile0, u.ntile, 15, out);
    if (threadIdx.x < 15) mom[(long long)t.unit * 24 + threadIdx.x] = out[threadIdx.x];
  }
}

// S(p,q; i) = sum_r x^(4-i) y^i with x = U R[:,p], y = U R[:,q], from the full
// (81-entry) moment tensor Mf.
__device__ double rot_moment(const double* Mf, const double* R, int p, int q, int i) {
  double s = 0.0;
  for (int a = 0; a < 3; ++a) {
    const double fa = R[a * 3 + (0 < 4 - i ? p : q)];
    for (int b = 0; b < 3; ++b) {
      const double fab = fa * R[b * 3 + (1 < 4 - i ? p : q)];
      for (int c = 0; c < 3; ++c) {
        const double fabc = fab * R[c * 3 + (2 < 4 - i ? p : q)];
        const double* row = Mf + ((a * 3 + b) * 3 + c) * 3;
        const int col = 3 < 4 - i ? p : q;
        s += fabc * (row[0] * R[0 * 3 + col] + row[1] * R[1 * 3 + col] + row[2] * R[2 * 3 + col]);
      }
    }
  }
  return s;
}

__global__ void k_quartic_rotation(Unit* units, int nunits, double* mom) {
  const int ui = blockIdx.x * blockDim.x + threadIdx.x;
  if (ui >= nunits) return;
  Unit& u = units[ui];
  if (!u.valid || u.ncand < 2) return;
  const int m = u.ncand;
  double* M = mom + (long long)ui * 24;
  double Mf[81];
  for (int a = 0; a < 3; ++a)
    for (int b = 0; b < 3; ++b)
      for (int c = 0; c < 3; ++c)
        for (int d = 0; d < 3; ++d) Mf[((a * 3 + b) * 3 + c) * 3 + d] = M[mom_index(a, b, c, d)];
  double R[9] = {1, 0, 0, 0, 1, 0, 0, 0, 1};
  const int sweeps = m > 2 ? 50 : 1;
  for (int sw = 0; sw < sweeps; ++sw) {
    double dmax = 0.0;
    for (int p = 0; p < m - 1; ++p)
      for (int q = p + 1; q < m; ++q) {
        const double x4 = rot_moment(Mf, R, p, q, 0);
        const double x3y = rot_moment(Mf, R, p, q, 1);
        const double x2y2 = rot_moment(Mf, R, p, q, 2);
        const double xy3 = rot_moment(Mf, R, p, q, 3);
        const double y4 = rot_moment(Mf, R, p, q, 4);
        // u = x^2 - y^2, w = 2 x y
        const double uu = x4 - 2.0 * x2y2 + y4;
        const double ww = 4.0 * x2y2;
        const double uw = 2.0 * (x3y - xy3);
        const double th = 0.25 * atan2(uw, 0.5 * (ww - uu));
        const double c = cos(th), s = sin(th);
        for (int a = 0; a < 3; ++a) {
          const double rp = R[a * 3 + p], rq = R[a * 3 + q];
          R[a * 3 + p] = c * rp - s * rq;
          R[a * 3 + q] = s * rp + c * rq;
        }
        dmax = fmax(dmax, fabs(th));
      }
    if (dmax < 1e-12) break;
  }
  for (int i = 0; i < 9; ++i) M[15 + i] = R[i];
}

__global__ void __launch_bounds__(RSB_BLOCK)
    k_quartic_apply(const Tile* __restrict__ tiles, const Unit* units, double* v0, double* v1,
                    double* v2, const double* mom) {
  const Tile t = tiles[blockIdx.x];
  const Unit& u = units[t.unit];
  if (!u.valid || u.ncand < 2) return;
  const int m = u.ncand;
  const double* R = mom + (long long)t.unit * 24 + 15;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    const double x[3] = {v0[r], v1[r], m > 2 ? v2[r] : 0.0};
    double y[3];
    for (int c = 0; c < m; ++c) {
      double s = 0.0;
      for (int a = 0; a < m; ++a) s += x[a] * R[a * 3 + c];
      y[c] = s;
    }
    v0[r] = y[0];
    v1[r] = y[1];
    if (m > 2) v2[r] = y[2];
  }
}

int solver_quartic(const Tile* tiles, int ntiles, Unit* units, int nunits, const uint64_t* ckey,
                   double* v0, double* v1, double* v2, double* partials, double* mom,
                   cudaStream_t s) {
  if (ntiles <= 0) return RSB_OK;
  k_quartic_moments<<<ntiles, RSB_BLOCK, 0, s>>>(tiles, units, ckey, v0, v1, v2, partials, ntiles,
                                                 mom);
  RSB_CKL("k_quartic_moments");
  k_quartic_rotation<<<(nunits + 63) / 64, 64, 0, s>>>(units, nunits, mom);
  RSB_CKL("k_quartic_rotation");
  k_quartic_apply<<<ntiles, RSB_BLOCK, 0, s>>>(tiles, units, v0, v1, v2, mom);
  RSB_CKL("k_quartic_apply");
  return RSB_OK;
}

// ----------------------------------------------------------------------------
// cluster test after a deflated solve (R5): candidate nd joins when its
// eigenvalue is within cluster_tol * lambda_a of the first.
// ----------------------------------------------------------------------------
__global__ void k_cluster_check(Unit* units, int nunits, int nd, double cluster_tol) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nunits) return;
  Unit& u = units[i];
  if (!u.valid || u.ncand != nd) return;
  if (u.status != U_CONVERGED && u.status != U_CAPPED) return;
  if (fabs(u.lam[nd] - u.lam[0]) <= cluster_tol * u.lam[0]) u.ncand = nd + 1;
}

int solver_cluster_check(Unit* units, int nunits, int nd, double cluster_tol, cudaStream_t s) {
  k_cluster_check<<<(nunits + 127) / 128, 128, 0, s>>>(units, nunits, nd, cluster_tol);
  RSB_CKL("k_cluster_check");
  return RSB_OK;
}

// Statistics of the finished solve: count capped units, max residual / dmax.
__global__ void k_solve_stats(const Unit* units, int nunits, int* capped, double* resid_max,
                              int cand) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nunits) return;
  const Unit& u = units[i];
  if (u.status == U_CAPPED) atomicAdd(capped, 1);
  if (u.status == U_CONVERGED || u.status == U_CAPPED) {
    const double r = u.resid / fmax(u.dmax, 1e-300);
    // non-negative doubles order like their bit patterns
    atomicMax((unsigned long long*)resid_max, (unsigned long long)__double_as_longlong(r));
  }
  (void)cand;
}

// CG iterations of the inverse-iteration solve just finished, summed over units
__global__ void k_sum_inner(const Unit* units, int nunits, long long* inner) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nunits) return;
  const Unit& u = units[i];
  if (u.status == U_CONVERGED || u.status == U_CAPPED)
    atomicAdd((unsigned long long*)inner, (unsigned long long)u.inner_total);
}

int solver_sum_inner(const Unit* units, int nunits, long long* inner, cudaStream_t s) {
  k_sum_inner<<<(nunits + 127) / 128, 128, 0, s>>>(units, nunits, inner);
  RSB_CKL("k_sum_inner");
  return RSB_OK;
}

int solver_stats(const Unit* units, int nunits, int* capped, double* resid_max, cudaStream_t s) {
  k_solve_stats<<<(nunits + 127) / 128, 128, 0, s>>>(units, nunits, capped, resid_max, 0);
  RSB_CKL("k_solve_stats");
  return RSB_OK;
}
