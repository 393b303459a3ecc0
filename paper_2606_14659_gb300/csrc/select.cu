// select.cu — the median split of Algorithm 1 (§4), done as a selection
// instead of the sort the paper describes:
//   * orientation of the Fiedler vector (reading R4: the smallest gid among
//     |v| >= max|v|/2 must come out negative),
//   * a segmented 8-bit-digit radix select of the k-th smallest key per unit
//     (keys: order-preserving bits of the FP64 value, a gid, or a component
//     key), which gives the same answer as sorting and taking k elements,
//   * the tie window of reading R7 (values within tie_rel * range of the k-th
//     value are ties and go left in ascending gid),
//   * the gid rule comparing two candidate splits of a repeated eigenvalue
//     (reading R5), and the final side of every row including whole
//     components placed by reading R8;
// in one cooperative launch per candidate where a level allows it.
#include <algorithm>

#include "rsb_internal.cuh"

// ----------------------------------------------------------------------------
// per-unit max weighted degree (the ||L|| scale of the stopping tests)
// ----------------------------------------------------------------------------
__device__ __forceinline__ void final_max(const double* partials, long long stride, int t0, int nt,
                                          double* out) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (w == 0) {
    double m = -1e300;
    for (int t = lane; t < nt; t += 32) m = fmax(m, __ldcg(partials + stride * 0 + t0 + t));
    m = warp_max(m);
    if (lane == 0) out[0] = m;
  }
  __syncthreads();
}

__global__ void __launch_bounds__(RSB_BLOCK)
    k_degree_max(const int32_t* __restrict__ deg, const Tile* __restrict__ tiles, Unit* units,
                 const uint64_t* __restrict__ ckey, double* partials, long long stride) {
  __shared__ double sm[RSB_WARPS];
  __shared__ double out[1];
  const Tile t = tiles[blockIdx.x];
  Unit& u = units[t.unit];
  if (!u.valid) return;
  double m = 0.0;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK)
    if (unit_has(u, ckey, r)) m = fmax(m, (double)deg[r]);
  m = warp_max(m);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    double b = 0.0;
    for (int i = 0; i < RSB_WARPS; ++i) b = fmax(b, sm[i]);
    partials[blockIdx.x] = b;
  }
  if (last_cta(&u.cnt, u.ntile)) {
    final_max(partials, stride, u.tile0, u.ntile, out);
    if (threadIdx.x == 0) u.dmax = out[0];
  }
}

int launch_degree_max(const LevelGraph& G, const Tile* tiles, int ntiles, Unit* units,
                      const uint64_t* ckey, double* partials, cudaStream_t s) {
  if (ntiles <= 0) return RSB_OK;
  k_degree_max<<<ntiles, RSB_BLOCK, 0, s>>>(G.deg, tiles, units, ckey, partials, ntiles);
  RSB_CKL("k_degree_max");
  return RSB_OK;
}

// ----------------------------------------------------------------------------
// orientation statistics: amax = max|v|, vmax, vmin over the unit
// ----------------------------------------------------------------------------
__global__ void __launch_bounds__(RSB_BLOCK)
    k_orient_stats(const Tile* __restrict__ tiles, Unit* units, const uint64_t* __restrict__ ckey,
                   const double* __restrict__ v, int cand, double* partials, long long stride) {
  __shared__ double sm[3][RSB_WARPS];
  __shared__ double out[3];
  const Tile t = tiles[blockIdx.x];
  Unit& u = units[t.unit];
  if (!u.valid || cand >= u.ncand) return;
  double a = 0.0, hi = -1e300, lo = 1e300;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    if (!unit_has(u, ckey, r)) continue;
    const double x = v[r];
    a = fmax(a, fabs(x));
    hi = fmax(hi, x);
    lo = fmin(lo, x);
  }
  a = warp_max(a);
  hi = warp_max(hi);
  lo = -warp_max(-lo);
  if ((threadIdx.x & 31) == 0) {
    sm[0][threadIdx.x >> 5] = a;
    sm[1][threadIdx.x >> 5] = hi;
    sm[2][threadIdx.x >> 5] = -lo;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    double b = -1e300;
    for (int i = 0; i < RSB_WARPS; ++i) b = fmax(b, sm[threadIdx.x][i]);
    partials[(long long)threadIdx.x * stride + blockIdx.x] = b;
  }
  if (last_cta(&u.cnt, u.ntile)) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (w < 3) {
      double m = -1e300;
      for (int i = lane; i < u.ntile; i += 32) m = fmax(m, __ldcg(partials + w * stride + u.tile0 + i));
      m = warp_max(m);
      if (lane == 0) out[w] = m;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      u.amax = out[0];
      u.vmax = out[1];
      u.vmin = -out[2];
    }
  }
}

// g* = smallest gid among rows with |v| >= amax / 2, and v at g*; then the
// sign that makes v[g*] negative and the tie window tau.
__global__ void __launch_bounds__(RSB_BLOCK)
    k_orient_gstar(const int64_t* __restrict__ gid, const Tile* __restrict__ tiles, Unit* units,
                   const uint64_t* __restrict__ ckey, const double* __restrict__ v, int cand,
                   double tie_rel, double* partials, long long stride, int fixed_sign) {
  __shared__ long long smg[RSB_WARPS];
  __shared__ double smv[RSB_WARPS];
  const Tile t = tiles[blockIdx.x];
  Unit& u = units[t.unit];
  if (!u.valid || cand >= u.ncand) return;
  const double thr = 0.5 * u.amax;
  long long g = LLONG_MAX;
  double gv = 0.0;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    if (!unit_has(u, ckey, r)) continue;
    const double x = v[r];
    if (fabs(x) >= thr && gid[r] < g) {
      g = gid[r];
      gv = x;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long og = __shfl_xor_sync(0xffffffffu, g, o);
    const double ov = __shfl_xor_sync(0xffffffffu, gv, o);
    if (og < g) { g = og; gv = ov; }
  }
  if ((threadIdx.x & 31) == 0) {
    smg[threadIdx.x >> 5] = g;
    smv[threadIdx.x >> 5] = gv;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < RSB_WARPS; ++i)
      if (smg[i] < g) { g = smg[i]; gv = smv[i]; }
    partials[blockIdx.x] = (double)g;
    partials[stride + blockIdx.x] = gv;
  }
  if (last_cta(&u.cnt, u.ntile)) {
    if (threadIdx.x < 32) {
      double bg = 1e300, bv = 0.0;
      for (int i = threadIdx.x; i < u.ntile; i += 32) {
        const double pg = __ldcg(partials + u.tile0 + i);
        const double pv = __ldcg(partials + stride + u.tile0 + i);
        if (pg < bg) { bg = pg; bv = pv; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double og = __shfl_xor_sync(0xffffffffu, bg, o);
        const double ov = __shfl_xor_sync(0xffffffffu, bv, o);
        if (og < bg) { bg = og; bv = ov; }
      }
      if (threadIdx.x != 0) return;
      u.gstar = (int64_t)bg;
      u.gstar_v = bv;
      u.sign = fixed_sign ? 1.0 : (bv > 0.0 ? -1.0 : 1.0);
      u.tau = tie_rel * (u.vmax - u.vmin);
    }
  }
}

// fixed_sign: keep v as it is (RCB: lower coordinates go left)
int launch_orient(const LevelGraph& G, const Tile* tiles, int ntiles, Unit* units,
                  const uint64_t* ckey, const double* v, int cand, double tie_rel,
                  double* partials, cudaStream_t s, int fixed_sign) {
  if (ntiles <= 0) return RSB_OK;
  k_orient_stats<<<ntiles, RSB_BLOCK, 0, s>>>(tiles, units, ckey, v, cand, partials, ntiles);
  RSB_CKL("k_orient_stats");
  k_orient_gstar<<<ntiles, RSB_BLOCK, 0, s>>>(G.gid, tiles, units, ckey, v, cand, tie_rel,
                                              partials, ntiles, fixed_sign);
  RSB_CKL("k_orient_gstar");
  return RSB_OK;
}

// ----------------------------------------------------------------------------
// segmented radix select
// ----------------------------------------------------------------------------
// The order of the values that are split: their integer keys, with -0 and +0 one value
// and every NaN (of either sign) one value above all others.  Coordinates are the
// caller's, and a unit's parts have their sizes whatever lies in them.
// The key of -x is 0 - the key of x.
__device__ __forceinline__ uint64_t split_key(double x, bool neg) {
  uint64_t b = (uint64_t)__double_as_longlong(x);
  // (the same test on k, which lies between the infinities' keys, by a subtraction and one
  // unsigned comparison, is compiled wrongly by nvcc 13.0)
  const bool nan = (b & 0x7FFFFFFFFFFFFFFFull) > 0x7FF0000000000000ull;
  if (neg) b ^= 0x8000000000000000ull;
  const uint64_t k = (b >> 63) ? 0ull - b : b | 0x8000000000000000ull;
  return nan ? ~0ull : k;
}
__device__ __forceinline__ double split_value(uint64_t k) {
  return __longlong_as_double(
      (long long)((k >> 63) ? k & 0x7FFFFFFFFFFFFFFFull : 0ull - k));
}

// Reading R7's window about the k-th value vk: a row below it goes left, a row in it is a
// tie.  A row of a key up to vk's is one or the other and at most k - 1 rows are below,
// so the ties always make up the k, also when vk or the range (and with it tau) is not
// finite: an infinite range makes every number a tie, a range that is no number leaves
// the exact ties.  Keys decide but for the rows just above vk, because an FP64
// comparison holds an SM sub-partition for 64 cycles.
struct TieWindow {
  uint64_t klim, kvk, khi;
  double vk, tau;
  __device__ __forceinline__ TieWindow(double v, double t) : vk(v), tau(t >= 0.0 ? t : 0.0) {
    klim = kvk = khi = split_key(vk, false);
    if (kvk == ~0ull) return;  // (nothing is computed from a NaN)
    if (isinf(tau)) {
      khi = split_key(tau, false);
      klim = 0ull - khi;
    } else {
      klim = split_key(vk - tau, false);
      khi = split_key(vk + 1.5 * tau, false);
    }
  }
  __device__ __forceinline__ bool below(uint64_t key) const { return key < klim; }
  // (x: the value of the key)
  __device__ __forceinline__ bool tie(uint64_t key, double x) const {
    return key >= klim && (key <= kvk || (key <= khi && x - vk <= tau));
  }
};

// mode 0: key = order bits of sign * v over unit rows, rank u.k -> u.vk
// mode 1: key = gid over tie rows (TieWindow), rank k-below     -> u.sel_prefix
// mode 2: key = component key over all unit rows, rank u.k           -> u.sel_prefix
enum { SEL_VALUE = 0, SEL_TIEGID = 1, SEL_COMP = 2 };

__device__ __forceinline__ bool sel_member(const Unit& u, int mode, int r, const uint64_t* ckey,
                                           const double* v, const int64_t* gid,
                                           const TieWindow& win, uint64_t& key) {
  if (mode == SEL_COMP) {
    key = ckey[r];
    return true;
  }
  if (!unit_has(u, ckey, r)) return false;
  key = split_key(v[r], u.sign < 0.0);
  if (mode == SEL_VALUE) return true;
  if (!win.tie(key, u.sign * v[r])) return false;
  key = (uint64_t)gid[r];
  return true;
}

__global__ void k_sel_init(Unit* units, int nunits, int mode, int cand) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nunits) return;
  Unit& u = units[i];
  if (!u.valid || (mode != SEL_COMP && cand >= u.ncand)) return;
  u.sel_prefix = 0;
  u.sel_below = 0;
  u.sel_eq = 0;
  u.sel_k = (mode == SEL_TIEGID) ? (u.k - u.below) : u.k;
}

__global__ void __launch_bounds__(RSB_BLOCK)
    k_sel_hist(const int64_t* __restrict__ gid, const Tile* __restrict__ tiles, const Unit* units,
               const uint64_t* __restrict__ ckey, const double* __restrict__ v, int mode, int cand,
               int shift, int* __restrict__ hist) {
  __shared__ int sh[256];
  const Tile t = tiles[blockIdx.x];
  const Unit& u = units[t.unit];
  if (!u.valid || (mode != SEL_COMP && cand >= u.ncand)) return;
  sh[threadIdx.x] = 0;
  __syncthreads();
  const uint64_t himask = shift >= 56 ? 0ull : (~0ull << (shift + 8));
  const uint64_t want = u.sel_prefix & himask;
  const TieWindow win(u.vk, u.tau);
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    uint64_t key;
    if (!sel_member(u, mode, r, ckey, v, gid, win, key)) continue;
    if ((key & himask) != want) continue;
    atomicAdd(&sh[(key >> shift) & 255u], 1);
  }
  __syncthreads();
  const int c = sh[threadIdx.x];
  if (c) atomicAdd(hist + (long long)t.unit * 256 + threadIdx.x, c);
}

__global__ void __launch_bounds__(256) k_sel_scan(Unit* units, int mode, int cand, int shift,
                                                  int* hist) {
  __shared__ int sc[256];
  Unit& u = units[blockIdx.x];
  if (!u.valid || (mode != SEL_COMP && cand >= u.ncand)) return;
  int* h = hist + (long long)blockIdx.x * 256;
  const int c = h[threadIdx.x];
  sc[threadIdx.x] = c;
  __syncthreads();
  for (int o = 1; o < 256; o <<= 1) {
    const int x = threadIdx.x >= (unsigned)o ? sc[threadIdx.x - o] : 0;
    __syncthreads();
    sc[threadIdx.x] += x;
    __syncthreads();
  }
  const long long incl = sc[threadIdx.x];
  const long long excl = incl - c;
  const long long k = u.sel_k;
  if (c > 0 && excl < k && k <= incl) {
    u.sel_k = k - excl;
    u.sel_below += excl;
    u.sel_prefix |= (uint64_t)threadIdx.x << shift;
    u.sel_eq = c;
    if (shift == 0 && mode == SEL_VALUE) u.vk = split_value(u.sel_prefix);
  }
  h[threadIdx.x] = 0;
}

int launch_select(const LevelGraph& G, const Tile* tiles, int ntiles, Unit* units, int nunits,
                  const uint64_t* ckey, const double* v, int mode, int cand, int* hist,
                  cudaStream_t s) {
  if (ntiles <= 0 || nunits <= 0) return RSB_OK;
  k_sel_init<<<(nunits + 255) / 256, 256, 0, s>>>(units, nunits, mode, cand);
  RSB_CKL("k_sel_init");
  for (int shift = 56; shift >= 0; shift -= 8) {
    k_sel_hist<<<ntiles, RSB_BLOCK, 0, s>>>(G.gid, tiles, units, ckey, v, mode, cand, shift, hist);
    RSB_CKL("k_sel_hist");
    k_sel_scan<<<nunits, 256, 0, s>>>(units, mode, cand, shift, hist);
    RSB_CKL("k_sel_scan");
  }
  return RSB_OK;
}

// ----------------------------------------------------------------------------
// R7: rows strictly below the tie window, then the side bit of candidate cand
// ----------------------------------------------------------------------------
__global__ void __launch_bounds__(RSB_BLOCK)
    k_split_below(const Tile* __restrict__ tiles, Unit* units, const uint64_t* __restrict__ ckey,
                  const double* __restrict__ v, int cand, double* partials, long long stride) {
  __shared__ double sm[RSB_WARPS];
  __shared__ double out[1];
  const Tile t = tiles[blockIdx.x];
  Unit& u = units[t.unit];
  if (!u.valid || cand >= u.ncand) return;
  const TieWindow win(u.vk, u.tau);
  int cnt = 0;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK)
    if (unit_has(u, ckey, r)) cnt += win.below(split_key(v[r], u.sign < 0.0));
  const double c = block_sum((double)cnt, sm);
  if (threadIdx.x == 0) partials[blockIdx.x] = c;
  if (last_cta(&u.cnt, u.ntile)) {
    final_reduce(partials, stride, u.tile0, u.ntile, 1, out);
    if (threadIdx.x == 0) u.below = (int64_t)out[0];
  }
}

int launch_split_below(const LevelGraph& G, const Tile* tiles, int ntiles, Unit* units,
                       const uint64_t* ckey, const double* v, int cand, double* partials,
                       cudaStream_t s) {
  (void)G;
  if (ntiles <= 0) return RSB_OK;
  k_split_below<<<ntiles, RSB_BLOCK, 0, s>>>(tiles, units, ckey, v, cand, partials, ntiles);
  RSB_CKL("k_split_below");
  return RSB_OK;
}

__global__ void __launch_bounds__(RSB_BLOCK)
    k_split_assign(const int64_t* __restrict__ gid, const Tile* __restrict__ tiles,
                   const Unit* units, const uint64_t* __restrict__ ckey,
                   const double* __restrict__ v, int cand, uint8_t* side) {
  const Tile t = tiles[blockIdx.x];
  const Unit& u = units[t.unit];
  if (!u.valid || cand >= u.ncand) return;
  const TieWindow win(u.vk, u.tau);
  const uint64_t gthr = u.sel_prefix;  // k''-th smallest tie gid
  const bool all_below = (u.k - u.below) <= 0;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    if (!unit_has(u, ckey, r)) continue;
    const uint64_t key = split_key(v[r], u.sign < 0.0);
    bool left = win.below(key);
    if (!left && !all_below && win.tie(key, u.sign * v[r])) left = (uint64_t)gid[r] <= gthr;
    const uint8_t bit = (uint8_t)(1u << cand);
    side[r] = left ? (uint8_t)(side[r] & ~bit) : (uint8_t)(side[r] | bit);
  }
}

int launch_split_assign(const LevelGraph& G, const Tile* tiles, int ntiles, Unit* units,
                        const uint64_t* ckey, const double* v, uint8_t* side, int cand,
                        cudaStream_t s) {
  if (ntiles <= 0) return RSB_OK;
  k_split_assign<<<ntiles, RSB_BLOCK, 0, s>>>(G.gid, tiles, units, ckey, v, cand, side);
  RSB_CKL("k_split_assign");
  return RSB_OK;
}

// ----------------------------------------------------------------------------
// The whole split of one candidate in one cooperative launch: orientation (R4), the
// k-th value, the tie window and the tie gid (R7), and the side bit of every row - the
// steps of k_orient_*, k_sel_*, k_split_below and k_split_assign above, which take 36
// launches and remain for levels of more tiles than SPLIT_MAXL a co-resident CTA.
// Bound: 20 grid barriers, 18 with a fixed sign (about 2 us each, whether or not a unit
// needs the pass), and, on large levels, one read of v from L2 for each radix pass.  A CTA
// walks its tiles in every phase and keeps their units' selection state; leading digits
// that all keys of a unit share (known from its smallest and largest key) take no read.  Values are compared as their integer keys, because an
// FP64 comparison holds an SM sub-partition for 64 cycles; only rows near the tie
// window take its FP64 test.  The split of a level of 512 rows 0.55 -> 0.12-0.26 ms (two
// or three candidates), of 2.1M rows by coordinates 0.5-0.9 -> 0.27-0.3 ms.
// ----------------------------------------------------------------------------
#define SPLIT_MAXL 32  // tiles of a CTA
#define SPLIT_BINS 256

// Per-unit scratch: zeroed (Z) and set to all ones (O) before the launch.
struct SplitZ {
  int hist[3][SPLIT_BINS];   // three buffers in turn: one filled, one read, one cleared
  unsigned long long kmax;   // largest key of a number
  unsigned long long nan;    // 1: there are NaNs
  unsigned long long tmax;
  unsigned long long below;
  unsigned long long sgn;    // 1: v[g*] <= 0, 2: v[g*] > 0
};
struct SplitO {
  unsigned long long kmin, tmin, gmin;
};

__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, x, o);
    x = y > x ? y : x;
  }
  return x;
}
__device__ __forceinline__ unsigned long long warp_min_u64(unsigned long long x) {
  return ~warp_max_u64(~x);
}
// first byte (0 = most significant) in which two keys differ; 8 when none does
__device__ __forceinline__ int first_byte(uint64_t a, uint64_t b) {
  return a == b ? 8 : __clzll((long long)(a ^ b)) >> 3;
}
__device__ __forceinline__ uint64_t top_bytes(uint64_t k, int n) {
  return n == 0 ? 0ull : n >= 8 ? k : k & ~(~0ull >> (8 * n));
}

__global__ void __launch_bounds__(RSB_BLOCK, 4)
    k_split(const int64_t* __restrict__ gid, const Tile* __restrict__ tiles, int ntiles, Unit* units,
            const uint64_t* __restrict__ ckey, const double* __restrict__ v, int cand, double tie_rel,
            int fixed_sign, uint8_t* side, SplitZ* Z, SplitO* O, unsigned* counter, GridBar* gb) {
  __shared__ int sh[SPLIT_BINS];
  __shared__ int wtot[RSB_WARPS];
  __shared__ uint64_t prefix[SPLIT_MAXL];
  __shared__ long long rank[SPLIT_MAXL];
  __shared__ int first[SPLIT_MAXL];       // passes before this one are decided; 8: none left
  __shared__ uint8_t neg[SPLIT_MAXL], on[SPLIT_MAXL];
  __shared__ uint64_t klim[SPLIT_MAXL], kvk[SPLIT_MAXL], khi[SPLIT_MAXL];
  __shared__ double vk[SPLIT_MAXL], tau[SPLIT_MAXL];
  __shared__ unsigned long long red[2][RSB_WARPS];
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int G = gridDim.x;
  UnitBar bar(counter, G, __ldcg(&gb->count), gb);
  // tiles blockIdx, blockIdx + G, ... of this CTA
  const int nl = (ntiles - (int)blockIdx.x + G - 1) / G;
  for (int l = tid; l < nl; l += RSB_BLOCK) {
    const Unit& u = units[tiles[blockIdx.x + l * G].unit];
    on[l] = u.valid && cand < u.ncand;
    neg[l] = 0;
  }
  __syncthreads();
  // smallest and largest key of every unit
  for (int l = 0; l < nl; ++l) {
    if (!on[l]) continue;
    const Tile t = tiles[blockIdx.x + l * G];
    const Unit& u = units[t.unit];
    unsigned long long hi = 0, lo = ~0ull;
    for (int r = t.row0 + tid; r < t.row1; r += RSB_BLOCK) {
      if (!unit_has(u, ckey, r)) continue;
      const uint64_t k = split_key(v[r], false);
      if (k == ~0ull) {
        Z[t.unit].nan = 1;
        continue;
      }
      hi = k > hi ? k : hi;
      lo = k < lo ? k : lo;
    }
    hi = warp_max_u64(hi);
    lo = warp_min_u64(lo);
    if (lane == 0) {
      red[0][w] = hi;
      red[1][w] = lo;
    }
    __syncthreads();
    if (w == 0) {
      hi = warp_max_u64(lane < RSB_WARPS ? red[0][lane] : 0ull);
      lo = warp_min_u64(lane < RSB_WARPS ? red[1][lane] : ~0ull);
      if (lane == 0 && lo <= hi) {
        atomicMax(&Z[t.unit].kmax, hi);
        atomicMin(&O[t.unit].kmin, lo);
      }
    }
    __syncthreads();
  }
  if (!bar.sync()) return;
  if (!fixed_sign) {
    // g*: the smallest gid with |v| >= max|v| / 2
    for (int l = 0; l < nl; ++l) {
      if (!on[l]) continue;
      const Tile t = tiles[blockIdx.x + l * G];
      const Unit& u = units[t.unit];
      const double amax = fmax(fabs(split_value(__ldcg(&Z[t.unit].kmax))),
                               fabs(split_value(__ldcg(&O[t.unit].kmin))));
      const uint64_t thr = split_key(0.5 * amax, false);
      unsigned long long g = ~0ull;
      for (int r = t.row0 + tid; r < t.row1; r += RSB_BLOCK) {
        if (!unit_has(u, ckey, r)) continue;
        const uint64_t key = split_key(v[r], false);
        if ((key >> 63 ? key : 0ull - key) >= thr && key != ~0ull) {
          const unsigned long long x = (unsigned long long)gid[r] ^ 0x8000000000000000ull;
          g = x < g ? x : g;
        }
      }
      g = warp_min_u64(g);
      if (lane == 0 && g != ~0ull) atomicMin(&O[t.unit].gmin, g);
    }
    if (!bar.sync()) return;
    for (int l = 0; l < nl; ++l) {  // the sign of v there (gids of a graph are distinct)
      if (!on[l]) continue;
      const Tile t = tiles[blockIdx.x + l * G];
      const Unit& u = units[t.unit];
      const int64_t g = (int64_t)(__ldcg(&O[t.unit].gmin) ^ 0x8000000000000000ull);
      for (int r = t.row0 + tid; r < t.row1; r += RSB_BLOCK)
        if (gid[r] == g && unit_has(u, ckey, r)) Z[t.unit].sgn = v[r] > 0.0 ? 2 : 1;
    }
    if (!bar.sync()) return;
  }
  // the k-th value, then among its ties the gid, a byte a pass
  for (int l = tid; l < nl; l += RSB_BLOCK) {
    first[l] = 8;
    if (!on[l]) continue;
    const int ui = tiles[blockIdx.x + l * G].unit;
    const bool ng = !fixed_sign && __ldcg(&Z[ui].sgn) == 2;
    uint64_t hi = __ldcg(&Z[ui].kmax), lo = __ldcg(&O[ui].kmin);
    if (ng) {  // keys of the negated values
      const uint64_t x = 0ull - lo;
      lo = 0ull - hi;
      hi = x;
    }
    if (__ldcg(&Z[ui].nan)) {  // (a unit of NaNs alone: one value)
      if (__ldcg(&O[ui].kmin) == ~0ull) lo = ~0ull;
      hi = ~0ull;
    }
    neg[l] = ng;
    rank[l] = units[ui].k;
    first[l] = first_byte(lo, hi);
    prefix[l] = top_bytes(lo, first[l]);
  }
  __syncthreads();
  for (int stage = 0; stage < 2; ++stage) {
    for (int p = 0; p < 8; ++p) {
      const int shift = 56 - 8 * p;
      const int buf = (stage * 8 + p) % 3, nxt = (buf + 1) % 3;
      const uint64_t himask = p == 0 ? 0ull : ~0ull << (shift + 8);
      for (int l = 0; l < nl; ++l) {
        if (!on[l]) continue;
        const Tile t = tiles[blockIdx.x + l * G];
        const Unit& u = units[t.unit];
        if (t.row0 == u.row0) Z[t.unit].hist[nxt][tid] = 0;  // read two passes ago
        if (p < first[l]) continue;
        sh[tid] = 0;
        __syncthreads();
        const uint64_t want = prefix[l] & himask;
        const bool ng = neg[l];
        for (int r = t.row0 + tid; r < t.row1; r += RSB_BLOCK) {
          if (!unit_has(u, ckey, r)) continue;
          uint64_t key = split_key(v[r], ng);
          if (stage == 1) {
            if (key < klim[l] || key > khi[l]) continue;
            if (key > kvk[l] && !((ng ? -v[r] : v[r]) - vk[l] <= tau[l])) continue;
            key = (uint64_t)gid[r];
          }
          if ((key & himask) == want) atomicAdd(&sh[(key >> shift) & 255u], 1);
        }
        __syncthreads();
        const int c = sh[tid];
        if (c) atomicAdd(&Z[t.unit].hist[buf][tid], c);
        __syncthreads();
      }
      if (!bar.sync()) return;
      for (int l = 0; l < nl; ++l) {
        if (!on[l] || p < first[l]) continue;
        const int ui = tiles[blockIdx.x + l * G].unit;
        const int c = __ldcg(&Z[ui].hist[buf][tid]);
        int x = c;  // inclusive sums over the bins
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, x, o);
          if (lane >= o) x += y;
        }
        if (lane == 31) wtot[w] = x;
        const long long k = rank[l];
        __syncthreads();
        for (int i = 0; i < w; ++i) x += wtot[i];
        if (c > 0 && x - c < k && k <= x) {
          rank[l] = k - (x - c);
          prefix[l] |= (uint64_t)tid << shift;
        }
        __syncthreads();
      }
    }
    if (stage == 1) break;
    // v_k, the rows below its tie window, the range of the ties' gids
    for (int l = tid; l < nl; l += RSB_BLOCK)
      if (on[l]) {
        const int ui = tiles[blockIdx.x + l * G].unit;
        // (of the numbers, and not beyond the starts of k_orient_stats)
        const double hi = fmax(-1e300, split_value(__ldcg(&Z[ui].kmax)));
        const double lo = fmin(1e300, split_value(__ldcg(&O[ui].kmin)));
        const TieWindow win(split_value(prefix[l]), tie_rel * (hi - lo));
        vk[l] = win.vk;
        tau[l] = win.tau;
        klim[l] = win.klim;
        kvk[l] = win.kvk;
        khi[l] = win.khi;
      }
    __syncthreads();
    for (int l = 0; l < nl; ++l) {
      if (!on[l]) continue;
      const Tile t = tiles[blockIdx.x + l * G];
      const Unit& u = units[t.unit];
      const bool ng = neg[l];
      int below = 0;
      unsigned long long hi = 0, lo = ~0ull;
      for (int r = t.row0 + tid; r < t.row1; r += RSB_BLOCK) {
        if (!unit_has(u, ckey, r)) continue;
        const uint64_t key = split_key(v[r], ng);
        below += key < klim[l];
        if (key >= klim[l] && key <= khi[l]) {
          if (key <= kvk[l] || (ng ? -v[r] : v[r]) - vk[l] <= tau[l]) {
            const unsigned long long g = (unsigned long long)gid[r];
            hi = g > hi ? g : hi;
            lo = g < lo ? g : lo;
          }
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) below += __shfl_xor_sync(0xffffffffu, below, o);
      hi = warp_max_u64(hi);
      lo = warp_min_u64(lo);
      if (lane == 0) {
        if (below) atomicAdd(&Z[t.unit].below, (unsigned long long)below);
        if (lo <= hi) {
          atomicMax(&Z[t.unit].tmax, hi);
          atomicMin(&O[t.unit].tmin, lo);
        }
      }
    }
    if (!bar.sync()) return;
    for (int l = tid; l < nl; l += RSB_BLOCK)
      if (on[l]) {
        const Tile t = tiles[blockIdx.x + l * G];
        Unit& u = units[t.unit];
        const long long below = (long long)__ldcg(&Z[t.unit].below);
        const uint64_t hi = __ldcg(&Z[t.unit].tmax), lo = __ldcg(&O[t.unit].tmin);
        rank[l] = u.k - below;
        // (no tie goes left: nothing to select)
        first[l] = rank[l] <= 0 || lo > hi ? 8 : first_byte(lo, hi);
        prefix[l] = rank[l] <= 0 || lo > hi ? 0ull : top_bytes(lo, first[l]);
        if (t.row0 == u.row0) {
          u.sign = neg[l] ? -1.0 : 1.0;
          u.vk = vk[l];
          u.tau = tau[l];
          u.below = below;
        }
      }
    __syncthreads();
  }
  // side bits
  for (int l = 0; l < nl; ++l) {
    if (!on[l]) continue;
    const Tile t = tiles[blockIdx.x + l * G];
    const Unit& u = units[t.unit];
    const bool ng = neg[l];
    // rank is 1-based among the ties until it is used up; a unit without a tie to its
    // left was given no passes and prefix 0
    const bool none = (long long)u.k - (long long)__ldcg(&Z[t.unit].below) <= 0;
    const uint64_t gthr = prefix[l];
    const uint8_t bit = (uint8_t)(1u << cand);
    for (int r = t.row0 + tid; r < t.row1; r += RSB_BLOCK) {
      if (!unit_has(u, ckey, r)) continue;
      const uint64_t key = split_key(v[r], ng);
      bool left = key < klim[l];
      if (!left && !none && key <= khi[l] &&
          (key <= kvk[l] || (ng ? -v[r] : v[r]) - vk[l] <= tau[l]))
        left = (uint64_t)gid[r] <= gthr;
      side[r] = left ? (uint8_t)(side[r] & ~bit) : (uint8_t)(side[r] | bit);
    }
  }
}

size_t split_scratch_bytes(int nunits) {
  return (sizeof(SplitZ) + sizeof(SplitO)) * (size_t)nunits + 256;
}

// scratch: split_scratch_bytes.  gb: its error word outlives the launch (a wait that ran
// out leaves the side bits unfinished; k_finalize_side then does not use them), its count
// is where the barrier's arrivals are expected to start, out of reach under the test hook.
// *done = 0 when the level has too many tiles for one
// co-resident launch (the caller then takes the steps one by one).
int launch_split(const LevelGraph& G, const Tile* tiles, int ntiles, Unit* units, int nunits,
                 const uint64_t* ckey, const double* v, int cand, double tie_rel, int fixed_sign,
                 uint8_t* side, void* scratch, GridBar* gb, cudaStream_t s, int* done) {
  *done = 0;
  if (ntiles <= 0 || nunits <= 0) {
    *done = 1;
    return RSB_OK;
  }
  int dev = 0, nsm = 0, occ = 0;
  RSB_CK(cudaGetDevice(&dev));
  RSB_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  RSB_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_split, RSB_BLOCK, 0));
  const int grid = std::min(ntiles, std::min(occ, 4) * nsm);  // (more only makes the barriers longer)
  if (grid <= 0 || (long long)grid * SPLIT_MAXL < ntiles) return RSB_OK;
  unsigned* counter = (unsigned*)scratch;
  SplitZ* Z = (SplitZ*)((char*)scratch + 256);
  SplitO* O = (SplitO*)(Z + nunits);
  RSB_CK(cudaMemsetAsync(scratch, 0, 256 + sizeof(SplitZ) * (size_t)nunits, s));
  RSB_CK(cudaMemsetAsync(O, 0xFF, sizeof(SplitO) * (size_t)nunits, s));
  if (g_rsb_poison_barrier)
    RSB_CK(cudaMemsetAsync(&gb->count, 0x40, sizeof(unsigned int), s));
  const int64_t* gid = G.gid;
  void* args[] = {(void*)&gid, (void*)&tiles, (void*)&ntiles, (void*)&units, (void*)&ckey, (void*)&v,
                  (void*)&cand, (void*)&tie_rel, (void*)&fixed_sign, (void*)&side, (void*)&Z,
                  (void*)&O, (void*)&counter, (void*)&gb};
  cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_split, grid, RSB_BLOCK, args, 0, s);
  rsb_count_launch();
  if (e != cudaSuccess) return rsb_set_cuda_error(e, "cudaLaunchCooperativeKernel(k_split)");
  *done = 1;
  return RSB_OK;
}

// ----------------------------------------------------------------------------
// R5 gid rule: smallest gid where candidates a and b disagree, and whether a
// has it on the left.  Result: u.best updated (a wins -> a, else b) among
// candidates of equal cut; the caller runs it after comparing cuts.
// ----------------------------------------------------------------------------
__global__ void __launch_bounds__(RSB_BLOCK)
    k_choose(const int64_t* __restrict__ gid, const Tile* __restrict__ tiles, Unit* units,
             const uint64_t* __restrict__ ckey, const uint8_t* __restrict__ side, int cb,
             double* partials, long long stride) {
  __shared__ long long smg[RSB_WARPS];
  __shared__ int sml[RSB_WARPS];
  const Tile t = tiles[blockIdx.x];
  Unit& u = units[t.unit];
  if (!u.valid || cb >= u.ncand) return;
  const int ca = u.best;
  long long g = LLONG_MAX;
  int aleft = 0;
  for (int r = t.row0 + threadIdx.x; r < t.row1; r += RSB_BLOCK) {
    if (!unit_has(u, ckey, r)) continue;
    const int sa = (side[r] >> ca) & 1, sb = (side[r] >> cb) & 1;
    if (sa != sb && gid[r] < g) {
      g = gid[r];
      aleft = sa == 0;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long og = __shfl_xor_sync(0xffffffffu, g, o);
    const int ol = __shfl_xor_sync(0xffffffffu, aleft, o);
    if (og < g) { g = og; aleft = ol; }
  }
  if ((threadIdx.x & 31) == 0) {
    smg[threadIdx.x >> 5] = g;
    sml[threadIdx.x >> 5] = aleft;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < RSB_WARPS; ++i)
      if (smg[i] < g) { g = smg[i]; aleft = sml[i]; }
    partials[blockIdx.x] = (double)g;
    partials[stride + blockIdx.x] = (double)aleft;
  }
  if (last_cta(&u.cnt, u.ntile)) {
    if (threadIdx.x < 32) {
      double bg = 1e300;
      int al = 1;
      for (int i = threadIdx.x; i < u.ntile; i += 32) {
        const double pg = __ldcg(partials + u.tile0 + i);
        const int pl = (int)__ldcg(partials + stride + u.tile0 + i);
        if (pg < bg) { bg = pg; al = pl; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double og = __shfl_xor_sync(0xffffffffu, bg, o);
        const int ol = __shfl_xor_sync(0xffffffffu, al, o);
        if (og < bg) { bg = og; al = ol; }
      }
      if (threadIdx.x != 0) return;
      const int64_t cut_a = u.cut[ca], cut_b = u.cut[cb];
      bool b_wins;
      if (cut_b != cut_a) b_wins = cut_b < cut_a;
      else b_wins = (bg < 1e300) && !al;  // equal cuts: the left set holding the smallest
                                          // differing gid wins (identical splits keep a)
      if (b_wins) u.best = cb;
    }
  }
}

int launch_choose(const LevelGraph& G, const Tile* tiles, int ntiles, Unit* units,
                  const uint64_t* ckey, const uint8_t* side, int cb, double* partials,
                  cudaStream_t s) {
  if (ntiles <= 0) return RSB_OK;
  k_choose<<<ntiles, RSB_BLOCK, 0, s>>>(G.gid, tiles, units, ckey, side, cb, partials, ntiles);
  RSB_CKL("k_choose");
  return RSB_OK;
}

// ----------------------------------------------------------------------------
// final side of every row of the level (0 left, 1 right)
// ----------------------------------------------------------------------------
// seg_split[s]: 1 when segment s is bisected at this level and connected, 2 when it
// is bisected and fell apart.
// seg_keystar[s]: component key of the straddling (or last fitting) component of a
// segment that fell apart.
// seg_unit[s]: unit solving the straddler, or -1 when components fit exactly.
// err: error word of the call's splits.  Once a wait of theirs ran out, the side bits may
// be anything; the call will fail, but its levels still run to the end, so every segment
// is then cut by row number, which gives the halves the sizes that the compaction relies on.
__global__ void k_finalize_side(const int32_t* __restrict__ row_seg, int32_t n,
                                const uint8_t* __restrict__ seg_split,
                                const uint64_t* __restrict__ seg_keystar,
                                const int32_t* __restrict__ seg_unit, const Unit* units,
                                const uint64_t* __restrict__ ckey,
                                const int64_t* __restrict__ seg_row0,
                                const int64_t* __restrict__ seg_nleft,
                                const int* __restrict__ err, uint8_t* side) {
  const int r = blockIdx.x * RSB_BLOCK + threadIdx.x;
  if (r >= n) return;
  const int s = row_seg[r];
  uint8_t out = 0;
  if (*err) {
    out = seg_split[s] && r - seg_row0[s] >= seg_nleft[s];
  } else if (seg_split[s]) {
    const uint64_t k = seg_split[s] == 2 ? ckey[r] : 0, ks = seg_split[s] == 2 ? seg_keystar[s] : 0;
    if (k < ks) out = 0;
    else if (k > ks) out = 1;
    else {
      const int ui = seg_unit[s];
      out = ui < 0 ? 0 : (uint8_t)((side[r] >> units[ui].best) & 1);
    }
  }
  side[r] = out;
}

int launch_finalize_side(const LevelGraph& G, const uint8_t* seg_split,
                         const uint64_t* seg_keystar, const int32_t* seg_unit, const Unit* units,
                         const uint64_t* ckey, const int64_t* seg_row0, const int64_t* seg_nleft,
                         const int* err, uint8_t* side, cudaStream_t s) {
  if (G.n <= 0) return RSB_OK;
  k_finalize_side<<<(G.n + RSB_BLOCK - 1) / RSB_BLOCK, RSB_BLOCK, 0, s>>>(
      G.row_seg, G.n, seg_split, seg_keystar, seg_unit, units, ckey, seg_row0, seg_nleft, err,
      side);
  RSB_CKL("k_finalize_side");
  return RSB_OK;
}
