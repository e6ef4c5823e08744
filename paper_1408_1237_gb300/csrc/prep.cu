// Point preparation (hot-path step A1): Hilbert- or Morton-order sort, scaling and
// tile-blocked packing of the points.
//
// The Gaussian of Eq. 2 becomes a base-2 exponential of scaled points:
//   exp(-|x_i - x_j|^2 / (2 sigma^2)) = 2^(-s^2 |x_i - x_j|^2),
//   s = sqrt(log2(e) / (2 sigma^2)),
// so the product kernels evaluate it with one MUFU.EX2 per pair.  (Under the
// Matern kernel of Sec. 6.1 the scale is s = sqrt(3) / h and the kernels form
// a = s |x_i - x_j|; every block takes the direct form.)  The packed
// copy keeps the caller's float32 coordinates unscaled: the kernels scale
// only after recentring or differencing, where no significant digits are
// lost (scaling first would round s*x at the magnitude of s*x).  Sorting the
// points along a Hilbert curve makes every block of consecutive
// points spatially compact, which the product kernels use to recentre their
// arithmetic (see mvp.cu).  K is invariant under a simultaneous permutation of
// rows and columns, so the solvers work in sorted order throughout and only
// the right-hand sides and solutions are permuted in and out.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "internal.h"

namespace krr {

namespace {

constexpr int SORT_THREADS = 256;
constexpr int SORT_ITEMS = 16;
constexpr int SORT_CHUNK = SORT_THREADS * SORT_ITEMS;  // elements per sort block
constexpr int SCAN_THREADS = 1024;
constexpr int BBOX_THREADS = 256;
constexpr int BBOX_BLOCKS = 152;                       // partial boxes, one block per SM
// Up to this many points one cluster of CL_SIZE CTAs sorts the keys in shared memory.
constexpr int CL_SIZE = 8;
constexpr int CL_THREADS = 1024;
constexpr int CL_MAX_ITEMS = 16;
constexpr int64_t CL_MAX_N = (int64_t)CL_SIZE * CL_THREADS * CL_MAX_ITEMS;

// Per-block partial bounding boxes: part[b*2d + k] = min, part[b*2d + d + k] = max.
// Non-finite coordinates raise DEV_NONFINITE.  X is read as one flat array: a
// block has a multiple of d threads, so a thread keeps one coordinate k and
// every load is coalesced (a strided loop per coordinate took 10.5 us at
// d = 25, 32768 points).
__global__ void bbox_kernel(const float* __restrict__ X, int64_t total, int d,
                            float* __restrict__ part, int* err) {
  __shared__ float slo[BBOX_THREADS], shi[BBOX_THREADS];
  const int tid = threadIdx.x;
  float lo = INFINITY, hi = -INFINITY;
  bool bad = false;
  for (int64_t f = (int64_t)blockIdx.x * blockDim.x + tid; f < total; f += (int64_t)gridDim.x * blockDim.x) {
    const float v = X[f];
    if (!isfinite(v)) bad = true;
    lo = fminf(lo, v);
    hi = fmaxf(hi, v);
  }
  if (bad) atomicExch(err, DEV_NONFINITE);
  slo[tid] = lo;
  shi[tid] = hi;
  __syncthreads();
  for (int t = tid; t < 2 * d; t += blockDim.x) {
    const bool is_min = t < d;
    float v = is_min ? INFINITY : -INFINITY;
    for (int e = is_min ? t : t - d; e < (int)blockDim.x; e += d) v = is_min ? fminf(v, slo[e]) : fmaxf(v, shi[e]);
    part[(int64_t)blockIdx.x * 2 * d + t] = v;
  }
}

// Hilbert-curve key over the first dk = min(d, 30) coordinates, `bits` bits
// each (J. Skilling, "Programming the Hilbert curve", AIP Conf. Proc. 707,
// 2004: the axes are turned into the transposed index in place, then its bits
// are interleaved, coordinate 0 most significant).  Consecutive cells of the
// curve are neighbours, where the Morton curve jumps across the cloud at every
// power of two, so runs of 256 points are more compact: of 131,072 points in
// the unit cube at sigma = 0.05, 38% of the super-blocks were too wide for the
// expanded form in Morton order and none are in Hilbert order; at 65,541
// points 84% and 32%; at 2^20 points 3% and none.
// hilbert = 0 interleaves the cells themselves (Morton order; the caller
// says why).  DK > 0: the coordinate count at compile time, the axes in
// registers; DK = 0: more than 8 coordinates (at most 3 bits each).
// Every block first folds the partial boxes (a few KB from L2) instead of
// waiting for one more launch.
template <int DK>
__global__ void __launch_bounds__(256)
    key_kernel(const float* __restrict__ X, int64_t N, int d, int dk_any, int bits, int hilbert,
               const float* __restrict__ part, int nparts, uint32_t* __restrict__ keys, int* __restrict__ vals) {
  __shared__ float box[60];  // lo of coordinates 0..dk-1, then hi
  const int dk = DK > 0 ? DK : dk_any;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int e = warp; e < 2 * dk; e += 8) {
    const bool is_min = e < dk;
    const int src = is_min ? e : d + e - dk;
    float v = is_min ? INFINITY : -INFINITY;
    for (int b = lane; b < nparts; b += 32) {
      const float u = part[(int64_t)b * 2 * d + src];
      v = is_min ? fminf(v, u) : fmaxf(v, u);
    }
    v = is_min ? warp_min(v) : warp_max(v);
    if (lane == 0) box[e] = v;
  }
  __syncthreads();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const uint32_t cells = 1u << bits;
  uint32_t x[DK > 0 ? DK : 30];
#pragma unroll
  for (int k = 0; k < dk; ++k) {
    const float lo = box[k], hi = box[dk + k];
    const float ext = hi - lo;
    uint32_t u = 0;
    if (ext > 0.f) {
      float f = (X[i * d + k] - lo) / ext * (float)cells;
      f = fminf(fmaxf(f, 0.f), (float)(cells - 1));
      u = (uint32_t)f;
    }
    x[k] = u;
  }
  if (hilbert) {
    // undo the rotations and reflections from the top bit down
    for (uint32_t q = cells >> 1; q > 1; q >>= 1) {
      const uint32_t low = q - 1;
#pragma unroll
      for (int k = 0; k < dk; ++k) {
        const uint32_t t = (x[0] ^ x[k]) & low;
        const bool set = (x[k] & q) != 0;
        x[0] ^= set ? low : t;
        if (k > 0) x[k] ^= set ? 0u : t;
      }
    }
    // Gray encode
#pragma unroll
    for (int k = 1; k < dk; ++k) x[k] ^= x[k - 1];
    uint32_t t = 0;
    for (uint32_t q = cells >> 1; q > 1; q >>= 1)
      if (x[dk - 1] & q) t ^= q - 1;
#pragma unroll
    for (int k = 0; k < dk; ++k) x[k] ^= t;
  }
  uint32_t key = 0;
#pragma unroll
  for (int k = 0; k < dk; ++k) {
    const int at = hilbert ? dk - 1 - k : k;
    for (int b = 0; b < bits; ++b) key |= ((x[k] >> b) & 1u) << (b * dk + at);
  }
  keys[i] = key;
  if (vals) vals[i] = (int)i;
}

// Stable ranks of a block's elements by one 8-bit digit.  The element order is
// (warp, item, lane); cnt holds 256 counters per warp.  The rank of item i is
// the element's rank among its warp's equal digits; after a barrier the
// caller scans the counters over the warps.  Elements whose bit of `valid` is
// clear are left out.  A warp ranks 32 elements per step: the lanes with equal
// digits come from 8 ballots (one match instruction took 24 us per pass at 16
// items); put(i, rank) takes the results.
template <int ITEMS, typename Put>
__device__ __forceinline__ void warp_digit_ranks(const uint32_t (&key)[ITEMS], uint32_t valid, int shift,
                                                 uint32_t* cnt, Put put) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const bool v = (valid >> i) & 1u;
    const uint32_t digit = (key[i] >> shift) & 0xFFu;
    uint32_t peers = __ballot_sync(0xffffffffu, v);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const bool set = (digit >> b) & 1u;
      const uint32_t have = __ballot_sync(0xffffffffu, set);
      peers &= set ? have : ~have;
    }
    const uint32_t below = __popc(peers & ((1u << lane) - 1u));
    uint32_t base = 0;
    if (v) base = cnt[digit];
    __syncwarp();
    if (v && below == 0) cnt[digit] = base + __popc(peers);
    __syncwarp();
    put(i, base + below);
  }
}

// Exclusive scan of one value per thread over the 256 threads of warps 0..7
// (all threads of the block call it; ws: 8 words of shared memory).
__device__ __forceinline__ uint32_t scan256(uint32_t v, uint32_t* ws) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  uint32_t x = v;
  if (t < 256) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) ws[warp] = x;
  }
  __syncthreads();
  uint32_t add = 0;
  if (t < 256) {
#pragma unroll
    for (int w = 0; w < 8; ++w)
      if (w < warp) add += ws[w];
  }
  return x - v + add;
}

// ---- cluster sort: the whole stable LSD radix sort of N <= CL_MAX_N keys in
// one launch.  The elements live in the shared memory of CL_SIZE CTAs (position
// p in CTA p / E, slot p % E, E = ITEMS * CL_THREADS); each 8-bit pass sorts a
// CTA's elements by digit in its own shared memory, exchanges the CTAs' digit
// counts and writes the digit runs to their places through distributed shared
// memory.  Two cluster barriers per pass replace three launches and a
// single-block scan, whose 4 x 46 us of kernels at 50,000 points were latency:
// the product over 4096 points went from 293 to 72 us, over 50,021 from 729
// to 539 us.  (Without the local sort every lane of a remote store has its
// own target row: the sort took 51 us at 50,021 points and 113 us at 131,072.)
template <int ITEMS>
constexpr size_t cluster_sort_smem() {
  return (size_t)ITEMS * CL_THREADS * 8 + (CL_THREADS / 32) * 256 * 4;
}

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_shared(const void* p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
  return r;
}

template <int ITEMS>
__global__ void __launch_bounds__(CL_THREADS, 1)
    cluster_sort_kernel(const uint32_t* __restrict__ keys, int N, int key_bits, int* __restrict__ perm) {
  constexpr int E = ITEMS * CL_THREADS;
  extern __shared__ __align__(16) uint2 sbuf[];  // E (key, value) pairs, then the warps' counters
  uint32_t* cnt = reinterpret_cast<uint32_t*>(sbuf + E);
  __shared__ uint32_t ctot[256], off[256], ws[8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cta = blockIdx.x;  // one cluster: the block index is the rank
  const int base = cta * E + warp * 32 * ITEMS + lane;
  // vr: the element's index (17 bits) and its rank in its warp (9 bits), one
  // register, so that 16 items fit the 64 registers of a 1024-thread block
  uint32_t key[ITEMS], vr[ITEMS];
  uint32_t valid = 0;
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const int p = base + 32 * i;
    if (p < N) valid |= 1u << i;
    key[i] = p < N ? keys[p] : 0u;
    vr[i] = (uint32_t)p;
  }
  for (int shift = 0; shift < key_bits; shift += 8) {
    const bool last = shift + 8 >= key_bits;
    if (shift > 0) {
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) {
        const uint2 kv = sbuf[warp * 32 * ITEMS + 32 * i + lane];
        key[i] = kv.x;
        vr[i] = kv.y;
      }
    }
    uint32_t* wc = cnt + warp * 256;
#pragma unroll
    for (int e = 0; e < 8; ++e) wc[lane + 32 * e] = 0u;
    __syncwarp();
    warp_digit_ranks<ITEMS>(key, valid, shift, wc, [&](int i, uint32_t r) { vr[i] |= r << 17; });
    __syncthreads();  // counters complete; every element of this CTA is in registers
    uint32_t total = 0;
    if (tid < 256) {
#pragma unroll 8
      for (int w = 0; w < CL_THREADS / 32; ++w) {
        const uint32_t c = cnt[w * 256 + tid];
        cnt[w * 256 + tid] = total;
        total += c;
      }
      ctot[tid] = total;
    }
    const uint32_t start = scan256(total, ws);  // this CTA's first slot of the digit
    if (tid < 256) off[tid] = start;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      if (!((valid >> i) & 1u)) continue;
      const uint32_t digit = (key[i] >> shift) & 0xFFu;
      sbuf[off[digit] + wc[digit] + (vr[i] >> 17)] = make_uint2(key[i], vr[i] & 0x1FFFFu);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      const uint2 kv = sbuf[warp * 32 * ITEMS + 32 * i + lane];
      key[i] = kv.x;
      vr[i] = kv.y;
    }
    cluster_barrier();  // counts published; every CTA's elements are in registers again
    uint32_t below = 0, all = 0;
    if (tid < 256) {
#pragma unroll
      for (int c = 0; c < CL_SIZE; ++c) {
        uint32_t v;
        asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(map_shared(&ctot[tid], c)) : "memory");
        if (c < cta) below += v;
        all += v;
      }
    }
    const uint32_t first = scan256(all, ws);
    // slot e of a digit's run goes to position off[digit] + e (modulo 2^32)
    if (tid < 256) off[tid] = first + below - start;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      if (!((valid >> i) & 1u)) continue;
      const uint32_t pos = off[(key[i] >> shift) & 0xFFu] + (uint32_t)(warp * 32 * ITEMS + 32 * i + lane);
      if (last) {
        perm[pos] = (int)vr[i];
      } else {
        const uint32_t a = map_shared(&sbuf[pos % E], pos / E);
        asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(key[i]), "r"(vr[i]) : "memory");
      }
    }
    cluster_barrier();  // scatter complete (and no CTA leaves while others read its counts)
  }
}

// ---- larger sorts: three launches per 8-bit pass.
// 1: digit histogram of each chunk, stored digit-major: hist[digit * nchunks + chunk].
__global__ void radix_hist_kernel(const uint32_t* __restrict__ keys, int64_t N, int shift,
                                  uint32_t* __restrict__ hist, int nchunks) {
  __shared__ uint32_t h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * SORT_CHUNK;
#pragma unroll
  for (int e = 0; e < SORT_ITEMS; ++e) {
    const int64_t i = base + e * SORT_THREADS + threadIdx.x;
    if (i < N) atomicAdd(&h[(keys[i] >> shift) & 0xFFu], 1u);
  }
  __syncthreads();
  hist[(int64_t)threadIdx.x * nchunks + blockIdx.x] = h[threadIdx.x];
}

// 2: exclusive scan of each digit's row over the chunks (one block per digit),
// with the digit's total in tot[digit]; the scatter scans the 256 totals.
// (One block scanning all 256 rows took 212 us per pass at 2^20 points.)
__global__ void __launch_bounds__(256) radix_scan_kernel(uint32_t* __restrict__ hist, int nchunks,
                                                         uint32_t* __restrict__ tot) {
  __shared__ uint32_t ws[8];
  __shared__ uint32_t carry_s;
  uint32_t* row = hist + (int64_t)blockIdx.x * nchunks;
  uint32_t carry = 0;
  for (int c0 = 0; c0 < nchunks; c0 += 256) {
    const int c = c0 + threadIdx.x;
    const uint32_t v = c < nchunks ? row[c] : 0u;
    const uint32_t ex = scan256(v, ws);
    if (c < nchunks) row[c] = carry + ex;
    if (threadIdx.x == 255) carry_s = ex + v;
    __syncthreads();
    carry += carry_s;
    __syncthreads();
  }
  if (threadIdx.x == 0) tot[blockIdx.x] = carry;
}

// 3: stable scatter (ranks as in the cluster sort; a thread per element
// instead of one per digit walking the whole chunk: 132 us per pass before at
// 2^20 points).
__global__ void __launch_bounds__(SORT_THREADS)
    radix_scatter_kernel(const uint32_t* __restrict__ keys_in, const int* __restrict__ vals_in, int64_t N, int shift,
                         const uint32_t* __restrict__ hist, int nchunks, const uint32_t* __restrict__ tot,
                         uint32_t* __restrict__ keys_out, int* __restrict__ vals_out) {
  __shared__ uint32_t cnt[SORT_THREADS / 32 * 256];
  __shared__ uint32_t ws[8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t base = (int64_t)blockIdx.x * SORT_CHUNK + warp * 32 * SORT_ITEMS + lane;
  uint32_t key[SORT_ITEMS], rank[SORT_ITEMS];
  int val[SORT_ITEMS];
  uint32_t valid = 0;
#pragma unroll
  for (int i = 0; i < SORT_ITEMS; ++i) {
    const int64_t p = base + 32 * i;
    if (p < N) valid |= 1u << i;
    key[i] = p < N ? keys_in[p] : 0u;
    val[i] = p < N ? vals_in[p] : 0;
  }
  uint32_t* wc = cnt + warp * 256;
#pragma unroll
  for (int e = 0; e < 8; ++e) wc[lane + 32 * e] = 0u;
  __syncwarp();
  warp_digit_ranks<SORT_ITEMS>(key, valid, shift, wc, [&](int i, uint32_t r) { rank[i] = r; });
  const uint32_t first = scan256(tot[tid], ws);  // holds a block barrier
  uint32_t run = first + hist[(int64_t)tid * nchunks + blockIdx.x];
#pragma unroll
  for (int w = 0; w < SORT_THREADS / 32; ++w) {
    const uint32_t c = cnt[w * 256 + tid];
    cnt[w * 256 + tid] = run;
    run += c;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < SORT_ITEMS; ++i) {
    if (!((valid >> i) & 1u)) continue;
    const uint32_t pos = wc[(key[i] >> shift) & 0xFFu] + rank[i];
    keys_out[pos] = key[i];
    vals_out[pos] = val[i];
  }
}

// Tile-blocked pack of one tile of TS points per block, and its metadata.
//   xs[(i/TS)*d*TS + k*TS + i%TS] = X[perm[i]*d_in + k]; the padded points
//   i >= N repeat the last sorted point (their weights are zero), so every
//   coordinate the product kernels meet is finite and nearby; they leave every
//   bounding box and radius below unchanged.
//   tbox: the tile's box, centre then half-width per dimension.
//   Warp blocks of 32*T points and super-blocks of SB = TS points: centre of
//   the bounding box (raw coordinates), and flag 1 when every point lies within
//   squared radius EXPANDED_R2 of it in scaled units s (x - c).
// One launch reads X once; five launches read the packed copy four times
// before (26 us of them at d = 25, 32768 points).
struct PackOut {
  float *xs, *tbox, *ctr, *sb_ctr;
  int *flag, *sb_flag;
};

__global__ void __launch_bounds__(TS)
    pack_kernel(const float* __restrict__ X, int64_t N, int d_in, int d, const int* __restrict__ perm, int T,
                int64_t nblk, int64_t nsb, float s, int allow_expanded, int allow_expanded_sb, const PackOut o) {
  __shared__ float wlo[8][64], whi[8][64], wctr[8][64], tctr[64];
  __shared__ float wr2[8], tr2[8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t tile = blockIdx.x;
  const int64_t i = tile * TS + tid;
  const float* row = X + (int64_t)perm[i < N ? i : N - 1] * d_in;
  float* dst = o.xs + tile * (int64_t)d * TS + tid;
  bool finite = true;
  for (int k = 0; k < d; ++k) {
    const float v = k < d_in ? row[k] : 0.f;  // padded coordinates: 0
    dst[(int64_t)k * TS] = v;
    finite = finite && isfinite(v);
    const float lo = warp_min(v), hi = warp_max(v);
    if (lane == 0) {
      wlo[warp][k] = lo;
      whi[warp][k] = hi;
    }
  }
  // min and max pass over NaN: the box of a tile with a coordinate that is not
  // finite is NaN (near to everything)
  const bool tile_finite = __syncthreads_and(finite);
  // the tile's box (and super-block centre), then each group of T warps
  for (int k = tid; k < d; k += TS) {
    float lo = wlo[0][k], hi = whi[0][k];
    for (int w = 1; w < 8; ++w) {
      lo = fminf(lo, wlo[w][k]);
      hi = fmaxf(hi, whi[w][k]);
    }
    const float c = 0.5f * (lo + hi);
    tctr[k] = c;
    o.tbox[tile * 2 * d + k] = tile_finite ? c : NAN;
    o.tbox[tile * 2 * d + d + k] = 0.5f * (hi - lo);
    if (tile < nsb) o.sb_ctr[tile * d + k] = c;
  }
  const int groups = 8 / T;
  for (int e = tid; e < groups * d; e += TS) {
    const int g = e / d, k = e % d;
    float lo = wlo[g * T][k], hi = whi[g * T][k];
    for (int w = 1; w < T; ++w) {
      lo = fminf(lo, wlo[g * T + w][k]);
      hi = fmaxf(hi, whi[g * T + w][k]);
    }
    const float c = 0.5f * (lo + hi);
    wctr[g][k] = c;
    const int64_t b = tile * groups + g;
    if (b < nblk) o.ctr[b * d + k] = c;
  }
  __syncthreads();
  const int g = warp / T;
  float aw = 0.f, at = 0.f;
  for (int k = 0; k < d; ++k) {
    const float v = k < d_in ? row[k] : 0.f;
    const float vw = s * (v - wctr[g][k]), vt = s * (v - tctr[k]);
    aw = fmaf(vw, vw, aw);
    at = fmaf(vt, vt, at);
  }
  aw = warp_max(aw);
  at = warp_max(at);
  if (lane == 0) {
    wr2[warp] = aw;
    tr2[warp] = at;
  }
  __syncthreads();
  if (tid < groups) {
    float r2 = wr2[tid * T];
    for (int w = 1; w < T; ++w) r2 = fmaxf(r2, wr2[tid * T + w]);
    const int64_t b = tile * groups + tid;
    if (b < nblk) o.flag[b] = (allow_expanded && r2 <= EXPANDED_R2) ? 1 : 0;
  }
  if (tid == 32 && tile < nsb) {
    float r2 = tr2[0];
    for (int w = 1; w < 8; ++w) r2 = fmaxf(r2, tr2[w]);
    o.sb_flag[tile] = (allow_expanded_sb && r2 <= EXPANDED_R2) ? 1 : 0;
  }
}

__global__ void unpack_kernel(const float* __restrict__ xs, int64_t N, int d_in, int d, const int* __restrict__ perm,
                              float* __restrict__ X) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const float* src = xs + i / TS * (int64_t)d * TS + i % TS;
  float* row = X + (int64_t)perm[i] * d_in;
  for (int k = 0; k < d_in; ++k) row[k] = src[(int64_t)k * TS];
}

// (Npad is a multiple of the block: no thread leaves early)
__global__ void __launch_bounds__(TS)
    gather_kernel(const float* __restrict__ in, int64_t N, int m, const int* __restrict__ perm, int64_t Npad,
                  float* __restrict__ out, int* __restrict__ qbad) {
  pdl_trigger();  // a product kernel reads only prepared points before its wait
  const int64_t i = (int64_t)blockIdx.x * TS + threadIdx.x;
  const int64_t p = i < N ? perm[i] : -1;
  bool bad = false;
  for (int c = 0; c < m; ++c) {
    const float v = p >= 0 ? in[(int64_t)c * N + p] : 0.f;
    out[(int64_t)c * Npad + i] = v;
    bad |= !(fabsf(v) < 65504.f);
  }
  if (qbad) {
    const int any = __syncthreads_or(bad);
    if (threadIdx.x == 0) qbad[blockIdx.x] = any ? 1 : 0;
  }
}

__global__ void scatter_kernel(const float* __restrict__ in, int64_t Npad, int64_t N, int m,
                               const int* __restrict__ perm, float* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int64_t p = perm[i];
  for (int c = 0; c < m; ++c) out[(int64_t)c * N + p] = in[(int64_t)c * Npad + i];
}

// Stable partition of the warp blocks (block 0) and the super-blocks (block 1):
// expanded-form blocks first.  *n_exp = number of expanded-form blocks, also
// written to the pinned host word host_n when there is one (the host sizes its
// grids from it).
struct OrderArgs {
  const int* flag;
  int64_t nblk;
  int *order, *n_exp, *host_n;
};

__global__ void __launch_bounds__(SCAN_THREADS) order_kernel(const OrderArgs warp_blocks, const OrderArgs super_blocks) {
  const OrderArgs a = blockIdx.x == 0 ? warp_blocks : super_blocks;
  __shared__ int wsum[SCAN_THREADS / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t per = (a.nblk + SCAN_THREADS - 1) / SCAN_THREADS;
  const int64_t lo = tid * per, hi = min(a.nblk, lo + per);
  int cnt = 0;
  for (int64_t b = lo; b < hi; ++b) cnt += a.flag[b];
  int x = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[warp] = x;
  __syncthreads();
  int before = 0, total = 0;
#pragma unroll
  for (int w = 0; w < SCAN_THREADS / 32; ++w) {
    if (w < warp) before += wsum[w];
    total += wsum[w];
  }
  int e = before + x - cnt;                          // expanded blocks before lo
  int64_t dpos = total + (min(lo, a.nblk) - e);      // direct blocks before lo, after all expanded
  for (int64_t b = lo; b < hi; ++b) {
    if (a.flag[b]) a.order[e++] = (int)b;
    else a.order[dpos++] = (int)b;
  }
  if (tid == 0) {
    *a.n_exp = total;
    if (a.host_n) {
      *(volatile int*)a.host_n = total;
      __threadfence_system();
    }
  }
}

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

template <int ITEMS>
cudaError_t cluster_sort_items(const uint32_t* keys, int N, int key_bits, int* perm, cudaStream_t st) {
  static bool done[128] = {};
  constexpr size_t smem = cluster_sort_smem<ITEMS>();
  int dev = 0;
  cudaGetDevice(&dev);
  cudaError_t e;
  if (dev >= 128 || !done[dev]) {
    if ((e = cudaFuncSetAttribute(cluster_sort_kernel<ITEMS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)))
      return e;
    if (dev < 128) done[dev] = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(CL_SIZE);
  cfg.blockDim = dim3(CL_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CL_SIZE;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, cluster_sort_kernel<ITEMS>, keys, N, key_bits, perm);
  count_launch();
  return e;
}

// Fewest items per thread that hold N elements (whole powers of two keep the
// register arrays short for small N).
cudaError_t cluster_sort(const uint32_t* keys, int N, int key_bits, int* perm, cudaStream_t st) {
  const int64_t per = CL_SIZE * CL_THREADS;
  if (N <= per) return cluster_sort_items<1>(keys, N, key_bits, perm, st);
  if (N <= 2 * per) return cluster_sort_items<2>(keys, N, key_bits, perm, st);
  if (N <= 4 * per) return cluster_sort_items<4>(keys, N, key_bits, perm, st);
  if (N <= 8 * per) return cluster_sort_items<8>(keys, N, key_bits, perm, st);
  return cluster_sort_items<CL_MAX_ITEMS>(keys, N, key_bits, perm, st);
}

}  // namespace

cudaError_t gather_sorted(const float* in, int64_t N, int m, const int* perm, int64_t Npad,
                          float* out, cudaStream_t st, int* qbad) {
  if (Npad == 0) return cudaSuccess;
  gather_kernel<<<blocks_for(Npad, TS), TS, 0, st>>>(in, N, m, perm, Npad, out, qbad); count_launch();
  return cudaGetLastError();
}

cudaError_t unpack_points(const PointsDev& P, float* X, cudaStream_t st) {
  if (P.N == 0) return cudaSuccess;
  unpack_kernel<<<blocks_for(P.N, 256), 256, 0, st>>>(P.xs, P.N, P.d_in, P.d, P.perm, X); count_launch();
  return cudaGetLastError();
}

cudaError_t scatter_orig(const float* in, int64_t Npad, int64_t N, int m, const int* perm,
                         float* out, cudaStream_t st) {
  if (N == 0) return cudaSuccess;
  scatter_kernel<<<blocks_for(N, 256), 256, 0, st>>>(in, Npad, N, m, perm, out); count_launch();
  return cudaGetLastError();
}

cudaError_t prepare_points(Ctx& c, const float* X, int64_t N, int d, float sigma,
                           const char* tag, PointsDev& P, cudaStream_t st, bool read_counts) {
  const std::string t(tag);
  const int d_in = d;
  d = padded_dim(d_in);
  P.N = N;
  P.d = d;
  P.d_in = d_in;
  P.Npad = round_up(std::max<int64_t>(N, 1), PAD);
  P.kfam = c.kernel_family;
  if (P.kfam == KRR_KERNEL_MATERN32)
    P.s2 = 3.0 / ((double)sigma * (double)sigma);  // (sqrt(3) / h)^2
  else
    P.s2 = 1.0 / (std::log(2.0) * 2.0 * (double)sigma * (double)sigma);  // log2(e) / (2 sigma^2)
  P.scale = (float)std::sqrt(P.s2);
  cudaError_t e;
  void *xs, *perm, *ka, *bbp;
  // a block's thread count is a multiple of d_in; d_in <= 64 leaves at least 192
  const int bbt = BBOX_THREADS / d_in * d_in;
  const int nbb = (int)std::min<int64_t>((N * d_in + 4LL * bbt - 1) / (4LL * bbt), BBOX_BLOCKS);
  // the expanded form factors the Gaussian; other kernels take the direct
  // form.  Warp blocks (the packed CUDA-core kernel, d <= 8) and super-blocks
  // (the tensor-core kernels, d <= 64) are classified separately.
  const bool gauss = P.kfam == KRR_KERNEL_GAUSSIAN;
  const int allow_expanded = (d <= 8 && gauss) ? 1 : 0;
  const int allow_expanded_sb = gauss ? 1 : 0;
  if ((e = c.ws.get(t + ".xs", sizeof(float) * P.Npad * d, &xs))) return e;
  if ((e = c.ws.get(t + ".perm", sizeof(int) * P.Npad, &perm))) return e;
  if ((e = c.ws.get("sort.ka", sizeof(uint32_t) * N, &ka))) return e;
  if ((e = c.ws.get("sort.bbp", sizeof(float) * 2 * d_in * (size_t)nbb, &bbp))) return e;
  P.xs = (float*)xs;
  P.perm = (int*)perm;

  bbox_kernel<<<nbb, bbt, 0, st>>>(X, N * d_in, d_in, (float*)bbp, c.d_err); count_launch();
  const int dk = std::min(d_in, 30);
  const int bits = std::max(1, std::min(16, 30 / dk));
  const int key_bits = bits * dk;
  // One cluster sorts up to CL_MAX_N = 131072 points in one launch; above, the
  // exchange outgrows the cluster's shared memory and the passes fill the
  // chip.
  const bool in_cluster = N <= CL_MAX_N;
  void* va = nullptr;
  if (!in_cluster && (e = c.ws.get("sort.va", sizeof(int) * N, &va))) return e;
  const unsigned kblocks = blocks_for(N, 256);
  switch (dk) {
#define KRR_KEY(DK, CASE) \
  CASE: key_kernel<DK><<<kblocks, 256, 0, st>>>(X, N, d_in, dk, bits, !c.morton, (const float*)bbp, nbb, (uint32_t*)ka, (int*)va); break;
    KRR_KEY(1, case 1) KRR_KEY(2, case 2) KRR_KEY(3, case 3) KRR_KEY(4, case 4)
    KRR_KEY(5, case 5) KRR_KEY(6, case 6) KRR_KEY(7, case 7) KRR_KEY(8, case 8)
    KRR_KEY(0, default)
#undef KRR_KEY
  }
  count_launch();
  if (in_cluster) {
    if ((e = cluster_sort((const uint32_t*)ka, (int)N, key_bits, P.perm, st))) return e;
  } else {
    void *kb, *vb, *hist;
    const int nchunks = (int)blocks_for(N, SORT_CHUNK);
    if ((e = c.ws.get("sort.kb", sizeof(uint32_t) * N, &kb))) return e;
    if ((e = c.ws.get("sort.vb", sizeof(int) * N, &vb))) return e;
    if ((e = c.ws.get("sort.hist", sizeof(uint32_t) * 256 * ((size_t)nchunks + 1), &hist))) return e;
    uint32_t* tot = (uint32_t*)hist + 256 * (size_t)nchunks;
    uint32_t *kin = (uint32_t*)ka, *kout = (uint32_t*)kb;
    int *vin = (int*)va, *vout = (int*)vb;
    for (int shift = 0; shift < key_bits; shift += 8) {
      if (shift + 8 >= key_bits) vout = P.perm;
      radix_hist_kernel<<<nchunks, SORT_THREADS, 0, st>>>(kin, N, shift, (uint32_t*)hist, nchunks); count_launch();
      radix_scan_kernel<<<256, 256, 0, st>>>((uint32_t*)hist, nchunks, tot); count_launch();
      radix_scatter_kernel<<<nchunks, SORT_THREADS, 0, st>>>(kin, vin, N, shift, (const uint32_t*)hist, nchunks, tot,
                                                             kout, vout); count_launch();
      std::swap(kin, kout);
      std::swap(vin, vout);
    }
  }

  P.T = mvp_targets_per_thread(d, N);
  P.nblk = (N + 32 * P.T - 1) / (32 * P.T);
  P.nsb = (N + SB - 1) / SB;
  const int64_t ntiles = P.Npad / TS;
  void *ctr, *flag, *order, *nexp, *tbox;
  if ((e = c.ws.get(t + ".ctr", sizeof(float) * P.nblk * d, &ctr))) return e;
  if ((e = c.ws.get(t + ".order", sizeof(int) * P.nblk, &order))) return e;
  if ((e = c.ws.get(t + ".nexp", sizeof(int), &nexp))) return e;
  if ((e = c.ws.get("sort.flag", sizeof(int) * P.nblk, &flag))) return e;
  P.ctr = (float*)ctr;
  P.order = (int*)order;
  P.n_exp = (int*)nexp;
  void* sbflag;
  if ((e = c.ws.get(t + ".sbctr", sizeof(float) * P.nsb * d, &ctr))) return e;
  if ((e = c.ws.get(t + ".sborder", sizeof(int) * P.nsb, &order))) return e;
  if ((e = c.ws.get(t + ".sbnexp", sizeof(int), &nexp))) return e;
  if ((e = c.ws.get(t + ".sbflag", sizeof(int) * P.nsb, &sbflag))) return e;
  if ((e = c.ws.get(t + ".tbox", sizeof(float) * 2 * d * ntiles, &tbox))) return e;
  P.sb_ctr = (float*)ctr;
  P.sb_order = (int*)order;
  P.sb_nexp = (int*)nexp;
  P.sb_flag = (int*)sbflag;
  P.tbox = (float*)tbox;
  const PackOut po{P.xs, P.tbox, P.ctr, P.sb_ctr, (int*)flag, P.sb_flag};
  pack_kernel<<<(unsigned)ntiles, TS, 0, st>>>(X, N, d_in, d, P.perm, P.T, P.nblk, P.nsb, P.scale, allow_expanded,
                                               allow_expanded_sb, po); count_launch();
  // the block counts size the product grids: the host reads them once (a short
  // wait for the preparation; never inside a graph capture), from pinned words
  // that the kernel writes, or by copies where the context has none.  Without
  // the wait the words are left alone: the kernel may run while another
  // preparation on the handle waits for its own counts.
  int counts[2] = {0, 0};
  int* hc = read_counts ? c.h_counts : nullptr;
  order_kernel<<<2, SCAN_THREADS, 0, st>>>(OrderArgs{(const int*)flag, P.nblk, P.order, P.n_exp, hc},
                                           OrderArgs{P.sb_flag, P.nsb, P.sb_order, P.sb_nexp, hc ? hc + 1 : nullptr});
  count_launch();
  if ((e = cudaGetLastError())) return e;
  P.counts_read = read_counts;
  if (!read_counts) return cudaSuccess;
  if (!hc) {
    if ((e = cudaMemcpyAsync(&counts[0], P.n_exp, sizeof(int), cudaMemcpyDeviceToHost, st))) return e;
    if ((e = cudaMemcpyAsync(&counts[1], P.sb_nexp, sizeof(int), cudaMemcpyDeviceToHost, st))) return e;
  }
  if ((e = cudaStreamSynchronize(st))) return e;
  if (hc) {
    counts[0] = ((volatile int*)hc)[0];
    counts[1] = ((volatile int*)hc)[1];
  }
  P.h_nexp = counts[0];
  P.h_sb_nexp = counts[1];
  return cudaSuccess;
}

}  // namespace krr
