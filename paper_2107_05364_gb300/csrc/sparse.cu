// Thresholded (sparse) tensor, Sec. 4.3.1 of the paper: the smallest
// fraction f of the nonzero tensor elements (by absolute value) is set to
// zero and the rest is stored as a sparse matrix, so the product reads only
// what is kept.
//
// Reading of the rule (drop the smallest fraction f of the nonzero elements): the elements
// are those of the full 3n x 3n matrix (an off-diagonal entry of a symmetric
// 3x3 block stands for two), ranked by magnitude of the stored FP32 value,
// ties in (row tile i, column tile j, entry) order with an off-diagonal
// entry's two copies adjacent; the first k = floor(f * nonzeros) are dropped,
// except that an entry whose two copies the cut splits stays (blocks stay
// symmetric).  The magnitude t of the element of rank k is found exactly by
// a three-pass radix select on the FP32 bit patterns (non-negative floats order
// like their bits); every element below t goes, and of the elements equal
// to t the first r = k - #(below t) in that order.
//
// Storage: block-sparse rows of tiles; a 3x3 block is kept if any of its
// entries survives, with its 6 unique entries (dropped ones zero), in
// increasing column order.  The threshold drops the blocks of distant tiles,
// so the kept columns of a row form long runs of consecutive tiles (about
// one per line of tiles): columns are stored as runs, not one index per
// block.  A run starts at a kept column; later kept columns join it while
// they are at most 4 columns past the last one (the gap is stored as zero
// blocks); each run is padded with zero blocks to a multiple of 4.  Row i
// holds K4 = ptr[i+1] - ptr[i] blocks as np planes of K4 floats,
// val[np ptr[i] + e K4 + a] (np = 6, or 4 when the source is a single-layer
// tensor without the xz and yz planes), and its runs rptr[i] .. rptr[i+1]-1
// as pairs (first block a0 within the row, first column c0): block a of the
// run has column c0 + (a - a0).  Every row and run starts on a 16-byte
// boundary, so a lane reads 4 blocks with np vector loads and their 4
// operands as one contiguous 64-byte stretch.
//
// Product: one warp per (tile row, simulation); the operand is a float4
// (Ms m, 0) per tile (n + 4 per simulation, the last 4 zero for padding that
// runs past the last tile), read from L2 in whole runs.  Partial sums are
// compensated (each addition's rounding error is kept by an error-free
// two-sum and added back at the end, Ogita, Rump and Oishi's Sum2), so the
// result does not depend on the long per-lane summation order to more than
// the FP32 storage error.
#include <algorithm>
#include <cstring>
#include <utility>
#include <vector>

#include "mt_internal.cuh"

namespace {

__device__ __forceinline__ uint32_t abs_bits(float v) { return __float_as_uint(v) & 0x7fffffffu; }
__device__ __forceinline__ float f4_at(const float4 &v, int q) { return q == 0 ? v.x : q == 1 ? v.y : q == 2 ? v.z : v.w; }

// Multiplicity of a stored plane's entry in the full matrix: an off-diagonal
// entry of a symmetric block stands for two elements (planes xx xy xz yy yz
// zz, or xx xy yy zz of a single-layer tensor).
template <int NP>
__device__ __forceinline__ constexpr int plane_mult(int pl) {
  return NP == 6 ? ((pl == 0 || pl == 3 || pl == 5) ? 1 : 2) : (pl == 1 ? 2 : 1);
}

// Radix select of the element of rank k, on the device: three passes over the
// 31 magnitude bits (11, 10, 10), each a histogram of the elements whose
// higher bits match the selection so far, then one block that finds the bin.
struct Select {
  unsigned long long nz;    // nonzero elements of the full matrix
  unsigned long long rest;  // rank within the selected prefix; at the end the copies of t to drop
  unsigned int prefix;      // selected high bits; at the end the bits of t
  int active;               // 0: nothing to drop (t = 0)
  unsigned long long kept;  // nonzero elements kept (k_rows)
};
__host__ __device__ constexpr int sel_shift(int pass) { return 20 - 10 * pass; }
__host__ __device__ constexpr int sel_bins(int pass) { return pass == 0 ? 2048 : 1024; }
constexpr int kHistCopies = 8, kHistThreads = 1024;
constexpr size_t kHistSmem = (size_t)kHistCopies * 2 * 2048 * sizeof(unsigned int);

// Adjacent tiles' entries have adjacent magnitudes, so a warp's atomics
// collide: they go to shared memory, a copy of the histogram per 4 warps, as
// plain increments (colliding lanes of an increment are counted together in
// hardware), off-diagonal entries to a second histogram that counts double at
// the end.  Global 64-bit atomics on 65,536 bins took 6.5 ms at n = 6,400
// (single layer), a pass of this 0.14-0.16 (0.097: its 655 MB at copy rate).
template <int NP>
__global__ void __launch_bounds__(kHistThreads) k_hist(const float *D, int64_t n, int TR, int TC, int64_t Q,
                                                       int64_t P, int pass, const Select *sel,
                                                       unsigned long long *hist) {
  extern __shared__ unsigned int sh[];  // [copy][2][bins]
  if (pass > 0 && !sel->active) return;
  const int bins = sel_bins(pass), shift = sel_shift(pass);
  const uint32_t prefix = pass > 0 ? sel->prefix : 0;
  for (int q = threadIdx.x; q < kHistCopies * 2 * bins; q += kHistThreads) sh[q] = 0;
  __syncthreads();
  unsigned int *mine = sh + (threadIdx.x >> 5) % kHistCopies * 2 * bins;
  // positions: 4 adjacent columns of one row of one chunk
  const int64_t c4 = TC / 4, per = TR * c4, plane = (int64_t)TR * TC, tot = P * Q * per;
  for (int64_t t = blockIdx.x * (int64_t)kHistThreads + threadIdx.x; t < tot; t += (int64_t)gridDim.x * kHistThreads) {
    const int64_t chunk = t / per, rc = t - chunk * per;
    const int64_t p = chunk / Q, q = chunk - p * Q;
    const int r = (int)(rc / c4), c = 4 * (int)(rc - (int64_t)r * c4);
    if (p * TR + r >= n) continue;
    const int64_t j = q * TC + c;
    const float *base = D + chunk * NP * plane + (int64_t)r * TC + c;
    float4 v[NP];
#pragma unroll
    for (int pl = 0; pl < NP; ++pl) v[pl] = __ldcs(reinterpret_cast<const float4 *>(base + pl * plane));
#pragma unroll
    for (int pl = 0; pl < NP; ++pl)
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t bits = abs_bits(f4_at(v[pl], u));
        if (bits == 0 || j + u >= n) continue;
        if (pass > 0 && (bits >> (shift + 10)) != prefix) continue;
        atomicAdd(&mine[(plane_mult<NP>(pl) - 1) * bins + ((bits >> shift) & (bins - 1))], 1u);
      }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < bins; q += kHistThreads) {
    unsigned long long h = 0;
    for (int k = 0; k < kHistCopies; ++k)
      h += (unsigned long long)sh[k * 2 * bins + q] + 2ull * sh[(k * 2 + 1) * bins + q];
    if (h) atomicAdd(&hist[q], h);
  }
}

// inclusive sum over the block of 1,024 threads
__device__ __forceinline__ unsigned long long block_scan(unsigned long long v, unsigned long long *sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  if (lane == 31) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    unsigned long long x = sh[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    sh[lane] = x;
  }
  __syncthreads();
  if (w > 0) v += sh[w - 1];
  __syncthreads();
  return v;
}

// one block: the bin holding rank `rest` (pass 0: the number of elements and
// the rank k = floor(fraction nz) first); clears the histogram for the next
// pass
__global__ void __launch_bounds__(1024) k_select(int pass, double fraction, unsigned long long *hist, Select *sel) {
  __shared__ unsigned long long sh[32], s_rest;
  __shared__ int s_active;
  const int t = threadIdx.x;
  // two adjacent bins per thread
  const unsigned long long h0 = hist[2 * t], h1 = hist[2 * t + 1];
  hist[2 * t] = hist[2 * t + 1] = 0;
  const unsigned long long incl = block_scan(h0 + h1, sh);
  if (pass == 0) {
    if (t == 1023) {
      sel->nz = incl;
      s_rest = (unsigned long long)(fraction * (double)incl);
      s_active = incl > 0 && s_rest > 0;
      sel->active = s_active;
      if (!s_active) {
        sel->prefix = 0;
        sel->rest = 0;
      }
    }
  } else if (t == 0) {
    s_rest = sel->rest;
    s_active = sel->active;
  }
  __syncthreads();
  if (!s_active) return;
  const unsigned long long k = s_rest, ex = incl - (h0 + h1);
  if (ex <= k && k < incl) {  // exactly one thread
    const int second = ex + h0 <= k ? 1 : 0;
    const unsigned int bin = 2 * t + second;
    sel->rest = k - ex - (second ? h0 : 0);
    sel->prefix = pass == 0 ? bin : (sel->prefix << 10) | bin;
  }
}

// copies of the cut value t in row tile i (counted for the tie order; not
// needed when none of them is dropped)
template <int NP>
__global__ void k_row_ties(const float *D, int64_t n, int TR, int TC, int64_t Q, const Select *sel,
                           unsigned long long *ties) {
  const int64_t i = blockIdx.x;
  const uint32_t tbits = sel->prefix;
  unsigned int local = 0;
  if (sel->rest > 0) {
    const int64_t p = i / TR, plane = (int64_t)TR * TC;
    const int r = (int)(i - p * TR);
    for (int64_t j = 4 * (int64_t)threadIdx.x; j < n; j += 4 * blockDim.x) {
      const int64_t q = j / TC;
      const float *base = D + (p * Q + q) * NP * plane + (int64_t)r * TC + (j - q * TC);
#pragma unroll
      for (int pl = 0; pl < NP; ++pl) {
        const float4 v = __ldcs(reinterpret_cast<const float4 *>(base + pl * plane));
#pragma unroll
        for (int u = 0; u < 4; ++u)  // the padding past column n is zero, t is not
          local += abs_bits(f4_at(v, u)) == tbits ? plane_mult<NP>(pl) : 0;
      }
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) local += __shfl_xor_sync(0xffffffffu, local, off);
  __shared__ unsigned int sh[32];
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = local;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long s = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += sh[w];
    ties[i] = s;
  }
}

// one block: out[i] = sum of in[0 .. i - 1], i = 0 .. n (in place allowed for
// 64-bit counts)
template <typename In, typename Out>
__global__ void __launch_bounds__(1024) k_scan(const In *in, int64_t n, Out *out) {
  __shared__ unsigned long long sh[32];
  unsigned long long carry = 0;
  for (int64_t i0 = 0; i0 < n; i0 += 1024) {
    const int64_t i = i0 + threadIdx.x;
    const unsigned long long v = i < n ? (unsigned long long)in[i] : 0;
    const unsigned long long incl = block_scan(v, sh);
    if (i < n) out[i] = (Out)(carry + incl - v);
    __shared__ unsigned long long s_tot;
    if (threadIdx.x == 1023) s_tot = incl;
    __syncthreads();
    carry += s_tot;
    __syncthreads();
  }
  if (threadIdx.x == 0) out[n] = (Out)carry;
}

// a later kept column joins the run when it lies at most this far past the
// run's last kept column (the columns between are stored as zero blocks)
constexpr int kRunJoin = 4;

// Row tile i in increasing column order, one warp per row, a chunk of 128
// columns per step as 4 words of 32 (lane = column), the next step's values
// loaded ahead.  An entry is kept if |v| > t, or if |v| == t and the copies
// of t up to and including it (counted from tie_start[i], in column and entry
// order) exceed r.  The kept columns are grouped into runs (see the storage
// note) from the word's ballot: the run state is the same in all lanes, and
// only the starts of new runs are walked one by one.  FILL = false: the row's
// stored blocks (runs padded to 4) into cnt[i], its runs into nrun[i], the
// kept elements of the full matrix added to sel->kept; FILL = true: each kept
// block at its slot and each run's (first block, first column) pair (the
// value planes were zeroed before).  With t = 0 every nonzero entry is kept.
// One 32-column word per step, walking every kept column, took 1.3 (count)
// and 1.5 ms (fill) at n = 6,400 (single layer, 40 % dropped); this 0.17 and
// 0.27 (0.10 and 0.16: the tensor read, the kept blocks written).
constexpr int kRowsPerCta = 4;
template <int NP, bool FILL>
__global__ void __launch_bounds__(32 * kRowsPerCta) k_rows(const float *D, int64_t n, int TR, int TC, int64_t Q,
                                                           const unsigned long long *tie_start, Select *sel, int *cnt,
                                                           int *nrun, const int64_t *ptr, const int64_t *rptr,
                                                           int32_t *run, float *val) {
  const int64_t i = blockIdx.x * (int64_t)kRowsPerCta + (threadIdx.x >> 5);
  if (i >= n) return;
  const int lane = threadIdx.x & 31;
  const int64_t p = i / TR, plane = (int64_t)TR * TC;
  const int rr = (int)(i - p * TR);
  const uint32_t tbits = sel->prefix;
  const unsigned long long r = sel->rest;
  const int64_t o = FILL ? ptr[i] : 0, K4 = FILL ? ptr[i + 1] - o : 0;
  float *rv = FILL ? val + NP * o : nullptr;  // NP value planes, as the source
  int32_t *rd = FILL ? run + 2 * rptr[i] : nullptr;
  unsigned long long carry = r > 0 ? tie_start[i] : 0;
  // run state: stored blocks before the open run, its first and last column
  int64_t ofs = 0, col0 = -1, last = -1;
  int64_t runs = 0;
  unsigned int kept = 0;
  const float *row = D + p * Q * NP * plane + (int64_t)rr * TC + lane;
  float nx[4][NP];
  auto load = [&](int64_t q) {
    const float *base = row + q * NP * plane;
#pragma unroll
    for (int w = 0; w < 4; ++w)
#pragma unroll
      for (int e = 0; e < NP; ++e) nx[w][e] = q * 128 + 32 * w + lane < n ? __ldcs(base + e * plane + 32 * w) : 0.0f;
  };
  load(0);
  for (int64_t q = 0; q < Q; ++q) {
    float v[4][NP];
#pragma unroll
    for (int w = 0; w < 4; ++w)
#pragma unroll
      for (int e = 0; e < NP; ++e) v[w][e] = nx[w][e];
    if (q + 1 < Q) load(q + 1);
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const int64_t j0 = q * 128 + 32 * w;
      unsigned tm = 0;  // copies of t in this lane's block
#pragma unroll
      for (int e = 0; e < NP; ++e) {
        const uint32_t bits = abs_bits(v[w][e]);
        tm += (bits != 0 && bits == tbits) ? plane_mult<NP>(e) : 0;
      }
      unsigned long long cum = carry;
      if (__any_sync(0xffffffffu, tm != 0)) {
        // inclusive scan of tm over the lanes (columns in order)
        unsigned incl = tm;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const unsigned y = __shfl_up_sync(0xffffffffu, incl, off);
          if (lane >= off) incl += y;
        }
        cum += incl - tm;
        carry += __shfl_sync(0xffffffffu, incl, 31);
      }
      bool keep = false;
#pragma unroll
      for (int e = 0; e < NP; ++e) {
        const uint32_t bits = abs_bits(v[w][e]);
        bool k = bits != 0 && bits > tbits;
        if (bits != 0 && bits == tbits) {
          cum += plane_mult<NP>(e);
          k = cum > r;
        }
        if (!k) v[w][e] = 0.0f;
        keep = keep || k;
        if (!FILL) kept += k ? plane_mult<NP>(e) : 0;
      }
      const unsigned mk = __ballot_sync(0xffffffffu, keep);
      if (mk == 0) continue;
      // a kept column starts a run when none of the kRunJoin columns before
      // it is kept (in this word, or in earlier ones through `last`)
      unsigned starts = mk & ~(mk << 1) & ~(mk << 2) & ~(mk << 3) & ~(mk << 4);
      const int first = __ffs(mk) - 1;
      if (col0 >= 0 && j0 + first - last <= kRunJoin) starts &= ~(1u << first);
      int64_t shift = ofs - col0;  // slot of column j of the open run: shift + j
      while (starts) {
        const int sc = __ffs(starts) - 1;
        starts &= starts - 1;
        const unsigned below = mk & ((1u << sc) - 1u);
        if (below) last = j0 + 31 - __clz(below);
        if (col0 >= 0) ofs += (last - col0 + 4) & ~(int64_t)3;  // close the open run, padded to 4
        col0 = j0 + sc;
        if (FILL && lane == 0) {
          rd[2 * runs] = (int32_t)ofs;
          rd[2 * runs + 1] = (int32_t)col0;
        }
        ++runs;
        if (lane >= sc) shift = ofs - col0;
      }
      last = j0 + 31 - __clz(mk);
      if (FILL && keep) {
#pragma unroll
        for (int e = 0; e < NP; ++e) rv[e * K4 + shift + j0 + lane] = v[w][e];
      }
    }
  }
  if (col0 >= 0) ofs += (last - col0 + 4) & ~(int64_t)3;
  if (!FILL) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) kept += __shfl_xor_sync(0xffffffffu, kept, off);
    if (lane == 0) {
      cnt[i] = (int)ofs;
      nrun[i] = (int)runs;
      atomicAdd(&sel->kept, (unsigned long long)kept);
    }
  }
}

// s + t = u + err exactly (Knuth's two-sum); the error goes to c
__device__ __forceinline__ void sum2_add(float &s, float &c, float t) {
  const float u = s + t;
  const float bp = u - s;
  c += (s - (u - bp)) + (t - bp);
  s = u;
}

// the warp's (sum, error) pairs combined into lane 0's (s, c) (and every
// lane's: butterfly), errors carried
__device__ __forceinline__ void warp_sum2_pair(float &s, float &c) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float so = __shfl_xor_sync(0xffffffffu, s, off);
    const float co = __shfl_xor_sync(0xffffffffu, c, off);
    c += co;
    sum2_add(s, c, so);
  }
}


// A row's blocks are taken 128 at a time (a step: 4 consecutive blocks of one
// run per lane).  The product may give a row to S = 1, 2, 4 or 8 warps, warp
// k taking steps floor(k st / S) .. floor((k + 1) st / S) - 1 of the row's
// st steps; seg[8 i + k'] holds the run (from the row's first) that contains
// the first block of eighth k', so a warp starts its cursor there.
constexpr int kSpSegMax = 8;

__global__ void k_seg_runs(int64_t n, const int64_t *__restrict__ ptr, const int64_t *__restrict__ rptr,
                           const int2 *__restrict__ run, int32_t *seg) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n * kSpSegMax) return;
  const int64_t i = t / kSpSegMax;
  const int k = (int)(t - i * kSpSegMax);
  const int64_t st = (ptr[i + 1] - ptr[i] + 127) / 128;
  const int64_t a = 128 * ((k * st) / kSpSegMax);
  int64_t lo = rptr[i], hi = rptr[i + 1] - 1;  // the last run starting at or before block a
  if (hi < lo) {
    seg[t] = 0;
    return;
  }
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) >> 1;
    if (run[mid].x <= a) lo = mid;
    else hi = mid - 1;
  }
  seg[t] = (int32_t)(lo - rptr[i]);
}

// H_i = -sum_kept N_ij Ms_j m_j, rows of one simulation consecutive; xs =
// float4 (Ms m, 0) per tile, n + 4 per simulation.  S = 1: one warp per
// (row, simulation), two per CTA.  S > 1: one CTA per (row, simulation), its
// S warps on consecutive step ranges, their compensated sums added in warp
// order in shared memory.  Each lane takes 4 consecutive blocks of one run
// per step (NP vector loads of the values and 4 contiguous operands) and
// follows the row's runs with a cursor of its own.  (Lanes on interleaved
// blocks, for wider contiguous loads, needed a cursor walk per block and
// measured 2.4x slower.)
template <int NP, int S>
__global__ void __launch_bounds__(S == 1 ? 64 : 32 * S) k_spmv(int64_t n, int B, const int64_t *__restrict__ ptr,
                                                               const int64_t *__restrict__ rptr,
                                                               const int2 *__restrict__ run,
                                                               const int32_t *__restrict__ seg,
                                                               const float *__restrict__ val,
                                                               const float4 *__restrict__ xs, float *H,
                                                               const int *active) {
  mtd::pdl_enter();
  const int lane = threadIdx.x & 31;
  int64_t rid;  // b n + i
  int k;        // this warp's part of the row
  if constexpr (S == 1) {
    rid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    k = 0;
    if (rid >= n * B) return;
  } else {
    rid = blockIdx.x;
    k = threadIdx.x >> 5;
  }
  const int64_t i = rid % n;
  const int b = (int)(rid / n);
  if (active && !active[b]) return;  // the whole CTA when S > 1
  const float4 *xb = xs + (size_t)b * sparse_x_stride(n);
  const int64_t o = ptr[i], K4 = ptr[i + 1] - o;
  const int64_t st = (K4 + 127) / 128;
  const int64_t a_lo = 128 * ((k * st) / S);
  const int64_t a_e = 128 * (((k + 1) * st) / S), a_hi = a_e < K4 ? a_e : K4;
  const float *rv = val + NP * o;
  const int64_t r1 = rptr[i + 1];
  int64_t rc = rptr[i] + (S == 1 ? 0 : seg[i * kSpSegMax + k * (kSpSegMax / S)]);  // this lane's run
  int2 cur = rc < r1 ? run[rc] : make_int2(0, 0);
  int64_t next = rc + 1 < r1 ? run[rc + 1].x : INT64_MAX;  // first block of the following run
  float sx = 0, cx = 0, sy = 0, cy = 0, sz = 0, cz = 0;
  for (int64_t a = a_lo + 4 * (int64_t)lane; a < a_hi; a += 128) {
    // the values stream past (read once: no L1 allocation); the operands,
    // read by every row, stay cached
    float4 v[NP];
#pragma unroll
    for (int e = 0; e < NP; ++e) v[e] = __ldcs(reinterpret_cast<const float4 *>(rv + e * K4 + a));
    while (a >= next) {
      ++rc;
      cur = run[rc];
      next = rc + 1 < r1 ? run[rc + 1].x : INT64_MAX;
    }
    const int64_t c = cur.y + (a - cur.x);  // column of block a
    float4 x[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) x[q] = xb[c + q];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if constexpr (NP == 6) {
        // per block: (v0 v1 v2; v1 v3 v4; v2 v4 v5) (x, y, z)
        const float n0 = f4_at(v[0], q), n1 = f4_at(v[1], q), n2 = f4_at(v[2], q);
        const float n3 = f4_at(v[3], q), n4 = f4_at(v[4], q), n5 = f4_at(v[5], q);
        sum2_add(sx, cx, fmaf(n0, x[q].x, fmaf(n1, x[q].y, n2 * x[q].z)));
        sum2_add(sy, cy, fmaf(n1, x[q].x, fmaf(n3, x[q].y, n4 * x[q].z)));
        sum2_add(sz, cz, fmaf(n2, x[q].x, fmaf(n4, x[q].y, n5 * x[q].z)));
      } else {
        // single-layer tensor: (v0 v1 0; v1 v2 0; 0 0 v3) (x, y, z)
        const float n0 = f4_at(v[0], q), n1 = f4_at(v[1], q);
        const float n3 = f4_at(v[2], q), n5 = f4_at(v[3], q);
        sum2_add(sx, cx, fmaf(n0, x[q].x, n1 * x[q].y));
        sum2_add(sy, cy, fmaf(n1, x[q].x, n3 * x[q].y));
        sum2_add(sz, cz, __fmul_rn(n5, x[q].z));  // a rounded product, as in the 6-plane form
      }
    }
  }
  warp_sum2_pair(sx, cx);
  warp_sum2_pair(sy, cy);
  warp_sum2_pair(sz, cz);
  float *Hb = H + (size_t)b * 3 * n + 3 * i;
  if constexpr (S == 1) {
    if (lane == 0) {
      Hb[0] = -(sx + cx);
      Hb[1] = -(sy + cy);
      Hb[2] = -(sz + cz);
    }
  } else {
    __shared__ float part[S][6];
    if (lane == 0) {
      part[k][0] = sx;
      part[k][1] = cx;
      part[k][2] = sy;
      part[k][3] = cy;
      part[k][4] = sz;
      part[k][5] = cz;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < S; ++w) {
        cx += part[w][1];
        sum2_add(sx, cx, part[w][0]);
        cy += part[w][3];
        sum2_add(sy, cy, part[w][2]);
        cz += part[w][5];
        sum2_add(sz, cz, part[w][4]);
      }
      Hb[0] = -(sx + cx);
      Hb[1] = -(sy + cy);
      Hb[2] = -(sz + cz);
    }
  }
}

// xs[b][j] = (Ms_j m_j, 0) (the 4 padding entries per simulation stay zero)
__global__ void k_prep_sparse_x(const float *m, const float *Ms, int64_t n, int B, float4 *xs) {
  mtd::pdl_enter();
  const int64_t tot = (int64_t)B * n;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = t / n, j = t - b * n;
    const float ms = Ms[j];
    const float *mj = m + 3 * t;
    xs[b * sparse_x_stride(n) + j] = make_float4(ms * mj[0], ms * mj[1], ms * mj[2], 0.0f);
  }
}

// Warps per row of the sparse product, a property of the tensor (so that a
// simulation's field does not depend on the batch it runs in): doubled while
// one simulation's rows give fewer than 4 waves of resident warps (32 per SM)
// and every warp keeps at least 6 steps of 128 blocks.  With one warp per row
// the last, partial wave runs a whole row's chain of dependent steps on
// mostly idle SMs.
int sparse_split(int64_t n, int64_t nnzb, int sms) {
  const double steps = n > 0 ? (double)nnzb / (double)n / 128.0 : 0.0;
  const int64_t resident = (int64_t)std::max(1, sms) * 32;
  int S = 1;
  while (S < kSpSegMax && n * S < 4 * resident && steps / (2 * S) >= 6.0) S *= 2;
  return S;
}

}  // namespace

namespace mt {

void launch_spmv(const mt_tensor *T, const float *xs, int B, float *H, const int *active, cudaStream_t s) {
  const int64_t rows = T->n * (int64_t)B;
  const int64_t *ptr = (const int64_t *)T->d_sp_ptr;
  const int64_t *rptr = (const int64_t *)T->d_sp_rptr;
  const int2 *run = reinterpret_cast<const int2 *>(T->d_sp_col);
  const int32_t *seg = T->d_sp_seg;
  const float *val = (const float *)T->d_sp_val;
  const float4 *x4 = reinterpret_cast<const float4 *>(xs);
  const int S = T->sp_split;
  const dim3 grid((unsigned)(S == 1 ? (rows + 1) / 2 : rows)), block(S == 1 ? 64 : 32 * S);
#define MT_SPMV(NP, SS) \
  mt::launch_pdl(k_spmv<NP, SS>, grid, block, 0, s, T->n, B, ptr, rptr, run, seg, val, x4, H, active)
  if (T->L.nplane == 4) {
    if (S == 8) MT_SPMV(4, 8);
    else if (S == 4) MT_SPMV(4, 4);
    else if (S == 2) MT_SPMV(4, 2);
    else MT_SPMV(4, 1);
  } else {
    if (S == 8) MT_SPMV(6, 8);
    else if (S == 4) MT_SPMV(6, 4);
    else if (S == 2) MT_SPMV(6, 2);
    else MT_SPMV(6, 1);
  }
#undef MT_SPMV
}

void launch_prep_sparse_x(const mt_tensor *T, const float *m, int B, float *xs, cudaStream_t s) {
  const int64_t tot = (int64_t)B * T->n;
  const int blocks = (int)std::min<int64_t>((tot + 255) / 256, 4096);
  mt::launch_pdl(k_prep_sparse_x, dim3(blocks), dim3(256), 0, s, m, (const float *)T->tiles->d_Ms, T->n, B,
                 reinterpret_cast<float4 *>(xs));
}

}  // namespace mt

extern "C" mt_status mt_tensor_threshold(mt_tensor *T, double fraction, mt_tensor **out, double *threshold,
                                         int64_t *kept_elements) {
  MT_CHECK(T && out, MT_EINVAL, "mt_tensor_threshold: NULL argument");
  MT_CHECK(T->prec == MT_F32 && T->layout == MT_LAYOUT_STREAM, MT_EINVAL,
           "mt_tensor_threshold: needs an FP32 tensor of the streaming layout");
  MT_CHECK(fraction >= 0.0 && fraction < 1.0, MT_EINVAL, "mt_tensor_threshold: fraction in [0, 1)");
  MT_CHECK(!T->L.half, MT_EINVAL,
           "mt_tensor_threshold: needs every block stored; assemble with MT_LAYOUT_STREAM_FULL");
  MT_CUDA(cudaSetDevice(T->tiles->ctx->device));
  const int64_t n = T->n;
  const mt_layout &L = T->L;
  const float *D = reinterpret_cast<const float *>(T->d_data);
  const int np = L.nplane;  // value planes: those the source stores (6, or 4 for a single layer)
  MT_CHECK(L.TC == 128 && (np == 6 || np == 4), MT_EINVAL, "mt_tensor_threshold: unexpected storage");
  // everything up to the sizes of the new arrays is decided on the device
  DevTemp<Select> sel;
  DevTemp<unsigned long long> hist, tie_start;
  DevTemp<int> cnt_rows, run_rows;
  DevTemp<int64_t> row_ptr, row_rptr;
  MT_CUDA(sel.alloc(1));
  MT_CUDA(hist.alloc(sel_bins(0)));
  MT_CUDA(tie_start.alloc(n + 1));
  MT_CUDA(cnt_rows.alloc(n));
  MT_CUDA(run_rows.alloc(n));
  MT_CUDA(row_ptr.alloc(n + 1));
  MT_CUDA(row_rptr.alloc(n + 1));
  MT_CUDA(cudaMemset(sel.p, 0, sizeof(Select)));
  MT_CUDA(cudaMemset(hist.p, 0, sizeof(unsigned long long) * sel_bins(0)));
  const auto hist_k = np == 6 ? k_hist<6> : k_hist<4>;
  MT_CUDA(cudaFuncSetAttribute(hist_k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kHistSmem));
  const int sms = T->tiles->ctx->num_sms;
  for (int pass = 0; pass < 3; ++pass) {
    hist_k<<<sms, kHistThreads, kHistSmem>>>(D, n, L.TR, L.TC, L.Q, L.P, pass, sel.p, hist.p);
    k_select<<<1, 1024>>>(pass, fraction, hist.p, sel.p);
  }
  (np == 6 ? k_row_ties<6> : k_row_ties<4>)<<<(unsigned)n, 256>>>(D, n, L.TR, L.TC, L.Q, sel.p, tie_start.p);
  k_scan<<<1, 1024>>>(tie_start.p, n, tie_start.p);
  const unsigned row_grid = (unsigned)((n + kRowsPerCta - 1) / kRowsPerCta);
  (np == 6 ? k_rows<6, false> : k_rows<4, false>)<<<row_grid, 32 * kRowsPerCta>>>(
      D, n, L.TR, L.TC, L.Q, tie_start.p, sel.p, cnt_rows.p, run_rows.p, nullptr, nullptr, nullptr, nullptr);
  k_scan<<<1, 1024>>>(cnt_rows.p, n, row_ptr.p);  // runs are padded to 4 blocks already
  k_scan<<<1, 1024>>>(run_rows.p, n, row_rptr.p);
  MT_CUDA(cudaGetLastError());
  Select hs;
  int64_t nnzb = 0, nruns = 0;
  MT_CUDA(cudaMemcpy(&hs, sel.p, sizeof(Select), cudaMemcpyDeviceToHost));
  MT_CUDA(cudaMemcpy(&nnzb, row_ptr.p + n, sizeof(int64_t), cudaMemcpyDeviceToHost));
  MT_CUDA(cudaMemcpy(&nruns, row_rptr.p + n, sizeof(int64_t), cudaMemcpyDeviceToHost));
  mt_ctx *ctx = T->tiles->ctx;
  mt_tensor *S = new mt_tensor();
  S->tiles = T->tiles;
  T->tiles->refs++;
  S->prec = MT_F32;
  S->layout = MT_LAYOUT_SPARSE;
  S->n = n;
  S->L = T->L;
  S->sp_blocks = nnzb;
  S->sp_runs = nruns;
  S->sp_split = sparse_split(n, nnzb, ctx->num_sms);
  S->bytes = 2 * sizeof(int64_t) * (n + 1) + 2 * sizeof(int32_t) * (size_t)std::max<int64_t>(1, nruns) +
             np * sizeof(float) * (size_t)std::max<int64_t>(1, nnzb) + sizeof(int32_t) * kSpSegMax * (size_t)n;
  {
    std::lock_guard<std::mutex> lk(ctx->mu);
    if (ctx->in_use + S->bytes > ctx->budget) {
      const size_t need = S->bytes;
      delete S;
      mt::tiles_release(T->tiles);
      mt::set_error("mt_tensor_threshold: %zu bytes exceed the context budget", need);
      return MT_ENOMEM;
    }
    ctx->in_use += S->bytes;
  }
  std::swap(S->d_sp_ptr, row_ptr.p);
  std::swap(S->d_sp_rptr, row_rptr.p);
  cudaError_t e = cudaMalloc(&S->d_sp_col, 2 * sizeof(int32_t) * std::max<int64_t>(1, nruns));
  if (e == cudaSuccess) e = cudaMalloc(&S->d_sp_val, np * sizeof(float) * std::max<int64_t>(1, nnzb));
  if (e == cudaSuccess) e = cudaMalloc(&S->d_sp_seg, sizeof(int32_t) * kSpSegMax * (size_t)n);
  // gap and padding blocks are zero
  if (e == cudaSuccess) e = cudaMemset(S->d_sp_val, 0, np * sizeof(float) * std::max<int64_t>(1, nnzb));
  if (e != cudaSuccess) {
    mt::tensor_release(S);
    return mt::cuda_fail(e, "mt_tensor_threshold allocation", __FILE__, __LINE__);
  }
  (np == 6 ? k_rows<6, true> : k_rows<4, true>)<<<row_grid, 32 * kRowsPerCta>>>(
      D, n, L.TR, L.TC, L.Q, tie_start.p, sel.p, nullptr, nullptr, S->d_sp_ptr, S->d_sp_rptr, S->d_sp_col,
      S->d_sp_val);
  e = cudaGetLastError();
  if (e == cudaSuccess)
    k_seg_runs<<<(unsigned)((n * kSpSegMax + 255) / 256), 256>>>(
        n, S->d_sp_ptr, S->d_sp_rptr, reinterpret_cast<const int2 *>(S->d_sp_col), S->d_sp_seg);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    mt::tensor_release(S);
    return mt::cuda_fail(e, "mt_tensor_threshold fill", __FILE__, __LINE__);
  }
  if (threshold) {
    float tf;
    std::memcpy(&tf, &hs.prefix, sizeof(tf));
    *threshold = (double)tf;
  }
  if (kept_elements) *kept_elements = (int64_t)hs.kept;
  *out = S;
  return MT_OK;
}

namespace mt {

// rows [i0, i1) of a thresholded tensor as dense FP64 blocks
mt_status read_rows_sparse(const mt_tensor *T, int64_t i0, int64_t i1, double *out) {
  const int64_t n = T->n;
  std::vector<int64_t> ptr(i1 - i0 + 1), rptr(i1 - i0 + 1);
  MT_CUDA(cudaMemcpy(ptr.data(), T->d_sp_ptr + i0, sizeof(int64_t) * (i1 - i0 + 1), cudaMemcpyDeviceToHost));
  MT_CUDA(cudaMemcpy(rptr.data(), T->d_sp_rptr + i0, sizeof(int64_t) * (i1 - i0 + 1), cudaMemcpyDeviceToHost));
  const int64_t a0 = ptr[0], a1 = ptr[i1 - i0], q0 = rptr[0], q1 = rptr[i1 - i0];
  std::vector<int32_t> run(2 * std::max<int64_t>(1, q1 - q0));
  const int np = T->L.nplane;
  std::vector<float> val(np * std::max<int64_t>(1, a1 - a0));
  if (a1 > a0) {
    MT_CUDA(cudaMemcpy(run.data(), T->d_sp_col + 2 * q0, 2 * sizeof(int32_t) * (q1 - q0), cudaMemcpyDeviceToHost));
    MT_CUDA(cudaMemcpy(val.data(), T->d_sp_val + np * a0, np * sizeof(float) * (a1 - a0), cudaMemcpyDeviceToHost));
  }
  std::memset(out, 0, sizeof(double) * 6 * (size_t)(i1 - i0) * n);
  for (int64_t i = i0; i < i1; ++i) {
    const int64_t o = ptr[i - i0], K4 = ptr[i - i0 + 1] - o;
    const float *rv = val.data() + np * (o - a0);
    const int64_t rb = rptr[i - i0] - q0, re = rptr[i - i0 + 1] - q0;
    for (int64_t q = rb; q < re; ++q) {
      const int64_t b0 = run[2 * q], c0 = run[2 * q + 1];
      const int64_t b1 = q + 1 < re ? run[2 * (q + 1)] : K4;
      for (int64_t a = b0; a < b1; ++a) {
        const int64_t j = c0 + (a - b0);
        if (j >= n) break;  // padding past the last tile (zero)
        for (int e = 0; e < 6; ++e) {
          const int pl = stream_plane(e, np);
          if (pl >= 0) out[((i - i0) * n + j) * 6 + e] += rv[pl * K4 + a];
        }
      }
    }
  }
  return MT_OK;
}

}  // namespace mt
