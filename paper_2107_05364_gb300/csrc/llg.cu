// Effective field, Landau-Lifshitz right-hand side and the Runge-Kutta (4,5)
// integrator (Sec. 2, Sec. 3.1 of the paper).
//
// One Dormand-Prince step of B simulations is a fixed sequence of kernels,
// captured once in a CUDA graph:
//   begin      commit the previous step if it was accepted (m <- |m_new|^-1
//              m_new, k1 <- k7), form the stage-2 input;
//   6 x [ streaming demag product ; stage kernel ]
//              a stage kernel adds exchange (Eq. 12), anisotropy (Eq. 16)
//              and applied field (Eq. 7) to H_d, evaluates Eq. 1 and forms
//              the next stage's input; the last one also reduces the
//              embedded error, the torque and the mean magnetisation, and its
//              last block decides accept/reject and the next step size on
//              the device.
// The host only replays the graph and polls a counter of unfinished
// simulations every few steps.
#include <algorithm>
#include <limits>
#include <cmath>
#include <cstring>
#include <vector>

#include "mt_internal.cuh"

namespace {

// Dormand & Prince (1980) RK5(4)7M: stage couplings, 5th-order weights
// (= last coupling row, first same as last) and the difference between the
// 5th- and the embedded 4th-order weights, which estimates the local error.
__constant__ double c_dp_a[7][7] = {
    {0, 0, 0, 0, 0, 0, 0},
    {1.0 / 5, 0, 0, 0, 0, 0, 0},
    {3.0 / 40, 9.0 / 40, 0, 0, 0, 0, 0},
    {44.0 / 45, -56.0 / 15, 32.0 / 9, 0, 0, 0, 0},
    {19372.0 / 6561, -25360.0 / 2187, 64448.0 / 6561, -212.0 / 729, 0, 0, 0},
    {9017.0 / 3168, -355.0 / 33, 46732.0 / 5247, 49.0 / 176, -5103.0 / 18656, 0, 0},
    {35.0 / 384, 0, 500.0 / 1113, 125.0 / 192, -2187.0 / 6784, 11.0 / 84, 0}};
__constant__ double c_dp_err[7] = {35.0 / 384 - 5179.0 / 57600,
                                   0.0,
                                   500.0 / 1113 - 7571.0 / 16695,
                                   125.0 / 192 - 393.0 / 640,
                                   -2187.0 / 6784 + 92097.0 / 339200,
                                   11.0 / 84 - 187.0 / 2100,
                                   -1.0 / 40};

// ---------------------------------------------------------------------------
// per-simulation control block (device memory)
// ---------------------------------------------------------------------------
struct SimCtl {
  double t, h, hs, t_next, t_out0, dt_out, t1, tol;
  double tau, err;
  double m_last[3];  // volume-averaged m of the last accepted (or starting) state
  int64_t iout, n_out;
  int64_t n_accept, n_reject, n_rhs, n_attempt, attempt_cap;
  int mode;      // 0 = fixed number of steps, 1 = integrate to t1, 2 = relax
  int accepted;  // last attempt accepted: begin/commit must adopt it
  int clipped;   // the current attempt ends exactly on t_next
  int status;
  int done;
  int fresh;  // admitted since the last k1 evaluation (serving slots)
};

enum { MODE_STEPS = 0, MODE_RUN = 1, MODE_RELAX = 2 };

struct StageArgs {
  int64_t n;
  int B;
  // geometry / material
  const int32_t *nbr;
  const float *wex, *kan, *axis, *Ms;
  const double *wvol;
  bool exch;
  // per-simulation equation parameters
  const float *g1, *g2, *Ha;
  const float *xsc;  // [B] factor on the exchange stiffness (nullptr: 1)
  // state
  float *y, *ys0, *ys1, *Hd, *xs;
  float *k[7];
  int64_t Q;
  int TC;
  // operand of the batched tensor-core product (dense layout; dense_x_index): BF16
  // (+ low part for the split precision); xs_mode 0 = streaming layout
  int xs_mode;  // 0 streaming FP32 chunks, 1 dense BF16, 2 dense split BF16, 3 sparse float4
  int64_t Kp;
  int Bp;
  __nv_bfloat16 *X;
  float *mT;  // simulation-fastest copy of the stage input (near blocks)
  // control
  SimCtl *ctl;
  int *active;
  int *n_active;
  float *red;      // [B][nblk][5]
  int *red_count;  // [B]
  double *mavg;    // [n_out][B][3]
  double rtol, atol, hmax, fixed_h;
  int fresh_only;  // stage 1: evaluate k1 only for freshly admitted simulations
};

constexpr int kStageThreads = 256;

__device__ __forceinline__ void cross3(const float a[3], const float b[3], float c[3]) {
  c[0] = a[1] * b[2] - a[2] * b[1];
  c[1] = a[2] * b[0] - a[0] * b[2];
  c[2] = a[0] * b[1] - a[1] * b[0];
}

// Effective field of tile i (Eq. 5/17): H_d (from the demag product) + exchange
// (finite volumes, Eq. 12; absent neighbour = Neumann, Eq. 3) + uniaxial
// anisotropy (Eq. 16) + applied field (Eq. 7).
// H holds H_d on entry.  ha, xs: the simulation's applied field and exchange
// factor; nbr6, wex6: the tile's six face neighbours (-1: none) and their
// weights; ka, e: its anisotropy prefactor and axis; yb: the simulation's
// state of all tiles (the neighbours' m).
__device__ __forceinline__ void local_fields(const float *ha, float xs, bool exch, const int32_t *nbr6,
                                             const float *wex6, float ka, const float *e, const float *yb,
                                             const float mi[3], float H[3]) {
  H[0] = H[0] + ha[0];
  H[1] = H[1] + ha[1];
  H[2] = H[2] + ha[2];
  if (exch) {
    float he[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      const int32_t p = nbr6[f];
      if (p >= 0) {
        const float w = wex6[f];
        he[0] += w * (yb[3 * p] - mi[0]);
        he[1] += w * (yb[3 * p + 1] - mi[1]);
        he[2] += w * (yb[3 * p + 2] - mi[2]);
      }
    }
    H[0] += xs * he[0];
    H[1] += xs * he[1];
    H[2] += xs * he[2];
  }
  if (ka != 0.0f) {
    const float me = mi[0] * e[0] + mi[1] * e[1] + mi[2] * e[2];
    H[0] += ka * me * e[0];
    H[1] += ka * me * e[1];
    H[2] += ka * me * e[2];
  }
}

__device__ __forceinline__ void add_local_fields(const StageArgs &A, const float *yb, int64_t i, int b,
                                                 const float mi[3], float H[3]) {
  local_fields(A.Ha + 3 * b, A.xsc ? A.xsc[b] : 1.0f, A.exch, A.nbr + 6 * i, A.wex + 6 * i, A.kan[i],
               A.axis + 3 * i, yb, mi, H);
}

__device__ __forceinline__ void effective_field(const StageArgs &A, const float *yin, const float *Hd, int64_t i,
                                                int b, const float mi[3], float H[3]) {
  const float *hd = Hd + (size_t)b * 3 * A.n + 3 * i;
  H[0] = hd[0];
  H[1] = hd[1];
  H[2] = hd[2];
  add_local_fields(A, yin + (size_t)b * 3 * A.n, i, b, mi, H);
}

// Eq. 1 with prefactors g1 (precession) and g2 (damping):
// dm/dt = -g1 m x H - g2 m x (m x H); returns |m x H|.
__device__ __forceinline__ float llg(float g1, float g2, const float m[3], const float H[3], float k[3]) {
  float a[3], c[3];
  cross3(m, H, a);
  cross3(m, a, c);
  k[0] = -g1 * a[0] - g2 * c[0];
  k[1] = -g1 * a[1] - g2 * c[1];
  k[2] = -g1 * a[2] - g2 * c[2];
  return sqrtf(a[0] * a[0] + a[1] * a[1] + a[2] * a[2]);
}

__device__ __forceinline__ void write_stage_input(const StageArgs &A, float *ysn, int64_t i, int b,
                                                  const float v[3]) {
  float *d = ysn + (size_t)b * 3 * A.n + 3 * i;
  d[0] = v[0];
  d[1] = v[1];
  d[2] = v[2];
  const float ms = A.Ms[i];
  if (A.xs_mode == 0) {
    const int64_t q = i / A.TC, t = i - q * A.TC;
    float *x = A.xs + ((size_t)(b * A.Q + q) * 3) * A.TC + t;
    x[0] = ms * v[0];
    x[A.TC] = ms * v[1];
    x[2 * A.TC] = ms * v[2];
  } else if (A.xs_mode == 3) {
    reinterpret_cast<float4 *>(A.xs)[(size_t)b * sparse_x_stride(A.n) + i] =
        make_float4(ms * v[0], ms * v[1], ms * v[2], 0.0f);
  } else {
    const size_t term = (size_t)3 * A.Kp * A.Bp;  // split: to the second and third operand terms
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float f = ms * v[c];
      const __nv_bfloat16 hi = __float2bfloat16(f);
      __nv_bfloat16 *x = A.X + dense_x_index(c, b, i, A.Bp);
      x[0] = hi;
      if (A.xs_mode == 2) {
        const float r = f - __bfloat162float(hi);
        const __nv_bfloat16 mid = __float2bfloat16(r);
        x[term] = mid;
        x[2 * term] = __float2bfloat16(r - __bfloat162float(mid));
      }
      A.mT[(size_t)(3 * i + c) * A.Bp + b] = v[c];
    }
  }
}

// Block-reduce NV floats (sum for all but index `max_idx`, which is a
// NaN-propagating max) and return them in thread 0.
template <int NV>
__device__ __forceinline__ void block_reduce(float v[NV], int max_idx) {
  __shared__ float sh[kStageThreads / 32][NV];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < NV; ++q) v[q] = (q == max_idx) ? mtd::warp_max(v[q]) : mtd::warp_sum(v[q]);
  if (lane == 0)
#pragma unroll
    for (int q = 0; q < NV; ++q) sh[w][q] = v[q];
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 0; q < NV; ++q) {
      float acc = sh[0][q];
      for (int ww = 1; ww < (int)(blockDim.x >> 5); ++ww)
        acc = (q == max_idx) ? mtd::nan_max(acc, sh[ww][q]) : acc + sh[ww][q];
      v[q] = acc;
    }
  }
  __syncthreads();
}

// Deterministic per-simulation reduction across blocks: every block writes
// its 5 values, the last block to arrive sums them in block order.  Returns
// true in thread 0 of the last block (with tot filled).  FP32 throughout:
// the sums (squared scaled errors, volume-weighted m) need no more, and FP64
// arithmetic on the one latency-critical thread is slow on this part.
__device__ bool reduce_across_blocks(const StageArgs &A, int b, float v[5], float tot[5]) {
  const int nblk = gridDim.x;
  __shared__ int s_last;
  block_reduce<5>(v, 1);
  if (threadIdx.x == 0) {
    float *dst = A.red + ((size_t)b * nblk + blockIdx.x) * 5;
    for (int q = 0; q < 5; ++q) dst[q] = v[q];
    __threadfence();
    const int old = atomicAdd(&A.red_count[b], 1);
    s_last = (old == nblk - 1);
  }
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
  float acc[5] = {0, 0, 0, 0, 0};
  for (int blk = threadIdx.x; blk < nblk; blk += blockDim.x) {
    const float *src = A.red + ((size_t)b * nblk + blk) * 5;
    acc[0] += __ldcg(&src[0]);
    acc[1] = mtd::nan_max(acc[1], __ldcg(&src[1]));
    acc[2] += __ldcg(&src[2]);
    acc[3] += __ldcg(&src[3]);
    acc[4] += __ldcg(&src[4]);
  }
  block_reduce<5>(acc, 1);
  if (threadIdx.x == 0) {
    A.red_count[b] = 0;
    for (int q = 0; q < 5; ++q) tot[q] = acc[q];
  }
  return threadIdx.x == 0;
}

__device__ __forceinline__ void finish_sim(SimCtl &c, int status) {
  c.done = 1;
  c.status = status;
}

// Step size for the next attempt: the proposal h capped by hmax, shortened to
// land on the next output (or end) time.
__device__ __forceinline__ void plan_attempt(const StageArgs &A, SimCtl &c) {
  double hs = c.h;
  if (A.fixed_h <= 0.0 && A.hmax > 0.0 && hs > A.hmax) hs = A.hmax;
  c.clipped = 0;
  if (c.t + hs >= c.t_next) {
    hs = c.t_next - c.t;
    c.clipped = 1;
  }
  c.hs = hs;
}

// After the first derivative of a run: its torque, and a relaxation that is
// already below tolerance ends here.
__device__ __forceinline__ void close_first(SimCtl &c, float tau) {
  c.tau = (double)tau;
  c.n_rhs += 1;
  c.fresh = 0;
  if (!isfinite(tau)) finish_sim(c, MT_ENONFINITE);
  else if (c.mode == MODE_RELAX && c.tau < c.tol) finish_sim(c, MT_OK);
}

// Step control after an attempt, from the simulation's reduced sums tot =
// (sum of squared scaled errors, max torque, volume-weighted <m>): accept or
// reject, advance the time, record an output (*out_row = its index, else
// -1), finish on the end time, on the torque tolerance or on the attempt
// cap, choose the next step size and plan the next attempt.
__device__ __forceinline__ void close_attempt(const StageArgs &A, SimCtl &c, const float tot[5], int64_t *out_row) {
  *out_row = -1;
  const bool fixed = A.fixed_h > 0.0;
  // the RMS of the scaled errors; its sum is an FP32 sum on both paths
  // (tests and the step factor in FP32 too: FP64 operations take many cycles
  // on this part, and one thread does all of this)
  const float err = sqrtf(tot[0] / (3.0f * (float)A.n));
  const double tau = (double)tot[1];
  c.err = (double)err;
  c.n_attempt += 1;
  c.n_rhs += 6;
  const bool finite = isfinite(err) && isfinite(tot[2]) && isfinite(tot[3]) && isfinite(tot[4]);
  const bool accept = finite && (fixed || err <= 1.0f);
  if (!finite) {
    c.accepted = 0;
    finish_sim(c, MT_ENONFINITE);
    return;
  }
  if (accept) {
    c.n_accept += 1;
    c.t = c.clipped ? c.t_next : c.t + c.hs;
    c.tau = tau;
    c.m_last[0] = tot[2];
    c.m_last[1] = tot[3];
    c.m_last[2] = tot[4];
    if (c.mode == MODE_RUN && c.clipped) {
      *out_row = c.iout;
      c.iout += 1;
      if (c.iout >= c.n_out) {
        finish_sim(c, MT_OK);
      } else {
        c.t_next = (c.iout + 1 == c.n_out) ? c.t1 : c.t_out0 + (double)(c.iout + 1) * c.dt_out;
      }
    } else if (c.mode == MODE_RELAX) {
      if (tau < c.tol) finish_sim(c, MT_OK);
      else if (c.clipped) finish_sim(c, MT_ENOCONV);
    }
  } else {
    c.n_reject += 1;
  }
  c.accepted = accept ? 1 : 0;
  if (fixed) {
    c.h = A.fixed_h;
  } else {
    // 0.9 err^(-1/5) clamped to [0.2, 5], in FP32 (a relative 1e-7 on the
    // proposal is immaterial; FP64 transcendentals are slow on this part)
    const float f = err > 0.0f ? 0.9f * exp2f(-0.2f * log2f(err)) : 5.0f;
    c.h = c.hs * (f > 5.0f ? 5.0 : f < 0.2f ? 0.2 : (double)f);
    if (A.hmax > 0.0 && c.h > A.hmax) c.h = A.hmax;
  }
  if (!c.done && c.mode != MODE_STEPS && c.n_attempt >= c.attempt_cap) finish_sim(c, MT_ENOCONV);
  plan_attempt(A, c);
}

// ---------------------------------------------------------------------------
// kernels
// ---------------------------------------------------------------------------
__global__ void k_begin(StageArgs A) {
  mtd::pdl_enter();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int b = blockIdx.y;
  if (i >= A.n) return;
  const SimCtl &c = A.ctl[b];
  const size_t o = (size_t)b * 3 * A.n + 3 * i;
  float m[3], k1[3];
  if (c.accepted) {
    const float *yn = A.ys1 + o;  // 5th-order solution of the previous attempt
    const float inv = rsqrtf(yn[0] * yn[0] + yn[1] * yn[1] + yn[2] * yn[2]);
    m[0] = yn[0] * inv;
    m[1] = yn[1] * inv;
    m[2] = yn[2] * inv;
    const float *k7 = A.k[6] + o;
    k1[0] = k7[0];
    k1[1] = k7[1];
    k1[2] = k7[2];
    A.y[o] = m[0];
    A.y[o + 1] = m[1];
    A.y[o + 2] = m[2];
    A.k[0][o] = k1[0];
    A.k[0][o + 1] = k1[1];
    A.k[0][o + 2] = k1[2];
  } else {
    m[0] = A.y[o];
    m[1] = A.y[o + 1];
    m[2] = A.y[o + 2];
    k1[0] = A.k[0][o];
    k1[1] = A.k[0][o + 1];
    k1[2] = A.k[0][o + 2];
  }
  if (!A.active[b]) return;
  const float h = (float)(c.hs * c_dp_a[1][0]);
  const float v[3] = {m[0] + h * k1[0], m[1] + h * k1[1], m[2] + h * k1[2]};
  write_stage_input(A, A.ys0, i, b, v);
}

// commit only (after the last replay)
__global__ void k_commit(StageArgs A) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int b = blockIdx.y;
  if (i >= A.n || !A.ctl[b].accepted) return;
  const size_t o = (size_t)b * 3 * A.n + 3 * i;
  const float *yn = A.ys1 + o;
  const float inv = rsqrtf(yn[0] * yn[0] + yn[1] * yn[1] + yn[2] * yn[2]);
  A.y[o] = yn[0] * inv;
  A.y[o + 1] = yn[1] * inv;
  A.y[o + 2] = yn[2] * inv;
  A.k[0][o] = A.k[6][o];
  A.k[0][o + 1] = A.k[6][o + 1];
  A.k[0][o + 2] = A.k[6][o + 2];
}

// Stage S (1..7).  S == 1 evaluates k1 at the state (start of a run);
// S in 2..6 also forms the input of stage S+1; S == 7 closes the attempt.
// A stage is a chain of dependent L2 loads between two products.  Only H_d
// comes from the kernel just ahead (the product, which lets this one start
// once it has waited for the stage before it): everything else is read and
// reduced before the wait, so that the chain after it is one load long
// (10,000-tile film, 8 attempts: 5,579 -> 5,527 us; 6,000
// tiles, 8 simulations on the dense tensor: 4,368 -> 4,224).
template <int S>
__global__ void __launch_bounds__(kStageThreads) k_stage(StageArgs A) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int b = blockIdx.y;
  const bool active = __ldcg(&A.active[b]) != 0 && !(S == 1 && A.fresh_only && !__ldcg(&A.ctl[b].fresh));
  const bool live = active && i < A.n;
  const float *yin = (S == 1) ? A.y : ((S & 1) ? A.ys1 : A.ys0);
  const size_t o = (size_t)b * 3 * A.n + 3 * i;
  float mi[3] = {0, 0, 0}, he[3] = {0, 0, 0}, kk[3] = {0, 0, 0};
  float y0[3] = {0, 0, 0}, acc[3] = {0, 0, 0};  // S in 2..6: y + sum of the earlier k's; S == 7: their error sum
  float a_last = 0.0f, ka = 0.0f, ms = 0.0f, ax[3] = {0, 0, 0}, hs = 0.0f;
  if (live) {
    const float *yb = yin + (size_t)b * 3 * A.n;
#pragma unroll
    for (int c = 0; c < 3; ++c) mi[c] = __ldcg(yb + 3 * i + c);
    if (A.exch) {
#pragma unroll
      for (int f = 0; f < 6; ++f) {
        const int32_t p = A.nbr[6 * i + f];
        if (p >= 0) {
          const float w = A.wex[6 * i + f];
#pragma unroll
          for (int c = 0; c < 3; ++c) he[c] += w * (__ldcg(yb + 3 * p + c) - mi[c]);
        }
      }
    }
    ka = A.kan[i];
    ms = A.Ms[i];
#pragma unroll
    for (int c = 0; c < 3; ++c) ax[c] = A.axis[3 * i + c];
    if constexpr (S >= 2) {
      const double h = __ldcg(&A.ctl[b].hs);
#pragma unroll
      for (int c = 0; c < 3; ++c) y0[c] = __ldcg(A.y + o + c);
#pragma unroll
      for (int j = 0; j < S - 1; ++j) {
        if constexpr (S <= 6) {
          const float a = (float)(h * c_dp_a[S][j]);
          if (a != 0.0f)
#pragma unroll
            for (int c = 0; c < 3; ++c) acc[c] += a * __ldcg(A.k[j] + o + c);
        } else if (c_dp_err[j] != 0.0) {
#pragma unroll
          for (int c = 0; c < 3; ++c) acc[c] = fmaf((float)c_dp_err[j], __ldcg(A.k[j] + o + c), acc[c]);
        }
      }
      if constexpr (S <= 6) a_last = (float)(h * c_dp_a[S][S - 1]);
      hs = (float)h;
    }
  }
  mtd::pdl_enter();
  if (!active) return;  // uniform per block
  float tau_i = 0.0f;
  if (live) {
    const float *hd = A.Hd + o, *ha = A.Ha + 3 * b;
    const float xs = A.xsc ? A.xsc[b] : 1.0f;
    float H[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      H[c] = hd[c] + ha[c];
      if (A.exch) H[c] += xs * he[c];
    }
    if (ka != 0.0f) {
      const float me = mi[0] * ax[0] + mi[1] * ax[1] + mi[2] * ax[2];
#pragma unroll
      for (int c = 0; c < 3; ++c) H[c] += ka * me * ax[c];
    }
    tau_i = llg(A.g1[b], A.g2[b], mi, H, kk) / ms;
    float *ko = A.k[S - 1] + o;
    ko[0] = kk[0];
    ko[1] = kk[1];
    ko[2] = kk[2];
  }
  if constexpr (S >= 2 && S <= 6) {
    if (live) {
      if (a_last != 0.0f)
#pragma unroll
        for (int c = 0; c < 3; ++c) acc[c] += a_last * kk[c];
      const float v[3] = {y0[0] + acc[0], y0[1] + acc[1], y0[2] + acc[2]};
      write_stage_input(A, (S + 1) & 1 ? A.ys1 : A.ys0, i, b, v);
    }
    return;
  }
  if constexpr (S == 1 || S == 7) {
    // torque and <m> (S == 1: of the starting state; a relaxation that is
    // already converged ends here with its mean recorded), for S == 7 at the
    // 5th-order solution together with the embedded error, in FP32
    float v[5] = {0.0f, tau_i, 0.0f, 0.0f, 0.0f};
    if (live) {
      if constexpr (S == 7) {
        const float atol = (float)A.atol, rtol = (float)A.rtol;
        float e2 = 0.0f;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float e = fmaf((float)c_dp_err[6], kk[c], acc[c]);
          const float r = e * hs / (atol + rtol * fmaxf(fabsf(y0[c]), fabsf(mi[c])));
          e2 = fmaf(r, r, e2);
        }
        v[0] = e2;
      }
      const float w = (float)A.wvol[i] / sqrtf(mi[0] * mi[0] + mi[1] * mi[1] + mi[2] * mi[2]);
      v[2] = w * mi[0];
      v[3] = w * mi[1];
      v[4] = w * mi[2];
    }
    float tot[5];
    if (reduce_across_blocks(A, b, v, tot)) {
      SimCtl c = A.ctl[b];
      if constexpr (S == 1) {
        c.m_last[0] = tot[2];
        c.m_last[1] = tot[3];
        c.m_last[2] = tot[4];
        close_first(c, tot[1]);
      } else {
        int64_t row = -1;
        close_attempt(A, c, tot, &row);
        if (row >= 0) {
          double *mo = A.mavg + ((size_t)row * A.B + b) * 3;
          mo[0] = tot[2];
          mo[1] = tot[3];
          mo[2] = tot[4];
        }
      }
      if (c.done) {
        A.active[b] = 0;
        atomicSub(A.n_active, 1);
      }
      A.ctl[b] = c;
    }
  }
}

// ---------------------------------------------------------------------------
// Small tile sets: a whole run in one cooperative kernel
// ---------------------------------------------------------------------------
// Below about two thousand tiles the FP32 tensor is a few tens of MB, a
// right-hand side is a few microseconds of work, and the step graph's 13
// dependent launches per attempt are what the step costs.  Here one CTA per
// SM keeps its rows of the tensor in shared memory for the whole call (or,
// when they do not fit, reads them from the L2-resident tensor), and every
// CTA takes the step-control decisions itself from the same per-CTA partial
// sums reduced in the same fixed order (so all CTAs agree bit for bit).  The
// stage arithmetic is the graph path's except that the error norm and <m> are
// summed over rows and CTAs in another order.
//
// What is left is bound by the latency of the exchanges between the CTAs, six
// per attempt: the inputs of stages 3..7 of all tiles, and k7 with the partial
// sums (the stage-2 input every CTA forms for all tiles itself).  A barrier
// after plain stores costs three L2 round trips in a row (the stores, the
// arrival counter, the reload of the data).  Instead every 64-bit word of an
// exchange carries the number of the exchange beside its data, and the reader
// polls the data itself: one trip out and one in.  64-bit accesses are single
// copies, so a word whose tag matches holds its data, and no ordering between
// words is needed.  400-tile film: 25.5 us
// per attempt with barriers and plain data, 20.7 with this exchange and one
// lane per row doing all that follows the row sums (about half of it the
// exchanges, the rest the serial chain of one stage).
constexpr int kSmallThreads = 256;
constexpr int kSmallWarps = kSmallThreads / 32;
constexpr int kSmallRed = 3 * 8 * kSmallWarps;       // floats of one simulation's row sums
constexpr int kSmallRedL2 = 3 * 16 * kSmallWarps;    // rows read from L2: those of 8 simulations

// one tile's vector: 3 floats and the 16-bit tag in each of two 64-bit words;
// a CTA's partial sums: 5 words of a float and the tag (padded to 6)
struct alignas(16) TagVec {
  unsigned long long a, b;
};
struct alignas(16) TagSum {
  unsigned long long v[6];
};

struct SmallArgs {
  StageArgs A;
  const float *N;  // stored FP32 tensor, streaming layout
  int TR, TC;
  int64_t Q;
  // exchanged words (zeroed before the launch; tags start at 1)
  TagVec *xg;       // 2 x B x n: stage inputs (ping-pong)
  TagVec *kx;       // 2 x B x n: the committed k1 and the k7 of the attempt
  TagVec *yx;       // B x n: the state of the last accepted attempt
  TagSum *part;     // [G][B] per-CTA partial sums
  int *abort_flag;  // a bounded wait gave up: every CTA leaves
  int *status;      // device status word (MT_DEV_TIMEOUT)
  int64_t iters;    // attempts at most (kSmallChunk: their 6 tags each fit 16 bits)
  int init;         // evaluate k1 and the torque at the state first
  int R;            // rows per CTA at most
  int group;        // rows in shared memory: simulations between two CTA barriers (1, 2, 4 or 8)
  int lanes;        // threads that poll one simulation's vectors (a power of two)
};

// byte offsets of the dynamic shared memory of k_small_run
struct SmallSmem {
  size_t ctl, red, y, k, coef, par, kc, Ms, M, N, total;
};
__host__ __device__ __forceinline__ size_t small_take(size_t &o, size_t bytes) {
  const size_t at = o;
  o += (bytes + 15) & ~(size_t)15;
  return at;
}
// floats of a simulation's state in shared memory: rows of 4 tiles are read as
// three float4 from 16-byte boundaries (12 floats past the last one's end are
// allocated for a last row of fewer tiles)
__host__ __device__ __forceinline__ int small_stride(int64_t n) { return (int)((3 * n + 3) & ~(int64_t)3); }
__host__ __device__ __forceinline__ SmallSmem small_smem(int64_t n, int B, int R, bool nsmem, int group) {
  SmallSmem s;
  size_t o = 0;
  s.ctl = small_take(o, sizeof(SimCtl) * B);
  s.red = small_take(o, sizeof(float) * 2 * (nsmem ? group * kSmallRed : kSmallRedL2));
  s.y = small_take(o, sizeof(float) * B * R * 3);
  s.k = small_take(o, sizeof(float) * 7 * B * R * 3);
  s.coef = small_take(o, sizeof(float) * B * 36);  // (float)(h a_sj), s = 1..6, j < s
  s.par = small_take(o, sizeof(float) * B * 6);    // g1, g2, Ha, exchange factor
  s.kc = small_take(o, sizeof(int) * B);           // where the committed k1 and y are (see SmallSh)
  s.Ms = small_take(o, sizeof(float) * n);
  s.M = small_take(o, sizeof(float) * ((size_t)B * small_stride(n) + 12));
  s.N = small_take(o, nsmem ? sizeof(float) * 6 * R * n : 0);
  s.total = o;
  return s;
}

struct SmallSh {
  SimCtl *ctl;
  float *red, *y, *k, *coef, *par, *Ms, *M, *N;
  // per simulation: the tag of the exchange that published the committed k1
  // (0: it is still in global memory, in k[0]), kKcBuf = its buffer of kx,
  // kKcY = the committed y is in yx under the same tag (else in global y)
  int *kc;
};
constexpr int kKcBuf = 1 << 30, kKcY = 1 << 29, kKcTag = 0xffff;

__device__ __forceinline__ void st_pair(void *p, unsigned long long a, unsigned long long b) {
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void ld_pair(const void *p, unsigned long long &a, unsigned long long &b) {
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ void publish_vec(TagVec *p, const float v[3], unsigned tag) {
  const unsigned y = __float_as_uint(v[1]);
  const unsigned hi_a = (y & 0xffffu) | (tag << 16), hi_b = (y >> 16) | (tag << 16);
  st_pair(p, __float_as_uint(v[0]) | ((unsigned long long)hi_a << 32),
          __float_as_uint(v[2]) | ((unsigned long long)hi_b << 32));
}
__device__ __forceinline__ bool vec_tagged(unsigned long long a, unsigned long long b, unsigned tag) {
  return (unsigned)(a >> 48) == tag && (unsigned)(b >> 48) == tag;
}
__device__ __forceinline__ void vec_of(unsigned long long a, unsigned long long b, float v[3]) {
  v[0] = __uint_as_float((unsigned)a);
  v[1] = __uint_as_float(((unsigned)(a >> 32) & 0xffffu) | ((unsigned)(b >> 32) << 16));
  v[2] = __uint_as_float((unsigned)b);
}

// Bound of every polling loop: after ~2 s (or once another CTA gave up) the
// status word gets MT_DEV_TIMEOUT, the abort flag is raised and the loop ends.
struct PollLimit {
  uint32_t it = 0;
  uint64_t t0 = 0;
  __device__ __forceinline__ bool expired(const SmallArgs &S) {
    if ((++it & 63u) != 0u) return false;
    if (*reinterpret_cast<volatile int *>(S.abort_flag)) return true;
    const uint64_t t = mtd::globaltimer_ns();
    if (t0 == 0) t0 = t;
    if (t - t0 <= 2000000000ull) return false;
    atomicExch(S.status, MT_DEV_TIMEOUT);
    atomicExch(S.abort_flag, 1);
    return true;
  }
};

// n tagged vectors from src: f(j, v) for this thread's j = first, first +
// lanes, ... (four in flight at once).  False when the wait gave up.
template <typename F>
__device__ __forceinline__ bool poll_vecs(const SmallArgs &S, const TagVec *src, int n, unsigned tag, int first,
                                          int lanes, F &&f) {
  constexpr int U = 4;
  PollLimit lim;
  for (int j0 = first; j0 < n; j0 += U * lanes) {
    unsigned long long a[U], b[U];
    for (;;) {
      bool all = true;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int j = j0 + u * lanes;
        if (j < n) ld_pair(src + j, a[u], b[u]);
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (j0 + u * lanes < n) all = all && vec_tagged(a[u], b[u], tag);
      if (all) break;
      if (lim.expired(S)) return false;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = j0 + u * lanes;
      if (j < n) {
        float v[3];
        vec_of(a[u], b[u], v);
        f(j, v);
      }
    }
  }
  return true;
}

// H_d row sums of simulation b for the CTA's rows, from the stage input of all
// tiles in sh.M, as partial sums in `red`.  Rows in shared memory: the CTA's
// threads over the columns, each warp's sums of row value v = 3 q + c at
// red[warp 3 RMAX + v].
template <int RMAX, bool PLANAR>
__device__ __forceinline__ void small_product(const SmallSh &sh, const float *mb, float *red, int R, int nr, int n) {
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  constexpr int NV = 3 * RMAX, NS = NV <= 8 ? 8 : NV <= 16 ? 16 : 32;
  const int pl = R * n;  // entries of one plane of the CTA's rows
  float acc[NS];
#pragma unroll
  for (int v = 0; v < NS; ++v) acc[v] = 0.0f;
  // rows past nr repeat the last one (their sums are dropped): no branch
  // between the loads of a column
  const float *e[RMAX];
#pragma unroll
  for (int q = 0; q < RMAX; ++q) e[q] = sh.N + (q < nr ? q : nr - 1) * n;
#pragma unroll 2
  for (int j = tid; j < n; j += kSmallThreads) {
    const float ms = sh.Ms[j];
    const float x0 = ms * mb[3 * j], x1 = ms * mb[3 * j + 1], x2 = ms * mb[3 * j + 2];
#pragma unroll
    for (int q = 0; q < RMAX; ++q) {
      const float *f = e[q] + j;
      if constexpr (PLANAR) {  // no xz, yz
        const float nxx = f[0], nxy = f[pl], nyy = f[3 * pl], nzz = f[5 * pl];
        acc[3 * q] = fmaf(nxx, x0, fmaf(nxy, x1, acc[3 * q]));
        acc[3 * q + 1] = fmaf(nxy, x0, fmaf(nyy, x1, acc[3 * q + 1]));
        acc[3 * q + 2] = fmaf(nzz, x2, acc[3 * q + 2]);
      } else {
        const float nxx = f[0], nxy = f[pl], nxz = f[2 * pl], nyy = f[3 * pl], nyz = f[4 * pl], nzz = f[5 * pl];
        acc[3 * q] = fmaf(nxx, x0, fmaf(nxy, x1, fmaf(nxz, x2, acc[3 * q])));
        acc[3 * q + 1] = fmaf(nxy, x0, fmaf(nyy, x1, fmaf(nyz, x2, acc[3 * q + 1])));
        acc[3 * q + 2] = fmaf(nxz, x0, fmaf(nyz, x1, fmaf(nzz, x2, acc[3 * q + 2])));
      }
    }
  }
  const float tot = mtd::warp_reduce_scatter<NS>(acc, lane);  // lane l: value l / (32 / NS)
  const int v = lane / (32 / NS);
  if (lane % (32 / NS) == 0 && v < 3 * nr) red[w * NV + v] = tot;
}

// The same for tile sets whose rows do not fit the shared memory but whose
// tensor stays in L2 (up to ~100 MB): each warp owns rows w and w + 8 of the
// CTA (at most 16) and reads them from the streaming layout, lanes over the
// columns (128 consecutive columns of an entry plane are contiguous, 16-byte
// aligned), so no cross-warp reduction is needed: simulation s of the SB that
// start at b at red[s 3 kSmallRowsL2 + 3 q + c].  The L2 reads bound it, so up
// to 4 simulations share them (2,016-tile prism, 4 simulations, 8 attempts:
// 2,302 us with a pass per simulation, 1,377 so; one simulation of an
// 1,190-tile film 568 -> 388).
constexpr int kSmallRowsL2 = 2 * kSmallWarps;
template <int SB, bool PLANAR>
__device__ __forceinline__ void small_product_l2(const SmallArgs &S, const SmallSh &sh, int b, float *red, int nr,
                                                 int64_t r0, int n) {
  constexpr int NP = PLANAR ? 4 : 6;
  constexpr int U = SB == 1 ? 2 : 1;  // groups of 128 columns in flight
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const size_t plane = (size_t)S.TR * S.TC, chunk = NP * plane;
  const float *rowp[2] = {nullptr, nullptr};
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int q = w + kSmallWarps * r;
    if (q < nr) {
      const int64_t i = r0 + q, p = i / S.TR;
      rowp[r] = S.N + (size_t)p * S.Q * chunk + (size_t)(i - p * S.TR) * S.TC;
    }
  }
  const float *mb[SB];  // (a group past the last simulation repeats it)
#pragma unroll
  for (int s = 0; s < SB; ++s) mb[s] = sh.M + (b + s < S.A.B ? b + s : S.A.B - 1) * small_stride(n);
  float acc[SB][2][3];
#pragma unroll
  for (int s = 0; s < SB; ++s)
#pragma unroll
    for (int r = 0; r < 2; ++r) acc[s][r][0] = acc[s][r][1] = acc[s][r][2] = 0.0f;
  // a lane takes 4 adjacent columns (one 16-byte load per entry plane; the
  // padding of the last column chunk holds zeros)
  for (int j0 = 4 * lane; j0 < n; j0 += 128 * U) {
    float4 ent[U][2][NP];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = j0 + 128 * u;
      const int cq = j / S.TC;
      const size_t off = (size_t)cq * chunk + (size_t)(j - cq * S.TC);
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int e = 0; e < NP; ++e)
          ent[u][r][e] = (rowp[r] && j < n) ? __ldg(reinterpret_cast<const float4 *>(rowp[r] + off + e * plane))
                                            : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = j0 + 128 * u;
      if (j >= n) break;
      float ms[4];
      *reinterpret_cast<float4 *>(ms) = *reinterpret_cast<const float4 *>(sh.Ms + j);
#pragma unroll
      for (int s = 0; s < SB; ++s) {
        float x[12];  // 4 tiles' vectors, times Ms (0 past the last tile)
#pragma unroll
        for (int q = 0; q < 3; ++q)
          reinterpret_cast<float4 *>(x)[q] = *reinterpret_cast<const float4 *>(mb[s] + 3 * j + 4 * q);
#pragma unroll
        for (int q = 0; q < 12; ++q) x[q] = j + q / 3 < n ? ms[q / 3] * x[q] : 0.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float x0 = x[3 * k], x1 = x[3 * k + 1], x2 = x[3 * k + 2];
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            const float *ex = reinterpret_cast<const float *>(&ent[u][r][0]) + k;  // plane e at ex[4 e]
            float *h = acc[s][r];
            if constexpr (PLANAR) {
              h[0] = fmaf(ex[0], x0, fmaf(ex[4], x1, h[0]));
              h[1] = fmaf(ex[4], x0, fmaf(ex[8], x1, h[1]));
              h[2] = fmaf(ex[12], x2, h[2]);
            } else {
              h[0] = fmaf(ex[0], x0, fmaf(ex[4], x1, fmaf(ex[8], x2, h[0])));
              h[1] = fmaf(ex[4], x0, fmaf(ex[12], x1, fmaf(ex[16], x2, h[1])));
              h[2] = fmaf(ex[8], x0, fmaf(ex[16], x1, fmaf(ex[20], x2, h[2])));
            }
          }
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    if (!rowp[r]) continue;  // the same in the whole warp
    const int q = w + kSmallWarps * r;
#pragma unroll
    for (int s = 0; s < SB; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float v = mtd::warp_sum(acc[s][r][c]);
        if (lane == 0) red[s * 3 * kSmallRowsL2 + 3 * q + c] = v;
      }
  }
}

// Warp: the sums of 5 values over its lanes (sum, max, sum, sum, sum)
__device__ __forceinline__ void small_warp_reduce(float v[5]) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    v[1] = mtd::nan_max(v[1], __shfl_xor_sync(0xffffffffu, v[1], o));
    v[2] += __shfl_xor_sync(0xffffffffu, v[2], o);
    v[3] += __shfl_xor_sync(0xffffffffu, v[3], o);
    v[4] += __shfl_xor_sync(0xffffffffu, v[4], o);
  }
}
// the CTA's 5 values of simulation b (one lane per row) to every CTA
__device__ __forceinline__ void small_partial(const SmallArgs &S, int b, float v[5], unsigned tag) {
  small_warp_reduce(v);
  if ((threadIdx.x & 31) < 3) {
    const int l = threadIdx.x & 31;  // lane l sends words 2 l and 2 l + 1
    const float lo = l == 0 ? v[0] : l == 1 ? v[2] : v[4], hi = l == 0 ? v[1] : l == 1 ? v[3] : 0.0f;
    TagSum *dst = S.part + (size_t)blockIdx.x * S.A.B + b;
    st_pair(&dst->v[2 * l], __float_as_uint(lo) | ((unsigned long long)tag << 32),
            __float_as_uint(hi) | ((unsigned long long)tag << 32));
  }
}
// A warp: the G partials of b added in a fixed order (lane-strided, then a
// butterfly), so all CTAs hold the same totals.  False when the wait gave up.
__device__ __forceinline__ bool small_total(const SmallArgs &S, int b, unsigned tag, float tot[5]) {
  float acc[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
  constexpr int U = 5;  // of one lane, in flight at once (152 CTAs: all)
  PollLimit lim;
  bool ok = true;
  for (int g0 = threadIdx.x & 31; ok && g0 < (int)gridDim.x; g0 += 32 * U) {
    unsigned long long w[U][6];
    for (;;) {
      bool all = true;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const TagSum *src = S.part + (size_t)(g0 + 32 * u) * S.A.B + b;
        if (g0 + 32 * u < (int)gridDim.x)
#pragma unroll
          for (int l = 0; l < 3; ++l) ld_pair(&src->v[2 * l], w[u][2 * l], w[u][2 * l + 1]);
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (g0 + 32 * u < (int)gridDim.x)
#pragma unroll
          for (int l = 0; l < 6; ++l) all = all && (unsigned)(w[u][l] >> 32) == tag;
      if (all) break;
      if (lim.expired(S)) {
        ok = false;
        break;
      }
    }
    if (!ok) break;
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (g0 + 32 * u < (int)gridDim.x) {
        acc[0] += __uint_as_float((unsigned)w[u][0]);
        acc[1] = mtd::nan_max(acc[1], __uint_as_float((unsigned)w[u][1]));
        acc[2] += __uint_as_float((unsigned)w[u][2]);
        acc[3] += __uint_as_float((unsigned)w[u][3]);
        acc[4] += __uint_as_float((unsigned)w[u][4]);
      }
  }
  ok = __all_sync(0xffffffffu, ok);
  small_warp_reduce(acc);
  for (int q = 0; q < 5; ++q) tot[q] = acc[q];
  return ok;
}

// m / |m| with every rounding pinned (no contraction freedom), so that the
// CTA committing a row and the CTAs forming the next stage input from it
// compute the same bits
__device__ __forceinline__ void small_unit(const float *v, float *out) {
  const float inv = rsqrtf(__fmaf_rn(v[2], v[2], __fmaf_rn(v[1], v[1], __fmul_rn(v[0], v[0]))));
  out[0] = __fmul_rn(v[0], inv);
  out[1] = __fmul_rn(v[1], inv);
  out[2] = __fmul_rn(v[2], inv);
}

// A warp: (float)(h a_sj) of every stage-input row s = 1..6 (the inputs of
// stages 2..7) and j < s of simulation b: coef[36 b + 6 (s - 1) + j]
__device__ __forceinline__ void small_coefficients(const SmallSh &sh, int b) {
  for (int rj = threadIdx.x & 31; rj < 36; rj += 32) {
    const int r = rj / 6, j = rj - r * 6;
    if (j <= r) sh.coef[36 * b + rj] = (float)(sh.ctl[b].hs * c_dp_a[r + 1][j]);
  }
}

// The constants of row q = lane of the CTA (every warp holds them: a warp owns
// simulations, its lanes the rows), a missing neighbour as the row itself
// with weight 0
struct SmallRow {
  int nbr[6];
  float wex[6], kan, axis[3], Ms, wv;
};

// One stage of every running simulation: the product, then by the warp that
// owns the simulation (b mod 8; lane q = row q of the CTA) the local fields,
// Eq. 1 (the arithmetic of k_stage) and what follows from it: after stages
// 1..6 k, for stages 2..6 also the next stage's input, published under
// `tag`; after stage 7 k7 and the sums of the error norm, the torque and <m>;
// after stage 1 (k1 at the state) k1 and the torque.  One CTA barrier between
// the product of a simulation (MANY: of S.group of them; rows read from L2: of
// eight) and the rest: sh.M is read only before it (a later exchange may
// overwrite it), and the two buffers of row sums alternate.
//
// What a row needs of the other tiles: m itself and the exchange sum.
struct SmallPre {
  float mi[3], he[3];
};
__device__ __forceinline__ void small_pre(const StageArgs &A, const SmallRow &rw, const float *mb, int i,
                                          SmallPre &pr) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    pr.mi[c] = mb[3 * i + c];
    pr.he[c] = 0.0f;
  }
  if (A.exch) {
#pragma unroll
    for (int f = 0; f < 6; ++f)
#pragma unroll
      for (int c = 0; c < 3; ++c) pr.he[c] += rw.wex[f] * (mb[3 * rw.nbr[f] + c] - pr.mi[c]);
  }
}

// the owning warp's part after the barrier; WSUM partial sums per row value
// (value v of part w at red[w WSTRIDE + v])
template <int WSUM, int WSTRIDE>
__device__ __forceinline__ void small_rows(const SmallArgs &S, const SmallSh &sh, const SmallRow &rw,
                                           const SmallPre &pr, const float *red, int b, int st, unsigned tag, int nr,
                                           int64_t r0) {
  const StageArgs &A = S.A;
  const int n = (int)A.n, B = A.B, R = S.R;
  const size_t kpl = (size_t)B * R * 3;  // floats of one derivative plane
  const int q = threadIdx.x & 31, i = (int)r0 + q;
  const bool row = q < nr;
  const float *mi = pr.mi, *he = pr.he;
  float k[3] = {0.0f, 0.0f, 0.0f}, tau = 0.0f;
  float *ks = sh.k + ((size_t)b * R + q) * 3;  // row q's k1; plane s at + s kpl
  const float *y0 = sh.y + ((size_t)b * R + q) * 3;
  if (row) {
    const float *pb = sh.par + 6 * b;
    float H[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float s = 0.0f;
#pragma unroll
      for (int w = 0; w < WSUM; ++w) s += red[w * WSTRIDE + 3 * q + c];
      H[c] = -s + pb[2 + c];
      if (A.exch) H[c] += pb[5] * he[c];
    }
    if (rw.kan != 0.0f) {
      const float me = mi[0] * rw.axis[0] + mi[1] * rw.axis[1] + mi[2] * rw.axis[2];
#pragma unroll
      for (int c = 0; c < 3; ++c) H[c] += rw.kan * me * rw.axis[c];
    }
    const float mxh = llg(pb[0], pb[1], mi, H, k);
    if (st == 1 || st == 7) tau = mxh / rw.Ms;
    for (int c = 0; c < 3; ++c) ks[(st - 1) * kpl + c] = k[c];
    if (st >= 2 && st <= 6) {
      // this row's input of the next stage: y + sum_j (h a_sj) k_j
      const float *cf = sh.coef + 36 * b + 6 * (st - 1);
      float acc[3] = {0.0f, 0.0f, 0.0f}, a[6], kj[6][3];
#pragma unroll
      for (int j = 0; j < 6; ++j) {  // all loads before the sums
        a[j] = j < st ? cf[j] : 0.0f;
#pragma unroll
        for (int c = 0; c < 3; ++c) kj[j][c] = j < st - 1 ? ks[j * kpl + c] : k[c];
      }
#pragma unroll
      for (int j = 0; j < 6; ++j)
        if (a[j] != 0.0f)
#pragma unroll
          for (int c = 0; c < 3; ++c) acc[c] += a[j] * kj[j][c];
      const float v[3] = {y0[0] + acc[0], y0[1] + acc[1], y0[2] + acc[2]};
      publish_vec(S.xg + (size_t)((st + 1) & 1) * B * n + (size_t)b * n + i, v, tag);
    }
  }
  if (st >= 2 && st <= 6) return;
  // k1 (stage 1) or k7 into the buffer that does not hold the committed k1
  const int into = st == 1 ? 0 : (sh.kc[b] & kKcBuf) ? 0 : 1;
  float v[5] = {0.0f, tau, 0.0f, 0.0f, 0.0f};
  if (row) {
    publish_vec(S.kx + (size_t)into * B * n + (size_t)b * n + i, k, tag);
    if (st == 7) {
      // embedded error, torque and <m> at the 5th-order solution (the
      // stage-7 input), in FP32
      const float hs = (float)sh.ctl[b].hs, atol = (float)A.atol, rtol = (float)A.rtol;
      for (int c = 0; c < 3; ++c) {
        float e = 0.0f;
#pragma unroll
        for (int j = 0; j < 7; ++j)
          if (c_dp_err[j] != 0.0) e = fmaf((float)c_dp_err[j], j == 6 ? k[c] : ks[j * kpl + c], e);
        const float r = e * hs / (atol + rtol * fmaxf(fabsf(y0[c]), fabsf(mi[c])));
        v[0] = fmaf(r, r, v[0]);
      }
      const float wv = rw.wv / sqrtf(mi[0] * mi[0] + mi[1] * mi[1] + mi[2] * mi[2]);
      for (int c = 0; c < 3; ++c) v[2 + c] = wv * mi[c];
    }
  }
  small_partial(S, b, v, tag);
}

template <int RMAX, bool NSMEM, bool PLANAR, bool MANY>
__device__ __forceinline__ void small_stage(const SmallArgs &S, const SmallSh &sh, const SmallRow &rw, int st,
                                            unsigned tag, int nr, int64_t r0, int &buf) {
  const StageArgs &A = S.A;
  const int n = (int)A.n, B = A.B;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  SmallPre pr = {{0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f}};
  if constexpr (MANY) {
    for (int base = 0; base < B; base += S.group) {
      const int end = base + S.group < B ? base + S.group : B;
      float *red = sh.red + buf * S.group * kSmallRed;
      buf ^= 1;
      bool live = false;  // the same in every thread
      for (int b = base; b < end; ++b) {
        if (sh.ctl[b].done) continue;
        live = true;
        small_product<RMAX, PLANAR>(sh, sh.M + b * small_stride(n), red + (b - base) * kSmallRed, S.R, nr, n);
      }
      if (!live) continue;
      const int b = base + ((warp - base) & (kSmallWarps - 1));  // this warp's simulation of the group
      const bool mine = b < end && !sh.ctl[b].done;
      if (mine && lane < nr) small_pre(A, rw, sh.M + b * small_stride(n), (int)r0 + lane, pr);
      __syncthreads();
      if (mine)
        small_rows<kSmallWarps, 3 * RMAX>(S, sh, rw, pr, red + (b - base) * kSmallRed, b, st, tag, nr, r0);
    }
  } else if constexpr (NSMEM) {
    for (int b = 0; b < B; ++b) {
      if (sh.ctl[b].done) continue;  // the same in every thread
      const float *mb = sh.M + b * small_stride(n);
      float *red = sh.red + buf * kSmallRed;
      buf ^= 1;
      small_product<RMAX, PLANAR>(sh, mb, red, S.R, nr, n);
      const bool mine = warp == (b & (kSmallWarps - 1));
      if (mine && lane < nr) small_pre(A, rw, mb, (int)r0 + lane, pr);
      __syncthreads();
      if (mine) small_rows<kSmallWarps, 3 * RMAX>(S, sh, rw, pr, red, b, st, tag, nr, r0);
    }
  } else {
    for (int base = 0; base < B; base += kSmallWarps) {
      const int end = base + kSmallWarps < B ? base + kSmallWarps : B;
      float *red = sh.red + buf * kSmallRedL2;
      buf ^= 1;
      for (int b = base; b < end; b += 4) {
        float *rb = red + (b - base) * 3 * kSmallRowsL2;
        bool live = false;  // the same in every thread
        for (int s = b; s < b + 4 && s < end; ++s) live = live || !sh.ctl[s].done;
        if (!live) continue;
        if (end - b >= 4) small_product_l2<4, PLANAR>(S, sh, b, rb, nr, r0, n);
        else if (end - b == 3) small_product_l2<3, PLANAR>(S, sh, b, rb, nr, r0, n);
        else if (end - b == 2) small_product_l2<2, PLANAR>(S, sh, b, rb, nr, r0, n);
        else small_product_l2<1, PLANAR>(S, sh, b, rb, nr, r0, n);
      }
      const int b = base + warp;
      const bool mine = b < end && !sh.ctl[b].done;
      if (mine && lane < nr) small_pre(A, rw, sh.M + b * small_stride(n), (int)r0 + lane, pr);
      __syncthreads();
      if (mine) small_rows<1, 0>(S, sh, rw, pr, red + warp * 3 * kSmallRowsL2, b, st, tag, nr, r0);
    }
  }
}

template <int RMAX, bool NSMEM, bool PLANAR, bool MANY>
__global__ void __launch_bounds__(kSmallThreads, 1) k_small_run(SmallArgs S) {
  extern __shared__ __align__(16) unsigned char smem[];
  const StageArgs &A = S.A;
  const int64_t n = A.n;
  const int B = A.B, R = S.R;
  const int G = gridDim.x, g = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t r0 = (int64_t)g * n / G, r1 = (int64_t)(g + 1) * n / G;
  const int nr = (int)(r1 - r0);
  const SmallSmem L = small_smem(n, B, R, NSMEM, MANY ? S.group : 1);
  SmallSh sh;
  sh.ctl = reinterpret_cast<SimCtl *>(smem + L.ctl);
  sh.red = reinterpret_cast<float *>(smem + L.red);
  sh.y = reinterpret_cast<float *>(smem + L.y);
  sh.k = reinterpret_cast<float *>(smem + L.k);
  sh.coef = reinterpret_cast<float *>(smem + L.coef);
  sh.par = reinterpret_cast<float *>(smem + L.par);
  sh.kc = reinterpret_cast<int *>(smem + L.kc);
  sh.Ms = reinterpret_cast<float *>(smem + L.Ms);
  sh.M = reinterpret_cast<float *>(smem + L.M);
  sh.N = reinterpret_cast<float *>(smem + L.N);
  const size_t kpl = (size_t)B * R * 3;
  // `lanes` threads poll the vectors of one simulation: this one b0, b0 + sims, ...
  const int lanes = MANY ? S.lanes : kSmallThreads, sims = MANY ? kSmallThreads / lanes : 1;
  const int b0 = MANY ? tid / lanes : 0, j0 = MANY ? tid & (lanes - 1) : tid;
  unsigned seq = 0;  // exchanges so far: the next one's tag is seq + 1
  int buf = 0;
  bool ok = true;

  // control blocks and parameters, Ms, the CTA's rows of N (plane e, row q,
  // column j) and their tile constants, the rows of y and of the derivative
  // the next attempt starts from
  for (int b = tid; b < B; b += kSmallThreads) {
    sh.ctl[b] = A.ctl[b];
    float *pb = sh.par + 6 * b;
    pb[0] = A.g1[b];
    pb[1] = A.g2[b];
    pb[2] = A.Ha[3 * b];
    pb[3] = A.Ha[3 * b + 1];
    pb[4] = A.Ha[3 * b + 2];
    pb[5] = A.xsc ? A.xsc[b] : 1.0f;
    sh.kc[b] = 0;
  }
  for (int64_t j = tid; j < n; j += kSmallThreads) sh.Ms[j] = A.Ms[j];
  if (NSMEM)
    for (int64_t q = tid; q < (int64_t)6 * nr * n; q += kSmallThreads) {
      const int64_t j = q % n, eq = q / n;
      const int e = (int)(eq / nr), r = (int)(eq % nr);
      constexpr int NP = PLANAR ? 4 : 6;
      const int pl = stream_plane(e, NP);
      if (pl >= 0) sh.N[((size_t)e * R + r) * n + j] = S.N[layout_index(r0 + r, j, pl, S.TR, S.TC, NP, S.Q)];
    }
  SmallRow rw;
  {
    const int64_t i = r0 + (lane < nr ? lane : 0);
    for (int f = 0; f < 6; ++f) {
      const int32_t p = A.nbr[6 * i + f];
      rw.nbr[f] = p >= 0 ? p : (int)i;
      rw.wex[f] = p >= 0 ? A.wex[6 * i + f] : 0.0f;
    }
    rw.kan = A.kan[i];
    for (int c = 0; c < 3; ++c) rw.axis[c] = A.axis[3 * i + c];
    rw.Ms = A.Ms[i];
    rw.wv = (float)A.wvol[i];
  }
  for (int p = tid; p < B * nr * 3; p += kSmallThreads) {
    const int b = p / (nr * 3), qc = p - b * nr * 3;
    const size_t o = (size_t)b * 3 * n + 3 * r0 + qc;
    sh.y[(size_t)b * R * 3 + qc] = A.y[o];
    sh.k[(size_t)b * R * 3 + qc] = A.k[0][o];
  }
  if (S.init)
    for (int b = 0; b < B; ++b)
      for (int q = tid; q < 3 * (int)n; q += kSmallThreads) sh.M[b * small_stride(n) + q] = A.y[(size_t)b * 3 * n + q];
  __syncthreads();

  if (S.init) {  // k1 and the torque at the state
    small_stage<RMAX, NSMEM, PLANAR, MANY>(S, sh, rw, 1, 1, nr, r0, buf);
    seq = 1;
    for (int b = warp; ok && b < B; b += kSmallWarps) {
      if (sh.ctl[b].done) continue;
      float tot[5];
      ok = small_total(S, b, 1, tot);
      if (ok && lane == 0) {
        close_first(sh.ctl[b], tot[1]);
        sh.kc[b] = 1;  // k1: tag 1 in buffer 0 of kx
      }
      __syncwarp();
    }
  }
  for (int b = warp; b < B; b += kSmallWarps)
    if (!sh.ctl[b].done) small_coefficients(sh, b);
  ok = __syncthreads_and(ok);

  for (int64_t it = 0; ok && it < S.iters; ++it) {
    bool any = false;
    for (int b = 0; b < B; ++b) any = any || !sh.ctl[b].done;
    if (!any) break;
    // stage 2 needs no exchange between CTAs: every CTA forms the input of
    // all tiles, y + (h a_21) k1, from the committed state (after an accepted
    // attempt: the normalised 5th-order solution still in sh.M and the k7
    // every CTA published; else the committed y and k1)
    for (int b = b0; b < B; b += sims) {
      if (sh.ctl[b].done) continue;
      const int kc = sh.kc[b];
      const bool adopt = it > 0 && sh.ctl[b].accepted;
      const float a21 = sh.coef[36 * b];
      float *mb = sh.M + b * small_stride(n);
      const float *yb = A.y + (size_t)b * 3 * n, *kb = A.k[0] + (size_t)b * 3 * n;
      if (!adopt) {  // the committed y into sh.M
        if (kc & kKcY)
          ok = poll_vecs(S, S.yx + (size_t)b * n, (int)n, kc & kKcTag, j0, lanes, [&](int j, const float *y) {
                 for (int c = 0; c < 3; ++c) mb[3 * j + c] = y[c];
               }) && ok;
        else
          for (int j = j0; j < n; j += lanes)
            for (int c = 0; c < 3; ++c) mb[3 * j + c] = __ldcg(yb + 3 * j + c);
      }
      auto form = [&](int j, const float *k1) {  // (the thread that wrote mb[j])
        float y[3] = {mb[3 * j], mb[3 * j + 1], mb[3 * j + 2]};
        if (adopt) small_unit(mb + 3 * j, y);
#pragma unroll
        for (int c = 0; c < 3; ++c) mb[3 * j + c] = __fadd_rn(y[c], __fmul_rn(a21, k1[c]));
      };
      if (kc & kKcTag)
        ok = poll_vecs(S, S.kx + (size_t)((kc & kKcBuf) ? 1 : 0) * B * n + (size_t)b * n, (int)n, kc & kKcTag, j0,
                       lanes, form) &&
             ok;
      else
        for (int j = j0; j < n; j += lanes) {
          const float k1[3] = {__ldcg(kb + 3 * j), __ldcg(kb + 3 * j + 1), __ldcg(kb + 3 * j + 2)};
          form(j, k1);
        }
    }
    ok = __syncthreads_and(ok);
    if (!ok) break;
    for (int st = 2; st <= 7; ++st) {
      if (st > 2) {  // all tiles' input of this stage
        for (int b = b0; b < B; b += sims) {
          if (sh.ctl[b].done) continue;
          float *mb = sh.M + b * small_stride(n);
          ok = poll_vecs(S, S.xg + (size_t)(st & 1) * B * n + (size_t)b * n, (int)n, seq + st - 2, j0, lanes,
                         [&](int j, const float *v) {
                           for (int c = 0; c < 3; ++c) mb[3 * j + c] = v[c];
                         }) && ok;
        }
        ok = __syncthreads_and(ok);
        if (!ok) break;
      }
      small_stage<RMAX, NSMEM, PLANAR, MANY>(S, sh, rw, st, seq + st - 1, nr, r0, buf);
    }
    if (!ok) break;
    seq += 6;  // the k7 and the partial sums went out under this tag
    for (int b = warp; ok && b < B; b += kSmallWarps) {
      if (sh.ctl[b].done) continue;
      float tot[5];
      ok = small_total(S, b, seq, tot);
      if (!ok) break;
      if (lane == 0) {
        int64_t out = -1;
        close_attempt(A, sh.ctl[b], tot, &out);
        if (g == 0 && out >= 0) {
          double *mo = A.mavg + ((size_t)out * B + b) * 3;
          mo[0] = tot[2];
          mo[1] = tot[3];
          mo[2] = tot[4];
        }
      }
      __syncwarp();
      small_coefficients(sh, b);
      if (!sh.ctl[b].accepted) continue;
      // adopt the normalised 5th-order solution (published for a stage-2
      // input after a later rejection); k7 is the next k1
      if (lane < nr) {
        float *y0 = sh.y + ((size_t)b * R + lane) * 3;
        float *k1 = sh.k + ((size_t)b * R + lane) * 3;
        small_unit(sh.M + b * small_stride(n) + 3 * (r0 + lane), y0);
        publish_vec(S.yx + (size_t)b * n + r0 + lane, y0, seq);
        for (int c = 0; c < 3; ++c) k1[c] = k1[6 * kpl + c];
      }
      if (lane == 0) sh.kc[b] = ((sh.kc[b] & kKcBuf) ^ kKcBuf) | kKcY | (int)seq;
    }
    ok = __syncthreads_and(ok);
  }
  if (!ok) return;  // timed out: the status word tells the host
  // write back: the state and the next derivative of this CTA's rows; CTA 0
  // the control blocks (nothing left to commit) and the active set.  (Every
  // CTA's partial sums of the last attempt have arrived, so none still reads
  // the global y and k1 for its stage 2.)
  for (int p = tid; p < B * nr * 3; p += kSmallThreads) {
    const int b = p / (nr * 3), qc = p - b * nr * 3;
    const size_t o = (size_t)b * 3 * n + 3 * r0 + qc;
    A.y[o] = sh.y[(size_t)b * R * 3 + qc];
    A.k[0][o] = sh.k[(size_t)b * R * 3 + qc];
  }
  if (g == 0 && tid == 0) {
    int na = 0;
    for (int b = 0; b < B; ++b) {
      SimCtl c = sh.ctl[b];
      c.accepted = 0;
      A.ctl[b] = c;
      A.active[b] = c.done ? 0 : 1;
      na += c.done ? 0 : 1;
    }
    *A.n_active = na;
  }
}

// failure-detection self-test: CTA 0 leaves without publishing its words, so
// the other CTAs' bounded wait for them runs out
__global__ void k_exchange_selftest(SmallArgs S) {
  if (blockIdx.x == 0) return;
  const float v[3] = {1.0f, 2.0f, 3.0f};
  if (threadIdx.x == 0) publish_vec(S.xg + blockIdx.x, v, 1);
  poll_vecs(S, S.xg, gridDim.x, 1, threadIdx.x, blockDim.x, [](int, const float *) {});
}

// put a prepared control block into slot b and make it active
__global__ void k_admit(SimCtl *ctl, int *active, int *n_active, int b, SimCtl c) {
  ctl[b] = c;
  if (!active[b]) {
    active[b] = 1;
    atomicAdd(n_active, 1);
  }
}

// Energy (Eqs. 4, 6, 8, 11, 15): every quadratic density is -(mu0 Ms/2) m.H
// of its field and the Zeeman one -mu0 Ms m.Ha, so per tile
//   e_i = -mu0 Ms_i V_i m_i.(Ha + (H_d + H_ex + H_an)/2)  split by term.
__global__ void k_energy(int64_t n, const int32_t *nbr, const float *wex, const float *kan, const float *axis,
                         const float *Ms, const double *wvol, double vol_total, bool exch, const float *m,
                         const float *Hd, const float *Ha, const float *xsc, double *E) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int b = blockIdx.y;
  double e[4] = {0, 0, 0, 0};
  if (i < n) {
    const size_t o = (size_t)b * 3 * n + 3 * i;
    const float mi[3] = {m[o], m[o + 1], m[o + 2]};
    double hex[3] = {0, 0, 0}, han[3] = {0, 0, 0};
    if (exch) {
      const float *mb = m + (size_t)b * 3 * n;
      for (int f = 0; f < 6; ++f) {
        const int32_t p = nbr[6 * i + f];
        if (p < 0) continue;
        for (int c = 0; c < 3; ++c) hex[c] += (double)wex[6 * i + f] * ((double)mb[3 * p + c] - (double)mi[c]);
      }
      for (int c = 0; c < 3; ++c) hex[c] *= (double)xsc[b];
    }
    const double me = (double)mi[0] * axis[3 * i] + (double)mi[1] * axis[3 * i + 1] + (double)mi[2] * axis[3 * i + 2];
    for (int c = 0; c < 3; ++c) han[c] = (double)kan[i] * me * axis[3 * i + c];
    const double w = MT_MU0 * (double)Ms[i] * wvol[i] * vol_total;
    for (int c = 0; c < 3; ++c) {
      e[0] += -w * mi[c] * (double)Ha[3 * b + c];
      e[1] += -0.5 * w * mi[c] * (double)Hd[o + c];
      e[2] += -0.5 * w * mi[c] * hex[c];
      e[3] += -0.5 * w * mi[c] * han[c];
    }
  }
  __shared__ double sh[8][4];
  for (int q = 0; q < 4; ++q) e[q] = mtd::warp_sum(e[q]);
  const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
  if (lane == 0)
    for (int q = 0; q < 4; ++q) sh[wq][q] = e[q];
  __syncthreads();
  if (threadIdx.x < 4) {
    double acc = 0;
    for (int ww = 0; ww < (int)(blockDim.x >> 5); ++ww) acc += sh[ww][threadIdx.x];
    atomicAdd(&E[4 * b + threadIdx.x], acc);
  }
}

// Standalone right-hand side: dmdt and per-simulation max torque.  The
// simulations' parameters travel with the launch, kRhsSims at a time: a call
// allocates nothing and copies nothing from the host (film of 2,500 tiles, one
// simulation: 60.8 -> 46.5 us for the call; with a device block of its own and
// four copies the host was what it waited for).
constexpr int kRhsSims = 64;
struct RhsParams {
  float g1[kRhsSims], g2[kRhsSims], Ha[3 * kRhsSims], xsc[kRhsSims];
};
__global__ void k_rhs_plain(int64_t n, const int32_t *nbr, const float *wex, const float *kan, const float *axis,
                            const float *Ms, bool exch, const float *m, const float *Hd,
                            const __grid_constant__ RhsParams P, float *dmdt, float *tau) {
  mtd::pdl_enter();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int b = blockIdx.y;
  const unsigned inside = __ballot_sync(~0u, i < n);
  if (i >= n) return;
  StageArgs A{};
  A.n = n;
  A.nbr = nbr;
  A.wex = wex;
  A.kan = kan;
  A.axis = axis;
  A.exch = exch;
  A.Ha = P.Ha;
  A.xsc = P.xsc;
  const size_t o = (size_t)b * 3 * n + 3 * i;
  const float mi[3] = {m[o], m[o + 1], m[o + 2]};
  float H[3], k[3];
  effective_field(A, m, Hd, i, b, mi, H);
  const float t = llg(P.g1[b], P.g2[b], mi, H, k) / Ms[i];
  dmdt[o] = k[0];
  dmdt[o + 1] = k[1];
  dmdt[o + 2] = k[2];
  if (tau) {  // t >= 0: its bits order as integers; one atomic for a warp
    const int top = __reduce_max_sync(inside, __float_as_int(t));
    if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<int *>(tau + b), top);
  }
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
namespace mt {

void launch_rhs_plain(const mt_tensor *T, const float *m, const float *Hd, int B, const float *g1,
                      const float *g2, const float *Ha, const float *xsc, float *dmdt, float *tau, cudaStream_t s) {
  const mt_tiles *t = T->tiles;
  for (int b0 = 0; b0 < B; b0 += kRhsSims) {
    const int nb = std::min(B - b0, kRhsSims);
    RhsParams P = {};
    std::copy_n(g1 + b0, nb, P.g1);
    std::copy_n(g2 + b0, nb, P.g2);
    std::copy_n(Ha + 3 * b0, 3 * nb, P.Ha);
    std::copy_n(xsc + b0, nb, P.xsc);
    const size_t o = (size_t)b0 * 3 * T->n;
    mt::launch_pdl(k_rhs_plain, dim3((unsigned)((T->n + 255) / 256), (unsigned)nb), dim3(256), 0, s, T->n,
                   (const int32_t *)t->d_nbr, (const float *)t->d_wex, (const float *)t->d_kan,
                   (const float *)t->d_axis, (const float *)t->d_Ms, t->has_exchange, m + o, Hd + o, P, dmdt + o,
                   tau ? tau + b0 : tau);
  }
}

void launch_energy(const mt_tensor *T, const float *m, const float *Hd, int B, const float *Ha, const float *xsc,
                   double *E, cudaStream_t s) {
  const mt_tiles *t = T->tiles;
  dim3 grid((unsigned)((T->n + 255) / 256), (unsigned)B);
  k_energy<<<grid, 256, 0, s>>>(T->n, t->d_nbr, t->d_wex, t->d_kan, t->d_axis, t->d_Ms, t->d_wvol, t->vol_total,
                                t->has_exchange, m, Hd, Ha, xsc, E);
}

void llg_prefactors(const mt_llg_params *p, int B, std::vector<float> &g1, std::vector<float> &g2,
                    std::vector<float> &ha, std::vector<float> &xsc) {
  g1.resize(B);
  g2.resize(B);
  ha.resize(3 * B);
  xsc.resize(B);
  for (int b = 0; b < B; ++b) {
    const double a = p->alpha[b];
    double G1, G2;
    if (p->form == MT_FORM_GILBERT) {
      G1 = p->gamma / (1.0 + a * a);
      G2 = G1 * a;
    } else {
      G1 = p->gamma;
      G2 = a;
    }
    if (!p->precess) G1 = 0.0;
    g1[b] = (float)G1;
    g2[b] = (float)G2;
    for (int c = 0; c < 3; ++c) ha[3 * b + c] = (float)p->Ha[3 * b + c];
    xsc[b] = p->exch_scale ? (float)p->exch_scale[b] : 1.0f;
  }
}

}  // namespace mt

struct mt_integrator {
  mt_tensor *T = nullptr;
  int B = 0;
  cudaStream_t stream = nullptr;       // private non-blocking stream: capture and replay
  cudaStream_t user_stream = nullptr;  // the caller's stream, ordered against `stream` by events
  cudaEvent_t order_ev = nullptr;
  mt_ode_opts o{};
  int form = 0, precess = 1;
  double gamma = 0;
  // device state
  float *y = nullptr, *ys0 = nullptr, *ys1 = nullptr, *Hd = nullptr, *xs = nullptr;
  float *k[7] = {};
  float *g1 = nullptr, *g2 = nullptr, *Ha = nullptr, *xsc = nullptr;
  float *part = nullptr;
  float *colpart = nullptr;  // half-stored tensor: column work area of the product
  int *count = nullptr;
  SimCtl *ctl = nullptr;
  int *active = nullptr;
  int *n_active = nullptr;
  float *red = nullptr;
  int *red_count = nullptr;
  double *mavg = nullptr;
  int64_t mavg_cap = 0;
  int *h_poll = nullptr;  // pinned, 2 slots
  float *h_slot_par = nullptr;  // pinned staging of per-slot parameters (g1, g2, Ha) for admissions
  cudaEvent_t ev[2] = {nullptr, nullptr};
  cudaGraphExec_t exec = nullptr;
  GemmPlan plan;  // dense layout: tensor maps of the batched product
  int nblk = 0;
  bool need_init = true;
  std::vector<void *> allocs;
  // small tile sets: the whole call in one cooperative kernel (k_small_run)
  int path = MT_PATH_GRAPH;  // the one in use
  bool small_ok = false;     // the tile set and batch fit it
  int small_G = 0, small_R = 0, small_rmax = 0, small_group = 1, small_lanes = kSmallThreads;
  bool small_many = false;  // its form for several simulations
  bool small_nsmem = true;  // tensor rows in shared memory (else read from L2)
  size_t small_smem_bytes = 0;
  unsigned char *sm_words = nullptr;  // words its CTAs exchange, then the abort flag (SmallWords)
};

namespace {

StageArgs stage_args(mt_integrator *I) {
  const mt_tensor *T = I->T;
  const mt_tiles *t = T->tiles;
  StageArgs A{};
  A.n = T->n;
  A.B = I->B;
  A.nbr = t->d_nbr;
  A.wex = t->d_wex;
  A.kan = t->d_kan;
  A.axis = t->d_axis;
  A.Ms = t->d_Ms;
  A.wvol = t->d_wvol;
  A.exch = t->has_exchange;
  A.g1 = I->g1;
  A.g2 = I->g2;
  A.Ha = I->Ha;
  A.xsc = I->xsc;
  A.y = I->y;
  A.ys0 = I->ys0;
  A.ys1 = I->ys1;
  A.Hd = I->Hd;
  A.xs = I->xs;
  for (int s = 0; s < 7; ++s) A.k[s] = I->k[s];
  A.Q = T->L.Q;
  A.TC = T->L.TC;
  A.xs_mode = T->layout == MT_LAYOUT_DENSE ? (T->prec == MT_BF16_SPLIT ? 2 : 1) : T->layout == MT_LAYOUT_SPARSE ? 3 : 0;
  A.Kp = T->Kp;
  A.Bp = mt::dense_pad_batch(I->B);
  A.X = reinterpret_cast<__nv_bfloat16 *>(I->xs);
  A.mT = T->layout == MT_LAYOUT_DENSE ? mt::dense_mT(T, I->B, I->xs) : nullptr;
  A.ctl = I->ctl;
  A.active = I->active;
  A.n_active = I->n_active;
  A.red = I->red;
  A.red_count = I->red_count;
  A.mavg = I->mavg;
  A.rtol = I->o.rtol;
  A.atol = I->o.atol;
  A.hmax = I->o.hmax;
  A.fixed_h = I->o.fixed_h;
  return A;
}

constexpr size_t kSmallSmemMax = 225 * 1024;  // of the 227 KB a CTA may opt in to
constexpr int kSmallSmemLimit = 227 * 1024;

using SmallKernel = void (*)(SmallArgs);
template <bool PLANAR, bool MANY>
SmallKernel small_kernel_of(int rmax) {
  return rmax == 2   ? k_small_run<2, true, PLANAR, MANY>
         : rmax == 4 ? k_small_run<4, true, PLANAR, MANY>
                     : k_small_run<8, true, PLANAR, MANY>;
}
SmallKernel small_kernel(const mt_tensor *T, bool nsmem, int rmax, bool many) {
  const bool planar = T->L.nplane == 4;
  if (!nsmem) return planar ? k_small_run<2, false, true, false> : k_small_run<2, false, false, false>;
  if (many) return planar ? small_kernel_of<true, true>(rmax) : small_kernel_of<false, true>(rmax);
  return planar ? small_kernel_of<true, false>(rmax) : small_kernel_of<false, false>(rmax);
}

// byte offsets of the exchanged words of k_small_run
struct SmallWords {
  size_t xg, kx, yx, part, abort_flag, total;
};
SmallWords small_words(int64_t n, int B, int G) {
  SmallWords w;
  const size_t vecs = sizeof(TagVec) * (size_t)B * n;
  w.xg = 0;
  w.kx = w.xg + 2 * vecs;
  w.yx = w.kx + 2 * vecs;
  w.part = w.yx + vecs;
  w.abort_flag = w.part + sizeof(TagSum) * (size_t)G * B;
  w.total = w.abort_flag + 128;
  return w;
}

// a tensor the one-kernel path reads from L2 every right-hand side must
// stay there (L2: 129 MB)
constexpr size_t kSmallL2Bytes = 96ull << 20;

// The bound on tile sets and batches of the one-kernel path, in bytes per CTA:
// the state of all tiles, 28 floats per row and simulation, 17 per row, the
// rows of the tensor (six planes) and 43 words and a control block per
// simulation, within 225 KB.  It is a rule of its own, wider than what the
// kernel takes, so that a tile set's path does not change with the kernel; near
// it the path has lost its lead (1,800 tiles, per attempt: 4 simulations 98 us
// against 117 of the step graph, 8 simulations 187 and 170).
size_t small_bound(int64_t n, int B, int R, bool nsmem) {
  size_t o = 0;
  small_take(o, sizeof(SimCtl) * B);
  for (const int64_t words : {(int64_t)kSmallRed, (int64_t)3 * B * R, (int64_t)21 * B * R, (int64_t)36 * B, (int64_t)6 * B,
                              (int64_t)B, n, (int64_t)3 * B * n, nsmem ? 6 * R * n : 0, (int64_t)3 * B * R,
                              (int64_t)B * R, (int64_t)6 * R, (int64_t)6 * R, (int64_t)R, (int64_t)3 * R, (int64_t)R})
    small_take(o, sizeof(float) * words);
  return o;
}

// Does the one-kernel path fit this tile set and batch?  An FP32 streaming
// tensor; one CTA per SM (or per tile) and a co-resident grid; either at
// most 8 rows per CTA whose tensor rows and the state of all tiles fit the
// shared memory, or at most 16 rows per CTA read from an L2-resident tensor
// with the state in shared memory.
bool small_plan(mt_integrator *I) {
  const mt_tensor *T = I->T;
  if (T->prec != MT_F32 || T->layout != MT_LAYOUT_STREAM || T->L.half) return false;
  const int64_t n = T->n;
  const int sms = T->tiles->ctx->num_sms;
  if (n < 1 || sms < 1) return false;
  const int64_t r_sm = (n + sms - 1) / sms;
  for (int pass = 0; pass < 2; ++pass) {
    const bool nsmem = pass == 0;
    // rows per CTA: enough to cover the tiles with one CTA per SM (fewer
    // CTAs meeting at each barrier measured no faster)
    const int R = (int)r_sm;
    if (R > (nsmem ? 8 : 2 * kSmallWarps)) continue;
    if (!nsmem && (T->bytes > kSmallL2Bytes || T->L.TC % 4 != 0)) continue;
    size_t bytes = small_smem(n, I->B, R, nsmem, 1).total;
    if (small_bound(n, I->B, R, nsmem) > kSmallSmemMax || bytes > (size_t)kSmallSmemLimit) continue;
    // Several simulations: `group` of them (as many as fit) between two CTA
    // barriers, one to a warp, and the threads divided among as many as keep
    // the poll of one a single round of four vectors per thread.  One after
    // the other, a barrier, a round trip and a chain each, 16 simulations of
    // 10 tiles took 114 us per attempt, so 46; 16 of 400 tiles 149, so 100
    // (one simulation: 12 and 20).  Three and four go two at a time: all at
    // once, the polls of 100 to 150 CTAs with a row each get in the way of
    // the stores (150 tiles, 4: 38 us against 29).  Two, and three whose poll
    // takes more than a round, are as fast one after the other (400 tiles, 2:
    // 23 us against 27; 1,000 tiles, 3: 46 and 47).
    const bool many = nsmem && (I->B >= 4 || (I->B == 3 && n <= 4 * kSmallThreads / 2));
    const int at_once = I->B <= 4 ? 2 : kSmallWarps;
    int group = 1, lanes = kSmallThreads;
    while (many && group < at_once && small_smem(n, I->B, R, nsmem, 2 * group).total <= kSmallSmemMax) group *= 2;
    while (many && kSmallThreads / lanes < (at_once == 2 ? 2 : I->B) && lanes > 1 && n <= 4 * (lanes / 2)) lanes /= 2;
    bytes = small_smem(n, I->B, R, nsmem, group).total;
    const int G = (int)((n + R - 1) / R);
    const int rmax = !nsmem ? 2 : R <= 2 ? 2 : R <= 4 ? 4 : 8;
    int per_sm = 0;
    const SmallKernel kern = small_kernel(T, nsmem, rmax, many);
    // the limit is the kernel's, for every integrator that uses it: a later and
    // smaller one must not lower it
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmallSmemLimit);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kSmallThreads, bytes);
    if (e != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    if (per_sm < 1 || (int64_t)per_sm * sms < G) continue;
    I->small_G = G;
    I->small_R = R;
    I->small_rmax = rmax;
    I->small_nsmem = nsmem;
    I->small_many = many;
    I->small_group = group;
    I->small_lanes = lanes;
    I->small_smem_bytes = bytes;
    return true;
  }
  return false;
}

mt_status launch_small(mt_integrator *I, int init, int64_t iters) {
  const mt_tensor *T = I->T;
  SmallArgs S{};
  S.A = stage_args(I);
  S.N = static_cast<const float *>(T->d_data);
  S.TR = T->L.TR;
  S.TC = T->L.TC;
  S.Q = T->L.Q;
  const SmallWords w = small_words(T->n, I->B, I->small_G);
  S.xg = reinterpret_cast<TagVec *>(I->sm_words + w.xg);
  S.kx = reinterpret_cast<TagVec *>(I->sm_words + w.kx);
  S.yx = reinterpret_cast<TagVec *>(I->sm_words + w.yx);
  S.part = reinterpret_cast<TagSum *>(I->sm_words + w.part);
  S.abort_flag = reinterpret_cast<int *>(I->sm_words + w.abort_flag);
  S.status = T->tiles->ctx->d_status;
  S.iters = iters;
  S.init = init;
  S.R = I->small_R;
  S.group = I->small_group;
  S.lanes = I->small_lanes;
  MT_CUDA(cudaMemsetAsync(I->sm_words, 0, w.total, I->stream));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)I->small_G);
  cfg.blockDim = dim3(kSmallThreads);
  cfg.dynamicSmemBytes = I->small_smem_bytes;
  cfg.stream = I->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  // after the context's previous one-kernel launch, whatever its stream: two
  // such grids resident together could each hold SMs the other waits for
  mt_ctx *ctx = T->tiles->ctx;
  std::lock_guard<std::mutex> lock(ctx->small_mu);
  cudaError_t e = cudaSuccess;
  if (!ctx->small_ev) e = cudaEventCreateWithFlags(&ctx->small_ev, cudaEventDisableTiming);
  else e = cudaStreamWaitEvent(I->stream, ctx->small_ev, 0);
  if (e == cudaSuccess) {
    e = cudaLaunchKernelEx(&cfg, small_kernel(T, I->small_nsmem, I->small_rmax, I->small_many), S);
  }
  if (e == cudaSuccess) e = cudaEventRecord(ctx->small_ev, I->stream);
  if (e != cudaSuccess) return mt::cuda_fail(e, "k_small_run launch", __FILE__, __LINE__);
  I->need_init = false;
  return MT_OK;
}

template <int S>
void launch_stage(mt_integrator *I, const StageArgs &A) {
  dim3 grid((unsigned)I->nblk, (unsigned)I->B);
  mt::launch_pdl(k_stage<S>, grid, dim3(kStageThreads), 0, I->stream, A);
}

// demag product of the stage input `m` into I->Hd (xs already formed)
void demag(mt_integrator *I, const float *m) {
  if (I->T->layout == MT_LAYOUT_SPARSE) {
    mt::launch_spmv(I->T, I->xs, I->B, I->Hd, I->active, I->stream);
    return;
  }
  if (I->T->layout == MT_LAYOUT_DENSE) {
    mt::launch_gemm(I->T, I->plan, I->Hd, I->part, I->count, I->n_active, I->T->tiles->ctx->d_status, I->stream);
    mt::launch_near(I->T, mt::dense_mT(I->T, I->B, I->xs), 1, mt::dense_pad_batch(I->B), I->B, I->Hd, I->active,
                    I->stream);
  } else {
    mt::launch_matvec(I->T, I->xs, I->B, I->Hd, I->part, I->count, I->active, I->T->tiles->ctx->d_status,
                      I->stream, I->colpart);
    mt::launch_near(I->T, m, 3 * I->T->n, 1, I->B, I->Hd, I->active, I->stream);
  }
}

void enqueue_attempt(mt_integrator *I) {
  StageArgs A = stage_args(I);
  dim3 grid((unsigned)I->nblk, (unsigned)I->B);
  mt::launch_pdl(k_begin, grid, dim3(kStageThreads), 0, I->stream, A);
  demag(I, I->ys0);
  launch_stage<2>(I, A);
  demag(I, I->ys1);
  launch_stage<3>(I, A);
  demag(I, I->ys0);
  launch_stage<4>(I, A);
  demag(I, I->ys1);
  launch_stage<5>(I, A);
  demag(I, I->ys0);
  launch_stage<6>(I, A);
  demag(I, I->ys1);
  launch_stage<7>(I, A);
}

mt_status enqueue_init(mt_integrator *I, int fresh_only = 0) {
  StageArgs A = stage_args(I);
  A.fresh_only = fresh_only;
  if (I->T->layout == MT_LAYOUT_DENSE)
    mt::launch_prep_dense_x(I->T, I->y, I->B, I->xs, I->stream);
  else
    mt::launch_prep_xs(I->T, I->y, I->B, I->xs, I->stream);
  demag(I, I->y);
  launch_stage<1>(I, A);
  MT_CUDA(cudaGetLastError());
  I->need_init = false;
  return MT_OK;
}

mt_status enqueue_commit(mt_integrator *I) {
  StageArgs A = stage_args(I);
  dim3 grid((unsigned)I->nblk, (unsigned)I->B);
  k_commit<<<grid, kStageThreads, 0, I->stream>>>(A);
  MT_CUDA(cudaGetLastError());
  return MT_OK;
}

template <typename P>
mt_status dalloc(mt_integrator *I, P **p, size_t bytes) {
  MT_CUDA(cudaMalloc((void **)p, bytes));
  MT_CUDA(cudaMemsetAsync(*p, 0, bytes, I->stream));
  I->allocs.push_back((void *)*p);
  return MT_OK;
}

mt_status read_ctl(mt_integrator *I, std::vector<SimCtl> &c) {
  c.resize(I->B);
  MT_CUDA(cudaMemcpyAsync(c.data(), I->ctl, sizeof(SimCtl) * I->B, cudaMemcpyDeviceToHost, I->stream));
  MT_CUDA(cudaStreamSynchronize(I->stream));
  return MT_OK;
}

mt_status write_ctl(mt_integrator *I, const std::vector<SimCtl> &c) {
  std::vector<int> act(I->B);
  int na = 0;
  for (int b = 0; b < I->B; ++b) {
    act[b] = c[b].done ? 0 : 1;
    na += act[b];
  }
  MT_CUDA(cudaMemcpyAsync(I->ctl, c.data(), sizeof(SimCtl) * I->B, cudaMemcpyHostToDevice, I->stream));
  MT_CUDA(cudaMemcpyAsync(I->active, act.data(), sizeof(int) * I->B, cudaMemcpyHostToDevice, I->stream));
  MT_CUDA(cudaMemcpyAsync(I->n_active, &na, sizeof(int), cudaMemcpyHostToDevice, I->stream));
  MT_CUDA(cudaStreamSynchronize(I->stream));  // host vectors go out of scope
  return MT_OK;
}

void fill_stats(const std::vector<SimCtl> &c, mt_stats *st, int B) {
  if (!st) return;
  for (int b = 0; b < B; ++b) {
    st[b].n_accept = c[b].n_accept;
    st[b].n_reject = c[b].n_reject;
    st[b].n_rhs = c[b].n_rhs;
    st[b].t = c[b].t;
    st[b].h = c[b].h;
    st[b].tau = c[b].tau;
    st[b].status = c[b].status;
    st[b].pad = 0;
  }
}

void plan_host(const mt_integrator *I, SimCtl &c) {
  double hs = c.h;
  if (I->o.fixed_h <= 0.0 && I->o.hmax > 0.0 && hs > I->o.hmax) hs = I->o.hmax;
  c.clipped = 0;
  if (c.t + hs >= c.t_next) {
    hs = c.t_next - c.t;
    c.clipped = 1;
  }
  c.hs = hs;
}

// The one-kernel path in launches of at most kSmallChunk attempts, so that
// no launch runs for long; between them the host reads the number of
// unfinished simulations (and stops on a device timeout).
constexpr int64_t kSmallChunk = 4096;
static_assert(6 * kSmallChunk + 1 < 1 << 15, "exchange tags of one launch");

mt_status small_steps(mt_integrator *I, int init, int64_t nsteps) {
  for (int64_t done = 0; done < nsteps || init;) {
    const int64_t todo = std::min<int64_t>(kSmallChunk, nsteps - done);
    mt_status st = launch_small(I, init, todo);
    if (st != MT_OK) return st;
    init = 0;
    done += todo;
  }
  return MT_OK;
}

mt_status small_until_done(mt_integrator *I, int64_t max_attempts) {
  int init = 1;
  for (int64_t done = 0;;) {
    const int64_t todo = std::min<int64_t>(kSmallChunk, max_attempts - done);
    mt_status st = launch_small(I, init, todo);
    if (st != MT_OK) return st;
    init = 0;
    done += todo;
    int h[2] = {0, 0};
    MT_CUDA(cudaMemcpyAsync(&h[0], I->n_active, sizeof(int), cudaMemcpyDeviceToHost, I->stream));
    MT_CUDA(cudaMemcpyAsync(&h[1], I->T->tiles->ctx->d_status, sizeof(int), cudaMemcpyDeviceToHost, I->stream));
    MT_CUDA(cudaStreamSynchronize(I->stream));
    if (h[0] == 0 || h[1] != 0 || done >= max_attempts) return MT_OK;
  }
}

// Replay the step graph until every simulation is finished (or a cap).
mt_status replay_until_done(mt_integrator *I, int64_t max_launches) {
  int64_t launched = 0;
  int chunk = 2;
  int slot = 0;
  bool pending[2] = {false, false};
  for (;;) {
    const int64_t todo = std::min<int64_t>(chunk, max_launches - launched);
    for (int64_t q = 0; q < todo; ++q) MT_CUDA(cudaGraphLaunch(I->exec, I->stream));
    launched += todo;
    MT_CUDA(cudaMemcpyAsync(&I->h_poll[slot], I->n_active, sizeof(int), cudaMemcpyDeviceToHost, I->stream));
    MT_CUDA(cudaEventRecord(I->ev[slot], I->stream));
    pending[slot] = true;
    const int prev = slot ^ 1;
    if (pending[prev]) {
      MT_CUDA(cudaEventSynchronize(I->ev[prev]));
      pending[prev] = false;
      if (I->h_poll[prev] == 0) break;
    }
    if (launched >= max_launches) {
      MT_CUDA(cudaEventSynchronize(I->ev[slot]));
      break;
    }
    slot = prev;
    if (chunk < 64) chunk *= 2;
  }
  MT_CUDA(cudaStreamSynchronize(I->stream));
  return MT_OK;
}

}  // namespace

// ---------------------------------------------------------------------------
// ABI
// ---------------------------------------------------------------------------
extern "C" {

mt_status mt_integrator_create(mt_tensor *T, const mt_llg_params *p, const mt_ode_opts *o, int B, void *stream,
                               mt_integrator **out) {
  MT_CHECK(T && p && o && out, MT_EINVAL, "mt_integrator_create: NULL argument");
  MT_CHECK(B >= 1 && B <= 4096, MT_EINVAL, "mt_integrator_create: B must be in [1, 4096]");
  MT_CHECK(T->prec != MT_F64, MT_EINVAL, "mt_integrator_create: the FP64 tensor serves field checks only");
  MT_CHECK(p->alpha && p->Ha, MT_EINVAL, "mt_integrator_create: alpha/Ha arrays required");
  MT_CHECK(o->fixed_h > 0.0 || (o->rtol > 0.0 && o->atol > 0.0 && o->h0 > 0.0), MT_EINVAL,
           "mt_integrator_create: rtol, atol and h0 must be positive");
  MT_CHECK(o->max_steps > 0, MT_EINVAL, "mt_integrator_create: max_steps must be positive");
  for (int b = 0; b < B; ++b)
    MT_CHECK(std::isfinite(p->alpha[b]) && std::isfinite(p->Ha[3 * b]) && std::isfinite(p->Ha[3 * b + 1]) &&
                 std::isfinite(p->Ha[3 * b + 2]),
             MT_EINVAL, "mt_integrator_create: non-finite parameter");
  MT_CUDA(cudaSetDevice(T->tiles->ctx->device));
  mt_integrator *I = new mt_integrator();
  I->T = T;
  T->refs++;
  I->B = B;
  I->user_stream = (cudaStream_t)stream;
  if (cudaStreamCreateWithFlags(&I->stream, cudaStreamNonBlocking) != cudaSuccess ||
      cudaEventCreateWithFlags(&I->order_ev, cudaEventDisableTiming) != cudaSuccess) {
    mt_integrator_destroy(I);
    mt::set_error("mt_integrator_create: stream/event creation failed");
    return MT_ECUDA;
  }
  I->o = *o;
  I->form = p->form;
  I->precess = p->precess;
  I->gamma = p->gamma;
  const int64_t n = T->n;
  const size_t vec = sizeof(float) * 3 * n * B;
  I->nblk = (int)((n + kStageThreads - 1) / kStageThreads);
  mt_status st = MT_OK;
#define MT_TRY(x)              \
  do {                         \
    if ((st = (x)) != MT_OK) { \
      mt_integrator_destroy(I); \
      return st;               \
    }                          \
  } while (0)
  MT_TRY(dalloc(I, &I->y, vec));
  MT_TRY(dalloc(I, &I->ys0, vec));
  MT_TRY(dalloc(I, &I->ys1, vec));
  MT_TRY(dalloc(I, &I->Hd, vec));
  for (int s = 0; s < 7; ++s) MT_TRY(dalloc(I, &I->k[s], vec));
  const bool dense = T->layout == MT_LAYOUT_DENSE;
  if (dense) {
    MT_TRY(dalloc(I, (unsigned char **)&I->xs, mt::dense_x_bytes(T, B)));
    MT_TRY(mt::gemm_plan(T, B, I->xs, &I->plan));
  } else {
    MT_TRY(dalloc(I, &I->xs, sizeof(float) * mt::xs_floats(T) * B));
  }
  MT_TRY(dalloc(I, &I->g1, sizeof(float) * B));
  MT_TRY(dalloc(I, &I->g2, sizeof(float) * B));
  MT_TRY(dalloc(I, &I->Ha, sizeof(float) * 3 * B));
  MT_TRY(dalloc(I, &I->xsc, sizeof(float) * B));
  MT_TRY(dalloc(I, &I->part, dense ? mt::dense_part_bytes(T, B) : mt::matvec_part_bytes(T)));
  MT_TRY(dalloc(I, &I->count, dense ? mt::dense_count_bytes(T) : mt::matvec_count_bytes(T, B)));
  if (!dense && T->L.half) MT_TRY(dalloc(I, &I->colpart, mt::matvec_colpart_bytes(T, B)));
  MT_TRY(dalloc(I, &I->ctl, sizeof(SimCtl) * B));
  MT_TRY(dalloc(I, &I->active, sizeof(int) * B));
  MT_TRY(dalloc(I, &I->n_active, sizeof(int)));
  MT_TRY(dalloc(I, &I->red, sizeof(float) * 5 * I->nblk * B));
  MT_TRY(dalloc(I, &I->red_count, sizeof(int) * B));
  I->mavg_cap = 1;
  MT_TRY(dalloc(I, &I->mavg, sizeof(double) * 3 * B));
  I->small_ok = small_plan(I);
  if (I->small_ok) {
    MT_TRY(dalloc(I, &I->sm_words, small_words(n, B, I->small_G).total));
    I->path = MT_PATH_PERSISTENT;
  }
  if (cudaMallocHost(&I->h_poll, 2 * sizeof(int)) != cudaSuccess) {
    mt_integrator_destroy(I);
    mt::set_error("mt_integrator_create: pinned allocation failed");
    return MT_ENOMEM;
  }
  if (cudaEventCreateWithFlags(&I->ev[0], cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&I->ev[1], cudaEventDisableTiming) != cudaSuccess) {
    mt_integrator_destroy(I);
    mt::set_error("mt_integrator_create: event creation failed");
    return MT_ECUDA;
  }
  MT_TRY(mt_integrator_set_params(I, p));
  if (dense) MT_TRY(mt::gemm_tune(T, &I->plan, I->Hd, I->part, I->count, T->tiles->ctx->d_status, I->stream));
  // capture one attempt
  cudaGraph_t g = nullptr;
  cudaError_t e = cudaStreamBeginCapture(I->stream, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    enqueue_attempt(I);
    e = cudaStreamEndCapture(I->stream, &g);
  }
  if (e == cudaSuccess) e = cudaGraphInstantiate(&I->exec, g, 0);
  if (g) cudaGraphDestroy(g);
  if (e != cudaSuccess) {
    mt_integrator_destroy(I);
    return mt::cuda_fail(e, "graph capture", __FILE__, __LINE__);
  }
#undef MT_TRY
  *out = I;
  return MT_OK;
}

void mt_integrator_destroy(mt_integrator *I) {
  if (!I) return;
  if (I->stream) cudaStreamSynchronize(I->stream);
  if (I->exec) cudaGraphExecDestroy(I->exec);
  for (void *p : I->allocs) cudaFree(p);
  if (I->h_poll) cudaFreeHost(I->h_poll);
  if (I->h_slot_par) cudaFreeHost(I->h_slot_par);
  for (auto &e : I->ev)
    if (e) cudaEventDestroy(e);
  if (I->order_ev) cudaEventDestroy(I->order_ev);
  if (I->stream) cudaStreamDestroy(I->stream);
  mt::tensor_release(I->T);
  delete I;
}

mt_status mt_integrator_set_params(mt_integrator *I, const mt_llg_params *p) {
  MT_CHECK(I && p && p->alpha && p->Ha, MT_EINVAL, "mt_integrator_set_params: NULL argument");
  std::vector<float> g1, g2, ha, xsc;
  mt::llg_prefactors(p, I->B, g1, g2, ha, xsc);
  for (int b = 0; b < I->B; ++b)
    MT_CHECK(std::isfinite(xsc[b]) && xsc[b] >= 0.0f, MT_EINVAL, "mt_integrator_set_params: bad exch_scale");
  MT_CUDA(cudaMemcpyAsync(I->g1, g1.data(), sizeof(float) * I->B, cudaMemcpyHostToDevice, I->stream));
  MT_CUDA(cudaMemcpyAsync(I->g2, g2.data(), sizeof(float) * I->B, cudaMemcpyHostToDevice, I->stream));
  MT_CUDA(cudaMemcpyAsync(I->Ha, ha.data(), sizeof(float) * 3 * I->B, cudaMemcpyHostToDevice, I->stream));
  MT_CUDA(cudaMemcpyAsync(I->xsc, xsc.data(), sizeof(float) * I->B, cudaMemcpyHostToDevice, I->stream));
  MT_CUDA(cudaStreamSynchronize(I->stream));
  I->need_init = true;
  return MT_OK;
}

mt_status mt_integrator_set_state(mt_integrator *I, const float *m, int m_is_host, double t0) {
  MT_CHECK(I && m, MT_EINVAL, "mt_integrator_set_state: NULL argument");
  const size_t bytes = sizeof(float) * 3 * I->T->n * I->B;
  if (!m_is_host) {  // the caller's stream may still be writing m
    MT_CUDA(cudaEventRecord(I->order_ev, I->user_stream));
    MT_CUDA(cudaStreamWaitEvent(I->stream, I->order_ev, 0));
  }
  MT_CUDA(cudaMemcpyAsync(I->y, m, bytes, m_is_host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice,
                          I->stream));
  std::vector<SimCtl> c(I->B);
  for (auto &x : c) {
    std::memset(&x, 0, sizeof(SimCtl));
    x.t = t0;
    x.h = I->o.fixed_h > 0 ? I->o.fixed_h : I->o.h0;
    x.t_next = 1e300;
    x.mode = MODE_STEPS;
    x.status = MT_OK;
    x.attempt_cap = INT64_MAX;
  }
  for (auto &x : c) plan_host(I, x);
  // write_ctl synchronises, which also orders the state copy
  mt_status st = write_ctl(I, c);
  if (st != MT_OK) return st;
  I->need_init = true;
  return MT_OK;
}

mt_status mt_integrator_get_state(mt_integrator *I, float *m, int m_is_host) {
  MT_CHECK(I && m, MT_EINVAL, "mt_integrator_get_state: NULL argument");
  const size_t bytes = sizeof(float) * 3 * I->T->n * I->B;
  MT_CUDA(cudaMemcpyAsync(m, I->y, bytes, m_is_host ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice,
                          I->stream));
  if (m_is_host) {
    MT_CUDA(cudaStreamSynchronize(I->stream));
  } else {  // later work on the caller's stream sees the copy
    MT_CUDA(cudaEventRecord(I->order_ev, I->stream));
    MT_CUDA(cudaStreamWaitEvent(I->user_stream, I->order_ev, 0));
  }
  return MT_OK;
}

void *mt_integrator_stream(mt_integrator *I) { return I ? (void *)I->stream : nullptr; }

mt_status mt_integrator_set_path(mt_integrator *I, int path) {
  MT_CHECK(I, MT_EINVAL, "mt_integrator_set_path: NULL integrator");
  MT_CHECK(path == MT_PATH_GRAPH || path == MT_PATH_PERSISTENT, MT_EINVAL, "mt_integrator_set_path: unknown path %d",
           path);
  MT_CHECK(path == MT_PATH_GRAPH || I->small_ok, MT_EINVAL,
           "mt_integrator_set_path: the one-kernel path needs an FP32 streaming tensor of a small tile set");
  // both paths leave the state committed between calls (y and k1 current)
  MT_CUDA(cudaStreamSynchronize(I->stream));
  I->path = path;
  return MT_OK;
}

int mt_integrator_get_path(mt_integrator *I) { return I ? I->path : 0; }

mt_status mt_selftest_grid_barrier_timeout(mt_ctx *ctx) {
  MT_CHECK(ctx, MT_EINVAL, "mt_selftest_grid_barrier_timeout: NULL context");
  MT_CUDA(cudaSetDevice(ctx->device));
  // 4 tagged vectors, the abort flag, a status word
  unsigned char *words = nullptr;
  MT_CUDA(cudaMalloc(&words, 256));
  cudaError_t e = cudaMemset(words, 0, 256);
  SmallArgs S{};
  S.xg = reinterpret_cast<TagVec *>(words);
  S.abort_flag = reinterpret_cast<int *>(words + 128);
  S.status = reinterpret_cast<int *>(words + 192);
  if (e == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(4);
    cfg.blockDim = dim3(32);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, k_exchange_selftest, S);
  }
  int h = 0;
  if (e == cudaSuccess) e = cudaMemcpy(&h, S.status, sizeof(int), cudaMemcpyDeviceToHost);
  cudaFree(words);
  if (e != cudaSuccess) return mt::cuda_fail(e, "mt_selftest_grid_barrier_timeout", __FILE__, __LINE__);
  if (h == MT_DEV_TIMEOUT) {
    mt::set_error("mt_selftest_grid_barrier_timeout: the bounded wait gave up as designed");
    return MT_ETIMEOUT;
  }
  mt::set_error("mt_selftest_grid_barrier_timeout: the wait did not report a timeout");
  return MT_ECUDA;
}

mt_status mt_integrator_step(mt_integrator *I, int64_t nsteps) {
  MT_CHECK(I && nsteps >= 0, MT_EINVAL, "mt_integrator_step: bad argument");
  if (I->need_init) {
    // fixed number of attempts: no time target, every simulation active
    std::vector<SimCtl> c;
    mt_status st = read_ctl(I, c);
    if (st != MT_OK) return st;
    for (auto &x : c) {
      x.mode = MODE_STEPS;
      x.t_next = 1e300;
      x.done = 0;
      x.status = MT_OK;
      plan_host(I, x);
    }
    if ((st = write_ctl(I, c)) != MT_OK) return st;
    if (I->path == MT_PATH_PERSISTENT) return small_steps(I, 1, nsteps);
    if ((st = enqueue_init(I)) != MT_OK) return st;
  }
  if (I->path == MT_PATH_PERSISTENT) return small_steps(I, 0, nsteps);
  for (int64_t q = 0; q < nsteps; ++q) MT_CUDA(cudaGraphLaunch(I->exec, I->stream));
  return enqueue_commit(I);
}

// cap_ok: in relax mode a simulation that reached its time cap with the
// torque above tol counts as finished (hysteresis values)
static mt_status run_common(mt_integrator *I, int mode, double t1, int64_t n_out, double tol, double *mavg,
                            mt_stats *stats, bool cap_ok = false, std::vector<SimCtl> *out_ctl = nullptr) {
  std::vector<SimCtl> c;
  mt_status st = read_ctl(I, c);
  if (st != MT_OK) return st;
  if (mode == MODE_RUN && n_out > I->mavg_cap) {
    cudaFree(I->mavg);
    I->allocs.erase(std::remove(I->allocs.begin(), I->allocs.end(), (void *)I->mavg), I->allocs.end());
    I->mavg = nullptr;
    if ((st = dalloc(I, &I->mavg, sizeof(double) * 3 * I->B * n_out)) != MT_OK) return st;
    I->mavg_cap = n_out;
    // the graph bakes the output pointer in: recapture
    cudaGraphExecDestroy(I->exec);
    I->exec = nullptr;
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(I->stream, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
      enqueue_attempt(I);
      e = cudaStreamEndCapture(I->stream, &g);
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&I->exec, g, 0);
    if (g) cudaGraphDestroy(g);
    if (e != cudaSuccess) return mt::cuda_fail(e, "graph capture", __FILE__, __LINE__);
  }
  for (auto &x : c) {
    x.mode = mode;
    x.done = 0;
    x.status = MT_OK;
    x.accepted = 0;
    x.attempt_cap = x.n_attempt + I->o.max_steps;
    if (mode == MODE_RUN) {
      x.n_out = n_out;
      x.iout = 0;
      x.t1 = t1;
      x.t_out0 = x.t;
      x.dt_out = (t1 - x.t) / (double)n_out;
      x.t_next = (n_out == 1) ? t1 : x.t + x.dt_out;
    } else {
      x.tol = tol;
      x.t1 = x.t + t1;
      x.t_next = x.t1;
    }
    plan_host(I, x);
  }
  if ((st = write_ctl(I, c)) != MT_OK) return st;
  if (I->path == MT_PATH_PERSISTENT) {
    if ((st = small_until_done(I, I->o.max_steps + 2)) != MT_OK) return st;
  } else {
    if ((st = enqueue_init(I)) != MT_OK) return st;
    if ((st = replay_until_done(I, I->o.max_steps + 2)) != MT_OK) return st;
    if ((st = enqueue_commit(I)) != MT_OK) return st;
  }
  if ((st = read_ctl(I, c)) != MT_OK) return st;
  int dev_status = 0;
  MT_CUDA(cudaMemcpy(&dev_status, I->T->tiles->ctx->d_status, sizeof(int), cudaMemcpyDeviceToHost));
  MT_CHECK(dev_status == 0, MT_ETIMEOUT, "integrator: a bounded device wait ran out");
  if (mavg && mode == MODE_RUN) {
    MT_CUDA(cudaMemcpy(mavg, I->mavg, sizeof(double) * 3 * I->B * n_out, cudaMemcpyDeviceToHost));
  }
  fill_stats(c, stats, I->B);
  if (out_ctl) *out_ctl = c;
  for (int b = 0; b < I->B; ++b) {
    if (!c[b].done) {
      mt::set_error("integrator: simulation %d not finished", b);
      return MT_ENOCONV;
    }
    if (cap_ok && c[b].status == MT_ENOCONV && c[b].t >= c[b].t1) continue;
    if (c[b].status != MT_OK) {
      mt::set_error("integrator: simulation %d ended with status %d", b, c[b].status);
      return (mt_status)c[b].status;
    }
  }
  return MT_OK;
}

mt_status mt_integrator_run(mt_integrator *I, double t1, int64_t n_out, double *mavg, mt_stats *stats) {
  MT_CHECK(I && n_out >= 1, MT_EINVAL, "mt_integrator_run: bad argument");
  return run_common(I, MODE_RUN, t1, n_out, 0.0, mavg, stats);
}

mt_status mt_integrator_relax(mt_integrator *I, double tol, double t_max, mt_stats *stats) {
  MT_CHECK(I && tol > 0 && t_max > 0, MT_EINVAL, "mt_integrator_relax: bad argument");
  return run_common(I, MODE_RELAX, t_max, 1, tol, nullptr, stats);
}

mt_status mt_integrator_hysteresis(mt_integrator *I, const double *dir, const double *H, int64_t S, double t_step,
                                   double tol, double *mavg, double *tau, double *hc, double *mr, mt_stats *stats) {
  MT_CHECK(I && dir && H && S >= 1 && t_step > 0 && tol >= 0, MT_EINVAL, "mt_integrator_hysteresis: bad argument");
  const int B = I->B;
  std::vector<double> d(3 * B);
  for (int b = 0; b < B; ++b) {
    const double nrm = std::sqrt(dir[3 * b] * dir[3 * b] + dir[3 * b + 1] * dir[3 * b + 1] +
                                 dir[3 * b + 2] * dir[3 * b + 2]);
    MT_CHECK(std::isfinite(nrm) && nrm > 0, MT_EINVAL, "mt_integrator_hysteresis: direction %d is zero", b);
    for (int c = 0; c < 3; ++c) d[3 * b + c] = dir[3 * b + c] / nrm;
  }
  for (int64_t s = 0; s < S; ++s)
    MT_CHECK(std::isfinite(H[s]), MT_EINVAL, "mt_integrator_hysteresis: non-finite field value");
  std::vector<double> pm(3 * B * (size_t)S), pt(B * (size_t)S);
  std::vector<float> ha(3 * B);
  std::vector<SimCtl> c;
  mt_status st0 = read_ctl(I, c);
  if (st0 != MT_OK) return st0;
  double t_end = 0.0;  // fixed-time values: every simulation ends on the same times
  for (int b = 0; b < B; ++b) t_end = std::max(t_end, c[b].t);
  for (int64_t s = 0; s < S; ++s) {
    for (int q = 0; q < 3 * B; ++q) ha[q] = (float)(H[s] * d[q]);
    MT_CUDA(cudaMemcpyAsync(I->Ha, ha.data(), sizeof(float) * 3 * B, cudaMemcpyHostToDevice, I->stream));
    MT_CUDA(cudaStreamSynchronize(I->stream));
    I->need_init = true;  // k1 belongs to the previous field
    t_end += t_step;
    mt_status st = tol > 0 ? run_common(I, MODE_RELAX, t_step, 1, tol, nullptr, stats, true, &c)
                           : run_common(I, MODE_RUN, t_end, 1, 0.0, nullptr, stats, false, &c);
    if (st != MT_OK) return st;
    for (int b = 0; b < B; ++b) {
      for (int q = 0; q < 3; ++q) pm[((size_t)s * B + b) * 3 + q] = c[b].m_last[q];
      pt[(size_t)s * B + b] = c[b].tau;
    }
  }
  if (mavg) std::memcpy(mavg, pm.data(), sizeof(double) * pm.size());
  if (tau) std::memcpy(tau, pt.data(), sizeof(double) * pt.size());
  const double nan = std::numeric_limits<double>::quiet_NaN();
  for (int b = 0; b < B; ++b) {
    auto proj = [&](int64_t s) {
      const double *m = &pm[((size_t)s * B + b) * 3];
      return m[0] * d[3 * b] + m[1] * d[3 * b + 1] + m[2] * d[3 * b + 2];
    };
    if (hc) {
      hc[b] = nan;
      for (int64_t s = 1; s < S; ++s) {
        const double p0 = proj(s - 1), p1 = proj(s);
        if (p0 > 0 && p1 <= 0) {
          hc[b] = H[s - 1] + (H[s] - H[s - 1]) * p0 / (p0 - p1);
          break;
        }
      }
    }
    if (mr) {
      for (int q = 0; q < 3; ++q) mr[3 * b + q] = nan;
      for (int64_t s = 1; s < S; ++s) {
        if (H[s - 1] >= 0 && H[s] <= 0 && H[s - 1] != H[s]) {
          const double w = H[s - 1] / (H[s - 1] - H[s]);
          for (int q = 0; q < 3; ++q)
            mr[3 * b + q] = (1 - w) * pm[((size_t)(s - 1) * B + b) * 3 + q] + w * pm[((size_t)s * B + b) * 3 + q];
          break;
        }
      }
    }
  }
  return MT_OK;
}

mt_status mt_integrator_crossover(mt_integrator *I, const double *lam, int K, const float *mA, const float *mB,
                                  double tol, double t_max, double *eA, double *eB, double *lam_cross,
                                  float *m_out, mt_stats *stats) {
  MT_CHECK(I && lam && mA && mB && K >= 1 && tol > 0 && t_max > 0, MT_EINVAL,
           "mt_integrator_crossover: bad argument");
  MT_CHECK(I->B == 2 * K, MT_EINVAL, "mt_integrator_crossover: the integrator must hold 2K = %d simulations", 2 * K);
  for (int k = 0; k < K; ++k)
    MT_CHECK(std::isfinite(lam[k]) && lam[k] > 0, MT_EINVAL, "mt_integrator_crossover: sizes must be positive");
  const int64_t n = I->T->n;
  const int B = I->B;
  // sizes enter as exchange factors (the point tensor is scale-invariant)
  std::vector<float> xsc(B);
  for (int k = 0; k < K; ++k) xsc[k] = xsc[K + k] = (float)(1.0 / (lam[k] * lam[k]));
  MT_CUDA(cudaMemcpyAsync(I->xsc, xsc.data(), sizeof(float) * B, cudaMemcpyHostToDevice, I->stream));
  // state: family A at every size, then family B
  std::vector<float> m0((size_t)3 * n * B);
  for (int k = 0; k < K; ++k) {
    std::memcpy(&m0[(size_t)3 * n * k], mA, sizeof(float) * 3 * n);
    std::memcpy(&m0[(size_t)3 * n * (K + k)], mB, sizeof(float) * 3 * n);
  }
  mt_status st = mt_integrator_set_state(I, m0.data(), 1, 0.0);
  if (st != MT_OK) return st;
  if ((st = run_common(I, MODE_RELAX, t_max, 1, tol, nullptr, stats, true)) != MT_OK) return st;
  // energies of the relaxed states: demag product of y for every simulation
  // (finished ones are inactive after the relaxation), then the densities
  {
    std::vector<int> act(B, 1);
    MT_CUDA(cudaMemcpyAsync(I->active, act.data(), sizeof(int) * B, cudaMemcpyHostToDevice, I->stream));
    MT_CUDA(cudaMemcpyAsync(I->n_active, &B, sizeof(int), cudaMemcpyHostToDevice, I->stream));
    MT_CUDA(cudaStreamSynchronize(I->stream));
  }
  double *d_E = nullptr;
  MT_CUDA(cudaMalloc(&d_E, sizeof(double) * 4 * B));
  cudaError_t e = cudaMemsetAsync(d_E, 0, sizeof(double) * 4 * B, I->stream);
  if (e == cudaSuccess) {
    if (I->T->layout == MT_LAYOUT_DENSE)
      mt::launch_prep_dense_x(I->T, I->y, B, I->xs, I->stream);
    else
      mt::launch_prep_xs(I->T, I->y, B, I->xs, I->stream);
    demag(I, I->y);
    mt::launch_energy(I->T, I->y, I->Hd, B, I->Ha, I->xsc, d_E, I->stream);
    e = cudaGetLastError();
  }
  std::vector<double> e4(4 * B);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(e4.data(), d_E, sizeof(double) * 4 * B, cudaMemcpyDeviceToHost, I->stream);
  if (e == cudaSuccess && m_out)
    e = cudaMemcpyAsync(m_out, I->y, sizeof(float) * 3 * n * B, cudaMemcpyDeviceToHost, I->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(I->stream);
  cudaFree(d_E);
  if (e != cudaSuccess) return mt::cuda_fail(e, "mt_integrator_crossover", __FILE__, __LINE__);
  I->need_init = true;  // the workspace now holds the relaxed state's product
  const double vol = I->T->tiles->vol_total;
  std::vector<double> ea(K), eb(K);
  for (int k = 0; k < K; ++k) {
    ea[k] = (e4[4 * k] + e4[4 * k + 1] + e4[4 * k + 2] + e4[4 * k + 3]) / vol;
    eb[k] = (e4[4 * (K + k)] + e4[4 * (K + k) + 1] + e4[4 * (K + k) + 2] + e4[4 * (K + k) + 3]) / vol;
  }
  if (eA) std::memcpy(eA, ea.data(), sizeof(double) * K);
  if (eB) std::memcpy(eB, eb.data(), sizeof(double) * K);
  if (lam_cross) {
    *lam_cross = std::numeric_limits<double>::quiet_NaN();
    for (int k = 1; k < K; ++k) {
      const double d0 = ea[k - 1] - eb[k - 1], d1 = ea[k] - eb[k];
      if ((d0 < 0) != (d1 < 0)) {
        *lam_cross = lam[k - 1] + (lam[k] - lam[k - 1]) * d0 / (d0 - d1);
        break;
      }
    }
  }
  return MT_OK;
}

mt_status mt_integrator_stats(mt_integrator *I, mt_stats *stats) {
  MT_CHECK(I && stats, MT_EINVAL, "mt_integrator_stats: NULL argument");
  std::vector<SimCtl> c;
  mt_status st = read_ctl(I, c);
  if (st != MT_OK) return st;
  fill_stats(c, stats, I->B);
  return MT_OK;
}

// ---------------------------------------------------------------------------
// checkpoint / resume: header | SimCtl[B] | m[3nB] | k1[3nB] | FNV-1a 64
// ---------------------------------------------------------------------------
namespace {

struct CkptHeader {
  char magic[8];
  uint32_t version;
  uint32_t k1_valid;  // the saved derivative belongs to the saved m
  int64_t n;
  int32_t B;
  int32_t prec;
  int32_t layout;
  uint32_t ctl_bytes;  // sizeof(SimCtl) of the writer
};
constexpr char kCkptMagic[8] = {'M', 'T', 'C', 'K', 'P', 'T', '0', '1'};
constexpr uint32_t kCkptVersion = 1;

uint64_t fnv1a64(const unsigned char *p, size_t len) {
  uint64_t h = 1469598103934665603ull;
  for (size_t q = 0; q < len; ++q) {
    h ^= p[q];
    h *= 1099511628211ull;
  }
  return h;
}

size_t ckpt_bytes(const mt_integrator *I) {
  const size_t state = sizeof(float) * 3 * (size_t)I->T->n * I->B;
  return sizeof(CkptHeader) + sizeof(SimCtl) * I->B + 2 * state + sizeof(uint64_t);
}

}  // namespace

mt_status mt_integrator_checkpoint_bytes(mt_integrator *I, size_t *bytes) {
  MT_CHECK(I && bytes, MT_EINVAL, "mt_integrator_checkpoint_bytes: NULL argument");
  *bytes = ckpt_bytes(I);
  return MT_OK;
}

mt_status mt_integrator_checkpoint(mt_integrator *I, void *buf, size_t bytes) {
  MT_CHECK(I && buf, MT_EINVAL, "mt_integrator_checkpoint: NULL argument");
  const size_t need = ckpt_bytes(I);
  MT_CHECK(bytes >= need, MT_EINVAL, "mt_integrator_checkpoint: buffer of %zu bytes, %zu needed", bytes, need);
  unsigned char *p = static_cast<unsigned char *>(buf);
  CkptHeader h{};
  std::memcpy(h.magic, kCkptMagic, sizeof(h.magic));
  h.version = kCkptVersion;
  h.k1_valid = I->need_init ? 0u : 1u;
  h.n = I->T->n;
  h.B = I->B;
  h.prec = I->T->prec;
  h.layout = I->T->layout;
  h.ctl_bytes = (uint32_t)sizeof(SimCtl);
  std::memcpy(p, &h, sizeof(h));
  std::vector<SimCtl> c;
  mt_status st = read_ctl(I, c);  // also orders after every queued step
  if (st != MT_OK) return st;
  // every public call ends with the commit of the last accepted attempt
  // (m and k1 already hold it), so the flag that asks the next begin to
  // adopt it again is dropped: the next attempt starts from the same bits
  for (auto &x : c) x.accepted = 0;
  unsigned char *q = p + sizeof(h);
  std::memcpy(q, c.data(), sizeof(SimCtl) * I->B);
  q += sizeof(SimCtl) * I->B;
  const size_t state = sizeof(float) * 3 * (size_t)I->T->n * I->B;
  MT_CUDA(cudaMemcpyAsync(q, I->y, state, cudaMemcpyDeviceToHost, I->stream));
  MT_CUDA(cudaMemcpyAsync(q + state, I->k[0], state, cudaMemcpyDeviceToHost, I->stream));
  MT_CUDA(cudaStreamSynchronize(I->stream));
  q += 2 * state;
  const uint64_t sum = fnv1a64(p, (size_t)(q - p));
  std::memcpy(q, &sum, sizeof(sum));
  return MT_OK;
}

mt_status mt_integrator_restore(mt_integrator *I, const void *buf, size_t bytes) {
  MT_CHECK(I && buf, MT_EINVAL, "mt_integrator_restore: NULL argument");
  const unsigned char *p = static_cast<const unsigned char *>(buf);
  MT_CHECK(bytes >= sizeof(CkptHeader), MT_EINVAL, "mt_integrator_restore: %zu bytes is no checkpoint", bytes);
  CkptHeader h;
  std::memcpy(&h, p, sizeof(h));
  MT_CHECK(std::memcmp(h.magic, kCkptMagic, sizeof(h.magic)) == 0 && h.version == kCkptVersion &&
               h.ctl_bytes == sizeof(SimCtl),
           MT_EINVAL, "mt_integrator_restore: not a checkpoint of this format version");
  MT_CHECK(h.n == I->T->n && h.B == I->B, MT_EINVAL,
           "mt_integrator_restore: checkpoint of n = %lld, B = %d into an integrator of n = %lld, B = %d",
           (long long)h.n, h.B, (long long)I->T->n, I->B);
  const size_t need = ckpt_bytes(I);
  MT_CHECK(bytes >= need, MT_EINVAL, "mt_integrator_restore: %zu bytes, %zu expected", bytes, need);
  uint64_t sum;
  std::memcpy(&sum, p + need - sizeof(sum), sizeof(sum));
  MT_CHECK(sum == fnv1a64(p, need - sizeof(sum)), MT_EINVAL, "mt_integrator_restore: checksum mismatch");
  std::vector<SimCtl> c(I->B);
  const unsigned char *q = p + sizeof(h);
  std::memcpy(c.data(), q, sizeof(SimCtl) * I->B);
  q += sizeof(SimCtl) * I->B;
  const size_t state = sizeof(float) * 3 * (size_t)I->T->n * I->B;
  // the state of a finished simulation is restored with it; the derivative
  // only when it was evaluated with this kind of tensor
  const bool keep_k1 = h.k1_valid && h.prec == I->T->prec && h.layout == I->T->layout;
  MT_CUDA(cudaMemcpyAsync(I->y, q, state, cudaMemcpyHostToDevice, I->stream));
  if (keep_k1) MT_CUDA(cudaMemcpyAsync(I->k[0], q + state, state, cudaMemcpyHostToDevice, I->stream));
  mt_status st = write_ctl(I, c);  // synchronises: the host image may go after this
  if (st != MT_OK) return st;
  I->need_init = !keep_k1;
  return MT_OK;
}

mt_status mt_integrate(mt_tensor *T, const mt_llg_params *p, const mt_ode_opts *o, float *m, int B, double t0,
                       double t1, int64_t n_out, double *mavg, mt_stats *stats, void *stream) {
  mt_integrator *I = nullptr;
  mt_status st = mt_integrator_create(T, p, o, B, stream, &I);
  if (st != MT_OK) return st;
  st = mt_integrator_set_state(I, m, 0, t0);
  mt_status st2 = (st == MT_OK) ? mt_integrator_run(I, t1, n_out, mavg, stats) : st;
  if (st == MT_OK) st = mt_integrator_get_state(I, m, 0);
  if (st == MT_OK) {
    cudaError_t e = cudaStreamSynchronize(I->stream);
    if (e != cudaSuccess) st = mt::cuda_fail(e, "sync", __FILE__, __LINE__);
  }
  mt_integrator_destroy(I);
  return st2 != MT_OK ? st2 : st;
}

mt_status mt_relax(mt_tensor *T, const mt_llg_params *p, const mt_ode_opts *o, double tol, double t_max, float *m,
                   int B, mt_stats *stats, void *stream) {
  mt_integrator *I = nullptr;
  mt_status st = mt_integrator_create(T, p, o, B, stream, &I);
  if (st != MT_OK) return st;
  st = mt_integrator_set_state(I, m, 0, 0.0);
  mt_status st2 = (st == MT_OK) ? mt_integrator_relax(I, tol, t_max, stats) : st;
  if (st == MT_OK) st = mt_integrator_get_state(I, m, 0);
  if (st == MT_OK) {
    cudaError_t e = cudaStreamSynchronize(I->stream);
    if (e != cudaSuccess) st = mt::cuda_fail(e, "sync", __FILE__, __LINE__);
  }
  mt_integrator_destroy(I);
  return st2 != MT_OK ? st2 : st;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// slot-level control used by the serving loop (one simulation per slot,
// admitted and retired while the others keep running)
// ---------------------------------------------------------------------------
namespace mt {

size_t integ_ctl_bytes(const mt_integrator *I) { return sizeof(SimCtl) * I->B; }
int integ_batch(const mt_integrator *I) { return I->B; }
void *integ_stream(const mt_integrator *I) { return I->stream; }

// Enqueue the admission of one simulation into slot b: its state (host,
// 3n floats, must stay valid until the stream reaches the copy), its
// equation parameters, and a relax goal (torque < tol, time cap t_max).
mt_status integ_admit(mt_integrator *I, int b, const float *m0_host, double alpha, const double *Ha, double tol,
                      double t_max) {
  MT_CHECK(b >= 0 && b < I->B, MT_EINVAL, "slot %d out of range", b);
  const int64_t n = I->T->n;
  MT_CUDA(cudaMemcpyAsync(I->y + (size_t)b * 3 * n, m0_host, sizeof(float) * 3 * n, cudaMemcpyHostToDevice,
                          I->stream));
  const double a = alpha;
  double G1, G2;
  if (I->form == MT_FORM_GILBERT) {
    G1 = I->gamma / (1.0 + a * a);
    G2 = G1 * a;
  } else {
    G1 = I->gamma;
    G2 = a;
  }
  if (!I->precess) G1 = 0.0;
  // pinned staging: slot b's entries are reused only after its previous
  // simulation finished, i.e. after the stream consumed them
  float *par = I->h_slot_par + 5 * b;
  par[0] = (float)G1;
  par[1] = (float)G2;
  par[2] = (float)Ha[0];
  par[3] = (float)Ha[1];
  par[4] = (float)Ha[2];
  MT_CUDA(cudaMemcpyAsync(I->g1 + b, par, sizeof(float), cudaMemcpyHostToDevice, I->stream));
  MT_CUDA(cudaMemcpyAsync(I->g2 + b, par + 1, sizeof(float), cudaMemcpyHostToDevice, I->stream));
  MT_CUDA(cudaMemcpyAsync(I->Ha + 3 * b, par + 2, 3 * sizeof(float), cudaMemcpyHostToDevice, I->stream));
  SimCtl c;
  std::memset(&c, 0, sizeof(c));
  c.t = 0.0;
  c.h = I->o.fixed_h > 0 ? I->o.fixed_h : I->o.h0;
  c.mode = MODE_RELAX;
  c.tol = tol;
  c.t1 = t_max;
  c.t_next = t_max;
  c.attempt_cap = I->o.max_steps;
  c.status = MT_OK;
  c.fresh = 1;
  plan_host(I, c);
  k_admit<<<1, 1, 0, I->stream>>>(I->ctl, I->active, I->n_active, b, c);
  MT_CUDA(cudaGetLastError());
  return MT_OK;
}

// Enqueue the next leg of slot b's simulation from the state it holds (a
// field sweep moves to its next applied field): new applied field, a fresh
// relax goal (torque < tol, time cap t_max from t = 0) and the first trial
// step h0, as a new relaxation would start; k1 is re-evaluated by the next
// integ_init_fresh.  The damping stays.
mt_status integ_readmit(mt_integrator *I, int b, const double *Ha, double tol, double t_max) {
  MT_CHECK(b >= 0 && b < I->B, MT_EINVAL, "slot %d out of range", b);
  // pinned staging: slot b's entries were consumed at its admission, which
  // the stream completed before the poll that reported the slot done
  float *par = I->h_slot_par + 5 * b;
  par[2] = (float)Ha[0];
  par[3] = (float)Ha[1];
  par[4] = (float)Ha[2];
  MT_CUDA(cudaMemcpyAsync(I->Ha + 3 * b, par + 2, 3 * sizeof(float), cudaMemcpyHostToDevice, I->stream));
  SimCtl c;
  std::memset(&c, 0, sizeof(c));
  c.t = 0.0;
  c.h = I->o.fixed_h > 0 ? I->o.fixed_h : I->o.h0;
  c.mode = MODE_RELAX;
  c.tol = tol;
  c.t1 = t_max;
  c.t_next = t_max;
  c.attempt_cap = I->o.max_steps;
  c.status = MT_OK;
  c.fresh = 1;
  plan_host(I, c);
  k_admit<<<1, 1, 0, I->stream>>>(I->ctl, I->active, I->n_active, b, c);
  MT_CUDA(cudaGetLastError());
  return MT_OK;
}

// volume-averaged m of slot b after its last accepted step, from a polled
// control copy
void integ_slot_mavg(const void *ctl_host, int b, double m[3]) {
  const SimCtl &c = reinterpret_cast<const SimCtl *>(ctl_host)[b];
  for (int q = 0; q < 3; ++q) m[q] = c.m_last[q];
}

// Device bytes of an integrator of B simulations (mt_integrator_create): states,
// fields and derivatives, operand and work areas of the product, and 4 MB for
// the rest (control blocks, reductions, the words of the one-kernel path, at
// most 2.5 MB as its states fit a CTA's shared memory, the step graph).
size_t integ_bytes(const mt_tensor *T, int B) {
  const bool dense = T->layout == MT_LAYOUT_DENSE;
  const size_t vec = sizeof(float) * 3 * T->n * B;
  const size_t product = dense ? dense_x_bytes(T, B) + dense_part_bytes(T, B) + dense_count_bytes(T)
                               : sizeof(float) * xs_floats(T) * B + matvec_part_bytes(T) + matvec_count_bytes(T, B) +
                                     matvec_colpart_bytes(T, B);
  return 11 * vec + product + ((size_t)4 << 20);
}

// k1 for the freshly admitted slots (one demag product for the batch)
mt_status integ_init_fresh(mt_integrator *I) { return enqueue_init(I, 1); }

mt_status integ_replay(mt_integrator *I, int k) {
  for (int q = 0; q < k; ++q) MT_CUDA(cudaGraphLaunch(I->exec, I->stream));
  return MT_OK;
}

// commit accepted states and copy every slot's control block to ctl_host
// (pinned); `ev` is recorded after the copy
mt_status integ_poll(mt_integrator *I, void *ctl_host, cudaEvent_t ev) {
  mt_status st = enqueue_commit(I);
  if (st != MT_OK) return st;
  MT_CUDA(cudaMemcpyAsync(ctl_host, I->ctl, sizeof(SimCtl) * I->B, cudaMemcpyDeviceToHost, I->stream));
  MT_CUDA(cudaEventRecord(ev, I->stream));
  return MT_OK;
}

// read slot b of a polled control copy
bool integ_slot_done(const void *ctl_host, int b, mt_stats *st) {
  const SimCtl &c = reinterpret_cast<const SimCtl *>(ctl_host)[b];
  if (st) {
    st->n_accept = c.n_accept;
    st->n_reject = c.n_reject;
    st->n_rhs = c.n_rhs;
    st->t = c.t;
    st->h = c.h;
    st->tau = c.tau;
    st->status = c.status;
    st->pad = 0;
  }
  return c.done != 0;
}

// enqueue the copy of slot b's committed state to host memory
mt_status integ_fetch_slot(mt_integrator *I, int b, float *m_host) {
  const int64_t n = I->T->n;
  MT_CUDA(cudaMemcpyAsync(m_host, I->y + (size_t)b * 3 * n, sizeof(float) * 3 * n, cudaMemcpyDeviceToHost,
                          I->stream));
  return MT_OK;
}

// an integrator whose slots all start empty (no active simulation)
mt_status integ_create_idle(mt_tensor *T, const mt_llg_params *p, const mt_ode_opts *o, int B,
                            mt_integrator **out) {
  mt_integrator *I = nullptr;
  mt_status st = mt_integrator_create(T, p, o, B, nullptr, &I);
  if (st != MT_OK) return st;
  I->path = MT_PATH_GRAPH;  // slots are admitted between graph replays
  std::vector<SimCtl> c(B);
  for (auto &x : c) {
    std::memset(&x, 0, sizeof(SimCtl));
    x.done = 1;
    x.status = MT_OK;
    x.t_next = 1e300;
  }
  if ((st = write_ctl(I, c)) != MT_OK) {
    mt_integrator_destroy(I);
    return st;
  }
  if (cudaMallocHost(&I->h_slot_par, sizeof(float) * 5 * B) != cudaSuccess) {
    mt_integrator_destroy(I);
    mt::set_error("serving engine: pinned allocation failed");
    return MT_ENOMEM;
  }
  I->need_init = false;
  *out = I;
  return MT_OK;
}

}  // namespace mt
