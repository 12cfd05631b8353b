// Batched demag product on the 5th-generation tensor cores (tcgen05).
//
// B simulations on one geometry turn the product H_d = -N (Ms m) (Eq. 9,
// Eq. 17) into GEMMs with X[b] = Ms m_b.  Every 3x3 block of N is symmetric,
// so the tensor is stored as its 6 entry planes (xx xy xz yy yz zz; 4, without
// xz and yz, for a single-layer tile set), each an n x n matrix in BF16 or as
// a BF16 hi + lo pair ("split"), and an off-diagonal plane is read once and
// multiplied twice: H_x += N_xy X_y and H_y += N_xy X_x.  The split product
// carries the operand as three BF16 terms x0 + x1 + x2 (24 significant bits: a
// relaxed, nearly uniform state would otherwise round every x the same way and
// leave a coherent error) and forms N_hi (x0 + x1 + x2) + N_lo (x0 + x1); the
// blocks of touching tiles are zero there and are applied with FP64-class
// accuracy by the near-field kernel.
//
// The product is HBM-bound for B <= ~200 (96 flop per tensor byte at B = 64),
// so the design streams the planes once per batched product:
//   * persistent CTAs, one per SM; the (row tile, K block, plane) units are
//     split evenly over the CTAs in storage order (stream-K);
//   * warp 0 issues 2-D TMA loads (128-byte swizzle): a 128 x 64 plane tile
//     (split: hi and lo together) per stage of a shared-memory ring, and the
//     64-wide operand slices of the K block's components, each once per row
//     tile and K block, in a ring of their own.  The first ring-full of plane
//     tiles is issued before the wait on the kernel ahead (which writes the
//     operand, never the tensor);
//   * warp 1 issues tcgen05.mma (M = 128, N = B ... 3 B, K = 16, BF16 -> FP32)
//     into one TMEM accumulator per component and K block (the tensor cores'
//     FP32 accumulation rounds with a bias, so chains stay short: at most 192
//     products), taken in rotation from a ring of accumulators, and releases
//     ring slots with tcgen05.commit;
//   * eight warps drain each finished accumulator with tcgen05.ld (one TMEM lane
//     = one row per thread, half of the batch per warp) into FP32 register
//     sums of the three components while the next ones fill; row tiles split
//     between CTAs are summed by whichever warp arrives last, in CTA order;
//   * the ring depth is chosen per tensor and batch width by timing
//     candidates on first use.
// Storing all 9 entries of a block moved 1.5 times the bytes (single layer:
// 2.25 times).  Fields, before and after: n = 6,000, B = 8, BF16 110 -> 84 us
// (product 98 -> 70, 0.92 of the copy bandwidth); n = 10,000, B = 64, BF16 328
// -> 226 us (product 188, 0.97); split, B = 16 521 -> 370 us (product at the
// copy bandwidth), B = 64 595 -> 537 us and at n = 20,000 2,187 -> 1,946 us:
// there the five products of every entry bound it, 1.3 PFLOP/s.
// Every wait is bounded; on a timeout the kernel records MT_DEV_TIMEOUT,
// still frees its TMEM and returns.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "mt_internal.cuh"

namespace {

constexpr int GM = 128;  // rows per tile (MMA M)
constexpr int GK = 64;   // K per ring stage: one 128-byte swizzle row of BF16
constexpr int EPI_WARPS = 8;
constexpr int A_TILE = GM * GK * 2;  // bytes of one plane tile

// Shape of one batch width.  GROUPS: column groups of an accumulator (the
// epilogue adds them).  The split product puts the operand terms side by side
// so that a tensor tile is read from shared memory twice per K step instead of
// five times (those reads, not the tensor pipe, would bound it):
//   BP <= 32: N_hi [x0 | x1 | x2] (N = 3 BP) and N_lo [x0 | x1] (N = 2 BP);
//   BP = 64:  three such groups of three components would not fit the 512 TMEM
//             columns twice over, so N_hi [x0 | x1] and N_lo [x0 | x1]
//             (N = 128), and N_hi x2 (N = 64) onto the second group;
//   BP = 128: five products onto one group.
// A ring stage holds one unit of 32 KB: a plane's hi and lo tiles, or two
// consecutive planes' tiles (16 KB stages left the handshakes of the TMA, MMA
// and commit path, a few hundred cycles each, above a tile's time in HBM).
// XG: the three operand slices of a K block share a slot and its barriers
// where two such slots fit, else each has its own.  AG: likewise the three
// accumulators of a K block; else they are taken in rotation, at least 4 (the
// next K block's first component starts while the last one's are drained).
template <bool SPLIT, int BP>
struct GemmShape {
  static constexpr int GROUPS = !SPLIT ? 1 : BP <= 32 ? 3 : BP == 64 ? 2 : 1;
  static constexpr int ACC_COLS = GROUPS * BP;
  static constexpr bool AG = 512 / ACC_COLS >= 6;
  static constexpr int NA = AG ? 2 : 512 / ACC_COLS;  // barriers: sets of three, or single accumulators
  static constexpr int ACCS = AG ? 6 : NA;
  static constexpr int TERMS = SPLIT ? 3 : 1;
  static constexpr int X_SLICE = TERMS * BP * GK * 2;  // bytes: one component of one K block
  static constexpr bool XG = !SPLIT || BP <= 32;
  static constexpr int NX = XG ? 2 : BP == 64 ? 4 : 3;
  static constexpr int X_SLOT = (XG ? 3 : 1) * X_SLICE;
  static constexpr int X_ROWS = XG && !SPLIT && 3 * BP <= 256 ? 3 * BP : BP;  // rows of one operand copy
  static constexpr int PPU = SPLIT ? 1 : 2;  // planes per unit
  static constexpr int A_STAGE = 2 * A_TILE;
  static constexpr int HB = BP / 2;  // simulations per epilogue warp
  // the 3 HB register sums of an epilogue thread at BP = 128 exceed what 10
  // warps may have (168): two warpgroups of epilogue warps then take over
  // registers of a first one that holds the TMA and MMA warps (56 + 2 x 224 =
  // 3 x 168)
  static constexpr bool REGSPLIT = BP == 128;
  static constexpr int EPI0 = REGSPLIT ? 4 : 2;  // first epilogue warp
  static constexpr int THREADS = 32 * (EPI0 + EPI_WARPS);
  static_assert(AG || NA >= 4, "accumulators of one K block and one spare");
};

// Planes in storage order (NP = 6, or 4 for a single layer): plane p couples
// the components pc(p) <= pd(p).
template <int NP>
constexpr __host__ __device__ int pc(int p) {
  return NP == 6 ? (p < 3 ? 0 : p < 5 ? 1 : 2) : (p < 2 ? 0 : p - 1);
}
template <int NP>
constexpr __host__ __device__ int pd(int p) {
  return NP == 6 ? (p < 3 ? p : p < 5 ? p - 2 : 2) : (p == 0 ? 0 : p < 3 ? 1 : 2);
}
// planes that a component takes part in, as a bit mask
template <int NP>
constexpr __host__ __device__ unsigned planes_of(int comp) {
  return NP == 6 ? (comp == 0 ? 0b000111u : comp == 1 ? 0b011010u : 0b110100u)
                 : (comp == 0 ? 0b0011u : comp == 1 ? 0b0110u : 0b1000u);
}
// does the component take part in none of the planes p + 1 .. e - 1?
template <int NP>
__device__ __forceinline__ bool last_plane(int comp, int p, int e) {
  return (planes_of<NP>(comp) & ~((2u << p) - 1u) & ((1u << e) - 1u)) == 0;
}

// ---- tcgen05 / TMA wrappers -------------------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(mtd::smem_u32(slot)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// one lane of the (converged) warp
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}

// D (tmem) = A (smem) * B (smem) [+ D]; BF16 inputs, FP32 accumulate
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// arrive on `bar` once every tcgen05.mma issued so far by this thread is done
__device__ __forceinline__ void umma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   mtd::smem_u32(bar))
               : "memory");
}
// 32 lanes x 32 bit, 16 consecutive columns per thread; the registers are
// valid only after tmem_wait_ld()
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t r[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t r[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tma_2d(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar,
                                       uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(mtd::smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(mtd::smem_u32(bar)), "l"(policy)
      : "memory");
}
// shared-memory matrix descriptor: K-major tile, 128-byte swizzle, rows of
// 128 bytes, 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

struct GemmArgs {
  int64_t n;     // tiles
  int64_t MT;    // row tiles
  int64_t KB;    // K blocks
  int B, Bp;     // batch, padded batch (MMA N)
  int stages;    // plane tiles in the ring
  uint32_t tmem_cols;
  float *H;      // [B][n][3]
  float *part;   // [2G][3][Bp][GM]
  int *count;    // [MT][EPI_WARPS]
  const int *n_active;
  int *status;
};

// f(integral_constant<0>) ... f(integral_constant<N - 1>)
template <int N, int I = 0, typename F>
__device__ __forceinline__ void static_for(F &&f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    static_for<N, I + 1>(f);
  }
}

// a ring position: slot and the parity of its current pass
template <int DEPTH>
struct RingPos {
  uint32_t s = 0, ph = 0;
  __device__ __forceinline__ void next(int depth = DEPTH) {
    if (++s == (uint32_t)depth) {
      s = 0;
      ph ^= 1u;
    }
  }
};

// W consecutive columns of an accumulator, its column groups added (the small
// ones first), onto run
template <int W, int GROUPS, int BP>
__device__ __forceinline__ void drain_cols(uint32_t acc, float *run) {
  uint32_t v[GROUPS][W];
#pragma unroll
  for (int g = 0; g < GROUPS; ++g) {
    if constexpr (W == 16) tmem_ld16(acc + (uint32_t)(g * BP), v[g]);
    else tmem_ld8(acc + (uint32_t)(g * BP), v[g]);
  }
  tmem_wait_ld();
#pragma unroll
  for (int j = 0; j < W; ++j) {
    float x = __uint_as_float(v[GROUPS - 1][j]);
#pragma unroll
    for (int g = GROUPS - 2; g >= 0; --g) x = __uint_as_float(v[g][j]) + x;
    run[j] += x;
  }
}

template <bool SPLIT, int BP, int NP>
__global__ void __launch_bounds__(GemmShape<SPLIT, BP>::THREADS, 1)
    k_gemm(const __grid_constant__ CUtensorMap tA, const __grid_constant__ CUtensorMap tX, GemmArgs P) {
  using SH = GemmShape<SPLIT, BP>;
  constexpr int NA = SH::NA, NX = SH::NX, HB = SH::HB;
  constexpr int NU = NP / SH::PPU;  // units of a (row tile, K block)
  extern __shared__ unsigned char smem_raw[];
  // 1024-byte aligned base for the swizzled tiles: the plane tiles, the
  // operand slices, the barriers
  const uint32_t raw = mtd::smem_u32(smem_raw);
  unsigned char *smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);
  unsigned char *smem_x = smem + (size_t)P.stages * SH::A_STAGE;
  uint64_t *full = reinterpret_cast<uint64_t *>(smem_x + NX * SH::X_SLOT);
  uint64_t *empty = full + P.stages;
  uint64_t *xfull = empty + P.stages;
  uint64_t *xempty = xfull + NX;
  uint64_t *accf = xempty + NX;
  uint64_t *acce = accf + NA;
  uint64_t *mma_done = acce + NA;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(mma_done + 1);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

  // (the same value in a form the compiler knows to be uniform)
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int64_t G = gridDim.x, k = blockIdx.x;
  const int64_t U = P.MT * P.KB * NU;
  const int64_t u0 = mtd::sk_begin(k, U, G), u1 = mtd::sk_begin(k + 1, U, G);

  if (threadIdx.x == 0) {
    for (int s = 0; s < P.stages; ++s) {
      mtd::mbar_init(&full[s], 1);
      mtd::mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < NX; ++s) {
      mtd::mbar_init(&xfull[s], 1);
      mtd::mbar_init(&xempty[s], 1);
    }
    for (int a = 0; a < NA; ++a) {
      mtd::mbar_init(&accf[a], 1);
      mtd::mbar_init(&acce[a], EPI_WARPS);
    }
    mtd::mbar_init(mma_done, 1);
    *abort_flag = 0;
    mtd::fence_mbar_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, P.tmem_cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // unit u into ring stage s
  auto load_a = [&](int64_t u, int s, uint64_t pol) {
    mtd::mbar_arrive_expect_tx(&full[s], SH::A_STAGE);
    tma_2d(smem + (size_t)s * SH::A_STAGE, &tA, 0, (int)(u * 2 * GM), &full[s], pol);
  };
  const int pre = (int)(u1 - u0 < P.stages ? u1 - u0 : P.stages);
  if (warp == 0 && elect_one()) {
    const uint64_t pol = mtd::policy_evict_first();
    for (int s = 0; s < pre; ++s) load_a(u0 + s, s, pol);
  }
  __syncwarp();
  mtd::pdl_enter();
  const bool idle = P.n_active && *P.n_active == 0;  // every simulation finished

  if (warp < SH::EPI0) {
    if constexpr (SH::REGSPLIT) asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    // (One thread each issues the copies and the products, and a few hundred
    // dependent instructions per plane tile would already exceed the tile's
    // time in HBM: the planes are unrolled, ring positions counted, and the
    // whole MMA warp walks the units, so that descriptors and addresses stay
    // in uniform registers, as the instruction takes them.)
    if (warp == 0) {
      // ---------------- TMA producer ----------------
      const bool leader = elect_one();
      const uint64_t pol_stream = mtd::policy_evict_first();
      const uint64_t pol_keep = mtd::policy_evict_last();
      RingPos<0> a;
      RingPos<NX> x;
      int it = 0, xi = 0;
      bool stop = idle;
      int64_t kb = (u0 / NU) % P.KB;
      int e0 = (int)(u0 % NU);
      auto wait = [&](uint64_t *bar, uint32_t parity) {
        if (*abort_flag || !mtd::mbar_wait_bounded(bar, parity, P.status)) {
          *abort_flag = 1;
          stop = true;
        }
      };
      // operand rows of (term t, K block kb, component c): ((t KB + kb) 3 + c) Bp
      auto copy_x = [&](uint32_t off, int t, int c) {
        tma_2d(smem_x + x.s * SH::X_SLOT + off, &tX, 0, (int)(((t * P.KB + kb) * 3 + c) * BP), &xfull[x.s], pol_keep);
      };
      for (int64_t u = u0; u < u1 && !stop;) {
        const int e1 = u1 - u < NU - e0 ? e0 + (int)(u1 - u) : NU;
        unsigned have = 0;  // components whose slice is loaded
        auto slice = [&](int comp) {
          if (have >> comp & 1 || stop) return;
          have |= SH::XG ? 7u : 1u << comp;
          wait(&xempty[x.s], x.ph ^ 1u);  // (passes on the first round)
          if (stop) return;
          if (leader) {
            mtd::mbar_arrive_expect_tx(&xfull[x.s], SH::X_SLOT);
            constexpr int TB = BP * GK * 2;  // bytes of one operand term
            if constexpr (SH::X_ROWS > BP) {
              copy_x(0, 0, 0);
            } else if constexpr (SH::XG) {
#pragma unroll
              for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int t = 0; t < SH::TERMS; ++t) copy_x(c * SH::X_SLICE + t * TB, t, c);
            } else {
#pragma unroll
              for (int t = 0; t < SH::TERMS; ++t) copy_x(t * TB, t, comp);
            }
          }
          x.next();
          ++xi;
        };
        static_for<NU>([&](auto uu) {
          constexpr int p0 = uu * SH::PPU;
          if (uu < e0 || uu >= e1 || stop) return;
          static_for<SH::PPU>([&](auto r) {
            slice(pc<NP>(p0 + r));
            slice(pd<NP>(p0 + r));
          });
          if (!stop && it >= pre) {
            wait(&empty[a.s], a.ph ^ 1u);
            if (!stop && leader) load_a(u + (uu - e0), (int)a.s, pol_stream);
          }
          if (!stop) {
            ++it;
            a.next(P.stages);
          }
        });
        u += e1 - e0;
        e0 = 0;
        if (++kb == P.KB) kb = 0;
      }
      // drain: every copy issued must have landed before the CTA may exit
      it = it > pre ? it : pre;
      for (int s = 0; s < P.stages && s < it; ++s) {
        const int last = it - 1 - ((it - 1 - s) % P.stages);  // last issue on stage s
        mtd::mbar_wait_bounded(&full[s], (uint32_t)(last / P.stages) & 1u, P.status);
      }
      for (int s = 0; s < NX && s < xi; ++s) {
        const int last = xi - 1 - ((xi - 1 - s) % NX);
        mtd::mbar_wait_bounded(&xfull[s], (uint32_t)(last / NX) & 1u, P.status);
      }
    } else if (!idle && warp == 1) {
      // ---------------- MMA issuer ----------------
      // D: FP32; A, B: BF16; M = 128; N in units of 8 columns
      constexpr uint32_t id0 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(GM >> 4) << 24);
      constexpr uint32_t id1 = id0 | ((uint32_t)(BP >> 3) << 17), id2 = id0 | ((uint32_t)(2 * BP >> 3) << 17),
                         id3 = id0 | ((uint32_t)(3 * BP >> 3) << 17);
      const uint64_t da0 = sw128_desc(mtd::smem_u32(smem)), dx0 = sw128_desc(mtd::smem_u32(smem_x));
      const bool leader = elect_one();
      RingPos<0> a;
      RingPos<NX> x;
      RingPos<NA> c;
      bool issued = false, ok = true;
      int e0 = (int)(u0 % NU);
      for (int64_t u = u0; u < u1 && ok;) {
        const int e1 = u1 - u < NU - e0 ? e0 + (int)(u1 - u) : NU;
        // per component: its operand (offset in the descriptor), its accumulator
        // (column), its barriers
        uint32_t opnd[3] = {0, 0, 0}, acc[3] = {0, 0, 0}, xbar[3] = {0, 0, 0}, abar[3] = {0, 0, 0};
        unsigned have = 0, begun = 0;
        // a component's first plane: its operand has arrived, an accumulator is free
        auto begin = [&](auto comp) {
          if (!SH::XG || have == 0) ok = ok && mtd::mbar_wait_bounded(&xfull[x.s], x.ph, P.status);
          if (!SH::AG || have == 0)
            ok = ok && mtd::mbar_wait_bounded(&acce[c.s], c.ph ^ 1u, P.status);  // (passes on the first round)
          opnd[comp] = (x.s * SH::X_SLOT + (SH::XG ? comp * SH::X_SLICE : 0)) >> 4;
          acc[comp] = (SH::AG ? 3 * c.s + comp : c.s) * SH::ACC_COLS;
          xbar[comp] = x.s;
          abar[comp] = c.s;
          have |= 1u << comp;
          if (!SH::XG) x.next();
          if (!SH::AG) c.next();
        };
        static_for<NU>([&](auto uu) {
          if (uu < e0 || uu >= e1 || !ok) return;
          static_for<SH::PPU>([&](auto r) {
            constexpr int p = uu * SH::PPU + r;
            constexpr std::integral_constant<int, pc<NP>(p)> pa{};
            constexpr std::integral_constant<int, pd<NP>(p)> pb{};
            if (!(have >> pa & 1)) begin(pa);
            if (!(have >> pb & 1)) begin(pb);
          });
          if (!ok || *abort_flag || !mtd::mbar_wait_bounded(&full[a.s], a.ph, P.status)) {
            ok = false;
            return;
          }
          tc_fence_after();
          static_for<SH::PPU>([&](auto r) {
            constexpr int p = uu * SH::PPU + r;
            constexpr std::integral_constant<int, pc<NP>(p)> pa{};
            constexpr std::integral_constant<int, pd<NP>(p)> pb{};
            const uint64_t da = da0 + ((a.s * SH::A_STAGE + (SPLIT ? 0 : r * A_TILE)) >> 4);
            // the plane times one component's operand, onto the other's accumulator
            auto product = [&](uint32_t to, uint32_t from, uint32_t keep) {
              const uint32_t dt = tmem_base + to;
              const uint64_t dx = dx0 + from;
              if (!leader) return;
  #pragma unroll
              for (int kk = 0; kk < GK / 16; ++kk) {
                // K advance inside the 128-byte swizzle row: 16 BF16 = 32 bytes
                const uint64_t dak = da + 2 * kk, dxk = dx + 2 * kk;
                const uint32_t k0 = kk == 0 ? keep : 1u;  // 0: the accumulator's first product
                if constexpr (!SPLIT) {
                  umma_bf16(dt, dak, dxk, id1, k0);
                } else {
                  const uint64_t dlo = dak + (A_TILE >> 4);
                  constexpr int TB = (BP * GK * 2) >> 4;  // one operand term
                  if constexpr (SH::GROUPS == 3) {
                    umma_bf16(dt, dak, dxk, id3, k0);  // N_hi [x0 | x1 | x2]
                    umma_bf16(dt, dlo, dxk, id2, 1u);  // N_lo [x0 | x1]
                  } else if constexpr (SH::GROUPS == 2) {
                    umma_bf16(dt, dak, dxk, id2, k0);                // N_hi [x0 | x1]
                    umma_bf16(dt + BP, dak, dxk + 2 * TB, id1, 1u);  // N_hi x2
                    umma_bf16(dt, dlo, dxk, id2, 1u);                // N_lo [x0 | x1]
                  } else {
                    umma_bf16(dt, dak, dxk, id1, k0);           // N_hi x0
                    umma_bf16(dt, dak, dxk + TB, id1, 1u);      // N_hi x1
                    umma_bf16(dt, dak, dxk + 2 * TB, id1, 1u);  // N_hi x2
                    umma_bf16(dt, dlo, dxk, id1, 1u);           // N_lo x0
                    umma_bf16(dt, dlo, dxk + TB, id1, 1u);      // N_lo x1
                  }
                }
              }
            };
            product(acc[pa], opnd[pb], begun >> pa & 1);
            if constexpr (pa != pb) product(acc[pb], opnd[pa], begun >> pb & 1);
            begun |= 1u << pa | 1u << pb;
          });
          issued = true;
          if (leader) umma_commit(&empty[a.s]);  // ring slot free once these MMAs are done
          a.next(P.stages);
          // a component's last plane: its slice is free, its accumulator complete
          static_for<3>([&](auto comp) {
            constexpr int pe = uu * SH::PPU + SH::PPU;  // planes so far
            if (!leader || !(planes_of<NP>(comp) >> (pe - SH::PPU) & ((1u << SH::PPU) - 1u)) ||
                !last_plane<NP>(comp, pe - 1, e1 * SH::PPU))
              return;
            if (!SH::XG) umma_commit(&xempty[xbar[comp]]);
            if (!SH::AG) umma_commit(&accf[abar[comp]]);
          });
        });
        if (!ok) break;
        if (SH::XG) {
          if (leader) umma_commit(&xempty[x.s]);
          x.next();
        }
        if (SH::AG) {
          if (leader) umma_commit(&accf[c.s]);
          c.next();
        }
        u += e1 - e0;
        e0 = 0;
      }
      if (!ok) *abort_flag = 1;
      if (leader) {
        if (issued) umma_commit(mma_done);
        else mtd::mbar_arrive(mma_done);
      }
    }
  } else {
    if constexpr (SH::REGSPLIT) asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
    if (!idle) {
      // ---------------- epilogue ----------------
      const int e = warp - SH::EPI0;
      const int lg = warp & 3;           // TMEM lane group accessible to this warp
      const int b0 = (e >> 2) * HB;      // this warp's half of the batch
      const int row = lg * 32 + lane;
      const int64_t KBU = P.KB * NU;
      const int64_t first_mt = u0 / KBU;
      RingPos<NA> c;
      float run[3][HB];  // FP32 sums of the current row tile
#pragma unroll
      for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int j = 0; j < HB; ++j) run[q][j] = 0.0f;
      bool ok = true;
      int64_t mt = first_mt, kb = (u0 / NU) % P.KB;
      int e0 = (int)(u0 % NU);
      for (int64_t u = u0; u < u1 && ok;) {
        const int e1 = u1 - u < NU - e0 ? e0 + (int)(u1 - u) : NU;
        // components in the order the MMA warp takes their accumulators (4 bits
        // each, + 1): x, y, z of a whole K block; of a partial one the planes tell
        unsigned order = 0x321;
        if (e0 != 0 || e1 != NU) {
          unsigned have = 0;
          int cnt = 0;
          order = 0;
#pragma unroll 1
          for (int p = e0 * SH::PPU; p < e1 * SH::PPU; ++p)
#pragma unroll 1
            for (int side = 0; side < 2; ++side) {
              const int comp = side ? pd<NP>(p) : pc<NP>(p);
              if (have >> comp & 1) continue;
              have |= 1u << comp;
              order |= (unsigned)(comp + 1) << (4 * cnt++);
            }
        }
        bool first = true;
#pragma unroll 1
        for (; order && ok; order >>= 4) {
          if (!SH::AG || first) {
            if (!mtd::mbar_wait_warp_relaxed(&accf[c.s], c.ph, P.status) || *abort_flag) {
              *abort_flag = 1;
              ok = false;
              break;
            }
            tc_fence_after();
          }
          first = false;
          const int comp = (int)(order & 15u) - 1;
          const uint32_t acc = tmem_base + ((uint32_t)(lg * 32) << 16) +
                               (uint32_t)((SH::AG ? 3 * c.s + comp : c.s) * SH::ACC_COLS + b0);
          constexpr int W = HB < 16 ? HB : 16;
          static_for<3>([&](auto q) {
            if (comp != q) return;
#pragma unroll
            for (int c0 = 0; c0 < HB; c0 += W) drain_cols<W, SH::GROUPS, BP>(acc + (uint32_t)c0, &run[q][c0]);
          });
          if (!SH::AG || (order >> 4) == 0) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mtd::mbar_arrive(&acce[c.s]);
            c.next();
          }
        }
        if (!ok) break;
        u += e1 - e0;
        const bool tile_ends = u == u1 || (kb == P.KB - 1 && e1 == NU);
        e0 = 0;
        if (!tile_ends) {
          ++kb;
          continue;
        }
        const int64_t next_mt = mt + 1;
        kb = 0;
        // the row tile's sums (this CTA's share of them)
        const int64_t kf = mtd::sk_owner(mt * KBU, U, G), kl = mtd::sk_owner(mt * KBU + KBU - 1, U, G);
        const int64_t r = mt * GM + row;
        const int nb = P.B - b0 < HB ? P.B - b0 : HB;  // simulations of this warp (may be <= 0)
        if (kf == kl) {
#pragma unroll
          for (int j = 0; j < HB; ++j)
            if (j < nb && r < P.n)
#pragma unroll
              for (int q = 0; q < 3; ++q) P.H[((size_t)(b0 + j) * P.n + r) * 3 + q] = -run[q][j];
        } else {
          const int64_t slot = (mt == first_mt) ? 2 * k : 2 * k + 1;
#pragma unroll
          for (int q = 0; q < 3; ++q)
#pragma unroll
            for (int j = 0; j < HB; ++j) P.part[(((size_t)slot * 3 + q) * BP + b0 + j) * GM + row] = run[q][j];
          __threadfence();
          __syncwarp();
          int last = 0;
          if (lane == 0) last = (atomicAdd(&P.count[mt * EPI_WARPS + e], 1) == (int)(kl - kf));
          last = __shfl_sync(0xffffffffu, last, 0);
          if (last) {
            __threadfence();
            // up to 16 simulations at a time, two parts' loads in flight (a
            // small tensor's row tile has a dozen parts, and the sums in CTA
            // order are a chain: 1,476-tile film, BF16, 29 simulations, four
            // attempts, 1,233 us with 8 simulations and one part at a time,
            // 833 with this).  Of the CTAs that share the tile only the first
            // may have begun before it.
            const int64_t slot_f = mtd::sk_begin(kf, U, G) / KBU == mt ? 2 * kf : 2 * kf + 1;
            constexpr int JW = HB < 16 ? HB : 16;
            for (int j0 = 0; j0 < nb; j0 += JW) {
              float tot[3][JW];
#pragma unroll
              for (int q = 0; q < 3; ++q)
#pragma unroll
                for (int j = 0; j < JW; ++j) tot[q][j] = 0.0f;
#pragma unroll 2
              for (int64_t kk = kf; kk <= kl; ++kk) {
                const float *src = P.part + ((size_t)(kk == kf ? slot_f : 2 * kk) * 3 * BP + b0 + j0) * GM + row;
#pragma unroll
                for (int q = 0; q < 3; ++q)
#pragma unroll
                  for (int j = 0; j < JW; ++j) tot[q][j] += __ldcg(src + (size_t)(q * BP + j) * GM);
              }
              if (r < P.n)
#pragma unroll
                for (int j = 0; j < JW; ++j)
                  if (j0 + j < nb)
#pragma unroll
                    for (int q = 0; q < 3; ++q) P.H[((size_t)(b0 + j0 + j) * P.n + r) * 3 + q] = -tot[q][j];
            }
            if (lane == 0) P.count[mt * EPI_WARPS + e] = 0;
          }
        }
        mt = next_mt;
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
          for (int j = 0; j < HB; ++j) run[q][j] = 0.0f;
      }
    }
  }
  __syncthreads();
  if (warp == 1) {
    if (!idle) mtd::mbar_wait_bounded(mma_done, 0u, P.status);
    tc_fence_after();
    tmem_dealloc(tmem_base, P.tmem_cols);
  }
}

// Operand of the batch: X_c[b][j] = BF16(Ms_j m_j,c), for the split product
// with the two further terms x1, x2 of x = x0 + x1 + x2 (zero for padding), and
// the simulation-fastest copy of m for the near blocks, mT[(3 j + c) Bp + b].
// A CTA takes the 64 tiles of one K block and up to SIMS simulations through
// shared memory, so that both sides of the transposition are whole rows: a warp
// reads a simulation's 192 floats, writes rows of 64 BF16, and rows of SIMS
// simulations of mT.  n = 20,000, B = 64, split: 28.5 us with one thread per
// value (mT stored with a stride), 12.1 with this.  SIMS = 32 fills a row of
// mT's 128 bytes; where that gives fewer CTAs than SMs the chain of a warp's
// simulations is the time, and SIMS = 8 gives each warp one
// (n = 729, B = 64: 6.9 us alone with 32).
constexpr int kPrepWarps = 8;
template <int SIMS>
__global__ void __launch_bounds__(32 * kPrepWarps) k_prep_dense_x(const float *m, const float *Ms, int64_t n,
                                                                  int64_t KB, int B, int Bp, int terms,
                                                                  __nv_bfloat16 *X, float *mT) {
  __shared__ float sm[SIMS][3 * GK + 1];
  const int64_t kb = blockIdx.x, j0 = kb * GK;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int b0 = blockIdx.y * SIMS, nb = B - b0 < SIMS ? B - b0 : SIMS;
  const int cols = (int)(n - j0 < GK ? n - j0 : GK);  // tiles of this block (may be <= 0: padding)
  const float ms[2] = {2 * lane < cols ? Ms[j0 + 2 * lane] : 0.0f, 2 * lane + 1 < cols ? Ms[j0 + 2 * lane + 1] : 0.0f};
  mtd::pdl_enter();
#pragma unroll
  for (int q = 0; q < SIMS / kPrepWarps; ++q) {
    const int b = w + kPrepWarps * q;
    if (b >= nb) break;
    const float *src = m + (size_t)(b0 + b) * 3 * n + 3 * j0;
#pragma unroll
    for (int t = lane; t < 3 * GK; t += 32) sm[b][t] = t < 3 * cols ? src[t] : 0.0f;
  }
  __syncthreads();
  const size_t term = (size_t)3 * KB * Bp * GK;
#pragma unroll
  for (int q = 0; q < SIMS / kPrepWarps; ++q) {
    const int b = w + kPrepWarps * q;
    if (b >= nb) break;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      __nv_bfloat162 *dst = reinterpret_cast<__nv_bfloat162 *>(X + dense_x_index(c, b0 + b, j0 + 2 * lane, Bp));
      float x[2] = {ms[0] * sm[b][6 * lane + c], ms[1] * sm[b][6 * lane + 3 + c]};
      __nv_bfloat162 hi = __floats2bfloat162_rn(x[0], x[1]);
      dst[0] = hi;
      for (int t = 1; t < terms; ++t) {
        x[0] -= __bfloat162float(hi.x);
        x[1] -= __bfloat162float(hi.y);
        hi = __floats2bfloat162_rn(x[0], x[1]);
        dst[t * term / 2] = hi;
      }
    }
  }
  const int b = lane % SIMS;
  if (b < nb)
#pragma unroll 4
    for (int t = threadIdx.x / SIMS; t < 3 * cols; t += 32 * kPrepWarps / SIMS)
      mT[(size_t)(3 * j0 + t) * Bp + b0 + b] = sm[b][t];
}

using EncodeFn = PFN_cuTensorMapEncodeTiled_v12000;

EncodeFn encode_fn() {
  static EncodeFn fn = nullptr;
  if (!fn) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeFn>(p);
  }
  return fn;
}

// 2-D BF16 map over a row-major [rows][cols] array, box (64 cols, box_rows)
mt_status make_map(CUtensorMap *map, const void *base, uint64_t cols, uint64_t rows, uint32_t box_rows) {
  EncodeFn fn = encode_fn();
  MT_CHECK(fn, MT_ECUDA, "cuTensorMapEncodeTiled is not available from the driver");
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {cols * 2};
  const cuuint32_t box[2] = {(cuuint32_t)GK, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  MT_CHECK(r == CUDA_SUCCESS, MT_ECUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
  return MT_OK;
}

// ring depth in plane tiles: what fits beside the operand slices
template <bool SPLIT, int BP>
constexpr int stages_max() {
  using SH = GemmShape<SPLIT, BP>;
  constexpr int fit = (224 * 1024 - SH::NX * SH::X_SLOT) / SH::A_STAGE;
  static_assert(fit >= 2, "at least a double-buffered ring");
  return fit < 12 ? fit : 12;
}
template <bool SPLIT, int BP>
constexpr size_t smem_for(int stages) {  // + alignment slack, barriers
  using SH = GemmShape<SPLIT, BP>;
  return (size_t)stages * SH::A_STAGE + SH::NX * SH::X_SLOT + 1024 + 512;
}
static_assert(8 * (2 * 12 + 2 * 6 + 2 * 8 + 1) + 8 <= 512, "barriers");

using GemmKernel = void (*)(const CUtensorMap, const CUtensorMap, GemmArgs);
struct GemmVariant {
  GemmKernel kernel;
  int stages, x_rows, planes_per_unit;
  size_t stage_bytes, fixed_bytes;
  uint32_t tmem_cols;
  int threads;
};
template <bool SPLIT, int BP>
GemmVariant variant(int np) {
  using SH = GemmShape<SPLIT, BP>;
  uint32_t cols = 32;
  while (cols < (uint32_t)(SH::ACCS * SH::ACC_COLS)) cols <<= 1;
  return {np == 6 ? k_gemm<SPLIT, BP, 6> : k_gemm<SPLIT, BP, 4>, stages_max<SPLIT, BP>(), SH::X_ROWS, SH::PPU, (size_t)SH::A_STAGE, smem_for<SPLIT, BP>(0), cols,
          SH::THREADS};
}
GemmVariant gemm_variant(bool split, int Bp, int np) {
  switch (Bp) {
    case 16: return split ? variant<true, 16>(np) : variant<false, 16>(np);
    case 32: return split ? variant<true, 32>(np) : variant<false, 32>(np);
    case 64: return split ? variant<true, 64>(np) : variant<false, 64>(np);
    default: return split ? variant<true, 128>(np) : variant<false, 128>(np);
  }
}

// CTAs of a product: one per SM, but at least four units to each (every CTA
// must own one, which the bookkeeping of split row tiles relies on): the last
// CTA of a row tile adds the parts of all others, a chain that grows with
// them.  Fields with a unit per CTA, with four (and with the nine-entry form
// that came before), split precision, 33 simulations: 130 tiles 29.1, 18.3
// (24.5) us, 392 tiles 56.5, 30.6 (46.1), 729 tiles 50.0, 40.8 (46.2); from
// 1,700 tiles on every SM has that many.  Eight gain more at some sizes (1,000
// tiles of a film 35.3 -> 29.9) and lose at others (350 tiles, BF16, 4
// simulations: 10.4 -> 13.9), as the ranges fall on the row tiles.  One row
// tile, up to 128 tiles, is left to one CTA (8 tiles, BF16, 128 simulations
// 21.3 -> 13.2 us; 64 tiles in a cube, split, 33: 26.0 -> 20.2).
constexpr int kMinUnits = 4;
int gemm_grid(const mt_tensor *T, int planes_per_unit) {
  const int64_t MT = T->Kp / GM, KB = T->Kp / GK, units = MT * KB * (T->L.nplane / planes_per_unit);
  return MT == 1 ? 1 : (int)std::min<int64_t>(mt::matvec_grid(T), std::max<int64_t>(1, units / kMinUnits));
}

}  // namespace

namespace mt {

// MMA N of a batch: 16, 32, 64 or 128 (one kernel instance each)
int dense_pad_batch(int B) {
  int bp = 16;
  while (bp < B && bp < 128) bp *= 2;
  return bp;
}

// operand: 3 components, 1 term (BF16) or 3 (split: x0, x1, x2)
static size_t dense_operand_bytes(const mt_tensor *T, int B) {
  return (size_t)dense_pad_batch(B) * 3 * T->Kp * 2 * (T->prec == MT_BF16_SPLIT ? 3 : 1);
}
size_t dense_x_bytes(const mt_tensor *T, int B) {  // + the simulation-fastest copy of m
  return dense_operand_bytes(T, B) + (size_t)3 * T->n * dense_pad_batch(B) * sizeof(float);
}
float *dense_mT(const mt_tensor *T, int B, void *X) {
  return reinterpret_cast<float *>(reinterpret_cast<unsigned char *>(X) + dense_operand_bytes(T, B));
}
size_t dense_part_bytes(const mt_tensor *T, int B) {
  return (size_t)2 * gemm_grid(T, T->prec == MT_BF16_SPLIT ? 1 : 2) * 3 * dense_pad_batch(B) * GM * sizeof(float);
}
size_t dense_count_bytes(const mt_tensor *T) { return (size_t)(T->Kp / GM) * EPI_WARPS * sizeof(int); }

cudaError_t gemm_prepare() {
  for (const bool split : {false, true})
    for (const int Bp : {16, 32, 64, 128})
      for (const int np : {4, 6}) {
        const cudaError_t e = cudaFuncSetAttribute(gemm_variant(split, Bp, np).kernel,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) return e;
      }
  return cudaSuccess;
}

void launch_prep_dense_x(const mt_tensor *T, const float *m, int B, void *X, cudaStream_t s) {
  const int64_t KB = T->Kp / GK;
  const bool wide = KB * ((B + 31) / 32) >= T->tiles->ctx->num_sms;
  const int sims = wide ? 32 : 8;
  const dim3 grid((unsigned)KB, (unsigned)((B + sims - 1) / sims));
  launch_pdl(wide ? k_prep_dense_x<32> : k_prep_dense_x<8>, grid, dim3(32 * kPrepWarps), 0, s, m,
             (const float *)T->tiles->d_Ms, T->n, KB, B, dense_pad_batch(B), T->prec == MT_BF16_SPLIT ? 3 : 1,
             reinterpret_cast<__nv_bfloat16 *>(X), dense_mT(T, B, X));
}

mt_status gemm_plan(const mt_tensor *T, int B, const void *X, GemmPlan *plan) {
  const int Bp = dense_pad_batch(B);
  MT_CHECK(B >= 1 && B <= 128, MT_EINVAL, "batched product: B = %d outside 1..128 simulations per pass", B);
  const bool split = T->prec == MT_BF16_SPLIT;
  const GemmVariant v = gemm_variant(split, Bp, T->L.nplane);
  const int64_t MT = T->Kp / GM, KB = T->Kp / GK, rows = MT * KB * (T->L.nplane / v.planes_per_unit) * 2 * GM;
  MT_CHECK(rows < ((int64_t)1 << 31), MT_EINVAL,
           "batched product: the dense tensor (n = %lld) exceeds the 32-bit TMA coordinate range", (long long)T->n);
  mt_status st;
  // blocked storage seen as a [units * 256][64] array and the operand as [terms * KB * 3 * Bp][64]
  if ((st = make_map(&plan->tA, T->d_data, GK, (uint64_t)rows, 2 * GM)) != MT_OK) return st;
  if ((st = make_map(&plan->tX, X, GK, (uint64_t)((split ? 9 : 3) * KB * Bp), (uint32_t)v.x_rows)) != MT_OK) return st;
  plan->B = B;
  plan->Bp = Bp;
  plan->split = split;
  plan->stages = v.stages;
  return MT_OK;
}

// The autotuner: per tensor and padded batch width, time the product for
// three ring depths (the deepest that fits in shared memory and one and two
// stages shallower) and keep the fastest; numerics do not depend on the choice.
mt_status gemm_tune(mt_tensor *T, GemmPlan *plan, float *H, float *part, int *count, int *status, cudaStream_t s) {
  int key = 0;
  while ((16 << key) < plan->Bp) ++key;
  if (T->gemm_stages[key] > 0) {
    plan->stages = T->gemm_stages[key];
    return MT_OK;
  }
  cudaEvent_t e0, e1;
  MT_CUDA(cudaEventCreate(&e0));
  MT_CUDA(cudaEventCreate(&e1));
  float best_ms = 1e30f;
  int best = plan->stages;
  const int smax = plan->stages;
  for (int st = smax; st >= std::max(2, smax - 2); --st) {
    plan->stages = st;
    launch_gemm(T, *plan, H, part, count, nullptr, status, s);  // warm
    MT_CUDA(cudaEventRecord(e0, s));
    for (int r = 0; r < 3; ++r) launch_gemm(T, *plan, H, part, count, nullptr, status, s);
    MT_CUDA(cudaEventRecord(e1, s));
    MT_CUDA(cudaEventSynchronize(e1));
    float ms = 0.0f;
    MT_CUDA(cudaEventElapsedTime(&ms, e0, e1));
    if (ms < best_ms) {
      best_ms = ms;
      best = st;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  MT_CUDA(cudaGetLastError());
  T->gemm_stages[key] = best;
  plan->stages = best;
  return MT_OK;
}

void launch_gemm(const mt_tensor *T, const GemmPlan &plan, float *H, float *part, int *count, const int *n_active,
                 int *status, cudaStream_t s) {
  const GemmVariant v = gemm_variant(plan.split, plan.Bp, T->L.nplane);
  GemmArgs P;
  P.n = T->n;
  P.MT = T->Kp / GM;
  P.KB = T->Kp / GK;
  P.B = plan.B;
  P.Bp = plan.Bp;
  P.stages = plan.stages;
  P.tmem_cols = v.tmem_cols;
  P.H = H;
  P.part = part;
  P.count = count;
  P.n_active = n_active;
  P.status = status;
  const int grid = gemm_grid(T, v.planes_per_unit);
  launch_pdl(v.kernel, dim3(grid), dim3(v.threads), plan.stages * v.stage_bytes + v.fixed_bytes, s, plan.tA,
             plan.tX, P);
}

}  // namespace mt
