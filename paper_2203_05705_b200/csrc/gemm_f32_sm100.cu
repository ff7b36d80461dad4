// fp32 layers on the tensor cores: every operand element is split into three bf16 numbers that add up to it,
// x = h + m + l (8 bits each, rounded to nearest, so 24 in all), and a product is taken as h h' + h m' + m h' + h l' + m m' + l h'.
// What is left out (m l', l m', l l') is below 2^-25 of |x y|, half of what rounding one fp32 product costs.  The
// tensor core truncates its sums, so the accumulators are taken out of tensor memory after every 64 contraction indices
// and added in fp32 registers, rounded to nearest, and h h' of a block's two halves has columns of its own: two truncations per
// sum instead of K / 16.  With four, operands of one sign, whose truncations add up, had a larger error than on the CUDA cores
// where those cut a contraction eight ways (512 x 384 x 512, uniform in 0 .. 1: 8.0e-8 against 6.1e-8, now 5.5e-8).
//
// One CTA per SM, 128 x 64 output tiles.  Warps 0..7 load (registers, the next block's piece requested as soon as this block's
// has been split) and write the six planes in the 128-byte-swizzled layout; warps 8 and 9 issue the products of the even and
// the odd blocks, each into accumulators of its own (an issued product costs its thread 136 cycles whatever its size, so one
// thread could not keep up); warps 10..13 take the accumulators out, add them up and write the tile.
// The three planes of B lie behind one another, so that one instruction multiplies a plane of A with up to all three:
//   A.h x [B.h B.m B.l] -> columns 0..191,  A.m x [B.h B.m] -> 64..191,  A.l x B.h -> 128..191;
// in the second half of a block A.h x B.h -> 192..255 and A.h x [B.m B.l] -> 64..191.
//
// Bound: shared memory.  A block (128 + 64 rows, 64 contraction indices) takes 48 KB through L1, 72 KB of stores of the planes
// and 106 KB of operand reads, 1810 cycles if all took turns at 128 bytes a cycle, next to 768 tensor-core cycles.  Measured 1724 (1024 x
// 4096 x 4096, forward), the threads' data pipe busy for 49 % of the time, the issue slots for 55 %, the tensor pipe for 39 %.
//
// Infinities, NaN and magnitudes that a bf16 cannot hold leave a NaN in l, and so in every sum they are part of.  Finite operands can
// leave an infinity or a NaN too where a product is near the largest fp32 number or beyond it: h h' may round past it, and h m'
// and m h' of an infinite product may have the other sign.  A tile whose sums are not all finite (its share of the contraction) is
// multiplied again on the CUDA cores.
//
// m and l of a small element would fall below the smallest bf16 (2^-133) and leave it with fewer bits: 2^-115 had an error of 1e-6,
// 2^-126 of 2e-3.  Operands are therefore taken times 2^16, which puts the last bit of the smallest fp32 number there, and the
// sums times 2^-32.  Elements from 2^111 on and sums from 2^96 on are not finite then, and are multiplied again.
#include "staged_product.h"

#include <math.h>

#include <type_traits>

namespace {

constexpr int F3_LOADERS = 256;
constexpr int F3_ISSUE_WARP = 8, F3_DRAIN_WARP = 10, F3_DRAINS = 4;
constexpr int F3_THREADS = 32 * (F3_DRAIN_WARP + F3_DRAINS);
constexpr int F3_BK = 64, F3_BN = 64;
constexpr int F3_A_PLANE = UMMA_BM * F3_BK * 2, F3_B_PLANE = F3_BN * F3_BK * 2;
constexpr int F3_STAGE = 3 * (F3_A_PLANE + F3_B_PLANE);
constexpr int F3_PITCH = F3_BN + 4;
constexpr int F3_TILE_OFF = 2 * F3_STAGE;
constexpr int AGAIN_K = 32, AGAIN_N = 32, AGAIN_PA = UMMA_BM + 4, AGAIN_PB = AGAIN_N + 4;  // multiply_again
constexpr int F3_AGAIN_OFF = F3_TILE_OFF + UMMA_BM * F3_PITCH * 4;
constexpr int F3_BAR_OFF = F3_AGAIN_OFF + AGAIN_K * (AGAIN_PA + AGAIN_PB) * 4;
constexpr int F3_SMEM = F3_BAR_OFF + 128 + 1024;
constexpr int F3_TMEM = 512;           // two blocks' accumulators of 4 * F3_BN columns each
constexpr double F3_LEAST_FLOPS = 1.5e8;  // kept operations, see f32_takes
constexpr float F3_UP = 65536.f, F3_DOWN = 1.f / (F3_UP * F3_UP);

struct F32Params {
  GemmArgs g;
  int ts;
  int cl;   // CTAs per cluster
  int vec;  // bit 0 / 1: rows of operand A / B start on 16-byte boundaries
};

// Four elements as two pairs; `pred`: zeros where it does not hold
struct Quad { uint64_t lo, hi; };
__device__ __forceinline__ Quad ld4(const float* p) {
  Quad v;
  asm volatile("ld.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.lo), "=l"(v.hi) : "l"(p));
  return v;
}
__device__ __forceinline__ Quad ld4(const float* p, bool pred) {
  Quad v;
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\tmov.b64 %0, 0;\n\tmov.b64 %1, 0;\n\t@p ld.global.v2.u64 {%0, %1}, [%2];\n\t}"
      : "=&l"(v.lo), "=&l"(v.hi) : "l"(p), "r"((int)pred));
  return v;
}
__device__ __forceinline__ float ld1(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ float ld1(const float* p, bool pred) {
  float v;
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\tmov.b32 %0, 0;\n\t@p ld.global.f32 %0, [%1];\n\t}"
               : "=&f"(v) : "l"(p), "r"((int)pred));
  return v;
}
__device__ __forceinline__ void sts8(uint32_t a, uint32_t x, uint32_t y) {
  asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ uint64_t pair(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint32_t round2(uint64_t x) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x));
  uint32_t h;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h) : "f"(b), "f"(a));
  return h;
}
// The pair rounded to bf16, and what that leaves of it (exact)
__device__ __forceinline__ uint32_t take_bf16(uint64_t& x) {
  const uint32_t h = round2(x);
  x = fma2(pair(__uint_as_float(h << 16), __uint_as_float(h & 0xffff0000u)), pair(-1.f, -1.f), x);
  return h;
}
__device__ __forceinline__ void split2(uint64_t x, uint32_t& h, uint32_t& m, uint32_t& l) {
  x = mul2(x, pair(F3_UP, F3_UP));
  h = take_bf16(x);
  m = take_bf16(x);
  l = round2(x);
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}

// Where operand elements are: r = position inside the tile, k = contraction index.
template <int KIND, int OP>
struct Operands {
  static constexpr bool A_MN = OP == OP_BWD_WEIGHT, B_MN = OP != OP_FWD;
  const float *PA, *PB;
  size_t ldb;
  int lda, step_a;          // step_a: columns of a full-width dY from one kept neuron to the next
  bool vec_a, vec_b;        // pieces of four contiguous elements are whole and on the 16-byte grid, or do not exist

  __device__ __forceinline__ Operands(const GemmArgs& g, const ProductPlan& s, int vec) {
    PA = reinterpret_cast<const float*>(g.A0);
    PB = reinterpret_cast<const float*>(g.A1);
    const bool strided_a = KIND == 0 && OP != OP_FWD && !g.flag0;
    lda = g.lda0;
    step_a = strided_a ? s.dp : 1;
    if (strided_a) PA += s.bb;
    // kept neurons are rows bb + i * dp of the weight (unless packed for a feeding pattern)
    const bool strided_b = KIND == 0 && OP != OP_BWD_WEIGHT && g.hdr_in == nullptr;
    ldb = strided_b ? (size_t)g.lda1 * s.dp : (size_t)g.lda1;
    if (strided_b) PB += (size_t)s.bb * g.lda1;
    const int along_a = KIND == 1 ? 0 : (A_MN ? s.M : s.K), along_b = KIND == 1 ? 0 : (B_MN ? s.N : s.K);
    vec_a = (vec & 1) && step_a == 1 && (along_a & 3) == 0;
    vec_b = (vec & 2) && (along_b & 3) == 0;
  }
  __device__ __forceinline__ int a_lim(const ProductPlan& s, const ProductTile& ti) const {
    return (KIND == 0 || OP != OP_BWD_WEIGHT ? s.M : ti.cnt * s.ts) - ti.m0;
  }
  __device__ __forceinline__ int b_lim(const ProductPlan& s, const ProductTile& ti) const {
    return (KIND == 0 ? s.N : (OP == OP_BWD_WEIGHT ? ti.len : ti.cnt) * s.ts) - ti.n0;
  }
  __device__ __forceinline__ const float* a(const ProductPlan& s, const ProductTile& ti, int r, int k) const {
    const int m = ti.m0 + r;
    if (KIND == 0) return PA + (A_MN ? (size_t)k * lda + (size_t)m * step_a : (size_t)m * lda + (size_t)k * step_a);
    return PA + (A_MN ? (size_t)k * lda + ti.class_pos(s, m) : (size_t)m * lda + ti.list_pos(s, k));
  }
  __device__ __forceinline__ const float* b(const ProductPlan& s, const ProductTile& ti, int r, int k) const {
    const int n = ti.n0 + r;
    if (KIND == 0) return PB + (B_MN ? (size_t)k * ldb + n : (size_t)n * ldb + k);
    if (OP == OP_FWD) return PB + (size_t)ti.class_pos(s, n) * ldb + ti.list_pos(s, k);
    if (OP == OP_BWD_DATA) return PB + (size_t)ti.list_pos(s, k) * ldb + ti.class_pos(s, n);
    return PB + (size_t)k * ldb + ti.list_pos(s, n);
  }
};

// True in all threads of the warps that add up if it is in any.
__device__ __forceinline__ bool any_drain(bool x) {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, 1, 128, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
               : "=r"(r) : "r"((uint32_t)x) : "memory");
  return r != 0;
}
__device__ __forceinline__ void sync_drain() { asm volatile("barrier.cta.sync 1, 128;" ::: "memory"); }

// The tile's sums over contraction indices [k0, k1) on the CUDA cores, for operands or sums that are not finite, into T, by the 128
// threads that add up (t: which of them): 32 columns at a time, 8 x 4 sums a thread, blocks of 32 indices of both operands through
// shared memory of its own at S.  Not more sums at a time: the registers of a function count for every warp of the kernel that calls
// it (64 a thread cost 128 x 2048 x 2048 1 us a product).  A training run that has diverged puts every tile through this (NaN in a
// column of each operand, 256 x 2048 x 2048, forward: 370 us; the CUDA-core kernel takes 76; a thread for a row's 64 sums, one
// after the other, took 4500).
template <int KIND, int OP>
__device__ __noinline__ void multiply_again(const Operands<KIND, OP>& o, const ProductPlan& s, const ProductTile& ti, int t, int k0, int k1,
                                            float* T, float* S) {
  using O = Operands<KIND, OP>;
  float* bB = S + AGAIN_K * AGAIN_PA;
  const int na = o.a_lim(s, ti), nb = o.b_lim(s, ti), r0 = t >> 3 << 3, c0 = (t & 7) << 2;
#pragma unroll 1
  for (int n0 = 0; n0 < F3_BN; n0 += AGAIN_N) {
    uint64_t acc[8][2] = {};
#pragma unroll 1
    for (int kk = k0; kk < k1; kk += AGAIN_K) {
      sync_drain();  // nobody reads the block before this one any more
      // eight elements on their way at a time: first those of A, then those of B
#pragma unroll 1
      for (int i0 = 0; i0 < AGAIN_K * (UMMA_BM + AGAIN_N) / 128; i0 += 8) {
        const bool is_a = i0 < AGAIN_K * UMMA_BM / 128;
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int e = (i0 + i) * 128 + t;
          if (is_a) {
            const int r = O::A_MN ? e & (UMMA_BM - 1) : e / AGAIN_K, k = kk + (O::A_MN ? e / UMMA_BM : e & (AGAIN_K - 1));
            v[i] = r < na && k < k1 ? ld1(o.a(s, ti, r, k)) : 0.f;
          } else {
            const int f = e - AGAIN_K * UMMA_BM, r = n0 + (O::B_MN ? f & (AGAIN_N - 1) : f / AGAIN_K), k = kk + (O::B_MN ? f / AGAIN_N : f & (AGAIN_K - 1));
            v[i] = r < nb && k < k1 ? ld1(o.b(s, ti, r, k)) : 0.f;
          }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int e = (i0 + i) * 128 + t, f = e - AGAIN_K * UMMA_BM;
          if (is_a) S[O::A_MN ? e / UMMA_BM * AGAIN_PA + (e & (UMMA_BM - 1)) : (e & (AGAIN_K - 1)) * AGAIN_PA + e / AGAIN_K] = v[i];
          else bB[O::B_MN ? f / AGAIN_N * AGAIN_PB + (f & (AGAIN_N - 1)) : (f & (AGAIN_K - 1)) * AGAIN_PB + f / AGAIN_K] = v[i];
        }
      }
      sync_drain();
#pragma unroll 2
      for (int k = 0; k < AGAIN_K; ++k) {
        const float4 x = *reinterpret_cast<const float4*>(S + k * AGAIN_PA + r0), y = *reinterpret_cast<const float4*>(S + k * AGAIN_PA + r0 + 4);
        const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(bB + k * AGAIN_PB + c0);
        const float a[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          acc[i][0] = fma2(pair(a[i], a[i]), w.x, acc[i][0]);
          acc[i][1] = fma2(pair(a[i], a[i]), w.y, acc[i][1]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) *reinterpret_cast<ulonglong2*>(T + (r0 + i) * F3_PITCH + n0 + c0) = make_ulonglong2(acc[i][0], acc[i][1]);
  }
}

template <int KIND, int OP>
__global__ void __launch_bounds__(F3_THREADS, 1) gemm_f32_kernel(const __grid_constant__ F32Params p) {
  using O = Operands<KIND, OP>;
  constexpr bool A_MN = O::A_MN, B_MN = O::B_MN;
  constexpr int NA = 8, NB = 4;  // four-element pieces per loading thread and block
  const GemmArgs& g = p.g;

  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t base = (raw_addr + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw_addr);
  const uint32_t bars = base + F3_BAR_OFF;
  // of half h of stage i and of accumulators i, i = block & 1: operands written; multiplied (for the loaders and, the second
  // half, for the warps that add up); added up
  auto full_bar = [&](int i, int h) { return bars + 8u * (2 * i + h); };
  auto done_bar = [&](int i, int h) { return bars + 8u * (4 + 2 * i + h); };
  auto free_bar = [&](int i) { return bars + 8u * (8 + i); };
  volatile uint32_t* tmem_ptr = reinterpret_cast<volatile uint32_t*>(smem + F3_BAR_OFF + 80);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + F3_BAR_OFF + 84);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  pdl_launch_dependents();
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      for (int h = 0; h < 2; ++h) {
        mbar_init(full_bar(i, h), F3_LOADERS / 64);
        mbar_init(done_bar(i, h), 1);
      }
      mbar_init(free_bar(i), F3_DRAINS);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == F3_ISSUE_WARP) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_ptr)), F3_TMEM);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_ptr;
  pdl_wait_prior_grids();

  const ProductPlan s = make_plan<KIND, OP, UMMA_BM, F3_BN, F3_BK>(g, p.ts, (int)gridDim.x, p.cl);
  const O o(g, s, p.vec);
  const int rank = (int)cluster_ctarank();
  const int lS = 31 - __clz(s.S), lG = 31 - __clz(s.G);
  const int part = rank & (s.S - 1);          // this CTA's share of the contraction
  const int lead = rank - part;               // first CTA of those that share it
  const int rows = rank & (s.G - 1);          // this CTA's part of the tile's rows
  const int group = rank >> lG, groups = p.cl >> lG;
  const int n_cl = (int)gridDim.x / p.cl, units = (s.tiles + groups - 1) / groups, u0 = (int)blockIdx.x / p.cl;

  // Unit u's tile and this CTA's blocks [kb0, kb1) of it; nkb < 0: nothing there.
  auto unit = [&](int u, int& kb0, int& kb1) {
    const int t = u * groups + group;
    ProductTile ti = {};
    ti.nkb = -1;
    if (t < s.tiles) ti = make_tile<KIND, OP, UMMA_BM, F3_BN, F3_BK>(g, s, t);
    kb0 = ti.nkb > 0 ? (ti.nkb * part) >> lS : 0;
    kb1 = ti.nkb > 0 ? (ti.nkb * (part + 1)) >> lS : 0;
    return ti;
  };
  float* T = reinterpret_cast<float*>(smem + F3_TILE_OFF);
  bool ok = true;

  if (warp < F3_ISSUE_WARP) {
    // ===================== loads =====================
    // Warps 0..3 bring the first half of every block (32 contraction indices), warps 4..7 the second: while one group waits for
    // its stage or its stores, the other splits.  A thread owns NA four-element pieces of A and NB of B.
    // K-major: 8 lanes read a row's 32 elements, piece i is row 16 i + r (the two rows of a half warp are four apart, so that
    // their halves of the 128-byte rows of the stage lie in different banks).  MN-major: 16 lanes read 64 columns of one
    // contraction row, piece i is row 8 (i & 3) + r of the half and, of A, box i / 4.
    const int h = warp >> 2, grp = (tid >> 3) & 15, kr = (grp >> 3) * 8 + (grp & 1) * 4 + ((grp >> 1) & 3);
    const int ra = A_MN ? (tid >> 4) & 7 : kr, rb = B_MN ? (tid >> 4) & 7 : kr;
    const int ca = 4 * (tid & (A_MN ? 15 : 7)), cb = 4 * (tid & (B_MN ? 15 : 7));
    ProductTile ti;
    int kb = 0, kb1 = 0, u = u0 - n_cl;     // the block in registers: block kb of unit u
    const float *ta[2] = {}, *tb[NB] = {};  // of the tile: see at()
    int na = 0, nb = 0;                     // K-major: rows that exist from the first piece's on; MN-major: columns
    Quad v[NA + NB];
    // Moves on to the next block; false: there is none.
    auto advance = [&]() {
      if (++kb < kb1) return true;
      for (;;) {
        u += n_cl;
        if (u >= units) return false;
        ti = unit(u, kb, kb1);
        if (kb < kb1) break;
      }
      na = o.a_lim(s, ti) - (A_MN ? ca : ra);
      nb = o.b_lim(s, ti) - (B_MN ? cb : rb);
      if (KIND == 0) {
        ta[0] = o.a(s, ti, A_MN ? ca : ra, A_MN ? ra : ca);
        tb[0] = o.b(s, ti, B_MN ? cb : rb, B_MN ? rb : cb);
      } else if (OP == OP_BWD_WEIGHT) {
#pragma unroll
        for (int i = 0; i < 2; ++i) ta[i] = o.PA + (size_t)ra * o.lda + (na > 64 * i ? ti.class_pos(s, ti.m0 + 64 * i + ca) : 0);
        tb[0] = o.PB + (size_t)rb * o.ldb + (nb > 0 ? ti.list_pos(s, ti.n0 + cb) : 0);
      } else {
        ta[0] = o.PA + (size_t)(ti.m0 + ra) * o.lda;
        if (OP == OP_FWD) {
#pragma unroll
          for (int i = 0; i < NB; ++i) tb[i] = o.PB + (size_t)(nb > 16 * i ? ti.class_pos(s, ti.n0 + 16 * i + rb) : 0) * o.ldb;
        } else {
          tb[0] = o.PB + (nb > 0 ? ti.class_pos(s, ti.n0 + cb) : 0);
        }
      }
      return true;
    };
    int kfirst = 0, kleft = 0;  // first contraction index of the half block, and how many there are from it on
    int kpos = 0;               // tile patterns: coordinate of contraction index kfirst + ca
    bool whole = false;         // every element of the half block exists
    auto begin_block = [&]() {
      kfirst = kb * F3_BK + 32 * h;
      kleft = ti.kext - kfirst;
      whole = kleft >= 32 && o.a_lim(s, ti) >= UMMA_BM && o.b_lim(s, ti) >= F3_BN;
      if (KIND == 1 && OP != OP_BWD_WEIGHT) kpos = ca < kleft ? ti.list_pos(s, kfirst + ca) : 0;
    };
    // Piece i: address, and whether / how many of its elements exist (<= 0: none).
    auto at = [&](int i, int& n) -> const float* {
      if (i < NA) {
        const int row = A_MN ? 8 * (i & 3) : 16 * i;
        if (A_MN) n = row + ra < kleft ? na - 64 * (i >> 2) : 0;
        else n = row < na ? kleft - ca : 0;
        if (KIND == 0) {
          if (A_MN) return ta[0] + (size_t)(kfirst + row) * o.lda + (size_t)((i >> 2) * 64) * o.step_a;
          return ta[0] + (size_t)row * o.lda + (size_t)kfirst * o.step_a;
        }
        if (A_MN) return ta[i >> 2] + (size_t)(kfirst + row) * o.lda;
        return ta[0] + (size_t)row * o.lda + kpos;
      }
      const int ib = i - NA, row = B_MN ? 8 * ib : 16 * ib;
      if (B_MN) n = row + rb < kleft ? nb : 0;
      else n = row < nb ? kleft - cb : 0;
      if (KIND == 0) return B_MN ? tb[0] + (size_t)(kfirst + row) * o.ldb : tb[0] + (size_t)row * o.ldb + kfirst;
      if (OP == OP_FWD) return tb[ib] + kpos;
      if (OP == OP_BWD_DATA) return tb[0] + (size_t)(row + rb < kleft ? ti.list_pos(s, kfirst + row + rb) : 0) * o.ldb;
      return tb[0] + (size_t)(kfirst + row) * o.ldb;
    };
    // VEC: 1 pieces on the 16-byte grid, 0 not, -1 to be looked at, and whether their elements exist too
    auto load = [&](auto vec, int i) {
      constexpr int VEC = decltype(vec)::value;
      int n;
      const float* q = at(i, n);
      const size_t st = i < NA ? o.step_a : 1;
      Quad& x = v[i];
      if (VEC == 1) {
        x = ld4(q);
      } else if (VEC == 0) {
        x.lo = pair(ld1(q), ld1(q + st));
        x.hi = pair(ld1(q + 2 * st), ld1(q + 3 * st));
      } else if (i < NA ? o.vec_a : o.vec_b) {
        x = ld4(q, n > 0);
      } else {
        x.lo = pair(ld1(q, n > 0), ld1(q + st, n > 1));
        x.hi = pair(ld1(q + 2 * st, n > 2), ld1(q + 3 * st, n > 3));
      }
    };
    auto place = [&](bool mn, int r, int c) {  // of piece 0
      const uint32_t d = (uint32_t)r * 128u + (uint32_t)(((c >> 3) ^ (r & 7)) << 4) + (uint32_t)(c & 4) * 2u;
      return base + (mn ? d + (uint32_t)h * 4096u : d ^ ((uint32_t)h * 64u));
    };
    const uint32_t pa = place(A_MN, ra, ca), pb = place(B_MN, rb, cb) + 3 * F3_A_PLANE;
    auto split = [&](int i, uint32_t stage) {
      uint32_t h0, m0, l0, h1, m1, l1;
      split2(v[i].lo, h0, m0, l0);
      split2(v[i].hi, h1, m1, l1);
      const int ib = i - NA;
      const uint32_t d = i < NA ? pa + stage + (uint32_t)(A_MN ? (i >> 2) * 8192 + (i & 3) * 1024 : i * 2048)
                                : pb + stage + (uint32_t)(B_MN ? ib * 1024 : ib * 2048);
      const uint32_t plane = i < NA ? F3_A_PLANE : F3_B_PLANE;
      sts8(d, h0, h1);
      sts8(d + plane, m0, m1);
      sts8(d + 2 * plane, l0, l1);
    };
    // The half block in registers goes to its stage while the next block's takes its place
    auto swap = [&](auto va, auto vb, uint32_t stage) {
#pragma unroll
      for (int i = 0; i < NA + NB; ++i) {
        split(i, stage);
        if (i < NA) load(va, i); else load(vb, i);
      }
    };
    using Yes = std::integral_constant<int, 1>;
    using No = std::integral_constant<int, 0>;
    using Look = std::integral_constant<int, -1>;
    int it = 0;
    bool more = advance();
    if (more) {
      begin_block();
#pragma unroll
      for (int i = 0; i < NA + NB; ++i) load(Look{}, i);
    }
    for (int w = u0; w < units; w += n_cl) {
      while (more && u == w && ok) {
        const int st = it & 1;
        const uint32_t stage = (uint32_t)st * F3_STAGE;
        more = advance();
        if (more) begin_block();
        else { whole = false; na = nb = kleft = 0; }  // nothing exists
        if (it >= 2 && !mbar_wait(done_bar(st, h), (uint32_t)((it >> 1) - 1) & 1u, abort_flag, g.status)) ok = false;
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        if (whole && o.vec_b && o.vec_a) swap(Yes{}, Yes{}, stage);
        else if (whole && o.vec_b) swap(No{}, Yes{}, stage);
        else if (whole && !o.vec_a) swap(No{}, No{}, stage);
        else swap(Look{}, Look{}, stage);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(full_bar(st, h));
        ++it;
      }
      __syncwarp();
      if (s.S > 1) {
        cluster_sync_all();  // the partial tiles of the group are complete
        int k0, k1;
        const ProductTile tw = unit(w, k0, k1);
        if (tw.nkb >= 0)
          write_tile<KIND, OP, UMMA_BM, F3_BN, F3_PITCH, F3_LOADERS / 32, true, float>(g, s, tw, T, base + F3_TILE_OFF, rows, lead, warp, lane);
        __syncwarp();
        cluster_sync_all();  // no CTA of the group reads this one's partial tile any more
      }
    }
  } else {
    const bool drain = warp >= F3_DRAIN_WARP;
    const int dw = warp - F3_DRAIN_WARP, quad = warp & 3;  // a warp reads the 32 lanes of tensor memory of its number modulo 4
    if (drain && OP == OP_BWD_WEIGHT && g.flag1 && s.dp > 1) {
      const int w = (int)blockIdx.x * F3_DRAINS + dw, ws = (int)gridDim.x * F3_DRAINS;
      if (KIND == 1) zero_dropped_tiles(g, p.ts, w, ws, lane);
      else zero_dropped_rows(g, s.N, w, ws, lane);
    }
    int it = 0;  // blocks of this CTA so far
    for (int u = u0; u < units; u += n_cl) {
      int kb0, kb1;
      const ProductTile ti = unit(u, kb0, kb1);
      if (!drain) {
        // ===================== products =====================
        const int mine = warp - F3_ISSUE_WARP;
        if (lane == 0 && ok) {
          const uint64_t desc_a = A_MN ? make_desc(0, 64 * F3_BK * 2, 1024) : make_desc(0, 16, 1024);
          const uint64_t desc_b = B_MN ? make_desc(0, 64 * F3_BK * 2, 1024) : make_desc(0, 16, 1024);
          const uint32_t sA = base + (uint32_t)mine * F3_STAGE, sB = sA + 3 * F3_A_PLANE;
          const uint64_t ad = desc_a | (uint64_t)((sA & 0x3FFFFu) >> 4), bd = desc_b | (uint64_t)((sB & 0x3FFFFu) >> 4);
          const uint32_t d = tmem + (uint32_t)mine * 256u;
          for (int b = it; b < it + kb1 - kb0; ++b) {
            if ((b & 1) != mine) continue;
            const uint32_t par = (uint32_t)(b >> 1) & 1u;
            if (!mbar_wait(free_bar(mine), par ^ 1u, abort_flag, g.status)) { ok = false; break; }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              if (!mbar_wait(full_bar(mine, h), par, abort_flag, g.status)) { ok = false; break; }
              tc_fence_after();
#pragma unroll
              for (int k = 2 * h; k < 2 * h + 2; ++k) {
                const uint64_t ak = ad + (uint64_t)(k * (A_MN ? 128 : 2)), bk = bd + (uint64_t)(k * (B_MN ? 128 : 2));
                if (h == 0) {
                  tc_mma_bf16(d, ak, bk, make_idesc(3 * F3_BN, A_MN, B_MN), k != 0 ? 1u : 0u);
                } else {
                  tc_mma_bf16(d + 3 * F3_BN, ak, bk, make_idesc(F3_BN, A_MN, B_MN), k != 2 ? 1u : 0u);
                  tc_mma_bf16(d + F3_BN, ak, bk + (F3_B_PLANE >> 4), make_idesc(2 * F3_BN, A_MN, B_MN), 1u);
                }
                tc_mma_bf16(d + F3_BN, ak + (F3_A_PLANE >> 4), bk, make_idesc(2 * F3_BN, A_MN, B_MN), 1u);
                tc_mma_bf16(d + 2 * F3_BN, ak + 2 * (F3_A_PLANE >> 4), bk, make_idesc(F3_BN, A_MN, B_MN), 1u);
              }
              tc_commit(done_bar(mine, h));
            }
            if (!ok) break;
          }
        }
        __syncwarp();
      } else if (ti.nkb >= 0) {
        // ===================== sums =====================
        uint64_t acc[F3_BN / 2];
#pragma unroll
        for (int i = 0; i < F3_BN / 2; ++i) acc[i] = 0ull;
        for (int b = it; b < it + kb1 - kb0 && ok; ++b) {
          const int i = b & 1;
          if (!mbar_wait(done_bar(i, 1), (uint32_t)(b >> 1) & 1u, abort_flag, g.status)) ok = false;
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          tc_fence_after();
          const uint32_t from = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)i * 256u;
#pragma unroll
          for (int cc = 0; cc < F3_BN; cc += 16) {
            uint32_t x[16], w[16], y[16], z[16];
            tmem_ld16(from + cc, x);
            tmem_ld16(from + 3 * F3_BN + cc, w);
            tmem_ld16(from + F3_BN + cc, y);
            tmem_ld16(from + 2 * F3_BN + cc, z);
            tmem_ld_wait();
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              auto two = [&](const uint32_t (&r)[16]) { return pair(__uint_as_float(r[2 * q]), __uint_as_float(r[2 * q + 1])); };
              acc[cc / 2 + q] = add2(acc[cc / 2 + q], add2(add2(two(x), two(w)), add2(two(y), two(z))));
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(free_bar(i));
        }
        float* row = T + (quad * 32 + lane) * F3_PITCH;
        uint64_t bad[4] = {};  // NaN once a sum is not finite, zero otherwise
#pragma unroll
        for (int i = 0; i < F3_BN / 2; ++i) bad[i & 3] = fma2(acc[i], 0ull, bad[i & 3]);
        if (any_drain((bad[0] | bad[1] | bad[2] | bad[3]) != 0ull)) {
          multiply_again(o, s, ti, tid - 32 * F3_DRAIN_WARP, kb0 * F3_BK, min(kb1 * F3_BK, ti.kext), T,
                         reinterpret_cast<float*>(smem + F3_AGAIN_OFF));
        } else {
#pragma unroll
          for (int i = 0; i < F3_BN / 4; ++i)
            *reinterpret_cast<ulonglong2*>(row + 4 * i) = make_ulonglong2(mul2(acc[2 * i], pair(F3_DOWN, F3_DOWN)), mul2(acc[2 * i + 1], pair(F3_DOWN, F3_DOWN)));
        }
        if (s.S == 1) sync_drain();
      }
      it += kb1 - kb0;
      __syncwarp();
      if (s.S > 1) {  // the loading warps, twice as many, add up the shares and write the tile
        cluster_sync_all();
        cluster_sync_all();
      } else if (drain && ti.nkb >= 0) {
        write_tile<KIND, OP, UMMA_BM, F3_BN, F3_PITCH, F3_DRAINS, true, float>(g, s, ti, T, base + F3_TILE_OFF, rows, lead, dw, lane);
        sync_drain();  // the tile has been read
        __syncwarp();
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == F3_ISSUE_WARP) {
    tc_fence_after();
    tmem_dealloc(tmem, F3_TMEM);
  }
}

inline int cdiv(int a, int b) { return (a + b - 1) / b; }

inline int cluster_size(const ard_ctx* ctx, int M, int N) { return (long long)cdiv(M, UMMA_BM) * cdiv(N, F3_BN) * 8 <= ctx->sm_count ? 8 : 4; }

// CTAs that the device holds at once in clusters of cl (all kernels here have the same registers, threads and shared memory)
int room(const ard_ctx* ctx, int cl) {
  static int known[2][64] = {};
  int& r = known[cl == 8][ctx->device & 63];
  if (r == 0) {
    auto kern = gemm_f32_kernel<0, OP_FWD>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, F3_SMEM) != cudaSuccess) (void)cudaGetLastError();
    r = ard_cluster_room(ctx, kern, cl, F3_THREADS, F3_SMEM);
  }
  return r;
}

// How make_plan cuts a product: blocks that a CTA takes one after the other, tiles among them, and blocks of all CTAs.
struct Cut { double serial, waves, total; };
Cut cut(double M, double N, double K, int BM, int BN, int BK, int places, int cl) {
  const double tiles = ceil(M / BM) * ceil(N / BN), nkb = ceil(K / BK);
  int S = cl;
  while (S > 1 && (tiles * S > places || nkb < 2 * S)) S >>= 1;
  const double waves = ceil(tiles * S / places), share = ceil(nkb / S);
  return {waves * share, waves, tiles * S * share};
}

template <int KIND, int OP>
ard_status launch_f32(ard_ctx* ctx, F32Params p, cudaStream_t s) {
  auto kern = gemm_f32_kernel<KIND, OP>;
  static bool attr_done[64] = {};
  const int dev = ctx->device & 63;
  if (!attr_done[dev]) {
    ARD_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, F3_SMEM));
    attr_done[dev] = true;
  }
  const GemmArgs& g = p.g;
  const int M = OP == OP_BWD_WEIGHT ? g.N : g.B, N = OP == OP_FWD ? g.N : g.K;
  const int nkb = cdiv(OP == OP_FWD ? g.K : (OP == OP_BWD_DATA ? g.N : g.B), F3_BK);
  const int tiles = cdiv(M, UMMA_BM) * cdiv(N, F3_BN);
  p.cl = cluster_size(ctx, M, N);
  int ctas = room(ctx, p.cl);
  if (KIND == 0) {  // no more than the densest pattern's tiles, cut as often as its contraction allows
    int S = p.cl;
    while (S > 1 && nkb < 2 * S) S >>= 1;
    const int n = cdiv(tiles * S, p.cl) * p.cl;
    if (n < ctas) ctas = n;
  }
  ARD_CUDA_OK(ard_launch_cluster(ctx, kern, p.cl, dim3(ctas), dim3(F3_THREADS), F3_SMEM, s, p));
  ctx->launches++;
  ARD_CUDA_OK(cudaGetLastError());
  return ARD_OK;
}

}  // namespace

// A product of up to 1.5e8 kept operations stays on the CUDA cores: about 5 us of every launch here go to the tables of the tile, the
// first loads and the way out, which the lighter kernel does faster.  Above, the rule is an estimate of both kernels' times from how
// they cut the product, its constants (us) fitted to 4400 products (batches of 16 to 4096, 128 to 4096 units, odd ones among
// them, periods of 1 to 16, both kinds of pattern, graph replays).  It is off by 14 % here and 11 % there (rms).
// Operations alone do not decide: a batch of 16 leaves a weight gradient a single block to a tile (16 x
// 4096 x 4096: 34 us there, 66 here), 94 tiles cannot be cut and leave 38 places idle (192 x 3000 x 3000, a period of 2, input gradient:
// 65, 79), columns of dY a period apart cost 8 sectors where one would do (512 x 3000 x 3000, a period of 16, weight gradient: 39, 80).
// Of 1452 others, operations alone made 135 slower than on the CUDA cores by a tenth and more, up to 2.2x, and this rule 20, up to 1.3x; the
// gain in the mean is 1.43x and 1.46x.  The margin of 5 % balances what is lost by being here (one in a hundred by a tenth) and there
// (two); a margin of a fifth 0.2 and 9.
// Three products of a dense layer, CUDA cores and here: 128 x 2048 x 2048 105 and 62 us, 1024 x 4096 x 4096 2730 and 951.
// Error against fp64 (2-norm) there and here, 12 shapes with contractions of 64 to 4096: operands of both signs 1.5e-7 .. 4.1e-7 and
// 5.4e-8 .. 1.0e-7, of one sign 6.1e-8 .. 2.5e-7 and 3.1e-8 .. 6.5e-8; at most 0.9 of the CUDA cores' in each.
bool f32_takes(const ard_ctx* ctx, ard_kind kind, GemmOp op, const GemmArgs& g, int ts) {
  if (ctx->path != ARD_PATH_AUTO || ctx->encode_fn == nullptr || g.B < 1 || g.K < 1 || g.N < 1) return false;
  if (kind == ARD_TILE && ts % 4 != 0) return false;  // four consecutive positions never leave a pattern tile
  const double kept = 2.0 * g.B * g.K * g.N * g.keep;
  if (kept < F3_LEAST_FLOPS) return false;
  const bool row = kind == ARD_ROW;
  const double n = row ? ceil(g.N * (double)g.keep) : g.N, keep_tile = row ? 1.0 : g.keep;
  const double M = op == OP_BWD_WEIGHT ? n : g.B, N = op == OP_FWD ? n : g.K * (op == OP_BWD_WEIGHT ? keep_tile : 1.0);
  const double K = op == OP_FWD ? g.K * keep_tile : (op == OP_BWD_DATA ? n * keep_tile : g.B);
  const int cl = cluster_size(ctx, op == OP_BWD_WEIGHT ? g.N : g.B, op == OP_FWD ? g.N : g.K);
  const Cut tc = cut(M, N, K, UMMA_BM, F3_BN, F3_BK, room(ctx, cl), cl), cc = cut(M, N, K, 64, 64, 16, 4 * ctx->sm_count, 8);
  const double cc_blocks = cc.total / (4 * ctx->sm_count);
  // columns of dY, a period apart (up to 8 elements to a sector) unless a compact copy will be read; zeros of dropped outputs, in MB
  const bool dropped = row && g.keep < 1.f, full_dy = op != OP_FWD && !g.flag0;
  const double apart = dropped && full_dy && kept < F32_COMPACT_FLOPS ? fmin(1.0 / g.keep, 8.0) - 1.0 : 0.0;
  const double mb_fwd = dropped && op == OP_FWD && g.flag0 == ARD_OUT_SCATTER_ZEROFILL ? 4e-6 * g.B * g.N : 0.0;
  const double mb_dw = op == OP_BWD_WEIGHT ? 4e-6 * g.N * g.K : 0.0;
  // contiguous pieces off the 16-byte grid
  auto off = [](const void* p, int ld, int along) { return ((reinterpret_cast<uintptr_t>(p) & 15) != 0 || ld % 4 != 0 || along % 4 != 0) ? 1.0 : 0.0; };
  const double off_a = row && apart == 0.0 ? off(g.A0, g.lda0, op == OP_FWD ? g.K : g.N) : 0.0;
  const double off_b = row ? off(g.A1, g.lda1, g.K) : 0.0;
  const double tc_off = op == OP_FWD ? 0.2 * off_a : (op == OP_BWD_DATA ? 0.55 * off_a + 0.15 * off_b : 0.9 * off_a + 0.3 * off_b);
  const double cc_off = op == OP_FWD ? 0.7 * off_a : 0.13 * (off_a + off_b);
  const double t_tc = 7.4 + 1.4 * tc.waves + tc.serial * (1.55 + 0.44 * apart + tc_off) + 1.3 * mb_fwd + 0.19 * mb_dw;
  const double t_cc = 7.4 + 0.74 * cc.serial + cc_blocks * (1.45 + 0.2 * apart + cc_off) + 0.36 * mb_fwd + 0.14 * mb_dw;
  return 1.05 * t_tc < t_cc;
}

ard_status launch_gemm_f32(ard_ctx* ctx, ard_kind kind, GemmOp op, const GemmArgs& g, int ts, cudaStream_t s) {
  F32Params p = {};
  p.g = g;
  p.ts = ts;
  p.vec = ((reinterpret_cast<uintptr_t>(g.A0) & 15) == 0 && g.lda0 % 4 == 0 ? 1 : 0) |
          ((reinterpret_cast<uintptr_t>(g.A1) & 15) == 0 && g.lda1 % 4 == 0 ? 2 : 0);
  if (kind == ARD_ROW) {
    if (op == OP_FWD) return launch_f32<0, OP_FWD>(ctx, p, s);
    if (op == OP_BWD_DATA) return launch_f32<0, OP_BWD_DATA>(ctx, p, s);
    return launch_f32<0, OP_BWD_WEIGHT>(ctx, p, s);
  }
  if (op == OP_FWD) return launch_f32<1, OP_FWD>(ctx, p, s);
  if (op == OP_BWD_DATA) return launch_f32<1, OP_BWD_DATA>(ctx, p, s);
  return launch_f32<1, OP_BWD_WEIGHT>(ctx, p, s);
}
