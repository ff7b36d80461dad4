// CUDA-core family of the compacted GEMMs: fp32 (or bf16) operands, fp32 FFMA accumulation.
//
// This is the path of the smaller fp32 layers (the larger ones: gemm_f32_sm100.cu) and the fall-back for bf16 shapes whose alignment no tensor-core kernel can take.
// One shared-memory tiled kernel; what differs per product is only how the logical operand element (m, k), (n, k)
// maps to memory and which contraction indices exist: dropped neurons / tiles are skipped through the pattern,
// never multiplied by zero.  Tiling, cut contractions and the rows' way out: staged_product.h.
#include "staged_product.h"

namespace {

template <typename T> __device__ __forceinline__ float to_f(T v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

__device__ __forceinline__ void store_out(void* out, size_t off, float v, int out_is_f32, int accumulate = 0) {
  if (out_is_f32) {
    float* p = reinterpret_cast<float*>(out) + off;
    *p = accumulate ? *p + v : v;
  } else {
    __nv_bfloat16* p = reinterpret_cast<__nv_bfloat16*>(out) + off;
    *p = __float2bfloat16_rn(accumulate ? __bfloat162float(*p) + v : v);
  }
}

// Four consecutive elements at p as fp32; the address is a multiple of four elements.
__device__ __forceinline__ float4 load4(const float* p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
  uint32_t a, b;
  asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(a), "=r"(b) : "l"(p));
  return make_float4(__uint_as_float(a << 16), __uint_as_float(a & 0xffff0000u), __uint_as_float(b << 16), __uint_as_float(b & 0xffff0000u));
}

__host__ __device__ constexpr int cc_threads(int R) { return R == 64 ? 128 : 64; }
constexpr int CC_CLUSTER = 8;
constexpr double CC_WIDE_FLOPS = 2e8;  // 64 x 64 tiles from here on, see launch_one
struct CcParams {
  GemmArgs g;
  int ts;
  int want;      // CTAs the device has room for at once
  int vec;       // bit 0 / 1: rows of operand A / B start on four-element boundaries
};

__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void fma2(uint64_t& d, uint64_t a, uint64_t b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b)); }

// A call, not inlined: inlined, the loops take registers from the product's (4096 x 33 x 4096 in fp32, a dense draw, 63 -> 79 us).
template <int KIND>
__device__ __noinline__ void cc_zeros(const GemmArgs& g, int ts, int cols, int warps) {
  const int warp = (int)blockIdx.x * warps + ((int)threadIdx.x >> 5), all = (int)gridDim.x * warps, lane = threadIdx.x & 31;
  if (KIND == 1) zero_dropped_tiles(g, ts, warp, all, lane);
  else zero_dropped_rows(g, cols, warp, all, lane);
}

// R: rows and columns of the output tile (64 or 32); a thread of the R / 4 x 8 grid owns 4 rows by R / 8 columns of it,
// multiplied two columns an instruction.  The operands of a KT-deep block are staged k-major as fp32, [k][row], through registers, one block ahead of the
// products.  KIND: 0 row, 1 tile.  OP: GemmOp.
// Bound: FFMA issue for the 64 x 64 tile (32 FFMA per three 16-byte shared-memory reads and thread), latency for the
// 32 x 32 one, which is for products that would otherwise occupy a few SMs.
template <typename T, int KIND, int OP, int R>
__global__ void __launch_bounds__(cc_threads(R)) gemm_cc_kernel(const __grid_constant__ CcParams p) {
  constexpr int CC_THREADS = cc_threads(R), KT = R == 64 ? 16 : 32, Q = R / 8, PITCH = R + 4;
  constexpr bool A_MN = OP == OP_BWD_WEIGHT, B_MN = OP != OP_FWD;
  constexpr int NCH = R * KT / 4 / CC_THREADS;  // four-element pieces per thread, operand and block
  __shared__ __align__(16) float sm[4 * KT * PITCH];  // [buffer][operand][k][row]; the finished tile overlays it
  static_assert(R <= 4 * KT, "the tile overlays the stages");
  const GemmArgs& g = p.g;
  // No __restrict__ / read-only loads on anything an earlier kernel of the stream wrote: this kernel may
  // become resident before that kernel has finished (see pdl_wait_prior_grids), and the non-coherent
  // load path may then serve a line another resident kernel brought in before the data was rewritten.
  pdl_launch_dependents();
  pdl_wait_prior_grids();

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, tx = tid & 7, ty = tid >> 3;
  const ProductPlan s = make_plan<KIND, OP, R, R, KT>(g, p.ts, p.want, CC_CLUSTER);
  const int rank = (int)cluster_ctarank();
  const int part = rank & (s.S - 1), lead = rank - part;
  const int group = rank / s.S, groups = CC_CLUSTER / s.S;
  const int n_cl = (int)gridDim.x / CC_CLUSTER, units = (s.tiles + groups - 1) / groups;
  const T* PA = reinterpret_cast<const T*>(g.A0);
  const T* PB = reinterpret_cast<const T*>(g.A1);
  // Kept neurons are bb + i * dp: columns of a full-width dY, rows of the weight (unless packed for a feeding pattern).
  const bool strided_a = KIND == 0 && OP != OP_FWD && !g.flag0;
  const size_t step_a = strided_a ? (size_t)s.dp : 1, off_a = strided_a ? (size_t)s.bb : 0;
  const bool strided_b = KIND == 0 && OP != OP_BWD_WEIGHT && g.hdr_in == nullptr;
  const size_t ldb = strided_b ? (size_t)g.lda1 * s.dp : (size_t)g.lda1;
  if (strided_b) PB += (size_t)s.bb * g.lda1;
  const bool whole = KIND == 0 || (p.ts & 3) == 0;  // four consecutive positions never leave a pattern tile
  const bool vec_a = (p.vec & 1) && step_a == 1 && whole, vec_b = (p.vec & 2) && whole;

  // Rows: dealt to all warps by the small tile where the contraction is not cut; else each row's zeros are left to the CTAs of
  // its tile (fp32, weight gradient, dealt and left: 16 x 2047 -> 2045, a period of 3, 15 and 23 us; 2000 x 129 -> 2047 39
  // and 30; and the call alone costs the large tile's loop 2 % and more).
  if (OP == OP_BWD_WEIGHT && g.flag1 && s.dp > 1 && (KIND == 1 || (R == 32 && s.S == 1))) cc_zeros<KIND>(g, p.ts, KIND == 0 ? s.N : 0, CC_THREADS / 32);
  for (int u = (int)blockIdx.x / CC_CLUSTER; u < units; u += n_cl) {
    const int t = u * groups + group;
    ProductTile ti = {};
    ti.nkb = -1;
    if (t < s.tiles) ti = make_tile<KIND, OP, R, R, KT>(g, s, t);
    const bool live = ti.nkb >= 0;
    const int kb0 = live ? (int)((long long)ti.nkb * part / s.S) : 0;
    const int kb1 = live ? (int)((long long)ti.nkb * (part + 1) / s.S) : 0;

    // Element offsets of operand elements; r = row inside the tile, k = contraction index.
    auto a_off = [&](int r, int k) -> size_t {
      const int m = ti.m0 + r;
      if (KIND == 0) return A_MN ? (size_t)k * g.lda0 + off_a + (size_t)m * step_a : (size_t)m * g.lda0 + off_a + (size_t)k * step_a;
      return A_MN ? (size_t)k * g.lda0 + ti.class_pos(s, m) : (size_t)m * g.lda0 + ti.list_pos(s, k);
    };
    auto b_off = [&](int r, int k) -> size_t {
      const int n = ti.n0 + r;
      if (KIND == 0) return B_MN ? (size_t)k * ldb + n : (size_t)n * ldb + k;
      if (OP == OP_FWD) return (size_t)ti.class_pos(s, n) * ldb + ti.list_pos(s, k);
      if (OP == OP_BWD_DATA) return (size_t)ti.list_pos(s, k) * ldb + ti.class_pos(s, n);
      return (size_t)k * ldb + ti.list_pos(s, n);
    };
    const int a_lim = (KIND == 0 || OP != OP_BWD_WEIGHT ? s.M : ti.cnt * s.ts) - ti.m0;
    const int b_lim = (KIND == 0 ? s.N : (OP == OP_BWD_WEIGHT ? ti.len : ti.cnt) * s.ts) - ti.n0;

    float4 va[NCH], vb[NCH];
    // Piece i of this thread: four k of one row (K-major) or four rows of one k (MN-major).
    auto load = [&](int kb) {
      const int kbase = kb * KT;
#pragma unroll
      for (int i = 0; i < NCH; ++i) {
        const int id = tid + i * CC_THREADS;
        auto fetch = [&](const T* P, bool mn, bool vec, int lim, auto off) {
          const int r = mn ? 4 * (id % (R / 4)) : id / (KT / 4), k = kbase + (mn ? id / (R / 4) : 4 * (id % (KT / 4)));
          const int n = mn ? (k < ti.kext ? lim - r : 0) : (r < lim ? ti.kext - k : 0);  // elements that exist
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          if (vec && n >= 4) {
            v = load4(P + off(r, k));
          } else {
            if (n > 0) v.x = to_f<T>(P[off(r, k)]);
            if (n > 1) v.y = to_f<T>(P[mn ? off(r + 1, k) : off(r, k + 1)]);
            if (n > 2) v.z = to_f<T>(P[mn ? off(r + 2, k) : off(r, k + 2)]);
            if (n > 3) v.w = to_f<T>(P[mn ? off(r + 3, k) : off(r, k + 3)]);
          }
          return v;
        };
        va[i] = fetch(PA, A_MN, vec_a, a_lim, a_off);
        vb[i] = fetch(PB, B_MN, vec_b, b_lim, b_off);
      }
    };
    auto stage = [&](int buf) {
      float* SA = sm + buf * 2 * KT * PITCH;
      float* SB = SA + KT * PITCH;
#pragma unroll
      for (int i = 0; i < NCH; ++i) {
        const int id = tid + i * CC_THREADS;
        auto put = [&](float* S, bool mn, const float4& v) {
          if (mn) {
            *reinterpret_cast<float4*>(S + (id / (R / 4)) * PITCH + 4 * (id % (R / 4))) = v;
          } else {
            float* d = S + 4 * (id % (KT / 4)) * PITCH + id / (KT / 4);
            d[0] = v.x; d[PITCH] = v.y; d[2 * PITCH] = v.z; d[3 * PITCH] = v.w;
          }
        };
        put(SA, A_MN, va[i]);
        put(SB, B_MN, vb[i]);
      }
    };

    uint64_t acc[4][Q / 2];  // column pairs
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < Q / 2; ++j) acc[i][j] = 0ull;
    if (kb1 > kb0) {
      load(kb0);
      stage(0);
      __syncthreads();
      for (int kb = kb0; kb < kb1; ++kb) {
        const int buf = (kb - kb0) & 1;
        const bool more = kb + 1 < kb1;
        if (more) load(kb + 1);
        const float* SA = sm + buf * 2 * KT * PITCH;
        const float* SB = SA + KT * PITCH;
#pragma unroll
        for (int k = 0; k < KT; ++k) {
          const float4 a = *reinterpret_cast<const float4*>(SA + k * PITCH + 4 * ty);
          const uint64_t a2[4] = {pack2(a.x, a.x), pack2(a.y, a.y), pack2(a.z, a.z), pack2(a.w, a.w)};
#pragma unroll
          for (int h = 0; h < Q / 4; ++h) {
            const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(SB + k * PITCH + 32 * h + 4 * tx);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              fma2(acc[i][2 * h], a2[i], b.x);
              fma2(acc[i][2 * h + 1], a2[i], b.y);
            }
          }
        }
        if (more) stage(buf ^ 1);
        __syncthreads();
      }
    }
    if (live) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int h = 0; h < Q / 4; ++h)
          *reinterpret_cast<ulonglong2*>(sm + (4 * ty + i) * PITCH + 32 * h + 4 * tx) = make_ulonglong2(acc[i][2 * h], acc[i][2 * h + 1]);
    }
    if (s.S > 1) cluster_sync_all();  // the partial tiles of the group are complete
    else __syncthreads();
    if (live) write_tile<KIND, OP, R, R, PITCH, CC_THREADS / 32, false, T>(g, s, ti, sm, smem_u32(sm), part, lead, warp, lane);
    __syncwarp();
    if (s.S > 1) cluster_sync_all();  // no CTA of the group reads this one's partial tile any more
    else __syncthreads();
  }
}

// ---- layers with at most 16 neurons (an output layer) -----------------------------------------------
// The tiled kernel above would give such a layer a handful of CTAs, each walking the whole fan-in alone.
// Forward: one CTA per batch row; every thread walks a strided share of the fan-in with one accumulator
// per kept neuron, then the CTA adds the shares (fixed order).  Backward-weight: 32 fan-in columns per CTA,
// the batch rows dealt to its 8 warps, one accumulator per kept neuron, warp sums added in warp order.
constexpr int SKINNY_N = ARD_SKINNY_N;

template <typename T>
__global__ void __launch_bounds__(256) skinny_fwd_kernel(GemmArgs g) {
  __shared__ float part[8][SKINNY_N];
  pdl_launch_dependents();
  pdl_wait_prior_grids();
  const int n_keep = g.hdr[HDR_NKEEP];
  const int kin = g.hdr_in != nullptr ? g.hdr_in[HDR_NKEEP] : g.K;
  const int m = blockIdx.x;
  const T* X = reinterpret_cast<const T*>(g.A0) + (size_t)m * g.lda0;
  const T* W = reinterpret_cast<const T*>(g.A1);
  float acc[SKINNY_N];
#pragma unroll
  for (int n = 0; n < SKINNY_N; ++n) acc[n] = 0.f;
  int rows[SKINNY_N];
#pragma unroll
  for (int n = 0; n < SKINNY_N; ++n) rows[n] = n < n_keep ? (g.hdr_in != nullptr ? n : g.idx[n]) : 0;
  for (int k = threadIdx.x; k < kin; k += 256) {
    const float x = to_f<T>(X[k]);
#pragma unroll
    for (int n = 0; n < SKINNY_N; ++n)
      if (n < n_keep) acc[n] = fmaf(x, to_f<T>(W[(size_t)rows[n] * g.lda1 + k]), acc[n]);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int n = 0; n < SKINNY_N; ++n) {
    float v = acc[n];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) part[warp][n] = v;
  }
  __syncthreads();
  if (threadIdx.x < n_keep) {
    const int n = threadIdx.x;
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) v += part[w][n];
    if (g.bias != nullptr) v += g.bias[g.idx[n]];
    if (g.relu) v = fmaxf(v, 0.f);
    v *= g.alpha;
    const size_t off = (size_t)m * g.ldo + (g.flag0 == ARD_OUT_SCATTER_ZEROFILL ? g.idx[n] : n);
    store_out(g.out, off, v, g.out_is_f32, g.accumulate);
  }
  if (g.flag0 == ARD_OUT_SCATTER_ZEROFILL && threadIdx.x >= 32 && threadIdx.x < 32 + g.N) {
    // full-width output: the dropped neurons' entries of this row are zero (no separate clearing pass)
    const int o = threadIdx.x - 32, dp = g.hdr[HDR_DP], bb = g.hdr[HDR_B] - 1;
    if (!(o >= bb && (o - bb) % dp == 0)) store_out(g.out, (size_t)m * g.ldo + o, 0.f, g.out_is_f32);
  }
}

template <typename T>
__global__ void __launch_bounds__(256) skinny_bwd_weight_kernel(GemmArgs g) {
  // 32 fan-in columns per CTA; its 8 warps take every eighth batch row and their sums are added in warp order
  __shared__ float part[8][SKINNY_N][33];
  pdl_launch_dependents();
  pdl_wait_prior_grids();
  const int n_keep = g.hdr[HDR_NKEEP];
  const int kin = g.hdr_in != nullptr ? g.hdr_in[HDR_NKEEP] : g.K;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int k = blockIdx.x * 32 + lane;
  if (blockIdx.x * 32 >= kin) return;
  const T* dY = reinterpret_cast<const T*>(g.A0);
  const T* X = reinterpret_cast<const T*>(g.A1);
  int cols[SKINNY_N];
#pragma unroll
  for (int n = 0; n < SKINNY_N; ++n) cols[n] = n < n_keep ? (g.flag0 ? n : g.idx[n]) : 0;
  float acc[SKINNY_N];
#pragma unroll
  for (int n = 0; n < SKINNY_N; ++n) acc[n] = 0.f;
  if (k < kin) {
#pragma unroll 4
    for (int r = warp; r < g.B; r += 8) {
      const float x = to_f<T>(X[(size_t)r * g.lda1 + k]);
      const T* dy = dY + (size_t)r * g.lda0;
#pragma unroll
      for (int n = 0; n < SKINNY_N; ++n)
        if (n < n_keep) acc[n] = fmaf(to_f<T>(dy[cols[n]]), x, acc[n]);
    }
  }
#pragma unroll
  for (int n = 0; n < SKINNY_N; ++n) part[warp][n][lane] = acc[n];
  __syncthreads();
  // 32 columns x up to 16 neurons = up to 512 outputs for 256 threads
  for (int o = threadIdx.x; o < 32 * n_keep; o += 256) {
    const int n = o >> 5, c = o & 31;
    const int kk = blockIdx.x * 32 + c;
    if (kk >= kin) continue;
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) v += part[w][n][c];
    store_out(g.out, (size_t)(g.hdr_in != nullptr ? n : g.idx[n]) * g.ldo + kk, g.alpha * v, g.out_is_f32, g.accumulate);
  }
  if (g.flag1) {
    // rows of dropped neurons, this CTA's 32 columns
    const int dp = g.hdr[HDR_DP], bb = g.hdr[HDR_B] - 1;
    for (int o = threadIdx.x; o < 32 * g.N; o += 256) {
      const int row = o >> 5, kk = blockIdx.x * 32 + (o & 31);
      if (kk < kin && !(row >= bb && (row - bb) % dp == 0)) store_out(g.out, (size_t)row * g.ldo + kk, 0.f, g.out_is_f32);
    }
  }
}

inline int cdiv(int a, int b) { return (a + b - 1) / b; }

template <typename T, int KIND, int OP>
void launch_one(const ard_ctx* ctx, const GemmArgs& g, int ts, cudaStream_t s) {
  CcParams p = {};
  p.g = g;
  p.ts = ts;
  const uintptr_t four = 4 * sizeof(T) - 1;
  p.vec = ((reinterpret_cast<uintptr_t>(g.A0) & four) == 0 && g.lda0 % 4 == 0 ? 1 : 0) |
          ((reinterpret_cast<uintptr_t>(g.A1) & four) == 0 && g.lda1 % 4 == 0 ? 2 : 0);
  const int M = OP == OP_BWD_WEIGHT ? g.N : g.B, N = OP == OP_FWD ? g.N : g.K;
  const double flops = 2.0 * g.B * g.K * g.N;
  // The grid covers the tiles of the densest pattern, cut or not; CTAs without work read the header and leave.
  auto launch = [&](auto kern, int R, int KT) {
    const int tiles = cdiv(M, R) * cdiv(N, R);
    p.want = 4 * ctx->sm_count;
    int n = min(16 * ctx->sm_count, max(p.want, tiles));
    if (KIND == 0) {  // no pattern cuts a tile into more shares than its longest contraction allows
      const int nkb = cdiv(OP == OP_FWD ? g.K : (OP == OP_BWD_DATA ? g.N : g.B), KT);
      int S = CC_CLUSTER;
      while (S > 1 && nkb < 2 * S) S >>= 1;
      n = min(n, tiles * S);
    }
    (void)ard_launch_cluster(ctx, kern, CC_CLUSTER, dim3(cdiv(n, CC_CLUSTER) * CC_CLUSTER), dim3(cc_threads(R)), 0, s, p);
  };
  if (flops > CC_WIDE_FLOPS) launch(gemm_cc_kernel<T, KIND, OP, 64>, 64, 16);
  else launch(gemm_cc_kernel<T, KIND, OP, 32>, 32, 32);
}  // errors: cudaGetLastError

template <typename T>
void dispatch(const ard_ctx* ctx, ard_kind kind, GemmOp op, const GemmArgs& a, int ts, cudaStream_t s) {
  if (kind == ARD_ROW) {
    if (op == OP_FWD) launch_one<T, 0, OP_FWD>(ctx, a, ts, s);
    else if (op == OP_BWD_DATA) launch_one<T, 0, OP_BWD_DATA>(ctx, a, ts, s);
    else launch_one<T, 0, OP_BWD_WEIGHT>(ctx, a, ts, s);
  } else {
    if (op == OP_FWD) launch_one<T, 1, OP_FWD>(ctx, a, ts, s);
    else if (op == OP_BWD_DATA) launch_one<T, 1, OP_BWD_DATA>(ctx, a, ts, s);
    else launch_one<T, 1, OP_BWD_WEIGHT>(ctx, a, ts, s);
  }
}

}  // namespace

ard_status launch_gemm_cc(ard_ctx* ctx, ard_kind kind, GemmOp op, ard_dtype dtype, const GemmArgs& a, int ts,
                          cudaStream_t s) {
  if ((a.B == 0 && op != OP_BWD_WEIGHT) || a.K == 0 || a.N == 0) return ARD_OK;
  if (kind == ARD_ROW && a.N <= SKINNY_N && op == OP_FWD && a.B > 0) {
    if (dtype == ARD_F32) (void)ard_launch(ctx, skinny_fwd_kernel<float>, dim3(a.B), dim3(256), 0, s, a);
    else (void)ard_launch(ctx, skinny_fwd_kernel<__nv_bfloat16>, dim3(a.B), dim3(256), 0, s, a);
  } else if (kind == ARD_ROW && a.N <= SKINNY_N && op == OP_BWD_WEIGHT) {
    if (dtype == ARD_F32) (void)ard_launch(ctx, skinny_bwd_weight_kernel<float>, dim3((a.K + 31) / 32), dim3(256), 0, s, a);
    else (void)ard_launch(ctx, skinny_bwd_weight_kernel<__nv_bfloat16>, dim3((a.K + 31) / 32), dim3(256), 0, s, a);
  } else if (dtype == ARD_F32 && f32_takes(ctx, kind, op, a, ts)) {
    return launch_gemm_f32(ctx, kind, op, a, ts, s);
  } else if (dtype == ARD_F32) {
    dispatch<float>(ctx, kind, op, a, ts, s);
  } else {
    dispatch<__nv_bfloat16>(ctx, kind, op, a, ts, s);
  }
  ctx->launches++;
  ARD_CUDA_OK(cudaGetLastError());
  return ARD_OK;
}
