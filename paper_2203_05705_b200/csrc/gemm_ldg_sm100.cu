// tcgen05 products whose operands no TMA descriptor can describe (bf16 operands, fp32 accumulation in tensor
// memory): rows that do not start on 16-byte boundaries (a fan-in of 1500, an odd width), periods beyond the
// TMA kernels' table, and pattern tiles narrower than the 64 columns of a swizzle row (the paper's 32 x 32 tiles).
//
// The CTA's own threads stage the operands in the 128-byte-swizzled layout that tcgen05.mma reads, a ninth warp issues
// the products.  Rows on the 4-, 8- or 16-byte grid are copied with asynchronous copies of that size, several blocks
// ahead.  An odd width puts every second row between two elements of that grid: such rows are read into registers as
// the aligned 16-byte units that cover them, one block ahead, and shifted into place with one exchange between
// neighbouring lanes.
// Tiling, cut contractions and the rows' way out: staged_product.h.
//
// Bound: the load unit and the latency of its copies (two CTAs share an SM); the tensor
// pipe is nearly idle.  Three products of a layer, against the CUDA-core kernel that took these shapes before:
// 700 x 1500 x 1500 under a row pattern of period 2 465 -> 69 us, 128 x 2048 x 2048 under 32 x 32 tiles of period 2
// 519 -> 49 us (with the sampler's launch).
#include "staged_product.h"

namespace {

constexpr int LG_LOADERS = 256;             // warps 0..7: loads, then the epilogue
constexpr int LG_THREADS = LG_LOADERS + 32; // warp 8: tensor memory, products
constexpr int LG_BK = 64;

struct LdgParams {
  GemmArgs g;
  int ts;
  int cl;  // CTAs per cluster
};

template <int BN>
struct LdgSmem {
  static constexpr int STAGES = BN == 64 ? 4 : 3;
  static constexpr int A_BYTES = UMMA_BM * LG_BK * 2;
  static constexpr int B_BYTES = BN * LG_BK * 2;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int PITCH = BN + 4;  // words per row of the fp32 tile (overlays the stages between two tiles)
  static constexpr int BAR_OFF = STAGES * STAGE_BYTES;
  static constexpr int TOTAL = BAR_OFF + 128 + 1024;
  static_assert(UMMA_BM * PITCH * 4 <= BAR_OFF, "the fp32 tile overlays the operand stages");
};

__device__ __forceinline__ uint4 ldg16(uintptr_t a, bool pred) {
  uint4 v;
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %5, 0;\n\tmov.b32 %0, 0;\n\tmov.b32 %1, 0;\n\tmov.b32 %2, 0;\n\tmov.b32 %3, 0;\n\t"
      "@p ld.global.v4.u32 {%0, %1, %2, %3}, [%4];\n\t}"
      : "=&r"(v.x), "=&r"(v.y), "=&r"(v.z), "=&r"(v.w) : "l"(a), "r"((int)pred));
  return v;
}
// AL bytes global -> shared, those beyond `bytes` zero (0: nothing is read)
template <int AL>
__device__ __forceinline__ void copy_async(uint32_t dst, uintptr_t src, int bytes) {
  if (AL == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], %3, %2;" ::"r"(dst), "l"(src), "r"(bytes), "n"(AL) : "memory");
}
__device__ __forceinline__ void sts16(uint32_t a, const uint4& v) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
// bytes sh .. sh + 15 of the 32 bytes lo | hi (sh even, 0 .. 14)
__device__ __forceinline__ uint4 shift_pair(const uint4& lo, const uint4& hi, int sh) {
  uint32_t w0 = lo.x, w1 = lo.y, w2 = lo.z, w3 = lo.w, w4 = hi.x, w5 = hi.y, w6 = hi.z, w7 = hi.w;
  if (sh & 8) { w0 = w2; w1 = w3; w2 = w4; w3 = w5; w4 = w6; w5 = w7; }
  if (sh & 4) { w0 = w1; w1 = w2; w2 = w3; w3 = w4; w4 = w5; }
  const uint32_t bits = (sh & 2) * 8;
  return make_uint4(__funnelshift_r(w0, w1, bits), __funnelshift_r(w1, w2, bits), __funnelshift_r(w2, w3, bits),
                    __funnelshift_r(w3, w4, bits));
}
// elements nv .. 7 of a 16-byte piece become zero
__device__ __forceinline__ uint4 keep_first(uint4 v, int nv) {
  if (nv >= 8) return v;
  uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (nv <= 2 * i) w[i] = 0u;
    else if (nv == 2 * i + 1) w[i] &= 0xffffu;
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// KIND: 0 row pattern, 1 tile pattern (ts a power of two from 8 to 64).  AL: every operand row starts on the AL-byte
// grid (16 for tile patterns; 16, 8, 4 or 2 for row patterns).
template <int KIND, int OP, int BN, int AL>
__global__ void __launch_bounds__(LG_THREADS, 2) gemm_ldg_kernel(const __grid_constant__ LdgParams p) {
  using L = LdgSmem<BN>;
  constexpr int LG_STAGES = L::STAGES;
  constexpr bool ASYNC = AL >= 4;
  constexpr bool A_MN = OP == OP_BWD_WEIGHT, B_MN = OP != OP_FWD;
  constexpr int NA = 4, NB = BN / 32;  // 16-byte pieces per loading thread and block, A and B
  const GemmArgs& g = p.g;

  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t base = (raw_addr + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw_addr);
  const uint32_t bars = base + L::BAR_OFF;
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (LG_STAGES + s); };
  const uint32_t done_bar = bars + 8u * (2 * LG_STAGES);
  volatile uint32_t* tmem_ptr = reinterpret_cast<volatile uint32_t*>(smem + L::BAR_OFF + 96);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::BAR_OFF + 100);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  pdl_launch_dependents();
  if (tid == 0) {
    for (int s = 0; s < LG_STAGES; ++s) {
      mbar_init(full_bar(s), ASYNC ? LG_LOADERS : LG_LOADERS / 32);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(done_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 8) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_ptr)), BN);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_ptr;
  pdl_wait_prior_grids();

  const ProductPlan s = make_plan<KIND, OP, UMMA_BM, BN, LG_BK>(g, p.ts, (int)gridDim.x, p.cl);
  const int rank = (int)cluster_ctarank();
  const int part = rank & (s.S - 1);          // this CTA's share of the contraction
  const int lead = rank - part;               // first CTA of those that share it
  const int rows = rank & (s.G - 1);          // this CTA's part of the tile's rows
  const int group = rank / s.G, groups = p.cl / s.G;
  const int n_cl = (int)gridDim.x / p.cl, units = (s.tiles + groups - 1) / groups;
  if (OP == OP_BWD_WEIGHT && g.flag1 && s.dp > 1 && warp < LG_LOADERS / 32) {
    const int w = (int)blockIdx.x * (LG_LOADERS / 32) + warp, ws = (int)gridDim.x * (LG_LOADERS / 32);
    if (KIND == 1) zero_dropped_tiles(g, p.ts, w, ws, lane);
    else zero_dropped_rows(g, s.N, w, ws, lane);
  }
  int blk = 0;        // blocks staged so far: stage = blk % STAGES
  int done = 0;       // accumulators finished so far
  bool ok = true;

  for (int u = (int)blockIdx.x / p.cl; u < units; u += n_cl) {
    const int t = u * groups + group;
    ProductTile ti = {};
    ti.nkb = -1;
    if (t < s.tiles) ti = make_tile<KIND, OP, UMMA_BM, BN, LG_BK>(g, s, t);
    const bool live = ti.nkb >= 0;
    const int kb0 = live ? (int)((long long)ti.nkb * part / s.S) : 0;
    const int kb1 = live ? (int)((long long)ti.nkb * (part + 1) / s.S) : 0;
    const bool has_acc = kb1 > kb0;

    if (warp == 8) {
      // ===================== products =====================
      if (lane == 0 && has_acc && ok) {
        const uint64_t desc_a = A_MN ? make_desc(0, 64 * LG_BK * 2, 1024) : make_desc(0, 16, 1024);
        const uint64_t desc_b = B_MN ? make_desc(0, 64 * LG_BK * 2, 1024) : make_desc(0, 16, 1024);
        const uint32_t idesc = make_idesc(BN, A_MN, B_MN);
        for (int kb = kb0; kb < kb1; ++kb) {
          const int it = blk + kb - kb0, st = it % LG_STAGES;
          if (!mbar_wait(full_bar(st), (uint32_t)(it / LG_STAGES) & 1u, abort_flag, g.status)) { ok = false; break; }
          if (ASYNC) fence_proxy_async_smem();  // the copies were made in the generic proxy
          tc_fence_after();
          const uint32_t sA = base + st * L::STAGE_BYTES;
          const uint64_t ad0 = desc_a | (uint64_t)((sA & 0x3FFFFu) >> 4);
          const uint64_t bd0 = desc_b | (uint64_t)(((sA + L::A_BYTES) & 0x3FFFFu) >> 4);
#pragma unroll
          for (int k = 0; k < LG_BK / 16; ++k)
            tc_mma_bf16(tmem, ad0 + (uint64_t)(k * (A_MN ? 128 : 2)), bd0 + (uint64_t)(k * (B_MN ? 128 : 2)), idesc,
                        (kb != kb0 || k != 0) ? 1u : 0u);
          tc_commit(empty_bar(st));
        }
        if (ok) tc_commit(done_bar);
      }
      __syncwarp();
    } else {
      // ===================== loads =====================
      // Thread (c, rsub) owns the 16-byte piece c of rows rsub, rsub + 32, ... of every block: rows of the operand
      // (K-major), or contraction rows of 64-column boxes (MN-major).  A block is 128 bytes further along the row, or
      // 64 rows further down, a multiple of 16 bytes either way, so what a thread's pieces look like (address,
      // phase `sh` on the 16-byte grid, elements that exist) is worked out once per tile.
      const int c = tid & 7, rsub = tid >> 3;
      uintptr_t ptr[NA + NB];      // first byte of the piece in block 0 (tile lists: without the listed coordinate)
      int rem[NA + NB];            // MN-major: columns from the piece's first to the last that exists; K-major: 0 = no such row
      const size_t ldb_row = (KIND == 0 && OP != OP_BWD_WEIGHT && g.hdr_in == nullptr) ? (size_t)g.lda1 * s.dp : (size_t)g.lda1;
      if (live) {
        const __nv_bfloat16* PA = reinterpret_cast<const __nv_bfloat16*>(g.A0);
        const __nv_bfloat16* PB = reinterpret_cast<const __nv_bfloat16*>(g.A1);
        // rows of the weight are the kept neurons, bb + i * dp; a weight packed for a feeding pattern has them in order
        if (KIND == 0 && OP != OP_BWD_WEIGHT && g.hdr_in == nullptr) PB += (size_t)s.bb * g.lda1;
#pragma unroll
        for (int j = 0; j < NA; ++j) {
          if (!A_MN) {
            const int m = ti.m0 + j * 32 + rsub;
            rem[j] = m < s.M ? 1 : 0;
            ptr[j] = reinterpret_cast<uintptr_t>(PA + (size_t)(m < s.M ? m : 0) * g.lda0 + (KIND == 0 ? 8 * c : 0));
          } else {
            const int m = ti.m0 + (j >> 1) * 64 + 8 * c, lim = KIND == 0 ? s.M : ti.cnt << s.lts;
            rem[j] = lim - m;
            const int col = KIND == 0 ? m : (m < lim ? ti.class_pos(s, m) : 0);
            ptr[j] = reinterpret_cast<uintptr_t>(PA + (size_t)((j & 1) * 32 + rsub) * g.lda0 + col);
          }
        }
#pragma unroll
        for (int j = 0; j < NB; ++j) {
          if (!B_MN) {
            const int n = ti.n0 + j * 32 + rsub, lim = KIND == 0 ? s.N : ti.cnt << s.lts;
            rem[NA + j] = n < lim ? 1 : 0;
            const int row = n < lim ? (KIND == 0 ? n : ti.class_pos(s, n)) : 0;
            ptr[NA + j] = reinterpret_cast<uintptr_t>(PB + (size_t)row * ldb_row + (KIND == 0 ? 8 * c : 0));
          } else {
            const int n = ti.n0 + (j >> 1) * 64 + 8 * c;
            const int lim = KIND == 0 ? s.N : (OP == OP_BWD_DATA ? ti.cnt : ti.len) << s.lts;
            rem[NA + j] = lim - n;
            int col = n;
            if (KIND == 1) col = n >= lim ? 0 : (OP == OP_BWD_DATA ? ti.class_pos(s, n) : ti.list_pos(s, n));
            const bool listed = KIND == 1 && OP == OP_BWD_DATA;  // its rows come from the list
            ptr[NA + j] = reinterpret_cast<uintptr_t>(PB + (listed ? (size_t)0 : (size_t)((j & 1) * 32 + rsub) * ldb_row) + col);
          }
        }
      }
      const size_t step_a = A_MN ? (size_t)g.lda0 * 128 : 128, step_b = B_MN ? ldb_row * 128 : 128;  // bytes per block
      uint4 v[NA + NB];
      uint4 x = make_uint4(0, 0, 0, 0);
      // Elements of a piece of row group j that exist in block kb (<= 0: none).
      auto exists = [&](int j, int kb, int piece) -> int {
        const bool mn = j < NA ? A_MN : B_MN;
        if (!mn) return rem[j] == 0 ? 0 : min(8, ti.kext - kb * LG_BK - 8 * piece);
        const int jj = j < NA ? j : j - NA;
        return kb * LG_BK + (jj & 1) * 32 + rsub < ti.kext ? min(8, rem[j] - 8 * (piece - c)) : 0;
      };
      auto address = [&](int j, int kb) -> uintptr_t {
        if (KIND == 0) return ptr[j] + (size_t)kb * (j < NA ? step_a : step_b);
        if (OP == OP_BWD_WEIGHT) return ptr[j] + (size_t)kb * (j < NA ? step_a : step_b);
        const bool mn = j < NA ? A_MN : B_MN;
        const int k = mn ? kb * LG_BK + ((j - NA) & 1) * 32 + rsub : kb * LG_BK + 8 * c;
        const size_t kp = k < ti.kext ? (size_t)ti.list_pos(s, k) : 0;
        return ptr[j] + (mn ? kp * (size_t)g.lda1 : kp) * 2;
      };
      // K-major: row 32 jj + rsub; MN-major: box jj / 2 (8 KiB each), row 32 (jj & 1) + rsub: the same offset
      auto place = [&](int j, uint32_t sA) {
        const int row = (j < NA ? j : j - NA) * 32 + rsub;
        return sA + (j < NA ? 0u : (uint32_t)L::A_BYTES) + (uint32_t)row * 128u + (uint32_t)((c ^ (row & 7)) << 4);
      };
      auto copy = [&](int kb, uint32_t sA) {
#pragma unroll
        for (int j = 0; j < NA + NB; ++j) {
          const int bytes = 2 * max(0, exists(j, kb, c));
          const uintptr_t a = bytes > 0 ? address(j, kb) : reinterpret_cast<uintptr_t>(j < NA ? g.A0 : g.A1);
          const uint32_t d = place(j, sA);
#pragma unroll
          for (int o = 0; o < 16; o += AL) {
            const int b = min(AL, max(0, bytes - o));
            copy_async<AL>(d + o, b > 0 ? a + o : a, b);
          }
        }
      };
      // AL == 2: loads of block kb in the aligned 16-byte units that cover the row: each lane the unit of its piece's first byte, and the unit after
      // the row's last piece is fetched by lane j of the row's eight lanes for the j-th row (x).  A unit is read only if it holds
      // an element that exists, so no load leaves the 16-byte unit of such an element.
      auto issue = [&](int kb) {
#pragma unroll
        for (int j = 0; j < NA + NB; ++j) {
          const int nv = exists(j, kb, c);
          const uintptr_t a = address(j, kb);
          // also when only the piece before it (same row) reaches into this unit
          const int sh = (int)(a & 15u);
          const int prev = exists(j, kb, c - 1);
          const bool before = c > 0 && sh != 0 && prev > 0 && 2 * prev > 16 - sh;
          v[j] = ldg16(a & ~(uintptr_t)15, nv > 0 || before);
        }
        {
          // the j-th row's end: this lane stands in for piece 7 of row group j = c
          uintptr_t a = 0;
          int nv = 0;
#pragma unroll
          for (int j = 0; j < NA + NB; ++j) {
            if (j == c) {
              a = address(j, kb) + (size_t)(7 - c) * 16;
              nv = exists(j, kb, 7);
            }
          }
          const int sh = (int)(a & 15u);
          x = ldg16((a & ~(uintptr_t)15) + 16, nv > 0 && sh != 0 && 2 * nv > 16 - sh);
        }
      };
      auto store = [&](int kb, uint32_t sA) {
#pragma unroll
        for (int j = 0; j < NA + NB; ++j) {
          const int sh = (int)(address(j, kb) & 15u);
          uint4 hi, e;
          hi.x = __shfl_down_sync(0xffffffffu, v[j].x, 1, 8);
          hi.y = __shfl_down_sync(0xffffffffu, v[j].y, 1, 8);
          hi.z = __shfl_down_sync(0xffffffffu, v[j].z, 1, 8);
          hi.w = __shfl_down_sync(0xffffffffu, v[j].w, 1, 8);
          e.x = __shfl_sync(0xffffffffu, x.x, j, 8);
          e.y = __shfl_sync(0xffffffffu, x.y, j, 8);
          e.z = __shfl_sync(0xffffffffu, x.z, j, 8);
          e.w = __shfl_sync(0xffffffffu, x.w, j, 8);
          if (c == 7) hi = e;
          sts16(place(j, sA), keep_first(shift_pair(v[j], hi, sh), exists(j, kb, c)));
        }
      };
      if (has_acc && ok && ASYNC) {
        for (int kb = kb0; kb < kb1; ++kb) {
          const int it = blk + kb - kb0, st = it % LG_STAGES;
          if (!mbar_wait(empty_bar(st), ((uint32_t)(it / LG_STAGES) & 1u) ^ 1u, abort_flag, g.status)) ok = false;
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          copy(kb, base + st * L::STAGE_BYTES);
          cp_async_mbar_arrive_noinc(full_bar(st));
        }
      } else if (has_acc && ok) {
        issue(kb0);
        for (int kb = kb0; kb < kb1; ++kb) {
          const int it = blk + kb - kb0, st = it % LG_STAGES;
          if (!mbar_wait(empty_bar(st), ((uint32_t)(it / LG_STAGES) & 1u) ^ 1u, abort_flag, g.status)) ok = false;
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          store(kb, base + st * L::STAGE_BYTES);
          if (kb + 1 < kb1) issue(kb + 1);
          fence_proxy_async_smem();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(full_bar(st));
        }
      }
      // ===================== fp32 tile to shared memory =====================
      if (live) {
        if (has_acc && ok) {
          if (!mbar_wait(done_bar, (uint32_t)done & 1u, abort_flag, g.status)) ok = false;
          ok = __all_sync(0xffffffffu, ok);
          tc_fence_after();
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");  // the stages are idle: every loading warp is past its last store
        float* T = reinterpret_cast<float*>(smem);
        const int row = (warp & 3) * 32 + lane, col0 = (warp >> 2) * (BN / 2);
#pragma unroll 1
        for (int cc = 0; cc < BN / 2; cc += 32) {
          uint32_t r[32];
          if (has_acc && ok) {
            tmem_ld32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(col0 + cc), r);
            tmem_ld_wait();
          }
          float4* dst = reinterpret_cast<float4*>(T + row * L::PITCH + col0 + cc);
#pragma unroll
          for (int i = 0; i < 8; ++i)
            dst[i] = has_acc && ok ? make_float4(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1]),
                                                 __uint_as_float(r[4 * i + 2]), __uint_as_float(r[4 * i + 3]))
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        tc_fence_before();
        if (s.S == 1) asm volatile("bar.sync 1, 256;" ::: "memory");
      }
    }
    blk += kb1 - kb0;
    if (has_acc) ++done;
    __syncwarp();
    if (s.S > 1) cluster_sync_all();  // the partial tiles of the group are complete

    if (warp < 8 && live) {
      // ===================== epilogue =====================
      write_tile<KIND, OP, UMMA_BM, BN, L::PITCH, LG_LOADERS / 32, true, __nv_bfloat16>(g, s, ti, reinterpret_cast<float*>(smem), base, rows,
                                                                                 lead, warp, lane);
      if (s.S == 1) asm volatile("bar.sync 1, 256;" ::: "memory");  // the tile has been read: the stages may be filled again
    }
    __syncwarp();
    if (s.S > 1) cluster_sync_all();  // no CTA of the group reads this one's partial tile any more
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    tmem_dealloc(tmem, BN);
  }
}

template <int KIND, int OP, int BN, int AL>
ard_status launch_ldg(ard_ctx* ctx, LdgParams p, int M, int N, int nkb, cudaStream_t s) {
  auto kern = gemm_ldg_kernel<KIND, OP, BN, AL>;
  static bool attr_done[64] = {};
  const int dev = ctx->device & 63;
  if (!attr_done[dev]) {
    ARD_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, LdgSmem<BN>::TOTAL));
    attr_done[dev] = true;
  }
  const int tiles = (M + UMMA_BM - 1) / UMMA_BM * ((N + BN - 1) / BN);
  // A cluster lives inside one GPC, and what is left of a GPC behind the last whole cluster stays empty: of two CTAs per SM
  // this GPU holds 37 clusters of 8 by count but 30 at once (15 by the occupancy query, which counts on one CTA per SM
  // for a kernel that allocates tensor memory), and a grid of 37 ran in two waves.  Hence a grid of what fits at once,
  // in clusters of 8 only where even eight shares of every tile find a place, else of 4.
  p.cl = tiles * 8 <= 2 * ctx->sm_count ? 8 : 4;
  static int room[2][64] = {};
  int& r = room[p.cl == 8][dev];
  if (r == 0) r = 2 * ard_cluster_room(ctx, kern, p.cl, LG_THREADS, LdgSmem<BN>::TOTAL);
  int ctas = r;
  if (KIND == 0) {  // no more than the densest pattern's tiles, cut as often as its contraction allows
    int S = p.cl;
    while (S > 1 && nkb < 2 * S) S >>= 1;
    const int n = (tiles * S + p.cl - 1) / p.cl * p.cl;
    if (n < ctas) ctas = n;
  }
  ARD_CUDA_OK(ard_launch_cluster(ctx, kern, p.cl, dim3(ctas), dim3(LG_THREADS), LdgSmem<BN>::TOTAL, s, p));
  ctx->launches++;
  ARD_CUDA_OK(cudaGetLastError());
  return ARD_OK;
}

inline int cdiv(int a, int b) { return (a + b - 1) / b; }

}  // namespace

bool ldg_takes(const ard_ctx* ctx, ard_kind kind, const GemmArgs& g, int ts) {
  if (ctx->encode_fn == nullptr || g.B < 1 || g.K < 1 || g.N < 1) return false;  // not sm_100, nothing to do
  if (kind == ARD_ROW) return true;
  return ts >= 8 && ts <= 64 && (ts & (ts - 1)) == 0 && ((reinterpret_cast<uintptr_t>(g.A0) | reinterpret_cast<uintptr_t>(g.A1)) & 15u) == 0 &&
         g.lda0 % 8 == 0 && g.lda1 % 8 == 0;
}

ard_status launch_gemm_ldg(ard_ctx* ctx, ard_kind kind, GemmOp op, const GemmArgs& g, int ts, cudaStream_t s) {
  LdgParams p = {};
  p.g = g;
  p.ts = ts;
  // 128 x 128 tiles once they fill the device without cutting the contraction, else 128 x 64
  const int M = op == OP_BWD_WEIGHT ? g.N : g.B, N = op == OP_FWD ? g.N : g.K;
  const bool wide = cdiv(M, UMMA_BM) * cdiv(N, 128) >= ctx->sm_count;
  const int nkb = cdiv(op == OP_FWD ? g.K : (op == OP_BWD_DATA ? g.N : g.B), LG_BK);
  const uintptr_t grid = reinterpret_cast<uintptr_t>(g.A0) | reinterpret_cast<uintptr_t>(g.A1) | (uintptr_t)(2 * g.lda0) | (uintptr_t)(2 * g.lda1);
#define ARD_LDG(KIND_, OP_, AL_) \
  return wide ? launch_ldg<KIND_, OP_, 128, AL_>(ctx, p, M, N, nkb, s) : launch_ldg<KIND_, OP_, 64, AL_>(ctx, p, M, N, nkb, s)
#define ARD_LDG_ROW(OP_)             \
  do {                               \
    if (grid % 16 == 0) ARD_LDG(0, OP_, 16);  \
    if (grid % 8 == 0) ARD_LDG(0, OP_, 8);    \
    if (grid % 4 == 0) ARD_LDG(0, OP_, 4);    \
    ARD_LDG(0, OP_, 2);                       \
  } while (0)
  if (kind == ARD_ROW) {
    if (op == OP_FWD) ARD_LDG_ROW(OP_FWD);
    if (op == OP_BWD_DATA) ARD_LDG_ROW(OP_BWD_DATA);
    ARD_LDG_ROW(OP_BWD_WEIGHT);
  }
  if (op == OP_FWD) ARD_LDG(1, OP_FWD, 16);
  if (op == OP_BWD_DATA) ARD_LDG(1, OP_BWD_DATA, 16);
  ARD_LDG(1, OP_BWD_WEIGHT, 16);
#undef ARD_LDG_ROW
#undef ARD_LDG
}
