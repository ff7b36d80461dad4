// What the product kernels whose threads stage the operands themselves have in common (gemm_ldg_sm100.cu and, for fp32 operands,
// gemm_f32_sm100.cu on the tensor cores, gemm_cc.cu on the CUDA cores): the tiling worked out from the pattern header on the device, the sum of the
// partial tiles of a cut contraction, and the rows' way out.  Everything is static to the including translation unit.
//
// A tile pattern (Sec. 3.2) keeps tile (r, c) iff r * Tc + c = b - 1 (mod dp), so tile-columns with equal c mod dp share
// one kept list, and tile-rows with equal r mod dp / gcd(Tc mod dp, dp) another: the members of such a class side by
// side are one dense product over their common list, whatever the size of a pattern tile.
//
// Work is dealt in clusters of 4 or 8 CTAs.  A product with fewer output tiles than the device has room for is cut
// along its contraction over S = 2, 4 or 8 CTAs of a cluster; S follows from the sampled pattern.
#pragma once

#include "ard_internal.h"
#include "dropped_zeros.h"
#include "sm100_ptx.h"

namespace {

struct ProductPlan {
  int dp, bb, n_keep;
  int M, N, K;         // extents of the product (tile patterns: K is the batch for the weight gradient, else unused)
  int Mt;              // tiles along M
  int tiles;           // output tiles (weight gradient of a tile pattern: an upper bound, some may turn out empty)
  int S;               // shares that a tile's contraction is cut into
  int G;               // CTAs per output tile: S, or more that compute the same shares and write other rows
  // tile patterns: class c (tiles with equal number mod cstep) has q + (c < rmd) members
  int ts, lts;         // pattern tile, its log2 (-1: not a power of two)
  int cstep, q, rmd, nclass;
  int nH, nL;          // output tiles of a class with q + 1 / q members
  int a, c0, mmax, nmax;       // weight gradient: non-empty classes c0, c0 + a, ...; tiles per class mmax x nmax

  __device__ __forceinline__ int tile_of(int i) const { return lts >= 0 ? i >> lts : i / ts; }
};

struct ProductTile {
  int m0, n0;           // tile patterns: along the gathered dimension a position among the class's members
  int nkb;              // contraction blocks (-1: no such tile)
  const int32_t* list;  // tile patterns: kept tiles along the contraction (weight gradient: along N)
  int len;
  int c, cnt;           // class and its members
  int kext;             // contraction length

  // coordinate of position i among the class's members / in the kept list
  __device__ __forceinline__ int class_pos(const ProductPlan& s, int i) const {
    const int m = s.tile_of(i);
    return (c + m * s.cstep) * s.ts + i - m * s.ts;
  }
  __device__ __forceinline__ int list_pos(const ProductPlan& s, int i) const {
    const int m = s.tile_of(i);
    return list[m] * s.ts + i - m * s.ts;
  }
};

__device__ __forceinline__ int sp_cdiv(int a, int b) { return (a + b - 1) / b; }

// want: CTAs the device has room for at once; cl: CTAs per cluster.
template <int KIND, int OP, int BM, int BN, int BK>
__device__ __forceinline__ ProductPlan make_plan(const GemmArgs& g, int ts, int want, int cl) {
  ProductPlan s = {};
  s.dp = g.hdr[HDR_DP];
  s.bb = g.hdr[HDR_B] - 1;
  s.n_keep = g.hdr[HDR_NKEEP];
  int nkb;
  if (KIND == 0) {
    // fan-in extent: all K inputs, or the kept outputs of the layer that produced the input
    const int kin = g.hdr_in != nullptr ? g.hdr_in[HDR_NKEEP] : g.K;
    s.M = OP == OP_BWD_WEIGHT ? s.n_keep : g.B;
    s.N = OP == OP_FWD ? s.n_keep : kin;
    s.K = OP == OP_FWD ? kin : (OP == OP_BWD_DATA ? s.n_keep : g.B);
    s.Mt = sp_cdiv(s.M, BM);
    s.tiles = s.Mt * sp_cdiv(s.N, BN);
    nkb = sp_cdiv(s.K, BK);
  } else {
    const int Tr = g.hdr[HDR_TR], Tc = g.hdr[HDR_TC];
    s.ts = ts;
    s.lts = (ts & (ts - 1)) == 0 ? 31 - __clz(ts) : -1;
    int gg = Tc % s.dp, a = s.dp;
    while (gg) { const int t = a % gg; a = gg; gg = t; }  // a = gcd(Tc mod dp, dp)
    const int extent = OP == OP_BWD_DATA ? Tr : Tc;
    s.cstep = OP == OP_BWD_DATA ? s.dp / a : s.dp;
    s.nclass = min(s.cstep, extent);
    s.q = extent / s.cstep;
    s.rmd = extent % s.cstep;
    s.nH = sp_cdiv((s.q + 1) * ts, BN);
    s.nL = sp_cdiv(s.q * ts, BN);
    s.M = OP == OP_BWD_WEIGHT ? g.N : g.B;
    s.N = OP == OP_FWD ? g.N : g.K;
    s.K = g.B;
    s.Mt = sp_cdiv(s.M, BM);
    if (OP == OP_BWD_WEIGHT) {
      s.a = a;
      s.c0 = s.bb % a;
      const int ncl = s.c0 < s.nclass ? (s.nclass - 1 - s.c0) / a + 1 : 0;
      s.mmax = sp_cdiv(sp_cdiv(extent, s.cstep) * ts, BM);
      s.nmax = sp_cdiv(sp_cdiv(Tr, s.dp / a) * ts, BN);
      s.tiles = ncl * s.mmax * s.nmax;
      nkb = sp_cdiv(g.B, BK);
    } else {
      s.tiles = s.Mt * (s.rmd * s.nH + (s.nclass - s.rmd) * s.nL);
      // longest kept list
      nkb = sp_cdiv(sp_cdiv(OP == OP_FWD ? Tr : Tc, OP == OP_FWD ? s.dp / a : s.dp) * ts, BK);
    }
  }
  // Cut the contraction only while the pieces still find an idle place and hold at least two blocks: a cut costs
  // two cluster barriers and a pass of the partial tiles through shared memory.
  s.S = cl;
  while (s.S > 1 && (s.tiles * s.S > want || nkb < 2 * s.S)) s.S >>= 1;
  // A full-width output under a long period is up to dp times as wide as what is multiplied: where the contraction is too
  // short to be cut, CTAs that would be idle compute the tile once more and write a part of its rows (forward, 2000 x 129 ->
  // 2047 under a period of 16: 103 -> 43 us).
  s.G = s.S;
  if (KIND == 0 && OP == OP_FWD && g.flag0 == ARD_OUT_SCATTER_ZEROFILL && s.dp > 1)
    while (s.G < cl && s.tiles * s.G * 2 <= want) s.G <<= 1;
  return s;
}

template <int KIND, int OP, int BM, int BN, int BK>
__device__ __forceinline__ ProductTile make_tile(const GemmArgs& g, const ProductPlan& s, int t) {
  ProductTile ti = {};
  if (KIND == 0) {
    ti.m0 = (t % s.Mt) * BM;
    ti.n0 = (t / s.Mt) * BN;
    ti.kext = s.K;
  } else if (OP == OP_BWD_WEIGHT) {
    const int per = s.mmax * s.nmax, ci = t / per, r = t - ci * per;
    ti.c = s.c0 + ci * s.a;
    ti.cnt = s.q + (ti.c < s.rmd ? 1 : 0);
    ti.m0 = (r % s.mmax) * BM;
    ti.n0 = (r / s.mmax) * BN;
    const int off = g.col_ptr[ti.c];
    ti.len = g.col_ptr[ti.c + 1] - off;
    ti.list = g.col_idx + off;
    ti.kext = s.K;
    if (ti.m0 >= ti.cnt * s.ts || ti.n0 >= ti.len * s.ts) { ti.nkb = -1; return ti; }
  } else {
    ti.m0 = (t % s.Mt) * BM;
    int j = t / s.Mt, v;
    if (j < s.rmd * s.nH) { ti.c = j / s.nH; v = j - ti.c * s.nH; }
    else { j -= s.rmd * s.nH; const int i = j / s.nL; ti.c = s.rmd + i; v = j - i * s.nL; }
    ti.cnt = s.q + (ti.c < s.rmd ? 1 : 0);
    ti.n0 = v * BN;
    const int32_t* ptr = OP == OP_FWD ? g.col_ptr : g.row_ptr;
    const int off = ptr[ti.c];
    ti.len = ptr[ti.c + 1] - off;
    ti.list = (OP == OP_FWD ? g.col_idx : g.row_idx) + off;
    ti.kext = ti.len * s.ts;
  }
  ti.nkb = sp_cdiv(ti.kext, BK);
  return ti;
}

__device__ __forceinline__ float4 ld_cluster_f4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
  return v;
}
// Adds the S partial tiles at `off` (the same shared-memory offset in CTAs lead .. lead + S - 1) in contraction order.
template <int S>
__device__ __forceinline__ float4 sum_shares(uint32_t off, int lead) {
  float4 v[S];
#pragma unroll
  for (int j = 0; j < S; ++j) v[j] = ld_cluster_f4(mapa_u32(off, (uint32_t)(lead + j)));
#pragma unroll
  for (int j = 1; j < S; ++j) { v[0].x += v[j].x; v[0].y += v[j].y; v[0].z += v[j].z; v[0].w += v[j].w; }
  return v[0];
}

// The CTA's rows of a finished tile (fp32, PITCH words per row in shared memory at T / address t_addr): rows
// [part * BM / G, (part + 1) * BM / G), dealt to NW warps.  With S > 1 the shares of CTAs lead .. lead + S - 1 are added
// into this CTA's own copy first.  T_: operand type (the saved activation's).  SPREAD: G may exceed S, and rows off
// the grid of four elements get wide stores between their edges (not for the CUDA-core kernels, whose loop lost a quarter of
// its speed to the code's registers; there G is S, and the CTAs that share a tile write the zeros that belong to its rows).
template <int KIND, int OP, int BM, int BN, int PITCH, int NW, bool SPREAD, typename T_>
__device__ __forceinline__ void write_tile(const GemmArgs& g, const ProductPlan& s, const ProductTile& ti, float* T, uint32_t t_addr,
                                           int part, int lead, int warp, int lane) {
  const int rows_per = BM / (SPREAD ? s.G : s.S), r0 = part * rows_per;
  if (s.S > 1) {
    for (int i = lane; i < rows_per / NW * (BN / 4); i += 32) {  // this warp's rows r0 + warp, r0 + warp + NW, ...
      const int row = r0 + warp + NW * (i / (BN / 4)), w = row * PITCH + 4 * (i % (BN / 4));
      const uint32_t off = t_addr + (uint32_t)w * 4u;
      *reinterpret_cast<float4*>(T + w) = s.S == 8 ? sum_shares<8>(off, lead) : (s.S == 4 ? sum_shares<4>(off, lead) : sum_shares<2>(off, lead));
    }
    __syncwarp();
  }
  const int es = g.out_is_f32 ? 4 : 2;
  const bool vec = !g.accumulate && (reinterpret_cast<uintptr_t>(g.out) & (uintptr_t)(4 * es - 1)) == 0 && (g.ldo & 3) == 0 &&
                   (KIND == 0 || (s.ts & 3) == 0);
  auto put = [&](size_t off, float val) {
    if (g.out_is_f32) {
      float* o = reinterpret_cast<float*>(g.out) + off;
      *o = g.accumulate ? *o + val : val;
    } else {
      __nv_bfloat16* o = reinterpret_cast<__nv_bfloat16*>(g.out) + off;
      *o = __float2bfloat16_rn(g.accumulate ? __bfloat162float(*o) + val : val);
    }
  };
  // v to four consecutive elements whose address is a multiple of four of them
  auto put4_aligned = [&](size_t off, const float (&v)[4]) {
    if (g.out_is_f32) {
      *reinterpret_cast<float4*>(reinterpret_cast<float*>(g.out) + off) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
      const __nv_bfloat162 lo = __floats2bfloat162_rn(v[0], v[1]), hi = __floats2bfloat162_rn(v[2], v[3]);
      *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(g.out) + off) =
          make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
    }
  };
  // v, the first nv of them, to four consecutive elements; off is a multiple of four
  auto put4 = [&](size_t off, const float (&v)[4], int nv) {
    if (vec && nv >= 4) {
      put4_aligned(off, v);
      return;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (i < nv) put(off + i, v[i]);
  };
  // compact column j of the tile: bias, then the activation, then the rescale (Sec. 3.2)
  auto fwd_value = [&](const float* row, int j) {
    float z = row[j];
    if (g.bias != nullptr) z += g.bias[s.bb + (ti.n0 + j) * s.dp];
    if (g.relu) z = fmaxf(z, 0.f);
    return z * g.alpha;
  };
  if (KIND == 0 && OP == OP_FWD && g.flag0 == ARD_OUT_SCATTER_ZEROFILL && s.dp > 1) {
    // output columns [n0 * dp, (n0 + BN) * dp), the last tile up to N: kept ones and the zeros between
    const int lo = ti.n0 * s.dp, hi = ti.n0 + BN >= s.N ? g.N : (ti.n0 + BN) * s.dp;
    for (int r = r0 + warp; r < r0 + rows_per && ti.m0 + r < s.M; r += NW) {
      const float* row = T + r * PITCH;
      const size_t base = (size_t)(ti.m0 + r) * g.ldo;
      int first = lo;  // of the pieces of four columns; off the grid the piece before the first one on it reaches back past lo
      if (SPREAD && !vec) {
        const uintptr_t at = reinterpret_cast<uintptr_t>(g.out) + (base + lo) * es;
        const int sh = (int)((0 - at) & (uintptr_t)(4 * es - 1)) / es;  // columns up to the grid
        first = sh == 0 ? lo : lo + sh - 4;
      }
      for (int c = first + 4 * lane; c < hi; c += 128) {
        const int rel = max(c, lo) - s.bb;
        int j = rel <= 0 ? 0 : (rel + s.dp - 1) / s.dp;  // first kept column at or after c
        int at = s.bb + j * s.dp - c;
        float v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          v[i] = 0.f;
          if (i == at) {
            if (j < s.n_keep) v[i] = fwd_value(row, j - ti.n0);
            ++j;
            at += s.dp;
          }
        }
        if (SPREAD && !vec) {
          if (c >= lo && hi - c >= 4 && !g.accumulate) {
            put4_aligned(base + c, v);
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (c + i >= lo && c + i < hi) put(base + c + i, v[i]);
          }
        } else {
          put4(base + c, v, hi - c);
        }
      }
    }
    return;
  }
  // Four consecutive columns per lane.
  constexpr int QR = BN / 4;
  const int col_lim = KIND == 0 ? s.N : (OP == OP_BWD_WEIGHT ? ti.len : ti.cnt) * s.ts;
  const int row_lim = KIND == 1 && OP == OP_BWD_WEIGHT ? ti.cnt * s.ts : s.M;
  for (int e = lane; e < rows_per / NW * QR; e += 32) {
    const int r = r0 + warp + NW * (e / QR), j0 = 4 * (e % QR);
    const int m = ti.m0 + r, n = ti.n0 + j0, nv = col_lim - n;
    if (m >= row_lim || nv <= 0) continue;
    const float* row = T + r * PITCH;
    float v[4];
    const float4 x = *reinterpret_cast<const float4*>(row + j0);
    v[0] = x.x * g.alpha; v[1] = x.y * g.alpha; v[2] = x.z * g.alpha; v[3] = x.w * g.alpha;
    if (KIND == 0 && OP == OP_FWD && (g.bias != nullptr || g.relu)) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < nv) v[i] = fwd_value(row, j0 + i);
    }
    if (KIND == 0 && OP == OP_BWD_DATA && g.act != nullptr) {
      // adjoint of the producing layer's ReLU: nothing flows where its output was not positive
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < nv && !((float)reinterpret_cast<const T_*>(g.act)[(size_t)m * g.ldact + n + i] > 0.f)) v[i] = 0.f;
    }
    size_t orow = m;
    if (KIND == 0 && OP == OP_BWD_WEIGHT && g.hdr_in == nullptr) orow = (size_t)s.bb + (size_t)m * s.dp;
    if (KIND == 1 && OP == OP_BWD_WEIGHT) orow = (size_t)ti.class_pos(s, m);
    auto pos = [&](int i) { return KIND == 0 ? i : (OP == OP_BWD_WEIGHT ? ti.list_pos(s, i) : ti.class_pos(s, i)); };
    if (KIND == 0 || (s.ts & 3) == 0) {
      put4(orow * g.ldo + pos(n), v, nv);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < nv) put(orow * g.ldo + pos(n + i), v[i]);
    }
    if (!SPREAD && KIND == 0 && OP == OP_BWD_WEIGHT && g.flag1 && s.dp > 1 && (BM == 64 || s.S > 1)) {
      // compact row m owns output rows [m * dp, (m + 1) * dp), the last one the tail: zeros but for its own
      const float zero[4] = {0.f, 0.f, 0.f, 0.f};
      const long long first = (long long)m * s.dp;
      const long long last = m == s.M - 1 ? g.N : min((long long)g.N, first + s.dp);
      for (long long z = first; z < last; ++z)
        if (z != (long long)orow) put4((size_t)z * g.ldo + n, zero, nv);
    }
  }
}

}  // namespace
