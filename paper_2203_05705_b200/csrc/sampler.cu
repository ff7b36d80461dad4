// Device-side pattern sampler (Sec. 3.4) and kept-unit list emitter (Sec. 3.1 Eq. 1, Sec. 3.2).
//
// One CTA per call.  Thread 0 runs Philox4x32-10 on the (seed, iteration, stream) counter, picks
// the period dp from the integer cumulative table of K and the bias b uniformly from {1..dp};
// all threads then write the header and the lists the GEMM kernels read.  Nothing returns to the
// host, so the GEMMs that follow on the same stream need no synchronisation.
#include "ard_internal.h"
#include "philox.h"

namespace {

constexpr int SAMPLER_THREADS = 1024;  // tile patterns; row patterns launch 256 (fewer lists to fill)

__global__ void __launch_bounds__(SAMPLER_THREADS)
ard_sample_kernel(int32_t* __restrict__ hdr, int32_t* __restrict__ idx, int32_t* __restrict__ col_ptr,
                  int32_t* __restrict__ col_idx, int32_t* __restrict__ row_ptr, int32_t* __restrict__ row_idx,
                  const unsigned long long* __restrict__ cdf, int ndp, unsigned long long seed,
                  unsigned long long iteration, uint32_t stream_id, int forced_dp, int forced_b, int kind,
                  int units, int Tr, int Tc, int ts, unsigned long long* __restrict__ counter, int advance) {
  __shared__ int s_dp, s_b;
  const int nthreads = (int)blockDim.x;
  __shared__ unsigned long long s_cdf[64];
  pdl_launch_dependents();
  pdl_wait_prior_grids();  // earlier kernels may still be reading the lists this kernel rewrites
  // The cumulative table is searched by one thread; short tables are fetched by all threads at once first,
  // so that the search does not pay one global-memory round trip per probe.
  const bool cdf_smem = forced_dp <= 0 && ndp <= 64;
  if (cdf_smem && (int)threadIdx.x < ndp) s_cdf[threadIdx.x] = cdf[threadIdx.x];
  __syncthreads();
  if (threadIdx.x == 0) {
    int dp, b;
    if (forced_dp > 0) {
      dp = forced_dp;
      b = forced_b;
    } else {
      // A device-resident counter lets a captured graph draw a fresh pattern at every replay.
      if (counter != nullptr) {
        const unsigned long long n = *counter;
        iteration += n;
        if (advance) *counter = n + 1ull;
      }
      uint32_t c[4] = {(uint32_t)iteration, (uint32_t)(iteration >> 32), stream_id, 0u};
      philox4x32_10(c, (uint32_t)seed, (uint32_t)(seed >> 32));
      // dp = smallest i with r0 < c_i; the table is non-decreasing and ends at 2^32.
      int lo = 0, hi = ndp - 1;  // answer index in [0, ndp-1]
      const unsigned long long r0 = c[0];
      while (lo < hi) {
        int mid = (lo + hi) >> 1;
        const unsigned long long cm = cdf_smem ? s_cdf[mid] : cdf[mid];
        if (r0 < cm) hi = mid; else lo = mid + 1;
      }
      dp = lo + 1;
      b = 1 + (int)(((unsigned long long)c[1] * (unsigned long long)dp) >> 32);
    }
    s_dp = dp;
    s_b = b;
  }
  __syncthreads();
  const int dp = s_dp, b = s_b;
  const int n_keep = (units - b) / dp + 1;
  if (threadIdx.x == 0) {
    hdr[HDR_KIND] = kind;
    hdr[HDR_DP] = dp;
    hdr[HDR_B] = b;
    hdr[HDR_NKEEP] = n_keep;
    hdr[HDR_UNITS] = units;
    hdr[HDR_TR] = Tr;
    hdr[HDR_TC] = Tc;
    hdr[HDR_TS] = ts;
    hdr[HDR_MAPIDX] = dp * (dp - 1) / 2 + (b - 1);
  }
  // Eq. 1 on the 1-based unit index i = b + j*dp  ->  0-based b-1 + j*dp, ascending.
  for (int j = threadIdx.x; j < n_keep; j += nthreads) idx[j] = b - 1 + j * dp;
  if (kind != ARD_TILE) return;

  // Tiles are numbered row-major, so the ascending list is already grouped by tile-row.
  for (int j = threadIdx.x; j < n_keep; j += nthreads) row_idx[j] = (b - 1 + j * dp) % Tc;
  for (int r = threadIdx.x; r <= Tr; r += nthreads) {
    // kept tiles with 0-based linear index < r*Tc
    const long long lim = (long long)r * Tc;  // count of j with b-1 + j*dp < lim
    int cnt = 0;
    if (lim > b - 1) cnt = (int)((lim - 1 - (b - 1)) / dp) + 1;
    row_ptr[r] = cnt;
  }
  // Grouped by tile-column.  Tile (r, c) is kept iff r * Tc + c = b - 1 (mod dp), so walking down a column adds Tc mod dp to a
  // residue: a thread per column finds its first kept row and the distance to the next in at most 2 dp steps, and the rest
  // follows.  Then a scan over the columns, and a warp per column writes its rows.  (4096 tiles, a period of 4: 5.0 us; ballots over
  // every tile of a column, twice, and one thread's running sum took 6.2.)
  __shared__ int s_first[SAMPLER_THREADS], s_step[SAMPLER_THREADS], s_ptr[SAMPLER_THREADS], s_sum[32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = nthreads / 32;
  const int t = Tc % dp;
  int before = 0;  // kept tiles in the columns of earlier rounds
  for (int c0 = 0; c0 < Tc; c0 += nthreads) {
    const int c = c0 + (int)threadIdx.x;
    int first = Tr, step = Tr, cnt = 0;
    if (c < Tc) {
      int v = (c - (b - 1)) % dp;
      if (v < 0) v += dp;
      int r = 0;
      auto down = [&]() { ++r; v += t; if (v >= dp) v -= dp; };
      const int most = min(dp, Tr);  // dp rows on, the residue is the same again
      while (v != 0 && r < most) down();
      if (v == 0 && r < Tr) {
        first = r;
        do down(); while (v != 0 && r < Tr);
        step = r - first;
        cnt = v == 0 ? (Tr - 1 - first) / step + 1 : 1;
      }
    }
    int x = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, d);
      if (lane >= d) x += y;
    }
    if (lane == 31) s_sum[warp] = x;
    __syncthreads();
    int base = before, all = 0;
    {
      int w = lane < nwarps ? s_sum[lane] : 0;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, w, d);
        if (lane >= d) w += y;
      }
      all = __shfl_sync(0xffffffffu, w, 31);
      const int mine = __shfl_sync(0xffffffffu, w, warp > 0 ? warp - 1 : 0);
      if (warp > 0) base += mine;
    }
    base += x - cnt;
    if (c < Tc) col_ptr[c] = base;
    s_first[threadIdx.x] = first;
    s_step[threadIdx.x] = step;
    s_ptr[threadIdx.x] = base;
    __syncthreads();
    auto fill = [&](auto zero) {  // ascending rows, counted in the type of `zero`
      using Row = decltype(zero);
      for (int i = warp; i < min(nthreads, Tc - c0); i += nwarps) {
        int32_t* to = col_idx + s_ptr[i];
        int j = lane;
        for (Row r = s_first[i] + lane * (Row)s_step[i]; r < Tr; r += 32 * (Row)s_step[i], j += 32) to[j] = (int)r;
      }
    };
    // beyond 2^25 rows 32 times a distance may be no int (64 bits, or entries counted instead of rows, for all: 0.2 us)
    if (Tr <= 1 << 25) fill(0);
    else fill(0ll);
    before += all;
    __syncthreads();
  }
  if (threadIdx.x == 0) col_ptr[Tc] = before;
}

}  // namespace

ard_status launch_sampler(ard_ctx* ctx, ard_pattern* pat, const unsigned long long* d_cdf, int ndp, uint64_t seed,
                          uint64_t iteration, uint32_t stream_id, int forced_dp, int forced_b, cudaStream_t s,
                          unsigned long long* d_counter, int advance) {
  ARD_CUDA_OK(ard_launch(ctx, ard_sample_kernel, dim3(1), dim3(pat->kind == ARD_TILE ? SAMPLER_THREADS : 256), 0, s, pat->d_hdr, pat->d_idx,
                         pat->d_col_ptr, pat->d_col_idx, pat->d_row_ptr, pat->d_row_idx, d_cdf, ndp,
                         (unsigned long long)seed, (unsigned long long)iteration, stream_id, forced_dp, forced_b,
                         (int)pat->kind, pat->units, pat->Tr, pat->Tc, pat->ts, d_counter, advance));
  ctx->launches++;
  ARD_CUDA_OK(cudaGetLastError());
  return ARD_OK;
}
