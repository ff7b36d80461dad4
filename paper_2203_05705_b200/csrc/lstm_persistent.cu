// Whole-sequence LSTM forward in one cooperative kernel (Sec. 7: the LSTM layer under a row pattern on
// its hidden units; one pattern serves every time step).
//
// The per-step path launches a gate product and a cell kernel per time step, and each launch costs
// more than the 64-row product itself.  Here the recurrence runs inside one kernel:
//   - the input half of the gate pre-activations does not depend on the recurrence: the caller computes
//     x_t . W_x for all steps with one large product beforehand and leaves it where the gate activations
//     of step t will be stored; the kernel adds it in its epilogue and handles the recurrent half only;
//   - every CTA owns U kept hidden units, i.e. 4 U gate columns (i|f|g|o x U), and keeps its slice of
//     the weight, [4 U rows][H] bf16, in shared memory.  The grid is sized for nothing dropped with U = 8 (12 for layers
//     of more than 8 units per SM); the drawn pattern then takes the smallest U of 4, 8, 12 with which the kept units
//     fit the grid: the cell update is a serial chain per (batch row, unit) pair, and a second pair per thread costs
//     more than the additional CTAs' reads of h (us per step: 64 rows, 512 of 1024 units kept, 4.7 with U = 8, 4.0 with
//     4; 20 rows, 750 of 1500 kept, 5.4 with 12, 4.4 with 8; 128 rows, 64 kept, 4.6 with 8, 3.6 with 4);
//   - per step it loads h_{t-1} (TMA boxes of up to 64 rows x 64 columns) into a ring of slots, one quarter of the
//     blocks per loading warp.  Usually every block of a step has a slot of its own, so all loads of a step are in
//     flight together; a slice so large that fewer slots fit re-uses them within the step.  The warp that loads a
//     quarter also issues its products (tcgen05.mma, M = 64 or 128, N = 4 U, accumulators in tensor memory,
//     double-buffered over steps): one thread issuing box after box paces at ~410 SM cycles per box, the lanes of a
//     warp ~70 cycles apart, and a tcgen05.mma this narrow costs its issuing thread ~110 cycles;
//   - the accumulator rows move to shared memory, then all 11 compute warps apply the cell
//     update to the (batch row, unit) pairs, keep c in registers, and write h_t (bf16) into the operand
//     of step t+1 and, after signalling, c_t and the gate activations for BPTT;
//   - the h columns wait for the grid-wide barrier that says h_{t-1} is complete;
//   - under a pattern (period > 1) the dropped units of h_{t-1} are exact zeros, so the contraction runs over
//     the kept units only: the cell update also writes h_t into a compact copy (column j = j-th kept unit, two
//     buffers in context scratch), which is the operand of step t+1, and the slice holds the kept fan-in
//     columns of the weight only.  Those stride the weight's contiguous dimension, which a TMA box cannot
//     follow, so the CTA gathers its slice with plain loads, once per sequence, straight into the swizzled
//     layout the MMA reads.  A step's loads and MMAs shrink with the kept count (forward of 35 steps, batch 64,
//     H = 1024: 218 -> 189 us at a period of 2, 204 -> 146 us at 8).  This form reads neither [x | h] nor the weight
//     through a descriptor, so it also serves layers whose rows are off the 16-byte grid, dense draws included
//     (1500 units, batch 20, 35 steps, a period of 2: see launch_lstm_forward_persistent).
// Patterns that keep 768 units or fewer run in lstm_cluster.cu where the device has room for its clusters (on 148 SMs it has).  The forms
// for few kept units here (U = 4; BPTT without the exchange) are for devices and partitions that have none, and for the option that refuses
// those launches, with which their tests reach them.
// The grid barrier is an arrival counter in global memory: after its stores and a fence each CTA adds 1,
// and the relay thread of each CTA polls for t * (number of CTAs with units) before step t.  The CTA that leaves
// last sets the counter back to zero.  The launch is cooperative, so all CTAs are resident; every wait is bounded
// (2 s) and a CTA that gives up sets the status word, which the others poll, so the kernel always returns.
#include "ard_internal.h"
#include "sm100_ptx.h"

namespace {

constexpr int LP_BK = 64;                    // contraction block: 64 bf16 = one 128-byte swizzle row
constexpr int LP_GROUPS = 4;                 // the blocks of a step are dealt to this many loading warps
constexpr int LP_SLOTS = 24;                 // most slots of a loading warp
constexpr int LP_ROW_BOX = 64 * LP_BK * 2;   // largest TMA box of the activations: 64 batch rows x 64 columns
constexpr int LP_THREADS = 512;              // warps 0-10 cell update (0-3 also read TMEM: lane quadrant = warp),
constexpr int LP_MATH = 352;                 //   warp 11 barrier relay, warps 12-15 loads and products
constexpr int LP_BAR_BYTES = 2048;           // barriers and flags at the start of shared memory
constexpr int LP_SMEM_MAX = 227 * 1024;

// Words of a context's barrier area (see ard_ctx::d_grid_bar): arrivals, CTAs that left.
constexpr int LP_BAR_WORD = 32;

// Batch rows are staged in 8-row groups of one KiB: bytes of one 64-column block of the activations.
__host__ __device__ inline int lstm_box_rows(int B) { return B >= 64 ? 64 : (B + 7) / 8 * 8; }
__host__ __device__ inline int lstm_a_block(int B) { return (B + 63) / 64 * lstm_box_rows(B) * LP_BK * 2; }

// Shared-memory plan of one recurrence: the ring of activation slots and the resident weight slice.  `blocks`
// contraction blocks per step, `w_block` bytes of the slice per block, `zs` bytes of staged sums.
struct LstmPlan {
  int gsz;        // blocks per loading warp
  int cap;        // slots per loading warp (== gsz: no slot is used twice in a step); 0: does not fit
  int zs_shared;  // the staged sums share the start of the ring
  int behind;     // bytes from the slice on, without the staged sums
  int bytes;      // everything behind the barriers
};
// An MMA reads 64 or 128 rows (lstm_mma_rows) however many the batch has, so what lies behind a slot has to exist: 16 KiB
// from the start of the last slot serve both.  tail: bytes that the MMA may read behind the slice.
__host__ __device__ inline LstmPlan lstm_plan(int blocks, int a_block, int w_block, int tail, int zs, int smem_bytes) {
  LstmPlan r;
  r.gsz = (blocks + LP_GROUPS - 1) / LP_GROUPS;
  const int want = r.gsz < LP_SLOTS ? r.gsz : LP_SLOTS;
  r.behind = blocks * w_block + tail > 16384 - a_block ? blocks * w_block + tail : 16384 - a_block;
  const int avail = smem_bytes - 1024 - LP_BAR_BYTES - r.behind;
  auto slots = [&](int bytes) {
    const int c = bytes <= 0 ? 0 : bytes / (LP_GROUPS * a_block);
    return c < want ? c : want;
  };
  r.cap = slots(avail);
  r.zs_shared = LP_GROUPS * r.cap * a_block >= zs;
  if (!r.zs_shared) r.cap = slots(avail - zs);
  r.bytes = LP_GROUPS * r.cap * a_block + r.behind + (r.zs_shared ? 0 : zs);
  return r;
}

// Rows of the products: an instruction of 64 reads half as much of the activations' slots as one of 128, and that is what
// paces these narrow products (us per step, forward / BPTT: 20 rows, 512 of 1024 units kept, 3.65 / 3.86 with 128, 3.48 /
// 3.65 with 64; 64 rows 4.02 / 4.20 and 3.95 / 4.10).  Its accumulator has 16 rows in each 32 lanes of tensor memory.
__host__ __device__ inline int lstm_mma_rows(int B) { return B <= 64 ? 64 : 128; }

struct LstmFwdParams {
  TcMap mapXH;    // [(T+1)*B][I+H], boxes of box_rows x 64 columns (used as encoded; not by the compact form)
  TcMap mapW[4];  // per gate: [H rows][I+H], boxes of 8 rows x 64 columns; specialised to the kept rows by the kernel
  TcMap mapHc;    // [2*B][ldhc]: the compact copies of h_{t-1} and h_t, boxes of box_rows x 64 columns
  CUtensorMap* tm_slots;  // this launch's descriptor scratch: ARD_TM_LSTM_SLOTS slots per block
  const int32_t* hdr;
  int T, B, I, H;
  const __nv_bfloat16* W;  // the weight itself, [4H][ldw]: its kept recurrent columns are gathered by the kernel
  int ldw;
  __nv_bfloat16* Hc;  // two buffers [B][ldhc]: column j = the j-th kept unit (nullptr: no compact recurrence)
  int ldhc;
  int always_compact; // the operands cannot be described to the TMA unit: the compact form for dense draws too
  int add_zx;         // the products of the other columns are waiting in G[t] (same layout as the gates)
  float alpha;
  __nv_bfloat16* XH;
  const float* bias;  // [4][H] or nullptr
  float* C;           // [T+1][B][H] compact
  float* G;           // [T][B][4H]: gate blocks of width H, compact inside a block
  unsigned int* bar;  // arrival counter, zero at launch; [1]: CTAs that left
  int* status;
  int smem_bytes;     // dynamic shared memory of this launch
  int above, up_to;   // a pattern that keeps no more than the one, or more than the other, is another kernel's
};

__device__ __forceinline__ unsigned int ld_acquire_u32(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Waits until the arrival counter reaches `target`.  Gives up after the time limit or when another CTA
// has already recorded a failure.
__device__ bool grid_wait(const unsigned int* bar, unsigned int target, volatile int* abort_flag, int* status) {
  if (ld_acquire_u32(bar) >= target) return true;
  const unsigned long long t0 = global_ns();
  for (int spin = 1;; ++spin) {
    if (ld_acquire_u32(bar) >= target) return true;
    if (*abort_flag) return false;
    if ((spin & 63) == 0) {
      if (*reinterpret_cast<volatile int*>(status) != 0) { *abort_flag = 1; return false; }
      if (global_ns() - t0 > WAIT_LIMIT_NS) {
        *abort_flag = 1;
        atomicMax(status, (int)ARD_ERR_TIMEOUT);
        return false;
      }
    }
  }
}

// The CTA that leaves last re-arms the grid-wide counter for the next launch.  Called by one thread per CTA after all
// of its waits and arrivals.
// Is the drawn pattern this launch's, with more than `above` units kept and at most `up_to`?  The same for all CTAs; asked before anything is
// set up, because a launch that does nothing stands in front of the next one's work.
__device__ __forceinline__ bool lstm_take_pattern(const int32_t* hdr, int above, int up_to) {
  pdl_wait_prior_grids();
  const int n_keep = hdr[HDR_NKEEP];
  return n_keep > above && n_keep <= up_to;
}

// With `above`, the kernel of the patterns that keep fewer units is enqueued behind this one and has nothing to do: it may be scheduled while
// this one runs, its CTAs then leave as soon as this one ends.  Only behind this one's allocation of tensor memory: a CTA of another kernel
// on the same SM that held the columns while it waits for this kernel's end would wait for good (that kernel's CTAs need an SM of their own).
// us of the whole pass, a dense draw of a distribution whose other draws are the clusters', 64 rows x 1024 units and 20 rows x 1500 over 35
// steps, 16 x 1024 over 8: with the grid-wide kernels alone 509, 596 and 151; with the others behind them, both kinds asking for the pattern
// once they are set up, 521, 609 and 156; as it is now 506, 595 and 151.
__device__ __forceinline__ void lstm_next_launch(int above) {
  if (above > 0) pdl_launch_dependents();
}

__device__ __forceinline__ void grid_leave(unsigned int* bar) {
  __threadfence();
  if (atomicAdd(bar + 1, 1u) == gridDim.x - 1) {
    bar[0] = 0u;
    bar[1] = 0u;
    __threadfence();
  }
}

// Sums of the first `groups` issuing warps' accumulators (`stride` columns apart) over N consecutive columns of this
// warp's 32 rows.
template <int N>
__device__ __forceinline__ void lstm_sum_groups(uint32_t taddr, int stride, int groups, float (&z)[N]) {
  static_assert(N == 4 || N == 8);
  uint32_t y[LP_GROUPS][N];
#pragma unroll
  for (int c = 0; c < LP_GROUPS; ++c) {
    if (c >= groups) continue;
    const uint32_t a = taddr + (uint32_t)(c * stride);
    if constexpr (N == 8)
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                   : "=r"(y[c][0]), "=r"(y[c][1]), "=r"(y[c][2]), "=r"(y[c][3]), "=r"(y[c][4]), "=r"(y[c][5]), "=r"(y[c][6]), "=r"(y[c][7])
                   : "r"(a) : "memory");
    else
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                   : "=r"(y[c][0]), "=r"(y[c][1]), "=r"(y[c][2]), "=r"(y[c][3]) : "r"(a) : "memory");
  }
  tmem_ld_wait();
#pragma unroll
  for (int i = 0; i < N; ++i) {
    z[i] = __uint_as_float(y[0][i]);
#pragma unroll
    for (int c = 1; c < LP_GROUPS; ++c)
      if (c < groups) z[i] += __uint_as_float(y[c][i]);
  }
}
// One step's blocks [0, n) of a loading warp, called by all its lanes: lane i requests block i into slot i while slots
// last; lane 0 multiplies the blocks as they arrive and requests the later ones into the slots that fell free.  A slot's
// barriers are phased by how often it has been used: `step` steps before this one.  request(block, slot) issues the
// copies of a block (and announces their bytes); multiply(block, slot, first) its products.  ok: lane 0's verdict.
template <typename Request, typename Multiply, typename FullBar, typename FreeBar>
__device__ __forceinline__ bool lstm_stream_blocks(int n, int cap, int step, int lane, bool ok, FullBar full_bar, FreeBar free_bar,
                                                   volatile int* abort_flag, int* status, Request request, Multiply multiply) {
  if (lane < n && lane < cap) request(lane, lane);
  __syncwarp();
  if (lane == 0 && ok) {
    auto count = [&](int slot, int i) { return (uint32_t)(step * ((n - 1 - slot) / cap + 1) + i / cap); };
    for (int i = 0; i < n; ++i) {
      const int slot = i % cap;
      if (!mbar_wait(full_bar(slot), count(slot, i) & 1u, abort_flag, status)) { ok = false; break; }
      tc_fence_after();
      multiply(i, slot, i == 0);
      if (n > cap) {
        // refill the slot of the block before this one, whose products were issued a block ago (with one slot: of this one)
        tc_commit(free_bar(slot));
        const int j = cap > 1 ? i - 1 : i;
        if (j >= 0 && j + cap < n) {
          const int sj = j % cap;
          if (!mbar_wait(free_bar(sj), count(sj, j) & 1u, abort_flag, status)) { ok = false; break; }
          request(j + cap, sj);
        }
      }
    }
  }
  __syncwarp();
  return ok;
}

// The gate functions of the per-step kernels (aux_kernels.cu), so that a layer's results do not depend on which of the two it takes (those in
// lstm_cluster.cu have a tanh of their own, as close to the exact one).
// 1 - 2 / (1 + exp(2x)) in tanhf's place cancels near zero: gates of size 0.01 were off by 7e-6 to 2e-5 of themselves, now by
// 1e-7 to 9e-7 (the sums of the pre-activations among it), and it was no faster (35 steps, 64 rows, 512 of 1024 units kept,
// forward plus BPTT 372.0 us, with tanhf 370.7; 20 rows, 750 of 1500 424.7 and 420.8).
__device__ __forceinline__ float sigmoid_fast(float x) { return 1.f / (1.f + __expf(-x)); }

// Barriers behind the slots' full and free ones (byte offsets): accumulators complete / read (two each), weight slice
// complete, h_{t-1} complete (relayed from the grid barrier); behind them the flags.
constexpr uint32_t LF_TFULL = 8 * 2 * LP_GROUPS * LP_SLOTS;
constexpr uint32_t LF_TEMPTY = LF_TFULL + 16;
constexpr uint32_t LF_WFULL = LF_TEMPTY + 16;
constexpr uint32_t LF_HREADY = LF_WFULL + 8;

// The recurrence with U units per CTA.  compact: see below.
template <int U>
__device__ __forceinline__ void lstm_forward_body(const LstmFwdParams& p, uint8_t* smem, uint32_t base, uint32_t tmem_base,
                                                  volatile int* abort_flag, int dp, int bb, int n_keep, bool compact) {
  constexpr int N = 4 * U;                             // gate columns per CTA
  constexpr int W_BLOCK = N * LP_BK * 2;               // one contraction block of the resident weight slice
  constexpr int ZS_LD = N + 1;                         // staged pre-activations: [rows][N + 1] floats
  constexpr int PAIRS = (128 * U + LP_MATH - 1) / LP_MATH;  // (row, unit) pairs per thread
  const int KH = p.I + p.H;
  const int box_rows = lstm_box_rows(p.B), row_boxes = (p.B + 63) / 64;
  const uint32_t a_block = (uint32_t)lstm_a_block(p.B);
  auto full_bar = [&](int g, int s) { return base + 8u * (g * LP_SLOTS + s); };
  auto free_bar = [&](int g, int s) { return base + 8u * ((LP_GROUPS + g) * LP_SLOTS + s); };
  auto tfull_bar = [&](int a) { return base + LF_TFULL + 8u * a; };
  auto tempty_bar = [&](int a) { return base + LF_TEMPTY + 8u * a; };
  const uint32_t wfull_bar = base + LF_WFULL, hready_bar = base + LF_HREADY;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  const int n_active = (n_keep + U - 1) / U;       // CTAs that own units (the others only tear down)
  const int j0 = (int)blockIdx.x * U;              // first kept unit (compact index) of this CTA
  const bool active = (int)blockIdx.x < n_active;
  // The dropped units of h_1 .. h_T, read by nobody before the kernel ends when the recurrence is compact: where enough
  // of the grid's CTAs have no units, these write the zeros meanwhile; otherwise the threads of the cell update do after
  // their CTA has signalled (as stores ahead of the signal they cost 0.3 us a step).
  const int n_idle = (int)gridDim.x - n_active;
  const bool idle_zeros = n_idle >= 8;
  // Under a pattern the dropped units of h_{t-1} are exact zeros (Sec. 3.1), so the recurrent contraction runs over
  // the kept units alone: the operand of a step is the compact copy of h_{t-1} (column j = j-th kept unit) that the
  // cell update writes beside the full-width one, and the weight slice holds the kept fan-in columns only.  Those
  // stride the weight's contiguous dimension, which no TMA box can follow, so the CTA gathers its slice itself,
  // once per sequence, straight into the swizzled layout the MMA reads.
  const int hs = compact ? 1 : 0;  // the compact h_0 is made by the kernel: one more grid-wide hand-over, before step 0
  const int nkb = ((compact ? n_keep : p.H) + LP_BK - 1) / LP_BK;
  // The staged pre-activations share the start of the ring where they fit: they are written after the step's MMAs
  // have completed and read before this CTA releases h_t, and the next loads are issued only after every CTA has
  // released.
  const LstmPlan plan = lstm_plan(nkb, (int)a_block, W_BLOCK, 0, (p.B + 31) / 32 * 32 * ZS_LD * 4, p.smem_bytes);
  const int gsz = plan.gsz, cap = plan.cap;
  const uint32_t sA = base + LP_BAR_BYTES;
  const uint32_t sW = sA + (uint32_t)(LP_GROUPS * cap) * a_block;
  float* zs = reinterpret_cast<float*>(smem + (plan.zs_shared ? sA - base : sW - base + (uint32_t)plan.behind));
  if (compact) {
    if (active) {
      const int nchunks = nkb * 8;  // 16-byte pieces of a slice row
      for (int task = threadIdx.x; task < N * nchunks; task += LP_THREADS) {
        const int r = task / nchunks, ch = task - r * nchunks;
        const int g = r / U, k = r - g * U, j = j0 + k;
        uint32_t w[4] = {0u, 0u, 0u, 0u};
        if (j < n_keep) {
          const __nv_bfloat16* src = p.W + ((size_t)g * p.H + bb + (size_t)j * dp) * p.ldw + p.I + bb + (size_t)ch * 8 * dp;
          uint32_t e[8];
#pragma unroll
          for (int q = 0; q < 8; ++q)
            e[q] = (ch * 8 + q < n_keep) ? (uint32_t)__ldg(reinterpret_cast<const unsigned short*>(src) + (size_t)q * dp) : 0u;
#pragma unroll
          for (int q = 0; q < 4; ++q) w[q] = e[2 * q] | (e[2 * q + 1] << 16);
        }
        // 128-byte swizzle: the 16-byte piece c of row k of an 8-row group sits at piece c ^ k
        uint8_t* dst = smem + (sW - base) + (size_t)(ch >> 3) * W_BLOCK + (r >> 3) * 1024 + (r & 7) * 128 + (((ch & 7) ^ (r & 7)) << 4);
        *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
      }
      fence_proxy_async_smem();  // generic-proxy stores -> the tensor core's reads
    }
    __syncthreads();
  }

  if (active) {
    if (warp == 11) {
      // ===================== weight loader and barrier relay =====================
      // Loads the weight slice (lane = contraction block), then relays the grid barrier of every step to
      // the warps of this CTA through a shared-memory barrier.
      // The gates' weight descriptors become those of the kept rows (the weight area, still empty, is the work area).
      if (compact) {
        // the slice is in place already (gathered by the whole CTA above)
        if (lane == 0) mbar_arrive(wfull_bar);
      } else {
        CUtensorMap* slots = p.tm_slots + (size_t)blockIdx.x * ARD_TM_LSTM_SLOTS;
        const CUtensorMap* mapW[4];
#pragma unroll
        for (int g = 0; g < 4; ++g)
          mapW[g] = tensormap_specialise(&p.mapW[g], dp, bb + 1, n_keep, smem + (sW - base) + 128 * g, slots + g, lane);
        fence_proxy_async_smem();
        if (lane < nkb && dp > 1) {
#pragma unroll
          for (int g = 0; g < 4; ++g) tensormap_acquire(mapW[g]);
        }
        if (lane == 0) mbar_arrive_expect_tx(wfull_bar, (uint32_t)nkb * W_BLOCK);
        __syncwarp();
        for (int kb = lane; kb < nkb; kb += 32) {
#pragma unroll
          for (int g = 0; g < 4; ++g)
            tma_load_2d(sW + kb * W_BLOCK + g * 1024, mapW[g], wfull_bar, p.I + kb * LP_BK, j0);
        }
      }
      if (lane == 0) {
        for (int t = 1 - hs; t < p.T; ++t) {
          // h_{t-1} is complete when every CTA with units has arrived t times (once more with a compact h_0)
          if (!grid_wait(p.bar, (unsigned)(t + hs) * (unsigned)n_active, abort_flag, p.status)) break;
          mbar_arrive(hready_bar);
        }
      }
    } else if (warp >= 12) {
      // ===================== loaders and MMA issuers: warp 12 + g owns the contraction blocks of group g =====================
      const int g = warp - 12;
      const int kb0 = g * gsz, n = max(0, min(nkb - kb0, gsz));
      const CUtensorMap* mapXH = compact ? &p.mapHc.tm : &p.mapXH.tm;  // kernel parameters, used as encoded
      const uint32_t idesc = make_idesc(N, false, false, lstm_mma_rows(p.B));
      bool ok = (lane != 0) || mbar_wait(wfull_bar, 0u, abort_flag, p.status);
      for (int t = 0; t < p.T; ++t) {
        const int acc = t & 1;
        // this group's slots are free once the MMAs of the previous step have completed
        if (ok && t > 0 && !mbar_wait(tfull_bar((t - 1) & 1), (uint32_t)((t - 1) >> 1) & 1u, abort_flag, p.status)) ok = false;
        if (ok && t + hs > 0 && n > 0) {
          if (!mbar_wait(hready_bar, (uint32_t)(t - 1 + hs) & 1u, abort_flag, p.status)) ok = false;
          asm volatile("fence.proxy.async.global;" ::: "memory");  // generic-proxy stores of other CTAs -> TMA reads
        }
        if (ok && lane == 0 && !mbar_wait(tempty_bar(acc), ((uint32_t)(t >> 1) & 1u) ^ 1u, abort_flag, p.status)) ok = false;
        if (!__all_sync(0xffffffffu, ok)) break;
        const uint32_t d_tmem = tmem_base + (uint32_t)((acc * LP_GROUPS + g) * N);
        auto request = [&](int i, int slot) {
          // full width: columns of h_{t-1} in [x_t | h_{t-1}], rows of step t; compact: the buffer that holds h_{t-1}
          const int x = compact ? (kb0 + i) * LP_BK : p.I + (kb0 + i) * LP_BK, y = compact ? (t & 1) * p.B : t * p.B;
          mbar_arrive_expect_tx(full_bar(g, slot), a_block);
          for (int rb = 0; rb < row_boxes; ++rb)
            tma_load_2d(sA + (uint32_t)(g * cap + slot) * a_block + rb * LP_ROW_BOX, mapXH, full_bar(g, slot), x, y + rb * box_rows);
        };
        auto multiply = [&](int i, int slot, bool first) {
          // descriptors by addition: the start-address field counts 16-byte units
          const uint64_t ad = make_desc(sA + (uint32_t)(g * cap + slot) * a_block, 16, 1024), bd = make_desc(sW + (kb0 + i) * W_BLOCK, 16, 1024);
#pragma unroll
          for (int s = 0; s < LP_BK / 16; ++s) tc_mma_bf16(d_tmem, ad + 2 * s, bd + 2 * s, idesc, (!first || s != 0) ? 1u : 0u);
        };
        ok = lstm_stream_blocks(n, cap, t, lane, ok, [&](int s) { return full_bar(g, s); }, [&](int s) { return free_bar(g, s); },
                                abort_flag, p.status, request, multiply);
        if (lane == 0 && ok) tc_commit(tfull_bar(acc));  // this quarter is complete
        __syncwarp();
      }
    } else {
      // ===================== cell update (warps 0-10) =====================
      const int tid = threadIdx.x;  // 0 .. LP_MATH-1
      const size_t ldxh = (size_t)KH;
      const int npairs = p.B * U;                    // (batch row, unit) pairs of this CTA; pair q = row * U + k
      const int nvalid = min(U, n_keep - j0);        // units this CTA really owns (>= 1)
      const int qrows = lstm_mma_rows(p.B) / 4;      // batch rows in each 32 lanes of tensor memory
      float creg[PAIRS];
#pragma unroll
      for (int i = 0; i < PAIRS; ++i) {
        const int q = tid + i * LP_MATH;
        const int row = q / U, k = q % U;
        creg[i] = (q < npairs && k < nvalid) ? p.C[(size_t)row * p.H + j0 + k] : 0.f;
      }
      if (compact) {
        // the compact copy of h_0 (buffer 0): this CTA's units of every row; the last CTA with units also clears
        // the columns up to the next multiple of 64 in both buffers (they meet the zeros of the weight slice)
        for (int q = tid; q < npairs; q += LP_MATH) {
          const int row = q / U, k = q % U;
          if (k < nvalid) p.Hc[(size_t)row * p.ldhc + j0 + k] = p.XH[(size_t)row * ldxh + p.I + bb + (size_t)(j0 + k) * dp];
        }
        if ((int)blockIdx.x == n_active - 1) {
          const int npad = nkb * LP_BK - n_keep;
          for (int q = tid; q < 2 * p.B * npad; q += LP_MATH) {
            const int row = q / npad, c = q - row * npad;
            p.Hc[(size_t)row * p.ldhc + n_keep + c] = __float2bfloat16_rn(0.f);
          }
        }
        asm volatile("bar.sync 1, 352;" ::: "memory");
        if (tid == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p.bar) : "memory");
      }
      // Zeros of h_t: the j-th kept unit owns the units [j * dp, (j + 1) * dp), the last one the tail.
      auto zeros_of = [&](int row, int t, int j) {
        const int first = j * dp, last = j == n_keep - 1 ? p.H : min(p.H, first + dp), own = bb + j * dp;
        __nv_bfloat16* hrow = p.XH + ((size_t)(t + 1) * p.B + row) * ldxh + p.I;
        for (int u = first; u < last; ++u)
          if (u != own) hrow[u] = __float2bfloat16_rn(0.f);
      };
      bool ok = true;
      for (int t = 0; t < p.T && ok; ++t) {
        const int acc = t & 1;
        // what does not depend on the recurrence is fetched before the wait: x_t . W_x and the bias
        float zadd[PAIRS][4];
#pragma unroll
        for (int i = 0; i < PAIRS; ++i) {
          const int q = tid + i * LP_MATH;
          const int row = q / U, k = q % U;
          zadd[i][0] = zadd[i][1] = zadd[i][2] = zadd[i][3] = 0.f;
          if (q < npairs && k < nvalid) {
            if (p.add_zx) {  // left in the slot of this step's gate activations
              const float* zx = p.G + ((size_t)t * p.B + row) * 4 * p.H + j0 + k;
#pragma unroll
              for (int g = 0; g < 4; ++g) zadd[i][g] = __ldcg(zx + (size_t)g * p.H);
            }
            if (p.bias) {
              const int u = bb + (j0 + k) * dp;
#pragma unroll
              for (int g = 0; g < 4; ++g) zadd[i][g] += p.bias[g * p.H + u];
            }
          }
        }
        if (warp < 8) {
          // accumulator rows -> shared memory; warps 4-7 take the second half of the columns
          if (!mbar_wait(tfull_bar(acc), (uint32_t)(t >> 1) & 1u, abort_flag, p.status)) ok = false;
          if (__all_sync(0xffffffffu, ok)) {
            tc_fence_after();
            const int quadrant = warp & 3;
            if (quadrant * qrows < p.B) {
              const uint32_t t_row = tmem_base + ((uint32_t)(quadrant * 32) << 16) + (uint32_t)(acc * LP_GROUPS * N);
              const int ngroups = (nkb + gsz - 1) / gsz;  // accumulators that received MMAs
              float* zr = zs + (quadrant * qrows + lane) * ZS_LD;
#pragma unroll
              for (int i0 = 0; i0 < N / 2; i0 += 8) {
                const int c0 = (warp >> 2) * (N / 2) + i0;
                float z[8];
                lstm_sum_groups<8>(t_row + (uint32_t)c0, N, ngroups, z);
                if (lane < qrows) {
#pragma unroll
                  for (int i = 0; i < 8; ++i) zr[c0 + i] = z[i];
                }
              }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(tempty_bar(acc));  // the accumulator has been read
          }
        }
        // every compute thread learns about a failed wait through the flag in shared memory
        asm volatile("bar.sync 2, 352;" ::: "memory");
        if (*abort_flag) { ok = false; break; }
        // Cell update (Sec. 7).  h first, because the other CTAs wait for it; c_t and the gate
        // activations, which only BPTT reads, after the CTA has signalled.
        float gi[PAIRS], gf[PAIRS], gg[PAIRS], go[PAIRS];
#pragma unroll
        for (int i = 0; i < PAIRS; ++i) {
          const int q = tid + i * LP_MATH;
          const int row = q / U, k = q % U;
          if (q < npairs && k < nvalid) {
            const int u = bb + (j0 + k) * dp;
            const float* zr = zs + row * ZS_LD;
            const float zi = zr[k] + zadd[i][0], zf = zr[U + k] + zadd[i][1];
            const float zg = zr[2 * U + k] + zadd[i][2], zo = zr[3 * U + k] + zadd[i][3];
            gi[i] = sigmoid_fast(zi);
            gf[i] = sigmoid_fast(zf);
            gg[i] = tanhf(zg);
            go[i] = sigmoid_fast(zo);
            creg[i] = gf[i] * creg[i] + gi[i] * gg[i];
            const __nv_bfloat16 h = __float2bfloat16_rn(p.alpha * go[i] * tanhf(creg[i]));
            p.XH[((size_t)(t + 1) * p.B + row) * ldxh + p.I + u] = h;
            if (compact) p.Hc[((size_t)((t + 1) & 1) * p.B + row) * p.ldhc + j0 + k] = h;
            else if (dp > 1) zeros_of(row, t, j0 + k);  // operands of the next step's product
          }
        }
        // publish h_t: all stores of the CTA, then one release-add for the CTA (the staged sums may lie in the
        // ring, which the TMA unit overwrites next: generic-proxy accesses first)
        fence_proxy_async_smem();
        asm volatile("bar.sync 1, 352;" ::: "memory");
        if (tid == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p.bar) : "memory");
#pragma unroll
        for (int i = 0; i < PAIRS; ++i) {
          const int q = tid + i * LP_MATH;
          const int row = q / U, k = q % U;
          if (q < npairs && k < nvalid) {
            p.C[((size_t)(t + 1) * p.B + row) * p.H + j0 + k] = creg[i];
            float* g_out = p.G + ((size_t)t * p.B + row) * 4 * p.H + j0 + k;
            g_out[0] = gi[i];
            g_out[p.H] = gf[i];
            g_out[2 * p.H] = gg[i];
            g_out[3 * p.H] = go[i];
            if (compact && dp > 1 && !idle_zeros) zeros_of(row, t, j0 + k);
          }
        }
      }
    }
  }

  if (!active && compact && dp > 1 && idle_zeros) {
    const int rows = p.T * p.B;
    for (int r = (int)blockIdx.x - n_active; r < rows; r += n_idle) {
      __nv_bfloat16* hrow = p.XH + ((size_t)p.B + r) * KH + p.I;
      for (int u = threadIdx.x; u < p.H; u += LP_THREADS)
        if (u < bb || (u - bb) % dp != 0) hrow[u] = __float2bfloat16_rn(0.f);
    }
  }
}

// U: units per CTA at most; the layer fits the grid with U units per CTA when nothing is dropped.
template <int U>
__global__ void __launch_bounds__(LP_THREADS, 1) ard_lstm_forward_kernel(const __grid_constant__ LstmFwdParams p) {
  constexpr uint32_t TMEM_COLS = 2 * LP_GROUPS * 4 * U <= 256 ? 256 : 512;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t base = (raw_addr + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw_addr);
  uint8_t* misc = smem + LF_HREADY + 8;
  volatile uint32_t* tmem_ptr_smem = reinterpret_cast<volatile uint32_t*>(misc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 4);
  const int warp = threadIdx.x >> 5;
  if (!lstm_take_pattern(p.hdr, p.above, p.up_to)) return;

  if (threadIdx.x < 2 * LP_GROUPS * LP_SLOTS) mbar_init(base + 8u * threadIdx.x, 1);  // slots: full, free
  if (threadIdx.x == 0) {
    for (int a = 0; a < 2; ++a) {
      mbar_init(base + LF_TFULL + 8u * a, LP_GROUPS);  // one commit per MMA issuer
      mbar_init(base + LF_TEMPTY + 8u * a, 8);       // one arrival per TMEM-reading warp
    }
    mbar_init(base + LF_WFULL, 1);
    mbar_init(base + LF_HREADY, 1);
    *abort_flag = 0;
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  if (warp == 15) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_ptr_smem)), TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_ptr_smem;
  lstm_next_launch(p.above);

  const int dp = p.hdr[HDR_DP], bb = p.hdr[HDR_B] - 1, n_keep = p.hdr[HDR_NKEEP], ctas = (int)gridDim.x;
  const bool compact = p.Hc != nullptr && (dp > 1 || p.always_compact);
  if (compact && n_keep <= 4 * ctas) lstm_forward_body<4>(p, smem, base, tmem_base, abort_flag, dp, bb, n_keep, compact);
  else if (U == 8 || (compact && n_keep <= 8 * ctas)) lstm_forward_body<8>(p, smem, base, tmem_base, abort_flag, dp, bb, n_keep, compact);
  else lstm_forward_body<U>(p, smem, base, tmem_base, abort_flag, dp, bb, n_keep, compact);

  // ---- teardown ----
  tc_fence_before();
  __syncwarp();  // lanes that left their role's loop one by one arrive at the block-wide barrier together
  __syncthreads();
  if (threadIdx.x == 0) grid_leave(p.bar);
  if (warp == 15) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
}


// ======================================================================================================
// Whole-sequence BPTT recurrence (Sec. 7), the counterpart of the kernel above.
//
// Per step t = T-1 .. 0 the recurrence needs  dh_t = upstream_t + dz_{t+1} . W_h  (contraction over the
// 4 * n_keep kept gate rows, output over the kept hidden units), then the cell adjoint gives dz_t.  A CTA owns U KEPT
// units: it keeps their cell gradient in registers and writes their columns of dz_t.  If it contracted for its own
// units only, every CTA would have to read all of dz_{t+1} in every step (256 KB at batch 64 and 512 kept units),
// which is what bounds a step then.  So CTAs work in clusters of LB_CLUSTER: the cluster owns LB_CLUSTER * U units and
// CTA r contracts the r-th share of the blocks of 64 gate rows for all of them.  A step is
//   1. dz_{t+1} is complete (grid barrier, relayed): TMA-load this CTA's blocks of it into the ring of slots of the
//      forward kernel and multiply (tcgen05.mma M = 64 or 128, N = LB_CLUSTER * U, four issuing warps with an accumulator
//      each) by the resident weight slice: the fan-out weights of the cluster's units, [units][gate rows] (K-major),
//      gathered by the kernel once per sequence;
//   2. send the sums of every CTA's units to that CTA's shared memory (st.async: the bytes themselves complete the
//      receiver's mbarrier, so the exchange costs one trip between SMs and no barrier);
//   3. the owner adds the shares in a fixed order and the upstream gradient, applies the cell adjoint with dc in a
//      register, stores dz_t (bf16, the operand of the next step and of the weight-gradient products), arrives.
// A pattern that keeps so few units that all of a step's blocks fit beside the slice of one CTA's own units may do
// without the exchange (see LB_WHOLE_BLOCKS): every CTA contracts whole rows for its own units.  The same form serves
// layers whose CTAs do not all fit the device in clusters.  After t = 0 one more product gives the gradient of h_0.
// The input half of d[x, h] and the weight gradient are large products over all T*B rows that the caller runs
// afterwards.  No operand of the caller but dz is read through a descriptor, and dz lives in a padded copy in context
// scratch where the caller's rows are off the 16-byte grid.
// The grid barrier is one arrival counter: every CTA that takes part arrives once per step, after all of its stores.
// us per step, before (partial sums through global memory and a second grid barrier, or whole contractions in every CTA;
// the cell adjoint formed behind the wait; 8 units per CTA) and now: 64 rows, 512 of 1024 units kept 7.4 -> 4.1, all
// kept 8.6 -> 6.1; 128 rows, 512 of 1024 kept 10.1 -> 5.6; 20 rows, 750 of 1500 kept 9.7 -> 4.8, all kept 25.4 -> 7.3.
// About 2.8 of it are what a step of any size costs: stores, barrier, TMA, a few narrow MMAs, the exchange.
constexpr int LB_CLUSTER = 4;     // of 148 SMs 132 can be used by clusters of 4, 120 by clusters of 8
constexpr int LB_COLS = 64;       // tensor-memory columns of an issuing warp's accumulator (at most LB_CLUSTER * 12 used)
constexpr int LB_THREADS = 512;   // warps 0-10 adjoint (0-7 also read TMEM), 11 relay, 12-15 load + MMA
constexpr int LB_MATH = 352;
// A step of this many blocks is contracted whole by every CTA: one block per issuing warp either way, and no exchange
// (64 rows, 64 of 1024 units kept: 3.22 us per step against 3.42 with it; 128 kept, 8 blocks: 3.68 against 3.44).
constexpr int LB_WHOLE_BLOCKS = 4;
constexpr uint32_t LB_TFULL = 8 * 2 * LP_GROUPS * LP_SLOTS;  // barriers behind the slots' full and free ones
constexpr uint32_t LB_HREADY = LB_TFULL + 8;                 // dz of the previous step is complete
constexpr uint32_t LB_PFULL = LB_TFULL + 16;                 // all shares of this CTA's sums are there; behind it: flags
constexpr int LC_N = 16;          // MMA width without the exchange (the instruction's minimum at 128 rows)
constexpr int LC_TAIL = 1024;     // ... whose slice has rows for the CTA's own units only: the read past its last block
// Rows of the weight slice, bytes of it per block, bytes of the staged sums (cl: CTAs sharing a contraction, or 1).
__host__ __device__ constexpr int lb_rows(int U, int cl) { return (cl * U + 7) / 8 * 8; }
__host__ __device__ constexpr int lb_w_block(int U, int cl) { return lb_rows(U, cl) * 128; }
__host__ __device__ inline LstmPlan lb_plan(int nblk, int B, int U, int cl, int smem_bytes) {
  if (cl == 1)  // the sums may share the ring: written once a step's products are complete, read before the CTA arrives
    return lstm_plan(nblk, lstm_a_block(B), lb_w_block(U, 1), LC_TAIL, (B + 31) / 32 * 32 * (U + 1) * 4, smem_bytes);
  // the other CTAs write here while this one's products may still read the ring: behind the slice
  return lstm_plan((nblk + cl - 1) / cl, lstm_a_block(B), lb_w_block(U, cl), cl * B * U * 4, 0, smem_bytes);
}

struct LstmBwdParams {
  TcMap mapDZ[4];  // per gate: [T*B rows][H columns], boxes of box_rows x 64; the kernel limits them to the n_keep compact columns
  CUtensorMap* tm_slots;  // this launch's descriptor scratch: ARD_TM_LSTM_SLOTS slots per block
  const int32_t* hdr;
  int T, B, I, H;
  float alpha;
  const float* C;        // [T+1][B][H] compact
  const float* G;        // [T][B][4H]
  const float* dH;       // [T][B][H] gradients of every h_t (then D and dc need not be prepared); nullptr: dH_last and D
  const float* dH_last;  // [B][H] full width
  float* D;              // [T][B][I+H]
  float* dc;             // [B][H] compact, in/out
  __nv_bfloat16* DZ;     // [T][B][4 * gs]: gate blocks of width gs, compact inside a block
  int gs;
  __nv_bfloat16* DZ_out; // a second copy for the caller, [T][B][4H] (nullptr: DZ is the caller's)
  unsigned int* bar;     // arrival counter, zero at launch; [1]: CTAs that left
  int* status;
  const __nv_bfloat16* W;  // [4H][ldw]
  int ldw;
  int whole_ok;            // a pattern that keeps few units may do without the exchange
  int smem_bytes;          // dynamic shared memory of this launch
  int above, up_to;        // a pattern that keeps no more than the one, or more than the other, is another kernel's
};

// What the cell adjoint of a (row, unit) pair reads besides the recurrent sum.
struct AdjointIn {
  float gi, gf, gg, go, cp, c, up;
};
__device__ __forceinline__ void fetch_saved(const LstmBwdParams& p, int t, int row, int j, int u, AdjointIn& in) {
  const float* gs = p.G + ((size_t)t * p.B + row) * 4 * p.H + j;
  in.gi = __ldcg(gs);
  in.gf = __ldcg(gs + p.H);
  in.gg = __ldcg(gs + 2 * p.H);
  in.go = __ldcg(gs + 3 * p.H);
  in.cp = __ldcg(p.C + ((size_t)t * p.B + row) * p.H + j);
  in.c = __ldcg(p.C + ((size_t)(t + 1) * p.B + row) * p.H + j);
  // upstream gradient of h_t (u: the unit's index in the layer)
  if (p.dH != nullptr) in.up = __ldcg(p.dH + ((size_t)t * p.B + row) * p.H + u);
  else if (t == p.T - 1) in.up = p.dH_last[(size_t)row * p.H + u];
  else in.up = __ldcg(p.D + ((size_t)(t + 1) * p.B + row) * (p.I + p.H) + p.I + u);
}
// The cell adjoint is linear in the total gradient dh of h_t: with dcv = dc + dh * c, the gradient of c_t, the gates'
// dz are dcv * i, dcv * f, dcv * g and dh * o, and dcv * next is the gradient of c_{t-1}.  These factors are formed
// while the recurrent sums are on their way
// (64 rows, 512 kept units: 4.27 -> 4.21 us per step; 64 kept: 3.29 -> 3.22).
struct Adjoint {
  float c, i, f, g, o, next, up;
};
__device__ __forceinline__ Adjoint adjoint_factors(const AdjointIn& in, float alpha) {
  Adjoint a;
  const float tc = tanhf(in.c);
  a.c = alpha * in.go * (1.f - tc * tc);
  a.i = in.gg * in.gi * (1.f - in.gi);
  a.f = in.cp * in.gf * (1.f - in.gf);
  a.g = in.gi * (1.f - in.gg * in.gg);
  a.o = alpha * tc * in.go * (1.f - in.go);
  a.next = in.gf;
  a.up = in.up;
  return a;
}
__device__ __forceinline__ void cell_adjoint(const Adjoint& a, float dh, float& dc, __nv_bfloat16 (&dz)[4]) {
  const float dcv = dc + dh * a.c;
  dc = dcv * a.next;
  dz[0] = __float2bfloat16_rn(dcv * a.i);
  dz[1] = __float2bfloat16_rn(dcv * a.f);
  dz[2] = __float2bfloat16_rn(dcv * a.g);
  dz[3] = __float2bfloat16_rn(dh * a.o);
}
__device__ __forceinline__ void store_dz(__nv_bfloat16* dst, size_t gs, const __nv_bfloat16 (&dz)[4]) {
#pragma unroll
  for (int g = 0; g < 4; ++g) dst[g * gs] = dz[g];
}

// Barrier ID of the LB_MATH adjoint threads; the same verdict for all of them: did anyone fail?
template <int ID>
__device__ __forceinline__ bool math_barrier_failed(bool failed) {
  uint32_t r;
  __syncwarp();
  asm volatile(
      "{\n\t.reg .pred P, Q;\n\t"
      "setp.ne.b32 Q, %1, 0;\n\t"
      "barrier.cta.red.or.pred.aligned P, %2, %3, Q;\n\t"
      "selp.b32 %0, 1, 0, P;\n\t}"
      : "=r"(r) : "r"((uint32_t)failed), "n"(ID), "n"(LB_MATH) : "memory");
  return r != 0;
}

// The recurrence with U units per CTA.
template <int U>
__device__ __forceinline__ void lstm_backward_body(const LstmBwdParams& p, uint8_t* smem, uint32_t base, uint32_t tmem_base,
                                                   volatile int* abort_flag, int cl, int dp, int bb, int n_keep) {
  constexpr int PAIRS = (128 * U + LB_MATH - 1) / LB_MATH;  // (row, unit) pairs per thread
  constexpr int GRAN = 4;                                   // columns read from tensor memory at a time
  auto full_bar = [&](int g, int s) { return base + 8u * (g * LP_SLOTS + s); };
  auto free_bar = [&](int g, int s) { return base + 8u * ((LP_GROUPS + g) * LP_SLOTS + s); };
  const uint32_t tfull_bar = base + LB_TFULL, hready_bar = base + LB_HREADY, pfull_bar = base + LB_PFULL;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int KH = p.I + p.H, T = p.T;
  const int box_rows = lstm_box_rows(p.B), row_boxes = (p.B + 63) / 64;
  const uint32_t a_block = (uint32_t)lstm_a_block(p.B);
  const int nb = (n_keep + 63) / 64;                  // contraction blocks per gate
  const int nblk_all = 4 * nb;                        // ... per step; block = gate * nb + jb
  int share = cl;                                     // CTAs that share a contraction
  LstmPlan plan = lb_plan(nblk_all, p.B, U, 1, p.smem_bytes);
  if (p.whole_ok && nblk_all <= LB_WHOLE_BLOCKS && plan.cap >= plan.gsz) share = 1;
  if (share > 1) plan = lb_plan(nblk_all, p.B, U, LB_CLUSTER, p.smem_bytes);
  const int gsz = plan.gsz, cap = plan.cap;
  const int per = (nblk_all + share - 1) / share;     // blocks of one share
  const int parts = (nblk_all + per - 1) / per;       // shares that have blocks
  // Without the exchange the first CTA of every cluster takes units before the second of any does: the CTAs of a
  // cluster are neighbours, and neighbours share their way to L2.
  const int cta = share > 1 ? (int)blockIdx.x : (int)(blockIdx.x % cl * (gridDim.x / cl) + blockIdx.x / cl);
  const int rank = cta % share;
  const int blk0 = rank * per, nblk = max(0, min(per, nblk_all - blk0));
  const int j0 = cta * U;                             // first kept unit (compact index) of this CTA
  const int s0 = j0 - rank * U;                       // ... of those whose sums it forms
  const int units = share * U;
  const int n_active = (n_keep + units - 1) / units * share;
  const bool active = cta < n_active;
  const int w_rows = share > 1 ? lb_rows(U, LB_CLUSTER) : lb_rows(U, 1);
  const uint32_t w_block = (uint32_t)w_rows * 128u;
  const uint32_t sA = base + LP_BAR_BYTES;            // the ring
  const uint32_t sW = sA + (uint32_t)(LP_GROUPS * cap) * a_block;  // the weight slice
  const uint32_t sZ = share > 1 ? sW + (uint32_t)per * w_block     // staged sums
                                : (plan.zs_shared ? sA : sW + (uint32_t)plan.behind);
  float* zs = reinterpret_cast<float*>(smem + (sZ - base));

  if (active) {
    // Weight slice, K-major: row r = unit s0 + r, column (gate, i) = W[gate * H + keep[i]][I + keep[s0 + r]], in the
    // 128-byte swizzle (16-byte piece c of row r of an 8-row group sits at piece c ^ r); rows beyond the units and
    // what lies beyond the kept counts are zeros.
    for (int task = threadIdx.x; task < nblk * w_rows * 8; task += LB_THREADS) {
      const int r = task % w_rows, c = task / w_rows & 7, kb = task / (w_rows * 8);
      const int blk = blk0 + kb, g = blk / nb, jb = blk - g * nb;
      uint32_t w[4] = {0u, 0u, 0u, 0u};
      if (r < units && s0 + r < n_keep) {
        const int i0 = jb * 64 + c * 8;
        const unsigned short* src = reinterpret_cast<const unsigned short*>(p.W) +
                                    ((size_t)g * p.H + bb + (size_t)i0 * dp) * p.ldw + p.I + bb + (size_t)(s0 + r) * dp;
        uint32_t e[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) e[q] = (i0 + q < n_keep) ? (uint32_t)__ldg(src + (size_t)q * dp * p.ldw) : 0u;
#pragma unroll
        for (int q = 0; q < 4; ++q) w[q] = e[2 * q] | (e[2 * q + 1] << 16);
      }
      uint8_t* dst = smem + (sW - base) + (size_t)kb * w_block + (r >> 3) * 1024 + (r & 7) * 128 + ((c ^ (r & 7)) << 4);
      *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    fence_proxy_async_smem();  // generic-proxy stores -> the tensor core's reads
  }
  __syncthreads();

  CUtensorMap* slots = p.tm_slots + (size_t)blockIdx.x * ARD_TM_LSTM_SLOTS;
  if (!active) {
  } else if (warp == 11) {
    // ===================== descriptors of the compact gradient columns, barrier relay =====================
#pragma unroll
    for (int g = 0; g < 4; ++g)  // the ring, still empty, is the work area
      tensormap_specialise(&p.mapDZ[g], dp, bb + 1, n_keep, smem + LP_BAR_BYTES + 128 * g, slots + g, lane);
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) {
      for (int ph = 1; ph <= T; ++ph) {
        // dz of time index T - ph is complete when every CTA that takes part has arrived ph times
        if (!grid_wait(p.bar, (unsigned)ph * (unsigned)n_active, abort_flag, p.status)) break;
        mbar_arrive(hready_bar);
      }
    }
  } else if (warp >= 12) {
    // ===================== loaders and MMA issuers (group g4 = warp - 12) =====================
    const int g4 = warp - 12;
    const int kb0 = g4 * gsz, n = max(0, min(nblk - kb0, gsz));
    // where dp == 1 the descriptors are used as encoded (tensormap_specialise returns the parameter)
    auto map_of = [&](int gate) -> const CUtensorMap* { return dp == 1 ? &p.mapDZ[gate].tm : slots + gate; };
    const uint32_t idesc = make_idesc(share > 1 ? LB_CLUSTER * U : LC_N, false, false, lstm_mma_rows(p.B));
    const uint32_t d_tmem = tmem_base + (uint32_t)(g4 * LB_COLS);
    bool ok = true;
    for (int k = 1; k <= T; ++k) {
      if (ok && !mbar_wait(hready_bar, (uint32_t)(k - 1) & 1u, abort_flag, p.status)) ok = false;
      if (!__all_sync(0xffffffffu, ok)) break;
      if (k == 1 && dp > 1) {  // written by warp 11 ahead of its first arrival on hready_bar
#pragma unroll
        for (int g = 0; g < 4; ++g) tensormap_acquire(slots + g);
      }
      asm volatile("fence.proxy.async.global;" ::: "memory");  // generic-proxy stores of other CTAs -> TMA reads
      auto request = [&](int i, int slot) {
        const int kb = blk0 + kb0 + i, gate = kb / nb, jb = kb - gate * nb;
        mbar_arrive_expect_tx(full_bar(g4, slot), a_block);
        for (int rb = 0; rb < row_boxes; ++rb)
          tma_load_2d(sA + (uint32_t)(g4 * cap + slot) * a_block + rb * LP_ROW_BOX, map_of(gate), full_bar(g4, slot), jb * 64,
                      (T - k) * p.B + rb * box_rows);
      };
      auto multiply = [&](int i, int slot, bool first) {
        const uint64_t ad = make_desc(sA + (uint32_t)(g4 * cap + slot) * a_block, 16, 1024), bd = make_desc(sW + (kb0 + i) * w_block, 16, 1024);
#pragma unroll
        for (int s = 0; s < LP_BK / 16; ++s) tc_mma_bf16(d_tmem, ad + 2 * s, bd + 2 * s, idesc, (!first || s != 0) ? 1u : 0u);
      };
      ok = lstm_stream_blocks(n, cap, k - 1, lane, ok, [&](int s) { return full_bar(g4, s); }, [&](int s) { return free_bar(g4, s); },
                              abort_flag, p.status, request, multiply);
      if (lane == 0 && ok) {
        if (n > 0) tc_commit(tfull_bar);
        else mbar_arrive(tfull_bar);
      }
      __syncwarp();
    }
  } else {
    // ===================== recurrent sums and cell adjoint (warps 0-10) =====================
    const int tid = threadIdx.x;
    const int npairs = p.B * U;  // (batch row, owned unit) pairs; pair q = row * U + kk
    const size_t ldd = (size_t)KH;
    const int ngroups = (nblk + gsz - 1) / gsz;  // issuing warps with blocks
    const int qrows = lstm_mma_rows(p.B) / 4;    // batch rows in each 32 lanes of tensor memory
    float dcreg[PAIRS];
    auto row_of = [&](int i) { return (tid + i * LB_MATH) / U; };
    auto unit_of = [&](int i) { return j0 + (tid + i * LB_MATH) % U; };  // kept index
    uint32_t own = 0;  // bit i: pair i exists (not beyond the kept count or the batch)
#pragma unroll
    for (int i = 0; i < PAIRS; ++i) {
      if (tid + i * LB_MATH < npairs && unit_of(i) < n_keep) own |= 1u << i;
      dcreg[i] = (own >> i & 1u) && p.dH == nullptr ? p.dc[(size_t)row_of(i) * p.H + unit_of(i)] : 0.f;
    }
    bool ok = true;
    for (int k = 0; k <= T; ++k) {
      const int t = T - 1 - k;  // time index whose dh is formed in this round (-1: the gradient of h_0)
      // what does not depend on the recurrence is fetched before the waits
      Adjoint adj[PAIRS];
#pragma unroll
      for (int i0 = 0; i0 < PAIRS; i0 += 3) {  // three pairs at a time: what fits the registers
        AdjointIn in[3];
#pragma unroll
        for (int i = i0; i < min(PAIRS, i0 + 3); ++i)
          if ((own >> i & 1u) && t >= 0) fetch_saved(p, t, row_of(i), unit_of(i), bb + unit_of(i) * dp, in[i - i0]);
#pragma unroll
        for (int i = i0; i < min(PAIRS, i0 + 3); ++i)
          if ((own >> i & 1u) && t >= 0) adj[i] = adjoint_factors(in[i - i0], p.alpha);
      }
      if (k >= 1 && share > 1) {
        const uint32_t phase = (uint32_t)(k - 1) & 1u;
        // j0 < n_keep: this CTA has units (the last ones of a cluster may have none: nobody sends to them)
        if (tid == 0 && j0 < n_keep) mbar_arrive_expect_tx(pfull_bar, (uint32_t)(parts * p.B * U * 4));
        if (warp < 8 && (warp & 3) * qrows < p.B && nblk > 0) {
          if (!mbar_wait(tfull_bar, phase, abort_flag, p.status)) ok = false;
          if (__all_sync(0xffffffffu, ok)) {
            tc_fence_after();
            const int row = lane < qrows ? (warp & 3) * qrows + lane : p.B;
            const uint32_t t_row = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
#pragma unroll
            for (int h = 0; h < LB_CLUSTER / 2; ++h) {  // warps 0-3: the units of CTAs 0 and 1, warps 4-7: of CTAs 2 and 3
              const int r = (warp >> 2) * (LB_CLUSTER / 2) + h;
              if (s0 + r * U >= n_keep) break;
              const uint32_t dst = mapa_u32(sZ + (uint32_t)((rank * p.B + row) * U * 4), (uint32_t)r), bar = mapa_u32(pfull_bar, (uint32_t)r);
#pragma unroll
              for (int u0 = 0; u0 < U; u0 += GRAN) {
                float z[GRAN];
                lstm_sum_groups<GRAN>(t_row + (uint32_t)(r * U + u0), LB_COLS, ngroups, z);
                if (row < p.B) {
#pragma unroll
                  for (int i = 0; i < GRAN; i += 4) st_async_f4(dst + 4u * (u0 + i), bar, z[i], z[i + 1], z[i + 2], z[i + 3]);
                }
              }
            }
            tc_fence_before();
          }
        }
        if (ok && j0 < n_keep && !mbar_wait_cluster(pfull_bar, phase, abort_flag, p.status)) ok = false;
      } else if (k >= 1) {
        if (warp < 4) {
          if (!mbar_wait(tfull_bar, (uint32_t)(k - 1) & 1u, abort_flag, p.status)) ok = false;
          if (__all_sync(0xffffffffu, ok)) {
            tc_fence_after();
            if (warp * qrows < p.B) {
              const uint32_t t_row = tmem_base + ((uint32_t)(warp * 32) << 16);
              float* zr = zs + (warp * qrows + lane) * (U + 1);
#pragma unroll
              for (int u0 = 0; u0 < U; u0 += GRAN) {
                float z[GRAN];
                lstm_sum_groups<GRAN>(t_row + (uint32_t)u0, LB_COLS, ngroups, z);
#pragma unroll
                for (int i = 0; i < GRAN; ++i)
                  if (lane < qrows) zr[u0 + i] = z[i];
              }
            }
            tc_fence_before();
          }
        }
        if (math_barrier_failed<2>(!ok)) { ok = false; break; }
      }
      float total[PAIRS];  // gradient of h_t, also handed back to the caller
#pragma unroll
      for (int i = 0; i < PAIRS; ++i) {
        if (!(own >> i & 1u)) continue;
        const int row = row_of(i), j = unit_of(i);
        float rec = 0.f;
        if (k >= 1 && share > 1) {
#pragma unroll
          for (int r = 0; r < LB_CLUSTER; ++r)  // fixed order: same bits every launch
            if (r < parts) rec += zs[r * p.B * U + tid + i * LB_MATH];
        } else if (k >= 1) {
          rec = zs[row * (U + 1) + j - j0];
        }
        if (t < 0) {  // gradient of h_0, added to what the caller left in the h half of D[0]
          float* d0 = p.D + (size_t)row * ldd + p.I;
          if (p.dH == nullptr) {
            d0[bb + j * dp] += rec;
          } else {  // nothing was there: zeros of the dropped units; the j-th kept one owns [j * dp, (j + 1) * dp), the last the tail
            const int last = j == n_keep - 1 ? p.H : min(p.H, (j + 1) * dp);
            for (int u = j * dp; u < last; ++u) d0[u] = u == bb + j * dp ? rec : 0.f;
          }
          continue;
        }
        total[i] = adj[i].up + rec;  // upstream gradient of h_t plus the recurrent part (none at T - 1)
        __nv_bfloat16 dz[4];
        cell_adjoint(adj[i], total[i], dcreg[i], dz);
        store_dz(p.DZ + ((size_t)t * p.B + row) * 4 * p.gs + j, p.gs, dz);
        if (p.DZ_out != nullptr) store_dz(p.DZ_out + ((size_t)t * p.B + row) * 4 * p.H + j, p.H, dz);
      }
      if (t >= 0) {
        // the staged sums may lie in the ring, which the TMA unit overwrites next
        fence_proxy_async_smem();
        if (math_barrier_failed<1>(!ok)) { ok = false; break; }
        if (tid == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p.bar) : "memory");
        if (t < T - 1 && p.dH == nullptr) {  // the caller's D holds the totals afterwards (with dH 10 us of a pass of 381)
#pragma unroll
          for (int i = 0; i < PAIRS; ++i)
            if (own >> i & 1u) p.D[((size_t)(t + 1) * p.B + row_of(i)) * ldd + p.I + bb + unit_of(i) * dp] = total[i];
        }
      }
    }
    if (ok) {
#pragma unroll
      for (int i = 0; i < PAIRS; ++i)
        if (own >> i & 1u) {
          float* dc = p.dc + (size_t)row_of(i) * p.H;
          dc[unit_of(i)] = dcreg[i];
          if (p.dH != nullptr)  // nothing was there: zeros behind the kept columns
            for (int c = unit_of(i) + n_keep; c < p.H; c += n_keep) dc[c] = 0.f;
        }
    }
  }

}

// U: units per CTA at most; the layer fits the grid with U units per CTA when nothing is dropped.
template <int U>
__global__ void __launch_bounds__(LB_THREADS, 1) ard_lstm_backward_kernel(const __grid_constant__ LstmBwdParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t base = (raw_addr + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw_addr);
  uint8_t* misc = smem + LB_PFULL + 8;
  volatile uint32_t* tmem_ptr_smem = reinterpret_cast<volatile uint32_t*>(misc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 4);
  const int warp = threadIdx.x >> 5;
  uint32_t cl;
  asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(cl));
  if (!lstm_take_pattern(p.hdr, p.above, p.up_to)) return;

  if (threadIdx.x < 2 * LP_GROUPS * LP_SLOTS) mbar_init(base + 8u * threadIdx.x, 1);
  if (threadIdx.x == 0) {
    mbar_init(base + LB_TFULL, LP_GROUPS);
    mbar_init(base + LB_HREADY, 1);
    mbar_init(base + LB_PFULL, 1);
    *abort_flag = 0;
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  if (warp == 15) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_ptr_smem)), LP_GROUPS * LB_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_ptr_smem;
  if (cl > 1) cluster_sync_all();  // every CTA's barriers exist before anyone sends
  lstm_next_launch(p.above);

  const int dp = p.hdr[HDR_DP], bb = p.hdr[HDR_B] - 1, n_keep = p.hdr[HDR_NKEEP];
  const int ctas = (int)gridDim.x;
  // as few units per CTA as the grid allows (see the forward kernel; 64 rows, 512 kept: 4.9 us per step with 8, 4.2 with 4)
  if (n_keep <= 4 * ctas) lstm_backward_body<4>(p, smem, base, tmem_base, abort_flag, (int)cl, dp, bb, n_keep);
  else if (U == 8 || n_keep <= 8 * ctas) lstm_backward_body<8>(p, smem, base, tmem_base, abort_flag, (int)cl, dp, bb, n_keep);
  else lstm_backward_body<U>(p, smem, base, tmem_base, abort_flag, (int)cl, dp, bb, n_keep);

  // ---- teardown ----
  tc_fence_before();
  __syncwarp();  // lanes that left their role's loop one by one arrive at the block-wide barrier together
  __syncthreads();
  if (threadIdx.x == 0) grid_leave(p.bar);
  if (warp == 15) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, LP_GROUPS * LB_COLS);
  }
  __syncwarp();
  if (cl > 1) cluster_sync_all();  // nobody leaves while its peers may still send to it
}

}  // namespace

namespace {

constexpr int lstm_units(int H, int sms) { return H <= 8 * sms ? 8 : 12; }

// Dynamic shared memory of a recurrence of `blocks` contraction blocks at most, everything resident if that fits.
int lstm_smem_bytes(int blocks, int B, int w_block, int tail, int zs) {
  const LstmPlan r = lstm_plan(blocks, lstm_a_block(B), w_block, tail, zs, LP_SMEM_MAX);
  return r.cap < 1 ? LP_SMEM_MAX + 1 : 1024 + LP_BAR_BYTES + r.bytes;
}
int lstm_fwd_smem_bytes(int B, int H, int U) {
  const int N = 4 * U;
  return lstm_smem_bytes((H + LP_BK - 1) / LP_BK, B, N * LP_BK * 2, 0, (B + 31) / 32 * 32 * (N + 1) * 4);
}
int lstm_bwd_smem_bytes(int B, int H, int U, int cl) {
  const LstmPlan r = lb_plan(4 * ((H + 63) / 64), B, U, cl, LP_SMEM_MAX);
  return r.cap < 1 ? LP_SMEM_MAX + 1 : 1024 + LP_BAR_BYTES + r.bytes;
}

// A kernel's dynamic shared memory limit raised once per device; false where that fails.
template <typename K>
bool lstm_probe(const ard_ctx* ctx, K kern, int* probed) {
  int& st = probed[ctx->device & 63];
  if (st == 0) st = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, LP_SMEM_MAX) == cudaSuccess ? 1 : -1;
  return st == 1;
}

// ARD_ERR_UNSUPPORTED (nothing enqueued) when the device cannot hold all CTAs at once right now (SMs taken by another
// context, a smaller partition).
template <typename K, typename P>
ard_status lstm_launch(ard_ctx* ctx, K kern, int cluster, int grid, int smem, const P& p, cudaStream_t s) {
  if (ctx->lstm_refuse & 2) return ARD_ERR_UNSUPPORTED;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(LP_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeCooperative;  // all CTAs resident: they wait for one another
  attr[0].val.cooperative = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  const cudaError_t err = cudaLaunchKernelEx(&cfg, kern, p);
  if (err == cudaErrorCooperativeLaunchTooLarge || err == cudaErrorLaunchOutOfResources) {
    (void)cudaGetLastError();
    return ARD_ERR_UNSUPPORTED;
  }
  if (err != cudaSuccess) return ARD_ERR_CUDA;
  ctx->launches++;
  ARD_CUDA_OK(cudaGetLastError());
  return ARD_OK;
}

}  // namespace

int lstm_box_rows_of(int B) { return lstm_box_rows(B); }

// Can the whole-sequence kernel run this layer on this device, whatever pattern is drawn?  (All units on as many CTAs
// as there are SMs, one slot per loading warp beside the densest weight slice, one 128-row tile of batch.)
bool lstm_persistent_fits(ard_ctx* ctx, int B, int H, bool tma) {
  if (B < 1 || B > 128 || H < 1 || ctx->d_lstm_hc == nullptr) return false;
  const int U = lstm_units(H, ctx->sm_count);
  if ((H + U - 1) / U > ctx->sm_count || (H + U - 1) / U > ARD_TM_LSTM_BLOCKS) return false;
  if ((U == 12 || !tma) && !ctx->lstm_compact_h) return false;
  if (H > ARD_LSTM_HC_LD - LP_BK) return false;
  return lstm_fwd_smem_bytes(B, H, U) <= LP_SMEM_MAX;
}

// tma: mapXH and mapW describe the operands (U = 8 only); otherwise they are not read and the compact form runs always.
// 35 steps, batch 20, 1500 -> 1500 units at a period of 2, forward and backward: 3.47 ms step by step with the products of
// gemm_ldg_sm100.cu, 0.45 ms with the whole-sequence kernels.
ard_status launch_lstm_forward_persistent(ard_ctx* ctx, const ard_pattern* pat, int T, int B, int I, int H, int add_zx, float alpha,
                                          const TcMap* mapXH, const TcMap* mapW, const TcMap* mapHc, const void* W, int ldw, void* XH,
                                          const float* bias, float* C, float* G, int above, int up_to, cudaStream_t s) {
  const int U = lstm_units(H, ctx->sm_count);
  LstmFwdParams p = {};
  p.always_compact = mapXH == nullptr || U != 8;
  if (p.always_compact && mapHc == nullptr) return ARD_ERR_UNSUPPORTED;
  p.mapXH = mapXH ? *mapXH : *mapHc;
  for (int g = 0; g < 4; ++g) p.mapW[g] = mapXH ? mapW[g] : *mapHc;
  p.mapHc = mapHc ? *mapHc : *mapXH;
  p.tm_slots = ctx->d_tm_slots + (size_t)ARD_TM_SM_MAX * ARD_TM_SLOTS;
  p.hdr = pat->d_hdr;
  p.T = T; p.B = B; p.I = I; p.H = H;
  p.add_zx = add_zx;
  p.W = reinterpret_cast<const __nv_bfloat16*>(W);
  p.ldw = ldw;
  p.Hc = mapHc ? reinterpret_cast<__nv_bfloat16*>(ctx->d_lstm_hc) : nullptr;
  p.ldhc = ARD_LSTM_HC_LD;
  p.alpha = alpha;
  p.XH = reinterpret_cast<__nv_bfloat16*>(XH);
  p.bias = bias;
  p.C = C;
  p.G = G;
  p.bar = ctx->d_grid_bar + LP_BAR_WORD;
  p.status = ctx->d_status;
  p.smem_bytes = lstm_fwd_smem_bytes(B, H, U);
  p.above = above;
  p.up_to = up_to;
  const int grid = (H + U - 1) / U;  // sized for dp = 1
  static int probed[2][64] = {};
  if (U == 8) {
    if (!lstm_probe(ctx, ard_lstm_forward_kernel<8>, probed[0])) return ARD_ERR_UNSUPPORTED;
    return lstm_launch(ctx, ard_lstm_forward_kernel<8>, 1, grid, p.smem_bytes, p, s);
  }
  if (!lstm_probe(ctx, ard_lstm_forward_kernel<12>, probed[1])) return ARD_ERR_UNSUPPORTED;
  return lstm_launch(ctx, ard_lstm_forward_kernel<12>, 1, grid, p.smem_bytes, p, s);
}

// ---- whole-sequence BPTT recurrence ----
namespace {
struct LstmBwdForm {
  int U, cl;  // units per CTA, cluster size; U == 0: the layer does not fit
  int smem;
};
}  // namespace

// In clusters while all CTAs of a dense draw can be resident that way, 8 units per CTA rather than 12; else without.
static LstmBwdForm lstm_bwd_form(ard_ctx* ctx, int B, int H) {
  static int probed[2][64] = {}, room[2][64] = {};
  const int dev = ctx->device & 63;
  for (int i = 0; i < 4; ++i) {
    const int u = i & 1, U = u ? 12 : 8, cl = i < 2 ? LB_CLUSTER : 1;
    auto kern = u ? ard_lstm_backward_kernel<12> : ard_lstm_backward_kernel<8>;
    if (!lstm_probe(ctx, kern, probed[u])) continue;
    int have = ctx->sm_count;
    if (cl > 1) {
      if (room[u][dev] == 0) room[u][dev] = ard_cluster_room(ctx, kern, cl, LB_THREADS, LP_SMEM_MAX);
      have = room[u][dev];
    }
    const int grid = ((H + U - 1) / U + cl - 1) / cl * cl, smem = lstm_bwd_smem_bytes(B, H, U, cl);
    if (grid <= have && grid <= ARD_TM_LSTM_BLOCKS && smem <= LP_SMEM_MAX) return LstmBwdForm{U, cl, smem};
  }
  return LstmBwdForm{0, 0, 0};
}

bool lstm_persistent_bwd_fits(ard_ctx* ctx, int B, int H) {
  return B >= 1 && B <= 128 && H >= 1 && lstm_bwd_form(ctx, B, H).U != 0;
}

ard_status launch_lstm_backward_persistent(ard_ctx* ctx, const ard_pattern* pat, int T, int B, int I, int H, float alpha,
                                           const TcMap mapDZ[4], const void* W, int ldw, const float* C, const float* G,
                                           const float* dH, const float* dH_last, float* D, float* dc, void* DZ, int gs,
                                           void* DZ_out, int above, int up_to, cudaStream_t s) {
  const LstmBwdForm f = lstm_bwd_form(ctx, B, H);
  if (f.U == 0) return ARD_ERR_UNSUPPORTED;
  LstmBwdParams p = {};
  for (int g = 0; g < 4; ++g) p.mapDZ[g] = mapDZ[g];
  p.tm_slots = ctx->d_tm_slots + (size_t)ARD_TM_SM_MAX * ARD_TM_SLOTS;
  p.hdr = pat->d_hdr;
  p.T = T; p.B = B; p.I = I; p.H = H;
  p.alpha = alpha;
  p.C = C; p.G = G; p.dH = dH; p.dH_last = dH_last; p.D = D; p.dc = dc;
  p.DZ = reinterpret_cast<__nv_bfloat16*>(DZ);
  p.gs = gs;
  p.DZ_out = reinterpret_cast<__nv_bfloat16*>(DZ_out);
  p.bar = ctx->d_grid_bar + LP_BAR_WORD;
  p.status = ctx->d_status;
  p.W = reinterpret_cast<const __nv_bfloat16*>(W);
  p.ldw = ldw;
  p.whole_ok = ctx->lstm_compact_h || f.cl == 1;
  p.smem_bytes = f.smem;
  p.above = above;
  p.up_to = up_to;
  const int grid = ((H + f.U - 1) / f.U + f.cl - 1) / f.cl * f.cl;
  return lstm_launch(ctx, f.U == 8 ? ard_lstm_backward_kernel<8> : ard_lstm_backward_kernel<12>, f.cl, grid, f.smem, p, s);
}
