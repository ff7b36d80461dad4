// Whole-sequence LSTM forward in one cooperative kernel (Sec. 7: the LSTM layer under a row pattern on
// its hidden units; one pattern serves every time step).
//
// The per-step path launches a gate product and a cell kernel per time step, and each launch costs
// more than the 64-row product itself.  Here the recurrence runs inside one kernel:
//   - the input half of the gate pre-activations does not depend on the recurrence: the caller computes
//     x_t . W_x for all steps with one large product beforehand and leaves it where the gate activations
//     of step t will be stored; the kernel adds it in its epilogue and handles the recurrent half only;
//   - every CTA owns U kept hidden units, i.e. 4 U gate columns (i|f|g|o x U), and keeps its slice of
//     the weight, [4 U rows][H] bf16, in shared memory.  U = 8; layers of more than 8 units per SM take U = 12;
//   - per step it loads h_{t-1} (TMA boxes of up to 64 rows x 64 columns) into a ring of slots, one quarter of the
//     blocks per loading warp.  Usually every block of a step has a slot of its own, so all loads of a step are in
//     flight together; a slice so large that fewer slots fit re-uses them within the step.  The warp that loads a
//     quarter also issues its products (tcgen05.mma, M = 128, N = 4 U, accumulators in tensor memory,
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
// The MMA always reads 128 rows, so what lies behind a slot has to exist: 16 KiB from the start of the last slot.  tail:
// bytes that the MMA may read behind the slice.
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
__device__ __forceinline__ void grid_leave(unsigned int* bar) {
  __threadfence();
  if (atomicAdd(bar + 1, 1u) == gridDim.x - 1) {
    bar[0] = 0u;
    bar[1] = 0u;
    __threadfence();
  }
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
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

__device__ __forceinline__ float sigmoid_fast(float x) { return 1.f / (1.f + __expf(-x)); }
__device__ __forceinline__ float tanh_fast(float x) { return 1.f - 2.f / (1.f + __expf(2.f * x)); }

template <int U>
__global__ void __launch_bounds__(LP_THREADS, 1) ard_lstm_forward_kernel(const __grid_constant__ LstmFwdParams p) {
  constexpr int N = 4 * U;                             // gate columns per CTA
  constexpr int W_BLOCK = N * LP_BK * 2;               // one contraction block of the resident weight slice
  constexpr int ZS_LD = N + 1;                         // staged pre-activations: [rows][N + 1] floats
  constexpr int PAIRS = (128 * U + LP_MATH - 1) / LP_MATH;  // (row, unit) pairs per thread
  constexpr uint32_t TMEM_COLS = 2 * LP_GROUPS * N <= 256 ? 256 : 512;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t base = (raw_addr + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw_addr);

  const int KH = p.I + p.H;
  const int box_rows = lstm_box_rows(p.B), row_boxes = (p.B + 63) / 64;
  const uint32_t a_block = (uint32_t)lstm_a_block(p.B);
  auto full_bar = [&](int g, int s) { return base + 8u * (g * LP_SLOTS + s); };
  auto free_bar = [&](int g, int s) { return base + 8u * ((LP_GROUPS + g) * LP_SLOTS + s); };
  const uint32_t bar_base = base + 8u * (2 * LP_GROUPS * LP_SLOTS);
  auto tfull_bar = [&](int a) { return bar_base + 8u * a; };
  auto tempty_bar = [&](int a) { return bar_base + 8u * (2 + a); };
  const uint32_t wfull_bar = bar_base + 8u * 4;
  const uint32_t hready_bar = bar_base + 8u * 5;  // h_{t-1} is complete (relayed from the grid barrier)
  uint8_t* misc = smem + (bar_base - base) + 8 * 6;
  volatile uint32_t* tmem_ptr_smem = reinterpret_cast<volatile uint32_t*>(misc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x < LP_GROUPS * LP_SLOTS) {
    mbar_init(full_bar(0, threadIdx.x), 1);
    mbar_init(free_bar(0, threadIdx.x), 1);
  }
  if (threadIdx.x == 0) {
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull_bar(a), LP_GROUPS);  // one commit per MMA issuer
      mbar_init(tempty_bar(a), 4);         // one arrival per TMEM-reading warp
    }
    mbar_init(wfull_bar, 1);
    mbar_init(hready_bar, 1);
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
  pdl_wait_prior_grids();

  const int dp = p.hdr[HDR_DP], bb = p.hdr[HDR_B] - 1, n_keep = p.hdr[HDR_NKEEP];
  const int n_active = (n_keep + U - 1) / U;       // CTAs that own units (the others only tear down)
  const int j0 = (int)blockIdx.x * U;              // first kept unit (compact index) of this CTA
  const bool active = (int)blockIdx.x < n_active;
  // Under a pattern the dropped units of h_{t-1} are exact zeros (Sec. 3.1), so the recurrent contraction runs over
  // the kept units alone: the operand of a step is the compact copy of h_{t-1} (column j = j-th kept unit) that the
  // cell update writes beside the full-width one, and the weight slice holds the kept fan-in columns only.  Those
  // stride the weight's contiguous dimension, which no TMA box can follow, so the CTA gathers its slice itself,
  // once per sequence, straight into the swizzled layout the MMA reads.
  const bool compact = p.Hc != nullptr && (dp > 1 || p.always_compact);
  const int hs = compact ? 1 : 0;  // the compact h_0 is made by the kernel: one more grid-wide hand-over, before step 0
  const int nkb = ((compact ? n_keep : p.H) + LP_BK - 1) / LP_BK;
  // The staged pre-activations share the start of the ring where they fit: they are written after the step's MMAs
  // have completed and read before this CTA releases h_t, and the next loads are issued only after every CTA has
  // released.  Without them the kernel stays below 196 KB of shared memory at H = 1024; one carve-out step higher
  // (228 KB, next to no L1 left) this kernel was measured 1.5 % slower and the BPTT kernel 4 %.
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
      const uint32_t idesc = make_idesc(N, false, false, 128);
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
        if (warp < 4) {
          // accumulator rows -> shared memory
          if (!mbar_wait(tfull_bar(acc), (uint32_t)(t >> 1) & 1u, abort_flag, p.status)) ok = false;
          if (ok) {
            tc_fence_after();
            if (warp * 32 < p.B) {
              const uint32_t t_row = tmem_base + ((uint32_t)(warp * 32) << 16) + (uint32_t)(acc * LP_GROUPS * N);
              const int ngroups = (nkb + gsz - 1) / gsz;  // accumulators that received MMAs
              float* zr = zs + (warp * 32 + lane) * ZS_LD;
#pragma unroll
              for (int c0 = 0; c0 < N; c0 += 16) {
                uint32_t y[LP_GROUPS][16];
#pragma unroll
                for (int c = 0; c < LP_GROUPS; ++c)
                  if (c < ngroups) tmem_ld16(t_row + (uint32_t)(c * N + c0), y[c]);
                tmem_ld_wait();
                float z[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) z[i] = __uint_as_float(y[0][i]);
#pragma unroll
                for (int c = 1; c < LP_GROUPS; ++c)
                  if (c < ngroups) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) z[i] += __uint_as_float(y[c][i]);
                  }
#pragma unroll
                for (int i = 0; i < 16; ++i) zr[c0 + i] = z[i];
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
            gg[i] = tanh_fast(zg);
            go[i] = sigmoid_fast(zo);
            creg[i] = gf[i] * creg[i] + gi[i] * gg[i];
            const __nv_bfloat16 h = __float2bfloat16_rn(p.alpha * go[i] * tanh_fast(creg[i]));
            p.XH[((size_t)(t + 1) * p.B + row) * ldxh + p.I + u] = h;
            if (compact) p.Hc[((size_t)((t + 1) & 1) * p.B + row) * p.ldhc + j0 + k] = h;
            else if (dp > 1) zeros_of(row, t, j0 + k);  // operands of the next step's product (compact: see below)
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
          }
        }
      }
    }
  }

  if (!active && compact && dp > 1) {
    // The dropped units of h_1 .. h_T, read by nobody before the kernel ends: under a period of dp all but 1 / dp of
    // the grid's CTAs have no units and write the zeros meanwhile (as stores of the cell update they cost 0.3 us a step).
    const int n_idle = (int)gridDim.x - n_active, rows = p.T * p.B;
    for (int r = (int)blockIdx.x - n_active; r < rows; r += n_idle) {
      __nv_bfloat16* hrow = p.XH + ((size_t)p.B + r) * KH + p.I;
      for (int u = threadIdx.x; u < p.H; u += LP_THREADS)
        if (u < bb || (u - bb) % dp != 0) hrow[u] = __float2bfloat16_rn(0.f);
    }
  }

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
// 4 * n_keep kept gate rows, output over the hidden units), then the cell adjoint gives dz_t.  Every SM
// would need all of dz_{t+1} if the output units were simply dealt out, so the product is cut both ways:
// CTA (s, r) owns the 64 hidden-unit COLUMNS 64 s .. 64 s + 63 of the recurrent weight (all of them, kept
// or not: the columns of a kept-unit set are strided and cannot be boxed) and the r-th eighth of the
// contraction blocks; its slice of the weight (at most 8 boxes of 64 gate rows x 64 columns, MN-major B
// operand straight from the neuron-major weight) stays in shared memory for the whole sequence.  A step is
//   A. wait until dz_{t+1} is complete (grid barrier), TMA-load this CTA's blocks of it, multiply
//      (tcgen05.mma M = 128, N = 64, four issuing warps with an accumulator each), park the 64-column
//      partial sums in global memory, arrive;
//   B. wait until all partial sums are there (grid barrier); the threads that own a kept unit among this
//      CTA's 8 columns 64 s + 8 r .. + 7 add the 8 partial sums in a fixed order, add the upstream gradient,
//      store the total (the caller's D holds it afterwards), apply the cell adjoint with dc in a register,
//      store dz_t (bf16, the operand of the next step and of the weight-gradient products), arrive.
// After t = 0 one more product gives the gradient of h_0.  The input half of d[x, h] and the weight
// gradient are large products over all T*B rows that the caller runs afterwards.
// Grid barriers are phases of one arrival counter: every CTA arrives exactly once per phase and only
// after it has passed the previous phase, so the count p * (number of CTAs) identifies phase p.
constexpr int LB_COLS = 64;    // weight columns (hidden units, kept or not) per CTA
constexpr int LB_KPARTS = 8;   // CTAs sharing the contraction of one column slice
constexpr int LB_OWN = LB_COLS / LB_KPARTS;  // columns whose cell adjoint this CTA computes
constexpr int LB_MAX_BLOCKS = 8;             // contraction blocks of one CTA (64 gate rows each)
constexpr int LB_W_BLOCK = 64 * LB_COLS * 2; // one resident weight box
constexpr int LB_THREADS = 512;              // warps 0-10 adjoint (0-3 also read TMEM), 11 relay, 12-15 load + MMA
constexpr int LB_MATH = 352;
constexpr int LB_PAIRS_MAX = (128 * LB_OWN + LB_MATH - 1) / LB_MATH;
// The compact form drops the cut along the contraction: a CTA owns U KEPT units, holds their fan-out weights over all
// 4 * n_keep kept gate rows (gathered by the kernel, K-major) and contracts the whole of dz_{t+1} itself, streamed
// through the same ring of slots as in the forward kernel: one grid-wide barrier per step instead of two, no partial
// sums through global memory.  Its slice needs only the rows of its U units: the instruction's columns beyond them
// are read from whatever follows and never used, so U = 8 takes one KiB per block (U = 12, for layers of more than 8
// units per SM, two).  It reads no operand of the caller through a descriptor but dz, which lives in a padded copy
// in context scratch where the caller's rows are off the 16-byte grid.
// Which form: the compact one while each of a step's blocks has a slot of its own (LB_ROUNDS; batch 64, H = 1024: up
// to 320 kept units), or where the other form cannot run at all.  Every CTA reads all of dz_{t+1} (256 KB of it at a
// period of 2): with slots re-used there the recurrence took 286 us against 264 with partial sums.
constexpr int LC_N = 16;                       // MMA width (the instruction's minimum at 128 rows)
constexpr int LB_ROUNDS = 1;
constexpr int LB_SMEM_BYTES = 195 * 1024;      // one carve-out step higher the form with partial sums was measured 4 - 8 % slower
constexpr int LC_TAIL = 1024;                  // the second 8-row group of the last block's read
__host__ __device__ constexpr int lc_w_block(int U) { return (U + 7) / 8 * 1024; }
__host__ __device__ inline int lc_zs_bytes(int U, int B) { return (B + 31) / 32 * 32 * (U + 1) * 4; }

struct LstmBwdParams {
  TcMap mapDZ[4];  // per gate: [T*B rows][H columns], boxes 64 x 64; the kernel limits them to the n_keep compact columns
  TcMap mapW[4];   // per gate: [H rows][I+H columns], boxes 64 x 64; the kernel turns them into the kept rows
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
  float* partial;        // [CTA][128][64]
  unsigned int* bar;     // arrival counter, zero at launch; [1]: CTAs that left
  int* status;
  const __nv_bfloat16* W;  // the weight itself, [4H][ldw] (the compact form gathers its slice from it)
  int ldw;
  int compact_ok;          // the compact form may be used when the drawn pattern allows it
  int always_compact;      // the operands do not allow the other form
  int smem_bytes;          // dynamic shared memory of this launch
};

// What the cell adjoint of a (row, unit) pair reads besides the recurrent sum.
struct AdjointIn {
  float gi, gf, gg, go, cp, c, up;
};
// Upstream gradient of h_t at (row, u).
__device__ __forceinline__ float upstream(const LstmBwdParams& p, int t, int row, int u) {
  if (p.dH != nullptr) return __ldcg(p.dH + ((size_t)t * p.B + row) * p.H + u);
  return t == p.T - 1 ? p.dH_last[(size_t)row * p.H + u] : __ldcg(p.D + ((size_t)(t + 1) * p.B + row) * (p.I + p.H) + p.I + u);
}
__device__ __forceinline__ void fetch_saved(const LstmBwdParams& p, int t, int row, int j, AdjointIn& in) {
  const float* gs = p.G + ((size_t)t * p.B + row) * 4 * p.H + j;
  in.gi = __ldcg(gs);
  in.gf = __ldcg(gs + p.H);
  in.gg = __ldcg(gs + 2 * p.H);
  in.go = __ldcg(gs + 3 * p.H);
  in.cp = __ldcg(p.C + ((size_t)t * p.B + row) * p.H + j);
  in.c = __ldcg(p.C + ((size_t)(t + 1) * p.B + row) * p.H + j);
}
// Cell adjoint: dz of the four gates from the total gradient dh of h_t; dc is updated to the gradient of c_{t-1}.
__device__ __forceinline__ void cell_adjoint(const LstmBwdParams& p, const AdjointIn& in, float dh, float& dc, __nv_bfloat16 (&dz)[4]) {
  const float tc = tanh_fast(in.c);
  const float d_o = dh * p.alpha * tc;
  const float dcv = dc + dh * p.alpha * in.go * (1.f - tc * tc);
  dc = dcv * in.gf;
  dz[0] = __float2bfloat16_rn(dcv * in.gg * in.gi * (1.f - in.gi));
  dz[1] = __float2bfloat16_rn(dcv * in.cp * in.gf * (1.f - in.gf));
  dz[2] = __float2bfloat16_rn(dcv * in.gi * (1.f - in.gg * in.gg));
  dz[3] = __float2bfloat16_rn(d_o * in.go * (1.f - in.go));
}
__device__ __forceinline__ void store_dz(__nv_bfloat16* dst, size_t gs, const __nv_bfloat16 (&dz)[4]) {
#pragma unroll
  for (int g = 0; g < 4; ++g) dst[g * gs] = dz[g];
}

// The compact form of the BPTT recurrence (see LC_N).
template <int U>
__device__ __forceinline__ void lstm_backward_compact(const LstmBwdParams& p, uint8_t* smem, uint32_t base, uint32_t tfull_bar,
                                                      uint32_t hready_bar, uint32_t tmem_base, volatile int* abort_flag, int dp,
                                                      int bb, int n_keep) {
  constexpr int W_BLOCK = lc_w_block(U), W_ROWS = W_BLOCK / 128;
  constexpr int ZS_LD = U + 1;                               // staged recurrent sums: [rows][U + 1] floats
  constexpr int PAIRS = (128 * U + LB_MATH - 1) / LB_MATH;
  auto full_bar = [&](int g, int s) { return base + 8u * (g * LP_SLOTS + s); };
  auto free_bar = [&](int g, int s) { return base + 8u * ((LP_GROUPS + g) * LP_SLOTS + s); };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int KH = p.I + p.H, T = p.T;
  const int box_rows = lstm_box_rows(p.B), row_boxes = (p.B + 63) / 64;
  const uint32_t a_block = (uint32_t)lstm_a_block(p.B);
  const int nb = (n_keep + 63) / 64;                  // contraction blocks per gate
  const int nblk = 4 * nb;                            // ... per step; block = gate * nb + jb
  const LstmPlan plan = lstm_plan(nblk, (int)a_block, W_BLOCK, LC_TAIL, lc_zs_bytes(U, p.B), p.smem_bytes);
  const int gsz = plan.gsz, cap = plan.cap;
  const int n_active = (n_keep + U - 1) / U;
  const bool active = (int)blockIdx.x < n_active;
  const int j0 = (int)blockIdx.x * U;                 // first kept unit (compact index) of this CTA
  const uint32_t sA = base + LP_BAR_BYTES;            // the ring
  const uint32_t sW = sA + (uint32_t)(LP_GROUPS * cap) * a_block;  // the weight slice
  // the sums share the ring where they fit: written once a step's products are complete, read before the CTA arrives
  float* zs = reinterpret_cast<float*>(smem + (plan.zs_shared ? sA - base : sW - base + (uint32_t)plan.behind));

  if (active) {
    // Weight slice, K-major: row r = unit j0 + r, column (gate, i) = W[gate * H + keep[i]][I + keep[j0 + r]], in the
    // 128-byte swizzle (16-byte piece c of row r of an 8-row group sits at piece c ^ r); rows beyond the CTA's units
    // and what lies beyond the kept counts are zeros.
    for (int task = threadIdx.x; task < nblk * W_ROWS * 8; task += LB_THREADS) {
      const int kb = task / (W_ROWS * 8), c = (task / W_ROWS) & 7, r = task % W_ROWS;
      const int g = kb / nb, jb = kb - g * nb;
      uint32_t w[4] = {0u, 0u, 0u, 0u};
      if (r < U && j0 + r < n_keep) {
        const int i0 = jb * 64 + c * 8;
        const unsigned short* src = reinterpret_cast<const unsigned short*>(p.W) +
                                    ((size_t)g * p.H + bb + (size_t)i0 * dp) * p.ldw + p.I + bb + (size_t)(j0 + r) * dp;
        uint32_t e[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) e[q] = (i0 + q < n_keep) ? (uint32_t)__ldg(src + (size_t)q * dp * p.ldw) : 0u;
#pragma unroll
        for (int q = 0; q < 4; ++q) w[q] = e[2 * q] | (e[2 * q + 1] << 16);
      }
      uint8_t* dst = smem + (sW - base) + (size_t)kb * W_BLOCK + (r >> 3) * 1024 + (r & 7) * 128 + ((c ^ (r & 7)) << 4);
      *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    fence_proxy_async_smem();  // generic-proxy stores -> the tensor core's reads
  }
  __syncthreads();
  if (!active) return;

  CUtensorMap* slots = p.tm_slots + (size_t)blockIdx.x * ARD_TM_LSTM_SLOTS;
  if (warp == 11) {
    // ===================== descriptors of the compact gradient columns, barrier relay =====================
#pragma unroll
    for (int g = 0; g < 4; ++g)  // the ring, still empty, is the work area
      tensormap_specialise(&p.mapDZ[g], dp, bb + 1, n_keep, smem + LP_BAR_BYTES + 128 * g, slots + 4 + g, lane);
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) {
      for (int ph = 1; ph <= T; ++ph) {
        // dz of time index T - ph is complete when every CTA with units has arrived ph times
        if (!grid_wait(p.bar, (unsigned)ph * (unsigned)n_active, abort_flag, p.status)) break;
        mbar_arrive(hready_bar);
      }
    }
  } else if (warp >= 12) {
    // ===================== loaders and MMA issuers (group g4 = warp - 12) =====================
    const int g4 = warp - 12;
    const int kb0 = g4 * gsz, n = max(0, min(nblk - kb0, gsz));
    // where dp == 1 the descriptors are used as encoded (tensormap_specialise returns the parameter)
    auto map_of = [&](int gate) -> const CUtensorMap* { return dp == 1 ? &p.mapDZ[gate].tm : slots + 4 + gate; };
    const uint32_t idesc = make_idesc(LC_N, false, false, 128);
    const uint32_t d_tmem = tmem_base + (uint32_t)(g4 * LB_COLS);
    bool ok = true;
    for (int k = 1; k <= T; ++k) {
      if (ok && !mbar_wait(hready_bar, (uint32_t)(k - 1) & 1u, abort_flag, p.status)) ok = false;
      if (!__all_sync(0xffffffffu, ok)) break;
      if (k == 1 && dp > 1) {  // written by warp 11 ahead of its first arrival on hready_bar
#pragma unroll
        for (int g = 0; g < 4; ++g) tensormap_acquire(slots + 4 + g);
      }
      asm volatile("fence.proxy.async.global;" ::: "memory");  // generic-proxy stores of other CTAs -> TMA reads
      auto request = [&](int i, int slot) {
        const int kb = kb0 + i, gate = kb / nb, jb = kb - gate * nb;
        mbar_arrive_expect_tx(full_bar(g4, slot), a_block);
        for (int rb = 0; rb < row_boxes; ++rb)
          tma_load_2d(sA + (uint32_t)(g4 * cap + slot) * a_block + rb * LP_ROW_BOX, map_of(gate), full_bar(g4, slot), jb * 64,
                      (T - k) * p.B + rb * box_rows);
      };
      auto multiply = [&](int i, int slot, bool first) {
        const uint64_t ad = make_desc(sA + (uint32_t)(g4 * cap + slot) * a_block, 16, 1024), bd = make_desc(sW + (kb0 + i) * W_BLOCK, 16, 1024);
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
    float dcreg[PAIRS];
    int jj[PAIRS];  // kept index of the pair's unit, -1 beyond the kept count or the batch
#pragma unroll
    for (int i = 0; i < PAIRS; ++i) {
      const int q = tid + i * LB_MATH;
      const int row = q / U, j = j0 + q % U;
      jj[i] = (q < npairs && j < n_keep) ? j : -1;
      dcreg[i] = jj[i] >= 0 && p.dH == nullptr ? p.dc[(size_t)row * p.H + j] : 0.f;
    }
    bool ok = true;
    for (int k = 0; k <= T && ok; ++k) {
      const int t = T - 1 - k;  // time index whose dh is formed in this round (-1: the gradient of h_0)
      AdjointIn in[PAIRS];
#pragma unroll
      for (int i = 0; i < PAIRS; ++i) {
        if (jj[i] >= 0 && t >= 0) {
          const int row = (tid + i * LB_MATH) / U;
          fetch_saved(p, t, row, jj[i], in[i]);
          in[i].up = upstream(p, t, row, bb + jj[i] * dp);
        }
      }
      if (k >= 1) {
        if (warp < 4) {
          if (!mbar_wait(tfull_bar, (uint32_t)(k - 1) & 1u, abort_flag, p.status)) ok = false;
          if (ok) {
            tc_fence_after();
            if (warp * 32 < p.B) {
              const uint32_t t_row = tmem_base + ((uint32_t)(warp * 32) << 16);
              const int ngroups = (nblk + gsz - 1) / gsz;
              uint32_t y[LP_GROUPS][16];
#pragma unroll
              for (int c = 0; c < LP_GROUPS; ++c)
                if (c < ngroups) tmem_ld16(t_row + (uint32_t)(c * LB_COLS), y[c]);
              tmem_ld_wait();
              float* zr = zs + (warp * 32 + lane) * ZS_LD;
#pragma unroll
              for (int i = 0; i < U; ++i) {
                float z = __uint_as_float(y[0][i]);
#pragma unroll
                for (int c = 1; c < LP_GROUPS; ++c)
                  if (c < ngroups) z += __uint_as_float(y[c][i]);
                zr[i] = z;
              }
            }
            tc_fence_before();
          }
        }
        asm volatile("bar.sync 2, 352;" ::: "memory");
        if (*abort_flag) { ok = false; break; }
      }
      float total[PAIRS];  // gradient of h_t, also handed back to the caller
#pragma unroll
      for (int i = 0; i < PAIRS; ++i) {
        if (jj[i] < 0) continue;
        const int q = tid + i * LB_MATH;
        const int row = q / U, j = jj[i];
        const float rec = k >= 1 ? zs[row * ZS_LD + q % U] : 0.f;
        if (t < 0) {  // gradient of h_0, added to what the caller left in the h half of D[0]
          float* d0 = p.D + (size_t)row * ldd + p.I + bb + j * dp;
          *d0 = p.dH == nullptr ? *d0 + rec : rec;
          continue;
        }
        total[i] = in[i].up + rec;  // upstream gradient of h_t plus the recurrent part (none at T - 1)
        __nv_bfloat16 dz[4];
        cell_adjoint(p, in[i], total[i], dcreg[i], dz);
        store_dz(p.DZ + ((size_t)t * p.B + row) * 4 * p.gs + j, p.gs, dz);
        if (p.DZ_out != nullptr) store_dz(p.DZ_out + ((size_t)t * p.B + row) * 4 * p.H + j, p.H, dz);
      }
      if (t >= 0) {
        // the staged sums may lie in the ring, which the TMA unit overwrites next
        fence_proxy_async_smem();
        asm volatile("bar.sync 1, 352;" ::: "memory");
        if (tid == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p.bar) : "memory");
        if (t < T - 1) {
#pragma unroll
          for (int i = 0; i < PAIRS; ++i)
            if (jj[i] >= 0) p.D[((size_t)(t + 1) * p.B + (tid + i * LB_MATH) / U) * ldd + p.I + bb + jj[i] * dp] = total[i];
        }
      }
    }
    if (ok) {
#pragma unroll
      for (int i = 0; i < PAIRS; ++i)
        if (jj[i] >= 0) p.dc[(size_t)((tid + i * LB_MATH) / U) * p.H + jj[i]] = dcreg[i];
    }
  }
}

// SUMS: the form with partial sums is available too (U = 8).
template <int U, bool SUMS>
__global__ void __launch_bounds__(LB_THREADS, 1) ard_lstm_backward_kernel(const __grid_constant__ LstmBwdParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t base = (raw_addr + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw_addr);

  const int KH = p.I + p.H;
  const int box_rows = lstm_box_rows(p.B), row_boxes = (p.B + 63) / 64;
  const uint32_t a_block = (uint32_t)lstm_a_block(p.B);
  // slots' full and free barriers of the compact form, then tfull, hready, wfull, pready, gfull[4]; flags
  const uint32_t bar_base = base + 8u * (2 * LP_GROUPS * LP_SLOTS);
  const uint32_t sA = base + LP_BAR_BYTES;                      // LB_MAX_BLOCKS blocks of dz
  const uint32_t sW = sA + LB_MAX_BLOCKS * a_block;             // LB_MAX_BLOCKS weight boxes (the MMA's 128-row read of
                                                                 // the last dz block ends inside this region)
  const uint32_t tfull_bar = bar_base;
  const uint32_t hready_bar = bar_base + 8u;                     // dz of the previous step is complete
  const uint32_t wfull_bar = bar_base + 8u * 2;
  const uint32_t pready_bar = bar_base + 8u * 3;                 // all partial sums of this step are parked
  auto gfull_bar = [&](int g) { return bar_base + 8u * (4 + g); };
  uint8_t* misc = smem + (bar_base - base) + 8 * (LP_GROUPS + 4);
  volatile uint32_t* tmem_ptr_smem = reinterpret_cast<volatile uint32_t*>(misc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x < 2 * LP_GROUPS * LP_SLOTS) mbar_init(base + 8u * threadIdx.x, 1);
  if (threadIdx.x == 0) {
    for (int g = 0; g < LP_GROUPS; ++g) mbar_init(gfull_bar(g), 1);
    mbar_init(tfull_bar, LP_GROUPS);
    mbar_init(wfull_bar, 1);
    mbar_init(hready_bar, 1);
    mbar_init(pready_bar, 1);
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
  pdl_wait_prior_grids();

  const int dp = p.hdr[HDR_DP], bb = p.hdr[HDR_B] - 1, n_keep = p.hdr[HDR_NKEEP];
  // Descriptors of this pattern: slots 0-3 the gates' kept weight rows, 4-7 the gates' compact gradient columns.
  // Warp 11 writes them (below) before its first arrival on hready_bar; the loading lanes acquire them after
  // their first wait on that barrier.
  CUtensorMap* slots = p.tm_slots + (size_t)blockIdx.x * ARD_TM_LSTM_SLOTS;
  auto map_of = [&](const TcMap* m, int slot) -> const CUtensorMap* { return dp == 1 ? &m->tm : slots + slot; };
  const int n_cta = (int)gridDim.x;
  const int s_idx = (int)blockIdx.x / LB_KPARTS, r_idx = (int)blockIdx.x % LB_KPARTS;
  const int c0 = s_idx * LB_COLS;                       // first weight column (hidden unit) of the slice
  const int nb = (n_keep + 63) / 64;                    // contraction blocks per gate
  const int per = (4 * nb + LB_KPARTS - 1) / LB_KPARTS; // blocks per CTA (<= LB_MAX_BLOCKS, checked by the host)
  const int blk0 = r_idx * per;
  const int nblk = max(0, min(per, 4 * nb - blk0));     // this CTA's blocks blk0 .. blk0 + nblk - 1; block = gate * nb + jb
  const int parts = (4 * nb + per - 1) / per;           // CTAs of a slice that have blocks
  const int gsz = (nblk + LP_GROUPS - 1) / LP_GROUPS;   // blocks per loader / MMA warp
  const int T = p.T;

  bool compact = p.always_compact || !SUMS;
  if (!compact && p.compact_ok && dp > 1) {
    const LstmPlan plan = lstm_plan(4 * nb, lstm_a_block(p.B), lc_w_block(U), LC_TAIL, lc_zs_bytes(U, p.B), p.smem_bytes);
    compact = LB_ROUNDS * plan.cap >= plan.gsz;
  }
  if (compact) {
    lstm_backward_compact<U>(p, smem, base, tfull_bar, hready_bar, tmem_base, abort_flag, dp, bb, n_keep);
  } else if (!SUMS) {
  } else if (warp == 11) {
    // ===================== weight loader and barrier relay =====================
    // the weight area, still empty, is the work area of the eight descriptors
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      tensormap_specialise(&p.mapW[g], dp, bb + 1, n_keep, smem + (sW - base) + 128 * g, slots + g, lane);
      tensormap_specialise(&p.mapDZ[g], dp, bb + 1, n_keep, smem + (sW - base) + 128 * (4 + g), slots + 4 + g, lane);
    }
    fence_proxy_async_smem();
    const int kb = lane;
    if (kb < nblk) {
      const int blk = blk0 + kb, g = blk / nb, jb = blk - g * nb;
      const CUtensorMap* mw = map_of(&p.mapW[g], g);
      if (dp > 1) tensormap_acquire(mw);
      if (lane == 0) mbar_arrive_expect_tx(wfull_bar, (uint32_t)nblk * LB_W_BLOCK);
      __syncwarp(__activemask());
      tma_load_2d(sW + kb * LB_W_BLOCK, mw, wfull_bar, p.I + c0, jb * 64);
    }
    __syncwarp();
    if (lane == 0) {
      for (int ph = 1; ph <= 2 * T; ++ph) {
        if (!grid_wait(p.bar, (unsigned)ph * (unsigned)n_cta, abort_flag, p.status)) break;
        mbar_arrive((ph & 1) ? hready_bar : pready_bar);
      }
    }
  } else if (warp >= 12) {
    // ===================== loaders and MMA issuers (group g = warp - 12) =====================
    const int g4 = warp - 12;
    const int kb0 = g4 * gsz, kb1 = min(nblk, kb0 + gsz);
    const int kb = kb0 + lane;
    const bool mine = kb < kb1;
    int gate = 0, jb = 0;
    if (mine) {
      const int blk = blk0 + kb;
      gate = blk / nb;
      jb = blk - gate * nb;
    }
    const CUtensorMap* mdz = map_of(&p.mapDZ[gate], 4 + gate);
    const uint32_t idesc = make_idesc(LB_COLS, false, true, 128);
    bool ok = (lane != 0) || nblk == 0 || mbar_wait(wfull_bar, 0u, abort_flag, p.status);
    for (int k = 1; k <= T; ++k) {
      // dz of time index T - k is complete
      if (ok && !mbar_wait(hready_bar, (uint32_t)(k - 1) & 1u, abort_flag, p.status)) ok = false;
      if (!__all_sync(0xffffffffu, ok)) break;
      if (k == 1 && mine && dp > 1) tensormap_acquire(mdz);  // written by warp 11 ahead of its first arrival on hready_bar
      if (kb0 < kb1) {
        asm volatile("fence.proxy.async.global;" ::: "memory");  // generic-proxy stores of other CTAs -> TMA reads
        if (lane == 0) mbar_arrive_expect_tx(gfull_bar(g4), (uint32_t)(kb1 - kb0) * a_block);
        __syncwarp();
        if (mine)
          for (int rb = 0; rb < row_boxes; ++rb)
            tma_load_2d(sA + kb * a_block + rb * LP_ROW_BOX, mdz, gfull_bar(g4), jb * 64,
                        (T - k) * p.B + rb * box_rows);
        if (lane == 0) {
          if (!mbar_wait(gfull_bar(g4), (uint32_t)(k - 1) & 1u, abort_flag, p.status)) ok = false;
          if (ok) {
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + (uint32_t)(g4 * LB_COLS);
            for (int k2 = kb0; k2 < kb1; ++k2) {
              const uint32_t a0 = sA + k2 * a_block, b0 = sW + k2 * LB_W_BLOCK;
#pragma unroll
              for (int s = 0; s < LP_BK / 16; ++s)  // A K-major: 32 bytes per step; B MN-major: 16 k-rows = 2048 bytes
                tc_mma_bf16(d_tmem, make_desc(a0 + s * 32, 16, 1024), make_desc(b0 + s * 2048, 64 * LP_BK * 2, 1024), idesc,
                            (k2 != kb0 || s != 0) ? 1u : 0u);
            }
          }
        }
      }
      if (lane == 0 && ok && nblk > 0) {
        if (kb0 < kb1) tc_commit(tfull_bar);
        else mbar_arrive(tfull_bar);
      }
      __syncwarp();
    }
  } else {
    // ===================== partial sums and cell adjoint (warps 0-10) =====================
    const int tid = threadIdx.x;  // 0 .. LB_MATH-1
    const int npairs = p.B * LB_OWN;  // (batch row, owned column) pairs; pair q = row * 8 + cc
    const size_t ldd = (size_t)KH;
    float dcreg[LB_PAIRS_MAX];
    int jj[LB_PAIRS_MAX];  // kept index of the pair's unit, -1 if the column is a dropped unit or out of range
#pragma unroll
    for (int i = 0; i < LB_PAIRS_MAX; ++i) {
      const int q = tid + i * LB_MATH;
      const int row = q >> 3, u = c0 + r_idx * LB_OWN + (q & 7);
      const int rel = u - bb;
      jj[i] = (q < npairs && u < p.H && rel >= 0 && rel % dp == 0) ? rel / dp : -1;
      dcreg[i] = jj[i] >= 0 && p.dH == nullptr ? p.dc[(size_t)row * p.H + jj[i]] : 0.f;
    }
    float* my_partial = p.partial + (size_t)blockIdx.x * 128 * LB_COLS;
    const float* slice_partial = p.partial + (size_t)(s_idx * LB_KPARTS) * 128 * LB_COLS;
    bool ok = true;
    for (int k = 0; k <= T && ok; ++k) {
      const int t = T - 1 - k;  // time index whose dh is formed in this round (-1: the gradient of h_0)
      // what does not depend on the recurrence is fetched before the waits: gate activations, cell states
      AdjointIn in[LB_PAIRS_MAX];
#pragma unroll
      for (int i = 0; i < LB_PAIRS_MAX; ++i)
        if (jj[i] >= 0 && t >= 0) fetch_saved(p, t, (tid + i * LB_MATH) >> 3, jj[i], in[i]);
      if (k >= 1) {
        // ---- phase A: park this CTA's partial sums ----
        // Every CTA passes the previous phase before it arrives for this one, also a CTA that has no
        // contraction blocks: the arrival count identifies a phase only if nobody is two arrivals ahead.
        if (!mbar_wait(hready_bar, (uint32_t)(k - 1) & 1u, abort_flag, p.status)) ok = false;
        if (ok && warp < 4 && nblk > 0) {
          if (!mbar_wait(tfull_bar, (uint32_t)(k - 1) & 1u, abort_flag, p.status)) ok = false;
          if (ok) {
            tc_fence_after();
            const int row = warp * 32 + lane;
            const uint32_t t_row = tmem_base + ((uint32_t)(warp * 32) << 16);
            const int ngroups = (nblk + gsz - 1) / gsz;
#pragma unroll 1
            for (int half = 0; half < 2; ++half) {
              uint32_t z[32], y[32];
              tmem_ld32(t_row + (uint32_t)(half * 32), z);
              tmem_ld_wait();
              for (int c = 1; c < ngroups; ++c) {
                tmem_ld32(t_row + (uint32_t)(c * LB_COLS + half * 32), y);
                tmem_ld_wait();
#pragma unroll
                for (int i = 0; i < 32; ++i) z[i] = __float_as_uint(__uint_as_float(z[i]) + __uint_as_float(y[i]));
              }
              if (row < p.B) {
                float4* dst = reinterpret_cast<float4*>(my_partial + (size_t)row * LB_COLS + half * 32);
#pragma unroll
                for (int i = 0; i < 8; ++i)
                  __stcg(dst + i, make_float4(__uint_as_float(z[4 * i]), __uint_as_float(z[4 * i + 1]),
                                              __uint_as_float(z[4 * i + 2]), __uint_as_float(z[4 * i + 3])));
              }
            }
            tc_fence_before();
          }
        }
        asm volatile("bar.sync 1, 352;" ::: "memory");
        if (*abort_flag) { ok = false; break; }
        if (tid == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p.bar) : "memory");
        // ---- all partial sums of the slice are parked ----
        if (!mbar_wait(pready_bar, (uint32_t)(k - 1) & 1u, abort_flag, p.status)) ok = false;
        asm volatile("bar.sync 2, 352;" ::: "memory");
        if (*abort_flag) { ok = false; break; }
      }
      // ---- phase B: total gradient of h_t, cell adjoint, dz_t ----
      // All loads of all owned (row, unit) pairs are issued before the first is consumed: the partial sums
      // come from L2 and a chain of dependent round trips would cost more than the whole product.
      float total[LB_PAIRS_MAX];  // recurrent part, then the gradient of h_t, also handed back to the caller
#pragma unroll
      for (int i = 0; i < LB_PAIRS_MAX; ++i) {
        total[i] = 0.f;
        if (jj[i] < 0) continue;
        const int q = tid + i * LB_MATH;
        const int row = q >> 3, cc = r_idx * LB_OWN + (q & 7), u = c0 + cc;
        float part[LB_KPARTS];
#pragma unroll
        for (int rp = 0; rp < LB_KPARTS; ++rp)
          part[rp] = (k >= 1 && rp < parts) ? __ldcg(slice_partial + ((size_t)rp * 128 + row) * LB_COLS + cc) : 0.f;
        in[i].up = t >= 0 ? upstream(p, t, row, u) : 0.f;
        float rec = 0.f;
#pragma unroll
        for (int rp = 0; rp < LB_KPARTS; ++rp) rec += part[rp];  // fixed order: same bits every launch
        total[i] = rec;
      }
#pragma unroll
      for (int i = 0; i < LB_PAIRS_MAX; ++i) {
        if (jj[i] < 0) continue;
        const int q = tid + i * LB_MATH;
        const int row = q >> 3, u = c0 + r_idx * LB_OWN + (q & 7), j = jj[i];
        if (t < 0) {  // gradient of h_0, added to what the caller left in the h half of D[0]
          float* d0 = p.D + (size_t)row * ldd + p.I + u;
          *d0 = p.dH == nullptr ? *d0 + total[i] : total[i];
          continue;
        }
        total[i] += in[i].up;  // upstream gradient of h_t plus the recurrent part (none at T - 1)
        __nv_bfloat16 dz[4];
        cell_adjoint(p, in[i], total[i], dcreg[i], dz);
        store_dz(p.DZ + ((size_t)t * p.B + row) * 4 * p.gs + j, p.gs, dz);
        if (p.DZ_out != nullptr) store_dz(p.DZ_out + ((size_t)t * p.B + row) * 4 * p.H + j, p.H, dz);
      }
      if (t >= 0) {
        asm volatile("bar.sync 1, 352;" ::: "memory");
        if (tid == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p.bar) : "memory");
        if (t < T - 1) {
#pragma unroll
          for (int i = 0; i < LB_PAIRS_MAX; ++i)
            if (jj[i] >= 0)
              p.D[((size_t)(t + 1) * p.B + ((tid + i * LB_MATH) >> 3)) * ldd + p.I + c0 + r_idx * LB_OWN + ((tid + i * LB_MATH) & 7)] = total[i];
        }
      }
    }
    if (ok) {
#pragma unroll
      for (int i = 0; i < LB_PAIRS_MAX; ++i)
        if (jj[i] >= 0) p.dc[(size_t)((tid + i * LB_MATH) >> 3) * p.H + jj[i]] = dcreg[i];
    }
  }

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
int lstm_bwd_compact_smem_bytes(int B, int n, int U) {
  return lstm_smem_bytes(4 * ((n + 63) / 64), B, lc_w_block(U), LC_TAIL, lc_zs_bytes(U, B));
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
ard_status lstm_launch(ard_ctx* ctx, K kern, int grid, int smem, const P& p, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(LP_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // all CTAs resident: they wait for one another
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
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
// gemm_ldg_sm100.cu.
ard_status launch_lstm_forward_persistent(ard_ctx* ctx, const ard_pattern* pat, int T, int B, int I, int H, int add_zx, float alpha,
                                          const TcMap* mapXH, const TcMap* mapW, const TcMap* mapHc, const void* W, int ldw, void* XH,
                                          const float* bias, float* C, float* G, cudaStream_t s) {
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
  // Sized for dp = 1.  Under a period of 2 or more at least one CTA has no units: it writes the zeros of dropped ones.
  const int grid = H > U ? (H + U - 1) / U : 2;
  static int probed[2][64] = {};
  if (U == 8) {
    if (!lstm_probe(ctx, ard_lstm_forward_kernel<8>, probed[0])) return ARD_ERR_UNSUPPORTED;
    return lstm_launch(ctx, ard_lstm_forward_kernel<8>, grid, p.smem_bytes, p, s);
  }
  if (!lstm_probe(ctx, ard_lstm_forward_kernel<12>, probed[1])) return ARD_ERR_UNSUPPORTED;
  return lstm_launch(ctx, ard_lstm_forward_kernel<12>, grid, p.smem_bytes, p, s);
}

// ---- whole-sequence BPTT recurrence ----
// Shared memory of the kernel with both forms.  The form is chosen on the device from the drawn pattern, so the launch
// asks for what either may need: 8 row blocks and 8 weight boxes behind the barriers for the form with partial sums,
// and below LB_SMEM_BYTES what the compact form can use.
static int lstm_bwd_sums_smem_bytes(int B) {
  static_assert((size_t)LB_MAX_BLOCKS * 2 * LP_ROW_BOX + (size_t)LB_MAX_BLOCKS * LB_W_BLOCK + LP_BAR_BYTES + 1024 <= LP_SMEM_MAX,
                "the form with partial sums does not fit");
  return LB_MAX_BLOCKS * lstm_a_block(B) + LB_MAX_BLOCKS * LB_W_BLOCK + LP_BAR_BYTES + 1024;
}

size_t lstm_bwd_partial_bytes(int sm_count) { return (size_t)sm_count * 128 * LB_COLS * sizeof(float); }

// The form with partial sums needs descriptors of the weight (tma) and at most 8 contraction blocks per CTA.
static bool lstm_bwd_sums_fits(const ard_ctx* ctx, int H, bool tma) {
  return tma && H <= 1024 && ctx->d_lstm_partial != nullptr && (H + LB_COLS - 1) / LB_COLS * LB_KPARTS <= ctx->sm_count;
}

bool lstm_persistent_bwd_fits(ard_ctx* ctx, int B, int H, bool tma) {
  if (B < 1 || B > 128 || H < 1) return false;
  if (lstm_bwd_sums_fits(ctx, H, tma)) return true;
  const int U = lstm_units(H, ctx->sm_count);
  if ((H + U - 1) / U > ctx->sm_count || (H + U - 1) / U > ARD_TM_LSTM_BLOCKS || !ctx->lstm_compact_h) return false;
  return lstm_bwd_compact_smem_bytes(B, H, U) <= LP_SMEM_MAX;
}

ard_status launch_lstm_backward_persistent(ard_ctx* ctx, const ard_pattern* pat, int T, int B, int I, int H, float alpha,
                                           const TcMap mapDZ[4], const TcMap* mapW, const void* W, int ldw, const float* C,
                                           const float* G, const float* dH, const float* dH_last, float* D, float* dc, void* DZ, int gs,
                                           void* DZ_out, cudaStream_t s) {
  LstmBwdParams p = {};
  const bool sums = lstm_bwd_sums_fits(ctx, H, mapW != nullptr);
  const int U = sums ? 8 : lstm_units(H, ctx->sm_count);
  for (int g = 0; g < 4; ++g) { p.mapDZ[g] = mapDZ[g]; p.mapW[g] = mapW ? mapW[g] : mapDZ[g]; }
  p.tm_slots = ctx->d_tm_slots + (size_t)ARD_TM_SM_MAX * ARD_TM_SLOTS;
  p.hdr = pat->d_hdr;
  p.T = T; p.B = B; p.I = I; p.H = H;
  p.alpha = alpha;
  p.C = C; p.G = G; p.dH = dH; p.dH_last = dH_last; p.D = D; p.dc = dc;
  p.DZ = reinterpret_cast<__nv_bfloat16*>(DZ);
  p.gs = gs;
  p.DZ_out = reinterpret_cast<__nv_bfloat16*>(DZ_out);
  p.partial = ctx->d_lstm_partial;
  p.bar = ctx->d_grid_bar + LP_BAR_WORD;
  p.status = ctx->d_status;
  p.W = reinterpret_cast<const __nv_bfloat16*>(W);
  p.ldw = ldw;
  p.compact_ok = ctx->lstm_compact_h;
  p.always_compact = !sums;
  static int probed[3][64] = {};
  if (sums) {
    p.smem_bytes = lstm_bwd_sums_smem_bytes(B);
    // the compact form of as many kept units as fit below the carve-out step (see LB_SMEM_BYTES)
    for (int nb = 1; p.compact_ok && pat->dp_bound > 1 && nb <= (H / 2 + 63) / 64; ++nb) {
      const int c = lstm_bwd_compact_smem_bytes(B, 64 * nb, 8);
      if (c > LB_SMEM_BYTES) break;
      if (c > p.smem_bytes) p.smem_bytes = c;
    }
    if (!lstm_probe(ctx, ard_lstm_backward_kernel<8, true>, probed[0])) return ARD_ERR_UNSUPPORTED;
    return lstm_launch(ctx, ard_lstm_backward_kernel<8, true>, (H + LB_COLS - 1) / LB_COLS * LB_KPARTS, p.smem_bytes, p, s);
  }
  p.smem_bytes = lstm_bwd_compact_smem_bytes(B, H, U);
  if (U == 8) {
    if (!lstm_probe(ctx, ard_lstm_backward_kernel<8, false>, probed[1])) return ARD_ERR_UNSUPPORTED;
    return lstm_launch(ctx, ard_lstm_backward_kernel<8, false>, (H + U - 1) / U, p.smem_bytes, p, s);
  }
  if (!lstm_probe(ctx, ard_lstm_backward_kernel<12, false>, probed[2])) return ARD_ERR_UNSUPPORTED;
  return lstm_launch(ctx, ard_lstm_backward_kernel<12, false>, (H + U - 1) / U, p.smem_bytes, p, s);
}
