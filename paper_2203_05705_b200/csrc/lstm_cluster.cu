// Whole-sequence LSTM recurrences whose hand-over between time steps stays inside a cluster of CTAs (Sec. 7).
//
// The batch rows of a layer are independent sequences.  Here a cluster of CTAs owns a few of them from the first step to the
// last: its CTAs hold the kept recurrent weights of the layer between them, and what a step hands to the next goes from SM to
// SM with st.async, whose bytes complete the receiver's mbarrier.  There is no grid-wide barrier, no trip through L2 and no
// descriptor in a step.  lstm_persistent.cu spreads the weights over the whole grid instead, so all SMs meet in L2 in every
// step (about 2.8 us of its 4); it remains for the layers whose kept weights do not fit a cluster.
//
// Bound: latency, a chain of T steps.  A step's products have 8 columns for every group of 8 batch rows that the cluster has, one to three
// groups.  Taken with one group: the narrowest tcgen05.mma has 128 rows and costs its issuing thread 136 cycles, with
// a commit, a wait and a load from tensor memory behind the last one; mma.sync leaves the sums in the registers of the threads
// that apply the cell update, at 8.1 cycles per 16 x 8 x 16 and SM quarter.  (With two and three groups, where mma.sync takes two and three
// times as long, they were not compared.)  The weights stay on the SM for the
// whole sequence, in TENSOR MEMORY used as a store: 12 warps with 48 operands each took 9.3 cycles per product with 8 operands in
// registers and 40 streamed from tensor memory by tcgen05.ld, 17.4 with the 40 in shared memory, which gives 128 bytes a cycle to
// the whole SM.  The exchange among 16 CTAs takes 400 cycles for one packet of 32 bytes each, and 1.7 cycles more for every packet
// that an SM sends or receives (bulk copies of the same bytes 1280 and more).
//
// us, forward and BPTT recurrence of a sequence of 35 steps, all SMs meeting in L2 / here, BPTT with the zeros of the weight gradient: 64 rows,
// 512 of 1024 units kept 138 and 157 / 98 and 81; 20 rows, 750 of 1500 kept 151 and 180 / 82 and 81; 64 rows, 64 of 1024 114 and 122 / 44 and 48;
// the whole pass of the first two, what lies before and behind the recurrences included, 384 / 254 and 437 / 247.  Of that the launch, the
// weights' way in, cold code and the zeros take 13 and 22, 18 and 27, 14 and 18, a step 2.4 and 1.7, 1.8 and 1.5, 0.85 and 0.86 (sequences of 35
// steps less those of 5).  Cycles of a forward step of 64 rows, 512 kept (two groups): products 1220, their sums through shared memory 300, cells
// 1080, shuffles and sends 600, stores and the next gates' loads 575, the wait for the other CTAs 250; of 20 rows, 750 kept (one group) 1290,
// 160, 680, 380, 700 and 220.
//
// Registers: 168 a thread in the forward kernels, of which all spill some.  With one and two groups the spills lie in front of the steps (as many
// local loads and stores with 4 steps as with 24, in clusters of 16); with three, the form of more than 16 rows a cluster, a warp makes 9 loads and 4 stores a step.
// Of the backward kernels only the one of 16 CTAs with three groups spills.
//
// Virtual units.  The kept units are numbered v = j + pad, j = 0 .. n_keep-1, with pad < 4 chosen so that at periods of 1 and
// 2 four consecutive units begin on an 8 or 16 byte boundary of the weight's rows, and are gathered with one load.
//
// Clusters: 16 CTAs, or 8 where the layer is known to keep few units (cluster_form).  A wait that expires
// sets the status word; both kernels end by a cluster barrier, behind which nobody sends.
#include <atomic>

#include "ard_internal.h"
#include "sm100_ptx.h"

namespace {

// W: warps of a CTA, 12, or 16 in one form of the backward kernel; each finishes the cells of 4 units.
__host__ __device__ constexpr int lc_units(int W) { return 4 * W; }  // units per CTA at most
constexpr int LC_REG = 8;                                     // 16 x 16 weight operands of a warp in registers; more in tensor memory,
__host__ __device__ constexpr int lc_tmem_warp(int W) { return W == 12 ? 160 : 128; }  // ... 4 columns each: W / 4 warps share the 512 of a quarter of its lanes
constexpr int LC_KQ = 12;             // forward: contraction steps (16 units) of a warp at most
constexpr int LC_HB = 4 * LC_KQ * 256;  // one copy of h for 8 batch rows, as the products read it
constexpr int LC_BARS = 128;          // barriers and flags at the start of shared memory
constexpr int LC_RING = 8;            // chunks of weight rows on their way at most
constexpr int LC_SWAP = 512;          // a warp's sums of 32 cells
constexpr int LC_SMEM_MAX = 227 * 1024;

struct LstmClusterParams {
  const int32_t* hdr;
  int T, B, I, H;
  int rows;    // batch rows per cluster
  int limit;   // kept units this launch takes; a pattern that keeps more leaves everything to another kernel
  int alone;   // ... which has not been enqueued: an error
  float alpha;
  const __nv_bfloat16* W;  // [4H][ldw]
  int ldw;
  int* status;
  float* C;    // [T+1][B][H] compact
  float* G;    // [T][B][4H]: gate blocks of width H, compact inside a block
  // forward
  int add_zx;  // the products of the other columns are waiting in G[t] (same layout as the gates)
  __nv_bfloat16* XH;
  const float* bias;     // [4][H] or nullptr
  // backward
  const float* dH;       // [T][B][H] gradients of every h_t (then D and dc need not be prepared); nullptr: dH_last and D
  const float* dH_last;  // [B][H] full width
  float* D;              // [T][B][I+H]
  float* dc;             // [B][H] compact, in/out
  __nv_bfloat16* DZ;     // [T][B][4 * gs]: gate blocks of width gs, compact inside a block
  int gs;
  __nv_bfloat16* DZ_out; // a second copy for the caller, [T][B][4H] (nullptr: DZ is the caller's)
  float* dW;             // weight gradient [4H][ld_dw]: the rows of dropped units become zero (the kernels that have it)
  int ld_dw, dw_cols;    // multiples of 4, as dW of 16 bytes
};

__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t* a, const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
__device__ __forceinline__ void lds64(uint32_t addr, uint32_t (&a)[2]) {
  asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(a[0]), "=r"(a[1]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void lds128(uint32_t addr, uint32_t (&a)[4]) {
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void sts128(uint32_t addr, const uint32_t (&a)[4]) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]) : "memory");
}
// Four operands of this warp, 16 columns of its lanes of tensor memory (a store takes its pipe 100 cycles and more whatever its width).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};"
      ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
        "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st4(uint32_t taddr, const uint32_t (&r)[4]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%4], {%0, %1, %2, %3};" ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// Loads and stores of one thread's cell: no branches, and they stay where they are written.
__device__ __forceinline__ float ld_if(bool yes, const void* at) {
  float v;
  asm volatile(
      "{\n\t.reg .pred P;\n\tsetp.ne.b32 P, %2, 0;\n\tmov.f32 %0, 0f00000000;\n\t@P ld.global.cg.f32 %0, [%1];\n\t}"
      : "=f"(v) : "l"(at), "r"((uint32_t)yes) : "memory");
  return v;
}
__device__ __forceinline__ void st_if(bool yes, void* at, float v) {
  asm volatile("{\n\t.reg .pred P;\n\tsetp.ne.b32 P, %2, 0;\n\t@P st.global.f32 [%0], %1;\n\t}" ::"l"(at), "f"(v), "r"((uint32_t)yes) : "memory");
}
__device__ __forceinline__ void st16_if(bool yes, void* at, uint32_t v) {
  asm volatile("{\n\t.reg .pred P;\n\tsetp.ne.b32 P, %2, 0;\n\t@P st.global.b16 [%0], %1;\n\t}" ::"l"(at), "h"((unsigned short)v), "r"((uint32_t)yes) : "memory");
}
// to = v where `yes`: an element of an array in registers chosen at run time (as an assignment the array went to local memory).
__device__ __forceinline__ void set_if(bool yes, uint32_t& to, uint32_t v) {
  asm("{\n\t.reg .pred P;\n\tsetp.ne.b32 P, %2, 0;\n\tselp.b32 %0, %1, %0, P;\n\t}" : "+r"(to) : "r"(v), "r"((uint32_t)yes));
}
// 8 bytes into another CTA's shared memory, counted on that CTA's barrier, where `yes`.
__device__ __forceinline__ void st_async_8(bool yes, uint32_t addr, uint32_t bar, uint32_t a, uint32_t b) {
  asm volatile(
      "{\n\t.reg .pred P;\n\t"
      "setp.ne.b32 P, %4, 0;\n\t"
      "@P st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%2, %3}, [%1];\n\t}"
      ::"r"(addr), "r"(bar), "r"(a), "r"(b), "r"((uint32_t)yes) : "memory");
}
// Barrier ID of `threads` threads; the same verdict for all of them: did anyone fail?
__device__ __forceinline__ bool barrier_failed(int id, int threads, bool failed) {
  uint32_t r;
  __syncwarp();
  asm volatile(
      "{\n\t.reg .pred P, Q;\n\t"
      "setp.ne.b32 Q, %1, 0;\n\t"
      "barrier.cta.red.or.pred.aligned P, %2, %3, Q;\n\t"
      "selp.b32 %0, 1, 0, P;\n\t}"
      : "=r"(r) : "r"((uint32_t)failed), "r"(id), "r"(threads) : "memory");
  return r != 0;
}

// A kernel enqueued beside the one that takes the patterns of more units: is the drawn one among them?  The same for all CTAs, and asked before
// anything is set up, because a launch that does nothing stands in front of the next one's work.  (These are kernels of their own: the question
// alone cost the others, which take their pattern, 0.2 - 0.7 % of the pass.)
__device__ __forceinline__ bool other_kernels_pattern(const LstmClusterParams& p) {
  pdl_wait_prior_grids();
  return p.hdr[HDR_NKEEP] > p.limit;
}

// Operand of 8 batch rows, 256 bytes for 16 contraction indices: thread (n = lane / 4, c = lane % 4) of a product reads the 8 bytes
// of the four indices 4 c .. 4 c + 3 of row n.  The 64 bytes of a c lie together (one sender writes them: 32-byte packets), and
// c = 2, 3 have their halves swapped so that 16 lanes' reads cover every bank once.
__device__ __forceinline__ uint32_t operand_offset(int c, int n) { return (uint32_t)(c * 64 + ((n * 8) ^ ((c >> 1) * 32))); }

// The kept units' place in the weight.
struct KeptWeights {
  const unsigned short* w0;  // element of virtual unit v in row r: w0[r * ldw + v * dp + sel]
  size_t ldw;
  int dp, bb, pad, sel, nv, H;
  int path;  // 1, 2: period 1, 2 with aligned groups of four; 0: element by element
};
__device__ __forceinline__ KeptWeights kept_weights(const LstmClusterParams& p, int dp, int bb, int n_keep) {
  KeptWeights k;
  k.ldw = (size_t)p.ldw;
  k.dp = dp;
  k.bb = bb;
  k.H = p.H;
  k.w0 = reinterpret_cast<const unsigned short*>(p.W) + p.I + bb;
  k.pad = k.sel = k.path = 0;
  const int m = (int)((reinterpret_cast<unsigned long long>(p.W) >> 1) + (unsigned)p.I) & 7;  // elements behind a 16-byte boundary
  const int first = dp == 1 ? m : (m + bb) >> 1, pad = first & 3;
  if (((dp == 1 && (p.ldw & 3) == 0) || (dp == 2 && (p.ldw & 7) == 0)) && n_keep + pad <= p.limit) {
    k.path = dp;
    k.pad = pad;
    k.sel = dp == 1 ? 0 : (m + bb) & 1;
    k.w0 += -bb - m + (first >> 2) * (4 * dp);
  }
  k.nv = n_keep + k.pad;
  return k;
}
// Row of unit v's gate from unit 0 on; units that do not exist get a row of one that does.
__device__ __forceinline__ const unsigned short* kept_row(const KeptWeights& k, int gate, int v) {
  const int j = min(max(v, k.pad), k.nv - 1) - k.pad;
  return k.w0 + ((size_t)gate * k.H + k.bb + (size_t)j * k.dp) * k.ldw;
}
// The weights pass through shared memory: whole rows by bulk copies, `rows` of them a chunk, the chunks in a ring over everything behind
// the barriers.  (Gathered by the threads, 8 rows x 64 bytes a request, an SM gets 15 - 26 bytes a cycle however much is in flight and the
// prologue of 750 of 1500 units takes 41,000 cycles; one row per copy and one copy per warp at a time 31 - 45.)  A row lies at its own phase
// of 16 bytes; the 16 bytes at either end hold a byte of a kept unit, so they lie where the weight does.
struct RowRing {
  uint32_t base, bars, row_bytes, pitch;  // `pitch`: apart in shared memory
  int rows, slots, chunks;
  int chunk, slot;       // the chunk that is read now, and its slot
  uint32_t phase;        // of that slot's barrier
};
// Row i of chunk `chunk` (its address in the weight: row(chunk, i)) into a slot, by lane i / W of warp i % W.
template <int W, typename Row>
__device__ __forceinline__ void ring_request(const RowRing& r, int chunk, int slot, Row row) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, i = lane * W + warp;
  const uint32_t bar = r.bars + 8u * (uint32_t)slot;
  if (i < r.rows) {
    const unsigned long long a = reinterpret_cast<unsigned long long>(row(chunk, i)), from = a & ~15ull;
    const uint32_t bytes = ((uint32_t)a & 15u) + r.row_bytes + 15u & ~15u;
    mbar_arrive_expect_tx(bar, bytes);
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(r.base + (uint32_t)(slot * r.rows + i) * r.pitch), "l"(from), "r"(bytes), "r"(bar) : "memory");
  }
}
template <int W, int PHASE, typename Row>  // PHASE: of the pitch modulo 128: conflict-free reads of two rows x 64 bytes (64) or four rows x 32 bytes (32)
__device__ __forceinline__ RowRing ring_start(const KeptWeights& k, uint32_t base, int rows, int chunks, Row row) {
  RowRing r;
  const int groups = ((k.nv - 1) >> 2) + 1;
  r.row_bytes = (uint32_t)(k.path == 2 ? 16 * groups : (k.path == 1 ? 8 * groups : ((k.nv - 1) * k.dp + 1) * 2));
  r.pitch = ((r.row_bytes + 30u) / 128u + 1u) * 128u + PHASE;
  r.base = base + LC_BARS;
  r.bars = base + 16;
  r.rows = rows;
  r.chunks = chunks;
  r.slots = min(min(LC_RING, chunks), (int)((LC_SMEM_MAX - LC_BARS) / (rows * r.pitch)));
  r.chunk = r.slot = 0;
  r.phase = 0u;
  if (threadIdx.x == 0)
    for (int i = 0; i < r.slots; ++i) mbar_init(r.bars + 8u * i, (uint32_t)rows);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  __syncthreads();
  for (int i = 0; i < r.slots; ++i) ring_request<W>(r, i, i, row);
  return r;
}
__device__ __forceinline__ bool ring_wait(const RowRing& r, volatile int* abort_flag, int* status) {
  const bool ok = mbar_wait(r.bars + 8u * (uint32_t)r.slot, r.phase, abort_flag, status);
  __syncwarp();
  return ok;
}
// All threads, when they have read the chunk: another takes its place.  False: someone's wait failed.
template <int W, typename Row>
__device__ __forceinline__ bool ring_next(RowRing& r, bool ok, Row row) {
  if (barrier_failed(0, 32 * W, !ok)) {  // copies on their way have another millisecond before the block may end
    for (int x = 0; x < 1000; ++x) __nanosleep(1000);
    return false;
  }
  if (r.chunk + r.slots < r.chunks) ring_request<W>(r, r.chunk + r.slots, r.slot, row);
  ++r.chunk;
  if (++r.slot == r.slots) {
    r.slot = 0;
    r.phase ^= 1u;
  }
  return true;
}
// Address of unit 0 of the chunk's row i, the row of unit v's gate.
__device__ __forceinline__ uint32_t ring_row(const KeptWeights& k, const RowRing& r, int i, int gate, int v) {
  const int j = min(max(v, k.pad), k.nv - 1) - k.pad;  // as in kept_row; the low bits of its address
  const uint32_t at = (uint32_t)reinterpret_cast<unsigned long long>(k.w0) + (uint32_t)(gate * k.H + k.bb + j * k.dp) * (uint32_t)k.ldw * 2u;
  return r.base + (uint32_t)(r.slot * r.rows + i) * r.pitch + (at & 15u);
}

// Which of the units v .. v + 3 (v a multiple of 4) exist, as masks of two bf16 each.
__device__ __forceinline__ void unit_masks(const KeptWeights& k, int v, uint32_t& lo, uint32_t& hi) {
  auto one = [&](int x) { return x >= k.pad && x < k.nv; };
  lo = (one(v) ? 0xffffu : 0u) | (one(v + 1) ? 0xffff0000u : 0u);
  hi = (one(v + 2) ? 0xffffu : 0u) | (one(v + 3) ? 0xffff0000u : 0u);
}
// Weights of the units v .. v + 3 (v a multiple of 4, v < nv) of a staged row, those of units that do not exist arbitrary.
__device__ __forceinline__ uint32_t lds_u16(uint32_t addr) {
  unsigned short x;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(x) : "r"(addr) : "memory");
  return x;
}
template <int PATH>
__device__ __forceinline__ void load_units4(const KeptWeights& k, uint32_t row, int v, uint32_t& lo, uint32_t& hi) {
  if (PATH == 2) {
    uint32_t q[4];
    lds128(row + (uint32_t)v * 4u, q);
    const uint32_t s = k.sel ? 0x7632u : 0x5410u;
    lo = __byte_perm(q[0], q[1], s);
    hi = __byte_perm(q[2], q[3], s);
  } else if (PATH == 1) {
    uint32_t q[2];
    lds64(row + (uint32_t)v * 2u, q);
    lo = q[0];
    hi = q[1];
  } else {
    uint32_t e[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) e[i] = lds_u16(row + (uint32_t)(min(v + i, k.nv - 1) * k.dp * 2));
    lo = e[0] | (e[1] << 16);
    hi = e[2] | (e[3] << 16);
  }
}
// Weights of the units v, v + 1 (v even, v < nv), v in the low half.
template <int PATH>
__device__ __forceinline__ uint32_t load_units2(const KeptWeights& k, uint32_t row, int v) {
  if (PATH == 2) {
    uint32_t q[2];
    lds64(row + (uint32_t)v * 4u, q);
    return __byte_perm(q[0], q[1], k.sel ? 0x7632u : 0x5410u);
  }
  if (PATH == 1) {
    uint32_t q;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(q) : "r"(row + (uint32_t)v * 2u) : "memory");
    return q;
  }
  return lds_u16(row + (uint32_t)(v * k.dp * 2)) | lds_u16(row + (uint32_t)(min(v + 1, k.nv - 1) * k.dp * 2)) << 16;
}
// run(path) with the path as a constant.
template <typename Run>
__device__ __forceinline__ void by_path(const KeptWeights& k, Run run) {
  if (k.path == 2) run(std::integral_constant<int, 2>{});
  else if (k.path == 1) run(std::integral_constant<int, 1>{});
  else run(std::integral_constant<int, 0>{});
}

// The gate functions, without branches: a step's cells are a serial chain per thread, and behind the branches of tanhf and of an
// IEEE division the chains of a thread's cells do not overlap (two cells 1150 cycles, so 400).  Errors against 64 bits in ulps:
// tanh at most 1.64 for |x| up to 12 (tanhf 1.82); the sigmoid as the per-step kernels' 1 / (1 + __expf(-x)), 2.6 up to |x| = 1
// and 14.4 at 12.
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// 1 / (1 + exp(-x)), the exponential of the per-step kernels, one Newton step on the reciprocal.
__device__ __forceinline__ float gate_sigmoid(float x) {
  const float d = 1.f + __expf(-x), r = rcp_approx(d);
  return d < 1e38f ? fmaf(r, fmaf(-d, r, 1.f), r) : r;  // infinite d: 0; NaN stays
}
// tanh x = e / (e + 2) with e = exp(2x) - 1: 2x = n ln 2 + r, exp(r) - 1 by its series up to r^7 (|r| <= ln 2 / 2: 1.5e-8 of r left out),
// e = 2^n (exp(r) - 1) + (2^n - 1); a quotient corrected by its remainder, what e + 2 was rounded by included.  Below 0.17 the series of
// tanh itself up to x^9 (8e-11 of x left out).
__device__ __forceinline__ float gate_tanh(float x) {
  const float a = fabsf(x), y = a > 10.f ? 20.f : a + a;                   // (beyond 9.1 the result is 1)
  const float shifted = fmaf(y, 1.4426950408889634f, 12582912.f), n = shifted - 12582912.f;
  const float r = fmaf(n, 4.787419e-7f, fmaf(n, -0.69314765930175781f, y));  // ln 2 = 363409 / 2^19 - 4.787e-7
  float q = fmaf(r, 1.f / 5040.f, 1.f / 720.f);
  q = fmaf(q, r, 1.f / 120.f);
  q = fmaf(q, r, 1.f / 24.f);
  q = fmaf(q, r, 1.f / 6.f);
  q = fmaf(q, r, 0.5f);
  const float p = fmaf(r * r, q, r);
  const float s = __int_as_float((__float_as_int(shifted) << 23) + 0x3f800000);  // 2^n: the low bits of `shifted` are n
  const float e = fmaf(s, p, s - 1.f), d = e + 2.f, lost = e - (d - 2.f), i = rcp_approx(d), h = e * i;
  const float large = fmaf(fmaf(-h, lost, fmaf(-h, d, e)), i, h);
  const float x2 = a * a;
  float t = fmaf(x2, 62.f / 2835.f, -17.f / 315.f);
  t = fmaf(t, x2, 2.f / 15.f);
  t = fmaf(t, x2, -1.f / 3.f);
  const float small = fmaf(a * x2, t, a);
  return copysignf(a < 0.17f ? small : large, x);
}

// ======================================================================================================
// Forward.  CTA r of a cluster owns U virtual units from r * U on, in groups of 16.  Four warps serve a group: each multiplies the
// group's four tiles (16 units x one gate) by a quarter of h, all four leave their sums in shared memory, and each warp finishes a
// quarter of the cells: 8 units x 4 batch rows, whose gate values lie in 32-byte pieces (two tiles of 4 units x 4 gates and halves of h
// made it 16-byte pieces in 8 rows, and the loads and stores of a step took 1300 of its 4500 cycles).  A thread has all four
// gates of its cell, keeps its c, and four threads put four units' h_t together (two shuffles), 8 bytes that go to every CTA of
// the cluster.  Column 2 c + b of a product is batch row c + 4 b of its group of 8, so that a warp's rows lie together.
// NT: groups of 8 batch rows.  BESIDE: enqueued with the kernel over the whole grid.
template <int CL, int NT, bool BESIDE>
__global__ void __launch_bounds__(384, 1) ard_lstm_cluster_forward_kernel(const __grid_constant__ LstmClusterParams p) {
  constexpr int W = 12, LC_THREADS = 32 * W, LC_WARPS = W, LC_UNITS = lc_units(W), LC_TMEM_WARP = lc_tmem_warp(W);
  extern __shared__ __align__(128) uint8_t smem[];
  const uint32_t base = smem_u32(smem);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + LC_BARS - 8);
  volatile uint32_t* tmem_ptr_smem = reinterpret_cast<volatile uint32_t*>(smem + LC_BARS - 16);
  const uint32_t s_h = base + LC_BARS;                      // [2][NT] copies of h
  const uint32_t s_x = s_h + 2 * NT * LC_HB;                // [group][NT][cells' quarter][contraction's quarter] sums
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  pdl_launch_dependents();
  if (BESIDE && other_kernels_pattern(p)) return;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) mbar_init(base + 8u * i, 1);  // one per copy: h is complete
    *abort_flag = 0;
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_ptr_smem)), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_ptr_smem, my_w = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * LC_TMEM_WARP);
  pdl_wait_prior_grids();

  const int dp = p.hdr[HDR_DP], bb = p.hdr[HDR_B] - 1, n_keep = p.hdr[HDR_NKEEP];
  const bool taken = n_keep <= p.limit;  // the same for all CTAs
  if (!taken && p.alone && threadIdx.x == 0) atomicMax(p.status, (int)ARD_ERR_UNSUPPORTED);
  const KeptWeights k = kept_weights(p, dp, bb, n_keep);
  const int U = ((k.nv + CL - 1) / CL + 15) & ~15;  // units per CTA
  const int n_act = (k.nv + U - 1) / U;             // CTAs with units
  const int kq = (((k.nv + 15) >> 4) + 3) >> 2;     // contraction steps (16 units) of a quarter
  const int row0 = (int)(blockIdx.x / CL) * p.rows, crows = min(p.rows, p.B - row0);
  const int KH = p.I + p.H;
  const int group = warp >> 2, quarter = warp & 3;
  const int v_group = rank * U + 16 * group;
  const bool active = taken && rank * U < k.nv;                  // the same for all threads
  bool working = active && group < (U >> 4) && v_group < k.nv;  // the same for the warps of a group
  const int q = lane >> 2, c = lane & 3;

  // The weights: block 4 (i / 4) + gate holds steps i .. i + 3 of this quarter, the first two blocks in registers.  A chunk holds one
  // gate's rows q or q + 8 of every group.
  const int blocks = (kq + 3) >> 2;  // of four steps
  uint32_t w[LC_REG * 4];
#pragma unroll
  for (int i = 0; i < LC_REG * 4; ++i) w[i] = 0u;
  if (active) {
    auto row = [&](int chunk, int i) { return kept_row(k, chunk >> 1, rank * U + 16 * (i >> 3) + 8 * (chunk & 1) + (i & 7)); };
    RowRing ring = ring_start<W, 64>(k, base, 8 * (U >> 4), 8, row);
    const int v0 = quarter * kq * 16 + 4 * c, last = (k.nv - 1) & ~3;
    const bool edge = (quarter == 0 && k.pad > 0) || (quarter + 1) * kq * 16 > k.nv || (kq & 3) != 0;  // some of this warp's units do not exist
    uint32_t a[LC_KQ][4];
    // half the registers of this gate's operands (rows of units that do not exist hold another unit's weights: nobody uses their sums)
    auto take = [&](int g, auto half_tag) {
      constexpr int HALF = decltype(half_tag)::value;
      const uint32_t from = ring_row(k, ring, 8 * group + q, g, v_group + 8 * HALF + q);
      by_path(k, [&](auto path) {
#pragma unroll
        for (int i0 = 0; i0 < LC_KQ; i0 += 4)
          if (i0 < kq) {
#pragma unroll
            for (int i = i0; i < i0 + 4; ++i) load_units4<decltype(path)::value>(k, from, min(v0 + 16 * i, last), a[i][HALF], a[i][2 + HALF]);
          }
      });
    };
    bool ok = true;
#pragma unroll 1
    for (int g = 0; g < 4 && ok; ++g) {
      ok = ring_wait(ring, abort_flag, p.status);
      if (working) take(g, std::integral_constant<int, 0>{});
      ok = ring_next<W>(ring, ok, row);
      if (!ok) break;
      ok = ring_wait(ring, abort_flag, p.status);
      if (working) {
        take(g, std::integral_constant<int, 1>{});
        if (edge) {
          uint32_t first_lo, first_hi, last_lo, last_hi;
          unit_masks(k, 0, first_lo, first_hi);
          unit_masks(k, last, last_lo, last_hi);
#pragma unroll
          for (int i = 0; i < LC_KQ; ++i) {
            const int v = i < kq ? v0 + 16 * i : k.nv;
            const uint32_t all = v < last ? 0xffffffffu : 0u, lo = v == last ? last_lo : all, hi = v == last ? last_hi : all;
#pragma unroll
            for (int x = 0; x < 4; ++x) a[i][x] &= x & 2 ? hi : lo;
          }
          if (v0 == 0) {
#pragma unroll
            for (int x = 0; x < 4; ++x) a[0][x] &= x & 2 ? first_hi : first_lo;
          }
        }
#pragma unroll
        for (int x = 0; x < 32; ++x) set_if(g == x >> 4, w[x], a[x >> 2 & 3][x & 3]);
        __syncwarp();
#pragma unroll
        for (int ib = 0; ib < LC_KQ / 4; ++ib)
          if (ib < blocks && 4 * ib + g >= 2) tmem_st16(my_w + (uint32_t)((4 * ib + g - 2) * 16), &a[4 * ib][0]);
      }
      ok = ring_next<W>(ring, ok, row);
    }
    if (!ok) working = false;
    tmem_st_wait();
  }
  __syncthreads();
  for (uint32_t o = threadIdx.x * 16u; o < 2u * NT * LC_HB; o += LC_THREADS * 16u)
    *reinterpret_cast<uint4*>(smem + LC_BARS + o) = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  // h_0 of the cluster's rows: every CTA reads all of it
  if (active) {
    const unsigned short* h0 = reinterpret_cast<const unsigned short*>(p.XH) + (size_t)row0 * KH + p.I + bb;
    for (int j = threadIdx.x; j < n_keep; j += LC_THREADS) {
      const int v = j + k.pad;
      const uint32_t at = (uint32_t)((v >> 4) * 256 + (v & 3) * 2) + operand_offset(v >> 2 & 3, 0);
      unsigned short x[8 * NT];
#pragma unroll
      for (int r = 0; r < 8 * NT; ++r) x[r] = h0[(size_t)min(r, crows - 1) * KH + (size_t)j * dp];
#pragma unroll
      for (int r = 0; r < 8 * NT; ++r)  // (row r of a group is row 0's place with r * 8 flipped in)
        if (r < crows) *reinterpret_cast<unsigned short*>(smem + (at ^ (uint32_t)((r & 7) * 8)) + LC_BARS + (r >> 3) * LC_HB) = x[r];
    }
  }
  __syncwarp();
  cluster_sync_all();  // everyone's barriers, zeros and h_0 are in place before anyone sends

  const bool idle_warps = U < LC_UNITS && dp > 1;  // warps without a group write the zeros of the dropped units
  if (working) {
    const int n = c + 4 * (quarter & 1);  // the cells of this thread: its unit of the group, row n of 8
    const int v = v_group + q + 8 * (quarter >> 1), j = v - k.pad, u = bb + j * dp;
    const bool unit_here = j >= 0 && v < k.nv, piece_here = (v & ~3) < k.nv;
    const uint32_t piece = (uint32_t)LC_BARS + (uint32_t)(v >> 4) * 256u + operand_offset(v >> 2 & 3, n);
    uint32_t peer[CL / 4];  // this thread's shared memory in the CTAs that it sends to
    bool send[NT][CL / 4], cell[NT], load_zx[NT];
    float creg[NT], zx[NT][4], bias[4] = {0.f, 0.f, 0.f, 0.f};
    if (p.bias != nullptr && unit_here) {
#pragma unroll
      for (int g = 0; g < 4; ++g) bias[g] = p.bias[g * p.H + u];
    }
    // this thread's places in step t of the first 8 rows; the next rows' and the next step's follow by constants
    const size_t row = (size_t)(row0 + n);
    char* gp = reinterpret_cast<char*>(p.G + row * 4 * p.H + j);
    char* cp = reinterpret_cast<char*>(p.C + ((size_t)p.B + row) * p.H + j);
    char* xp = reinterpret_cast<char*>(p.XH + ((size_t)p.B + row) * KH + p.I + u);
    const size_t g_step = (size_t)p.B * 16 * p.H, c_step = (size_t)p.B * 4 * p.H, x_step = (size_t)p.B * 2 * KH;
    const int g_gate = 4 * p.H, g_rows = 8 * 16 * p.H, c_rows = 8 * 4 * p.H, x_rows = 8 * 2 * KH;
#pragma unroll
    for (int i = 0; i < CL / 4; ++i) peer[i] = mapa_u32(base, (uint32_t)((q & 3) + 4 * i));
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      const bool row_here = n < crows - 8 * nt;
      cell[nt] = unit_here && row_here;
      load_zx[nt] = cell[nt] && p.add_zx;
#pragma unroll
      for (int i = 0; i < CL / 4; ++i) send[nt][i] = piece_here && row_here && (q & 3) + 4 * i < n_act;
      creg[nt] = cell[nt] ? p.C[(row + 8 * nt) * p.H + j] : 0.f;
#pragma unroll
      for (int g = 0; g < 4; ++g) zx[nt][g] = ld_if(load_zx[nt], gp + nt * g_rows + g * g_gate);
    }
    const int col = lane >> 2;  // the column of the products that this lane brings: batch row (col >> 1) + 4 (col & 1)
    const uint32_t lane_h = s_h + (uint32_t)(quarter * kq * 256) + operand_offset(c, (col >> 1) + 4 * (col & 1));
    const uint32_t s_g = s_x + (uint32_t)(group * NT * 16 * LC_SWAP + lane * 16);
    const uint32_t bytes = (uint32_t)(((k.nv + 3) >> 2) * 8 * crows);
    bool ok = true;
    for (int t = 0; t < p.T; ++t) {
      const int buf = t & 1;
      uint32_t r[2][16];
      tmem_ld16(my_w, r[0]);
      if (threadIdx.x == 0 && t + 1 < p.T) mbar_arrive_expect_tx(base + 8u * (buf ^ 1), bytes);
      if (t > 0 && !mbar_wait_cluster(base + 8u * buf, (uint32_t)((t - 1) >> 1) & 1u, abort_flag, p.status)) ok = false;
      __syncwarp();
      constexpr int CH = NT == 1 ? 2 : 1;  // independent sums of a gate
      float acc[4][CH][NT][4] = {};
      const uint32_t hb = lane_h + (uint32_t)(buf * NT * LC_HB);
      uint32_t b[4][NT][2];
      auto multiply = [&](int g, const uint32_t* a) {  // four steps of one gate
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) mma_16816(acc[g][e % CH][nt], &a[4 * e], b[e][nt]);
      };
      auto operands = [&](int ib) {
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) lds64(hb + (uint32_t)(nt * LC_HB + (4 * ib + e) * 256), b[e][nt]);
      };
      operands(0);
      multiply(0, &w[0]);
      multiply(1, &w[16]);
      tmem_ld_wait();
      tmem_ld16(my_w + 16u, r[1]);
      multiply(2, r[0]);
      tmem_ld_wait();
      if (blocks > 1) tmem_ld16(my_w + 32u, r[0]);
      multiply(3, r[1]);
#pragma unroll 1
      for (int ib = 1; ib < blocks; ++ib) {
        const uint32_t at = my_w + (uint32_t)((4 * ib - 2) * 16);
        operands(ib);
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          tmem_ld_wait();
          if (g < 3 || ib + 1 < blocks) tmem_ld16(at + (uint32_t)((g + 1) * 16), r[(g + 1) & 1]);
          multiply(g, r[g & 1]);
        }
      }
      // The sums of the four quarters meet in shared memory: element e of a tile's sums belongs to the cells of warp e.  One buffer will
      // do: a warp reads before it sends its pieces of h_t, without which nobody gets to the next step.
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          uint32_t give[4];
#pragma unroll
          for (int g = 0; g < 4; ++g) give[g] = __float_as_uint(CH == 2 ? acc[g][0][nt][e] + acc[g][CH - 1][nt][e] : acc[g][0][nt][e]);
          sts128(s_g + (uint32_t)((nt * 16 + e * 4 + quarter) * LC_SWAP), give);
        }
      if (barrier_failed(1 + group, 128, !ok)) break;
      float z[NT][4];
      uint32_t h[NT];
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        uint32_t got[4][4];
#pragma unroll
        for (int x = 0; x < 4; ++x) lds128(s_g + (uint32_t)((nt * 16 + quarter * 4 + x) * LC_SWAP), got[x]);
#pragma unroll
        for (int g = 0; g < 4; ++g)
          z[nt][g] = (__uint_as_float(got[0][g]) + __uint_as_float(got[1][g])) + (__uint_as_float(got[2][g]) + __uint_as_float(got[3][g])) + (zx[nt][g] + bias[g]);
      }
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        z[nt][0] = gate_sigmoid(z[nt][0]);
        z[nt][1] = gate_sigmoid(z[nt][1]);
        z[nt][2] = gate_tanh(z[nt][2]);
        z[nt][3] = gate_sigmoid(z[nt][3]);
        creg[nt] = z[nt][1] * creg[nt] + z[nt][0] * z[nt][2];
      }
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) h[nt] = cell[nt] ? __bfloat16_as_ushort(__float2bfloat16_rn(p.alpha * z[nt][3] * gate_tanh(creg[nt]))) : 0u;
      if (t + 1 < p.T) {
        const uint32_t bar = 8u * (uint32_t)(buf ^ 1);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          const uint32_t a1 = __shfl_xor_sync(0xffffffffu, h[nt], 4);
          const uint32_t two = q & 1 ? a1 | (h[nt] << 16) : h[nt] | (a1 << 16);
          const uint32_t a2 = __shfl_xor_sync(0xffffffffu, two, 8);
          const uint32_t lo = q & 2 ? a2 : two, hi = q & 2 ? two : a2, dst = piece + (uint32_t)(((buf ^ 1) * NT + nt) * LC_HB);
#pragma unroll
          for (int i = 0; i < CL / 4; ++i) st_async_8(send[nt][i], peer[i] + dst, peer[i] + bar, lo, hi);
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
          for (int g = 0; g < 4; ++g) zx[nt][g] = ld_if(load_zx[nt], gp + g_step + nt * g_rows + g * g_gate);
      }
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
        for (int g = 0; g < 4; ++g) st_if(cell[nt], gp + nt * g_rows + g * g_gate, z[nt][g]);
        st_if(cell[nt], cp + nt * c_rows, creg[nt]);
        st16_if(cell[nt], xp + nt * x_rows, h[nt]);
      }
      if (dp > 1 && !idle_warps) {  // the j-th kept unit owns the units [j * dp, (j + 1) * dp), the last one the tail
        const int first = -bb, last = (j == n_keep - 1 ? p.H : (j + 1) * dp) - u;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
          for (int x = first; x < last; ++x) st16_if(cell[nt] && x != 0, xp + nt * x_rows + 2 * x, 0u);
      }
      gp += g_step;
      cp += c_step;
      xp += x_step;
    }
  } else if (taken && idle_warps && 16 * group >= U) {
    const int seg = (p.H + CL - 1) / CL, c0 = rank * seg, c1 = min(p.H, c0 + seg);
    for (int x = warp - (U >> 2); x < p.T * crows; x += LC_WARPS - (U >> 2)) {
      const int t = x / crows, r = x - t * crows;
      __nv_bfloat16* hrow = p.XH + ((size_t)(t + 1) * p.B + row0 + r) * KH + p.I;
      for (int u = c0 + lane; u < c1; u += 32)
        if (u < bb || (u - bb) % dp != 0) hrow[u] = __float2bfloat16_rn(0.f);
    }
  }
  __syncwarp();
  tc_fence_before();
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

// ======================================================================================================
// BPTT.  CTA r owns U units (U = 4 KS): their cell adjoint gives 4 U gate gradients, which stay in the CTA: it multiplies them by
// its rows of the weight for ALL kept units and sends every CTA the partial sums of that one's units (an all-gather of the
// gradients would move twice the bytes).  The receiver adds the shares in the order of the CTAs.  The contraction index is
// (unit, gate), so a thread's four gate gradients are the 8 bytes of the operand that another thread reads whole.
// Tiles of 16 output units are dealt to the warps round-robin; row g of a tile is unit 2 g, row g + 8 unit 2 g + 1.  A tile's sums
// lie as [column pair c][g][4]: 16 bytes of one thread, and the cells of warp (tile, c) are consecutive words.
__host__ __device__ constexpr int lcb_tiles(int CL, int KS, int W) { return (CL * KS / 4 + W - 1) / W; }  // per warp
__host__ __device__ constexpr int lcb_sums(int CL, int KS) { return CL * (KS / 4) * 512; }  // partial sums of 8 rows, one step
__host__ __device__ constexpr int lcb_smem(int CL, int KS, int NT) { return LC_BARS + 2 * NT * lcb_sums(CL, KS) + 2 * NT * KS * 256; }

struct SavedCell {
  float gi, gf, gg, go, cp, up;
};

// The zeros of the weight gradient's dropped rows are bulk copies from LC_ZERO bytes of zeros at the end of shared memory; this is the i-th
// row of the CTA.
constexpr int LC_ZERO = 16 * 1024;
__device__ __forceinline__ void zero_dropped_weight_row(const LstmClusterParams& p, uint32_t zeros, int i, int dp, int bb) {
  const int x = (int)blockIdx.x + (int)gridDim.x * i;
  if (x >= 4 * p.H) return;
  const int u = x % p.H;
  if (u >= bb && (u - bb) % dp == 0) return;
  char* d = reinterpret_cast<char*>(p.dW + (size_t)x * p.ld_dw);
  for (int left = 4 * p.dw_cols; left > 0; left -= LC_ZERO, d += LC_ZERO) bulk_store(d, zeros, (uint32_t)min(left, LC_ZERO));
}

// ZEROS: with those of the weight gradient (a kernel of its own: the code alone costs the others 1.5 us, cold as it is).
template <int CL, int NT, int W, int KS, bool ZEROS>
__device__ __forceinline__ void lstm_cluster_backward_body(const LstmClusterParams& p, uint8_t* smem, uint32_t base, uint32_t tmem_base,
                                                           volatile int* abort_flag, int rank, const KeptWeights& k, int n_keep) {
  constexpr int LC_THREADS = 32 * W, LC_WARPS = W, LC_TMEM_WARP = lc_tmem_warp(W);
  constexpr int U = 4 * KS, TPC = KS / 4;  // units and tiles of a CTA
  constexpr int TILES = lcb_tiles(CL, KS, W), OPS = TILES * KS, QUADS = OPS / 4;  // weight operands of a warp, fours of them
  static_assert(OPS >= LC_REG && 4 * (OPS - LC_REG) <= LC_TMEM_WARP, "weight operands");
  constexpr int SUMS = lcb_sums(CL, KS);
  const uint32_t s_p = base + LC_BARS, s_dz = s_p + 2 * NT * SUMS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int T = p.T, KH = p.I + p.H, dp = k.dp, bb = k.bb;
  const int row0 = (int)(blockIdx.x / CL) * p.rows, crows = min(p.rows, p.B - row0);
  const int n_act = (k.nv + U - 1) / U, tt = (k.nv + 15) >> 4;
  const int v_first = rank * U;
  const bool active = v_first < k.nv;
  const int q = lane >> 2, c = lane & 3;
  const uint32_t my_w = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * LC_TMEM_WARP);

  // Weights: rows = output units, contraction = (own unit, gate).  Operand i * KS + ks is step ks of tile warp + W i, the first LC_REG in
  // registers.  A chunk holds the four gates' rows of the four units of a step.
  uint32_t w[LC_REG * 4];
#pragma unroll
  for (int i = 0; i < LC_REG * 4; ++i) w[i] = 0u;
  bool ok = true;
  if (active) {
    auto from_weight = [&](int ks, int i) { return kept_row(k, i >> 2, v_first + 4 * ks + (i & 3)); };
    RowRing ring = ring_start<W, 32>(k, base, 16, KS, from_weight);
#pragma unroll 1
    for (int ks = 0; ks < KS && ok; ++ks) {
      ok = ring_wait(ring, abort_flag, p.status);
      const int vc = v_first + 4 * ks + c;
      const uint32_t exists = vc >= k.pad && vc < k.nv ? 0xffffffffu : 0u;
      uint32_t from[4];
#pragma unroll
      for (int g = 0; g < 4; ++g) from[g] = ring_row(k, ring, 4 * g + c, g, vc);
      by_path(k, [&](auto path) {
        uint32_t e[TILES][4];
#pragma unroll
        for (int i = 0; i < TILES; ++i) {  // (columns of units that do not exist: nobody uses their sums)
          const int at = min((warp + i * LC_WARPS) * 16 + 2 * q, (k.nv - 1) & ~1);
#pragma unroll
          for (int g = 0; g < 4; ++g) e[i][g] = load_units2<decltype(path)::value>(k, from[g], at) & exists;
        }
#pragma unroll
        for (int i = 0; i < TILES; ++i) {
          const int op = i * KS + ks;
          const uint32_t a[4] = {__byte_perm(e[i][0], e[i][1], 0x5410), __byte_perm(e[i][0], e[i][1], 0x7632), __byte_perm(e[i][2], e[i][3], 0x5410),
                                 __byte_perm(e[i][2], e[i][3], 0x7632)};
          if (i * KS < LC_REG) {
#pragma unroll
            for (int x = i * KS; x < i * KS + KS && x < LC_REG; ++x)
#pragma unroll
              for (int y = 0; y < 4; ++y) set_if(x == op, w[4 * x + y], a[y]);
          }
          if (op >= LC_REG) tmem_st4(my_w + (uint32_t)((op - LC_REG) * 4), a);
        }
      });
      ok = ring_next<W>(ring, ok, from_weight);
    }
    tmem_st_wait();
  }
  __syncthreads();
  for (uint32_t o = threadIdx.x * 16u; o < 2u * NT * SUMS; o += LC_THREADS * 16u)
    *reinterpret_cast<uint4*>(smem + LC_BARS + o) = make_uint4(0u, 0u, 0u, 0u);
  if constexpr (ZEROS) {
    for (uint32_t o = threadIdx.x * 16u; o < (uint32_t)LC_ZERO; o += LC_THREADS * 16u)
      *reinterpret_cast<uint4*>(smem + LC_SMEM_MAX - LC_ZERO + o) = make_uint4(0u, 0u, 0u, 0u);
    fence_proxy_async_smem();  // (read by bulk copies)
  }
  __syncwarp();
  cluster_sync_all();  // everyone's barriers and zeros are in place before anyone sends
  // Zeros of the weight gradient: a burst of rows in every eighth step, or all here where a step has as many products as to have no room for
  // the code (64 rows, 512 of 1024 units kept, us of the recurrence: 78 without zeros, 80.6 all here, 94 in bursts; 20 rows, 188 of 1500: 45, 61
  // and 53; some rows in every step 56).
  constexpr int BURST = KS <= 8 ? 8 : 0;
  const uint32_t s_zeros = base + (uint32_t)(LC_SMEM_MAX - LC_ZERO);
  const int zero_rows = dp > 1 ? (4 * p.H + (int)gridDim.x - 1) / (int)gridDim.x : 0;  // of this CTA
  const int bursts = BURST > 0 ? (T + BURST - 1) / BURST : 1, zero_burst = (zero_rows + bursts - 1) / bursts;
  if (ZEROS && (BURST == 0 || !active))
    for (int i = warp + W * lane; i < zero_rows; i += 32 * W) zero_dropped_weight_row(p, s_zeros, i, dp, bb);

  // the cells of this thread: warps 0 .. 4 TPC - 1, unit lane / 2 of tile warp / 4, row 2 (warp % 4) + lane % 2 of a group
  const int ct = warp >> 2, n = 2 * (warp & 3) + (lane & 1);
  const int v = v_first + 16 * ct + (lane >> 1), j = v - k.pad, u = bb + j * dp;
  const bool unit_here = active && ct < TPC && j >= 0 && v < k.nv;
  const uint32_t dz_piece = (uint32_t)((4 * ct + (lane >> 3)) * 256) + operand_offset(lane >> 1 & 3, n);
  const uint32_t my_sums = s_p + (uint32_t)(ct * 512 + (warp & 3) * 128 + lane * 4);
  // this thread's places in step t of the first group of rows; the next group's and the step's before follow by constants
  const size_t row = (size_t)(row0 + n);
  const char* gp = reinterpret_cast<const char*>(p.G + ((size_t)(T - 1) * p.B + row) * 4 * p.H + j);
  const char* cp = reinterpret_cast<const char*>(p.C + ((size_t)(T - 1) * p.B + row) * p.H + j);
  const char* hp = p.dH != nullptr ? reinterpret_cast<const char*>(p.dH + ((size_t)(T - 1) * p.B + row) * p.H + u)
                                   : reinterpret_cast<const char*>(p.D + ((size_t)T * p.B + row) * KH + p.I + u);
  char* zp = reinterpret_cast<char*>(p.DZ + ((size_t)(T - 1) * p.B + row) * 4 * p.gs + j);
  const size_t g_step = (size_t)p.B * 16 * p.H, c_step = (size_t)p.B * 4 * p.H, h_step = (size_t)p.B * 4 * (p.dH != nullptr ? p.H : KH);
  const size_t z_step = (size_t)p.B * 8 * p.gs;
  const int g_gate = 4 * p.H, g_rows = 8 * 16 * p.H, c_rows = 8 * 4 * p.H, h_rows = 8 * 4 * (p.dH != nullptr ? p.H : KH), z_rows = 8 * 8 * p.gs;
  bool cell[NT] = {};
  float dcreg[NT], c_now[NT];
  SavedCell next[NT];
  auto fetch = [&](int nt, SavedCell& s) {  // what the adjoint of the step that the places stand for reads besides the recurrent sums
    const char* g = gp + nt * g_rows;
    s.gi = ld_if(cell[nt], g);
    s.gf = ld_if(cell[nt], g + g_gate);
    s.gg = ld_if(cell[nt], g + 2 * g_gate);
    s.go = ld_if(cell[nt], g + 3 * g_gate);
    s.cp = ld_if(cell[nt], cp + nt * c_rows);
  };
  uint32_t share_bytes = 0;  // of one step
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    cell[nt] = unit_here && n < crows - 8 * nt;
    const size_t at = row + 8 * nt;
    dcreg[nt] = cell[nt] && p.dH == nullptr ? p.dc[at * p.H + j] : 0.f;
    c_now[nt] = ld_if(cell[nt], cp + c_step + nt * c_rows);
    fetch(nt, next[nt]);
    next[nt].up = p.dH != nullptr ? ld_if(cell[nt], hp + nt * h_rows) : ld_if(cell[nt], p.dH_last + at * p.H + u);
    if (active) share_bytes += (uint32_t)(min(TPC, tt - rank * TPC) * ((min(8, max(0, crows - 8 * nt)) + 1) / 2) * 128 * n_act);
  }
  for (int s = 0; s <= T && active && ok; ++s) {
    const int t = T - 1 - s, buf = s & 1;  // time index whose dh is formed in this round (-1: the gradient of h_0)
    // The cell adjoint is linear in dh: with dcv = dc + dh * fc, the gradient of c_t, the gates' dz are dcv * i, dcv * f,
    // dcv * g and dh * o.  The factors are formed, and the next step's values asked for, while the sums are on their way.
    float fc[NT], fi[NT], ff[NT], fg[NT], fo[NT], fnext[NT], total[NT], rec[NT];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      const SavedCell in = next[nt];
      const float tc = gate_tanh(c_now[nt]);
      fc[nt] = p.alpha * in.go * (1.f - tc * tc);
      fi[nt] = in.gg * in.gi * (1.f - in.gi);
      ff[nt] = in.cp * in.gf * (1.f - in.gf);
      fg[nt] = in.gi * (1.f - in.gg * in.gg);
      fo[nt] = p.alpha * tc * in.go * (1.f - in.go);
      fnext[nt] = in.gf;
      total[nt] = in.up;
      rec[nt] = 0.f;
      c_now[nt] = in.cp;
    }
    gp -= g_step;
    cp -= c_step;
    hp -= h_step;
    if (t > 0) {
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        fetch(nt, next[nt]);
        next[nt].up = ld_if(cell[nt], hp + nt * h_rows);
      }
    }
    if (threadIdx.x == 0 && t >= 0) mbar_arrive_expect_tx(base + 8u * (buf ^ 1), share_bytes);
    if (s > 0 && ct < TPC) {
      if (!mbar_wait_cluster(base + 8u * buf, (uint32_t)((s - 1) >> 1) & 1u, abort_flag, p.status)) ok = false;
      // (what lies in rows that do not exist is not used; CTAs without units have left zeros)
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        const float* sums = reinterpret_cast<const float*>(smem + (my_sums - base) + (buf * NT + nt) * SUMS);
        float x[CL];
#pragma unroll
        for (int r = 0; r < CL; ++r) x[r] = sums[r * TPC * 128];
#pragma unroll
        for (int r = 0; r < CL; ++r) rec[nt] += x[r];
      }
    }
    if (t < 0) {  // gradient of h_0
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        if (!cell[nt] || !ok) continue;
        float* d0 = p.D + (row + 8 * nt) * KH + p.I;
        if (p.dH == nullptr) {
          d0[u] += rec[nt];  // to what the caller left there
        } else {  // nothing was there: zeros of the dropped units; the j-th kept one owns [j * dp, (j + 1) * dp), the last the tail
          const int last = j == n_keep - 1 ? p.H : min(p.H, (j + 1) * dp);
          for (int x = j * dp; x < last; ++x) d0[x] = x == u ? rec[nt] : 0.f;
        }
      }
      break;
    }
    uint32_t dz[NT][2];  // i | f, g | o
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      total[nt] += rec[nt];
      const float dcv = dcreg[nt] + total[nt] * fc[nt];
      dcreg[nt] = dcv * fnext[nt];
      const __nv_bfloat162 a = __floats2bfloat162_rn(dcv * fi[nt], dcv * ff[nt]), b = __floats2bfloat162_rn(dcv * fg[nt], total[nt] * fo[nt]);
      dz[nt][0] = cell[nt] ? *reinterpret_cast<const uint32_t*>(&a) : 0u;
      dz[nt][1] = cell[nt] ? *reinterpret_cast<const uint32_t*>(&b) : 0u;
      if (ct < TPC)
        asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(s_dz + (uint32_t)((buf * NT + nt) * KS * 256) + dz_piece), "r"(dz[nt][0]), "r"(dz[nt][1]) : "memory");
    }
    if (barrier_failed(1, LC_THREADS, !ok)) { ok = false; break; }
    {
      uint32_t r[2][16];
      if (OPS > LC_REG) tmem_ld16(my_w, r[0]);
      uint32_t b[NT][KS][2];
#pragma unroll
      for (int ks = 0; ks < KS; ++ks)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) lds64(s_dz + (uint32_t)((buf * NT + nt) * KS * 256 + ks * 256) + operand_offset(c, q), b[nt][ks]);
      float acc[NT][2][4];  // two independent sums
#pragma unroll
      for (int f = 0; f < QUADS; ++f) {  // operands 4 f .. 4 f + 3, of one tile
        const int i = 4 * f / KS, tile = warp + i * LC_WARPS;
        if (4 * f >= LC_REG) {
          tmem_ld_wait();
          if (f + 1 < QUADS) tmem_ld16(my_w + (uint32_t)((4 * (f + 1) - LC_REG) * 4), r[(f + 1) & 1]);
        }
        if (4 * f % KS == 0) {
#pragma unroll
          for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int x = 0; x < 4; ++x) acc[nt][0][x] = acc[nt][1][x] = 0.f;
        }
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int nt = 0; nt < NT; ++nt)
            mma_16816(acc[nt][x & 1], 4 * f < LC_REG ? &w[(4 * f + x) * 4 % (LC_REG * 4)] : &r[f & 1][4 * x], b[nt][(4 * f + x) % KS]);
        if (4 * (f + 1) % KS == 0 && tile < tt) {  // the tile is complete
          const uint32_t dst = (uint32_t)(tile / TPC), local = (uint32_t)(tile % TPC), peer = mapa_u32(base, dst);
#pragma unroll
          for (int nt = 0; nt < NT; ++nt)
            if (2 * c < crows - 8 * nt)
              st_async_f4(peer + (s_p - base) + (uint32_t)(((buf ^ 1) * NT + nt) * SUMS) + ((uint32_t)(rank * TPC) + local) * 512u + (uint32_t)(c * 128 + q * 16),
                          peer + 8u * (buf ^ 1), acc[nt][0][0] + acc[nt][1][0], acc[nt][0][1] + acc[nt][1][1], acc[nt][0][2] + acc[nt][1][2],
                          acc[nt][0][3] + acc[nt][1][3]);
          __syncwarp();
        }
      }
    }
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      char* d = zp + nt * z_rows;
#pragma unroll
      for (int g = 0; g < 4; ++g) st16_if(cell[nt], d + 2 * g * p.gs, dz[nt][g >> 1] >> (16 * (g & 1)));
    }
    zp -= z_step;
    if constexpr (ZEROS && BURST > 0) {
      if (s % BURST == 0)
        for (int i = warp + W * lane; i < zero_burst; i += 32 * W) zero_dropped_weight_row(p, s_zeros, s / BURST * zero_burst + i, dp, bb);
    }
    if (p.dH == nullptr || p.DZ_out != nullptr) {
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        if (!cell[nt]) continue;
        const size_t at = (size_t)t * p.B + row + 8 * nt;
        if (p.DZ_out != nullptr) {
          unsigned short* o = reinterpret_cast<unsigned short*>(p.DZ_out) + at * 4 * p.H + j;
#pragma unroll
          for (int g = 0; g < 4; ++g) o[(size_t)g * p.H] = (unsigned short)(dz[nt][g >> 1] >> (16 * (g & 1)));
        }
        if (t < T - 1 && p.dH == nullptr) p.D[(at + p.B) * KH + p.I + u] = total[nt];  // the caller's D holds the totals afterwards
      }
    }
    __syncwarp();
  }
  if (ok) {
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
      if (cell[nt]) {
        float* dc = p.dc + (row + 8 * nt) * p.H;
        dc[j] = dcreg[nt];
        if (p.dH != nullptr)  // nothing was there: zeros behind the kept columns
          for (int x = j + n_keep; x < p.H; x += n_keep) dc[x] = 0.f;
      }
  }
  if constexpr (ZEROS) {
    bulk_commit();
    bulk_wait_all();
  }
}

template <int CL, int NT, int W, bool ZEROS, bool BESIDE>
__global__ void __launch_bounds__(32 * W, 1) ard_lstm_cluster_backward_kernel(const __grid_constant__ LstmClusterParams p) {
  extern __shared__ __align__(128) uint8_t smem[];
  const uint32_t base = smem_u32(smem);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + LC_BARS - 8);
  volatile uint32_t* tmem_ptr_smem = reinterpret_cast<volatile uint32_t*>(smem + LC_BARS - 16);
  const int warp = threadIdx.x >> 5;
  const int rank = (int)cluster_ctarank();
  pdl_launch_dependents();
  if (BESIDE && other_kernels_pattern(p)) return;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) mbar_init(base + 8u * i, 1);  // one per set of partial sums: they are complete
    *abort_flag = 0;
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_ptr_smem)), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_ptr_smem;
  pdl_wait_prior_grids();
  const int dp = p.hdr[HDR_DP], bb = p.hdr[HDR_B] - 1, n_keep = p.hdr[HDR_NKEEP];
  if (n_keep <= p.limit) {  // the same for all CTAs
    const KeptWeights k = kept_weights(p, dp, bb, n_keep);
    bool done = false;  // four units a step: the fewest steps that the units fit
    if constexpr (CL == 16) {
      done = k.nv <= 16 * CL;
      if (done) lstm_cluster_backward_body<CL, NT, W, 4, ZEROS>(p, smem, base, tmem_base, abort_flag, rank, k, n_keep);
    }
    if (done) {
    } else if (k.nv <= 32 * CL) {
      lstm_cluster_backward_body<CL, NT, W, 8, ZEROS>(p, smem, base, tmem_base, abort_flag, rank, k, n_keep);
    } else if (W == 12 || k.nv <= 48 * CL) {
      lstm_cluster_backward_body<CL, NT, W, 12, ZEROS>(p, smem, base, tmem_base, abort_flag, rank, k, n_keep);
    } else if constexpr (W == 16) {
      lstm_cluster_backward_body<CL, NT, W, 16, ZEROS>(p, smem, base, tmem_base, abort_flag, rank, k, n_keep);
    }
  } else if (p.alone && threadIdx.x == 0) {
    atomicMax(p.status, (int)ARD_ERR_UNSUPPORTED);
  }
  __syncwarp();
  tc_fence_before();
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

// ---- launch ----------------------------------------------------------------------------------------------------------
constexpr int lcf_smem(int NT) { return LC_BARS + 2 * NT * LC_HB + 12 * NT * 4 * LC_SWAP; }
static_assert(lcf_smem(3) <= LC_SMEM_MAX && lcb_smem(16, 12, 3) + LC_ZERO <= LC_SMEM_MAX && lcb_smem(8, 16, 1) + LC_ZERO <= LC_SMEM_MAX,
              "shared memory of the cluster recurrences");

using ClusterKernel = void (*)(LstmClusterParams);
struct ClusterForm {
  ClusterKernel kern, kern_zeros, kern_beside;  // nullptr: not taken; the one that also writes zeros of the weight gradient; BESIDE
  int cl, threads, nt, limit;
  int clusters, rows;
};

// Clusters of this form that the device holds at once; 0 where it holds none.
int cluster_count(const ard_ctx* ctx, const ClusterForm& f) {
  for (ClusterKernel kern : {f.kern, f.kern_zeros, f.kern_beside})
    if (kern != nullptr && (cudaFuncSetAttribute((const void*)kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
                            cudaFuncSetAttribute((const void*)kern, cudaFuncAttributeMaxDynamicSharedMemorySize, LC_SMEM_MAX) != cudaSuccess)) {
      (void)cudaGetLastError();
      return 0;
    }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctx->sm_count / f.cl * f.cl);
  cfg.blockDim = dim3(f.threads);
  cfg.dynamicSmemBytes = LC_SMEM_MAX;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = f.cl;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, (const void*)f.kern, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return n;
}

// (the other kernel is needed only where 16 CTAs may not hold the kept units: cluster_form)
template <int CL, int NT>
ClusterForm forward_form() {
  ClusterForm f = {ard_lstm_cluster_forward_kernel<CL, NT, false>, nullptr, nullptr, CL, 384, NT, CL * lc_units(12), 0, 0};
  if constexpr (CL == 16) f.kern_beside = ard_lstm_cluster_forward_kernel<CL, NT, true>;
  return f;
}
template <int CL, int NT, int W>
ClusterForm backward_form() {
  ClusterForm f = {ard_lstm_cluster_backward_kernel<CL, NT, W, false, false>, ard_lstm_cluster_backward_kernel<CL, NT, W, true, false>, nullptr, CL,
                   32 * W, NT, CL * lc_units(W), 0, 0};
  if constexpr (CL == 16) f.kern_beside = ard_lstm_cluster_backward_kernel<CL, NT, W, false, true>;
  return f;
}

// The form for a layer that keeps n_max units at most, in the order in which they are preferred: clusters of 8 where the weights fit eight
// CTAs (more clusters, so fewer rows in each, and fewer CTAs to send to).  For 385 to 512 units the backward kernel has a form of 8 CTAs of 16
// warps, better than 16 CTAs with a second group of rows (64 rows, 512 of 1024 units kept, 35 steps: 85 -> 78 us; the forward kernel that way
// 99 -> 106: its exchange is not hidden), not better than 16 CTAs with one.
template <bool BWD>
ClusterForm cluster_form(const ard_ctx* ctx, int B, int n_max) {
  static const ClusterForm forward[] = {forward_form<8, 1>(), forward_form<8, 2>(), forward_form<16, 1>(), forward_form<16, 2>(), forward_form<16, 3>(), {}};
  static const ClusterForm backward[] = {backward_form<8, 1, 12>(), backward_form<8, 2, 12>(), backward_form<16, 1, 12>(),
                                         backward_form<8, 1, 16>(), backward_form<16, 2, 12>(), backward_form<16, 3, 12>()};
  constexpr int FORMS = 6;
  const ClusterForm* forms = BWD ? backward : forward;
  static std::atomic<int> room[64][FORMS];  // clusters at once, plus one; 0: not asked yet
  for (int i = 0; i < FORMS; ++i) {
    ClusterForm f = forms[i];
    if (f.kern == nullptr || (n_max > f.limit && f.cl == 8)) continue;
    std::atomic<int>& known = room[ctx->device & 63][i];
    int have = known.load(std::memory_order_relaxed);
    if (have == 0) known.store(have = 1 + cluster_count(ctx, f), std::memory_order_relaxed);
    if (have <= 1) continue;
    f.rows = (B + have - 2) / (have - 1);
    if (f.rows > 8 * f.nt) continue;
    f.clusters = (B + f.rows - 1) / f.rows;
    return f;
  }
  return {};
}

ard_status launch_cluster(ard_ctx* ctx, const ClusterForm& f, const LstmClusterParams& p, cudaStream_t s) {
  if (ctx->lstm_refuse & 1) return ARD_ERR_UNSUPPORTED;
  const cudaError_t err = ard_launch_cluster(ctx, f.kern, f.cl, dim3(f.cl * f.clusters), dim3(f.threads), LC_SMEM_MAX, s, p);
  if (err != cudaSuccess) {
    (void)cudaGetLastError();
    return err == cudaErrorLaunchOutOfResources || err == cudaErrorInvalidClusterSize ? ARD_ERR_UNSUPPORTED : ARD_ERR_CUDA;
  }
  ctx->launches++;
  return ARD_OK;
}

}  // namespace

int lstm_cluster_limit(const ard_ctx* ctx, int B, int n_max, bool backward) {
  const ClusterForm f = backward ? cluster_form<true>(ctx, B, n_max) : cluster_form<false>(ctx, B, n_max);
  return f.kern ? f.limit : 0;
}

ard_status launch_lstm_forward_cluster(ard_ctx* ctx, const ard_pattern* pat, int n_max, int T, int B, int I, int H, int add_zx, float alpha,
                                       const void* W, int ldw, void* XH, const float* bias, float* C, float* G, cudaStream_t s) {
  ClusterForm f = cluster_form<false>(ctx, B, n_max);
  if (!f.kern) return ARD_ERR_UNSUPPORTED;
  LstmClusterParams p = {};
  p.hdr = pat->d_hdr;
  p.T = T; p.B = B; p.I = I; p.H = H;
  p.rows = f.rows;
  p.limit = f.limit;
  p.alone = n_max <= f.limit;
  if (!p.alone) f.kern = f.kern_beside;
  p.alpha = alpha;
  p.W = reinterpret_cast<const __nv_bfloat16*>(W);
  p.ldw = ldw;
  p.status = ctx->d_status;
  p.C = C;
  p.G = G;
  p.add_zx = add_zx;
  p.XH = reinterpret_cast<__nv_bfloat16*>(XH);
  p.bias = bias;
  return launch_cluster(ctx, f, p, s);
}

ard_status launch_lstm_backward_cluster(ard_ctx* ctx, const ard_pattern* pat, int n_max, int T, int B, int I, int H, float alpha,
                                        const void* W, int ldw, const float* C, const float* G, const float* dH, const float* dH_last,
                                        float* D, float* dc, void* DZ, int gs, void* DZ_out, float* dW, int ld_dw, int dw_cols, bool* zeros,
                                        cudaStream_t s) {
  *zeros = false;
  ClusterForm f = cluster_form<true>(ctx, B, n_max);
  if (!f.kern) return ARD_ERR_UNSUPPORTED;
  LstmClusterParams p = {};
  p.hdr = pat->d_hdr;
  p.T = T; p.B = B; p.I = I; p.H = H;
  p.rows = f.rows;
  p.limit = f.limit;
  p.alone = n_max <= f.limit;
  if (!p.alone) f.kern = f.kern_beside;
  p.alpha = alpha;
  p.W = reinterpret_cast<const __nv_bfloat16*>(W);
  p.ldw = ldw;
  p.status = ctx->d_status;
  p.C = const_cast<float*>(C);
  p.G = const_cast<float*>(G);
  p.dH = dH; p.dH_last = dH_last; p.D = D; p.dc = dc;
  p.DZ = reinterpret_cast<__nv_bfloat16*>(DZ);
  p.gs = gs;
  p.DZ_out = reinterpret_cast<__nv_bfloat16*>(DZ_out);
  // The zeros of dW's dropped rows pay here: the product that computes the kept rows takes 31.5 -> 25 us without them (33 MB of dW, half of it
  // zero), 38 -> 25 (72 MB, half), 44 -> 17.5 (72 MB, seven eighths), this kernel 2.5, 6 and 8 us more with them.  The smallest layers that
  // gained had 0.8 MB (12 steps, 87.3 -> 85.9 the whole pass); 0.5 MB lost (29 steps, 109.7 -> 111.7).
  constexpr size_t least = 640u << 10;
  if (p.alone && dW != nullptr && (uintptr_t)dW % 16 == 0 && ld_dw % 4 == 0 && dw_cols % 4 == 0 && (size_t)16 * H * dw_cols >= least) {
    p.dW = dW;
    p.ld_dw = ld_dw;
    p.dw_cols = dw_cols;
    f.kern = f.kern_zeros;
  }
  const ard_status st = launch_cluster(ctx, f, p, s);
  *zeros = st == ARD_OK && p.dW != nullptr;
  return st;
}
