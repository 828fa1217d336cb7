// QK4PV8 prefill (Algorithm 1 lines 6-20) for sm_100a.
//
// A work item is one 128-row query tile of one q head; its KV blocks (128 keys) are visited from the last
// visible block down to block 0 (Section 4.1).  One persistent CTA per SM walks a static list of work items
// (struct TileWalk) and keeps its pipeline running across item boundaries.  Roles (640 threads):
//   warp 0       producer: K codes (tensor map, 64B swizzle), K scale factors and Delta_S (bulk copies)
//                and V (tensor map, 128B swizzle) into rings of 4 stages; in the paged variant (template
//                parameter PAGED, entry point mpfa_prefill_paged) every tile half is one bulk copy of a
//                64-token page slab, found through the page table;
//   warp 2       paged variant only: re-tiles the pages' row-major K scales for tcgen05.cp and un-swizzles
//                their Delta_S rows (idle otherwise; it also owns the tensor-memory allocation);
//   warp 1       Q K^T issuer: per block a rank-one BF16 MMA seeds S with 1 x Delta_S
//                (Eq. 11) and two block-scaled FP4 MMAs (K = 64 each) accumulate Q K^T into
//                the same TMEM columns, block c in score buffer c & 1;
//   warp 3       P V issuer: four FP8 MMAs per block (A = P_hat from TMEM, B = V from
//                shared memory, MN-major) accumulate P V into O;
//   warps 12-15  running row maximum (Algorithm 1 lines 11-12), one thread per row, into a shared-memory ring;
//   warps 4-7    exponentials of the even-numbered blocks of the traversal, warps 8-11 of the odd-numbered ones.  One
//                thread per row: the whole 128-column row in registers (so the score buffer is handed back before the
//                first exponential), mask, 2^(lam S - lam m), row sum from the unquantized P, P -> E4M3 at the fixed
//                scale 448 into the group's own 32 TMEM columns (lines 13-14);
//   warps 16-19  correction + epilogue: the rescale of O (Eq. 6, only when some row's maximum moved) and
//                O / (448 l) * v_scale as BF16 (line 17).
// Tensor memory (512 columns): S0 [0,128) S1 [128,256) O [256,384), P_hat0 [384,416) P_hat1 [416,448), scale factors of two
// query tiles [448,464) and of two K blocks [464,480).
//
// Why this split.  The exponentials bound a block: 128 x 128 of them take 1024 cycles of each SM quarter's special-function
// unit, 1130 with the conversions and stores around them (both exponent warps of a quarter together, alone on the SM; 1465 with
// maximum, rescale and MMAs beside them).  The maximum passes on a serial chain from block to block, and with both on the
// same thread (two groups that alternate over the blocks and hand the maximum to one another) the chain held up every item's
// first and last blocks and every causal diagonal.  Warps of their own run the chain ahead of the exponentials; the second
// reading of the scores costs 72 cycles of the tensor-memory port.  Two score buffers and one accumulator take the place of
// one and two.  Measured, the kernel alone (us, back to back), alternating groups / this as it is now: 256 keys x 1 head 11.3 / 7.4;
// 8 x 577 keys x 16 heads, not causal, 48.2 / 35.7; 4 x 777 x 8 heads 20.5 / 14.2; causal 1999 x 40 heads 61.4 / 51.2; 4096 x 32 133.8 /
// 117.8; 16384 x 32 1636 / 1558; 131072 x 32 96.8 / 97.2 ms (where the power limit sets the clock); chunks of 512 queries on
// pages 424 / 310; 16384 x 32 from pages 1782 / 1720.
// What must not be in the exponentials: one straight run of 128 took 1130 cycles where the same code with a mask test or a wait
// per 32 scores took 2200.
//
// Every mbarrier wait is bounded; on expiry the CTA raises MPFA_DEV_TIMEOUT in
// *device_status, all roles leave their loops, outstanding TMA copies are drained and
// tensor memory is released.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "common.cuh"
#include "sm100_ptx.cuh"
#include "prefill_common.cuh"

namespace mpfa {
namespace {

constexpr int KST = 4, VST = 4, MST = 8;   // stages: K, V, row maxima
constexpr int NTHREADS = 640;
// setmaxnreg only moves registers inside the pool the CTA got at launch (640 threads x the 96 registers of the launch bound); a
// request beyond the pool would block forever, so the split is checked here.
constexpr int LAUNCH_REGS = 96;
// exponentials / maxima / correction / utility.  The paged instance's producer and re-tiling warps need more, see below.
// Measured without runs (whole passes with stage 1, us; causal 1999 x 40 heads, 16384 x 32): short instance 144/48/80/64 75.7, 1625;
// 152/48/72/56 75.4, 1630; 144/64/80/48 76.3, 1640; 136/56/88/64 75.7, 1635.  Paged (chunks of 512): 152/48/72/56 423, 144/56/72/64
// 435, 144/64/80/48 427.  Less than 48 for the maxima or 72 for the correction spills heavily.
// With runs (RUNS; the kernel alone, us, 16384 x 32 / 131072 x 32 / chunks of 512 on pages / 16384 x 32 from pages): 144/56/88/48 1553,
// 96.6 ms, 310, 1720; 152/48/80/48 1556, 96.4 ms, 312, 1742; 144/48/88/56 1549, 97.0 ms, 315, 1737; 144/48/80/64 1564, 97.1 ms, 314,
// 1752; 152/48/72/56 1598, 96.7 ms, 318, 1771.
template <bool PAGED, bool LONG, bool RUNS> constexpr int REGS_EXP = RUNS ? (LONG && !PAGED ? 152 : 144) : (PAGED ? 152 : 144);
template <bool PAGED, bool LONG, bool RUNS> constexpr int REGS_MAX = RUNS ? (LONG && !PAGED ? 48 : 56) : (PAGED || !LONG ? 48 : 56);
template <bool PAGED, bool LONG, bool RUNS> constexpr int REGS_CORR = RUNS ? (LONG && !PAGED ? 80 : 88) : (PAGED || LONG ? 72 : 80);
template <bool PAGED, bool LONG, bool RUNS> constexpr int REGS_UTIL = RUNS ? 48 : (PAGED ? 56 : 64);
template <bool PAGED, bool LONG, bool RUNS>
constexpr bool regs_ok() {
  constexpr int e = REGS_EXP<PAGED, LONG, RUNS>, m = REGS_MAX<PAGED, LONG, RUNS>, c = REGS_CORR<PAGED, LONG, RUNS>, u = REGS_UTIL<PAGED, LONG, RUNS>;
  // the exponent warps take registers (setmaxnreg.inc: not below the launch's), the others give them back (setmaxnreg.dec: not
  // above the launch's, or the instruction is illegal)
  return 8 * e + 4 * (m + c + u) <= 20 * LAUNCH_REGS && e >= LAUNCH_REGS && m <= LAUNCH_REGS && c <= LAUNCH_REGS && u <= LAUNCH_REGS &&
         u >= 24 && e % 8 == 0 && m % 8 == 0 && c % 8 == 0 && u % 8 == 0;
}
static_assert(regs_ok<false, false, false>() && regs_ok<false, false, true>() && regs_ok<false, true, true>() && regs_ok<true, true, false>() &&
              regs_ok<true, true, true>(), "setmaxnreg split");

enum {
  BAR_Q_FULL = 0,                       // [2] query tile of work item i in buffer i & 1
  BAR_Q_EMPTY = 2,                      // [2] every Q K^T MMA of that work item has completed
  BAR_K_FULL = 4,
  BAR_K_EMPTY = BAR_K_FULL + KST,
  BAR_V_FULL = BAR_K_EMPTY + KST,
  BAR_V_EMPTY = BAR_V_FULL + VST,
  BAR_S_FULL = BAR_V_EMPTY + VST,       // [2] scores of block c in buffer c & 1
  BAR_S_EMPTY = BAR_S_FULL + 2,         // [2] the exponent warps have them in registers (the maximum was taken before)
  BAR_M_FULL = BAR_S_EMPTY + 2,         // [MST] running maximum after block c in slot c % MST.  The maximum warps are at most two
                                        //     blocks ahead of the exponent warps, and those (P_hat of block c needs P V of block
                                        //     c-2, which needs the correction warps) at most three ahead of the correction
                                        //     warps, whose hand-over of the accumulator for an item's first block comes
                                        //     before they read that block's maximum: a slot is never two phases ahead of a
                                        //     reader with five slots or more
  BAR_P_FULL = BAR_M_FULL + MST,        // [2] P_hat of block c written
  BAR_P_EMPTY = BAR_P_FULL + 2,         // [2] P V of block c has consumed P_hat
  BAR_O_FULL = BAR_P_EMPTY + 2,         // P V of block c accumulated into O
  BAR_O_READY = BAR_O_FULL + 1,         // O rescaled for block c (an item's first block: the previous item's output has been read)
  BAR_L_FULL = BAR_O_READY + 1,         // [4] row sums of the u-th item that has KV blocks (T > 0), slot u & 3.  The exponent
                                        //     warps can be at most three (one-block) such items ahead of the epilogue, so a
                                        //     slot is never two phases ahead of its reader.  Items without blocks stay out of
                                        //     the ring: nothing bounds how many of them those warps could run through
  BAR_SF_READY = BAR_L_FULL + 4,        // [KST] paged source only: scales and Delta_S of the stage re-tiled
  NUM_BARS = BAR_SF_READY + KST
};
static_assert(NUM_BARS <= 64, "barrier table");

// Contiguous operands: the most keys that the short instance takes (measured at the kernel: the shorter side's last clear gain)
constexpr int LONG_KEYS = 49152;

// RUNS: an item of RUN_BLOCKS KV blocks or more accumulates them in two runs, from 256 blocks in four.  The tensor core drops what
// does not fit behind the accumulator's last bit, so O comes out too small by an amount that grows with the number of additions
// into one accumulator.  Relative error of the FP32 result against a 64-bit recomputation (2-norm), in one run / in these / with the
// blocks alternating between two accumulators: causal 16384 keys 1.7e-6 / 1.1e-6 / 8.3e-7, 2048 queries on 65536 keys 4.0e-5 / 2.5e-5 /
// 2.9e-5, on 131072 keys 8.0e-5 / 6.0e-5 / 6.4e-5.  After a run the correction warps move O to shared memory (added to what is
// there, scaled to the present maximum), the next P V starts from zero, and the epilogue adds the sum of the earlier runs.  It costs
// (us, kernel alone, one run / these) 16384 x 32 heads 1539 / 1558, 131072 x 32 96.8 / 97.2 ms, chunks of 512 on pages 299 / 312.
// Shorter items stay in one run, within 8e-7.  (Runs from 16 blocks on would make 8.9e-7 of the 1.1e-6 above, but the pass over 1999
// keys x 40 heads 87.7 us instead of 82.4, the kernel alone 52.4 instead of 51.2: with the copy's 64 KB of shared memory its CTAs
// do not fit beside the last ones of stage 1.)  Launches that have no longer items take an instance without this code.
constexpr int RUN_BLOCKS = 32;
template <bool RUNS>
__device__ __forceinline__ int run_length(int T) { return !RUNS || T < RUN_BLOCKS ? T : T < 256 ? (T + 1) >> 1 : (T + 3) >> 2; }

constexpr uint32_t OFF_Q = 0;                              // 2 tiles (the next tile's queries are prefetched)
constexpr uint32_t OFF_K = OFF_Q + 2 * 8192;
constexpr uint32_t OFF_V = OFF_K + KST * 8192;
constexpr uint32_t OFF_DELTA = OFF_V + VST * 16384;
constexpr uint32_t OFF_ONES = OFF_DELTA + KST * 4096;
constexpr uint32_t OFF_SFQ = OFF_ONES + 4096;
constexpr uint32_t OFF_SFK = OFF_SFQ + 2 * 1024;
constexpr uint32_t OFF_M = OFF_SFK + KST * 1024;           // running maximum after block c, [c % MST][128]
constexpr uint32_t OFF_L = OFF_M + MST * 128 * 4;          // final (l, m) of the two exponent groups, [item & 3][2][2][128]
constexpr uint32_t OFF_BAR = OFF_L + 4 * 4 * 128 * 4;
constexpr uint32_t OFF_MISC = OFF_BAR + 64 * 8;            // tmem base, abort flag (NUM_BARS <= 64)
constexpr uint32_t OFF_TAIL = OFF_MISC + 128;              // what only some instances have
// paged source only: per K stage the two pages' scale bytes (2 x 512) and Delta_S rows (2 x 128) as stored; groups by length
constexpr uint32_t RAW_STAGE = 1280;
constexpr uint32_t OFF_RAW = OFF_TAIL;
constexpr uint32_t OFF_ORDER = OFF_RAW + KST * RAW_STAGE;
// O of the runs so far of an item's blocks, [32 groups of 4 columns][128 rows] x 16 bytes
template <bool PAGED> constexpr uint32_t OFF_RUN = PAGED ? OFF_ORDER + 2 * MAX_GROUPS : OFF_TAIL;
template <bool PAGED, bool RUNS>
constexpr uint32_t SMEM_BYTES = OFF_RUN<PAGED> + (RUNS ? HEAD_DIM * 128 * 4 : 0) + 1024;   // + slack for the 1024-byte alignment
static_assert(OFF_TAIL % 128 == 0 && OFF_RUN<true> % 16 == 0 && SMEM_BYTES<true, true> <= 227 * 1024, "shared memory");

constexpr uint32_t TM_S = 0 /* 2 x 128 */, TM_O = 256, TM_P = 384 /* 2 x 32 */, TM_SFQ = 448 /* 2 x 8 */, TM_SFK = 464 /* 2 x 8 */;
constexpr uint32_t TMEM_COLS = 512;

// Keeps every use of freshly loaded tensor-memory registers behind the wait that stands before it.
__device__ __forceinline__ void pin32(uint32_t (&r)[32]) {
  asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
                    "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]),
                    "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]),
                    "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31]));
}
__device__ __forceinline__ void pin16(uint32_t (&r)[16]) {
  asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
                    "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]));
}

// x += w * (16 columns of the copy in shared memory)
__device__ __forceinline__ void add_copy(uint32_t (&x)[16], const uint4 *copy, float w) {
#pragma unroll
  for (int i = 0; i < 16; i += 4) {
    const uint4 o = copy[(i >> 2) * 128];
    x[i] = __float_as_uint(__fmaf_rn(w, __uint_as_float(o.x), __uint_as_float(x[i])));
    x[i + 1] = __float_as_uint(__fmaf_rn(w, __uint_as_float(o.y), __uint_as_float(x[i + 1])));
    x[i + 2] = __float_as_uint(__fmaf_rn(w, __uint_as_float(o.z), __uint_as_float(x[i + 2])));
    x[i + 3] = __float_as_uint(__fmaf_rn(w, __uint_as_float(o.w), __uint_as_float(x[i + 3])));
  }
}

// last key that a query row sees.  Rows past a request's own query count take the last row's (the epilogue writes their zeros):
// with nothing visible they would have every block of their tile masked (8 requests x 612 queries on 1445 to 9983 tokens: 704 us
// that way, now 508).
template <bool PAGED>
__device__ __forceinline__ int last_key(const PrefillParams &p, const Tile &tl, int r_abs) {
  const int n_kv = PAGED ? tl.nkv : p.N_kv, n_q = PAGED ? tl.nq : p.N_q;
  return p.causal ? min(n_kv - 1, (PAGED ? min(r_abs, n_q - 1) : r_abs) + (n_kv - n_q)) : n_kv - 1;
}

__device__ __forceinline__ float exponent_unit(const PrefillParams &p, int b) {
  return __fmul_rn(__fmul_rn(__fmul_rn(p.softmax_scale, 1.4426950408889634f), p.q_gscale[b]), p.k_gscale[b]);
}

// LONG: who masks and how P_hat is stored.  false: the maximum warps write masked scores back to tensor memory, so the code of the
// exponentials has no mask in it (it is read by every pass and competes for the instruction cache with the other roles'), and
// P_hat goes out in one store.  true: the exponent warps mask, P_hat in two stores.  The arithmetic is the same.  Measured, the kernel
// alone, false / true (us): 8 x 577 keys x 16 heads, not causal, 35.5 / 37.9; causal 1999 x 40 50.6 / 53.4; 4096 x 32 117.6 / 126.9;
// 8192 x 32 413 / 437; 16384 x 32 1580 / 1629; 32768 x 32 5933 / 6002; 49152 x 32 13.54 / 13.71 ms; 57344 x 32 18.71 / 18.69; 65536 x 32 24.4 /
// 24.6; 131072 x 32 102.6 / 97.7.  Not causal: 32768 x 16 5.97 / 6.03 ms, 49152 x 8 6.67 / 6.70, 65536 x 8 11.90 / 11.83.  From pages the
// second form is ahead at every length (chunks of 512 on 4120 to 15011 tokens 314 / 310 us, 16384 x 32 1764 / 1720).  Neither
// result is explained beyond the compiler's schedules, which differ in every role: the rule is what was measured.
template <bool PAGED, bool LONG, bool RUNS>
__global__ void __launch_bounds__(NTHREADS, 1)
prefill_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
               const __grid_constant__ CUtensorMap tm_v, const PrefillParams p, const PagedSrc pg) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sbase = smem_u32(smem);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  Ctx cx;
  cx.bars = sbase + OFF_BAR;
  cx.abort_flag = reinterpret_cast<volatile int *>(smem + OFF_MISC + 4);
  cx.status = p.status;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + OFF_MISC);

  // ---- one-time setup
  launch_dependents();
  if (tid == 0) {
    *cx.abort_flag = 0;
    for (int i = 0; i < 2; ++i) { mbar_init(cx.bar(BAR_Q_FULL + i), 1); mbar_init(cx.bar(BAR_Q_EMPTY + i), 1); }
    for (int i = 0; i < KST; ++i) {
      mbar_init(cx.bar(BAR_K_FULL + i), 1);
      mbar_init(cx.bar(BAR_K_EMPTY + i), 1);
      mbar_init(cx.bar(BAR_SF_READY + i), 1);
    }
    for (int i = 0; i < VST; ++i) { mbar_init(cx.bar(BAR_V_FULL + i), 1); mbar_init(cx.bar(BAR_V_EMPTY + i), 1); }
    for (int i = 0; i < 2; ++i) {
      mbar_init(cx.bar(BAR_S_FULL + i), 1);
      mbar_init(cx.bar(BAR_S_EMPTY + i), 4);   // one arrival per warp (lane 0 after __syncwarp)
      mbar_init(cx.bar(BAR_P_FULL + i), 4);
      mbar_init(cx.bar(BAR_P_EMPTY + i), 1);
    }
    for (int i = 0; i < MST; ++i) mbar_init(cx.bar(BAR_M_FULL + i), 4);
    for (int i = 0; i < 4; ++i) mbar_init(cx.bar(BAR_L_FULL + i), 8);
    mbar_init(cx.bar(BAR_O_FULL), 1);
    mbar_init(cx.bar(BAR_O_READY), 4);
    mbar_init_fence();
    prefetch_tmap(&tm_q);
    if (!PAGED) {
      prefetch_tmap(&tm_k);
      prefetch_tmap(&tm_v);
    }
  }
  // rank-one operands: MN-major, 128B swizzle, K = 16.  Row k = 0 of each 64-element half
  // holds the data (ones / Delta_S), every other row stays zero for the CTA's lifetime.
  for (int i = tid; i < (KST * 4096 + 4096) / 16; i += NTHREADS)
    reinterpret_cast<uint4 *>(smem + OFF_DELTA)[i] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  if (tid < 128) reinterpret_cast<uint16_t *>(smem + OFF_ONES)[(tid >> 6) * 1024 + (tid & 63)] = 0x3F80;  // 1.0
  fence_proxy_async_smem();
  if (warp == 2) {
    tmem_alloc(smem_u32(tmem_slot), TMEM_COLS);
    tmem_relinquish();
  }
  // everything above touches this CTA only and overlaps the end of the preceding kernel; everything below reads memory
  grid_dependency_wait();
  const bool ordered = PAGED && p.B > 1 && p.B * p.nq_tiles <= MAX_GROUPS;
  if (ordered)   // the row-sum ring is not in use yet
    length_order(p, pg, reinterpret_cast<uint16_t *>(smem + OFF_L), reinterpret_cast<uint16_t *>(smem + OFF_ORDER), tid, NTHREADS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = *tmem_slot;
  const bool has_delta = p.delta != nullptr;   // operand of the seed MMA

  // Every role walks the same list of work items (q tile x q head) and keeps the same running count of
  // KV blocks; ring slots and barrier phases are functions of those two counters, so the pipeline runs
  // straight through item boundaries: the next item's Q/K/V arrive and its first scores are computed while
  // the correction warps write the previous item's output.
  TileWalk walk;
  walk.init(PAGED && ordered ? reinterpret_cast<const uint16_t *>(smem + OFF_ORDER) : nullptr);
  Tile tl;
  uint32_t gb = 0;   // KV blocks of the items already walked
  uint32_t ti = 0;   // index of the current item in this CTA's list

  if (warp < 4) setmaxnreg_dec<REGS_UTIL<PAGED, LONG, RUNS>>();
  if (warp == 0) {
    // =========================== TMA producer ===========================
    // The whole warp runs the loop (uniform control flow keeps addresses and barrier handles in
    // uniform registers); a single elected lane issues each copy.
    bool ok = true;
    uint32_t nk_armed = 0, nv_armed = 0, nq_armed = 0;
    for (; ok && walk.template next<PAGED>(p, pg, tl); gb += tl.T, ++ti) {
      const uint32_t qb = ti & 1;
      if (ti >= 2) ok = cx.wait(BAR_Q_EMPTY + qb, ((ti >> 1) - 1) & 1u);
      if (!ok) break;
      const size_t q_row = ((size_t)tl.b * p.H_q + tl.hq) * (size_t)(p.nq_tiles * TILE) + tl.row0;
      const size_t k_row = ((size_t)tl.b * p.H_kv + tl.hk) * (size_t)(p.nk_tiles * TILE);
      if (elect_one()) {
        mbar_expect_tx(cx.bar(BAR_Q_FULL + qb), 8192 + 1024);
        tma_load_2d(sbase + OFF_Q + qb * 8192, &tm_q, 0, (int)q_row, cx.bar(BAR_Q_FULL + qb));
        bulk_load(sbase + OFF_SFQ + qb * 1024, p.q_sf + (((size_t)tl.b * p.H_q + tl.hq) * p.nq_tiles + tl.qt) * 1024, 1024,
                  cx.bar(BAR_Q_FULL + qb));
      }
      nq_armed = ti + 1;
      PageLookup look;
      for (int t = 0; t < tl.T && ok; ++t) {
        const uint32_t c = gb + t;
        const int jb = tl.T - 1 - t;
        const uint32_t ks = c % KST, vs = c % VST;
        int page_lo = 0, page_hi = 0;
        if (PAGED) look.get(pg, p.status, tl.b, tl.nkv, t, jb, lane, page_lo, page_hi);
        if (c >= (uint32_t)KST) ok = cx.wait(BAR_K_EMPTY + ks, (c / KST - 1) & 1u);
        if (!ok) break;
        if (PAGED) {
          if (elect_one()) {
            const uint32_t bar = cx.bar(BAR_K_FULL + ks);
            mbar_expect_tx(bar, 8192 + 1024 + (has_delta ? 256 : 0));
            const size_t s_lo = (size_t)page_lo * p.H_kv + tl.hk, s_hi = (size_t)page_hi * p.H_kv + tl.hk;
            bulk_load(sbase + OFF_K + ks * 8192, pg.k_codes + s_lo * 4096, 4096, bar);
            bulk_load(sbase + OFF_K + ks * 8192 + 4096, pg.k_codes + s_hi * 4096, 4096, bar);
            bulk_load(sbase + OFF_RAW + ks * RAW_STAGE, pg.k_sf + s_lo * 512, 512, bar);
            bulk_load(sbase + OFF_RAW + ks * RAW_STAGE + 512, pg.k_sf + s_hi * 512, 512, bar);
            if (has_delta) {
              bulk_load(sbase + OFF_RAW + ks * RAW_STAGE + 1024, pg.delta + ((size_t)page_lo * p.H_q + tl.hq) * 64, 128, bar);
              bulk_load(sbase + OFF_RAW + ks * RAW_STAGE + 1152, pg.delta + ((size_t)page_hi * p.H_q + tl.hq) * 64, 128, bar);
            }
          }
        } else if (elect_one()) {
          mbar_expect_tx(cx.bar(BAR_K_FULL + ks), 8192 + 1024 + (has_delta ? 256 : 0));
          tma_load_2d(sbase + OFF_K + ks * 8192, &tm_k, 0, (int)(k_row + (size_t)jb * TILE), cx.bar(BAR_K_FULL + ks));
          bulk_load(sbase + OFF_SFK + ks * 1024, p.k_sf + (((size_t)tl.b * p.H_kv + tl.hk) * p.nk_tiles + jb) * 1024, 1024,
                    cx.bar(BAR_K_FULL + ks));
          if (has_delta) {
            const __nv_bfloat16 *d = p.delta + ((size_t)tl.b * p.H_q + tl.hq) * (size_t)(p.nk_tiles * TILE) + (size_t)jb * TILE;
            bulk_load(sbase + OFF_DELTA + ks * 4096, d, 128, cx.bar(BAR_K_FULL + ks));
            bulk_load(sbase + OFF_DELTA + ks * 4096 + 2048, d + 64, 128, cx.bar(BAR_K_FULL + ks));
          }
        }
        nk_armed = c + 1;
        if (c >= (uint32_t)VST) ok = cx.wait(BAR_V_EMPTY + vs, (c / VST - 1) & 1u);
        if (!ok) break;
        if (MPFA_DROP_V(c)) {
          // test build: this copy is left out on purpose
        } else if (PAGED) {
          if (elect_one()) {
            const uint32_t bar = cx.bar(BAR_V_FULL + vs);
            mbar_expect_tx(bar, 16384);
            bulk_load(sbase + OFF_V + vs * 16384, pg.v_fp8 + ((size_t)page_lo * p.H_kv + tl.hk) * 8192, 8192, bar);
            bulk_load(sbase + OFF_V + vs * 16384 + 8192, pg.v_fp8 + ((size_t)page_hi * p.H_kv + tl.hk) * 8192, 8192, bar);
          }
        } else if (elect_one()) {
          mbar_expect_tx(cx.bar(BAR_V_FULL + vs), 16384);
          tma_load_2d(sbase + OFF_V + vs * 16384, &tm_v, 0, (int)(k_row + (size_t)jb * TILE), cx.bar(BAR_V_FULL + vs));
        }
        if (!MPFA_DROP_V(c)) nv_armed = c + 1;
      }
    }
    if (*cx.abort_flag) {
      // Drain: copies still in flight must land before the CTA's shared memory is released.
      for (uint32_t c = nk_armed - min(nk_armed, (uint32_t)KST); c < nk_armed; ++c)
        mbar_wait_ns(cx.bar(BAR_K_FULL + c % KST), (c / KST) & 1u, WAIT_LIMIT_NS);
      for (uint32_t c = nv_armed - min(nv_armed, (uint32_t)VST); c < nv_armed; ++c)
        if (!MPFA_DROP_V(c)) mbar_wait_ns(cx.bar(BAR_V_FULL + c % VST), (c / VST) & 1u, WAIT_LIMIT_NS);
      for (uint32_t i = nq_armed - min(nq_armed, 2u); i < nq_armed; ++i)
        mbar_wait_ns(cx.bar(BAR_Q_FULL + (i & 1)), (i >> 1) & 1u, WAIT_LIMIT_NS);
    }
  } else if (warp == 1) {
    // =========================== Q K^T issuer ===========================
    // Whole warp in uniform control flow; lane 0 (always the elected lane of a full warp) issues
    // every tcgen05 instruction, so the commits track the MMAs of the same thread.
    // All shared-memory descriptors are built once; a ring stage or K step only adds a
    // constant to the 14-bit start-address field (shared addresses stay below 256 KB).
    const uint32_t id_fp4 = idesc_nvfp4(128, 128), id_bf16 = idesc_bf16(128, 128, 1, 1);
    const uint64_t d_ones = smem_desc(sbase + OFF_ONES, 2048, 1024, SWZ_128B);
    const uint64_t d_delta0 = smem_desc(sbase + OFF_DELTA, 2048, 1024, SWZ_128B);
    const uint64_t d_q00 = smem_desc(sbase + OFF_Q, 16, 512, SWZ_64B);
    const uint64_t d_k0 = smem_desc(sbase + OFF_K, 16, 512, SWZ_64B);
    const uint64_t d_sfq00 = smem_desc(sbase + OFF_SFQ, 0, 128, SWZ_NONE);
    const uint64_t d_sfk0 = smem_desc(sbase + OFF_SFK, 0, 128, SWZ_NONE);
    bool ok = true;
    for (; ok && walk.template next<PAGED>(p, pg, tl); gb += tl.T, ++ti) {
      const uint32_t qb = ti & 1;
      ok = cx.wait(BAR_Q_FULL + qb, (ti >> 1) & 1u);
      if (!ok) break;
      const uint64_t d_q0 = d_q00 + (uint64_t)((qb * 8192) >> 4);
      const uint32_t tSFQ = tm + TM_SFQ + qb * 8;
      tc_fence_after();
      if (elect_one()) {
        const uint64_t d_sfq0 = d_sfq00 + (uint64_t)((qb * 1024) >> 4);
        tmem_cp_32x128b_warpx4(tSFQ, d_sfq0);
        tmem_cp_32x128b_warpx4(tSFQ + 4, d_sfq0 + (512 >> 4));
      }
      for (int t = 0; t < tl.T && ok; ++t) {
        const uint32_t c = gb + t, ks = c % KST, sb = c & 1;
        ok = cx.wait(BAR_K_FULL + ks, (c / KST) & 1u);
        if (PAGED) ok = ok && cx.wait(BAR_SF_READY + ks, (c / KST) & 1u);
        if (c >= 2) ok = ok && cx.wait(BAR_S_EMPTY + sb, ((c >> 1) - 1) & 1u);
        if (!ok) break;
        const uint32_t tSFK = tm + TM_SFK + sb * 8, tS = tm + TM_S + sb * 128;
        const uint64_t d_sfk = d_sfk0 + (uint64_t)((ks * 1024) >> 4), d_k = d_k0 + (uint64_t)((ks * 8192) >> 4);
        const uint64_t d_delta = d_delta0 + (uint64_t)((ks * 4096) >> 4);
        tc_fence_after();
        if (elect_one()) {
          tmem_cp_32x128b_warpx4(tSFK, d_sfk);
          tmem_cp_32x128b_warpx4(tSFK + 4, d_sfk + (512 >> 4));
          if (has_delta) mma_bf16_ss(tS, d_ones, d_delta, id_bf16, 0);
          mma_nvfp4_ss(tS, d_q0, d_k, id_fp4, tSFQ, tSFK, has_delta ? 1u : 0u);
          mma_nvfp4_ss(tS, d_q0 + (32 >> 4), d_k + (32 >> 4), id_fp4, tSFQ + 4, tSFK + 4, 1u);
          mma_commit(cx.bar(BAR_S_FULL + sb));
          mma_commit(cx.bar(BAR_K_EMPTY + ks));
        }
      }
      if (ok && elect_one()) mma_commit(cx.bar(BAR_Q_EMPTY + qb));   // after every MMA that reads this query tile
      __syncwarp();
    }
  } else if (PAGED && warp == 2) {
    // ==== paged source: re-tile the K scales and un-swizzle Delta_S of every stage ====
    const int G = p.H_q / p.H_kv;
    bool ok = true;
    for (; ok && walk.template next<PAGED>(p, pg, tl); gb += tl.T, ++ti) {
      const int rsw = tl.hq % G;
      for (int t = 0; t < tl.T && ok; ++t) {
        const uint32_t c = gb + t;
        const uint32_t ks = c % KST;
        ok = cx.wait(BAR_K_FULL + ks, (c / KST) & 1u);
        if (!ok) break;
        const uint8_t *raw = smem + OFF_RAW + ks * RAW_STAGE;
        // scales: row-major [key][8] -> the 32x128b tile layout tcgen05.cp expects (lane = key mod 32)
        uint2 v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = *reinterpret_cast<const uint2 *>(raw + (q >> 1) * 512 + ((q & 1) * 32 + lane) * 8);
        uint8_t *dst = smem + OFF_SFK + ks * 1024 + lane * 16;
        *reinterpret_cast<uint4 *>(dst) = make_uint4(v[0].x, v[1].x, v[2].x, v[3].x);
        *reinterpret_cast<uint4 *>(dst + 512) = make_uint4(v[0].y, v[1].y, v[2].y, v[3].y);
        // Delta_S: 16-byte group c of a page is stored at c ^ (q head mod G); row 0 of the operand wants them in order
        if (has_delta && lane < 16) {
          const int half = lane >> 3, cg = lane & 7;
          const uint4 d = *reinterpret_cast<const uint4 *>(raw + 1024 + half * 128 + ((cg ^ rsw) << 4));
          *reinterpret_cast<uint4 *>(smem + OFF_DELTA + ks * 4096 + half * 2048 + (cg << 4)) = d;
        }
        fence_proxy_async_smem();
        warp_arrive(cx.bar(BAR_SF_READY + ks), lane);
      }
    }
  } else if (warp == 3) {
    // =========================== P V issuer ===========================
    const uint32_t id_fp8 = idesc_e4m3(128, 128, 0, 1);
    const uint64_t d_v0 = smem_desc(sbase + OFF_V, 16, 1024, SWZ_128B);
    bool ok = true;
    for (; ok && walk.template next<PAGED>(p, pg, tl); gb += tl.T, ++ti) {
      const int run = run_length<RUNS>(tl.T);
      int begin = 0;   // of the run
      for (int t = 0; t < tl.T && ok; ++t) {
        const uint32_t c = gb + t, sb = c & 1, vs = c % VST;
        ok = cx.wait(BAR_V_FULL + vs, (c / VST) & 1u);
        ok = ok && cx.wait(BAR_P_FULL + sb, (c >> 1) & 1u);
        ok = ok && cx.wait(BAR_O_READY, c & 1u);
        if (!ok) break;
        tc_fence_after();
        const uint32_t tP = tm + TM_P + sb * 32;
        const uint64_t d_v = d_v0 + (uint64_t)((vs * 16384) >> 4);
        if (RUNS && t == begin + run) begin = t;
        if (elect_one()) {
#pragma unroll
          for (int k4 = 0; k4 < 4; ++k4)
            mma_e4m3_ts(tm + TM_O, tP + 8 * k4, d_v + (uint64_t)((4096 * k4) >> 4), id_fp8, ((RUNS ? t != begin : t > 0) || k4 > 0) ? 1u : 0u);
          mma_commit(cx.bar(BAR_O_FULL));
          mma_commit(cx.bar(BAR_P_EMPTY + sb));
          mma_commit(cx.bar(BAR_V_EMPTY + vs));
        }
      }
    }
  } else if (warp >= 12 && warp < 16) {
    // =========================== running maximum ===========================
    setmaxnreg_dec<REGS_MAX<PAGED, LONG, RUNS>>();
    const int row = (warp & 3) * 32 + lane;
    const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
    float *s_m = reinterpret_cast<float *>(smem + OFF_M);
    bool ok = true;
    for (; ok && walk.template next<PAGED>(p, pg, tl); gb += tl.T, ++ti) {
      const int limit = last_key<PAGED>(p, tl, tl.row0 + row);
      float m = -INFINITY;
      for (int t = 0; t < tl.T; ++t) {
        const uint32_t c = gb + t;
        const int key0 = (tl.T - 1 - t) * TILE;
        const uint32_t tS = tm + TM_S + (c & 1) * 128 + lane_off;
        if (!__all_sync(0xffffffffu, cx.wait(BAR_S_FULL + (c & 1), (c >> 1) & 1u))) { ok = false; break; }
        tc_fence_after();
        float mx[4] = {m, -INFINITY, -INFINITY, -INFINITY};
        bool ragged = key0 + TILE - 1 > limit;
        if (!LONG) ragged = __any_sync(0xffffffffu, ragged);   // the stores below are the whole warp's
#pragma unroll 1
        for (int c0 = 0; c0 < 128; c0 += 32) {
          uint32_t x[32];
          tmem_ld32(tS + c0, x);
          tmem_ld_wait();
          pin32(x);
          if (ragged) {   // diagonal / ragged block only
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (key0 + c0 + i > limit) x[i] = 0xFF800000u;   // -inf
            if (!LONG) tmem_st32(tS + c0, x);
          }
#pragma unroll
          for (int i = 0; i < 32; i += 8) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
              mx[j] = max3(mx[j], __uint_as_float(x[i + 2 * j]), __uint_as_float(x[i + 2 * j + 1]));
          }
        }
        m = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
        s_m[(c % MST) * 128 + row] = m;
        if (!LONG && ragged) tmem_st_wait();
        tc_fence_before();
        warp_arrive(cx.bar(BAR_M_FULL + c % MST), lane);
      }
    }
  } else if (warp >= 4 && warp < 12) {
    // =========================== exponentials ===========================
    setmaxnreg_inc<REGS_EXP<PAGED, LONG, RUNS>>();
    const int grp = (warp - 4) >> 2;   // takes the KV blocks whose running count has this parity
    const int row = (warp & 3) * 32 + lane;
    const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
    const float *s_m = reinterpret_cast<const float *>(smem + OFF_M);
    const uint32_t tS = tm + TM_S + grp * 128 + lane_off, tP = tm + TM_P + grp * 32 + lane_off;
    bool ok = true;
    uint32_t n_used = 0;   // items so far with T > 0: only those go through the row-sum ring
    for (; ok && walk.template next<PAGED>(p, pg, tl); gb += tl.T, ++ti) {
      const int TT = tl.T;
      if (TT == 0) continue;   // nothing to attend to: the epilogue writes zeros without waiting for this role
      const int limit = last_key<PAGED>(p, tl, tl.row0 + row);
      const float lam = exponent_unit(p, tl.b);
      float m_own = -INFINITY;   // running maximum after this group's previous block
      float l_own = 0.0f;        // sum of 448 P over this group's blocks, relative to m_own
      for (int t = (grp ^ (int)gb) & 1; t < TT; t += 2) {
        const uint32_t c = gb + t;
        const int key0 = (TT - 1 - t) * TILE;
        // both of the block's conditions in one vote: the maximum is there, P V of block c-2 has consumed the group's P_hat
        const uint32_t par_m = (c / MST) & 1u, par_pe = ((c >> 1) - 1) & 1u;
        const bool both = cx.probe(BAR_M_FULL + c % MST, par_m) & (c < 2 || cx.probe(BAR_P_EMPTY + grp, par_pe));
        if (!__all_sync(0xffffffffu, both)) {
          bool w = cx.wait(BAR_M_FULL + c % MST, par_m);
          if (c >= 2) w = w && cx.wait(BAR_P_EMPTY + grp, par_pe);
          if (!__all_sync(0xffffffffu, w)) { ok = false; break; }
        }
        tc_fence_after();
        uint32_t s[4][32];
#pragma unroll
        for (int i = 0; i < 4; ++i) tmem_ld32(tS + 32 * i, s[i]);
        const float m_t = s_m[(c % MST) * 128 + row];
        const float a_own = (m_t == m_own) ? 1.0f : ex2_approx(__fmul_rn(m_own - m_t, lam));
        // P = 2^(lam S - lam m) (Eq. 4)
        // the factor 448 of the E4M3 operand is folded into the exponent: q = 448 P = 2^(lam S - lam m + log2 448); the row
        // sum is taken over q and the factor is divided out once in the epilogue
        const float cc = (m_t == -INFINITY) ? 0.0f : __fsub_rn(8.8073549220576042f, __fmul_rn(m_t, lam));
        m_own = m_t;
        tmem_ld_wait();
        pin32(s[0]), pin32(s[1]), pin32(s[2]), pin32(s[3]);
        tc_fence_before();
        warp_arrive(cx.bar(BAR_S_EMPTY + grp), lane);
        if (LONG && key0 + TILE - 1 > limit) {
#pragma unroll
          for (int i = 0; i < 128; ++i)
            if (key0 + i > limit) s[i >> 5][i & 31] = 0xFF800000u;
        }
        uint32_t packed[2][16];
        float sum[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int c0 = 0; c0 < 4; ++c0) {
          uint32_t(&x)[32] = s[c0];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            float x0, x1, x2, x3;
            fma2(x0, x1, __uint_as_float(x[4 * i]), __uint_as_float(x[4 * i + 1]), lam, cc);
            fma2(x2, x3, __uint_as_float(x[4 * i + 2]), __uint_as_float(x[4 * i + 3]), lam, cc);
            const float q0 = ex2_approx(x0), q1 = ex2_approx(x1), q2 = ex2_approx(x2), q3 = ex2_approx(x3);
            acc2(sum[0], sum[1], q0, q1);
            acc2(sum[2], sum[3], q2, q3);
            // two conversions written into the halves of one register (no separate merge instruction)
            asm("{.reg .b16 lo, hi;\n\t"
                "cvt.rn.satfinite.e4m3x2.f32 lo, %2, %1;\n\t"
                "cvt.rn.satfinite.e4m3x2.f32 hi, %4, %3;\n\t"
                "mov.b32 %0, {lo, hi};}"
                : "=r"(packed[c0 >> 1][8 * (c0 & 1) + i])
                : "f"(q0), "f"(q1), "f"(q2), "f"(q3));
          }
          if (LONG && (c0 & 1)) tmem_st16(tP + 8 * (c0 - 1), packed[c0 >> 1]);
        }
        if (!LONG) tmem_st32(tP, reinterpret_cast<uint32_t(&)[32]>(packed));
        l_own = __fadd_rn(__fmul_rn(a_own, l_own), (sum[0] + sum[1]) + (sum[2] + sum[3]));
        tmem_st_wait();
        tc_fence_before();
        warp_arrive(cx.bar(BAR_P_FULL + grp), lane);
      }
      if (!ok) break;
      float *s_fin = reinterpret_cast<float *>(smem + OFF_L) + (n_used & 3) * 512;
      s_fin[(grp * 2 + 0) * 128 + row] = l_own;
      s_fin[(grp * 2 + 1) * 128 + row] = m_own;
      warp_arrive(cx.bar(BAR_L_FULL + (n_used & 3)), lane);
      ++n_used;
    }
  } else if (warp >= 16) {
    // =========================== correction + epilogue ===========================
    setmaxnreg_dec<REGS_CORR<PAGED, LONG, RUNS>>();
    const int row = (warp & 3) * 32 + lane;
    const float *s_m = reinterpret_cast<const float *>(smem + OFF_M);
    uint4 *const s_run = reinterpret_cast<uint4 *>(smem + OFF_RUN<PAGED>) + row;   // this thread's row: written and read by it alone
    const uint32_t tO = tm + TM_O + ((uint32_t)((warp & 3) * 32) << 16);
    bool ok = true;
    uint32_t n_used = 0;   // items so far with T > 0 (slot and phase of the row-sum ring)
    warp_arrive(cx.bar(BAR_O_READY), lane);
    for (; walk.template next<PAGED>(p, pg, tl); gb += tl.T, ++ti) {
      const int TT = tl.T, r_abs = tl.row0 + row;
      const float lam = exponent_unit(p, tl.b);
      const bool past = PAGED && r_abs >= tl.nq;   // nobody reads these rows: they ask for no rescale
      float m_before = -INFINITY, m_run = -INFINITY;
      int t = 0, end = run_length<RUNS>(TT);
      for (;;) {   // the item's runs of blocks
        for (const int first = t; ok && t < end; ++t) {
          const uint32_t c = gb + t;
          ok = __all_sync(0xffffffffu, cx.wait(BAR_M_FULL + c % MST, (c / MST) & 1u));
          if (!ok) break;
          // alpha_t = 2^(lam (m_{t-1} - m_t)) (Eq. 5/6)
          const float m_now = s_m[(c % MST) * 128 + row];
          const float alpha = (m_now == m_before || past) ? 1.0f : ex2_approx(__fmul_rn(m_before - m_now, lam));
          m_before = m_now;
          if (t == first) continue;   // handed over by the previous item's epilogue, or when the run before was copied
          ok = __all_sync(0xffffffffu, cx.wait(BAR_O_FULL, (c - 1) & 1u));
          if (!ok) break;
          tc_fence_after();
          if (__any_sync(0xffffffffu, alpha != 1.0f)) {   // identical result when every factor is exactly 1
            // 16 columns on the way while 16 are multiplied, in a short loop: unrolled over 32-column halves the rescale took
            // 260-495 cycles instead of 590-770, but the kernel 1780 us instead of 1715 (16384 keys): the exponentials beside it
            // ran slower
            uint32_t r[2][16];
            tmem_ld16(tO, r[0]);
#pragma unroll 1
            for (int c0 = 0; c0 < 8; c0 += 2) {
#pragma unroll
              for (int u = 0; u < 2; ++u) {
                uint32_t(&x)[16] = r[u];
                tmem_ld_wait();
                pin16(x);
                if (c0 + u < 7) tmem_ld16(tO + 16 * (c0 + u + 1), r[u ^ 1]);
#pragma unroll
                for (int i = 0; i < 16; i += 2) {
                  float y0, y1;
                  mul2(y0, y1, __uint_as_float(x[i]), __uint_as_float(x[i + 1]), alpha);
                  x[i] = __float_as_uint(y0), x[i + 1] = __float_as_uint(y1);
                }
                tmem_st16(tO + 16 * (c0 + u), x);
              }
            }
            tmem_st_wait();
          }
          tc_fence_before();
          warp_arrive(cx.bar(BAR_O_READY), lane);
        }
        if (!RUNS || end == TT || !ok) break;
        // the run's O goes to shared memory, the first as it is, a later one added to the sum of those before
        ok = __all_sync(0xffffffffu, cx.wait(BAR_O_FULL, (gb + end - 1) & 1u));
        if (!ok) break;
        tc_fence_after();
        const bool more = end > run_length<RUNS>(TT);
        const float w = m_run == m_before ? 1.0f : ex2_approx(__fmul_rn(m_run - m_before, lam));
        m_run = m_before;
#pragma unroll 1
        for (int c0 = 0; c0 < HEAD_DIM; c0 += 16) {
          uint32_t x[16];
          tmem_ld16(tO + c0, x);
          tmem_ld_wait();
          pin16(x);
          if (more) add_copy(x, s_run + c0 / 4 * 128, w);
#pragma unroll
          for (int i = 0; i < 4; ++i) s_run[(c0 / 4 + i) * 128] = make_uint4(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]);
        }
        tc_fence_before();
        warp_arrive(cx.bar(BAR_O_READY), lane);
        end = min(end + run_length<RUNS>(TT), TT);
      }
      // final normalisation (Algorithm 1 line 17).  The two exponent groups hold partial sums relative to their own last
      // maximum; bring both to the final one.
      float l = 0.0f, w_run = 0.0f;
      if (ok && TT > 0) {
        ok = cx.wait(BAR_O_FULL, (gb + TT - 1) & 1u);
        ok = ok && cx.wait(BAR_L_FULL + (n_used & 3), (n_used >> 2) & 1u);
        tc_fence_after();
        if (ok) {
          const float *s_fin = reinterpret_cast<const float *>(smem + OFF_L) + (n_used & 3) * 512;
          const float l0 = s_fin[0 * 128 + row], m0 = s_fin[1 * 128 + row];
          const float l1 = s_fin[2 * 128 + row], m1 = s_fin[3 * 128 + row];
          const float mf = fmaxf(m0, m1);
          if (mf != -INFINITY && !past) {
            const float w0 = (m0 == mf) ? 1.0f : ex2_approx(__fmul_rn(m0 - mf, lam));
            const float w1 = (m1 == mf) ? 1.0f : ex2_approx(__fmul_rn(m1 - mf, lam));
            l = __fadd_rn(__fmul_rn(w0, l0), __fmul_rn(w1, l1));
            if (RUNS) w_run = (m_run == mf) ? 1.0f : ex2_approx(__fmul_rn(m_run - mf, lam));
          }
        }
      }
      // tcgen05.ld is warp-collective: every lane loads, only the stores are predicated.
      const bool warp_ok = __all_sync(0xffffffffu, ok);
      const bool store = r_abs < p.N_q && (warp_ok || TT == 0);
      const size_t o_off = (((size_t)tl.b * p.N_q + (store ? r_abs : 0)) * p.H_q + tl.hq) * HEAD_DIM;
      // one IEEE reciprocal per row; 128 divisions per thread would cost more than ten KV blocks
      const float inv_denom = (l > 0.0f) ? __frcp_rn(l) : 0.0f;
#pragma unroll 1
      for (int c0 = 0; c0 < HEAD_DIM; c0 += 16) {
        uint32_t r[16];
        if (TT > 0 && warp_ok) {
          tmem_ld16(tO + c0, r);
          tmem_ld_wait();
          pin16(r);
        }
        if (RUNS && TT >= RUN_BLOCKS) add_copy(r, s_run + c0 / 4 * 128, w_run);
        if (c0 == HEAD_DIM - 16 && TT > 0) {   // O is in registers: the next item's P V may overwrite it
          tc_fence_before();
          warp_arrive(cx.bar(BAR_O_READY), lane);
        }
#pragma unroll
        for (int i = 0; i < 16; ++i)
          r[i] = (l > 0.0f) ? __float_as_uint(__fmul_rn(__fmul_rn(__uint_as_float(r[i]), inv_denom), p.v_scale)) : 0u;
        if (store) {
          if (p.out_f32) {
#pragma unroll
            for (int i = 0; i < 16; i += 4)
              *reinterpret_cast<uint4 *>(p.out_f32 + o_off + c0 + i) = make_uint4(r[i], r[i + 1], r[i + 2], r[i + 3]);
          }
#pragma unroll
          for (int i = 0; i < 16; i += 8) {
            uint32_t h[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              __nv_bfloat162 v = __floats2bfloat162_rn(__uint_as_float(r[i + 2 * j]), __uint_as_float(r[i + 2 * j + 1]));
              h[j] = *reinterpret_cast<uint32_t *>(&v);
            }
            *reinterpret_cast<uint4 *>(p.out + o_off + c0 + i) = make_uint4(h[0], h[1], h[2], h[3]);
          }
        }
      }
      if (TT > 0) ++n_used;
      if (!ok) break;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 2) tmem_dealloc(tm, TMEM_COLS);
}
}  // namespace
}  // namespace mpfa

using namespace mpfa;

// 0: one query tile per CTA (the faster one on B200, see
// prefill_pair.cu's header for the measured comparison); 1: two query tiles per CTA (prefill_pair.cu)
static int g_arrangement = 0;
extern "C" int mpfa_set_prefill_arrangement(int a) {
  if (a != 0 && a != 1) return MPFA_ERR_INVALID_ARG;
  g_arrangement = a;
  return MPFA_OK;
}

extern "C" mpfa_status mpfa_prefill(const mpfa_fp4_tensor *q, const mpfa_fp4_tensor *k, const uint8_t *v_fp8,
                                    const void *delta_s_bf16, const mpfa_stats *st, float v_scale, int causal,
                                    float softmax_scale, void *out_bf16, float *out_f32, int32_t *device_status,
                                    void *stream) {
  return mpfa_prefill_variant(q, k, v_fp8, delta_s_bf16, st, v_scale, causal, softmax_scale, 0, out_bf16, out_f32,
                              device_status, stream);
}

extern "C" mpfa_status mpfa_prefill_variant(const mpfa_fp4_tensor *q, const mpfa_fp4_tensor *k, const uint8_t *v_fp8,
                                            const void *delta_s_bf16, const mpfa_stats *st, float v_scale, int causal,
                                            float softmax_scale, int variant, void *out_bf16, float *out_f32,
                                            int32_t *device_status, void *stream) {
  if (variant != 0 && variant != MPFA_VARIANT_COMP_ELEMENTWISE && variant != MPFA_VARIANT_PV_BF16 && variant != MPFA_VARIANT_PV_FP4)
    return MPFA_ERR_INVALID_ARG;
  const bool ew = variant == MPFA_VARIANT_COMP_ELEMENTWISE && delta_s_bf16 != nullptr;
  if (!q || !k || !v_fp8 || !st || !out_bf16 || !device_status) return MPFA_ERR_INVALID_ARG;
  if (!q->codes || !q->sf || !k->codes || !k->sf || !st->q_gscale || !st->k_gscale) return MPFA_ERR_INVALID_ARG;
  if (q->B <= 0 || q->B != k->B || q->H <= 0 || k->H <= 0 || q->N <= 0 || k->N <= 0) return MPFA_ERR_INVALID_ARG;
  if (!(softmax_scale > 0.0f) || !(v_scale > 0.0f)) return MPFA_ERR_INVALID_ARG;
  if (q->H % k->H != 0 || q->H / k->H > 8) return MPFA_ERR_UNSUPPORTED;
  if (!aligned(q->codes, 1024) || !aligned(k->codes, 1024) || !aligned(q->sf, 1024) || !aligned(k->sf, 1024) ||
      !aligned(v_fp8, 1024) || !aligned(delta_s_bf16, 256) || !aligned(out_bf16, 16) || !aligned(out_f32, 16))
    return MPFA_ERR_ALIGNMENT;
  const int nq_tiles = pad128(q->N) / TILE, nk_tiles = pad128(k->N) / TILE;
  const uint64_t q_rows = (uint64_t)q->B * q->H * nq_tiles * TILE, k_rows = (uint64_t)k->B * k->H * nk_tiles * TILE;
  if (q_rows >= (1ull << 31) || k_rows >= (1ull << 31)) return MPFA_ERR_UNSUPPORTED;
  const uint64_t n_cta = (uint64_t)q->B * q->H * nq_tiles;
  if (n_cta >= (1ull << 31)) return MPFA_ERR_UNSUPPORTED;
  int dev = 0, n_sm = 0;
  mpfa_status rc = device_info(&dev, &n_sm);
  if (rc != MPFA_OK) return rc;
  PrefillParams p;
  p.q_sf = q->sf;
  p.k_sf = k->sf;
  p.delta = static_cast<const __nv_bfloat16 *>(delta_s_bf16);
  p.q_gscale = st->q_gscale;
  p.k_gscale = st->k_gscale;
  p.out = static_cast<__nv_bfloat16 *>(out_bf16);
  p.out_f32 = out_f32;
  p.status = device_status;
  p.B = q->B;
  p.N_q = q->N;
  p.N_kv = k->N;
  p.H_q = q->H;
  p.H_kv = k->H;
  p.nq_tiles = nq_tiles;
  p.nk_tiles = nk_tiles;
  p.causal = causal ? 1 : 0;
  p.softmax_scale = softmax_scale;
  p.v_scale = v_scale;
  p.n_items = (int)n_cta;
  const unsigned grid = (unsigned)(n_cta < (uint64_t)n_sm ? n_cta : (uint64_t)n_sm);   // one persistent CTA per SM
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const bool other_pv = variant == MPFA_VARIANT_PV_BF16 || variant == MPFA_VARIANT_PV_FP4;
  if (g_arrangement == 1 && !other_pv) return launch_prefill_pair(q, k, v_fp8, p, ew, s);
  if (ew || other_pv) return launch_prefill_variant(q, k, v_fp8, p, variant, grid, s);
  EncodeTiledFn enc;
  rc = get_encoder(&enc);
  if (rc != MPFA_OK) return rc;
  CUtensorMap tq, tk, tv;
  if ((rc = make_map(enc, &tq, q->codes, q_rows, 64)) != MPFA_OK) return rc;
  if ((rc = make_map(enc, &tk, k->codes, k_rows, 64)) != MPFA_OK) return rc;
  if ((rc = make_map(enc, &tv, v_fp8, k_rows, 128)) != MPFA_OK) return rc;
  if (nk_tiles < RUN_BLOCKS) return start<prefill_kernel<false, false, false>, SMEM_BYTES<false, false>>(grid, NTHREADS, s, tq, tk, tv, p, PagedSrc{});
  if (k->N <= LONG_KEYS) return start<prefill_kernel<false, false, true>, SMEM_BYTES<false, true>>(grid, NTHREADS, s, tq, tk, tv, p, PagedSrc{});
  return start<prefill_kernel<false, true, true>, SMEM_BYTES<false, true>>(grid, NTHREADS, s, tq, tk, tv, p, PagedSrc{});
}

extern "C" mpfa_status mpfa_prefill_paged(const mpfa_fp4_tensor *q, const mpfa_paged_kv *kv, const int32_t *page_table,
                                          int max_pages_per_req, const int32_t *seq_lens, const int32_t *q_lens,
                                          const mpfa_stats *st,
                                          float v_scale, float softmax_scale, void *out_bf16, float *out_f32,
                                          int32_t *device_status, void *stream) {
  if (!q || !kv || !page_table || !seq_lens || !st || !out_bf16 || !device_status) return MPFA_ERR_INVALID_ARG;
  if (!q->codes || !q->sf || !kv->k_codes || !kv->k_sf || !kv->v_fp8 || !st->q_gscale || !st->k_gscale)
    return MPFA_ERR_INVALID_ARG;
  if (q->B <= 0 || q->H <= 0 || q->N <= 0 || kv->num_pages <= 0 || max_pages_per_req <= 0) return MPFA_ERR_INVALID_ARG;
  if (q->H != kv->H_q || kv->H_kv <= 0) return MPFA_ERR_INVALID_ARG;
  if (!(softmax_scale > 0.0f) || !(v_scale > 0.0f)) return MPFA_ERR_INVALID_ARG;
  if (kv->page_size != 64 || q->H % kv->H_kv != 0 || q->H / kv->H_kv > 8) return MPFA_ERR_UNSUPPORTED;
  if (!aligned(q->codes, 1024) || !aligned(q->sf, 1024) || !aligned(kv->k_codes, 256) || !aligned(kv->k_sf, 256) ||
      !aligned(kv->v_fp8, 256) || !aligned(kv->delta_s_bf16, 256) || !aligned(out_bf16, 16) || !aligned(out_f32, 16))
    return MPFA_ERR_ALIGNMENT;
  const int nq_tiles = pad128(q->N) / TILE;
  const uint64_t q_rows = (uint64_t)q->B * q->H * nq_tiles * TILE;
  if (q_rows >= (1ull << 31)) return MPFA_ERR_UNSUPPORTED;
  const uint64_t n_cta = (uint64_t)q->B * q->H * nq_tiles;
  int dev = 0, n_sm = 0;
  mpfa_status rc = device_info(&dev, &n_sm);
  if (rc != MPFA_OK) return rc;
  PrefillParams p;
  p.q_sf = q->sf;
  p.k_sf = nullptr;
  p.delta = static_cast<const __nv_bfloat16 *>(kv->delta_s_bf16);   // the kernel only tests it against null
  p.q_gscale = st->q_gscale;
  p.k_gscale = st->k_gscale;
  p.out = static_cast<__nv_bfloat16 *>(out_bf16);
  p.out_f32 = out_f32;
  p.status = device_status;
  p.B = q->B;
  p.N_q = q->N;
  p.N_kv = 0;
  p.H_q = q->H;
  p.H_kv = kv->H_kv;
  p.nq_tiles = nq_tiles;
  p.nk_tiles = 0;
  p.causal = 1;
  p.softmax_scale = softmax_scale;
  p.v_scale = v_scale;
  p.n_items = (int)n_cta;
  PagedSrc pg;
  pg.k_codes = kv->k_codes;
  pg.k_sf = kv->k_sf;
  pg.v_fp8 = kv->v_fp8;
  pg.delta = static_cast<const __nv_bfloat16 *>(kv->delta_s_bf16);
  pg.page_table = page_table;
  pg.seq_lens = seq_lens;
  pg.q_lens = q_lens;
  pg.max_pages = max_pages_per_req;
  pg.num_pages = kv->num_pages;
  if (g_arrangement == 1) return launch_prefill_pair_paged(q, p, pg, static_cast<cudaStream_t>(stream));
  EncodeTiledFn enc;
  rc = get_encoder(&enc);
  if (rc != MPFA_OK) return rc;
  CUtensorMap tq;
  if ((rc = make_map(enc, &tq, q->codes, q_rows, 64)) != MPFA_OK) return rc;
  const unsigned grid = (unsigned)(n_cta < (uint64_t)n_sm ? n_cta : (uint64_t)n_sm);
  if (max_pages_per_req < RUN_BLOCKS * (TILE / PAGE) - 1)   // no request can have RUN_BLOCKS blocks
    return start<prefill_kernel<true, true, false>, SMEM_BYTES<true, false>>(grid, NTHREADS, static_cast<cudaStream_t>(stream), tq, tq, tq, p, pg);
  return start<prefill_kernel<true, true, true>, SMEM_BYTES<true, true>>(grid, NTHREADS, static_cast<cudaStream_t>(stream), tq, tq, tq, p, pg);
}
