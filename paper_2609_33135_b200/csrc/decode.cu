// QK4PV8 decode over a paged low-bit KV cache (Section 5.3) for sm_100a.
//
// The path is bound by streaming the cache from HBM (200 bytes per token and kv head plus
// 2 of Delta_S per q head), so the kernel is a persistent streaming pipeline: one CTA per SM walks a list of
// (request, kv head, 1024-token partition) work items, and a producer warp keeps two rings of
// 128-key blocks in flight with bulk asynchronous copies: a K ring (codes, block scales,
// Delta_S) that runs one item AHEAD of a V ring.  The cache's physical byte order
// (include/mpfa.h) is the swizzled shared-memory image the tensor-core descriptors read, so a
// page needs one copy per tensor and no thread touches the bytes.
//
// The problem is transposed so that the long axis is the MMA's M dimension and the GQA group
// (Section 5.3 packs it into one MMA tile) is the N dimension, padded to 16:
//   S^T[key, head] = K Q^T       tcgen05.mma kind::mxf4nvf4 (E2M1 codes, UE4M3 block scales),
//                                M = 128 keys, N = 16, K = 2 x 64 channels, FP32 in TMEM,
//                                one 16-column slot per block of the item;
//   softmax        one thread per key.  As each S^T lands: + Delta_S (Eq. 11), warp maximum.
//                  After the item's last block one exchange gives every block u the running
//                  maximum m_u of the reverse traversal (max over the blocks visited so far),
//                  then P = 2^(lam S - lam m_u), P_hat = E4M3(448 P) for all blocks at once,
//                  written to shared memory as the B operands of the PV MMAs;
//   O_u^T[ch, head] = V_u^T P_hat_u^T   tcgen05.mma kind::f8f6f4, M = 128 channels, N = 16,
//                                K = 4 x 32 keys, V read MN-major straight from the ring, one
//                                accumulator slot per block.
// Because the scores of an item are finished while the previous item's V is still streaming,
// a V block is consumed the moment it lands, and the softmax never sits on the critical path.
// The sequential rescaling O <- 2^(lam (m_old - m_new)) O + P_hat V becomes
// O = sum_u 2^(lam (m_u - m)) O_u at the end of the item (one thread per channel), the same
// sum with the factors multiplied out.  Two groups of four warps take the softmax of alternate blocks of an item and a
// third one the O of every item: the P_hat of an item has to be ready when the V of the item before it has been consumed,
// so a group that also wrote O out would have one item's time (5.3 us at memory speed) for both.
//
// A request that fits one partition is finished right there.  Otherwise the partition state (m, l, O) goes to the
// workspace and decode_merge_kernel merges the partitions by log-sum-exp.  Its blocks fit beside a CTA of this kernel and
// are launched while it runs, so the merge starts the moment the last state is written.  (Merging inside this kernel, by
// the warp that completes a request's last partition, was slower in every form tried: a few CTAs end up with most of the
// merges, 190 us instead of 160 for 16 requests of 32K.)
//
// Measured (call alone, before / after the two softmax groups, the O group and the rolled passes over the scores):
// 16 requests x 32K, 8 kv heads, groups of 1 / 4 / 5 / 8 heads: 148 / 164 / 670 / 904 -> 144 / 156 / 158 / 173 us
// (5.9 / 5.6 / 5.6 / 5.2 TB/s of cache); 64 requests of 100..4000 tokens, 40:8 heads: 227 -> 59 us.  The running maxima and
// block weights held in the lanes and handed out by shuffles, where every thread took them from shared memory for every
// block: 256 requests of 100..2000 tokens with append and query 137 -> 130 us, one request of 4097 22.6 -> 21.7 us.
// K blocks by two warps in turn, each lane issuing its own block, MMAs issued by one thread that also waits, both softmax groups on every
// item, V held back until the first item's K is on its way, and then one waiting loop for all roles (replayed back to back): one request of
// 4097 keys 15.5 -> 12.9 -> 12.6 us, 64 of 100..4000 63.1 -> 59.2 -> 53.8, 32 of 16K..128K 703 -> 649 -> 634 (4.06 GB of cache, 6.4 TB/s).
// Not kept: K rings of 5, 6 and 7 stages (1 to 3 us more on short batches, nothing on long ones), small pieces by 16-byte copies of all
// lanes (no gain), partitions shorter than 1024 keys drawn last (2 us more on 64 requests), items of one block by one softmax group alone
// (no gain on them, 1 to 3 % more on 512 requests of 100..2000).
//
// Warps: 18 draws work items and stages their query tiles, 0 and 17 K producers (alternate blocks),
// 16 V producer, 1 QK issue (+ TMEM allocation), 2 PV issue, 3 rewrites the K scales of each block from
// [token][8] into the 32 x 16-byte tiles tcgen05.cp expects, 4-7 and 8-11 the two softmax groups, 12-15 O (TMEM lane
// quadrant = warp % 4).  Every wait is bounded.
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace mpfa {
namespace {

constexpr int MAXG = 8;
constexpr int NCOL = 16;          // MMA N: the GQA group padded to 16 columns
constexpr int MAXBLK = DECODE_SPLIT / TILE;   // 8 blocks per item

constexpr int D_NK = 4;           // K ring stages
constexpr int D_NV = 8;           // V ring stages
constexpr int D_THREADS = 608;
constexpr int D_NITEM = 4;        // slots of the work-item ring

// one K stage
constexpr uint32_t KST_K = 0;          // 2 pages x 4096 B of codes: 64-byte rows, 64-byte swizzle
constexpr uint32_t KST_SF = 8192;      // 2 pages x 512 B of K scales, [token][8]
constexpr uint32_t KST_DELTA = 9216;   // 2 pages x 8 rows x 128 B of Delta_S (BF16, 128-byte swizzle; rows G..7 stay zero)
constexpr uint32_t KST_BYTES = 11264;
constexpr uint32_t VST_BYTES = 16384;  // 2 pages x 8192 B: 128-byte rows, 128-byte swizzle
constexpr uint32_t D_OFF_K = 0;
constexpr uint32_t D_OFF_V = D_OFF_K + D_NK * KST_BYTES;
constexpr uint32_t D_OFF_P = D_OFF_V + D_NV * VST_BYTES;   // [2 items][8 blocks] x 1024: P_hat^T, 8 rows of 128 keys (rows 8..15: zero block)
constexpr uint32_t D_OFF_Q = D_OFF_P + 2 * MAXBLK * 1024;  // 2 x 1024: Q codes, 16 rows of 64 B, 64-byte swizzle
constexpr uint32_t D_OFF_SFQ = D_OFF_Q + 2048;             // 2 x (2 x 512): Q scales, one tile per 64 channels
constexpr uint32_t D_OFF_SFK = D_OFF_SFQ + 2048;           // D_NK x (2 x 512): K scales
constexpr uint32_t D_OFF_ZERO = D_OFF_SFK + D_NK * 1024;    // 2048 B of zeros: second K group of the Delta_S operand, rows 8..15 of P_hat^T
constexpr uint32_t D_OFF_IDENT = D_OFF_ZERO + 2048;        // 16 x 16 BF16 identity, MN-major, 128-byte swizzle
constexpr uint32_t D_OFF_BAR = D_OFF_IDENT + 2048;
constexpr uint32_t D_OFF_XMAX = D_OFF_BAR + 1024;           // [2][8 blocks][MAXG][4 warps] floats
constexpr uint32_t D_OFF_WTAB = D_OFF_XMAX + 2 * MAXBLK * MAXG * 16;   // [2][8 blocks][MAXG] floats
constexpr uint32_t D_OFF_MFIN = D_OFF_WTAB + 2 * MAXBLK * MAXG * 4;    // [2][MAXG]
constexpr uint32_t D_OFF_XL = D_OFF_MFIN + 2 * MAXG * 4;               // [2][8 warps][MAXG]
constexpr uint32_t D_OFF_MISC = D_OFF_XL + 2 * 8 * MAXG * 4;           // TMEM address, abort flag
constexpr int D_MAXREQ = 768;                                          // requests whose length / lambda are cached
constexpr uint32_t D_OFF_LEN = D_OFF_MISC + 64;                        // [D_MAXREQ] int32 lengths
constexpr uint32_t D_OFF_LAM = D_OFF_LEN + D_MAXREQ * 4;               // [D_MAXREQ] float
constexpr uint32_t D_OFF_RING = D_OFF_LAM + D_MAXREQ * 4;              // [D_NITEM] int4 work items {b, hk, sp, L}
constexpr uint32_t D_OFF_PRE = D_OFF_RING + D_NITEM * 16;              // [D_MAXREQ + 1] items of the requests before b
constexpr uint32_t D_SMEM_USED = D_OFF_PRE + (D_MAXREQ + 4) * 4;
constexpr uint32_t D_SMEM = D_SMEM_USED + 1024;     // slack for the 1024-byte alignment of the base

// barriers (8 bytes each)
constexpr int B_K_FULL = 0;                      // [D_NK] K stage landed (bytes)
constexpr int B_K_EMPTY = B_K_FULL + D_NK;       // [D_NK] QK commit
constexpr int B_V_FULL = B_K_EMPTY + D_NK;       // [D_NV]
constexpr int B_V_EMPTY = B_V_FULL + D_NV;       // [D_NV] PV commit
constexpr int B_SF_READY = B_V_EMPTY + D_NV;     // [D_NK] K scales formatted
constexpr int B_S_FULL = B_SF_READY + D_NK;      // [2] QK commit after the item's last block
constexpr int B_S_FREE = B_S_FULL + 2;           // [2] 8 warps: the item's scores have been read
constexpr int B_P_READY = B_S_FREE + 2;          // [2] 8 warps: P_hat, block weights and row sums of the item written
constexpr int B_Q_READY = B_P_READY + 2;         // [2] query tile of the item staged
constexpr int B_O_FULL = B_Q_READY + 2;          // [1] PV commit after the item's last block
constexpr int B_T_FREE = B_O_FULL + 1;           // [2] 4 warps: the item's tables (and, after its PV, P_hat) may be overwritten
constexpr int B_O_FREE = B_T_FREE + 2;           // [1] 4 warps
constexpr int B_XCHG = B_O_FREE + 1;             // [2] 8 softmax warps: block maxima of the item exchanged
constexpr int B_ITEM_FULL = B_XCHG + 2;          // [D_NITEM] work item published
constexpr int B_ITEM_EMPTY = B_ITEM_FULL + D_NITEM;   // [D_NITEM] read by all eighteen consumer warps
constexpr int B_DRAW = B_ITEM_EMPTY + D_NITEM;   // [2] warp 0 has begun item k (slot k & 1): the next one may be drawn
constexpr int B_V_GO = B_DRAW + 2;               // [1] warp 0 has issued its K blocks of the CTA's first item (when to begin, nothing more)
constexpr int B_COUNT = B_V_GO + 1;
static_assert(B_COUNT * 8 <= 1024, "barrier block");
static_assert(D_SMEM <= 232448, "shared memory");
static_assert(KST_BYTES % 1024 == 0 && D_OFF_V % 1024 == 0 && D_OFF_P % 1024 == 0, "swizzle atoms");

// tensor-memory columns
constexpr uint32_t TM_S = 0;       // [2 items][8 blocks] x 16
constexpr uint32_t TM_O = 256;     // [8 blocks] x 16
constexpr uint32_t TM_SFQ = 384;   // 2 x 8
constexpr uint32_t TM_SFK = 400;   // D_NK x 8
static_assert(TM_SFK + D_NK * 8 <= 512, "tensor memory");
constexpr uint32_t TM_COLS = 512;

#ifndef MPFA_WAIT_LIMIT_CYCLES
#define MPFA_WAIT_LIMIT_CYCLES 4000000000ll   // about two seconds of SM clock
#endif
constexpr long long D_WAIT_CYCLES = MPFA_WAIT_LIMIT_CYCLES;
// Test builds only (-DMPFA_TEST_DROP_V_COPY with a short limit): every CTA's V producer leaves out its first copy,
// so the give-up path runs (status bit, roles leave, copies in flight awaited, tensor memory released).

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The first G (1..8) TMEM columns at `taddr` of this thread's lane; the load width is the next power of two.
template <int G>
__device__ __forceinline__ void tmem_ld_g(uint32_t taddr, uint32_t (&r)[G]) {
  static_assert(G >= 1 && G <= 8, "group size");
  if constexpr (G == 1) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r[0]) : "r"(taddr) : "memory");
  } else if constexpr (G == 2) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(taddr) : "memory");
  } else if constexpr (G <= 4) {
    uint32_t x[4];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3])
                 : "r"(taddr)
                 : "memory");
#pragma unroll
    for (int g = 0; g < G; ++g) r[g] = x[g];
  } else {
    uint32_t x[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]), "=r"(x[4]), "=r"(x[5]), "=r"(x[6]), "=r"(x[7])
                 : "r"(taddr)
                 : "memory");
#pragma unroll
    for (int g = 0; g < G; ++g) r[g] = x[g];
  }
}

__device__ __forceinline__ float warp_max(float x) {
  asm("redux.sync.max.f32 %0, %0, 0xffffffff;" : "+f"(x));
  return x;
}

struct DecodeParams {
  const uint8_t *q_codes;  // tile layout, N = 1: row 0 of each (b, hq) tile
  const uint8_t *q_sf;
  const uint8_t *k_codes, *k_sf, *v_fp8;
  const __nv_bfloat16 *delta;  // may be null
  const int32_t *page_table;
  const int32_t *seq_lens;
  const float *q_gscale, *k_gscale;
  float *part_o;           // [B, H_q, n_split, 128]
  float2 *part_ml;         // [B, H_q, n_split]: (m, l)
  unsigned int *ticket;    // global work counter, zero at launch; null: the first tickets cover all items
  __nv_bfloat16 *out;
  float *out_f32;          // may be null
  int32_t *status;
  int B, H_q, H_kv, max_pages, num_pages, n_split;
  float softmax_scale, v_scale;
  __device__ __forceinline__ int n_parts(int L) const { return min((max(L, 0) + DECODE_SPLIT - 1) / DECODE_SPLIT, n_split); }
};

// Work items (request, kv head, 1024-token partition) are handed out dynamically: one warp per CTA draws
// tickets from a global counter (its first one is its block index) and publishes the decoded items in a small
// shared-memory ring; every other warp walks that ring.  SMs do not stream at the same rate (those far from the memory
// they read are up to 8 % slower), so a static split leaves the fast ones idle at the end.  An item is drawn when the K
// producer begins the one before it: drawn further ahead, a short batch is shared out unevenly (64 requests of one
// partition, 512 items on 148 CTAs, drawn eight ahead: the first 64 CTAs could take them all).  After an item of at most half a
// partition it is drawn one earlier, since such an item's K is issued before the next ticket is there (decode alone, one / two ahead: 512
// requests of 257..512 tokens, 32:8 heads 80.1 / 73.3 us, 40:8 83.4 / 79.2; of 100..2000 169 / 164; of 16..256 the same within 1 %).
struct WorkIter;

struct DCtx {
  uint32_t bar0;
  volatile int *abort_flag;
  int32_t *status;
  __device__ __forceinline__ uint32_t bar(int i) const { return bar0 + 8u * (uint32_t)i; }
  // Bounded wait; a timeout (or another role's abort) ends in a status bit and `false`.  The waiting itself is one function for all
  // roles: nineteen warps run ten different pieces of code once per item, and with the loop copied into each of its thirty places they
  // pushed each other out of the instruction cache (stamps: every step of an item of one block took two to three times as long on some SMs
  // as on others).  Decode alone, copied / called: 512 requests of 16..128 tokens, 32:8 heads 84.1 / 62.4 us, 40:8 95.1 / 68.0, of
  // 100..2000 209 / 181; one request of 4097 13.0 / 12.6; 16 of 30000..33000 144.9 / 142.5.
  __device__ __forceinline__ bool wait(int i, uint32_t parity) const {
    const uint32_t a = bar(i);
    return mbar_try_wait(a, parity) || wait_longer(a, parity, abort_flag, status);
  }
  static __device__ __noinline__ bool wait_longer(uint32_t a, uint32_t parity, volatile int *abort_flag, int32_t *status) {
    const long long t0 = clock64();
    for (uint32_t n = 1;; ++n) {
      if (mbar_try_wait_hint(a, parity, 2000u)) return true;   // the hardware may park the thread meanwhile
      if ((n & 255u) == 0u) {
        if (*abort_flag) return false;
        if (clock64() - t0 > D_WAIT_CYCLES) {
          *abort_flag = 1;
          atomicOr(status, MPFA_DEV_TIMEOUT);
          return false;
        }
      }
    }
  }
  // the same for a whole warp: every lane waits, the result is uniform
  __device__ __forceinline__ bool wait_warp(int i, uint32_t parity) const {
    return __all_sync(0xffffffffu, wait(i, parity));
  }
  __device__ __forceinline__ void warp_arrive(int i) const {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(bar(i));
  }
};

struct WorkIter {
  uint32_t n = 0;      // items taken so far
  int b, hk, sp, L, nblk;
  // Whole warp, or the one thread that stands for its warp.  false: no more items (or the CTA is giving up).
  template <bool ONE_THREAD = false>
  __device__ bool next(const DCtx &cx, const int4 *ring) {
    const uint32_t slot = n % D_NITEM, parity = (n / D_NITEM) & 1;
    if (!(ONE_THREAD ? cx.wait(B_ITEM_FULL + slot, parity) : cx.wait_warp(B_ITEM_FULL + slot, parity))) return false;
    const int4 it = ring[slot];
    if (it.x < 0) return false;   // end marker: stays in its slot, nobody moves past it
    if (ONE_THREAD)
      mbar_arrive(cx.bar(B_ITEM_EMPTY + slot));
    else
      cx.warp_arrive(B_ITEM_EMPTY + slot);
    ++n;
    b = it.x, hk = it.y, sp = it.z, L = it.w;
    nblk = (min(L - sp * DECODE_SPLIT, DECODE_SPLIT) + TILE - 1) / TILE;
    return true;
  }
};

// Page ids of the blocks of one item, lane l holding block l's two table entries (loads only: the values
// are range-checked where they are used, so that nothing waits for them here).
__device__ __forceinline__ void lookup_pages(const DecodeParams &p, const WorkIter &w, int lane, int &pid0, int &pid1) {
  pid0 = -1, pid1 = -1;
  if (lane < w.nblk) {
    const int pg = (w.sp * DECODE_SPLIT + lane * TILE) / PAGE;
    const int32_t *row = p.page_table + (size_t)w.b * p.max_pages;
    if (pg < p.max_pages) pid0 = row[pg];
    if (pg + 1 < p.max_pages) pid1 = row[pg + 1];
  }
}

// Registers of a thread: a block of 256 threads and 64 registers of the small kernels before and after fits on an SM beside a CTA of this
// one, and its set-up runs meanwhile, if five warps of a sub-partition leave two of those their registers: 5 x 32 R + 2 x 2048 <= 16384, so
// R <= 72.  Groups of up to four heads need no more (a bound of 896 threads asks for it); the function call in the waits had raised
// them to 80 and more.  Append, query and decode at 80 / 72: 16 requests of 16..128 tokens, 16:16 heads 17.9 / 14.8 us; 100 of 100..700, 8:2
// 23.4 / 19.0; 64 of 100..1000, 32:8 31.6 / 30.0.  Larger groups spill there (groups of eight, 64 of 100..2000 21.0 / 21.9).
template <int G>
__global__ void __launch_bounds__(G <= 4 ? 896 : D_THREADS, 1) decode_split_kernel(const __grid_constant__ DecodeParams p) {
  extern __shared__ uint8_t dsm_raw[];
  uint8_t *dsm = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(dsm_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sbase = smem_u32(dsm);
  float *xmax = reinterpret_cast<float *>(dsm + D_OFF_XMAX);
  float *wtab = reinterpret_cast<float *>(dsm + D_OFF_WTAB);
  float *mfin = reinterpret_cast<float *>(dsm + D_OFF_MFIN);
  float *xl = reinterpret_cast<float *>(dsm + D_OFF_XL);
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(dsm + D_OFF_MISC);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(dsm + D_OFF_MISC + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  launch_dependents();   // the merge's blocks
  DCtx cx{sbase + D_OFF_BAR, abort_flag, p.status};

  // ---- set-up: barriers, zeroed operand tiles (rows G..15 stay zero for good), TMEM
  if (threadIdx.x == 0) {
    for (int i = 0; i < D_NK; ++i) {
      mbar_init(cx.bar(B_K_FULL + i), 1);
      mbar_init(cx.bar(B_K_EMPTY + i), 1);
      mbar_init(cx.bar(B_SF_READY + i), 1);
    }
    for (int i = 0; i < D_NV; ++i) {
      mbar_init(cx.bar(B_V_FULL + i), 1);
      mbar_init(cx.bar(B_V_EMPTY + i), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(cx.bar(B_S_FULL + i), 1);
      mbar_init(cx.bar(B_XCHG + i), 8);
      mbar_init(cx.bar(B_T_FREE + i), 4);
      mbar_init(cx.bar(B_DRAW + i), 1);
      mbar_init(cx.bar(B_S_FREE + i), 8);
      mbar_init(cx.bar(B_P_READY + i), 8);
      mbar_init(cx.bar(B_Q_READY + i), 1);
    }
    mbar_init(cx.bar(B_V_GO), 1);
    mbar_init(cx.bar(B_O_FULL), 1);
    mbar_init(cx.bar(B_O_FREE), 4);
    for (int i = 0; i < D_NITEM; ++i) {
      mbar_init(cx.bar(B_ITEM_FULL + i), 1);
      mbar_init(cx.bar(B_ITEM_EMPTY + i), 18);
    }
    mbar_init_fence();
    *abort_flag = 0;
  }
  // zeroed once: the K ring (Delta_S rows G..7 are never written), P, Q and scale tiles, zero and identity blocks
  for (uint32_t o = threadIdx.x * 16; o < D_NK * KST_BYTES; o += D_THREADS * 16)
    *reinterpret_cast<uint4 *>(dsm + D_OFF_K + o) = make_uint4(0u, 0u, 0u, 0u);
  for (uint32_t o = threadIdx.x * 16; o < D_OFF_BAR - D_OFF_P; o += D_THREADS * 16)
    *reinterpret_cast<uint4 *>(dsm + D_OFF_P + o) = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  if (threadIdx.x < 16) {   // identity[n][k]: element (n, k) at (k/8)*1024 + (k%8)*128 + ((n/8) ^ (k%8))*16 + (n%8)*2
    const int k = threadIdx.x;
    *reinterpret_cast<uint16_t *>(dsm + D_OFF_IDENT + (k >> 3) * 1024 + (k & 7) * 128 + (((k >> 3) ^ (k & 7)) << 4) + (k & 7) * 2) = 0x3F80;
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), TM_COLS);
    tmem_relinquish();
  }
  // everything above touches this CTA only and overlaps the end of the preceding kernel; everything below reads memory
  grid_dependency_wait();
  int32_t *len_tab = reinterpret_cast<int32_t *>(dsm + D_OFF_LEN);
  float *lam_tab = reinterpret_cast<float *>(dsm + D_OFF_LAM);
  for (int i = threadIdx.x; i < min(p.B, D_MAXREQ); i += D_THREADS) {
    len_tab[i] = p.seq_lens[i];
    lam_tab[i] = __fmul_rn(__fmul_rn(__fmul_rn(p.softmax_scale, 1.4426950408889634f), p.q_gscale[i]), p.k_gscale[i]);
  }
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = *tmem_slot;
  const int4 *ring = reinterpret_cast<const int4 *>(dsm + D_OFF_RING);

  if (warp == 18) {
    // ================= work distribution: tickets from the global counter, decoded and published; then the query tile
    // (codes and scales of the group's G heads) of the same item is staged, in the slot that item k-2 has left.
    // With at most D_MAXREQ requests the tickets number only the partitions that exist (prefix sums of
    // ceil(L / 1024) * H_kv per request, request found by bisection); otherwise they number every
    // (request, kv head, partition slot) and the empty ones are drawn again.
    int4 *ring_w = reinterpret_cast<int4 *>(dsm + D_OFF_RING);
    int32_t *pre = reinterpret_cast<int32_t *>(dsm + D_OFF_PRE);
    const bool compact = p.B <= D_MAXREQ;
    uint32_t total;
    if (compact) {
      // pre[b] = items of requests 0..b-1: every lane sums a contiguous run of requests, the warp scans the runs
      const int per = (p.B + 31) / 32, lo = min(p.B, lane * per), hi = min(p.B, lo + per);
      int run = 0;
      for (int i = lo; i < hi; ++i) run += p.n_parts(len_tab[i]) * p.H_kv;
      int incl = run;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      int acc = incl - run;
      for (int i = lo; i < hi; ++i) {
        pre[i] = acc;
        acc += p.n_parts(len_tab[i]) * p.H_kv;
      }
      total = (uint32_t)__shfl_sync(0xffffffffu, incl, 31);
      if (lane == 31) pre[p.B] = (int)total;
      __syncwarp();
    } else {
      total = (uint32_t)p.B * p.H_kv * p.n_split;
    }
    bool ok = true, prev_short = false;
    for (uint32_t k = 0; ok; ++k) {
      const uint32_t slot = k % D_NITEM;
      if (k >= 2) {   // the K producer has begun item k-1, or k-2 where item k-1 is over before the next one could be drawn
        const uint32_t begun = prev_short ? k - 2 : k - 1;
        ok = cx.wait_warp(B_DRAW + (begun & 1), (begun >> 1) & 1);
      }
      if (ok && k >= (uint32_t)D_NITEM) ok = cx.wait_warp(B_ITEM_EMPTY + slot, ((k / D_NITEM) - 1) & 1);
      if (!ok) break;
      int4 item = make_int4(-1, 0, 0, 0);
      if (lane == 0) {
        for (bool first = k == 0;; first = false) {
          if (!first && !p.ticket) break;
          const uint32_t tkt = first ? blockIdx.x : gridDim.x + atomicAdd(p.ticket, 1u);
          if (tkt >= total) break;
          if (compact) {
            int lo = 0, hi = p.B;   // largest b with pre[b] <= tkt
            while (hi - lo > 1) {
              const int mid = (lo + hi) >> 1;
              if ((uint32_t)pre[mid] <= tkt) lo = mid; else hi = mid;
            }
            const int L = len_tab[lo], nsp = p.n_parts(L);
            const int r = (int)tkt - pre[lo];
            item = make_int4(lo, r / nsp, r % nsp, L);
            break;
          }
          const int sp = (int)(tkt % (uint32_t)p.n_split), r = (int)(tkt / (uint32_t)p.n_split);
          const int b = r / p.H_kv, L = p.seq_lens[b];
          if (L - sp * DECODE_SPLIT > 0) {
            item = make_int4(b, r % p.H_kv, sp, L);
            break;
          }
        }
        ring_w[slot] = item;
        mbar_arrive(cx.bar(B_ITEM_FULL + slot));
      }
      item.x = __shfl_sync(0xffffffffu, item.x, 0);
      if (item.x < 0) break;   // the end marker is in the ring; this CTA draws no more
      item.y = __shfl_sync(0xffffffffu, item.y, 0);
      item.z = __shfl_sync(0xffffffffu, item.z, 0);
      item.w = __shfl_sync(0xffffffffu, item.w, 0);
      prev_short = item.w - item.z * DECODE_SPLIT <= DECODE_SPLIT / 2;
      const size_t head0 = (size_t)item.x * p.H_q + (size_t)item.y * G;
      uint4 qv = make_uint4(0u, 0u, 0u, 0u);
      uint32_t qs0 = 0, qs1 = 0;
      if (lane < G * 4) qv = *reinterpret_cast<const uint4 *>(p.q_codes + (head0 + (lane >> 2)) * (TILE * 64) + (lane & 3) * 16);
      if (lane < G) {
        const uint8_t *src = p.q_sf + (head0 + lane) * 1024;
        qs0 = *reinterpret_cast<const uint32_t *>(src);
        qs1 = *reinterpret_cast<const uint32_t *>(src + 512);
      }
      const uint32_t par = k & 1;
      if (k >= 2) ok = cx.wait_warp(B_S_FULL + par, ((k >> 1) - 1) & 1);   // the MMAs of item k-2 have read the slot
      if (!ok) break;
      if (lane < G * 4) {
        const int n = lane >> 2, c = lane & 3;
        *reinterpret_cast<uint4 *>(dsm + D_OFF_Q + par * 1024 + n * 64 + ((c ^ ((n & 7) >> 1)) << 4)) = qv;
      }
      if (lane < G) {
        uint8_t *dst = dsm + D_OFF_SFQ + par * 1024 + lane * 16;
        *reinterpret_cast<uint32_t *>(dst) = qs0;
        *reinterpret_cast<uint32_t *>(dst + 512) = qs1;
      }
      fence_proxy_async_smem();
      cx.warp_arrive(B_Q_READY + par);
    }
  } else if (warp == 0 || warp >= 16) {
    // ================= producers: warps 0 and 17 stream the K ring, a block each in turn, warp 16 the V ring.  Lane u holds
    // block u of the item, its addresses and what of it exists, and issues that block's copies itself: with page ids handed around and
    // addresses made for each block, codes on one warp and the small pieces on the other, a block cost the warps 700 and 950 cycles,
    // next to the 1180 that its bytes take at the rate of the memory, and the K of a CTA's first item took 8300 with the memory idle.
    // Nothing orders the two streams but the data flow: a K stage is released by its QK MMAs, a V stage
    // only after the item's softmax, so K runs about one item ahead.  The next item is taken up, and its page ids
    // requested, before the last two blocks of the current one.
    const bool is_k = warp != 16;
    WorkIter w, wn;
    uint32_t c = 0, j = 0;   // blocks and items of this ring
    bool ok = true;
    const uint32_t d_bytes = p.delta ? (uint32_t)G * PAGE * 2 : 0u;
    const uint32_t page_bytes = is_k ? 4096u + 512u + d_bytes : 8192u;
    const uint32_t n_ring = is_k ? D_NK : D_NV;
    const int b_full = is_k ? B_K_FULL : B_V_FULL, b_empty = is_k ? B_K_EMPTY : B_V_EMPTY;
    static_assert(D_NK % 2 == 0, "each K producer has its own stages");
    int pc0 = -1, pc1 = -1, pn0 = -1, pn1 = -1;
    bool vw = w.next(cx, ring), vn = false;
    if (vw) lookup_pages(p, w, lane, pc0, pc1);
    for (; ok && vw; ++j) {
      if (warp == 0) cx.warp_arrive(B_DRAW + (j & 1));
      // Nothing can be done with V before the first item's softmax, and while all CTAs start at once its copies only keep K waiting, of
      // which warp 17's last block may still be to come.
      if (!is_k && j == 0) ok = cx.wait_warp(B_V_GO, 0);
      const bool in = lane < w.nblk, want1 = w.sp * DECODE_SPLIT + lane * TILE + PAGE < w.L;
      const bool has0 = in && pc0 >= 0 && pc0 < p.num_pages, has1 = in && want1 && pc1 >= 0 && pc1 < p.num_pages;
      if (in && (!has0 || (want1 && !has1))) atomicOr(p.status, MPFA_DEV_BAD_PAGE);
      const size_t slab0 = (size_t)(has0 ? pc0 : 0) * p.H_kv + w.hk, slab1 = (size_t)(has1 ? pc1 : 0) * p.H_kv + w.hk;
      const uint8_t *const big0 = is_k ? p.k_codes + slab0 * 4096 : p.v_fp8 + slab0 * 8192;
      const uint8_t *const big1 = is_k ? p.k_codes + slab1 * 4096 : p.v_fp8 + slab1 * 8192;
      const uint8_t *const sf0 = p.k_sf + slab0 * 512, *const sf1 = p.k_sf + slab1 * 512;
      const __nv_bfloat16 *const del0 = p.delta + slab0 * (G * PAGE), *const del1 = p.delta + slab1 * (G * PAGE);
      const uint32_t bytes = ((has0 ? 1u : 0u) + (has1 ? 1u : 0u)) * page_bytes;
      const uint32_t absent = __ballot_sync(0xffffffffu, in && !(has0 && has1));
      for (int t = 0; ok && t < w.nblk; ++t, ++c) {
        const uint32_t st = c % n_ring;
        const bool mine = !is_k || (c & 1) == (warp == 17 ? 1u : 0u);
        if (mine && c >= n_ring && !cx.wait_warp(b_empty + st, ((c / n_ring) - 1) & 1)) {
          ok = false;
          break;
        }
        const int u = w.nblk - 1 - t;
        const uint32_t full = cx.bar(b_full + st);
        if (!is_k && (absent >> u & 1u)) {
          // a page that is not there contributes P_hat = 0 times V: V must be finite, so zero it
          const bool h0 = __shfl_sync(0xffffffffu, has0, u), h1 = __shfl_sync(0xffffffffu, has1, u);
          uint8_t *stage = dsm + D_OFF_V + st * VST_BYTES;
#pragma unroll 1
          for (int half = 0; half < 2; ++half) {
            if (half == 0 ? h0 : h1) continue;
            for (int i = 0; i < 16; ++i)
              *reinterpret_cast<uint4 *>(stage + half * 8192 + i * 512 + lane * 16) = make_uint4(0u, 0u, 0u, 0u);
          }
          fence_proxy_async_smem();
          __syncwarp();
        }
#ifdef MPFA_TEST_DROP_V_COPY
        if (!is_k && c == 0) {
          // left out on purpose (work items are drawn dynamically: any CTA may be the one that gets work)
        } else
#endif
        if (mine && lane == u) {
          mbar_expect_tx(full, bytes);
          if (is_k) {
            const uint32_t dst = sbase + D_OFF_K + st * KST_BYTES;
            if (has0) {
              bulk_load(dst + KST_K, big0, 4096, full);
              bulk_load(dst + KST_SF, sf0, 512, full);
              if (d_bytes) bulk_load(dst + KST_DELTA, del0, d_bytes, full);
            }
            if (has1) {
              bulk_load(dst + KST_K + 4096, big1, 4096, full);
              bulk_load(dst + KST_SF + 512, sf1, 512, full);
              if (d_bytes) bulk_load(dst + KST_DELTA + 1024, del1, d_bytes, full);
            }
          } else {
            const uint32_t dst = sbase + D_OFF_V + st * VST_BYTES;
            if (has0) bulk_load(dst, big0, 8192, full);
            if (has1) bulk_load(dst + 8192, big1, 8192, full);
          }
        }
        __syncwarp();
        if (t == max(0, w.nblk - 3)) {
          wn = w;
          vn = wn.next(cx, ring);
          if (vn) lookup_pages(p, wn, lane, pn0, pn1);
        }
      }
      if (warp == 0 && j == 0) cx.warp_arrive(B_V_GO);
      vw = vn;
      w = wn;
      pc0 = pn0, pc1 = pn1;
    }
    // The last copies of this ring land before the warp leaves: where all goes well their consumers wait for them too, and where a
    // role gives up, before or after this loop has ended, shared memory must not go away under them.
    for (uint32_t i = c - min(c, n_ring); i < c; ++i) {
      const long long t0 = clock64();
      while (!mbar_try_wait(cx.bar(b_full + i % n_ring), (i / n_ring) & 1) && clock64() - t0 < D_WAIT_CYCLES) {
      }
    }
  } else if (warp == 1) {
    // ================= QK issue: S^T[item parity][block] = K Q^T as K stages land
    // One thread waits and issues: with the waits taken by the whole warp a block cost it 600 cycles, as long as the block's
    // bytes take.
    if (elect_one()) {
      const uint32_t id_qk = idesc_nvfp4(128, NCOL);
      const uint32_t id_ds = idesc_bf16(128, NCOL, 1, 1);
      const uint64_t d_ident = smem_desc(sbase + D_OFF_IDENT, 2048, 1024, SWZ_128B);
      const uint64_t d_sfq0 = smem_desc(sbase + D_OFF_SFQ, 0, 128, SWZ_NONE), d_sfk0 = smem_desc(sbase + D_OFF_SFK, 0, 128, SWZ_NONE);
      const uint64_t d_k0 = smem_desc(sbase + D_OFF_K + KST_K, 16, 512, SWZ_64B), d_q0 = smem_desc(sbase + D_OFF_Q, 16, 512, SWZ_64B);
      const bool has_delta = p.delta != nullptr;
      WorkIter w;
      uint32_t kc = 0, j = 0;
      bool ok = true;
      while (ok && w.next<true>(cx, ring)) {
        const uint32_t par = j & 1;
        ok = cx.wait(B_Q_READY + par, (j >> 1) & 1);
        if (ok && j >= 2) ok = cx.wait(B_S_FREE + par, ((j >> 1) - 1) & 1);   // scores of item j-2 have been read
        const uint32_t tSFQ = tm + TM_SFQ + par * 8;
        const uint64_t d_q = d_q0 + par * (1024 >> 4), d_sfq = d_sfq0 + par * (1024 >> 4);
        for (int t = 0; ok && t < w.nblk; ++t, ++kc) {
          const uint32_t st = kc % D_NK;
          ok = cx.wait(B_SF_READY + st, (kc / D_NK) & 1) && cx.wait(B_K_FULL + st, (kc / D_NK) & 1);
          if (!ok) break;
          tc_fence_after();
          const uint32_t tSFK = tm + TM_SFK + st * 8;
          if (t == 0) {
            tmem_cp_32x128b_warpx4(tSFQ, d_sfq);
            tmem_cp_32x128b_warpx4(tSFQ + 4, d_sfq + (512 >> 4));
          }
          const uint64_t d_sfk = d_sfk0 + st * (1024 >> 4);
          tmem_cp_32x128b_warpx4(tSFK, d_sfk);
          tmem_cp_32x128b_warpx4(tSFK + 4, d_sfk + (512 >> 4));
          const uint64_t d_k = d_k0 + st * (KST_BYTES >> 4);
          const uint32_t tS = tm + TM_S + (par * MAXBLK + t) * 16;
          if (has_delta) {
            // S^T = Delta_S^T I (Eq. 11 seed): A = the stage's Delta_S rows, MN-major (keys contiguous), its
            // second group of eight K rows read from the zero block; B = identity
            const uint32_t a_ds = sbase + D_OFF_K + st * KST_BYTES + KST_DELTA;
            mma_bf16_ss(tS, smem_desc(a_ds, 1024, sbase + D_OFF_ZERO - a_ds, SWZ_128B), d_ident, id_ds, 0u);
          }
          mma_nvfp4_ss(tS, d_k, d_q, id_qk, tSFK, tSFQ, has_delta ? 1u : 0u);
          mma_nvfp4_ss(tS, d_k + (32 >> 4), d_q + (32 >> 4), id_qk, tSFK + 4, tSFQ + 4, 1u);
          if (t == w.nblk - 1) mma_commit(cx.bar(B_S_FULL + par));
          mma_commit(cx.bar(B_K_EMPTY + st));
        }
        ++j;
      }
    }
    __syncwarp();
  } else if (warp == 2) {
    // ================= PV issue: O_u^T = V_u^T P_hat_u^T as V stages land
    // a request without keys has no work item: its zeros are written here, while this warp has nothing to issue
    for (int b = blockIdx.x; b < p.B; b += gridDim.x)
      if (p.seq_lens[b] <= 0)
        for (int i = lane; i < p.H_q * HEAD_DIM; i += 32) {
          p.out[(size_t)b * p.H_q * HEAD_DIM + i] = __float2bfloat16_rn(0.0f);
          if (p.out_f32) p.out_f32[(size_t)b * p.H_q * HEAD_DIM + i] = 0.0f;
        }
    if (elect_one()) {   // one thread, as for Q K^T
      const uint32_t id_pv = idesc_e4m3(128, NCOL, 1, 0);
      const uint64_t d_v0 = smem_desc(sbase + D_OFF_V, 16, 1024, SWZ_128B);
      WorkIter w;
      uint32_t vc = 0, j = 0;
      bool ok = true;
      while (ok && w.next<true>(cx, ring)) {
        const uint32_t par = j & 1;
        ok = cx.wait(B_P_READY + par, (j >> 1) & 1);
        if (ok && j >= 1) ok = cx.wait(B_O_FREE, (j - 1) & 1);   // the previous item's O has been read
        for (int t = 0; ok && t < w.nblk; ++t, ++vc) {
          const uint32_t st = vc % D_NV;
          ok = cx.wait(B_V_FULL + st, (vc / D_NV) & 1);
          if (!ok) break;
          tc_fence_after();
          const uint64_t d_v = d_v0 + st * (VST_BYTES >> 4);
          // rows 0..7 of P_hat^T in the block's tile, rows 8..15 (the next 8-row group) from the zero block
          const uint32_t a_p = sbase + D_OFF_P + (par * MAXBLK + t) * 1024;
          const uint64_t d_p = smem_desc(a_p, 16, sbase + D_OFF_ZERO - a_p, SWZ_128B);
#pragma unroll
          for (int k4 = 0; k4 < 4; ++k4)   // 32 keys per MMA
            mma_e4m3_ss(tm + TM_O + t * 16, d_v + (uint64_t)((4096 * k4) >> 4), d_p + (uint64_t)((32 * k4) >> 4), id_pv,
                        k4 > 0 ? 1u : 0u);
          mma_commit(cx.bar(B_V_EMPTY + st));
          if (t == w.nblk - 1) mma_commit(cx.bar(B_O_FULL));
        }
        ++j;
      }
    }
    __syncwarp();
  } else if (warp == 3) {
    // ================= K scales of a block: [token][8 blocks] -> two 32 x 16-byte tiles
    // (tile h = blocks 4h..4h+3; row i holds tokens i, 32+i, 64+i, 96+i), the form tcgen05.cp spreads.
    // The tile of stage st is free: the copy into the stage waited for the MMAs that read it.
    WorkIter w;
    uint32_t kc = 0;
    bool ok = true;
    while (ok && w.next(cx, ring)) {
      for (int t = 0; t < w.nblk; ++t, ++kc) {
        const uint32_t st = kc % D_NK;
        ok = cx.wait_warp(B_K_FULL + st, (kc / D_NK) & 1);
        if (!ok) break;
        const uint8_t *raw = dsm + D_OFF_K + st * KST_BYTES + KST_SF;
        uint2 v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = *reinterpret_cast<const uint2 *>(raw + (q >> 1) * 512 + ((q & 1) * 32 + lane) * 8);
        uint8_t *dst = dsm + D_OFF_SFK + st * 1024 + lane * 16;
        *reinterpret_cast<uint4 *>(dst) = make_uint4(v[0].x, v[1].x, v[2].x, v[3].x);
        *reinterpret_cast<uint4 *>(dst + 512) = make_uint4(v[0].y, v[1].y, v[2].y, v[3].y);
        fence_proxy_async_smem();
        cx.warp_arrive(B_SF_READY + st);
      }
    }
  } else if (warp < 12) {
    // ================= softmax, one thread per key of a block; two groups of four warps, group `grp` takes every item's
    // blocks of that parity
    const int grp = (warp - 4) >> 2;
    const int quad = warp & 3;                  // TMEM lane quadrant this warp may touch
    const int r = quad * 32 + lane;             // key within the block
    const uint32_t tlane = (uint32_t)(quad * 32) << 16;
    constexpr int CH = G <= 2 ? 4 : 2;          // blocks whose tensor-memory loads are in flight together
    constexpr int GP = G <= 4 ? 4 : 8, TPV = 32 / GP, NV = MAXBLK / TPV;   // heads padded; blocks to a warp's lanes; such sets
    bool ok = true;
    WorkIter w;
    for (uint32_t j = 0; ok && w.next(cx, ring); ++j) {
      const uint32_t par = j & 1, ph = (j >> 1) & 1;
      const uint32_t tS = tm + TM_S + par * (MAXBLK * 16) + tlane;
      uint8_t *const pt = dsm + D_OFF_P + par * MAXBLK * 1024 + (r & 15);
      float *xm = xmax + par * MAXBLK * MAXG * 4, *wt = wtab + par * MAXBLK * MAXG, *xlg = xl + par * 8 * MAXG;
      const float lam = w.b < D_MAXREQ ? lam_tab[w.b]
                                       : __fmul_rn(__fmul_rn(__fmul_rn(p.softmax_scale, 1.4426950408889634f), p.q_gscale[w.b]), p.k_gscale[w.b]);
      const int k_part = w.sp * DECODE_SPLIT;
      // ---- all scores of the item at once.  They are read from tensor memory twice, once for the maxima and once for the
      // exponentials: held in registers in between, MAXBLK x G of them and as many maxima went to local memory for groups
      // of five heads and more (24 us per item instead of 6).
      ok = cx.wait_warp(B_S_FULL + par, ph);
      if (!ok) break;
      tc_fence_after();
      // block maxima of this warp's keys, CH blocks at a time
#pragma unroll 1
      for (int t0 = grp; t0 < w.nblk; t0 += 2 * CH) {
        uint32_t sr[CH][G];
#pragma unroll
        for (int u = 0; u < CH; ++u)
          if (t0 + 2 * u < w.nblk) tmem_ld_g<G>(tS + (t0 + 2 * u) * 16, sr[u]);
        tmem_ld_wait();
#pragma unroll
        for (int u = 0; u < CH; ++u) {
          const int t = t0 + 2 * u;
          if (t < w.nblk) {
            const bool valid = k_part + (w.nblk - 1 - t) * TILE + r < w.L;
#pragma unroll
            for (int g = 0; g < G; ++g) {
              const float wm = warp_max(valid ? __uint_as_float(sr[u][g]) : -INFINITY);
              if (lane == 0) xm[(t * MAXG + g) * 4 + quad] = wm;
            }
          }
        }
      }
      cx.warp_arrive(B_XCHG + par);
      ok = cx.wait_warp(B_XCHG + par, ph);
      if (!ok) break;
      // running maxima m_t of the reverse traversal, -lam m_t and the weights 2^(lam (m_t - m)) of the item's end, in the lanes
      float mt[NV], nml[NV], wl[NV], m_end;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const int t = v * TPV + lane / GP;
        const float4 q = *reinterpret_cast<const float4 *>(&xm[(t * MAXG + (lane & (GP - 1))) * 4]);
        mt[v] = t < w.nblk ? fmaxf(fmaxf(fmaxf(q.x, q.y), fmaxf(q.z, q.w)), -INFINITY) : -INFINITY;   // NaNs are passed over
#pragma unroll
        for (int o = GP; o < 32; o <<= 1) {
          const float before = __shfl_up_sync(0xffffffffu, mt[v], o);
          if (lane >= o) mt[v] = fmaxf(mt[v], before);
        }
        if (v > 0) mt[v] = fmaxf(mt[v], m_end);
        m_end = __shfl_sync(0xffffffffu, mt[v], 32 - GP + (lane & (GP - 1)));
      }
      // the item two before this one, which used the same tables and P_hat tiles, is through with them
      if (j >= 2) ok = cx.wait_warp(B_T_FREE + par, ph ^ 1);
      if (!ok) break;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        nml[v] = -__fmul_rn(mt[v], lam);
        wl[v] = mt[v] == m_end ? 1.0f : ex2_approx(__fmul_rn(mt[v] - m_end, lam));
        if (warp == 4 && (lane & (GP - 1)) < G) wt[(v * TPV + lane / GP) * MAXG + (lane & (GP - 1))] = wl[v];
      }
      if (warp == 4 && lane < G) mfin[par * MAXG + lane] = m_end;
      // all P_hat of the item; l = sum of the blocks' sums times their weights
      float lsum[G];
#pragma unroll
      for (int g = 0; g < G; ++g) lsum[g] = 0.0f;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
#pragma unroll 1
        for (int t0 = grp; t0 < TPV && v * TPV + t0 < w.nblk; t0 += 2 * CH) {
          uint32_t sr[CH][G];
#pragma unroll
          for (int u = 0; u < CH; ++u)
            if (v * TPV + t0 + 2 * u < w.nblk) tmem_ld_g<G>(tS + (v * TPV + t0 + 2 * u) * 16, sr[u]);
          tmem_ld_wait();
#pragma unroll
          for (int u = 0; u < CH; ++u) {
            const int t = v * TPV + t0 + 2 * u;
            if (t < w.nblk) {
              const bool valid = k_part + (w.nblk - 1 - t) * TILE + r < w.L;
              float pq[G + 1];
#pragma unroll
              for (int g = 0; g < G; ++g) {
                const float c = __shfl_sync(0xffffffffu, nml[v], (t0 + 2 * u) * GP + g), wg = __shfl_sync(0xffffffffu, wl[v], (t0 + 2 * u) * GP + g);
                const float e = ex2_approx(__fmaf_rn(__uint_as_float(sr[u][g]), lam, c));
                const float pv = valid ? e : 0.0f;
                lsum[g] = __fmaf_rn(wg, pv, lsum[g]);
                pq[g] = __fmul_rn(pv, 448.0f);
              }
              pq[G] = 0.0f;
              uint8_t *const pb = pt + t * 1024;
#pragma unroll
              for (int g = 0; g < G; g += 2) {
                const uint32_t two = (uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(pq[g], pq[g + 1]), __NV_SATFINITE, __NV_E4M3);
                pb[g * 128 + (((r >> 4) ^ g) << 4)] = (uint8_t)two;
                if (g + 1 < G) pb[(g + 1) * 128 + (((r >> 4) ^ (g + 1)) << 4)] = (uint8_t)(two >> 8);
              }
            }
          }
        }
      }
      tc_fence_before();
      cx.warp_arrive(B_S_FREE + par);
#pragma unroll
      for (int g = 0; g < G; ++g) {
        float ls = lsum[g];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ls += __shfl_xor_sync(0xffffffffu, ls, o);
        if (lane == 0) xlg[(warp - 4) * MAXG + g] = ls;
      }
      fence_proxy_async_smem();
      cx.warp_arrive(B_P_READY + par);
    }
  } else {
    // ================= O of every item, one thread per channel, as soon as its V has been consumed
    constexpr int CH = G <= 2 ? 4 : 2;
    const int quad = warp & 3, r = quad * 32 + lane;
    const uint32_t tO = tm + TM_O + ((uint32_t)(quad * 32) << 16);
    bool ok = true;
    WorkIter w;
    for (uint32_t j = 0; ok && w.next(cx, ring); ++j) {
      const int par = j & 1;
      const float *wt = wtab + par * MAXBLK * MAXG, *xlg = xl + par * 8 * MAXG;
      ok = cx.wait_warp(B_P_READY + par, (j >> 1) & 1) && cx.wait_warp(B_O_FULL, j & 1);   // the item's tables; its accumulators
      if (!ok) break;
      tc_fence_after();
      float acc[G], l[G], m[G];
#pragma unroll
      for (int g = 0; g < G; ++g) {
        acc[g] = 0.0f;
        m[g] = mfin[par * MAXG + g];
        l[g] = ((xlg[g] + xlg[MAXG + g]) + (xlg[2 * MAXG + g] + xlg[3 * MAXG + g])) +
               ((xlg[4 * MAXG + g] + xlg[5 * MAXG + g]) + (xlg[6 * MAXG + g] + xlg[7 * MAXG + g]));
      }
#pragma unroll 1
      for (int t0 = 0; t0 < w.nblk; t0 += CH) {
        uint32_t o[CH][G];
#pragma unroll
        for (int u = 0; u < CH; ++u)
          if (t0 + u < w.nblk) tmem_ld_g<G>(tO + (t0 + u) * 16, o[u]);
        tmem_ld_wait();
#pragma unroll
        for (int u = 0; u < CH; ++u)
          if (t0 + u < w.nblk) {
#pragma unroll
            for (int g = 0; g < G; ++g) acc[g] = __fmaf_rn(wt[(t0 + u) * MAXG + g], __uint_as_float(o[u][g]), acc[g]);
          }
      }
      tc_fence_before();
      cx.warp_arrive(B_O_FREE);
      cx.warp_arrive(B_T_FREE + par);
      const size_t head0 = (size_t)w.b * p.H_q + (size_t)w.hk * G;
      const int n_parts = p.n_parts(w.L);
      if (n_parts == 1) {
#pragma unroll
        for (int g = 0; g < G; ++g) {
          const float y = l[g] > 0.0f ? __fmul_rn(__fdiv_rn(acc[g], __fmul_rn(448.0f, l[g])), p.v_scale) : 0.0f;
          p.out[(head0 + g) * HEAD_DIM + r] = __float2bfloat16_rn(y);
          if (p.out_f32) p.out_f32[(head0 + g) * HEAD_DIM + r] = y;
        }
        continue;
      }
#pragma unroll
      for (int g = 0; g < G; ++g) {
        p.part_o[((head0 + g) * p.n_split + w.sp) * HEAD_DIM + r] = acc[g];
        if (r == g) p.part_ml[(head0 + g) * p.n_split + w.sp] = make_float2(m[g], l[g]);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tm, TM_COLS);
}

// The work counter, zeroed in stream order.  A kernel and not a memory set, so that the split kernel's set-up overlaps
// the end of whatever precedes the call.
__global__ void decode_prep_kernel(unsigned int *ticket) {
  launch_dependents();
  grid_dependency_wait();
  *ticket = 0u;
}

// Merge of the partition states (Section 5.3): M = max m_s, w_s = 2^(lam (m_s - M)),
// l = sum w_s l_s, O = sum w_s O_s, out = O / (448 l) * v_scale.  grid (H_q, B).  Warp w takes the partitions s = w,
// w + 4, ... in ascending order, a lane four channels (one 512-byte row per warp and load, four rows in flight), and the
// four sums are added in warp order: a fixed order, so the result is reproducible.  128 threads of at most 56 registers
// fit beside a CTA of the split kernel.  Requests of one partition or without keys are complete already.
__global__ void __launch_bounds__(128, 9) decode_merge_kernel(const __grid_constant__ DecodeParams p) {
  __shared__ float s_l[4];
  __shared__ __align__(16) float s_o[4][HEAD_DIM];
  grid_dependency_wait();
  const int hq = blockIdx.x, b = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const size_t head = (size_t)b * p.H_q + hq;
  const float2 *ml = p.part_ml + head * p.n_split;
  const float4 *po = reinterpret_cast<const float4 *>(p.part_o + head * p.n_split * HEAD_DIM) + lane;
  // The first states are requested before the length is known: the request's slots of the workspace exist whatever it is, and
  // what stands in those past its last partition is not used.  (One load after the other, length, maxima, states, the merge of a
  // single request took 4.2 us alone.)  Sixteen of them where there are few heads, which wait for one another's latency only; four where
  // there are many, since a table that is wider than the requests are long makes the others reads for nothing.  Append, query and decode with
  // sixteen / four: one request of 4097 keys, 32 heads 18.57 / 18.76 us; 8 x 40 heads the same; 16 requests of 30000..33000, 32 heads 145.8 /
  // 145.1; 64 x 40 heads of 100..4000 keys in tables of 2048 pages 68.3 / 66.6.
  const bool few = gridDim.x * gridDim.y <= 320;
  float2 a[4];
  float4 x[4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
    if (u == 0 || few) {
      const int s = min(warp + 4 * u, p.n_split - 1);
      a[u] = ml[s];
      x[u] = po[(size_t)s * (HEAD_DIM / 4)];
    }
  const float first_max = ml[min(lane, p.n_split - 1)].x;
  const int n = p.n_parts(p.seq_lens[b]);
  const float lam = __fmul_rn(__fmul_rn(__fmul_rn(p.softmax_scale, 1.4426950408889634f), p.q_gscale[b]), p.k_gscale[b]);
  if (n <= 1) return;
  float M = lane < n ? first_max : -INFINITY;
  for (int s = lane + 32; s < n; s += 32) M = fmaxf(M, ml[s].x);   // every warp takes the maximum of all
  M = warp_max(M);
  float l = 0.0f, o[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 1
  for (int s0 = warp; s0 < n; s0 += 16) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (s0 != warp || (u > 0 && !few)) {
        const int s = min(s0 + 4 * u, n - 1);
        a[u] = ml[s];
        x[u] = po[(size_t)s * (HEAD_DIM / 4)];
      }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (s0 + 4 * u >= n) a[u].x = -INFINITY;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (a[u].x == -INFINITY) continue;   // no score above -infinity: left out, its sums need not be finite
      const float w = ex2_approx(__fmul_rn(a[u].x - M, lam));
      l = __fmaf_rn(w, a[u].y, l);
      o[0] = __fmaf_rn(w, x[u].x, o[0]);
      o[1] = __fmaf_rn(w, x[u].y, o[1]);
      o[2] = __fmaf_rn(w, x[u].z, o[2]);
      o[3] = __fmaf_rn(w, x[u].w, o[3]);
    }
  }
  if (lane == 0) s_l[warp] = l;
  *reinterpret_cast<float4 *>(&s_o[warp][lane * 4]) = make_float4(o[0], o[1], o[2], o[3]);
  __syncthreads();
  const int c = threadIdx.x;
  const float lt = (s_l[0] + s_l[1]) + (s_l[2] + s_l[3]), ot = (s_o[0][c] + s_o[1][c]) + (s_o[2][c] + s_o[3][c]);
  const float y = lt > 0.0f ? __fmul_rn(__fdiv_rn(ot, __fmul_rn(448.0f, lt)), p.v_scale) : 0.0f;
  p.out[head * HEAD_DIM + c] = __float2bfloat16_rn(y);
  if (p.out_f32) p.out_f32[head * HEAD_DIM + c] = y;
}

// The same merge where no request can have more than FEW_PARTS partitions: a warp per (request, head), all states in flight, nothing to
// exchange.  (Four warps of which each had one state, append + query + decode: 256 requests of 100..2000 tokens 126 us, now 122.5; 64
// of 100..4000 66 both ways.)
constexpr int FEW_PARTS = 4;
__global__ void __launch_bounds__(128) decode_merge_few_kernel(const __grid_constant__ DecodeParams p) {
  grid_dependency_wait();
  const int head = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (head >= p.B * p.H_q) return;
  const int b = head / p.H_q;
  const float2 *ml = p.part_ml + (size_t)head * p.n_split;
  const float4 *po = reinterpret_cast<const float4 *>(p.part_o + (size_t)head * p.n_split * HEAD_DIM) + lane;
  float2 a[FEW_PARTS];
  float4 x[FEW_PARTS];
#pragma unroll
  for (int s = 0; s < FEW_PARTS; ++s) {   // requested before the length is known, as above
    const int at = min(s, p.n_split - 1);
    a[s] = ml[at];
    x[s] = po[(size_t)at * (HEAD_DIM / 4)];
  }
  const int n = p.n_parts(p.seq_lens[b]);
  const float lam = __fmul_rn(__fmul_rn(__fmul_rn(p.softmax_scale, 1.4426950408889634f), p.q_gscale[b]), p.k_gscale[b]);
  if (n <= 1) return;
  float M = -INFINITY;
#pragma unroll
  for (int s = 0; s < FEW_PARTS; ++s)
    if (s < n) M = fmaxf(M, a[s].x);
  float l = 0.0f, o[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
  for (int s = 0; s < FEW_PARTS; ++s) {
    if (s >= n || a[s].x == -INFINITY) continue;   // no score above -infinity: left out, its sums need not be finite
    const float w = ex2_approx(__fmul_rn(a[s].x - M, lam));
    l = __fmaf_rn(w, a[s].y, l);
    o[0] = __fmaf_rn(w, x[s].x, o[0]);
    o[1] = __fmaf_rn(w, x[s].y, o[1]);
    o[2] = __fmaf_rn(w, x[s].z, o[2]);
    o[3] = __fmaf_rn(w, x[s].w, o[3]);
  }
  __align__(8) __nv_bfloat16 h[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    o[i] = l > 0.0f ? __fmul_rn(__fdiv_rn(o[i], __fmul_rn(448.0f, l)), p.v_scale) : 0.0f;
    h[i] = __float2bfloat16_rn(o[i]);
  }
  const size_t at = (size_t)head * HEAD_DIM + lane * 4;
  if ((reinterpret_cast<uintptr_t>(p.out) & 7) == 0) {   // the interface asks for no alignment of the outputs
    *reinterpret_cast<uint2 *>(p.out + at) = *reinterpret_cast<const uint2 *>(h);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) p.out[at + i] = h[i];
  }
  if (p.out_f32) {
#pragma unroll
    for (int i = 0; i < 4; ++i) p.out_f32[at + i] = o[i];
  }
}

}  // namespace
}  // namespace mpfa

using namespace mpfa;

// Workspace: partition accumulators, partition (m, l), work counter; each part 256-byte aligned.
struct DecodeWorkspace {
  size_t ml, ticket, bytes;
};
static DecodeWorkspace decode_workspace(int B, int H_q, size_t n_split) {
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  DecodeWorkspace w;
  w.ml = up((size_t)B * H_q * n_split * HEAD_DIM * sizeof(float));
  w.ticket = w.ml + up((size_t)B * H_q * n_split * sizeof(float2));
  w.bytes = w.ticket + 256;
  return w;
}

extern "C" size_t mpfa_decode_workspace_bytes(int B, int H_q, int H_kv, int max_pages_per_req) {
  if (B <= 0 || H_q <= 0 || H_kv <= 0 || max_pages_per_req <= 0) return 0;
  const size_t n_split = ((size_t)max_pages_per_req * PAGE + DECODE_SPLIT - 1) / DECODE_SPLIT;
  return decode_workspace(B, H_q, n_split).bytes;
}

extern "C" mpfa_status mpfa_decode(const mpfa_fp4_tensor *q, const mpfa_paged_kv *kv, const int32_t *page_table,
                                   int max_pages_per_req, const int32_t *seq_lens, const mpfa_stats *st, float v_scale,
                                   float softmax_scale, void *out_bf16, float *out_f32, void *workspace,
                                   size_t workspace_bytes, int32_t *device_status, void *stream) {
  if (!q || !kv || !page_table || !seq_lens || !st || !out_bf16 || !workspace || !device_status)
    return MPFA_ERR_INVALID_ARG;
  if (!q->codes || !q->sf || q->B <= 0 || q->H <= 0 || q->N != 1 || max_pages_per_req <= 0)
    return MPFA_ERR_INVALID_ARG;
  if (!kv->k_codes || !kv->k_sf || !kv->v_fp8 || kv->num_pages <= 0 || !st->q_gscale || !st->k_gscale)
    return MPFA_ERR_INVALID_ARG;
  if (!(softmax_scale > 0.0f) || !(v_scale > 0.0f)) return MPFA_ERR_INVALID_ARG;
  if (kv->page_size != PAGE) return MPFA_ERR_UNSUPPORTED;
  const int B = q->B, H_q = q->H, H_kv = kv->H_kv;
  if (H_kv <= 0 || kv->H_q != H_q) return MPFA_ERR_INVALID_ARG;
  if (H_q % H_kv != 0 || H_q / H_kv > MAXG) return MPFA_ERR_UNSUPPORTED;
  const size_t n_split = ((size_t)max_pages_per_req * PAGE + DECODE_SPLIT - 1) / DECODE_SPLIT;
  const DecodeWorkspace ws = decode_workspace(B, H_q, n_split);
  if (workspace_bytes < ws.bytes) return MPFA_ERR_WORKSPACE;
  if ((size_t)B * H_kv * n_split > 0x7FFFFFFFull || B > 65535) return MPFA_ERR_UNSUPPORTED;
  if (!aligned(q->codes, 16) || !aligned(q->sf, 16) || !aligned(kv->k_codes, 256) || !aligned(kv->k_sf, 256) ||
      !aligned(kv->v_fp8, 256) || !aligned(kv->delta_s_bf16, 256) || !aligned(workspace, 16))
    return MPFA_ERR_ALIGNMENT;
  int dev = 0, n_sm = 0;
  mpfa_status rc = device_info(&dev, &n_sm);
  if (rc != MPFA_OK) return rc;
  DecodeParams p;
  p.q_codes = q->codes;
  p.q_sf = q->sf;
  p.k_codes = kv->k_codes;
  p.k_sf = kv->k_sf;
  p.v_fp8 = kv->v_fp8;
  p.delta = static_cast<const __nv_bfloat16 *>(kv->delta_s_bf16);
  p.page_table = page_table;
  p.seq_lens = seq_lens;
  p.q_gscale = st->q_gscale;
  p.k_gscale = st->k_gscale;
  p.part_o = static_cast<float *>(workspace);
  p.part_ml = reinterpret_cast<float2 *>(static_cast<uint8_t *>(workspace) + ws.ml);
  p.out = static_cast<__nv_bfloat16 *>(out_bf16);
  p.out_f32 = out_f32;
  p.status = device_status;
  p.B = B;
  p.H_q = H_q;
  p.H_kv = H_kv;
  p.max_pages = max_pages_per_req;
  p.num_pages = kv->num_pages;
  p.n_split = (int)n_split;
  p.softmax_scale = softmax_scale;
  p.v_scale = v_scale;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const size_t items = (size_t)B * H_kv * n_split;
  const unsigned grid = (unsigned)(items < (size_t)n_sm ? items : (size_t)n_sm);   // one persistent CTA per SM
  void (*kern)(const DecodeParams) = nullptr;
  switch (H_q / H_kv) {
    case 1: kern = decode_split_kernel<1>, rc = allow_smem<decode_split_kernel<1>>(D_SMEM); break;
    case 2: kern = decode_split_kernel<2>, rc = allow_smem<decode_split_kernel<2>>(D_SMEM); break;
    case 3: kern = decode_split_kernel<3>, rc = allow_smem<decode_split_kernel<3>>(D_SMEM); break;
    case 4: kern = decode_split_kernel<4>, rc = allow_smem<decode_split_kernel<4>>(D_SMEM); break;
    case 5: kern = decode_split_kernel<5>, rc = allow_smem<decode_split_kernel<5>>(D_SMEM); break;
    case 6: kern = decode_split_kernel<6>, rc = allow_smem<decode_split_kernel<6>>(D_SMEM); break;
    case 7: kern = decode_split_kernel<7>, rc = allow_smem<decode_split_kernel<7>>(D_SMEM); break;
    case 8: kern = decode_split_kernel<8>, rc = allow_smem<decode_split_kernel<8>>(D_SMEM); break;
    default: return MPFA_ERR_UNSUPPORTED;
  }
  if (rc != MPFA_OK) return rc;
  // Kernels that a small call does not need are not launched (each costs a few microseconds of host time and one to two of
  // latency): no counter where every CTA gets at most one item, no merge where no request can have two partitions.
  p.ticket = items > (size_t)n_sm ? reinterpret_cast<unsigned int *>(static_cast<uint8_t *>(workspace) + ws.ticket) : nullptr;
  if (p.ticket) MPFA_CUDA_OK(launch(decode_prep_kernel, dim3(1), dim3(1), 0, s, p.ticket));
  MPFA_CUDA_OK(launch(kern, dim3(grid), dim3(D_THREADS), D_SMEM, s, p));
  if (n_split > FEW_PARTS)
    MPFA_CUDA_OK(launch(decode_merge_kernel, dim3(H_q, B), dim3(128), 0, s, p));
  else if (n_split > 1)
    MPFA_CUDA_OK(launch(decode_merge_few_kernel, dim3((unsigned)(((long long)B * H_q + 3) / 4)), dim3(128), 0, s, p));
  return MPFA_OK;
}
