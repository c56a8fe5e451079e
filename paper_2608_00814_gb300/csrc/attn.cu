// Tree attention of the verify step.
//
// Node i, query head h (kv head g = h / (nq/nkv)) attends to the committed
// cache positions [0, ctx) and to the tree slots ctx + a for every ancestor a
// of i (itself included): softmax(q k / sqrt(d)) v.  The tree's own K/V sit in
// slots ctx .. ctx+T-1 right after the committed ones, so the keys of one
// (node, head) are a masked prefix of the contiguous slot range [0, ctx+T).
//
// bf16 path (tcgen05), split-K over the keys inside one thread-block cluster.
// A block owns up to 128 query rows of one kv head -- the (node, q-head) pairs
// of the group, so GQA reuses every K/V tile for nq/nkv heads, and 128 rows
// are the MMA's M -- and one contiguous range of 128-key tiles of [0, ctx+T).
// The blocks of the different ranges of the same rows form one cluster (up to
// 16 blocks, non-portable size, chosen so that every cluster is resident at
// once).  Per tile:
//   - S = q K^T on the tensor cores into TMEM, N = 128 keys, q as hi + lo
//     bf16 halves (two MMA chains), the A operand straight from the shared
//     memory TMA staged it in;
//   - softmax, two threads per query row, 64 keys each (one warp per SM quarter
//     left the exponentials waiting on their own latency): the row's S from TMEM,
//     the valid-key mask (cache keys, then the node's ancestors), the two halves'
//     maxima exchanged through shared memory, exp2, and P (bf16 pairs) written back
//     to TMEM;
//   - O += P V on the tensor cores (P the A operand from TMEM, V in the
//     MN-major layout TMA writes, [key][d]).
// Two threads issue the MMAs (S, and P.V) so neither waits behind the other's
// barriers; K/V tiles come by TMA through a two-stage ring.  The running
// maximum moves only when a tile exceeds it by more than 2^8 (O is rescaled
// in TMEM then).
// Merge: each block stages its unnormalised O rows and (max, sum) in its own
// shared memory over the K/V ring; after a cluster barrier a warp per owned row
// pulls it from every split, adds the splits by log-sum-exp in split order
// (deterministic) and writes the hi/lo bf16 GEMM input.
//
// The slot range is read through tensor maps over the cache's whole capacity,
// and ctx comes from device memory (written by the step's tree preparation), so
// one launch serves any ctx.  Keys past ctx + T in the last tile are masked,
// and their V rows are zeroed in shared memory before the P.V product, so
// whatever the cache holds there cannot reach the output.
//
// Prefill runs the same kernel on a chunk of consecutive tokens (CAUSAL): row i
// attends to every slot up to its own, ctx + i, so a block's keys end at its last
// row's slot and the mask is a length, not an ancestor set.
#include <math.h>
#include <string.h>
#include <stdlib.h>

#include "common.cuh"
#include "internal.h"

// Step timeline (built only with -DOOS_TIMELINE, see timeline.py): per block
// of the last attention launch, the globaltimer at entry (0), at the end of the
// loader's dependency wait (1), when q has landed (2), at the start and end of
// the softmax of tiles 0..5 (3 + 2t, 4 + 2t), when all MMAs are done (15), when
// the merge rows are staged (21), past the cluster barrier (22) and at exit (18);
// slots 19 and 20 hold the block's tile count and the split count.
#ifdef OOS_TIMELINE
namespace oos {
__device__ unsigned long long g_tl_attn[2048][24];
}
#define TL_ATTN(ev)                                                                      \
  do {                                                                                   \
    const unsigned bid_ = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z); \
    if (bid_ < 2048) oos::g_tl_attn[bid_][ev] = oos::globaltimer();                      \
  } while (0)
#define TL_ATTN_VAL(ev, v)                                                               \
  do {                                                                                   \
    const unsigned bid_ = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z); \
    if (bid_ < 2048) oos::g_tl_attn[bid_][ev] = (unsigned long long)(v);                 \
  } while (0)
#else
#define TL_ATTN(ev) \
  do {              \
  } while (0)
#define TL_ATTN_VAL(ev, v) \
  do {                     \
  } while (0)
#endif

namespace oos {

constexpr int kAttnRows = 128;     // query rows per block (tcgen05 M)
constexpr int kAttnKeys = 128;     // keys per tile (N of the S MMAs)
constexpr int kAttnD = 128;        // head dim of the bf16 path
constexpr int kKvStages = 2;       // K and V tiles in flight
// shared memory (bytes): operand tiles in the 128-byte-swizzled layout TMA
// writes: per tile two 64-wide d blocks of 128 keys x 128 bytes
constexpr int kDBlock = kAttnKeys * 128;                  // 16 KB
constexpr int kTileBytes = 2 * kDBlock;                   // 32 KB
constexpr int kOffK = 0;                                  // [kKvStages]
constexpr int kOffV = kOffK + kKvStages * kTileBytes;     // [kKvStages]
constexpr int kMaxSplits = 16;
// a merge row: the unnormalised O row (128 fp32), then (max, sum), padded to 16 bytes
constexpr int kMergeLd = kAttnD + 4;                      // floats
constexpr int kMergeRowBytes = kMergeLd * 4;              // 528
constexpr int kOffStage = kOffK;                          // merge: this block's rows, staged over the K/V ring
constexpr int kOffQ = kOffV + kKvStages * kTileBytes;     // q hi and lo, two 64-wide d blocks of 128 rows each
constexpr int kOffMax = kOffQ + 4 * kAttnRows * 128;      // [tile parity][key half][row] softmax exchange
constexpr int kOffBar = kOffMax + 4 * kAttnRows * 4;
static_assert(kAttnRows * kMergeRowBytes <= kKvStages * 2 * kTileBytes, "merge staging");
static_assert((kOffQ & 1023) == 0, "swizzled q staging is 1024-aligned");
constexpr int kAttnSmem = kOffBar + 256 + 1024;           // + barriers + alignment slack
constexpr int kAttnThreads = 384;                         // 12 warps, roles below
constexpr int kSoftWarp0 = 4;                             // softmax warps 4..11
// prefill: registers a thread keeps in the loaders' and issuers' warps and in the
// softmax warps (setmaxnreg), of the 384 * 168 the block is launched with
constexpr int kPfRegsIo = 56, kPfRegsSoft = 224, kPfRegsLaunch = 168;
static_assert(128 * kPfRegsIo + (kAttnThreads - 128) * kPfRegsSoft <= kAttnThreads * kPfRegsLaunch, "register split");
static_assert(kAttnSmem <= 227 * 1024, "shared memory per block");
static_assert(kMaxSplits <= 16, "cluster size");
// TMEM columns (lane = query row): S[2] fp32 scores of a tile, O fp32, P[2] bf16
// pairs.  With P apart from S the next S MMAs into a buffer wait only until its
// scores are in registers, not for the P.V product (8 k cached positions, T = 128:
// a tile every 1.2 us, 1.35 before).  In prefill P overwrites the first 64 columns of
// its S buffer, and there are two O, of the even and the odd tiles.
//
// Prefill's blocks go through every key unsplit or nearly.  Under one running maximum
// only its own key's weight is exact in 16 bits, and the tensor core truncates every
// addition to an O that collects all tiles: the K/V of the layers above were up to
// 15 % (FP16 cache) and 12 % (bf16) further from the exact ones than with trees of 128
// tokens, whose keys are cut over up to 16 splits, each with a maximum and an O of its own.
// So every tile has its own maximum and its own P.V, and the softmax threads add the
// tiles' O up in registers, scaled, in fp32: errors 0 .. 25 % below the trees' in seven
// shapes, for 101 -> 114 us (2048 tokens, 8B shape) and 21 -> 23 us (0.6B, 333).
constexpr int kTmS = 0;                            // [2] x 128
constexpr int kTmO = 2 * kAttnKeys;                // verify: 128, prefill: [2] x 128
constexpr int kTmP = kTmO + kAttnD;                // verify: [2] x 64
constexpr int kAttnTmemCols = 512;                 // allocation unit: a power of two
static_assert(kTmO + 2 * kAttnD <= kAttnTmemCols, "TMEM columns");

struct AttnArgs {
  CUtensorMap kmap, vmap;   // cache [capacity][nkv][d] as (d, kv head, slot)
  CUtensorMap qhi, qlo;     // q [node][nq][d] as (d, head in group, kv head, node), hi and lo halves
  const unsigned long long* anc;
  const int* ctx_dev;       // committed positions of the step (written by tree preparation)
  int T, nq, group;
  int npc;                  // nodes per block: its rows are (node, head in group), npc * group <= 128
  int splits;               // blocks per cluster (key ranges of the same rows)
  float scale_log2;         // log2(e) / sqrt(d)
  __nv_bfloat16* out;       // [T][nq*d] hi rows, lo rows at out_lo_off
  size_t out_lo_off;
  uint32_t* status;         // step status word (pipeline waits that give up)
};

// D[tmem] (+)= A[tmem] * B[smem]: A (M = 128 rows, one per lane) as packed
// bf16 pairs, K index 2c and 2c + 1 in column c (low half first)
OOS_DEV void tc_mma_bf16_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(tmem_d),
      "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Shared-memory descriptor of an MN-major operand in the 128-byte-swizzled
// layout: 64 consecutive MN elements (bf16) per 128-byte row, one row per K
// index, 8-row / 1024-byte swizzle atoms.  `lbo` is the byte distance between
// consecutive 64-element MN blocks, the stride between 8-row K groups is 1024.
OOS_DEV uint64_t smem_desc_sw128_mn(uint32_t saddr, uint32_t lbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)(1024u >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
OOS_DEV void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// 2^x by the hardware approximation (relative error ~2^-22; -inf gives +0)
OOS_DEV float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// 16-byte chunk c of row r of a 128-byte-swizzled tile (rows 128 bytes apart,
// 8-row / 1024-byte swizzle atoms, tile base 1024-aligned)
OOS_DEV uint32_t sw128(int r, int c) { return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4)); }
// 32 lanes x 32 bit, 16 consecutive columns per thread, TMEM <- raw words
OOS_DEV void tmem_st16u(uint32_t taddr, const uint32_t* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
          taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
      "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}
OOS_DEV void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// 32 lanes x 32 bit, 32 consecutive columns per thread, without waiting: the
// caller issues several, then tmem_wait_ld_regs over every register loaded
OOS_DEV void tmem_ld32_nowait(uint32_t taddr, float* v) {
  uint32_t* r = reinterpret_cast<uint32_t*>(v);
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
// wait for the thread's outstanding TMEM loads; the empty statements after it
// make every later use of v[0..n) depend on the wait
template <int N>
OOS_DEV void tmem_wait_ld_regs(float (&v)[N]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < N; ++i) asm volatile("" : "+f"(v[i]));
}
// 64 columns of one lane row starting at taddr
OOS_DEV void tmem_ld64(uint32_t taddr, float (&v)[64]) {
  tmem_ld32_nowait(taddr, v);
  tmem_ld32_nowait(taddr + 32, v + 32);
  tmem_wait_ld_regs(v);
}
OOS_DEV float4 ld_cluster4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}
OOS_DEV float2 ld_cluster2(uint32_t addr) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
  return v;
}
// the 64 threads of the two softmax warps that share 32 query rows
OOS_DEV void row_pair_bar(int q4) { asm volatile("bar.sync %0, 64;" ::"r"(1 + q4) : "memory"); }

// 128-bit masks as (lo: bits 0..63, hi: bits 64..127)
OOS_DEV void shr128(unsigned long long lo, unsigned long long hi, int s, unsigned long long& rlo,
                    unsigned long long& rhi) {
  if (s >= 128) { rlo = 0; rhi = 0; }
  else if (s >= 64) { rlo = s == 64 ? hi : hi >> (s - 64); rhi = 0; }
  else if (s == 0) { rlo = lo; rhi = hi; }
  else { rlo = (lo >> s) | (hi << (64 - s)); rhi = hi >> s; }
}
OOS_DEV void shl128(unsigned long long lo, unsigned long long hi, int s, unsigned long long& rlo,
                    unsigned long long& rhi) {
  if (s >= 128) { rlo = 0; rhi = 0; }
  else if (s >= 64) { rhi = s == 64 ? lo : lo << (s - 64); rlo = 0; }
  else if (s == 0) { rlo = lo; rhi = hi; }
  else { rhi = (hi << s) | (lo >> (64 - s)); rlo = lo << s; }
}

template <int N>
struct Int {
  static constexpr int value = N;
};

// sites of the bounded waits (recorded on the status word when one expires)
enum { AW_KEMPTY = 21, AW_VEMPTY, AW_QFULL, AW_KFULL, AW_SFREE, AW_PFULL, AW_VFULL, AW_SFULL, AW_PV_RESCALE,
       AW_VZERO, AW_PFREE };
OOS_DEV bool attn_wait(uint64_t* bar, uint32_t parity, volatile int* abort, uint32_t* status, uint32_t site, int ti) {
  if (mbar_wait(bar, parity, abort, status)) return true;
  if (*(volatile uint32_t*)(status + 1) == 0u && (*(volatile uint32_t*)status & ST_TIMEOUT))
    record_timeout(status, site, ti, blockIdx.y, (int)blockIdx.z);
  return false;
}
// a CTA's own copies or MMAs draining after an abort: bounded by the default limit
OOS_DEV void drain_wait(uint64_t* bar, uint32_t parity) {
  const unsigned long long t0 = globaltimer();
  while (!mbar_test(smem_addr(bar), parity) && globaltimer() - t0 < kWaitLimitNs) {
  }
}

// Block roles: warp 0 lane 0 loads K tiles and q, warp 3 lane 0 V tiles (TMA into
// the swizzled layouts; apart, so that a K tile does not queue behind a V tile whose
// stage is still in use); warp 1 lane 0 issues the S MMAs, warp 2 lane 0 the P.V MMAs;
// warps 4..11 run the softmax (lane = query row = TMEM lane, warps 4..7 on the
// first 64 keys of a tile, 8..11 on the others); all warps take part in the merge
// (prefill: the softmax warps, the others having given up their registers).
// F16: the KV cache (and q) are IEEE binary16 -- every product runs in f16;
// otherwise bf16.  CAUSAL: a prefill chunk.
template <bool F16, bool CAUSAL>
__global__ void __launch_bounds__(kAttnThreads, 1) k_attn_tc(const __grid_constant__ AttnArgs a) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm + kOffBar);
  uint64_t* kfull = bar;          // [2] TMA transaction bytes
  uint64_t* kempty = bar + 2;     // [2] S MMAs of the stage's tile done
  uint64_t* vfull = bar + 4;      // [2] TMA transaction bytes
  uint64_t* vempty = bar + 6;     // [2] P.V MMAs of the stage's tile done
  uint64_t* sfull = bar + 8;      // [2] S MMAs done
  uint64_t* pfull = bar + 10;     // [2] 8 softmax warps: P written
  uint64_t* pvdone = bar + 12;    // [2] P.V MMAs done (S/P buffer free, O current)
  uint64_t* odone = bar + 15;     // both MMA issuers done
  uint64_t* qfull = bar + 17;     // q tile landed (transaction bytes)
  uint64_t* sread = bar + 18;     // [2] 8 softmax warps: S in registers (verify)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar + 20);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  static_assert(20 * 8 + 8 <= 256, "barrier block");
  constexpr bool P_APART = !CAUSAL;

  if (threadIdx.x == 0) TL_ATTN(0);
  const int T = a.T, nq = a.nq, G = a.group, npc = a.npc, S = a.splits;
  const float scale_log2 = a.scale_log2;
  uint32_t* status = a.status;
  // causal row blocks late in the chunk have the most keys: they start first
  const int rb = CAUSAL ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x, g = blockIdx.y, split = blockIdx.z;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int node0 = rb * npc;
  const int rows = npc * G;                                   // query rows of the block
  const int vrows = max(0, min(rows, (T - node0) * G));       // rows of real nodes

  // Committed positions of the step.  The step's tree preparation wrote them
  // and has completed: every kernel of the step lets its dependents launch
  // only after its own dependency wait, so when this kernel starts the kernel
  // two launches back and everything before it are complete.
  const int ctx = *a.ctx_dev;
  const int n_keys = ctx + (CAUSAL ? min(T, node0 + npc) : T);
  const int n_all = (n_keys + kAttnKeys - 1) / kAttnKeys;   // tiles over the block's keys, slots [0, n_keys)
  const int t0 = (int)((long long)split * n_all / S);
  const int n_tiles = (int)((long long)(split + 1) * n_all / S) - t0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(&kfull[s], 1);
      mbar_init(&kempty[s], 1);
      mbar_init(&vfull[s], 1);
      mbar_init(&vempty[s], 1);
      mbar_init(&sfull[s], 1);
      mbar_init(&pfull[s], 8);
      mbar_init(&sread[s], 8);
      mbar_init(&pvdone[s], 1);
    }
    mbar_init(odone, 2);
    mbar_init(qfull, 1);
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 2) tmem_alloc(tmem_slot, kAttnTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t tmem_o = tmem + kTmO;

  // every role is done with the rings and TMEM past this
  auto block_done = [&]() {
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
  };
  float* stage = reinterpret_cast<float*>(sm + kOffStage);   // [row][kMergeLd]

  // ------------------------------------------------------------ merge
  // Each block stages its O row, max and sum of every real row in its own
  // shared memory (over the K/V ring, idle by then).  Rows [0, vrows) are dealt to the S
  // blocks of the cluster; past the cluster barrier a warp takes an owned row at a
  // time, pulls it from every split and adds the splits by log-sum-exp, in order.
  // Every thread of the cluster arrives twice, whatever happened before: its
  // block's rows are staged, and it has pulled (a stage must outlive its readers).
  auto finish = [&]() {
    if (threadIdx.x == 128) TL_ATTN(21);
    cluster_arrive_release();
    __syncwarp();
    cluster_wait_acquire();
    if (threadIdx.x == 128) TL_ATTN(22);
    {
      // A warp takes KR owned rows at a time, so that about 16 pulls of a lane are in
      // flight whatever the split count (one row at a time: 4.4 us from the barrier to
      // the exit of 6 splits).
      const int lr0 = (int)((long long)vrows * split / S);
      const int n_mine = (int)((long long)vrows * (split + 1) / S) - lr0;
      constexpr int kWarp0 = CAUSAL ? kSoftWarp0 : 0, kWarps = kAttnThreads / 32 - kWarp0;
      auto merge = [&](auto kr, auto sm_max) {
        constexpr int KR = decltype(kr)::value, SM = decltype(sm_max)::value;
        bool arrived = false;
        for (int i0 = warp - kWarp0; i0 < n_mine || !arrived; i0 += KR * kWarps) {
          float2 ml[KR];
          float4 v[KR][SM];
#pragma unroll
          for (int k = 0; k < KR; ++k) {
            const int i = i0 + k * kWarps;
            const bool on = i < n_mine;
            const uint32_t off = (uint32_t)((lr0 + (on ? i : 0)) * kMergeRowBytes);
            // lane s: (max, sum) of split s; then every split's four values of this lane
            ml[k] = make_float2(-INFINITY, 0.f);
            if (on && lane < S) ml[k] = ld_cluster2(dsmem_addr(stage, (uint32_t)lane) + off + kAttnD * 4);
#pragma unroll
            for (int s = 0; s < SM; ++s)
              v[k][s] = on && s < S ? ld_cluster4(dsmem_addr(stage, (uint32_t)s) + off + (uint32_t)lane * 16u)
                                    : make_float4(0.f, 0.f, 0.f, 0.f);
          }
          float4 acc[KR];
#pragma unroll
          for (int k = 0; k < KR; ++k) {
            const float M = warp_max(ml[k].x);
            const float w = ml[k].x == -INFINITY ? 0.f : exp2f(ml[k].x - M);
            const float den = warp_sum(w * ml[k].y);
            const float wn = den > 0.f ? w / den : 0.f;
            acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int s = 0; s < SM; ++s) {
              const float ws = __shfl_sync(0xffffffffu, wn, s);   // 0 past the splits
              acc[k].x += ws * v[k][s].x;
              acc[k].y += ws * v[k][s].y;
              acc[k].z += ws * v[k][s].z;
              acc[k].w += ws * v[k][s].w;
            }
          }
          if (i0 + KR * kWarps >= n_mine) {   // the last pull: the barrier need not await this round's stores
            cluster_arrive_release();
            arrived = true;
          }
#pragma unroll
          for (int k = 0; k < KR; ++k) {
            const int i = i0 + k * kWarps;
            if (i < n_mine) {
              const int lr = lr0 + i;
              const size_t grow = (size_t)(node0 + lr / G) * nq + g * G + lr % G;
              store_act4(a.out, grow * kAttnD + 4 * lane, a.out_lo_off, acc[k]);
            }
          }
        }
      };
      if (S <= 5) merge(Int<3>{}, Int<5>{});
      else if (S <= 8) merge(Int<2>{}, Int<8>{});
      else merge(Int<1>{}, Int<kMaxSplits>{});
    }
  };

  if (warp < kSoftWarp0) {
    if constexpr (CAUSAL) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kPfRegsIo));
    if (warp == 0 || warp == 3) {
      // ------------------------------------------------------------ loaders (one thread each, TMA)
      if (lane == 0) {
        const bool v = warp == 3;
        const CUtensorMap* map = v ? &a.vmap : &a.kmap;
        uint64_t* full = v ? vfull : kfull;
        uint64_t* empty = v ? vempty : kempty;
        tma_prefetch_desc(map);
        const uint64_t pol_kv = policy_evict_first();
        auto load = [&](int ti) {   // two 64-wide d blocks of 128 slots
          const int st = ti & 1;
          const int key0 = (t0 + ti) * kAttnKeys;
          unsigned char* dst = sm + (v ? kOffV : kOffK) + st * kTileBytes;
          mbar_arrive_expect_tx(&full[st], kTileBytes);
          tma_load_3d(dst, map, &full[st], 0, g, key0, pol_kv);
          tma_load_3d(dst + kDBlock, map, &full[st], 64, g, key0, pol_kv);
        };
        // tiles of committed slots only do not depend on the producing kernel:
        // the first stages are fetched before waiting for it
        int n = 0;   // tiles issued
        while (n < n_tiles && n < kKvStages && (t0 + n + 1) * kAttnKeys <= ctx) load(n++);
        pdl_wait();
        pdl_trigger();
        if (!v) {
          TL_ATTN(1);
          // q rows of the block's nodes, hi and lo halves, two 64-wide d blocks each
          tma_prefetch_desc(&a.qhi);
          tma_prefetch_desc(&a.qlo);
          const uint64_t pol_q = policy_evict_last();
          unsigned char* qs = sm + kOffQ;
          mbar_arrive_expect_tx(qfull, (uint32_t)(4 * rows * 128));
          tma_load_4d(qs, &a.qhi, qfull, 0, 0, g, node0, pol_q);
          tma_load_4d(qs + kAttnRows * 128, &a.qhi, qfull, 64, 0, g, node0, pol_q);
          tma_load_4d(qs + 2 * kAttnRows * 128, &a.qlo, qfull, 0, 0, g, node0, pol_q);
          tma_load_4d(qs + 3 * kAttnRows * 128, &a.qlo, qfull, 64, 0, g, node0, pol_q);
        }
        for (int ti = n; ti < n_tiles; ++ti) {
          if (!attn_wait(&empty[ti & 1], ((uint32_t)(ti >> 1) & 1u) ^ 1u, abort_flag, status, v ? AW_VEMPTY : AW_KEMPTY, ti))
            break;
          load(ti);
          ++n;
        }
        // every copy this thread issued has landed before the block can exit,
        // whoever gave up (immediate on the normal path, where all were consumed)
        for (int ti = n > 2 ? n - 2 : 0; ti < n; ++ti) drain_wait(&full[ti & 1], (uint32_t)(ti >> 1) & 1u);
        if (!v) drain_wait(qfull, 0);
      }
    } else if (warp == 1 || warp == 2) {
      // ------------------------------------------------------------ MMA issuers
      // Operands reach the tensor cores through the async proxy only: q, K and
      // V by TMA, P from threads that wait for their TMEM stores before they
      // arrive, the zeroed V rows fenced by the threads that wrote them.
      // Descriptors: the start address is the low field (16-byte units), so a
      // byte offset o inside an operand region is added as o >> 4.
      if (lane == 0 && warp == 1) {
        constexpr uint32_t idesc_s = F16 ? idesc_f16_f32(kAttnRows, kAttnKeys) : idesc_bf16_f32(kAttnRows, kAttnKeys);
        bool ok = attn_wait(qfull, 0, abort_flag, status, AW_QFULL, 0);
        TL_ATTN(2);
        tc_fence_after();
        const uint64_t kdesc0 = smem_desc_sw128(smem_addr(sm + kOffK));
        // q as staged by TMA: [hi d0, hi d1, lo d0, lo d1], each 128 rows x 128
        // bytes in the swizzled K-major layout (rows of padding nodes hold
        // whatever the q buffer holds; every row of S, P and O is its own)
        const uint64_t qdesc0 = smem_desc_sw128(smem_addr(sm + kOffQ));
        for (int ti = 0; ti < n_tiles && ok; ++ti) {
          const int b = ti & 1;
          const uint32_t use = (uint32_t)(ti >> 1);
          // S buffer b holds tile ti - 2's scores until they are read, or its P until
          // that tile's P.V is done
          if (!attn_wait(&kfull[b], use & 1u, abort_flag, status, AW_KFULL, ti) ||
              !attn_wait(P_APART ? &sread[b] : &pvdone[b], (use & 1u) ^ 1u, abort_flag, status, AW_SFREE, ti))
            break;
          tc_fence_after();
          const uint64_t kd0 = kdesc0 + (uint64_t)((b * kTileBytes) >> 4);
          const uint32_t d = tmem + kTmS + b * kAttnKeys;
          // S = q_hi K^T + q_lo K^T over the 128 head dims: q and K both from
          // their two 64-wide d blocks (32 bytes of d per MMA)
#pragma unroll
          for (int half = 0; half < 2; ++half) {
#pragma unroll
            for (int k = 0; k < kAttnD / 16; ++k) {
              const uint64_t kd = kd0 + (uint64_t)(((k >> 2) * kDBlock) >> 4) + 2 * (k & 3);
              const uint64_t qd = qdesc0 + (uint64_t)(((2 * half + (k >> 2)) * (kAttnRows * 128)) >> 4) + 2 * (k & 3);
              tc_mma_bf16(d, qd, kd, idesc_s, (half > 0 || k > 0) ? 1u : 0u);
            }
          }
          tc_commit(&kempty[b]);
          tc_commit(&sfull[b]);
        }
        tc_commit(odone);
      } else if (lane == 0 && warp == 2) {
        constexpr uint32_t idesc_pv =
            (F16 ? idesc_f16_f32(kAttnRows, kAttnD) : idesc_bf16_f32(kAttnRows, kAttnD)) | (1u << 16);   // B (V) MN-major
        // V tile: d blocks of 64 (kDBlock apart) along N, 16 keys (2 KB) per MMA along K
        const uint64_t vdesc0 = smem_desc_sw128_mn(smem_addr(sm + kOffV), kDBlock);
        for (int ti = 0; ti < n_tiles; ++ti) {
          const int b = ti & 1;
          const uint32_t use = (uint32_t)(ti >> 1);
          if (!attn_wait(&pfull[b], use & 1u, abort_flag, status, AW_PFULL, ti) ||
              !attn_wait(&vfull[b], use & 1u, abort_flag, status, AW_VFULL, ti))
            break;
          tc_fence_after();
          // P: 8 columns = 16 keys per MMA
          const uint32_t pt = tmem + (P_APART ? kTmP + b * 64 : kTmS + b * kAttnKeys);
          const uint64_t vd = vdesc0 + (uint64_t)((b * kTileBytes) >> 4);
#pragma unroll
          for (int kk = 0; kk < kAttnKeys / 16; ++kk)
            tc_mma_bf16_ts(tmem_o + (CAUSAL ? b * kAttnD : 0), pt + 8 * kk, vd + (uint64_t)((kk * 16 * 128) >> 4),
                           idesc_pv, (kk > 0 || (!CAUSAL && ti > 0)) ? 1u : 0u);
          tc_commit(&pvdone[b]);
          tc_commit(&vempty[b]);
        }
        tc_commit(odone);
      }
    }
    block_done();
    if (CAUSAL) {   // their registers are given up: the softmax warps merge
      cluster_arrive_release();
      __syncwarp();
      cluster_wait_acquire();
      cluster_arrive_release();
    }
  } else {
    if constexpr (CAUSAL) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kPfRegsSoft));   // half an O row each
    // ------------------------------------------------------------ softmax (warps 4..11)
    float m_used = -INFINITY, l_sum = 0.f;            // l_sum: of this thread's keys
    const int q4 = warp & 3;
    const int hf = warp >= kSoftWarp0 + 4 ? 1 : 0;    // key half
    const int lrow = q4 * 32 + lane;                  // local row = TMEM lane
    const uint32_t lane_off = (uint32_t)(q4 * 32) << 16;
    float* s_max = reinterpret_cast<float*>(sm + kOffMax);
    // Prefill: this thread's half of its O row, of the tiles taken so far, and the
    // maximum it is scaled by (m_used: the last tile's own).
    float o_sum[CAUSAL ? 64 : 1], m_sum = -INFINITY;
#pragma unroll
    for (int i = 0; i < (CAUSAL ? 64 : 1); ++i) o_sum[i] = 0.f;
    // tile t, complete by now, whose maximum is m and whose weights sum to l (of this
    // thread's keys)
    auto take_o = [&](int t, float m, float l) {
      if constexpr (CAUSAL) {
        const float to = fmaxf(m_sum, m);
        const float fo = m_sum == -INFINITY ? 0.f : exp2f(m_sum - to), ft = m == -INFINITY ? 0.f : exp2f(m - to);
        m_sum = to;
        l_sum = l_sum * fo + l * ft;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          float ov[32];
          tmem_ld32_nowait(tmem_o + lane_off + (t & 1) * kAttnD + hf * 64 + c * 32, ov);
          tmem_wait_ld_regs(ov);
#pragma unroll
          for (int i = 0; i < 32; ++i) o_sum[c * 32 + i] = fmaf(ov[i], ft, o_sum[c * 32 + i] * fo);
        }
      }
    };
    float l_tile = 0.f, m_prev = -INFINITY, l_prev = 0.f;   // prefill: of the tile at hand, and the one before it
    const bool real = lrow < vrows;
    const int node = real ? node0 + lrow / G : node0;
    unsigned long long anc0 = 0ull, anc1 = 0ull;
    bool waited = false;
    // A wait that gives up ends the warp's work, but it still meets the warp that
    // shares its rows at the barrier of every tile.
    bool dead = false;
    // Iteration -1 is a dry pass of the tile body, run before the dependency
    // wait while the block has nothing else to do: it brings the body's code
    // into the SM's instruction caches (the step's other kernels have evicted
    // it since the previous layer), reads whatever S buffer 0 holds, and
    // discards everything -- no wait, store, arrive or state update.
#pragma unroll 1
    for (int ti = -1; ti < n_tiles; ++ti) {
      asm volatile("" : "+r"(ti));   // one loop body for every iteration: none is specialised
      const bool dry = ti < 0;         // warp-uniform
      if (ti == 0) {
        pdl_wait();
        pdl_trigger();
        waited = true;
        if (!CAUSAL) {
          anc0 = a.anc[2 * node];
          anc1 = a.anc[2 * node + 1];
        }
      }
      const int tt = dry ? 0 : ti;
      const int b = tt & 1;
      const uint32_t use = (uint32_t)(tt >> 1);
      if (!dry && !dead) {
        // every wait's outcome is made warp-uniform: the .sync.aligned TMEM
        // accesses and __syncwarp below need the whole warp on one path
        dead = !__all_sync(0xffffffffu, attn_wait(&sfull[b], use & 1u, abort_flag, status, AW_SFULL, ti));
        tc_fence_after();
      }
      const int key0 = dry ? ctx : (t0 + ti) * kAttnKeys;
      if (!dry && warp == kSoftWarp0 && lane == 0 && ti < 6) TL_ATTN(3 + 2 * ti);
      // valid keys of this row in the tile's half: committed slots, then the tree
      // slots of the node's ancestors (slot ctx + j for ancestor j); slots at
      // or past ctx + T are never ancestors (the dry pass takes the masked path)
      const bool full_tile = !dry && key0 + kAttnKeys <= ctx + (CAUSAL ? node0 + 1 : 0);   // tile-uniform
      unsigned long long mask = ~0ull;
      if (!full_tile) {
        // leading valid slots: the committed ones (< 128), or those up to the row's own
        const int c = CAUSAL ? max(0, min(kAttnKeys, ctx + node + 1 - key0)) : max(0, ctx - key0);
        unsigned long long tlo = 0ull, thi = 0ull;
        if (!CAUSAL) {
          if (key0 >= ctx) shr128(anc0, anc1, key0 - ctx, tlo, thi);
          else shl128(anc0, anc1, c, tlo, thi);
        }
        const unsigned long long clo = c >= 64 ? ~0ull : (c == 0 ? 0ull : (~0ull >> (64 - c)));
        const unsigned long long chi = c <= 64 ? 0ull : (~0ull >> (128 - c));
        mask = hf ? chi | thi : clo | tlo;
      }
      // the row's 64 scores, masked keys at -inf
      float sv[64];
      tmem_ld64(tmem + lane_off + kTmS + b * kAttnKeys + hf * 64, sv);
      if (P_APART && !dry && !dead) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sread[b]);
      }
      if (!full_tile) {
#pragma unroll
        for (int i = 0; i < 64; ++i)
          if (!((mask >> i) & 1ull)) sv[i] = -INFINITY;
      }
      float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int i = 0; i < 64; ++i) mx[i & 3] = fmaxf(mx[i & 3], sv[i]);
      float tmax = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
      // the row's maximum over both halves; past the barrier both have also read S,
      // whose columns P overwrites where they are not apart
      float* sx = s_max + b * 2 * kAttnRows + lrow;
      sx[hf * kAttnRows] = tmax;
      row_pair_bar(q4);
      tmax = fmaxf(tmax, sx[(hf ^ 1) * kAttnRows]) * scale_log2;   // scale > 0
      if (dead) continue;
      // move the running maximum only when this tile exceeds it by 2^8 (a
      // lane that moves its maximum rescales its half of the O row; the whole warp
      // takes part in the TMEM accesses, lanes that keep theirs scale by 1)
      // (prefill: every tile its own maximum)
      const bool move = CAUSAL ? !dry : !dry && tmax > m_used + 8.f;
      const bool rescale = !CAUSAL && move && m_used != -INFINITY;
      if (!CAUSAL && __any_sync(0xffffffffu, rescale)) {
        // O holds P.V of tiles < ti: wait for the last of them, then rescale
        const int pb = (ti - 1) & 1;
        dead = !__all_sync(0xffffffffu, attn_wait(&pvdone[pb], (uint32_t)((ti - 1) >> 1) & 1u, abort_flag, status,
                                                  AW_PV_RESCALE, ti));
        if (dead) continue;
        tc_fence_after();
        const float f = rescale ? exp2f(m_used - tmax) : 1.f;
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {   // 32 columns at a time: the scores stay in registers
          const uint32_t col = tmem_o + lane_off + hf * 64 + c * 32;
          float ov[32];
          tmem_ld32_nowait(col, ov);
          tmem_wait_ld_regs(ov);
#pragma unroll
          for (int i = 0; i < 32; ++i) ov[i] *= f;
          tmem_st16u(col, reinterpret_cast<const uint32_t*>(ov));
          tmem_st16u(col + 16, reinterpret_cast<const uint32_t*>(ov + 16));
          tmem_wait_st();
        }
        l_sum *= f;
      }
      if (move) m_used = tmax;
      // p = 2^(s * scale - m): one FMA and one ex2 per score; a masked score
      // (-inf) gives 0, and a row with nothing valid yet (m = -inf) gives 0
      uint32_t pk[32];
      float ps[4] = {0.f, 0.f, 0.f, 0.f};
      const bool live = dry || m_used != -INFINITY;
      const float neg_m = (live && !dry) ? -m_used : 0.f;
#pragma unroll
      for (int i = 0; i < 64; i += 2) {
        const float p0 = live ? ex2_approx(fmaf(sv[i], scale_log2, neg_m)) : 0.f;
        const float p1 = live ? ex2_approx(fmaf(sv[i + 1], scale_log2, neg_m)) : 0.f;
        // P in the operand format of V; the sum uses the rounded weights that P.V multiplies
        if constexpr (F16) {
          const __half2 pp = __floats2half2_rn(p0, p1);
          ps[(i >> 1) & 3] += __low2float(pp) + __high2float(pp);
          pk[i / 2] = *reinterpret_cast<const uint32_t*>(&pp);
        } else {
          const __nv_bfloat162 pp = __floats2bfloat162_rn(p0, p1);
          ps[(i >> 1) & 3] += __low2float(pp) + __high2float(pp);
          pk[i / 2] = *reinterpret_cast<const uint32_t*>(&pp);
        }
      }
      if (dry) {   // the weights count as used, so that the dry pass computes them
#pragma unroll
        for (int i = 0; i < 32; ++i) asm volatile("" ::"r"(pk[i]));
        asm volatile("" ::"f"(ps[0]), "f"(ps[1]), "f"(ps[2]), "f"(ps[3]));
        continue;
      }
      if (CAUSAL) l_tile = (ps[0] + ps[1]) + (ps[2] + ps[3]);
      else l_sum += (ps[0] + ps[1]) + (ps[2] + ps[3]);
      // Tile ti - 2's P.V has read this P buffer and this V buffer.  Waited for before
      // the V wait below, whose parity alone would also match a phase two back.
      if (P_APART && ti >= 2) {
        dead = !__all_sync(0xffffffffu, attn_wait(&pvdone[b], (use & 1u) ^ 1u, abort_flag, status, AW_PFREE, ti));
        if (dead) continue;
        tc_fence_after();
      }
      // slots at or past ctx + T in this tile hold whatever the cache holds
      // there: zero their V rows (P is 0 for them, but 0 * NaN is not 0), each
      // half of the warps one 64-wide d block
      const int n_ok = ctx + T - key0;                   // tile-uniform
      if (n_ok < kAttnKeys) {
        dead = !__all_sync(0xffffffffu, attn_wait(&vfull[b], use & 1u, abort_flag, status, AW_VZERO, ti));
        if (dead) continue;
        if (lrow >= n_ok) {
          unsigned char* vt = sm + kOffV + b * kTileBytes + hf * kDBlock + lrow * 128;
#pragma unroll
          for (int c = 0; c < 8; ++c) *reinterpret_cast<uint4*>(vt + c * 16) = make_uint4(0, 0, 0, 0);
          fence_async_smem();
        }
      }
#pragma unroll
      for (int part = 0; part < 2; ++part)
        tmem_st16u(tmem + lane_off + (P_APART ? kTmP + b * 64 : kTmS + b * kAttnKeys) + hf * 32 + part * 16, pk + part * 16);
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&pfull[b]);
      if (warp == kSoftWarp0 && lane == 0 && ti < 6) TL_ATTN(4 + 2 * ti);
      if (CAUSAL) {   // the tile before, whose O columns tile ti + 1 takes (it waits for these threads' P)
        if (ti > 0) {
          dead = !__all_sync(0xffffffffu, attn_wait(&pvdone[b ^ 1], (uint32_t)((ti - 1) >> 1) & 1u, abort_flag, status,
                                                    AW_PFREE, ti));
          if (dead) continue;
          tc_fence_after();
          take_o(ti - 1, m_prev, l_prev);
          tc_fence_before();
        }
        m_prev = m_used;
        l_prev = l_tile;
      }
    }
    if (!waited) {   // no tile: the dependency wait is still owed
      pdl_wait();
      pdl_trigger();
    }
    // every role is done with the rings and TMEM once all MMAs have completed;
    // both issuers always commit this barrier, and TMEM must not be released
    // under a running MMA, so the wait is not cut short by the handle's limit
    drain_wait(odone, 0);
    if (warp == kSoftWarp0 && lane == 0) TL_ATTN(15);
    block_done();
    const bool have_o = n_tiles > 0 && !*abort_flag;   // block-uniform after the barrier
    float ov[64];
    if (have_o && CAUSAL) {
      take_o(n_tiles - 1, m_prev, l_prev);
      m_used = m_sum;
#pragma unroll
      for (int i = 0; i < 64; ++i) ov[i] = o_sum[CAUSAL ? i : 0];
    } else if (have_o) {
      tmem_ld64(tmem_o + lane_off + hf * 64, ov);
    } else {
#pragma unroll
      for (int i = 0; i < 64; ++i) ov[i] = 0.f;
    }
    if (hf) s_max[lrow] = l_sum;
    if (lrow < vrows) {
      float* row = stage + (size_t)lrow * kMergeLd + hf * 64;
#pragma unroll
      for (int i = 0; i < 64; i += 4) *reinterpret_cast<float4*>(row + i) = make_float4(ov[i], ov[i + 1], ov[i + 2], ov[i + 3]);
    }
    row_pair_bar(q4);
    if (!hf && lrow < vrows) {
      const float l = l_sum + s_max[lrow];
      *reinterpret_cast<float2*>(stage + (size_t)lrow * kMergeLd + kAttnD) =
          make_float2(have_o ? m_used : -INFINITY, have_o ? l : 0.f);
    }
    if (CAUSAL) finish();
  }
  if (!CAUSAL) finish();
  __syncwarp();
  cluster_wait_acquire();
  if (threadIdx.x == 128) {
    TL_ATTN(18);
    TL_ATTN_VAL(19, n_tiles);
    TL_ATTN_VAL(20, S);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc(tmem, kAttnTmemCols);
  }
}

int attn_nodes_per_block(int group) { return group >= kAttnRows ? 1 : kAttnRows / group; }

static bool encode_q_maps(const Model& m, const void* q, int nodes, CUtensorMap* hi, CUtensorMap* lo) {
  const auto& c = m.cfg;
  const int group = c.n_q_heads / c.n_kv_heads;
  // q [node][nq][d] viewed as (d, head in group, kv head, node); a box is the
  // (node, head in group) rows of one kv head, 64 of d at a time
  const uint64_t dims[4] = {(uint64_t)kAttnD, (uint64_t)group, (uint64_t)c.n_kv_heads, (uint64_t)nodes};
  const uint64_t strides[3] = {(uint64_t)kAttnD * 2, (uint64_t)group * kAttnD * 2, (uint64_t)c.n_q_heads * kAttnD * 2};
  const uint32_t box[4] = {64, (uint32_t)group, 1, (uint32_t)attn_nodes_per_block(group)};
  const __nv_bfloat16* qp = (const __nv_bfloat16*)q;
  const bool f16 = c.kv_f16 != 0;
  return encode_bf16_map(hi, qp, 4, dims, strides, box, f16) &&
         encode_bf16_map(lo, qp + (size_t)nodes * c.n_q_heads * kAttnD, 4, dims, strides, box, f16);
}
bool attn_encode_q_maps(Model& m) {
  return encode_q_maps(m, m.ws.q, kMaxT, &m.qmap_hi, &m.qmap_lo) &&
         encode_q_maps(m, m.ws.pf_q, kPfTokens, &m.pf_qmap_hi, &m.pf_qmap_lo);
}

// clusters of `sp` attention blocks resident at once on this device (occupancy query, cached)
static int attn_max_clusters(int sp) {
  static int cached[kMaxSplits + 1] = {0};
  if (sp < 1 || sp > kMaxSplits) return 0;
  if (cached[sp] == 0) {
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(1, 1, sp);
    lc.blockDim = dim3(kAttnThreads);
    lc.dynamicSmemBytes = (size_t)kAttnSmem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = sp;
    lc.attrs = attr;
    lc.numAttrs = 1;
    int n = 0;
    cached[sp] = cudaOccupancyMaxActiveClusters(&n, (const void*)k_attn_tc<false, false>, &lc) == cudaSuccess && n > 0 ? n : -1;
    cudaGetLastError();
  }
  return cached[sp];
}

template <bool F16, bool CAUSAL>
static cudaError_t attn_setup_one() {
  cudaError_t e = cudaFuncSetAttribute(k_attn_tc<F16, CAUSAL>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAttnSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_attn_tc<F16, CAUSAL>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  // the register split must not ask for more than the block is launched with
  return e == cudaSuccess && CAUSAL ? check_launch_regs((const void*)k_attn_tc<F16, CAUSAL>, kPfRegsLaunch) : e;
}

cudaError_t attn_setup() {
  cudaError_t e = attn_setup_one<false, false>();
  if (e == cudaSuccess) e = attn_setup_one<true, false>();
  if (e == cudaSuccess) e = attn_setup_one<false, true>();
  return e == cudaSuccess ? attn_setup_one<true, true>() : e;
}

int attn_splits(Model& m, int ctx_hint, int T) {
  const auto& c = m.cfg;
  const int npc = attn_nodes_per_block(c.n_q_heads / c.n_kv_heads);
  const int pairs = c.n_kv_heads * ((T + npc - 1) / npc);
  const int tiles = (ctx_hint + T + kAttnKeys - 1) / kAttnKeys;
  // the most splits (one cluster of them per row block and kv head) such that
  // every cluster is resident at once -- one wave -- and no block is without a tile
  for (int sp = kMaxSplits; sp >= 1; --sp) {
    if (sp > tiles || pairs * sp > m.num_sms) continue;
    if (attn_max_clusters(sp) >= pairs) return sp;
  }
  return 1;
}

// one bf16-path launch over T nodes: a.qhi/qlo, a.out and a.out_lo_off are the caller's
template <bool CAUSAL>
static cudaError_t launch_attn_tc(Model& m, int layer, const void* kc, const void* vc, int capacity, int ctx, int T,
                                  AttnArgs& a, cudaStream_t st) {
  const auto& c = m.cfg;
  // this layer's cache over its whole capacity, (d, kv head, slot); encoded
  // again only when the cache buffers change
  {
    if ((int)m.kv_maps.size() != c.n_layers) m.kv_maps.assign(c.n_layers, Model::KvMaps());
    Model::KvMaps& km = m.kv_maps[layer];
    if (km.k != kc || km.v != vc || km.extent != capacity) {
      const uint64_t dims[3] = {(uint64_t)kAttnD, (uint64_t)c.n_kv_heads, (uint64_t)capacity};
      const uint64_t strides[2] = {(uint64_t)kAttnD * 2, (uint64_t)c.n_kv_heads * kAttnD * 2};
      const uint32_t box[3] = {64, 1, (uint32_t)kAttnKeys};
      if (!encode_bf16_map(&km.kmap, kc, 3, dims, strides, box, c.kv_f16 != 0) ||
          !encode_bf16_map(&km.vmap, vc, 3, dims, strides, box, c.kv_f16 != 0)) {
        km.k = km.v = nullptr;
        return cudaErrorInvalidValue;
      }
      km.k = kc;
      km.v = vc;
      km.extent = capacity;
    }
    a.kmap = km.kmap;
    a.vmap = km.vmap;
  }
  a.anc = m.ws.anc;
  a.ctx_dev = m.ws.ctx;
  a.T = T;
  a.nq = c.n_q_heads;
  a.group = c.n_q_heads / c.n_kv_heads;
  a.npc = attn_nodes_per_block(a.group);
  const int RB = (T + a.npc - 1) / a.npc;
  a.splits = attn_splits(m, ctx, T);
  a.scale_log2 = 1.4426950408889634f / sqrtf((float)kAttnD);
  a.status = m.ws.status;

  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(RB, c.n_kv_heads, a.splits);
  lc.blockDim = dim3(kAttnThreads);
  lc.dynamicSmemBytes = (size_t)kAttnSmem;
  lc.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = a.splits;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = attr;
  lc.numAttrs = m.pdl ? 2 : 1;
  return c.kv_f16 ? cudaLaunchKernelEx(&lc, k_attn_tc<true, CAUSAL>, a)
                  : cudaLaunchKernelEx(&lc, k_attn_tc<false, CAUSAL>, a);
}

cudaError_t launch_attention(Model& m, int layer, const void* kc, const void* vc, int capacity, int ctx, int T,
                             cudaStream_t st) {
  if (m.cfg.dtype != OOS_DTYPE_BF16) return launch_f32_attention(m, kc, vc, T, st);
  AttnArgs a;
  memset(&a, 0, sizeof(a));
  a.qhi = m.qmap_hi;
  a.qlo = m.qmap_lo;
  a.out = (__nv_bfloat16*)m.ws.attn;
  a.out_lo_off = (size_t)kMaxT * m.cfg.n_q_heads * kAttnD;
  return launch_attn_tc<false>(m, layer, kc, vc, capacity, ctx, T, a, st);
}

cudaError_t launch_attention_pf(Model& m, int layer, const void* kc, const void* vc, int capacity, int ctx, int T,
                                cudaStream_t st) {
  AttnArgs a;
  memset(&a, 0, sizeof(a));
  a.qhi = m.pf_qmap_hi;
  a.qlo = m.pf_qmap_lo;
  a.out = (__nv_bfloat16*)m.ws.pf_attn;
  a.out_lo_off = (size_t)kPfTokens * m.cfg.n_q_heads * kAttnD;
  return launch_attn_tc<true>(m, layer, kc, vc, capacity, ctx, T, a, st);
}

}  // namespace oos

#ifdef OOS_TIMELINE
// timeline accessors (the OOS_TIMELINE library only)
extern "C" int oos_timeline_attn_read(void* out, size_t bytes) {
  return cudaMemcpyFromSymbol(out, oos::g_tl_attn, bytes < sizeof(oos::g_tl_attn) ? bytes : sizeof(oos::g_tl_attn)) ==
                 cudaSuccess
             ? 0
             : OOS_ECUDA;
}
extern "C" int oos_timeline_attn_clear() {
  void* p = nullptr;
  if (cudaGetSymbolAddress(&p, oos::g_tl_attn) != cudaSuccess) return OOS_ECUDA;
  return cudaMemset(p, 0, sizeof(oos::g_tl_attn)) == cudaSuccess ? 0 : OOS_ECUDA;
}
#endif
