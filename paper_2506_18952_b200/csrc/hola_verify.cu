// hola_verify.cu - sm_100a kernels and C ABI for the entropy-aware verify step of Hierarchical Speculative
// Decoding (HSD section, Eq. 1, the HSD loop of Algorithm 1).  See include/hola_verify.h for the contract.
//
// Kernels
//   lm_head_entropy_kernel      persistent, warp-specialised weight-streaming GEMM run by pairs of CTAs (clusters of
//       two).  The vocabulary lies on the 128 tensor-memory lanes of each CTA, the verify positions on the N
//       dimension of the MMA:  D[v, r] = sum_h W_lm[v, h] * hidden[r, h].  A pair owns up to 256 vocabulary rows
//       per tile; each CTA streams its (up to 128) rows of W_lm and HALF of the hidden rows per K block with TMA, and one
//       thread of the leader CTA issues tcgen05.mma.cta_group::2 (bf16 x bf16 -> fp32 in tensor memory) that reads
//       both halves.  Sixteen epilogue warps copy finished accumulators to the fp32 logits buffer and, from the
//       same registers transposed through a small shared-memory buffer, keep per verify position the running
//       softmax statistics (m, s, t) = (max, sum e^(l-m), sum e^(l-m)(l-m)) and the arg-max in registers, in the
//       shadow of the next tile's MMAs.  W_lm is read from HBM once; the logits are never read back.  More verify
//       rows than one pass holds (at most 512): all passes run in the same launch, on groups of neighbouring pairs
//       that walk the same vocabulary tiles in step, one pass each, so that a tile still leaves HBM once and reaches
//       the other pairs of its group out of the L2.
//       With 257..384 verify rows the accumulators rotate over the four 128-column units of the tensor memory and a
//       unit is handed back as soon as its chunk has gone to the logits buffer and a staging buffer.  In its
//       on-chip-expansion mode the kernel streams groups of 256 vocabulary rows stored at 4, 8 or 16 bits and
//       converter warps (groups of four, each owning whole K blocks) expand the codes exactly to bf16 in tensor memory,
//       from where the MMA reads them (mixed-precision quantiser of the Lo-Bi Optimization section).
//   quantize_rows_kernel        the Lo-Bi quantiser on W_lm ahead of time: rows at 8 bits, at 4 bits (codes in [-7, 7], one
//       shared exponent per sub-block of 128 channels) or in groups of mixed width, one launch for the whole head.
//   quantize_hidden_kernel      the hidden rows of a call as one or two 8-bit planes.
//   align_hidden_kernel         the hidden rows of a call once more, on 128-byte lines.
//   bounded_wait_selftest_kernel, staged_wait_selftest_kernel  waits that are made to run out, to exercise the give-up paths
//       without breaking anything; quotient_selftest_kernel, the division behind every entropy.
//   draft_entropy_kernel        H(q_j) of the draft rows, for the gate on the draft distribution.
//   shard_record_kernel         vocabulary-parallel form: a rank's statistics record for the first all-gather.
//   finalize_kernel             merges the per-CTA statistics:  logZ = m + ln s,  H = ln s - t/s  (entropy
//       definition of the HSD section, rearranged around the running maximum).
//   accept_sample_kernel        one cluster of CTAs, or one large CTA, per sequence: merges the statistics for its k+1 positions (warp
//       shuffles), applies the entropy gate and the ratio test in draft order, then makes one vectorised pass
//       over the logits row and the draft row of the first rejected position: residual max(0, p - q), per-chunk
//       sums, a scan, and the inverse-CDF pick with the supplied uniform.
//
// Every on-chip wait is bounded: when a wait runs out the CTA raises HOLA_FLAG_TIMEOUT, leaves its loops,
// releases its tensor memory and returns.

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <cooperative_groups.h>

#include <mutex>

#include "../../include/hola_verify.h"

namespace cg = cooperative_groups;

namespace {

// ------------------------------------------------------------------------------------------------ constants
constexpr int kBlockK = 64;                      // bf16 elements per K block = one 128-byte swizzle row
constexpr int kLanes = 128;                      // vocabulary rows per CTA per tile = tensor-memory lanes
constexpr int kPairTile = 2 * kLanes;            // vocabulary rows per CTA pair per tile
constexpr int kWBlockBytes = kLanes * kBlockK * 2;
constexpr int kMaxN = 256;                       // verify rows per MMA
constexpr int kMaxRowsPerPass = 2 * kMaxN;       // two MMAs per K step fill the 512 tensor-memory columns
constexpr int kEpiWarps = 16;                    // warps 2..17: tensor memory -> logits buffer + softmax statistics
constexpr int kK1Warps = 2 + kEpiWarps;          // warp 0 TMA, warp 1 MMA + tensor-memory owner
constexpr int kK1Threads = kK1Warps * 32;
constexpr int kEpiSlots = 4;                     // 32-column chunks of a tile one epilogue warp handles at most
constexpr int kTransRows = 16;                   // verify rows per transposition step of an epilogue warp
constexpr int kTransBytes = kTransRows * 32 * 4; // its staging buffer: [16 rows][32 vocabulary entries] fp32
// 8-bit and 4-bit W_lm, expanded on chip (mode 1): the codes of a K block land in the ring slot and converter warps
// expand them, through registers, into the bf16 operand in TENSOR MEMORY that the MMA reads (64 columns hold the 128
// channels of a K block, one lane per vocabulary row).  Warps 2..9 are epilogue warps, warps 10..17 convert: two groups
// of four warps (one per quarter of the tensor-memory lanes) take the K blocks in turn.  With at most 32 verify rows (one
// chunk per lane quarter) four epilogue warps do, and there are three groups of converters: the chain of one block, some
// 1600 cycles, then no longer bounds (whole step of one sequence, V = 32000, H = 4096: widths 20 / 70 / 10 % 39.3 -> 37.4 us).
constexpr int kExpandK = 128;                     // channels per K block of 4- and 8-bit rows (16-bit rows: kBlockK)
constexpr int kExpandMaxN = 192;                  // two accumulators of 192 columns leave 128 columns for the operand
constexpr int kOperandCols = kExpandK / 2;        // tensor-memory columns of one K block of the expanded operand
constexpr int kGroupRows = 256;                   // vocabulary rows per group of one width
constexpr int kSubBlock = 128;                    // hidden channels per 4-bit sub-block (one shared exponent each)
constexpr int kW8EpiWarps = 8, kW8FewEpiWarps = 4;
constexpr int kConvGroup = 4;                     // converter warps per K block: one per tensor-memory lane quarter
constexpr int kConvGroups = (kK1Warps - 2 - kW8EpiWarps) / kConvGroup, kConvGroupsFew = (kK1Warps - 2 - kW8FewEpiWarps) / kConvGroup;
// What the expansion leaves in the operand is the code times a power of two (see expand_*); the epilogue takes it out
// of the accumulators together with the row's scale.  Both are exact.
constexpr float kExpandUnscale8 = 64.f, kExpandUnscale4 = 1024.f;
constexpr int kTmemCols = 512;
constexpr int kMaxStages = 12;
constexpr int kMaxPaceGroups = 128;              // groups of CTA pairs of a launch that holds all passes
constexpr int kSmemBudget = 227 * 1024;          // dynamic shared memory per CTA on sm_100
constexpr int kBarrierBytes = 512;
constexpr long long kWaitLimitCycles = 4000000000ll;   // about 2 s of SM clock per wait, far above any legitimate wait

constexpr int kK3Threads = 256;
constexpr int kSoloThreads = 1024;               // its form with one CTA per sequence
constexpr int kFewEntries = 8192;                // vocabulary up to which half of them stay
constexpr int kK3MaxPerSm = 4;                   // CTAs of the accept/sample kernel an SM holds (register budget: 64 per thread)
constexpr int kChunk = 128;                      // vocabulary entries per warp step (32 lanes x 4)
constexpr int kMaxChunks = 4096;                 // => V <= 524288
constexpr int kMaxK1 = 64;                       // k + 1 <= 64
constexpr int kK3MaxDynSmem = 200 * 1024;        // rows staged in shared memory (kStaged)
constexpr int kK3Unroll = 4;                     // vocabulary chunks a warp has in flight per step

constexpr int kHqSlices = 8;                     // CTAs that share one draft row in draft_entropy_kernel

constexpr float kLog2e = 1.4426950408889634f, kLn2 = 0.6931471805599453f;

struct K1Params {
  int M;          // total verify rows B(k+1)
  int row0;       // first row of this pass
  int rows;       // rows of this pass (<= n_sub * N)
  int n_pass;     // > 1: all passes in this launch; CTA pair i works on pass i % n_pass (rows from row0 + that many
  int rows_per_pass;   // times rows_per_pass on) and shares the vocabulary tiles with the pairs i / n_pass, see the kernel
  int V, n_ptiles, n_kblocks, stages, nbuf;
  int n_sub, N;   // MMAs per K step and their N (verify rows each; multiple of 16)
  int rot;        // 1: three MMAs of N <= 128 per K step whose accumulators rotate over the four 128-column units
  int pair256;    // rot with N = 128 exactly: two of the three units of a tile are adjacent and take ONE MMA of N = 256
  int kpb;        // K blocks per ring slot (1, 2 or 4); > 1: the tensor maps are three-dimensional and one copy brings them all;
                  // a K block that H fills only in part then has a slot of its own, through two-dimensional maps (tmap_w4 of
                  // W_lm, tmap_w16 of the hidden rows)
  int k_tail;     // kpb > 1: 1 if there is such a block
  int acc_cols;   // tensor-memory columns from one accumulator buffer to the next
  int conv_groups, a_slots;   // (on-chip expansion) groups of converter warps that take part, K blocks of expanded operand
                              // that tensor memory holds (at most as many as ring slots)
  int tile_rows;  // vocabulary rows per CTA per tile (<= 128, multiple of 4): balances the tiles over the pairs
  int ldl;        // row pitch of the logits buffer, in floats
  const float* w_scale;   // 8-bit W_lm: fp32 scale per vocabulary row, applied to the accumulators
  const float* h_scale;   // 8-bit activations (modes 2, 3): fp32 scale per verify row (mode 3: of the coarse plane)
  const float* h_scale2;  // mode 3: scale of the second plane
  // Mode 1 with vocabulary groups of mixed width (null: every row is 8-bit and lives at its own index in W_lm): width
  // (4, 8 or 16) of each group of 256 vocabulary rows, first row of the group inside the buffer of its width, and the
  // exponents of the 4-bit sub-blocks, [sub-block][row of the 4-bit buffer].
  const uint8_t* group_width;
  const int* group_row;
  const uint8_t* shift4;
  int rows4;
  int want_arg;           // 1: the arg-max of every row is wanted too (greedy verifier, records of the vocabulary-parallel form)
  int clear_status;       // 1: the status word holds anything; CTA 0 clears it (what sets bits comes seconds later, when a
                          // wait runs out, or in a later kernel)
  int bulk_logits;        // (rotating units) 1: the logits buffer has a tensor map (rows of whole 16-byte pieces), full blocks
                          // leave by bulk stores
  int stream_logits;      // 1: store the logits with the streaming hint (they exceed what the L2 keeps until they are read)
  float* logits;      // null: nobody reads them, none are stored
  float4* partials;   // [M][part_stride] (m, s, t, arg-max index): a row's partials side by side, one per CTA of its pass
  int part_stride;
  unsigned* status;
  // What the accept/sample kernel behind this one will gather (null: nothing): draft tokens, uniforms and the entries
  // q_j(x_j), and all of q when it is small.  An idle warp asks for it early on, so that the chain of dependent reads there
  // finds it in the L2 instead of in DRAM.
  const int* next_tok;
  const float* next_u;
  const char* next_q;
  int next_n, next_q_elem;      // B * k; bytes per draft probability
  unsigned next_q_bytes;        // bytes of q to ask for whole (0: only the entries)
  const void* draft_q;          // draft-entropy gate (else null; not with rotating units): the epilogue warps make the pass over the draft rows while
  int draft_q_dtype, draft_units;   // the first tile's MMAs run; a unit is one slice of one row (draft_rows * kHqSlices)
  double* draft_part;
  int prefetch_blocks;  // K blocks of its first tile a CTA asks into the L2 before it waits for the kernel before
  unsigned* pace;     // n_pass > 1, several tiles: two words per group of pairs (zero at launch, and again at the end), by which
                      // the group keeps in step
};

struct K3Params {
  int B, k, V, ldl;
  const float* logits;
  const float4* partials;       // partial i of row r at [r * row_stride + i * part_stride]
  int nparts, row_stride, part_stride, combine;
  const int* tok;
  const void* q;
  int q_dtype;
  const float* q_tok;           // optional fp32 [B][k]: q_j(x_j) already gathered (then q is read at row n only)
  const void* q_far;            // optional: the same draft tensor in pinned HOST memory, as the device sees it; rows
  int q_far_from;               //   n >= q_far_from of a sequence are read from there (rows before it were copied to q)
  int inputs_settled;           // 1: launched right behind this call's own GEMM kernel, whose CTAs have waited for the
                                // kernel before the call: tokens, uniforms and draft probabilities may be read
                                // before this grid's dependency wait.  0: wait first.
  int phase;                    // 0: the whole step; 1: stop after the accept test (accept_len, statistics written);
                                // vocabulary-parallel form: 3: stop after the masses of row n inside this shard,
                                // 4: the draw, by the shard that holds the point u * R
  // Vocabulary-parallel form (shard_world > 0): V, logits and q cover this rank's V entries starting at v_offset;
  // draft tokens and next_tok are global indices below V_global.
  int shard_world, shard_rank, v_offset, V_global;
  const float* lx_all;          // [world] records, rec_stride floats apart: logit of x_j where its owner found it, else -inf
  int rec_stride;               // floats from one rank's record to the next
  double* mass_out;             // phase 3: [B][2] mass of max(0, p_n - q_n) and of p_n inside this shard
  const double* mass_all;       // phase 4: [world][B][2], the same from every rank
  const float* u;
  float tau;
  int gate_source;          // hola_gate_source
  int fallback;             // hola_fallback
  const double* hq_part;        // [B][k][kHqSlices] slice sums of q ln q, read when the draft entropy gates
  float* draft_entropy;         // [B][k] optional output of H(q_j)
  int* accept_len;
  int* next_tok;
  float* entropy;
  float* logZ;
  unsigned* status;
  unsigned* flags_out;      // optional [B], in host memory: every sequence's flags, with what is in the status word, by plain
                            // stores instead of OR-ing them into the status word
};

// ------------------------------------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ uint32_t cluster_cta_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Address, in the cluster's shared window, of the same shared-memory offset in CTA `rank` of this cluster.
__device__ __forceinline__ uint32_t map_to_cta(uint32_t smem_addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
// Execution barrier only: orders no memory operations.  For the end of the kernel, where the point is that the peer CTA
// has stopped using this CTA's barriers and tensor memory; a release here would make every thread wait until its last
// stores of logits (hundreds of KB per CTA) have drained to L2 before the CTA may leave.
__device__ __forceinline__ void cluster_sync_execution_only() {
  asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");
  asm volatile("barrier.cluster.wait;" ::: "memory");
}

// True in exactly one lane of a converged warp.  Unlike a lane-id test, the compiler knows that a single thread
// runs the guarded region, so TMA / tcgen05 operands can stay in uniform registers.
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile("{\n .reg .pred P;\n elect.sync _|P, 0xffffffff;\n selp.u32 %0, 1, 0, P;\n}" : "=r"(pred));
  return pred != 0;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Arrivals on a barrier that may live in the peer CTA (address from map_to_cta).  Default (CTA-scope release)
// semantics on purpose: a cluster-scope release here acts as a fence that waits for the thread's earlier
// outstanding operations and serialises the pipeline.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx_cluster(uint32_t cluster_bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cluster.b64 _, [%0], %1;" ::"r"(cluster_bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred P1;\n mbarrier.try_wait.parity.shared::cta.b64 P1, [%1], %2;\n selp.u32 %0, 1, 0, P1;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// One look, no waiting.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred P1;\n mbarrier.test_wait.parity.shared::cta.b64 P1, [%1], %2;\n selp.u32 %0, 1, 0, P1;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait.  Returns false when the CTA is aborting (this wait or another one ran out of time).
// The clock is the SM's cycle counter (cheap to read), looked at only every 256 unsuccessful polls.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag,
                                          unsigned* status, long long limit_cycles = kWaitLimitCycles) {
  if (mbar_try_wait(bar, parity)) return true;
  long long t0 = 0;
  uint32_t spins = 0;
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((++spins & 255u) == 0u) {
      if (*abort_flag) return false;
      const long long now = clock64();
      if (t0 == 0) t0 = now;
      if (now - t0 > limit_cycles) {
        *abort_flag = 1u;
        if (status) atomicOr(status, HOLA_FLAG_TIMEOUT);
        return false;
      }
    }
  }
}

// The same for a converged warp that polls together: no lane is singled out and nothing has to be handed round, which
// takes a wait that is satisfied already from about 300 to about 50 cycles.
__device__ __forceinline__ bool mbar_wait_together(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag,
                                                   unsigned* status) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  long long t0 = 0;
  uint32_t spins = 0;
  while (true) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    if ((++spins & 255u) == 0u) {
      const long long now = clock64();
      if (t0 == 0) t0 = now;
      const bool late = now - t0 > kWaitLimitCycles;
      if (late) {
        *abort_flag = 1u;
        if (status) atomicOr(status, HOLA_FLAG_TIMEOUT);
      }
      if (__any_sync(0xffffffffu, late || *abort_flag)) return false;
    }
  }
}

// Whole-warp form: lane 0 polls, every lane gets the same answer (and, through the shuffle, the same ordering).
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag,
                                               unsigned* status, long long limit_cycles = kWaitLimitCycles) {
  int r = 1;
  if ((threadIdx.x & 31) == 0) r = mbar_wait(bar, parity, abort_flag, status, limit_cycles) ? 1 : 0;
  r = __shfl_sync(0xffffffffu, r, 0);
  return r != 0;
}

__device__ __forceinline__ uint64_t l2_policy_evict_first() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ uint64_t l2_policy_evict_normal() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}

// 2-D tiled TMA load, global -> this CTA's shared memory.  The completion is counted on an mbarrier that may
// live in either CTA of the pair (cta_group::2 form); no multicast: each CTA fetches its own bytes.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t cluster_bar, int x, int y,
                                            uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%3, %4}], [%2], %5;"
      ::"r"(dst), "l"(map), "r"(cluster_bar), "r"(x), "r"(y), "l"(policy)
      : "memory");
}

// A block of 16 rows x 32 logits from its (128-byte-swizzled) staging buffer to the logits buffer.  The rows past the last
// one and the entries past the vocabulary fall outside the map and are dropped.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int x, int y, uint64_t policy) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group.L2::cache_hint [%0, {%2, %3}], [%1], %4;"
               ::"l"(map), "r"(src), "r"(x), "r"(y), "l"(policy)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Three-dimensional form: (element of a K block, row, K block).
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t cluster_bar, int row, int kb,
                                            uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%3, %4, %5}], [%2], %6;"
      ::"r"(dst), "l"(map), "r"(cluster_bar), "r"(0), "r"(row), "r"(kb), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap* map, int row, int kb, uint64_t policy) {
  asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile.L2::cache_hint [%0, {%1, %2, %3}], %4;"
               ::"l"(map), "r"(0), "r"(row), "r"(kb), "l"(policy)
               : "memory");
}
// The same box into the L2 only.  A hint: it moves nothing that the program can see, so it may run ahead of the kernel
// that this grid depends on even if that kernel writes the lines (the L2 is where writes land).
__device__ __forceinline__ void tma_prefetch_2d(const CUtensorMap* map, int x, int y, uint64_t policy) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile.L2::cache_hint [%0, {%1, %2}], %3;"
               ::"l"(map), "r"(x), "r"(y), "l"(policy)
               : "memory");
}
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p) : "memory"); }
__device__ __forceinline__ void bulk_prefetch_l2(const void* p, unsigned bytes) {      // both multiples of 16
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
// A table entry that the kernel before may still be writing, past the L1 (which must not keep what is read ahead of the
// dependency wait).
__device__ __forceinline__ int load_past_l1(const int* p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ int load_past_l1(const uint8_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u8 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return static_cast<int>(v);
}

// All passes in one launch: the pairs of a group read the same tile of W_lm, and only those that read it within the
// few tens of microseconds a line stays in the L2 are spared the trip to HBM.  So before a new tile every producer
// thread of the group counts itself in and waits, for a bounded time, until the others have done so too.  A pace
// maker, not a barrier: when the time is up the thread goes on, and nothing depends on the others having arrived.
constexpr long long kPaceLimitCycles = 60000;
__device__ __forceinline__ void keep_pace(unsigned* counter, unsigned target) {
  atomicAdd(counter, 1u);
  const long long t0 = clock64();
  while (true) {
    unsigned seen;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(counter) : "memory");
    if (seen >= target || clock64() - t0 > kPaceLimitCycles) break;
  }
}
// Behind its last tile: the last of the group's `members` leaves both of the group's words at zero for the next launch.
// (A memset ahead of the launch did so before: an operation of its own in the stream, which also keeps the launch from being put
// in place early.  us: 660 rows, V = 3920 28.7 -> 23.7, 196 rows of mixed widths, V = 2656 18.5 -> 13.9, which have one tile per
// pair and no pace at all; 765 8-bit rows, V = 22752 56.6 -> 50.6.)
__device__ __forceinline__ void leave_pace(unsigned* counter, unsigned members) {
  __threadfence();
  if (atomicAdd(counter + kMaxPaceGroups, 1u) == members - 1) {
    counter[kMaxPaceGroups] = 0u;
    *counter = 0u;
  }
}

// Programmatic dependent launch: the grid may have been started while the kernel before it in the stream was still
// running.  grid_dependency_wait returns once that kernel has completed and its writes are visible; it must precede
// every global-memory access of the calling thread that could touch what that kernel reads or writes.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Tensor memory of the CTA pair: executed by one warp of EACH CTA of the pair.
__device__ __forceinline__ void tmem_alloc(uint32_t holder_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(holder_smem), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// D[tmem of both CTAs] (+)= A[smem of both CTAs] * B[smem of both CTAs]^T.  bf16 inputs with fp32 accumulation
// (K = 16 per instruction) or, with kInt8, signed 8-bit inputs with int32 accumulation (K = 32 per instruction).
// Issued by one thread of the pair's leader CTA; descriptors are shared-memory offsets valid in both CTAs.
template <bool kInt8>
__device__ __forceinline__ void umma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                     uint32_t accumulate) {
  if (kInt8) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::2.kind::i8 [%0], %1, %2, %3, p;\n}"
        ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  } else {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}"
        ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  }
}
// The same with A in tensor memory: lane i of each CTA holds row i of its half of A, two bf16 channels per column.
__device__ __forceinline__ void umma_tmem_a(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n}"
      ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// The mbarrier at this shared-memory offset in BOTH CTAs of the pair gets one arrival once every MMA issued so far
// by this thread has completed.
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  const uint16_t mask = 3;
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"(mask)
               : "memory");
}

// 32 consecutive fp32 columns of this thread's tensor-memory lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// 32 words into 32 consecutive columns of this thread's tensor-memory lane (tmem_st_wait: they are there).
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]),
        "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]),
        "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// 16 consecutive 32-bit columns of this thread's tensor-memory lane, as raw words (no wait: the caller waits once
// for all loads it has issued).
__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Shared-memory matrix descriptor: K-major tile whose rows are 128 bytes, 128-byte swizzle, 8-row groups
// 1024 bytes apart (stride byte offset), descriptor version 1 (sm_100).
__device__ __forceinline__ uint64_t make_kmajor_sw128_desc(uint32_t smem_addr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((smem_addr & 0x3FFFFu) >> 4);      // start address, 16-byte units
  d |= static_cast<uint64_t>(1) << 16;                          // leading byte offset: unused with swizzled K-major
  d |= static_cast<uint64_t>(1024 >> 4) << 32;                  // stride byte offset
  d |= static_cast<uint64_t>(1) << 46;                          // version
  d |= static_cast<uint64_t>(2) << 61;                          // layout: 128-byte swizzle
  return d;
}

// Instruction descriptor, kind::f16: D fp32, A and B bf16, both K-major, M = 256 (the pair), N = n.
__device__ __forceinline__ uint32_t make_idesc_bf16_m256(uint32_t n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((256u >> 4) << 24);
}
// Instruction descriptor, kind::i8: D int32, A and B signed 8-bit, both K-major, M = 256, N = n (multiple of 32).
__device__ __forceinline__ uint32_t make_idesc_s8_m256(uint32_t n) {
  return (2u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((256u >> 4) << 24);
}

// ------------------------------------------------------------------------------------------------ softmax statistics
// Statistics of a set of logits around its maximum m:  s = sum e^(l-m),  t = sum e^(l-m) (l-m).
// logZ = m + ln s;  H = -sum p ln p = ln s - t/s.
struct Stats {
  float m, s, t;
  int arg;        // vocabulary index of the maximum (lowest index among equals): the greedy verifier's token
};
__device__ __forceinline__ Stats stats_empty() { return Stats{-CUDART_INF_F, 0.f, 0.f, 0x7fffffff}; }

__device__ __forceinline__ Stats stats_merge(Stats a, Stats b) {
  if (b.m == -CUDART_INF_F) return a;
  if (a.m == -CUDART_INF_F) return b;
  const float m = fmaxf(a.m, b.m);
  const float da = a.m - m, db = b.m - m;
  const float ea = __expf(da), eb = __expf(db);
  Stats r;
  r.m = m;
  r.s = ea * a.s + eb * b.s;
  r.t = ea * (a.t + da * a.s) + eb * (b.t + db * b.s);
  r.arg = a.m > b.m ? a.arg : (b.m > a.m ? b.arg : min(a.arg, b.arg));
  return r;
}

// Fold the first `n` (1..16) of sixteen logits into the running statistics; element i is vocabulary entry vocab0 + i.  The
// arg-max, a comparison and a selection per entry whenever a maximum moves, only where it is wanted.  (The read-out of the last
// tile is exposed, and in the first tiles a maximum moves in nearly every warp.  us, with it -> without: V = 32000, 5 rows
// 46.6 -> 46.4, mixed widths 34.9 -> 34.8; 80 rows, V = 11000 14.94 -> 14.83; 500 rows, V = 3000 26.3 -> 26.0; 384 rows,
// V = 32000 106.8 -> 106.1.)
template <bool kFull>
__device__ __forceinline__ void stats_fold16(const float* v, int n, int vocab0, int want_arg, Stats& st) {
  float cmax = v[0];
#pragma unroll
  for (int i = 1; i < 16; ++i)
    if (kFull || i < n) cmax = fmaxf(cmax, v[i]);
  if (cmax > st.m) {
    if (st.m != -CUDART_INF_F) {
      const float d = st.m - cmax;
      const float sc = ex2_approx(d * kLog2e);
      st.t = sc * (st.t + d * st.s);
      st.s *= sc;
    }
    st.m = cmax;
    if (want_arg) {
      int first = 0;
#pragma unroll
      for (int i = 15; i > 0; --i)
        if ((kFull || i < n) && v[i] == cmax) first = i;
      if (v[0] == cmax) first = 0;
      st.arg = vocab0 + first;
    }
  }
  const float m = st.m;
  const float mneg2 = -m * kLog2e;
  float s = st.s, t = st.t;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    if (kFull || i < n) {
      const float e = ex2_approx(fmaf(v[i], kLog2e, mneg2));
      s += e;
      t = fmaf(e, v[i] - m, t);
    }
  }
  st.s = s;
  st.t = t;
}

// Two fp32 values in one 64-bit register, for the packed fp32 instructions of sm_100 (two results per issue slot).
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t r, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(r));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// stats_fold16<true> with half the issue slots: the maximum by three-input comparisons, the exponents' arguments
// x = (l - m) log2 e, the sum of the exponentials and the sum of e * x two at a time.  The centred sum is ln 2 times the
// last one.  What the rounding of m log2 e puts on every x (up to 2^-24 |m|) then counts as a shift of the reference in s and
// t alike and leaves H = ln s - t / s alone.  (Taken as  sum e l - m sum e  the centred sum has a rounding error of that size
// relative to s: entropies of rows with logits of +-40 were 1.3e-6 off in the 2-norm at V = 1000 instead of 3e-7.)
__device__ __forceinline__ void stats_fold16_packed(const float* v, int vocab0, int want_arg, Stats& st) {
  const float c0 = max3(v[0], v[1], v[2]), c1 = max3(v[3], v[4], v[5]), c2 = max3(v[6], v[7], v[8]),
              c3 = max3(v[9], v[10], v[11]), c4 = max3(v[12], v[13], v[14]);
  const float cmax = fmaxf(max3(c0, c1, c2), max3(c3, c4, v[15]));
  if (cmax > st.m) {
    if (st.m != -CUDART_INF_F) {
      const float d = st.m - cmax;
      const float sc = ex2_approx(d * kLog2e);
      st.t = sc * (st.t + d * st.s);
      st.s *= sc;
    }
    st.m = cmax;
    if (want_arg) {
      int first = 0;
#pragma unroll
      for (int i = 15; i > 0; --i)
        if (v[i] == cmax) first = i;
      if (v[0] == cmax) first = 0;
      st.arg = vocab0 + first;
    }
  }
  const float m = st.m;
  const float mneg2 = -m * kLog2e;
  const uint64_t l2e = pack2(kLog2e, kLog2e), mn = pack2(mneg2, mneg2);
  uint64_t s2 = pack2(0.f, 0.f), a2 = pack2(0.f, 0.f);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint64_t xp = fma2(pack2(v[2 * j], v[2 * j + 1]), l2e, mn);
    float x0, x1;
    unpack2(xp, x0, x1);
    const uint64_t ep = pack2(ex2_approx(x0), ex2_approx(x1));
    s2 = add2(s2, ep);
    a2 = fma2(ep, xp, a2);
  }
  float sa, sb, aa, ab;
  unpack2(s2, sa, sb);
  unpack2(a2, aa, ab);
  st.s += sa + sb;
  st.t = fmaf(kLn2, aa + ab, st.t);
}

// Integer codes to bf16 without conversion instructions.  A byte u in the low half of a 16-bit lane, high half zero, IS
// the bf16 number u * 2^-133 (subnormal below 128, first binade above: the spacing is the same on both sides), so one
// packed multiply-add per two codes scales and centres them; every result is an integer of at most eight bits times a
// power of two, exact in bf16.
__device__ __forceinline__ uint32_t bf16x2_fma(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

// Sixteen int8 codes -> sixteen bf16 values code / 64, in channel order, two per word: with the sign bit flipped a byte
// is u = code + 128, and u 2^-133 * 2^127 - 2 = code / 64.  Three integer-pipe instructions and two multiply-adds per
// four codes.
__device__ __forceinline__ void expand_int8x16(const uint4 x, uint32_t* o) {
  const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t u = w[j] ^ 0x80808080u;
    o[2 * j] = bf16x2_fma(__byte_perm(u, 0u, 0x4140), 0x7F007F00u, 0xC000C000u);
    o[2 * j + 1] = bf16x2_fma(__byte_perm(u, 0u, 0x4342), 0x7F007F00u, 0xC000C000u);
  }
}

// Thirty-two 4-bit codes (two's complement nibbles, even channel in the low one) -> thirty-two bf16 values
// code * 2^(shift - 10): a byte goes into both 16-bit lanes, the low lane keeps its low nibble and the high lane its high
// nibble (sixteen times the code, which that lane's multiplier takes out), both with the sign bit flipped (code + 8).
// Two integer-pipe instructions and one multiply-add per two codes.
__device__ __forceinline__ void expand_int4x32(const uint4 x, uint32_t* o, uint32_t shift) {
  const uint32_t w[4] = {x.x, x.y, x.z, x.w};
  const uint32_t mul = ((250u + shift) << 7) | ((246u + shift) << 23);     // 2^(123 + shift), 2^(119 + shift)
  const uint32_t add1 = 0x8000u | ((120u + shift) << 7);                    // -2^(shift - 7) = -8 * 2^(shift - 10)
  const uint32_t add = add1 | (add1 << 16);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
#pragma unroll
    for (int b = 0; b < 4; ++b)
      o[4 * j + b] = bf16x2_fma((__byte_perm(w[j], 0u, 0x4040 + 0x101 * b) & 0x00F0000Fu) ^ 0x00800008u, mul, add);
  }
}

// A logit on its way to the buffer.  Only one verify row per sequence is ever read back (row accept_len, by the
// accept/sample kernel); when the buffer is much larger than the L2 the streaming hint lets the lines leave early
// instead of displacing what the next kernel reads.
__device__ __forceinline__ void store_logit(float* dst, float x, int streaming) {
  if (streaming) __stcs(dst, x);
  else *dst = x;
}

// One accumulator on its way to the logits buffer.  Mode 0: as is.  Mode 1: times the scale of the vocabulary row.
// Mode 2: the accumulator is an int32 (bit pattern in `acc`); times the scales of the vocabulary row and of the
// verify row.
template <int kMode>
__device__ __forceinline__ float scaled(float acc, float w_scale, const float* h_scale, int row) {
  if (kMode == 1) return acc * w_scale;
  if (kMode == 2) return static_cast<float>(__float_as_int(acc)) * (w_scale * h_scale[row]);
  return acc;
}

__device__ __forceinline__ float warp_max_f32(float x) {       // (of numbers; -inf among them)
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));       // (volatile: whole warps, stays where it is)
  return r;
}
__device__ __forceinline__ double warp_sum_f64(double x) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
  return x;
}

// ------------------------------------------------------------------------------------------------ draft entropy, a slice
// H(q) = -sum_v q ln q of a draft row: the gate value when the gate looks at the draft distribution, as the HSD section words
// it.  q is used as stored; entries with q <= 0 contribute nothing.
// q ln q for q > 0, else 0.  The fast logarithm (absolute error about 2^-21 near 1, a few ulp elsewhere) is
// ample here: every term is weighted by q <= 1 and the sum is compared at 1e-4.
__device__ __forceinline__ float qlnq(float a) { return a > 0.f ? a * __logf(a) : 0.f; }
__device__ __forceinline__ float qlnq8(const uint4 raw) {     // sum over eight bf16 values
  const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
  float part = 0.f;
#pragma unroll
  for (int j = 0; j < 4; ++j) part += qlnq(__uint_as_float(w[j] << 16)) + qlnq(__uint_as_float(w[j] & 0xFFFF0000u));
  return part;
}
__device__ __forceinline__ float qlnq4(const uint4 x) {        // sum over four fp32 values
  return (qlnq(__uint_as_float(x.x)) + qlnq(__uint_as_float(x.y))) + (qlnq(__uint_as_float(x.z)) + qlnq(__uint_as_float(x.w)));
}

// This thread's share (of `nthr`) of sum q ln q over slice `slice` of a row: the 16-byte pieces of the row are cut into
// kHqSlices runs; what lies before the first piece and behind the last goes to slice 0.
__device__ __noinline__ double draft_slice_sum(const void* q, int q_dtype, int V, size_t row, int slice, int tid, int nthr) {
  const bool half = q_dtype == HOLA_Q_BF16;
  const int elem = half ? 2 : 4, per16 = 16 / elem;
  const char* qr = static_cast<const char*>(q) + row * V * elem;
  const int head = min(V, static_cast<int>((16u - (reinterpret_cast<uintptr_t>(qr) & 15u)) & 15u) / elem);
  const int nvec = (V - head) / per16;
  const uint4* q16 = reinterpret_cast<const uint4*>(qr + head * elem);
  const int per = (nvec + kHqSlices - 1) / kHqSlices, end = min(nvec, (slice + 1) * per);
  constexpr int kInFlight = 4;                           // independent 16-byte loads per thread and step
  double acc = 0.0;
  int i = slice * per + tid;
  for (; i + (kInFlight - 1) * nthr < end; i += kInFlight * nthr) {
    uint4 raw[kInFlight];
#pragma unroll
    for (int u = 0; u < kInFlight; ++u) raw[u] = q16[i + u * nthr];
#pragma unroll
    for (int u = 0; u < kInFlight; ++u) acc += half ? qlnq8(raw[u]) : qlnq4(raw[u]);
  }
  for (; i < end; i += nthr) acc += half ? qlnq8(q16[i]) : qlnq4(q16[i]);
  if (slice == 0) {
    const int tail = head + nvec * per16;
    for (int n = tid; n < head + V - tail; n += nthr) {
      const int v = n < head ? n : tail + n - head;
      acc += qlnq(half ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(qr)[v]) : reinterpret_cast<const float*>(qr)[v]);
    }
  }
  return acc;
}

// ------------------------------------------------------------------------------------------------ K1
// Shared memory: `stages` ring slots of [W_lm block 128 x 64 | hidden block(s) n_sub x (N/2) x 64], then the
// barrier area.  Barriers (8 bytes each, offsets in the barrier area):
//   full[12]   @0    leader CTA's copy is the live one: 2 arrivals (one producer per CTA) + the bytes of both CTAs
//   empty[12]  @96   per CTA: the MMAs that read this slot have completed (commit, delivered to both CTAs)
//   tfull[2]   @192  per CTA: the accumulators of a tile are complete (commit, delivered to both CTAs)
//   tempty[4]  @208  leader's copy: all epilogue warps of the pair have read their accumulators (per buffer; per
//                    128-column unit when the accumulators rotate)
//   tensor-memory base @256, abort flag @260
//   on-chip expansion only: rawfull[12] @272 per CTA: the codes of the slot have landed.  full[] then counts the hidden
//   bytes (and, for 16-bit rows, their bytes) and one arrival per converter warp of the pair that owns the K block: the
//   operand is in tensor memory.
// After the barrier area (with rotating units before it): one transposition buffer of 2 KB (4 KB) per epilogue warp.
// kMode 3 is kMode 2 with every verify row present twice in the hidden operand (coarse 8-bit plane and the plane of
// its remainder, in alternating blocks of 32 rows): the epilogue adds the two int32 sums with their scales.
// kMode: 0 bf16 x bf16; 1 int8 W_lm expanded to bf16 on chip (exact); 2 int8 W_lm x int8 hidden on the 8-bit MMA
// kind (K blocks of 128 elements, so that a block is 128 bytes per row exactly as in mode 0; int32 accumulators).
// kRot: 257..384 rows per pass, three MMAs of N <= 128 per K step on rotating 128-column accumulator units (a
// specialisation of its own because its epilogue holds a different set of values in registers).
// kFew (mode 1): at most 32 verify rows, four epilogue warps and three groups of converters.
// (tmap_w4 is the map of the logits buffer with kRot.)
// kWide: logits leave the staging buffer 16 bytes per lane (see the epilogue).
template <int kMode, bool kRot, bool kFew = false, bool kWide = false>
__global__ void __launch_bounds__(kK1Threads, 1)
lm_head_entropy_kernel(const __grid_constant__ CUtensorMap tmap_hidden, const __grid_constant__ CUtensorMap tmap_w,
                       const __grid_constant__ CUtensorMap tmap_w4, const __grid_constant__ CUtensorMap tmap_w16,
                       const K1Params p) {
  constexpr bool kW8 = kMode == 1;
  constexpr bool kI8 = kMode >= 2;                       // both operands 8-bit, 8-bit MMA kind
  constexpr bool kTwoPlane = kMode == 3;                 // hidden rows as two 8-bit planes, 64 operand rows per 32 verify rows
  constexpr int kKStep = kI8 ? 2 * kBlockK : kBlockK;    // elements of K per ring slot
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;          // 128-byte swizzle wants 1024-byte aligned tiles
  uint8_t* smem = smem_raw + (base - raw);

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);   // same value in all lanes, and the compiler knows it
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_cta_rank();              // 0 = leader of the pair
  // One pass per launch: pair i of npairs takes the vocabulary tiles i, i + npairs, ...  All passes in one launch
  // (n_pass > 1): n_pass neighbouring pairs form a group that walks the same tiles at the same time, one pass of the
  // verify rows each, so that a tile of W_lm comes from HBM once and reaches the other pairs of the group out of the L2.
  const int pair_of_grid = blockIdx.x >> 1;
  const int pair = p.n_pass > 1 ? pair_of_grid / p.n_pass : pair_of_grid;          // which tiles
  const int npairs = p.n_pass > 1 ? (gridDim.x >> 1) / p.n_pass : gridDim.x >> 1;
  const int row0 = p.n_pass > 1 ? (pair_of_grid - pair * p.n_pass) * p.rows_per_pass : p.row0;
  const int rows = p.n_pass > 1 ? min(p.rows_per_pass, p.M - row0) : p.rows;
  const int half_n = p.N >> 1;                           // hidden rows this CTA supplies per MMA
  const uint32_t hid_block_bytes = static_cast<uint32_t>(half_n) * 128u;
  // Bytes of a K block's rows of W_lm in the slot (the MMA reads 128 rows from its start: what follows only reaches lanes
  // that hold nothing) and of the slot.
  const uint32_t w_block_bytes = kW8 || kRot ? kWBlockBytes : (static_cast<uint32_t>(p.tile_rows) * 128u + 1023u) & ~1023u;
  const uint32_t stage_bytes = kW8 ? kWBlockBytes + 2 * hid_block_bytes : p.kpb * (w_block_bytes + p.n_sub * hid_block_bytes);
  const int n_slots = kRot || kW8 || p.kpb == 1 ? p.n_kblocks        // slots' worth of K blocks per tile
                                                : (p.n_kblocks - p.k_tail + p.kpb - 1) / p.kpb + p.k_tail;
  const uint32_t hid_tx_bytes = p.n_sub * hid_block_bytes;
  const uint32_t tx_bytes = static_cast<uint32_t>(p.tile_rows) * 128u + hid_tx_bytes;   // bf16 W_lm: per CTA and slot
  const int code_blocks = (p.n_kblocks + 1) >> 1;        // (on-chip expansion) K blocks of a tile of 4- or 8-bit rows
  const int pair_rows = 2 * p.tile_rows;                 // vocabulary rows of a pair's tile
  constexpr int kWarpTransBytes = kRot ? 2 * kTransBytes : kTransBytes;   // rotating units: a whole 32-row chunk at once
  // Staging buffers: behind the barrier area; with rotating units before it, on 1024-byte boundaries, as the swizzle of the
  // bulk stores wants them.
  constexpr int kTransFirst = kRot ? kEpiWarps * kWarpTransBytes : 0;
  const uint32_t bar_off = p.stages * stage_bytes + kTransFirst;
  const uint32_t bar_base = base + bar_off;
  const uint32_t full_bar = bar_base, empty_bar = bar_base + 96, tfull_bar = bar_base + 192,
                 tempty_bar = bar_base + 208, rawfull_bar = bar_base + 272;
  constexpr int kNumEpi = kFew ? kW8FewEpiWarps : kW8 ? kW8EpiWarps : kEpiWarps;      // epilogue warps 2 .. 2 + kNumEpi - 1
  constexpr int kGroups = kNumEpi / 4;                        // warps per tensor-memory lane quarter
  float* trans_base = reinterpret_cast<float*>(smem + (kRot ? bar_off - kTransFirst : bar_off + kBarrierBytes));
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + bar_off + 256);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + bar_off + 260);

  if (threadIdx.x == 0) {
    for (int i = 0; i < p.stages; ++i) {
      mbar_init(full_bar + 8 * i, kW8 ? 2 + 2 * kConvGroup : 2);     // (+ the converter warps of a K block, both CTAs)
      mbar_init(empty_bar + 8 * i, 1);
      if (kW8) mbar_init(rawfull_bar + 8 * i, 1);
    }
    for (int i = 0; i < 2; ++i) mbar_init(tfull_bar + 8 * i, 1);
    for (int i = 0; i < 4; ++i) mbar_init(tempty_bar + 8 * i, 2 * kNumEpi);
    *abort_flag = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_hidden) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_w) : "memory");
  }
  __syncwarp();
  if (warp == 1) tmem_alloc(smem_u32(tmem_holder), kTmemCols);
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                                    // the peer's barriers are initialised too
  tc_fence_after();
  const uint32_t tmem_base = *tmem_holder;

  const int my_tiles = (p.n_ptiles - pair + npairs - 1) / npairs;
  const int sub_chunks = (p.N + 31) >> 5;                // 32-column chunks per MMA's accumulator
  // Accumulators.  rot == 0: MMA s of buffer b starts at column b * 256 + s * 256 (two buffers only when
  // n_sub == 1; with two MMAs the next tile waits until the whole tile has been read out).  rot == 1 (257..384 rows):
  // three MMAs of N <= 128; MMA s of tile t owns the 128-column unit (3 t + s) % 4, so a tile's first unit is always
  // free and its second and third are the first two the epilogue of the tile before it reads out: the tensor pipe
  // restarts after one epilogue round instead of after the whole read-out.

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (one per CTA)
    if (elect_one()) {
      // W_lm is streamed once.  (With all passes in one launch the other pairs of the group read the tile out of the L2
      // within microseconds, the group keeping in step; measured, the lines still do best as the first to be evicted:
      // they then never displace the hidden rows, which every pair re-reads for every tile.)
      const uint64_t pol_w = l2_policy_evict_first();
      const uint64_t pol_h = l2_policy_evict_last();     // hidden is re-read for every tile
      const uint32_t leader_full = map_to_cta(full_bar, 0);
      const uint32_t own_rawfull = map_to_cta(rawfull_bar, rank);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      // While the kernel before still runs (in a loop of calls: the accept/sample kernel, some 10 us of latency in which
      // HBM would idle), the first blocks of this CTA's rows move into the L2.
      if (p.prefetch_blocks > 0 && my_tiles > 0) {
        int width = 0, w_row = pair * pair_rows + static_cast<int>(rank) * p.tile_rows;
        if (kW8 && p.group_width) {
          width = load_past_l1(p.group_width + pair);
          w_row = load_past_l1(p.group_row + pair) + static_cast<int>(rank) * p.tile_rows;
        }
        const CUtensorMap* map = width == 4 ? &tmap_w4 : width == 16 ? &tmap_w16 : &tmap_w;
        const int step = width == 4 || width == 16 ? kBlockK : (kW8 ? kExpandK : kKStep);   // box width, in map elements
        if (!kRot && !kW8 && p.kpb > 1) {
          for (int kb = 0; kb < p.prefetch_blocks; kb += p.kpb) tma_prefetch_3d(map, w_row, kb, pol_w);
        } else
        for (int kb = 0; kb < p.prefetch_blocks; ++kb) tma_prefetch_2d(map, kb * step, w_row, pol_w);
      }
      grid_dependency_wait();                            // W_lm and the hidden rows may come from the kernel before
      if (p.clear_status && blockIdx.x == 0) *p.status = 0u;
      if (kW8) {
        // On-chip expansion: codes (or 16-bit rows as they are) and hidden rows of a K block into one slot, which is free
        // again once the MMAs of its previous use are done: those have waited for the converters.
        for (int t = 0; t < my_tiles && ok; ++t) {
          if (p.n_pass > 1 && p.pace && t > 0) keep_pace(p.pace + pair, static_cast<unsigned>(2 * p.n_pass * t));
          int tile_width = 8;                              // width of this tile's rows and where they are stored
          int w_row = (pair + t * npairs) * pair_rows + static_cast<int>(rank) * p.tile_rows;
          if (p.group_width) {
            const int g = pair + t * npairs;
            tile_width = p.group_width[g];
            w_row = p.group_row[g] + static_cast<int>(rank) * p.tile_rows;
          }
          const int h_row = row0 + static_cast<int>(rank) * half_n;
          const int n_blocks = tile_width == 16 ? p.n_kblocks : code_blocks;
          int kx = 0;
          for (int kb = 0; kb < n_blocks; ++kb) {
            if (!mbar_wait(empty_bar + 8 * stage, phase ^ 1u, abort_flag, p.status)) { ok = false; break; }
            const uint32_t sa = base + stage * stage_bytes;
            const uint32_t rb = own_rawfull + 8 * stage, fb = leader_full + 8 * stage;
            if (tile_width == 16) {                        // 16-bit rows: the tile the MMA reads from shared memory
              mbar_arrive(rawfull_bar + 8 * stage);        // (every barrier moves on by one phase per use of the slot)
              mbar_expect_tx_cluster(fb, tx_bytes);
              tma_load_2d(sa, &tmap_w16, fb, kx, w_row, pol_w);
              tma_load_2d(sa + kWBlockBytes, &tmap_hidden, fb, kx, h_row, pol_h);
              kx += kBlockK;
            } else {
              if (tile_width == 8) {                       // a byte per code: 128 bytes per row and K block
                mbar_expect_tx_cluster(rb, static_cast<uint32_t>(p.tile_rows) * 128u);
                tma_load_2d(sa, &tmap_w, rb, kx, w_row, pol_w);
              } else {                                     // two codes per byte: 64 bytes
                mbar_expect_tx_cluster(rb, static_cast<uint32_t>(p.tile_rows) * 64u);
                tma_load_2d(sa, &tmap_w4, rb, kx >> 1, w_row, pol_w);
              }
              mbar_expect_tx_cluster(fb, 2 * hid_block_bytes);
              tma_load_2d(sa + kWBlockBytes, &tmap_hidden, fb, kx, h_row, pol_h);
              tma_load_2d(sa + kWBlockBytes + hid_block_bytes, &tmap_hidden, fb, kx + kBlockK, h_row, pol_h);
              kx += kExpandK;
            }
            if (++stage == p.stages) { stage = 0; phase ^= 1u; }
          }
        }
      } else
      for (int t = 0; t < my_tiles && ok; ++t) {
        const int v0 = (pair + t * npairs) * pair_rows + static_cast<int>(rank) * p.tile_rows;
        if (p.n_pass > 1 && p.pace && t > 0) keep_pace(p.pace + pair, static_cast<unsigned>(2 * p.n_pass * t));
        if (!kRot && p.kpb > 1) {
          // Several K blocks per slot: one wait, one announcement and two copies for all of them.  A producer that does
          // this per K block needs some 450 cycles for it, which bounds narrow tiles (and tiles that are in the L2).
          const uint32_t hid_off = p.kpb * w_block_bytes;
          for (int i = 0; i < n_slots; ++i) {
            const uint32_t sa = base + stage * stage_bytes;
            if (!mbar_wait(empty_bar + 8 * stage, phase ^ 1u, abort_flag, p.status)) { ok = false; break; }
            const uint32_t fb = leader_full + 8 * stage;
            const int h_row = (kTwoPlane ? 2 : 1) * row0 + static_cast<int>(rank) * half_n;
            if (p.k_tail && i == n_slots - 1) {
              const int kx = (p.n_kblocks - 1) * kKStep;
              mbar_expect_tx_cluster(fb, tx_bytes);
              tma_load_2d(sa, &tmap_w4, fb, kx, v0, pol_w);
              tma_load_2d(sa + hid_off, &tmap_w16, fb, kx, h_row, pol_h);
            } else {
              mbar_expect_tx_cluster(fb, p.kpb * tx_bytes);
              tma_load_3d(sa, &tmap_w, fb, v0, i * p.kpb, pol_w);
              tma_load_3d(sa + hid_off, &tmap_hidden, fb, h_row, i * p.kpb, pol_h);
            }
            if (++stage == p.stages) { stage = 0; phase ^= 1u; }
          }
          continue;
        }
        int kx = 0;                                      // K coordinate of the block, in elements
        for (int kb = 0; kb < p.n_kblocks; ++kb, kx += kKStep) {
          const uint32_t sa = base + stage * stage_bytes;
          if (!mbar_wait(empty_bar + 8 * stage, phase ^ 1u, abort_flag, p.status)) { ok = false; break; }
          const uint32_t fb = leader_full + 8 * stage;
          mbar_expect_tx_cluster(fb, tx_bytes);
          tma_load_2d(sa, &tmap_w, fb, kx, v0, pol_w);
          if (kRot && p.pair256) {
            // Row blocks 0, 1, 2 (128 rows each) sit on units (3t, 3t+1, 3t+2) mod 4.  Two of them that are adjacent
            // without wrapping (blocks 0, 1, or blocks 1, 2 when the tile starts on unit 3) share one MMA of N = 256:
            // this CTA then supplies ONE of the two blocks whole, and its half of the third block as before.
            const bool late_pair = ((3 * t) & 3) == 3;
            const int pair_row = (late_pair ? 128 : 0) + static_cast<int>(rank) * 128;
            const int single_row = (late_pair ? 0 : 256) + static_cast<int>(rank) * 64;
            tma_load_2d(sa + kWBlockBytes, &tmap_hidden, fb, kx, row0 + pair_row, pol_h);
            tma_load_2d(sa + kWBlockBytes + hid_block_bytes, &tmap_hidden, fb, kx, row0 + pair_row + 64, pol_h);
            tma_load_2d(sa + kWBlockBytes + 2 * hid_block_bytes, &tmap_hidden, fb, kx, row0 + single_row, pol_h);
          } else {
            for (int s = 0; s < p.n_sub; ++s)
              tma_load_2d(sa + w_block_bytes + s * hid_block_bytes, &tmap_hidden, fb, kx,
                          (kTwoPlane ? 2 : 1) * row0 + s * p.N + static_cast<int>(rank) * half_n, pol_h);
          }
          if (++stage == p.stages) { stage = 0; phase ^= 1u; }
        }
      }
      if (p.n_pass > 1 && p.pace && my_tiles > 1) leave_pace(p.pace + pair, static_cast<unsigned>(2 * p.n_pass));
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (leader CTA only)
    if (rank == 1 && p.next_tok) {
      grid_dependency_wait();
      const int w = pair_of_grid, nw = gridDim.x >> 1;
      for (int i = w * 32 + lane; i < p.next_n; i += nw * 32) {
        const int x = p.next_tok[i];
        prefetch_l2(p.next_u + i);
        if (x >= 0 && x < p.V) prefetch_l2(p.next_q + (static_cast<size_t>(i) * p.V + x) * p.next_q_elem);
      }
      if (p.next_q_bytes && lane == 0) {
        const unsigned piece = ((p.next_q_bytes + nw - 1) / nw + 15u) & ~15u, at = piece * w;
        if (at < p.next_q_bytes) bulk_prefetch_l2(p.next_q + at, min(piece, p.next_q_bytes - at));
      }
    }
    if (rank == 0 && elect_one()) {
      const uint32_t idesc = kI8 ? make_idesc_s8_m256(static_cast<uint32_t>(p.N))
                                 : make_idesc_bf16_m256(static_cast<uint32_t>(p.N));
      const uint32_t idesc_pair = kI8 ? make_idesc_s8_m256(256u) : make_idesc_bf16_m256(256u);
      const uint64_t desc0 = make_kmajor_sw128_desc(base);
      const bool two_mmas = p.n_sub == 2;
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      if (kRot) {
        uint32_t used = 0;                               // bit u: parity of the number of tiles that used unit u
        for (int t = 0; t < my_tiles && ok; ++t) {
          for (int kb = 0; kb < p.n_kblocks && ok; ++kb) {
            if (!mbar_wait(full_bar + 8 * stage, phase, abort_flag, p.status)) { ok = false; break; }
            tc_fence_after();
            const uint64_t adesc = desc0 + ((stage * stage_bytes) >> 4);
            const uint64_t bdesc0 = adesc + (kWBlockBytes >> 4);
            if (p.pair256) {
              // one MMA of N = 256 over the two adjacent units, one of N = 128 over the third: the W_lm block is read
              // from shared memory twice per K step instead of three times
              const uint32_t a0 = static_cast<uint32_t>(3 * t) & 3u;
              const bool late_pair = a0 == 3u;
              const uint32_t unit_pair = late_pair ? 0u : a0, unit_single = late_pair ? 3u : ((a0 + 2u) & 3u);
              if (kb == 0) {                             // the epilogue must have read these units' previous tiles
#pragma unroll
                for (int u = 0; u < 3; ++u) {
                  const uint32_t unit = (a0 + u) & 3u;
                  const uint32_t par = (used >> unit) & 1u;
                  if (!mbar_wait(tempty_bar + 8 * unit, par ^ 1u, abort_flag, p.status)) { ok = false; break; }
                  used ^= 1u << unit;
                }
                if (!ok) break;
                tc_fence_after();
              }
              const uint32_t acc = kb != 0 ? 1u : 0u;
              const uint32_t dp = tmem_base + unit_pair * 128u, ds = tmem_base + unit_single * 128u;
              const uint64_t bdesc_s = bdesc0 + 2 * (hid_block_bytes >> 4);
#pragma unroll
              for (int kk = 0; kk < kBlockK / 16; ++kk) {
                umma<kI8>(dp, adesc + 2 * kk, bdesc0 + 2 * kk, idesc_pair, kk == 0 ? acc : 1u);
                umma<kI8>(ds, adesc + 2 * kk, bdesc_s + 2 * kk, idesc, kk == 0 ? acc : 1u);
              }
            } else
#pragma unroll
            for (int u = 0; u < 3; ++u) {
              const uint32_t unit = static_cast<uint32_t>(3 * t + u) & 3u;
              if (kb == 0) {                             // the epilogue must have read this unit's previous tile
                const uint32_t par = (used >> unit) & 1u;
                if (!mbar_wait(tempty_bar + 8 * unit, par ^ 1u, abort_flag, p.status)) { ok = false; break; }
                used ^= 1u << unit;
                tc_fence_after();
              }
              const uint32_t d = tmem_base + unit * 128u;
              const uint64_t bdesc = bdesc0 + u * (hid_block_bytes >> 4);
              umma<kI8>(d, adesc, bdesc, idesc, kb != 0 ? 1u : 0u);
#pragma unroll
              for (int kk = 1; kk < kBlockK / 16; ++kk) umma<kI8>(d, adesc + 2 * kk, bdesc + 2 * kk, idesc, 1u);
            }
            if (!ok) break;
            umma_commit_pair(empty_bar + 8 * stage);
            if (++stage == p.stages) { stage = 0; phase ^= 1u; }
          }
          if (ok) umma_commit_pair(tfull_bar);           // all three units of this tile are complete in both CTAs
        }
      } else
      if (kW8) {
        // A K block's operand is in tensor memory (4- and 8-bit rows) or in the slot's shared memory (16-bit rows); in
        // either case the converters report for it, so that all barriers move on block by block.
        const uint32_t operand0 = tmem_base + 2 * p.acc_cols;
        int aslot = 0;
        bool ready = false;                                // the next block has been seen complete
        if (p.group_width) grid_dependency_wait();         // the width table may come from the kernel before
        int width_next = p.group_width && my_tiles > 0 ? p.group_width[pair] : 8;
        for (int t = 0; t < my_tiles && ok; ++t) {
          const int buf = t & 1;
          const uint32_t acc_phase = static_cast<uint32_t>(t >> 1) & 1u;
          const bool in_smem = width_next == 16;
          if (p.group_width && t + 1 < my_tiles) width_next = p.group_width[pair + (t + 1) * npairs];
          if (!mbar_wait(tempty_bar + 8 * buf, acc_phase ^ 1u, abort_flag, p.status)) { ok = false; break; }
          tc_fence_after();
          const uint32_t d0 = tmem_base + buf * p.acc_cols;
          const int n_blocks = in_smem ? p.n_kblocks : code_blocks;
          for (int kb = 0; kb < n_blocks; ++kb) {
            if (!ready && !mbar_wait(full_bar + 8 * stage, phase, abort_flag, p.status)) { ok = false; break; }
            // a look at the next block's barrier, whose answer (some 90 cycles) arrives while this block's MMAs are issued
            const int next = stage + 1 == p.stages ? 0 : stage + 1;
            ready = mbar_test(full_bar + 8 * next, next ? phase : phase ^ 1u);
            tc_fence_after();
            const uint64_t adesc = desc0 + ((stage * stage_bytes) >> 4);
            const uint64_t bdesc = adesc + (kWBlockBytes >> 4);
            const uint32_t acc = kb != 0 ? 1u : 0u;
            if (in_smem) {
              umma<false>(d0, adesc, bdesc, idesc, acc);
#pragma unroll
              for (int kk = 1; kk < kBlockK / 16; ++kk) umma<false>(d0, adesc + 2 * kk, bdesc + 2 * kk, idesc, 1u);
            } else {
              const uint32_t a = operand0 + aslot * kOperandCols;
              umma_tmem_a(d0, a, bdesc, idesc, acc);
#pragma unroll
              for (int kk = 1; kk < kBlockK / 16; ++kk) umma_tmem_a(d0, a + 8 * kk, bdesc + 2 * kk, idesc, 1u);
              const uint64_t bdesc2 = bdesc + (hid_block_bytes >> 4);
#pragma unroll
              for (int kk = 0; kk < kBlockK / 16; ++kk)
                umma_tmem_a(d0, a + kBlockK / 2 + 8 * kk, bdesc2 + 2 * kk, idesc, 1u);
            }
            umma_commit_pair(empty_bar + 8 * stage);
            if (++stage == p.stages) { stage = 0; phase ^= 1u; }
            if (++aslot == p.a_slots) aslot = 0;
          }
          if (ok) umma_commit_pair(tfull_bar + 8 * buf);
        }
      } else
      for (int t = 0; t < my_tiles && ok; ++t) {
        const int buf = t % p.nbuf;
        const uint32_t acc_phase = static_cast<uint32_t>(t / p.nbuf) & 1u;
        if (!mbar_wait(tempty_bar + 8 * buf, acc_phase ^ 1u, abort_flag, p.status)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d0 = tmem_base + buf * 256;
        for (int kb = 0; kb < n_slots; ++kb) {
          if (!mbar_wait(full_bar + 8 * stage, phase, abort_flag, p.status)) { ok = false; break; }
          tc_fence_after();
          // descriptors of this slot: only the 14-bit address field changes (16-byte units)
          const uint64_t adesc = desc0 + ((stage * stage_bytes) >> 4);
          const uint64_t bdesc0 = adesc + ((p.kpb * w_block_bytes) >> 4);
          const uint32_t acc = kb != 0 ? 1u : 0u;
          // 16 bf16 = 32 bytes further along K inside the swizzled row: +2 in 16-byte address units
          if (two_mmas) {
            const uint64_t bdesc1 = bdesc0 + (hid_block_bytes >> 4);
            umma<kI8>(d0, adesc, bdesc0, idesc, acc);
            umma<kI8>(d0 + 256, adesc, bdesc1, idesc, acc);
#pragma unroll
            for (int kk = 1; kk < kBlockK / 16; ++kk) {
              umma<kI8>(d0, adesc + 2 * kk, bdesc0 + 2 * kk, idesc, 1u);
              umma<kI8>(d0 + 256, adesc + 2 * kk, bdesc1 + 2 * kk, idesc, 1u);
            }
          } else {
            umma<kI8>(d0, adesc, bdesc0, idesc, acc);
#pragma unroll
            for (int kk = 1; kk < kBlockK / 16; ++kk) umma<kI8>(d0, adesc + 2 * kk, bdesc0 + 2 * kk, idesc, 1u);
            // (whole K blocks past the last one are zeros in both operands)
            const int blocks = p.k_tail && kb == n_slots - 1 ? 1 : p.kpb;
            for (int n = 1; n < blocks; ++n) {
              const uint64_t an = adesc + n * (w_block_bytes >> 4), bn = bdesc0 + n * (hid_block_bytes >> 4);
#pragma unroll
              for (int kk = 0; kk < kBlockK / 16; ++kk) umma<kI8>(d0, an + 2 * kk, bn + 2 * kk, idesc, 1u);
            }
          }
          umma_commit_pair(empty_bar + 8 * stage);       // frees the slot in both CTAs once these MMAs have read it
          if (++stage == p.stages) { stage = 0; phase ^= 1u; }
        }
        if (ok) umma_commit_pair(tfull_bar + 8 * buf);   // accumulators of this tile are complete in both CTAs
      }
    }
  } else if (warp < 2 + kNumEpi) {
    // ------------------------------------------------------------------ epilogue warps
    // Tensor memory -> registers (thread = vocabulary entry, register = verify row) -> logits buffer, and the same
    // values, transposed through a small shared-memory buffer 16 rows at a time (thread = verify row and half of the
    // warp's 32 vocabulary entries), into thread-private softmax statistics that live in registers for the whole
    // kernel.  A warp owns one lane quarter (fixed by its id) and every kGroups-th 32-column chunk (with rotating
    // accumulators: chunk `group` of every unit, so that all warps read unit after unit and free each at once).
    const int quarter = warp & 3;                        // tensor-memory lanes 32*quarter .. +31
    const int group = (warp - 2) >> 2;
    const uint32_t leader_tempty = map_to_cta(tempty_bar, 0);
    const int n_chunks = p.n_sub * sub_chunks;
    constexpr bool rot = kRot;
    const int my_chunks = rot ? (group < sub_chunks ? p.n_sub : 0)
                              : (group < n_chunks ? (n_chunks - 1 - group) / kGroups + 1 : 0);
    float* tbuf = trans_base + (warp - 2) * (kWarpTransBytes / 4);
    const int trow = lane & 15, thalf = lane >> 4;       // row of a transposition step; which 16 of the 32 entries
    // Rotating units: logits leave by bulk stores out of the staging buffer, 16 rows each, where the lane quarter is all this
    // CTA's (rows past the last one fall outside the map; a pass ends on a multiple of 16); otherwise lane by lane.  The 32
    // store instructions of a chunk, their addresses and their way through the L1 bound the read-out of a tile, which a
    // small H does not hide: us, 384 rows, V = 32000, H = 128 29.9 -> 25.7, 512 34.8 -> 32.9 (8-bit 40.7 -> 37.1),
    // 4096 110.4 -> 108.5; 2304 rows, V = 128256, H = 8192 3715 -> 3685.  (With at most 256 rows the read-out hides under the
    // next tile, and its bulk stores stand in the way of the next tile's loads: one sequence 47.3 -> 49.0, 240 rows 79 -> 86, 192 rows
    // at 8 bits 136 -> 147.)
    // kWide: they leave out of the staging buffer too, 16 bytes per lane, and half of the warps fold their statistics first and
    // store then: in step, all sixteen wait for the store path (1400 cycles per chunk) and then for the exponentials (1400).
    // From 128 rows on; fewer leave too little to store for the longer code (us, V = 32000: 240 rows, H = 512 25.8 -> 25.3, 1024
    // 33.5 -> 32.7, 4096 80.8 -> 79.8; 96 rows 18.7 -> 18.9, one sequence 47.4 -> 47.8).
    const bool bulk = kRot && p.bulk_logits && quarter * 32 + 32 <= p.tile_rows;
    const uint32_t tbuf_addr = smem_u32(tbuf);
    const uint64_t pol_l = p.stream_logits ? l2_policy_evict_first() : l2_policy_evict_normal();
    constexpr int kSlots = kFew ? 1 : (kRot || kW8) ? 3 : kEpiSlots;   // chunks per tile this warp keeps statistics for
    Stats st[kSlots][2];
#pragma unroll
    for (int i = 0; i < kSlots; ++i) { st[i][0] = stats_empty(); st[i][1] = stats_empty(); }
    bool ok = true;
    grid_dependency_wait();                              // the logits buffer may still be read by the kernel before
    if (!kRot && p.draft_q) {
      // Nothing else for these warps to do until the first tile is complete.
      for (int u = blockIdx.x + static_cast<int>(gridDim.x) * (warp - 2); u < p.draft_units; u += gridDim.x * kNumEpi) {
        const double sum = warp_sum_f64(draft_slice_sum(p.draft_q, p.draft_q_dtype, p.V, u / kHqSlices, u % kHqSlices, lane, 32));
        if (lane == 0) p.draft_part[u] = sum;
      }
    }
    for (int t = 0; t < my_tiles && ok; ++t) {
      // (one buffer or two.  What depends on the tile alone is worked out, and loaded, ahead of the wait; with 8-bit hidden rows
      // behind it: there it would be spilled)
      constexpr bool kAhead = !kI8 || kRot;
      const int buf = p.nbuf == 2 ? t & 1 : 0;
      const uint32_t acc_phase = static_cast<uint32_t>(p.nbuf == 2 ? t >> 1 : t) & 1u;
      if (!kAhead) {
        if (!mbar_wait_warp(tfull_bar + 8 * buf, acc_phase, abort_flag, p.status)) { ok = false; break; }
        tc_fence_after();
      }
      const int vbase = (pair + t * npairs) * pair_rows + static_cast<int>(rank) * p.tile_rows;
      const int tile_lane = quarter * 32 + lane;         // lanes at or beyond tile_rows hold nothing
      const int vocab = vbase + tile_lane;
      const bool vocab_ok = tile_lane < p.tile_rows && vocab < p.V;
      // vocabulary entries of this quarter that exist (a prefix of its 32 lanes), and of this thread's 16
      const int nv = max(0, min(32, min(p.tile_rows, p.V - vbase) - quarter * 32));
      const int n16 = max(0, min(16, nv - thalf * 16));
      const int vocab16 = vbase + quarter * 32 + thalf * 16;
      float w_scale = ((kW8 || kI8) && vocab_ok) ? p.w_scale[vocab] : 1.f;   // 8-bit W_lm: the row's scale
      if (kW8) {                                         // and the power of two the expansion put in (exact)
        const int width = p.group_width ? p.group_width[pair + t * npairs] : 8;
        w_scale *= width == 8 ? kExpandUnscale8 : (width == 4 ? kExpandUnscale4 : 1.f);
      }
      const uint32_t lane_addr = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
      if (kAhead) {
        if (!mbar_wait_warp(tfull_bar + 8 * buf, acc_phase, abort_flag, p.status)) { ok = false; break; }
        tc_fence_after();
      }
      if (kTwoPlane) {
        // Two planes: 64 consecutive accumulator columns hold the coarse-plane sums (first 32) and the remainder-plane
        // sums (last 32) of the same 32 verify rows.  Read 16 + 16 columns at a time, add them with their scales, and
        // go on as in the other modes (16 rows are exactly one transposition step).
        const int n_pairs = p.n_sub * p.N / 64;
        const int my_pairs = group < n_pairs ? (n_pairs - 1 - group) / kGroups + 1 : 0;
        if (my_pairs == 0) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(leader_tempty + 8 * buf);
        }
#pragma unroll
        for (int slot = 0; slot < 2; ++slot) {
          if (slot < my_pairs) {
            const int pr = group + slot * kGroups;
            const int sub = 64 * pr >= p.N ? 1 : 0, col = 64 * pr - sub * p.N;      // (at most two MMAs)
            const uint32_t taddr = lane_addr + buf * 256 + sub * 256 + col;
            const int vr0 = row0 + 32 * pr;            // verify row of the pair's first column
            const int n_ok = min(32, p.M - vr0);
#pragma unroll
            for (int half = 0; half < 2; ++half) {
              uint32_t a[16], c[16];
              __syncwarp();
              tmem_ld16_nowait(taddr + 16 * half, a);
              tmem_ld16_nowait(taddr + 32 + 16 * half, c);
              tmem_ld_wait();
              if (slot == my_pairs - 1 && half == 1) {   // this warp's accumulators may be overwritten
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(leader_tempty + 8 * buf);
              }
              const int rows_here = n_ok - 16 * half;    // real rows among these 16
              if (rows_here > 0) {
                float f[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                  f[i] = 0.f;
                  if (i < rows_here) {
                    const int r = vr0 + 16 * half + i;
                    f[i] = fmaf(static_cast<float>(static_cast<int>(c[i])), w_scale * p.h_scale2[r],
                                static_cast<float>(static_cast<int>(a[i])) * (w_scale * p.h_scale[r]));
                  }
                }
                if (vocab_ok && p.logits) {
                  float* dst = p.logits + static_cast<size_t>(vr0 + 16 * half) * p.ldl + vocab;
#pragma unroll
                  for (int i = 0; i < 16; ++i)
                    if (i < rows_here) store_logit(dst + static_cast<size_t>(i) * p.ldl, f[i], p.stream_logits);
                }
                if (nv > 0) {
                  __syncwarp();
#pragma unroll
                  for (int i = 0; i < kTransRows; ++i)
                    tbuf[i * 32 + ((((lane >> 2) ^ (i & 7))) << 2) + (lane & 3)] = f[i];
                  __syncwarp();
                  float e[16];
#pragma unroll
                  for (int jj = 0; jj < 4; ++jj) {
                    const float4 x = *reinterpret_cast<const float4*>(
                        tbuf + trow * 32 + (((thalf * 4 + jj) ^ (trow & 7)) << 2));
                    e[4 * jj] = x.x; e[4 * jj + 1] = x.y; e[4 * jj + 2] = x.z; e[4 * jj + 3] = x.w;
                  }
                  if (n16 == 16) stats_fold16_packed(e, vocab16, p.want_arg, st[slot][half]);
                  else if (n16 > 0) stats_fold16<false>(e, n16, vocab16, p.want_arg, st[slot][half]);
                }
              }
            }
          }
        }
        continue;
      }
      if (my_chunks == 0) {                              // nothing to read: the accumulators are free as far as this
        tc_fence_before();                               // warp is concerned
        __syncwarp();
        if (lane == 0) {
          if (rot) {
            for (int u = 0; u < p.n_sub; ++u) mbar_arrive_cluster(leader_tempty + 8 * ((3 * t + u) & 3));
          } else {
            mbar_arrive_cluster(leader_tempty + 8 * buf);
          }
        }
      }
      if (kRot) {
        // Rotating units.  The next tile's MMAs wait for this tile's first two units, so a unit is read and handed back
        // as early as possible: a chunk goes from the registers to the logits buffer and, whole, into the warp's
        // 4 KB staging buffer; the registers then take the next unit's chunk at once, and the statistics of the chunk
        // before are folded from the staging buffer while that unit is already free.
        if (my_chunks > 0) {
          float v[32];
          __syncwarp();
          tmem_ld32(lane_addr + ((3 * t) & 3) * 128 + group * 32, v);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(leader_tempty + 8 * ((3 * t) & 3));
#pragma unroll
          for (int slot = 0; slot < 3; ++slot) {
            const int c0 = group * 32;                   // first column of the chunk inside its MMA
            const int r0 = row0 + slot * p.N + c0;     // verify row of column c0
            const int n_ok = min(32, min(p.N - c0, p.M - r0));   // columns that are real rows
            if (n_ok > 0) {
#pragma unroll
              for (int i0 = 0; i0 < 32; i0 += 8) {
#pragma unroll
                for (int i = i0; i < i0 + 8; ++i)
                  if (i < n_ok) v[i] = scaled<kMode>(v[i], w_scale, p.h_scale, r0 + i);
                if (kMode >= 2) asm volatile("" ::: "memory");   // the row scales eight at a time, not all 32 ahead
              }
              if (vocab_ok && !bulk && p.logits) {
                float* dst = p.logits + static_cast<size_t>(r0) * p.ldl + vocab;
#pragma unroll
                for (int i = 0; i < 32; ++i)
                  if (i < n_ok) store_logit(dst + static_cast<size_t>(i) * p.ldl, v[i], p.stream_logits);
              }
            }
            const bool out = bulk && n_ok > 0 && nv > 0;
            if (bulk && lane == 0) bulk_wait_read();     // (the stores of the chunk before have left the buffer)
            const bool fold = n_ok > 0 && nv > 0;
            __syncwarp();                                // every lane has folded the chunk before out of the buffer
            if (fold) {
              // two blocks of 16 rows, each laid out as in the 16-row scheme: entry (row i, vocabulary lane l) at
              // 16-byte group (l / 4) ^ (i % 8) of row i
#pragma unroll
              for (int i = 0; i < 32; ++i)
                tbuf[i * 32 + ((((lane >> 2) ^ (i & 7))) << 2) + (lane & 3)] = v[i];
              if (out) fence_async_shared();
            }
            __syncwarp();
            if (out && lane == 0) {
              tma_store_2d(&tmap_w4, tbuf_addr, vbase + quarter * 32, r0, pol_l);
              if (n_ok > kTransRows)
                tma_store_2d(&tmap_w4, tbuf_addr + kTransBytes, vbase + quarter * 32, r0 + kTransRows, pol_l);
              bulk_commit();
            }
            if (slot < 2) {                              // the registers are free: take the next unit's chunk, free the unit
              const int unit = (3 * t + slot + 1) & 3;
              tmem_ld32(lane_addr + unit * 128 + group * 32, v);
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive_cluster(leader_tempty + 8 * unit);
            }
            if (fold) {
#pragma unroll
              for (int half = 0; half < 2; ++half) {
                if (half * kTransRows < n_ok) {
                  float e[16];
#pragma unroll
                  for (int jj = 0; jj < 4; ++jj) {
                    const float4 x = *reinterpret_cast<const float4*>(
                        tbuf + (half * kTransRows + trow) * 32 + (((thalf * 4 + jj) ^ (trow & 7)) << 2));
                    e[4 * jj] = x.x; e[4 * jj + 1] = x.y; e[4 * jj + 2] = x.z; e[4 * jj + 3] = x.w;
                  }
                  if (n16 == 16) stats_fold16_packed(e, vocab16, p.want_arg, st[slot][half]);
                  else if (n16 > 0) stats_fold16<false>(e, n16, vocab16, p.want_arg, st[slot][half]);
                }
              }
            }
          }
        }
        continue;
      }
#pragma unroll
      for (int slot = 0; slot < kSlots; ++slot) {
        if (slot < my_chunks) {
          const int ch = group + slot * kGroups;
          const int sub = kI8 ? ch / sub_chunks : ch >= sub_chunks ? 1 : 0, j = ch - sub * sub_chunks;      // (at most two MMAs)
          float v[32];
          __syncwarp();                                  // tcgen05.ld is warp-collective: reconverge first
          tmem_ld32(lane_addr + (kW8 ? buf * p.acc_cols : buf * 256 + sub * 256) + j * 32, v);
          if (slot == my_chunks - 1) {                   // this warp's accumulators may be overwritten
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(leader_tempty + 8 * buf);
          }
          const int c0 = j * 32;                         // first column of the chunk inside its MMA
          const int r0 = row0 + sub * p.N + c0;        // verify row of column c0
          const int n_ok = min(32, min(p.N - c0, p.M - r0));   // columns that are real rows
          if (n_ok > 0) {
#pragma unroll
            for (int i0 = 0; i0 < 32; i0 += 8) {
#pragma unroll
              for (int i = i0; i < i0 + 8; ++i)
                if (i < n_ok) v[i] = scaled<kMode>(v[i], w_scale, p.h_scale, r0 + i);
              if (kMode >= 2) asm volatile("" ::: "memory");     // the row scales eight at a time, not all 32 ahead
            }
            if (vocab_ok && !kWide && p.logits) {
              float* dst = p.logits + static_cast<size_t>(r0) * p.ldl + vocab;
              if (n_ok == 32 && p.stream_logits) {       // (the common cases without a test per store)
#pragma unroll
                for (int i = 0; i < 32; ++i) __stcs(dst + static_cast<size_t>(i) * p.ldl, v[i]);
              } else if (n_ok == 32) {
#pragma unroll
                for (int i = 0; i < 32; ++i) dst[static_cast<size_t>(i) * p.ldl] = v[i];
              } else {                                   // (left at the last row: small batches have few, and wait for this)
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                  if (!kI8 && i >= n_ok) break;          // (8-bit hidden rows: that, and the selection above, would spill)
                  if (!kI8 || i < n_ok) store_logit(dst + static_cast<size_t>(i) * p.ldl, v[i], p.stream_logits);
                }
              }
            }
            if (nv > 0) {
#pragma unroll
              for (int half = 0; half < 2; ++half) {
                if (half * kTransRows < n_ok) {
                  // entry (row i, vocabulary lane l) at 16-byte group (l / 4) ^ (i % 8) of row i: stores of one
                  // row and the 16-byte loads of eight neighbouring rows both touch every bank once
                  __syncwarp();
#pragma unroll
                  for (int i = 0; i < kTransRows; ++i)
                    tbuf[i * 32 + ((((lane >> 2) ^ (i & 7))) << 2) + (lane & 3)] = v[half * kTransRows + i];
                  __syncwarp();
                  auto put = [&]() {                     // the 16 rows out of the staging buffer, 16 bytes per lane and row group
                    float* dst = p.logits + static_cast<size_t>(r0 + half * kTransRows + (lane >> 3)) * p.ldl + vbase +
                                 quarter * 32 + (lane & 7) * 4;
#pragma unroll
                    for (int it = 0; it < 4; ++it) {
                      const int row = it * 4 + (lane >> 3);
                      if (half * kTransRows + row < n_ok && (lane & 7) * 4 < nv) {
                        const float4 x = *reinterpret_cast<const float4*>(tbuf + row * 32 + (((lane & 7) ^ (row & 7)) << 2));
                        float4* d4 = reinterpret_cast<float4*>(dst + static_cast<size_t>(it * 4) * p.ldl);
                        if (p.stream_logits) __stcs(d4, x);
                        else *d4 = x;
                      }
                    }
                  };
                  if (kWide && p.logits && !(group & 1)) put();
                  float e[16];
#pragma unroll
                  for (int jj = 0; jj < 4; ++jj) {
                    const float4 x = *reinterpret_cast<const float4*>(
                        tbuf + trow * 32 + (((thalf * 4 + jj) ^ (trow & 7)) << 2));
                    e[4 * jj] = x.x; e[4 * jj + 1] = x.y; e[4 * jj + 2] = x.z; e[4 * jj + 3] = x.w;
                  }
                  // (rows at or beyond n_ok fold whatever the unused columns held; they are never written out)
                  if (n16 == 16) stats_fold16_packed(e, vocab16, p.want_arg, st[slot][half]);
                  else if (n16 > 0) stats_fold16<false>(e, n16, vocab16, p.want_arg, st[slot][half]);
                  if (kWide && p.logits && (group & 1)) put();
                }
              }
            }
          }
        }
      }
    }
    if (bulk && lane == 0) bulk_wait_all();
    // ---- the CTA's statistics of every row: the eight contributions (lane quarter, half) side by side where the ring was
    // (this warp has seen the last tile's MMAs complete, so every slot has been filled and read for the last time)
    float4* merge = reinterpret_cast<float4*>(smem);                // [8][rows of the pass]
#pragma unroll
    for (int slot = 0; slot < kSlots; ++slot) {
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const Stats a = st[slot][half];
        const float4 x = make_float4(a.m, a.s, a.t, __int_as_float(a.arg));
        if (kTwoPlane) {
          const int r = 32 * (group + slot * kGroups) + half * kTransRows + trow;   // row inside the pass
          if (slot < 2 && r < rows) merge[(quarter * 2 + thalf) * rows + r] = x;
        } else if (slot < my_chunks) {
          const int ch = rot ? slot * sub_chunks + group : group + slot * kGroups;
          const int sub = ch / sub_chunks, j = ch - sub * sub_chunks;
          const int c = j * 32 + half * kTransRows + trow;           // column inside its MMA
          const int r = sub * p.N + c;                               // row inside the pass
          if (c < p.N && r < rows) merge[(quarter * 2 + thalf) * rows + r] = x;
        }
      }
    }
  } else if (kW8) {
    // ------------------------------------------------------------------ on-chip expansion: converter warps
    // Codes of a K block, [tile_rows][128] in the slot -> bf16 operand in tensor memory, thread = vocabulary row = lane:
    // 128 (8-bit) or 64 (4-bit) bytes of the row come in as 16-byte pieces (the TMA swizzle of 128 / 64 bytes spreads
    // eight neighbouring rows over all banks), are expanded in registers and go out 32 columns per tcgen05.st.  The
    // expanded operand never touches shared memory.  Two groups of four warps (a warp reaches only its own quarter of the
    // lanes) take the blocks in turn.
    // What bounds it: with few verify rows the thread that issues the MMAs (some 650 cycles per block: its look at the
    // barrier, eight MMAs, two commits), close to the 700 cycles that HBM needs for a block at 8 bits; with 129..192 rows
    // the MMAs (768 cycles per block) and, in long loops, the power cap.  Measured (whole step, widths 20/70/10 %): one
    // sequence, H = 4096, V = 32000 68.3 us with the operand expanded into shared memory by groups of two warps, K blocks of
    // 64 and a byte permute or more per code; 44.0 in this form, 41.0 with the tail and the accept/sample kernel
    // shortened, 37.4 with three groups, 35.3 with one barrier per block for hidden rows and operand and an early look at
    // the next one (all 8-bit: 58.1 -> 31.6).  192 rows, V = 128256: 331 -> 220.  Operand slots of half a block (four of
    // 32 columns next to two accumulators of 192): no gain at 192 rows, 39.4 -> 47.6 with one sequence.
    const int quarter = warp & 3;
    const int grp = (warp - (2 + kNumEpi)) / kConvGroup;
    const int row = quarter * 32 + lane;
    const int G = p.conv_groups;
    const uint32_t leader_full = map_to_cta(full_bar, 0);
    const uint32_t operand_lane = tmem_base + 2 * p.acc_cols + (static_cast<uint32_t>(quarter * 32) << 16);
    grid_dependency_wait();                              // the width table and the exponents may come from the kernel before
    // Where this lane's row starts in the slot, and what the swizzle does to the index of its 16-byte pieces.
    const uint32_t off8 = static_cast<uint32_t>(row) * 128u, x8 = (static_cast<uint32_t>(row) & 7u) << 4;
    const uint32_t off4 = static_cast<uint32_t>(row) * 64u, x4 = (static_cast<uint32_t>(row >> 1) & 3u) << 4;
    // Ring slot and phase of block i of the CTA's sequence; operand slot of block i; ring slot and phase of block
    // i - a_slots, whose MMAs must be done before the operand slot is overwritten.  a_slots <= stages, so having waited
    // for that block implies that the slot's previous codes have been used up, and no wait is more than a phase behind.
    int stage = grp, aslot = grp;                        // (grp < conv_groups <= a_slots <= stages)
    int old_stage = (grp + G * kMaxStages - p.a_slots) % G;       // first block >= a_slots of this group, less a_slots
    uint32_t phase = 0, old_phase = 0;
    int i = grp, kb = grp;                               // block i is block kb of tile t
    bool ok = grp < G;
    for (int t = 0; t < my_tiles && ok; ++t) {
      const int g = pair + t * npairs;
      const int width = p.group_width ? p.group_width[g] : 8;
      const int n_blocks = width == 16 ? p.n_kblocks : code_blocks;
      // (4-bit) exponents of this lane's row, one per K block, fetched two of the group's blocks ahead
      const uint8_t* sh = nullptr;
      if (width == 4) {
        const int r4 = p.group_row[g] + static_cast<int>(rank) * p.tile_rows + row;
        if (r4 < p.rows4) sh = p.shift4 + r4;
      }
      uint32_t sh0 = sh && kb < n_blocks ? sh[static_cast<size_t>(kb) * p.rows4] : 0u;
      uint32_t sh1 = sh && kb + G < n_blocks ? sh[static_cast<size_t>(kb + G) * p.rows4] : 0u;
      for (; kb < n_blocks; kb += G, i += G) {
        const uint32_t sh2 = sh && kb + 2 * G < n_blocks ? sh[static_cast<size_t>(kb + 2 * G) * p.rows4] : 0u;
        if (i >= p.a_slots) {
          if (!mbar_wait_together(empty_bar + 8 * old_stage, old_phase, abort_flag, p.status)) { ok = false; break; }
          tc_fence_after();
          old_stage += G;
          if (old_stage >= p.stages) { old_stage -= p.stages; old_phase ^= 1u; }
        }
        if (width != 16) {
          if (!mbar_wait_together(rawfull_bar + 8 * stage, phase, abort_flag, p.status)) { ok = false; break; }
          const uint8_t* slot = smem + stage * stage_bytes;
          const uint32_t dst = operand_lane + aslot * kOperandCols;
          if (width == 8) {
#pragma unroll
            for (int half = 0; half < 2; ++half) {
              uint4 x[4];
              uint32_t o[32];
#pragma unroll
              for (int c = 0; c < 4; ++c)
                x[c] = *reinterpret_cast<const uint4*>(slot + off8 + ((16u * (4 * half + c)) ^ x8));
#pragma unroll
              for (int c = 0; c < 4; ++c) expand_int8x16(x[c], o + 8 * c);
              tmem_st32(dst + 32 * half, o);
            }
          } else {
            const uint32_t shift = min(sh0, 4u);
#pragma unroll
            for (int half = 0; half < 2; ++half) {
              uint4 x[2];
              uint32_t o[32];
#pragma unroll
              for (int c = 0; c < 2; ++c)
                x[c] = *reinterpret_cast<const uint4*>(slot + off4 + ((16u * (2 * half + c)) ^ x4));
#pragma unroll
              for (int c = 0; c < 2; ++c) expand_int4x32(x[c], o + 16 * c, shift);
              tmem_st32(dst + 32 * half, o);
            }
          }
          tmem_st_wait();
          tc_fence_before();
        }
        __syncwarp();
        if (elect_one()) mbar_arrive_cluster(leader_full + 8 * stage);
        sh0 = sh1; sh1 = sh2;
        stage += G;
        if (stage >= p.stages) { stage -= p.stages; phase ^= 1u; }
        aslot += G;
        if (aslot >= p.a_slots) aslot -= p.a_slots;
      }
      kb -= n_blocks;                                    // where this group starts in the next tile
    }
  }

  // ------------------------------------------------------------------ common tail
  __syncwarp();                                          // warps 0 and 1 ran one lane apart from the others
  tc_fence_before();
  __syncthreads();
  grid_dependency_wait();                                // (every thread that writes below; long since satisfied)
  // 8-bit modes: what the tail needs is worked out anew.  Values that lived through the epilogue's loops on its account were
  // spilled (72 and 108 bytes of reloads, some of them per K block, by the threads that feed the tensor cores).  us: 192 rows,
  // V = 128256 137.8 -> 135.6, two planes, V = 32000 118.9 -> 117.8.  (The other modes do not spill on its account and gain nothing.)
  constexpr bool kAnew = kMode >= 2 && !kRot;
  int bid = blockIdx.x, tid = threadIdx.x, pair_end = pair, row0_end = row0, rows_end = rows;
  if (kAnew) {
    asm volatile("mov.u32 %0, %%ctaid.x;" : "=r"(bid));
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
    pair_end = p.n_pass > 1 ? (bid >> 1) / p.n_pass : bid >> 1;
    row0_end = p.n_pass > 1 ? ((bid >> 1) - pair_end * p.n_pass) * p.rows_per_pass : p.row0;
    rows_end = p.n_pass > 1 ? min(p.rows_per_pass, p.M - row0_end) : p.rows;
  }
  if (!*abort_flag) {
    // one partial per CTA and row: the eight contributions merged around their maximum
    const float4* merge = reinterpret_cast<const float4*>(smem);
    for (int r = tid; r < rows_end; r += kK1Threads) {
      float4 x[8];
      float m = -CUDART_INF_F, sum = 0.f, sum_t = 0.f;
      int arg = 0x7fffffff;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        x[q] = merge[q * rows_end + r];
        m = fmaxf(m, x[q].x);
      }
      // (No branches: they kept the eight exponentials from overlapping, 900 cycles at the end of every launch.  With that, the
      // stores that stop at the last row and what moved ahead of the wait for a tile, us: one sequence, V = 8000 11.66 -> 11.15,
      // V = 32000 46.9 -> 46.2, mixed widths 34.7 -> 33.8; 4, V = 20000 16.45 -> 16.0; 64, V = 16000 18.3 -> 17.9.)
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (x[q].x == m) arg = min(arg, __float_as_int(x[q].w));
        const bool some = x[q].x != -CUDART_INF_F;
        const float d = some ? x[q].x - m : 0.f, y = some ? x[q].y : 0.f, z = some ? x[q].z : 0.f, e = __expf(d);
        sum = fmaf(e, y, sum);
        sum_t = fmaf(e, fmaf(d, y, z), sum_t);
      }
      p.partials[static_cast<size_t>(row0_end + r) * p.part_stride + 2 * pair_end + (kAnew ? bid & 1 : static_cast<int>(rank))] =
          make_float4(m, sum, sum_t, __int_as_float(arg));
    }
  }
  cluster_sync_execution_only();                         // the peer no longer signals this CTA's barriers or tensor memory
  if ((kAnew ? tid >> 5 : warp) == 1) {
    if (*abort_flag) __nanosleep(200000);                // let copies already in flight land before leaving
    tmem_dealloc(kAnew ? *reinterpret_cast<volatile uint32_t*>(tmem_holder) : tmem_base, kTmemCols);
  }
}

// ------------------------------------------------------------------------------------------------ self-test
// The way a GEMM CTA pair gives up, in miniature and on purpose: a pair of CTAs sets up barriers and tensor memory as
// the GEMM kernel does, then one thread and one whole warp of each CTA wait (with the limit given) on a barrier that
// nothing ever arrives on.  The wait must run out, raise HOLA_FLAG_TIMEOUT and the CTA's abort flag, the other waiters
// must see that flag, and every thread must reach the common tail, where the tensor memory is released.
// out[0] counts the threads that got there, out[1] the waits that returned "give up".
__global__ void __launch_bounds__(64, 1) bounded_wait_selftest_kernel(long long limit_cycles, unsigned* status,
                                                                      unsigned* out) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t tmem_holder;
  __shared__ uint32_t abort_word;
  volatile uint32_t* abort_flag = &abort_word;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    abort_word = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (warp == 1) tmem_alloc(smem_u32(&tmem_holder), 32);
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem_base = tmem_holder;
  unsigned gave_up = 0;
  if (warp == 0) {
    if (lane == 0) gave_up = mbar_wait(smem_u32(&bar), 0u, abort_flag, status, limit_cycles) ? 0u : 1u;
  } else {
    gave_up = mbar_wait_warp(smem_u32(&bar), 0u, abort_flag, status, limit_cycles) ? 0u : (lane == 0 ? 1u : 0u);
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (gave_up) atomicAdd(out + 1, 1u);
  atomicAdd(out, 1u);
  cluster_sync_execution_only();
  if (warp == 1) tmem_dealloc(tmem_base, 32);
}

// ------------------------------------------------------------------------------------------------ K2
// The statistics of one row over all CTAs, by a warp, the same bits in every lane.  Six loads per lane in flight (192
// partials per round: one round on a 148-SM part; a GEMM launch leaves a row's partials side by side, part_stride 1).  The
// maximum first (one instruction), so that the exponentials of the partials are independent of one another and only additions
// remain to be passed round: five shuffles instead of eleven merges of a hundred cycles each.  No branch per partial (an empty one
// counts as zeros): they kept the exponentials from overlapping.  The arg-max only for whoever reads it.
constexpr int kPartsPerLane = 6;
__device__ __forceinline__ void load_partials(const float4* partials, int base, int nparts, int part_stride, int lane,
                                              float4 x[kPartsPerLane]) {
#pragma unroll
  for (int u = 0; u < kPartsPerLane; ++u) {
    const int i = base + lane + 32 * u;
    x[u] = i < nparts ? partials[static_cast<size_t>(i) * part_stride]
                      : make_float4(-CUDART_INF_F, 0.f, 0.f, __int_as_float(0x7fffffff));
  }
}
__device__ __forceinline__ Stats merge_loaded(const float4 x[kPartsPerLane], bool want_arg) {
  const float m = warp_max_f32(fmaxf(max3(x[0].x, x[1].x, x[2].x), max3(x[3].x, x[4].x, x[5].x)));
  float s = 0.f, t = 0.f;
#pragma unroll
  for (int u = 0; u < kPartsPerLane; ++u) {
    const bool some = x[u].x != -CUDART_INF_F;
    const float d = some ? x[u].x - m : 0.f, y = some ? x[u].y : 0.f, z = some ? x[u].z : 0.f, e = __expf(d);
    s = fmaf(e, y, s);
    t = fmaf(e, fmaf(d, y, z), t);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, off);
    t += __shfl_xor_sync(0xffffffffu, t, off);
  }
  int arg = 0x7fffffff;
  if (want_arg) {
#pragma unroll
    for (int u = 0; u < kPartsPerLane; ++u)
      if (x[u].x == m) arg = min(arg, __float_as_int(x[u].w));
    arg = __reduce_min_sync(0xffffffffu, arg);
  }
  return Stats{m, s, t, arg};
}
// (x: the first round, loaded)
__device__ __forceinline__ Stats warp_merge_partials(float4 x[kPartsPerLane], const float4* partials, int nparts, int part_stride,
                                                     int lane, bool want_arg) {
  Stats st = merge_loaded(x, want_arg);
  for (int base = 32 * kPartsPerLane; base < nparts; base += 32 * kPartsPerLane) {
    load_partials(partials, base, nparts, part_stride, lane, x);
    st = stats_merge(st, merge_loaded(x, want_arg));
  }
  return st;
}
__device__ __forceinline__ Stats warp_merge_row(const float4* partials, int nparts, int row_stride, int row, int lane, bool want_arg) {
  partials += static_cast<size_t>(row) * row_stride;
  float4 x[kPartsPerLane];
  load_partials(partials, 0, nparts, 1, lane, x);
  return warp_merge_partials(x, partials, nparts, 1, lane, want_arg);
}

// t / s for 1 <= s <= V and t = 0 or |t| >= 2^-100: the product with the approximate reciprocal, corrected once by its remainder
// (Newton's step on the quotient).  The reciprocal is within 2^-23 (relative), the product then within 1.5 * 2^-23, the corrected
// quotient within 1.5 * 2^-46, to which the rounding of the remainder adds half of that at most: less than 2^-20 of a unit in the
// last place ahead of its one rounding, hence t / s rounded or, where that is as close to a tie, its neighbour.  (An IEEE division
// takes 260 cycles here, of a chain that small batches wait for; this 35.)
__device__ __forceinline__ float quotient(float t, float s) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(s));
  const float q = t * y;
  return fmaf(fmaf(-q, s, t), y, q);
}
__global__ void quotient_selftest_kernel(const float* t, const float* s, int n, float* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = quotient(t[i], s[i]);
}
__device__ __forceinline__ void stats_to_outputs(Stats st, float* logZ, float* H) {
  const float ls = logf(st.s);
  *logZ = st.m + ls;
  *H = fmaxf(0.f, ls - quotient(st.t, st.s));
}

__global__ void __launch_bounds__(256) finalize_kernel(const float4* partials, int nparts, int row_stride, int M,
                                                       float* logZ, float* entropy) {
  // (launched like the accept/sample kernel: the next kernel in the stream may be put in place behind this one)
  grid_dependency_release();
  const int row = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  grid_dependency_wait();
  if (row >= M) return;
  Stats st = warp_merge_row(partials, nparts, row_stride, row, lane, false);
  if (lane == 0) stats_to_outputs(st, &logZ[row], &entropy[row]);
}

// Vocabulary-parallel form, first exchange record of a rank: per verify row the statistics of this shard's logits
// (m, s, t, arg-max as a GLOBAL vocabulary index), then per draft position the logit of the draft token if this shard
// owns it (-inf otherwise).  Blocks 0 .. ceil(M/8)-1 merge the per-CTA partials, the others gather the logits.
__global__ void __launch_bounds__(256) shard_record_kernel(const float4* partials, int nparts, int row_stride, int M,
                                                           int v_offset, int V, const float* logits, int ldl,
                                                           const int* tok, int B, int k, float4* stats_out,
                                                           float* lx_out) {
  const int row_blocks = (M + 7) / 8;
  if (static_cast<int>(blockIdx.x) < row_blocks) {
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (row >= M) return;
    Stats st = warp_merge_row(partials, nparts, row_stride, row, lane, true);
    if (lane == 0) {
      const int arg = st.arg == 0x7fffffff ? st.arg : st.arg + v_offset;
      stats_out[row] = make_float4(st.m, st.s, st.t, __int_as_float(arg));
    }
  } else {
    const int i = (blockIdx.x - row_blocks) * 256 + threadIdx.x;
    if (i >= B * k) return;
    const int b = i / k, j = i - b * k;
    const int x = tok[i] - v_offset;
    lx_out[i] = (x >= 0 && x < V) ? logits[static_cast<size_t>(b * (k + 1) + j) * ldl + x] : -CUDART_INF_F;
  }
}

// ------------------------------------------------------------------------------------------------ K3
// Four sums over the warp at once (lanes 8 i .. 8 i + 7 return the sum of v[i]): the first two rounds halve the
// number of values a lane carries instead of adding all of them everywhere, six shuffles in all.
__device__ __forceinline__ float warp_sum4_f32(const float v[4], int lane) {
  const bool hi16 = (lane & 16) != 0;
  const float a = (hi16 ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, hi16 ? v[0] : v[2], 16);
  const float b = (hi16 ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, hi16 ? v[1] : v[3], 16);
  const bool hi8 = (lane & 8) != 0;
  float c = (hi8 ? b : a) + __shfl_xor_sync(0xffffffffu, hi8 ? a : b, 8);
#pragma unroll
  for (int off = 4; off > 0; off >>= 1) c += __shfl_xor_sync(0xffffffffu, c, off);
  return c;
}

// Logits and draft probabilities of vocabulary entries base..base+3 of one row (q = 0 when the row is drawn
// from p itself; entries at or beyond V get l = -inf, q = 0 and so no mass).  Loads only: a caller can issue
// several of these before using any, which keeps more requests in flight.
template <bool kVec, bool kHalf>
__device__ __forceinline__ void fetch4(const float* lrow, const void* qrow, bool residual, int base, int V, float l[4], float q[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) { l[i] = -CUDART_INF_F; q[i] = 0.f; }
  if (kVec) {                                            // (V is a multiple of 4)
    if (base < V) {
      const float4 l4 = *reinterpret_cast<const float4*>(lrow + base);
      l[0] = l4.x; l[1] = l4.y; l[2] = l4.z; l[3] = l4.w;
      if (residual) {
        if (kHalf) {
          const uint2 raw = *reinterpret_cast<const uint2*>(static_cast<const __nv_bfloat16*>(qrow) + base);
          q[0] = __uint_as_float(raw.x << 16); q[1] = __uint_as_float(raw.x & 0xFFFF0000u);
          q[2] = __uint_as_float(raw.y << 16); q[3] = __uint_as_float(raw.y & 0xFFFF0000u);
        } else {
          const float4 q4 = *reinterpret_cast<const float4*>(static_cast<const float*>(qrow) + base);
          q[0] = q4.x; q[1] = q4.y; q[2] = q4.z; q[3] = q4.w;
        }
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int v = base + i;
      if (v < V) {
        l[i] = lrow[v];
        if (residual)
          q[i] = kHalf ? __bfloat162float(static_cast<const __nv_bfloat16*>(qrow)[v]) : static_cast<const float*>(qrow)[v];
      }
    }
  }
}

// The four residual masses  r = max(0, p - q)  with  p = e^(l - logZ)  (q = 0: r = p).  The exponential is the
// hardware's 2^x on (l - logZ) log2 e: relative error about 1e-6 at l - logZ = -30, against a decision margin of 1e-4
// on the cumulative mass; the pass over the row and the final search inside a chunk both come through here.
__device__ __forceinline__ void resid4(const float l[4], const float q[4], float logZ, float r[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) r[i] = fmaxf(0.f, ex2_approx((l[i] - logZ) * kLog2e) - q[i]);
}

// The residual masses of up to four chunks, c0 and every kStride-th after it as long as they are among n, by a warp: into csum[],
// and as the result in lanes 8 i .. 8 i + 7 (0 where there is no i-th).  In fp32 (128 non-negative terms added pairwise: relative
// error a few 1e-7), kept as fp64 for the sums that follow.  lrow, qrow: entry 0 of the row, which a staged slice does not hold.
// (Once per type of q: us, 50 rows, V = 60000 53.2 -> 52.4, 32 rows, V = 128256 61.0 -> 59.7, 5 rows, V = 32000 46.67 -> 46.46.  A
// form for two chunks, and packed fp32 arithmetic, took fewer instructions and longer.)
template <bool kVec, bool kHalf, int kStride>
__device__ __forceinline__ double sum_step(const float* lrow, const void* qrow, bool residual, int c0, int n, int V, float logZ,
                                           double* csum, int lane) {
  float l[kK3Unroll][4], q[kK3Unroll][4];
#pragma unroll
  for (int i = 0; i < kK3Unroll; ++i)                    // all loads first
    fetch4<kVec, kHalf>(lrow, qrow, residual, i * kStride < n ? (c0 + i * kStride) * kChunk + lane * 4 : V, V, l[i], q[i]);
  float part[kK3Unroll];
#pragma unroll
  for (int i = 0; i < kK3Unroll; ++i) {
    part[i] = 0.f;
    if (i * kStride < n) {
      float r[4];
      resid4(l[i], q[i], logZ, r);
      part[i] = (r[0] + r[1]) + (r[2] + r[3]);
    }
  }
  const double sum = static_cast<double>(warp_sum4_f32(part, lane));
  if ((lane & 7) == 0 && (lane >> 3) * kStride < n) csum[(lane >> 3) * kStride] = sum;
  return sum;
}

// Untiled bulk copy into this CTA's shared memory (addresses and size multiples of 16 bytes), counted on an mbarrier.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
// A double into a CTA of the cluster (addresses from map_to_cta), counted on a barrier there.
__device__ __forceinline__ void store_async(uint32_t cluster_addr, double x, uint32_t cluster_bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];"
               ::"r"(cluster_addr), "l"(__double_as_longlong(x)), "r"(cluster_bar)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile("{\n .reg .pred P;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 P, [%1], %2;\n selp.u32 %0, 1, 0, P;\n}"
               : "=r"(done) : "r"(bar), "r"(parity) : "memory");
  return done != 0;
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void report_flags(const K3Params& p, int b, unsigned flags) {
  if (p.flags_out) p.flags_out[b] = flags | (p.status ? *reinterpret_cast<volatile unsigned*>(p.status) : 0u);
  else if (flags && p.status) atomicOr(p.status, flags);
}

__device__ __forceinline__ float clamp_uniform(float u, unsigned& flags) {
  if (!(u >= 0.f)) { flags |= HOLA_FLAG_BAD_UNIFORM; return 0.f; }
  if (u >= 1.f) { flags |= HOLA_FLAG_BAD_UNIFORM; return 1.f - 5.9604645e-8f; }   // 1 - 2^-24
  return u;
}

// Waits for what is counted on a barrier of this CTA: its staged rows, or the masses of all warps of the cluster.  When the time is
// up the status word is told at once: the CTA that draws the token, and reports, may be another one of the cluster, whose rows did
// land (it looks at the status word behind the exchange of masses).  What is waited for then has as long again before the CTA goes
// on (and sooner or later leaves the memory that copies write to).  False: gave up, nothing arrived in that time either.
__device__ __forceinline__ bool wait_bulk(uint32_t bar, unsigned* status, long long limit_cycles) {
  const long long t0 = clock64();
  bool late = false;
  while (!mbar_try_wait_cluster(bar, 0u)) {
    const long long waited = clock64() - t0;
    if (waited > limit_cycles && !late) {
      late = true;
      if (status) atomicOr(status, HOLA_FLAG_TIMEOUT);
    }
    if (waited > 2 * limit_cycles) return false;
  }
  return true;
}

// The exchange of masses: each CTA of the cluster has room for the masses of all, and a barrier that counts their bytes.
// A warp's mass to every CTA, lane i to CTA i (`lane` < cluster size only).
__device__ __forceinline__ void send_mass(double* slot, uint64_t* all, double mass, int lane) {
  store_async(map_to_cta(smem_u32(slot), lane), mass, map_to_cta(smem_u32(all), lane));
}
// The wait for them, twice as long as that for staged rows: a CTA whose rows do not land sends what it has behind that wait.
__device__ __forceinline__ bool wait_masses(uint64_t* all, unsigned* status, long long limit_cycles) {
  return wait_bulk(smem_u32(all), status, 2 * limit_cycles);
}
// The way out for a CTA whose wait gave up (all of its threads).  The others may still be sending to it: it stays until each of
// them has left (threads that have exited are not waited for) or has come here too, and until what they sent has landed.
__device__ __forceinline__ void leave_behind_the_others() {
  cluster_sync_all();
  __nanosleep(200000);
}

// The ways those waits give up, in miniature: a cluster of two CTAs, of which the second waits for staged rows that nothing ever
// brings and sends its mass behind that.  kEarly: the first, whose rows are there, gives up on the second one's mass long before,
// and has to stay until it has landed; otherwise it gets it, and must find the time-out in the status word when it reports.
// out[0] counts the threads that reached the end, out[1] the waits that gave up, out[2] is the word of flags that the first
// CTA leaves, out[3] (kEarly) counts the CTAs in whose memory both masses have landed when they leave.
template <bool kEarly>
__global__ void __launch_bounds__(64, 1) staged_wait_selftest_kernel(long long limit_cycles, unsigned* status, unsigned* out) {
  __shared__ __align__(8) uint64_t bar, all;
  __shared__ double masses[2];
  __shared__ int sh_gave_up;
  const uint32_t rank = cluster_cta_rank();
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    mbar_init(smem_u32(&all), 1);
    mbar_expect_tx(smem_u32(&all), 2 * 8u);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (rank == 0) mbar_arrive(smem_u32(&bar));
    masses[0] = masses[1] = 0.0;
    sh_gave_up = 0;
  }
  __syncthreads();
  cluster_sync_all();
  if (!wait_bulk(smem_u32(&bar), status, limit_cycles)) { sh_gave_up = 1; atomicAdd(out + 1, 1u); }
  if (threadIdx.x < 2) send_mass(&masses[rank], &all, 1.0 + rank, threadIdx.x);
  if (threadIdx.x < 32 && !wait_masses(&all, status, kEarly && rank == 0 ? limit_cycles / 16 : limit_cycles)) {
    sh_gave_up = 1;
    atomicAdd(out + 1, 1u);
  }
  __syncthreads();
  if (sh_gave_up) leave_behind_the_others();
  if (kEarly && threadIdx.x == 0 && *const_cast<volatile double*>(&masses[0]) == 1.0 && *const_cast<volatile double*>(&masses[1]) == 2.0)
    atomicAdd(out + 3, 1u);
  if (rank == 0 && threadIdx.x == 0) {
    K3Params p;
    p.status = status; p.flags_out = out + 2;
    report_flags(p, 0, 0u);
  }
  atomicAdd(out, 1u);
}

// Whether the run of accepted drafts ends at a position, and what it flags.
constexpr unsigned kStop = 1u << 31;
__device__ __forceinline__ unsigned decide(const K3Params& p, int x, int Vtok, float u, float lx, float qx, float hq, float logZ,
                                           float H, int amax) {
  if (x < 0 || x >= Vtok) return HOLA_FLAG_BAD_TOKEN | kStop;
  if ((p.gate_source == HOLA_GATE_DRAFT_ENTROPY ? hq : H) < p.tau) return 0u;        // entropy gate: fast path keeps the draft token
  if (p.fallback == HOLA_FALLBACK_GREEDY) return x != amax ? kStop : 0u;             // the verifier's own token, or the run ends here
  unsigned flags = 0;
  u = clamp_uniform(u, flags);
  const float px = expf(lx - logZ);
  const bool keep = (qx > 0.f) ? (u * qx < px) : (px > 0.f);
  return flags | (keep ? 0u : kStop);
}

// One cluster of S CTAs per sequence.  Every CTA derives accept_len on its own (same inputs, same arithmetic,
// same result), a warp per position from the statistics to the decision, sums the residual mass of its slice of the
// vocabulary chunk by chunk, and every warp sends what it summed to all CTAs of the cluster through distributed shared memory.
// Once all of it has arrived each CTA knows the total mass R and which slice holds the point u*R; that CTA alone finishes the
// inverse-CDF search, with one warp: chunk, lane, entry.
// On small batches a chain of dependent steps bounds it, a few hundred cycles each (a shuffle is 29, one of a double with its
// addition 35, a vote 21, an IEEE division 260), and where one SM has 32 warps at it the instructions of all of them: nothing is
// worked out by more warps than need it, nor ahead of a barrier if one warp can do it behind.  Before, every warp made all
// decisions behind the first barrier, warp 0 of each CTA scanned its chunks ahead of a cluster barrier, and every warp scanned the
// slices behind it.  Cycles from entry to token, V = 1000 9030 -> 7090, V = 32000 9890 -> 8820; us, one sequence, V = 1000
// 9.6 -> 8.7, V = 8000 11.06 -> 10.85, V = 32000 45.8 -> 45.2, mixed widths 33.8 -> 33.2; 8 sequences of 9 positions, V = 30000
// 18.6 -> 17.9; 200, V = 12000 41.0 -> 39.9; 250, V = 30000 47.4 -> 44.2; 64, V = 16000 18.0 -> 17.9; 8, V = 128256 38.65 -> 38.8.
// The chunks of a step alternate between the warps: side by side in one warp (so that a warp's mass is that of a run of the
// vocabulary, and one scan less is needed) rows that start on no line are fetched twice, 60 sequences, V = 50003 33.2 -> 36.9.
// kAsk: the slice of row n is asked into the L2 as soon as n is known.
// kSoloWarps: one CTA of 1024 threads instead of the cluster (see sample_solo).  All 32 warps of it take part or, for up to
// kFewEntries entries and sequences for half of the SMs, the first 16: the others leave at once, and the instructions of the rest
// find more room.  us, 32 -> 16 warps: V = 2000, 16 sequences 10.4 -> 10.0; V = 3000, 1 9.7 -> 9.4; V = 5000, 2 / 32 10.15 -> 9.8,
// 11.55 -> 11.25; V = 8000, 1 / 64 / 75 / 140 10.5 -> 10.25, 13.2 -> 13.0, 15.0 -> 15.0, 18.35 -> 18.45; V = 8191, 5 12.25 -> 11.95;
// V = 11000, 16 13.2 -> 13.6; V = 16000, 64 17.7 -> 18.8.  (Launched with 512 threads they take 0.05 to 0.15 less again; the
// launch is one of 1024, as hola_sample_plan_for_shape reports it.)
// kStaged: this CTA's slice of ALL k + 1 rows is brought into shared memory while the statistics are merged and the accept test
// is made, instead of row n afterwards.
template <bool kVec, bool kAsk, int kSoloWarps = 0, bool kStaged = false>
__global__ void __launch_bounds__(kSoloWarps ? kSoloThreads : kK3Threads, kSoloWarps ? 1 : kK3MaxPerSm) accept_sample_kernel(const K3Params p) {
  constexpr bool kSolo = kSoloWarps > 0;
  constexpr int kWarps = kSolo ? kSoloWarps : kK3Threads / 32;
  if (kSolo && threadIdx.x >= kWarps * 32) return;
  extern __shared__ __align__(16) double csum[];                       // per-chunk residual mass of this CTA's slice
  __shared__ __align__(16) double sh_tot[2][kSolo ? kWarps : 8 * kWarps];      // masses of all warps' runs, per attempt
  __shared__ float sh_logZ[kMaxK1], sh_uk;
  __shared__ int sh_amax[kMaxK1];
  __shared__ unsigned sh_dec[kMaxK1];                    // decide()'s results
  __shared__ __align__(8) uint64_t sh_bar;               // staged rows have landed
  __shared__ __align__(8) uint64_t sh_all[2];            // all runs' masses have arrived, per attempt
  __shared__ int sh_gave_up;                             // a wait of this CTA ran out

  // The next kernel in the stream (normally the next call's GEMM kernel, which waits for this grid before it touches
  // memory) may be scheduled from now on: its launch and prologue then hide behind this kernel.
  grid_dependency_release();
  cg::cluster_group cluster = cg::this_cluster();
  const int S = kSolo ? 1 : static_cast<int>(cluster.num_blocks());
  const int rank = kSolo ? 0 : static_cast<int>(cluster.block_rank());
  const int b = kSolo ? static_cast<int>(blockIdx.x) : static_cast<int>(blockIdx.x) >> (31 - __clz(S));   // (S is 1, 2, 4 or 8)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = p.k, V = p.V;
  const int row_first = b * (k + 1);

  // ---- the draft tokens and uniforms.  The k + 1 positions are dealt to the warps from the last warp down, and lane i of a
  // warp looks after the warp's i-th position.  These come from the caller, not from the GEMM kernel.  Behind this call's own
  // GEMM kernel they are known to be in place (its CTAs waited for whatever ran before the call) and are asked for before this
  // grid's dependency wait; in every other launch the wait comes first.  Nothing looks at a loaded value before everything
  // that does not depend on it has been asked for: each look costs a round trip to the L2 (or, where the GEMM kernel's idle
  // warps have not asked ahead, to DRAM).
  if (!p.inputs_settled) grid_dependency_wait();
  const bool shard = p.shard_world > 0;
  const int Vtok = shard ? p.V_global : V;               // range of valid token ids
  const int j_first = kWarps - 1 - warp, j_mine = j_first + lane * kWarps;
  int x_mine = -1;
  float u_mine = 0.f;
  if (j_mine < k) x_mine = p.tok[b * k + j_mine];
  if (j_mine <= k) u_mine = p.u[b * (k + 1) + j_mine];
  // From here on the GEMM kernel's results are read.
  if (p.inputs_settled) grid_dependency_wait();
  // (statistics first: what follows looks at the tokens)
  const float4* row_parts = p.partials + static_cast<size_t>(row_first + j_first) * p.row_stride;
  float4 x[kPartsPerLane];
  if (p.combine && j_first <= k) load_partials(row_parts, 0, p.nparts, p.part_stride, lane, x);
  // (waited for behind the decisions, ahead of the first remote store.  Relaxed: a release here would first wait for the loads)
  if (!kSolo && S > 1) {
    if (threadIdx.x == 0) {
      for (int i = 0; i < 2; ++i) {
        mbar_init(smem_u32(&sh_all[i]), 1);
        mbar_expect_tx(smem_u32(&sh_all[i]), S * kWarps * 8u);
      }
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");
  }
  if (!kSolo && threadIdx.x == 0) sh_gave_up = 0;
  const int nchunks = (V + kChunk - 1) / kChunk;
  const int cpc = kSolo ? nchunks : (nchunks + S - 1) >> (31 - __clz(S));      // chunks per CTA
  const int c_first = rank * cpc;
  const int mine = max(0, min(nchunks, c_first + cpc) - c_first);
  const size_t q_elem = (p.q_dtype == HOLA_Q_BF16) ? 2 : 4;
  // Staged rows, behind the chunk sums: [k + 1][cpc * 128] logits, then [k][cpc * 128] draft probabilities, each row's
  // slice by one bulk copy, a lane of the first warp per copy, while the other warps merge statistics (with eight rows and more
  // that one does so too: then the last warp).  (One thread after the other, in a warp that merges as well, they held the merge
  // up by 0.7 us; us, 5 rows, V = 32000: 46.67 -> 46.31, mixed widths 34.84 -> 34.47.)
  const int slice = cpc * kChunk;
  float* sl = reinterpret_cast<float*>(csum + (cpc + 1) / 2 * 2);      // (16-byte boundary whatever the number of chunks)
  char* sq = reinterpret_cast<char*>(sl + static_cast<size_t>(k + 1) * slice);
  const int here = min(V - c_first * kChunk, mine * kChunk);           // entries of this slice (0 or less: none)
  if (kStaged && warp == (k + 1 < kWarps ? 0 : kWarps - 1) && here > 0) {
    const uint32_t bar = smem_u32(&sh_bar), lbytes = here * 4u, qbytes = static_cast<uint32_t>(here * q_elem);
    if (lane == 0) {
      mbar_init(bar, 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      mbar_expect_tx(bar, (k + 1) * lbytes + k * qbytes);
    }
    __syncwarp();
    const float* l = p.logits + static_cast<size_t>(row_first) * p.ldl + c_first * kChunk;
    const char* q = static_cast<const char*>(p.q) + (static_cast<size_t>(b) * k * V + c_first * kChunk) * q_elem;
    for (int i = lane; i <= 2 * k; i += 32) {
      if (i <= k) bulk_load(smem_u32(sl + static_cast<size_t>(i) * slice), l + static_cast<size_t>(i) * p.ldl, lbytes, bar);
      else bulk_load(smem_u32(sq + static_cast<size_t>(i - k - 1) * slice * q_elem), q + static_cast<size_t>(i - k - 1) * V * q_elem, qbytes, bar);
    }
    __syncwarp();
  }
  // the draft token's logit and probability
  float lx = 0.f, hq = 0.f;
  uint32_t q_bits = 0;                                   // (as loaded: converted where it is used)
  if (j_mine < k) {
    const int j = j_mine;
    if (x_mine >= 0 && x_mine < Vtok && p.fallback != HOLA_FALLBACK_GREEDY) {     // (greedy: compared by its index alone)
      const size_t qi = (static_cast<size_t>(b) * k + j) * V + x_mine;
      if (p.q_tok) q_bits = __float_as_uint(p.q_tok[b * k + j]);
      else if (p.q_dtype == HOLA_Q_BF16) q_bits = static_cast<const uint16_t*>(p.q)[qi];
      else q_bits = static_cast<const uint32_t*>(p.q)[qi];
      if (shard) {                                       // exactly one shard owns x and left its logit there
        lx = -CUDART_INF_F;
        for (int r = 0; r < p.shard_world; ++r) lx = fmaxf(lx, p.lx_all[static_cast<size_t>(r) * p.rec_stride + b * k + j]);
      } else {
        lx = p.logits[static_cast<size_t>(row_first + j) * p.ldl + x_mine];
      }
    }
    if (p.gate_source == HOLA_GATE_DRAFT_ENTROPY) {
      double tot = 0.0;
      for (int sl = 0; sl < kHqSlices; ++sl) tot += p.hq_part[(static_cast<size_t>(b) * k + j) * kHqSlices + sl];
      hq = fmaxf(0.f, static_cast<float>(-tot));
      if (rank == 0 && p.draft_entropy) p.draft_entropy[b * k + j] = hq;
    }
  }
  // ---- softmax statistics of this sequence's k+1 positions; gate and ratio test of each
  for (int i = 0, j = j_first; j <= k; ++i, j += kWarps) {
    float lz, h;
    int amax = 0;
    if (p.combine) {
      if (i > 0) {
        row_parts += static_cast<size_t>(kWarps) * p.row_stride;
        load_partials(row_parts, 0, p.nparts, p.part_stride, lane, x);
      }
      const Stats st = warp_merge_partials(x, row_parts, p.nparts, p.part_stride, lane, p.fallback == HOLA_FALLBACK_GREEDY);
      stats_to_outputs(st, &lz, &h);
      amax = st.arg;
    } else {
      lz = p.logZ[row_first + j];
      h = p.entropy[row_first + j];
    }
    if (lane == i) {
      const float qx = __uint_as_float(!p.q_tok && p.q_dtype == HOLA_Q_BF16 ? q_bits << 16 : q_bits);
      sh_dec[j] = j < k ? decide(p, x_mine, Vtok, u_mine, lx, qx, hq, lz, h, amax) : 0u;
      sh_logZ[j] = lz; sh_amax[j] = amax;
      if (j == k) sh_uk = u_mine;
      if (rank == 0 && p.combine) { p.logZ[row_first + j] = lz; p.entropy[row_first + j] = h; }
    }
  }
  __syncthreads();

  // ---- in draft order, the first position that is not accepted ends the run (what a position past it flags does not count)
  unsigned flags = 0;                                    // (of the first and the last warp, which report)
  int n = k;
  for (int j0 = 0; j0 < k && n == k; j0 += 32) {
    const unsigned dec = j0 + lane < k ? sh_dec[j0 + lane] : 0u;
    const unsigned stops = __ballot_sync(0xffffffffu, (dec & kStop) != 0u);
    if (stops) n = j0 + __ffs(stops) - 1;
    if (warp == 0 || warp == kWarps - 1) flags |= __reduce_or_sync(0xffffffffu, j0 + lane <= n ? dec & ~kStop : 0u);
  }
  if (rank == 0 && threadIdx.x == (kWarps - 1) * 32) {   // (the first warp goes on to the token)
    p.accept_len[b] = n;
    if (p.fallback == HOLA_FALLBACK_GREEDY) {            // greedy: argmax p_n follows the accepted run; no draw
      p.next_tok[b] = min(max(sh_amax[n], 0), Vtok - 1);
      report_flags(p, b, flags);
    } else if (p.phase == 1) {
      report_flags(p, b, flags);
    }
  }
  if (p.fallback == HOLA_FALLBACK_GREEDY || p.phase == 1) return;   // same decision in every CTA of the cluster

  // ---- this CTA's slice of row n: per-chunk residual mass
  const float logZ = sh_logZ[n];
  const char* qbase = static_cast<const char*>(p.q);
  const float* lrow;
  const void* qrow;
  if (kStaged) {                                         // (as if the slice were the whole row, entry v at row + v)
    lrow = sl + static_cast<size_t>(n) * slice - c_first * kChunk;
    qrow = n >= k ? sq : sq + static_cast<size_t>(n) * slice * q_elem - c_first * kChunk * q_elem;
  } else {
    if (p.q_far && n >= p.q_far_from) qbase = static_cast<const char*>(p.q_far);
    lrow = p.logits + static_cast<size_t>(row_first + n) * p.ldl;
    qrow = n >= k ? nullptr : static_cast<const void*>(qbase + (static_cast<size_t>(b) * k + n) * V * q_elem);
  }
  const bool half = p.q_dtype == HOLA_Q_BF16;
  if (!kSolo && S > 1) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  // (rows that never land: their sums mean nothing, but the other CTAs wait for them)
  if (kStaged && here > 0 && !wait_bulk(smem_u32(&sh_bar), p.status, kWaitLimitCycles)) sh_gave_up = 1;
  // Several CTAs per SM and short slices (up to 8192 entries): a slice into the L2 by two bulk requests instead of by the loads
  // alone.  us, V = 32000, H = 512, 384 rows 33.2 -> 32.5, 240 rows 25.3 -> 24.7; V = 128256 (16032 entries) no gain.  With a CTA
  // per SM the loads are all out at once, and the code alone costs 0.2 us, hence a kernel without it.
  if (kAsk && threadIdx.x == (kWarps - 1) * 32 && here > 0) {
    bulk_prefetch_l2(lrow + c_first * kChunk, static_cast<unsigned>(here) * 4u);
    if (n < k && qbase == static_cast<const char*>(p.q)) {
      const uintptr_t q0 = reinterpret_cast<uintptr_t>(qrow) + c_first * kChunk * q_elem;
      const uintptr_t q1 = (q0 + here * q_elem) & ~static_cast<uintptr_t>(15), qa = (q0 + 15) & ~static_cast<uintptr_t>(15);
      if (q1 > qa) bulk_prefetch_l2(reinterpret_cast<const void*>(qa), static_cast<unsigned>(q1 - qa));
    }
  }
  bool residual = n < k;

  // Vocabulary-parallel draw: every rank holds every rank's two masses of row n, so all of them agree on which mass
  // counts (the residual's unless it vanishes everywhere), on the total R and on the shard that holds the point u * R.
  double shard_target = 0.0;
  if (shard && p.phase == 4) {
    const double* mass = p.mass_all + static_cast<size_t>(b) * 2;
    const size_t rs = static_cast<size_t>(p.B) * 2;
    double tot_res = 0.0;
    for (int r = 0; r < p.shard_world; ++r) tot_res += mass[r * rs];
    const bool use_p = !residual || !(tot_res > 0.0);
    if (use_p && residual) {
      residual = false;
      flags |= HOLA_FLAG_R_ZERO;
    }
    const int idx = use_p ? 1 : 0;
    double total = 0.0;
    for (int r = 0; r < p.shard_world; ++r) total += mass[r * rs + idx];
    unsigned uflags = 0;
    const double target = static_cast<double>(clamp_uniform(sh_uk, uflags)) * total;
    int owner = -1, last_mass = 0;
    double before = 0.0, cum = 0.0;
    for (int r = 0; r < p.shard_world; ++r) {
      const double m = mass[r * rs + idx];
      if (m > 0.0) last_mass = r;
      if (owner < 0 && cum + m > target) { owner = r; before = cum; }
      cum += m;
    }
    shard_target = target - before;
    if (owner < 0) { owner = last_mass; shard_target = CUDART_INF; }     // rounding: the last entry with mass
    if (owner != p.shard_rank) {
      if (rank == 0 && threadIdx.x == 0) p.next_tok[b] = -1;
      return;                                            // same decision in every CTA of the cluster
    }
    __syncthreads();
  }

  for (int attempt = 0; attempt < 2; ++attempt) {
    double mass = 0.0;
    for (int c = warp; c < mine; c += kWarps * kK3Unroll) {
      const int len = mine - c;                          // (a warp's chunks are kWarps apart)
      mass += half ? sum_step<kVec, true, kWarps>(lrow, qrow, residual, c_first + c, len, V, logZ, csum + c, lane)
                   : sum_step<kVec, false, kWarps>(lrow, qrow, residual, c_first + c, len, V, logZ, csum + c, lane);
    }
    mass += __shfl_xor_sync(0xffffffffu, mass, 8);
    mass += __shfl_xor_sync(0xffffffffu, mass, 16);
    if (kSolo || S == 1) {
      if (lane == 0) sh_tot[attempt][warp] = mass;
    } else {
      // To all CTAs, counted on a barrier of theirs: half the way of stores and a cluster barrier behind them.
      if (lane < S) send_mass(&sh_tot[attempt][rank * kWarps + warp], &sh_all[attempt], mass, lane);
      if (warp == 0 && !wait_masses(&sh_all[attempt], p.status, kWaitLimitCycles)) sh_gave_up = 1;
    }
    __syncthreads();                                     // (and this CTA's chunk masses, for the first warp)
    // Lane i has masses 2 i and 2 i + 1.  Every warp learns whether there is any; the first one of every CTA goes on.
    double2 two = make_double2(0.0, 0.0);
    if (2 * lane < (kSolo ? kWarps : S * kWarps)) two = reinterpret_cast<const double2*>(sh_tot[attempt])[lane];
    const bool any = __any_sync(0xffffffffu, two.x > 0.0 || two.y > 0.0) &&
                     !__any_sync(0xffffffffu, two.x != two.x || two.y != two.y);
    if (!kSolo && sh_gave_up) {                          // no draw: some token, and the time-out
      leave_behind_the_others();
      if (threadIdx.x == 0) {
        if (shard && p.phase == 3) p.mass_out[b * 2] = p.mass_out[b * 2 + 1] = 0.0;
        else p.next_tok[b] = shard ? p.v_offset : 0;
        report_flags(p, b, flags | HOLA_FLAG_TIMEOUT);
      }
      return;
    }
    if (shard && p.phase == 3) {
      // the shard's masses of row n: of the residual, then (second pass, q taken as 0) of p itself
      if (rank == 0 && warp == 0) {
        const double R = warp_sum_f64(two.x + two.y);
        if (lane == 0) {
          p.mass_out[b * 2 + attempt] = R;
          if (!residual && attempt == 0) p.mass_out[b * 2 + 1] = R;        // bonus position: both are the mass of p
          if (attempt == 1 || !residual) report_flags(p, b, flags);
        }
      }
      if (residual) {
        residual = false;
        __syncthreads();
        continue;
      }
      return;
    }
    if (!any && residual && !shard) {                    // p <= q everywhere: draw from p instead
      residual = false;
      flags |= HOLA_FLAG_R_ZERO;
      __syncthreads();
      continue;
    }
    if (warp != 0) return;
    const float uk = clamp_uniform(sh_uk, flags);
    double target = shard_target, before = 0.0;
    bool take_last = false;                              // rounding left the running sum a hair below u*R
    if (!kSolo && S > 1) {
      // the slice that holds u * R, with identical arithmetic in every CTA: lanes 4 r .. 4 r + 3 have slice r
      constexpr int kPer = kK3Threads / 64;
      double sum = two.x + two.y;
#pragma unroll
      for (int off = 1; off < kPer; off <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
      double incl = sum;
      for (int off = kPer; off < kPer * S; off <<= 1) {
        const double o = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += o;
      }
      const double R = __shfl_sync(0xffffffffu, incl, kPer * S - 1);
      if (!shard) target = static_cast<double>(uk) * R;
      const unsigned over = __ballot_sync(0xffffffffu, sum > 0.0 && incl > target);
      const unsigned has_mass = __ballot_sync(0xffffffffu, sum > 0.0);
      take_last = over == 0u;
      const int at = over ? __ffs(over) - 1 : (has_mass ? 31 - __clz(has_mass) : 0);
      before = __shfl_sync(0xffffffffu, incl - sum, at);
      if (at / kPer != rank) return;
    }
    // the chunk: lane i has chunks [a, z) of the slice
    const int per_lane = (cpc + 31) / 32, a = min(mine, lane * per_lane), z = min(mine, a + per_lane);
    constexpr int kHeld = 4;                             // (that few stay in registers)
    double m[kHeld], tot = 0.0;
#pragma unroll
    for (int i = 0; i < kHeld; ++i) {
      m[i] = a + i < z ? csum[a + i] : 0.0;
      tot += m[i];
    }
    for (int c = a + kHeld; c < z; ++c) tot += csum[c];
    double upto = tot;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const double o = __shfl_up_sync(0xffffffffu, upto, off);
      if (lane >= off) upto += o;
    }
    if ((kSolo || S == 1) && !shard) target = static_cast<double>(uk) * __shfl_sync(0xffffffffu, upto, 31);
    const unsigned lane_over = __ballot_sync(0xffffffffu, tot > 0.0 && before + upto > target);
    const unsigned lane_mass = __ballot_sync(0xffffffffu, tot > 0.0);
    take_last = take_last || lane_over == 0u;
    const int from = !take_last ? __ffs(lane_over) - 1 : (lane_mass ? 31 - __clz(lane_mass) : 0);
    int cstar = -1, last = a;
    double cum = before + (upto - tot), start = cum;
    auto look = [&](int c, double mc) {                  // (every lane in its own chunks; that of lane `from` counts)
      if (mc > 0.0) {
        last = c;
        if (cstar < 0 && !take_last && cum + mc > target) { cstar = c; start = cum; }
      }
      cum += mc;
    };
#pragma unroll
    for (int i = 0; i < kHeld; ++i) look(a + i, m[i]);
    for (int c = a + kHeld; c < z; ++c) look(c, csum[c]);
    if (cstar < 0) { cstar = last; take_last = true; }
    cstar = __shfl_sync(0xffffffffu, cstar, from);
    before = __shfl_sync(0xffffffffu, start, from);
    take_last = __shfl_sync(0xffffffffu, take_last ? 1 : 0, from) != 0;
    // inside the chunk: lane prefix, then the lane's four entries in ascending order
    const int base = (c_first + cstar) * kChunk + lane * 4;
    float l4[4], q4[4], r4[4];
    if (half) fetch4<kVec, true>(lrow, qrow, residual, base, V, l4, q4);
    else fetch4<kVec, false>(lrow, qrow, residual, base, V, l4, q4);
    resid4(l4, q4, logZ, r4);
    const double mine4 = ((static_cast<double>(r4[0]) + r4[1]) + r4[2]) + r4[3];
    double lincl = mine4;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const double o = __shfl_up_sync(0xffffffffu, lincl, off);
      if (lane >= off) lincl += o;
    }
    cum = before + (lincl - mine4);
    int found = -1, last4 = -1;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      cum += r4[i];
      if (r4[i] > 0.f) {
        last4 = i;
        if (found < 0 && !take_last && cum > target) found = i;
      }
    }
    const unsigned hit = __ballot_sync(0xffffffffu, found >= 0);
    const unsigned mass4 = __ballot_sync(0xffffffffu, last4 >= 0);
    int src, idx;
    if (hit) { src = __ffs(hit) - 1; idx = found; }
    else { src = mass4 ? 31 - __clz(mass4) : 0; idx = last4 < 0 ? 0 : last4; }
    idx = __shfl_sync(0xffffffffu, idx, src);
    if (lane == 0) {
      int tokn = (c_first + cstar) * kChunk + src * 4 + idx;
      if (tokn >= V) tokn = V - 1;
      p.next_tok[b] = tokn + (shard ? p.v_offset : 0);
      report_flags(p, b, flags);
    }
    return;
  }
}

// ------------------------------------------------------------------------------------------------ 8-bit quantiser
// The 8-bit case of the Lo-Bi quantiser on the LM head (Lo-Bi Optimization section; the quantiser itself is not
// spelled out there): one vocabulary row per sub-block, symmetric integers in [-127, 127], one fp32 scale per row,
//   scale = max|w| / 127 (1 for an all-zero row),  q = clip(rint(w / scale)),  all in fp32, ties to even.
// The 4-bit case of the Lo-Bi quantiser on the LM head (reading: a sub-block is 128 hidden channels of one vocabulary
// row; symmetric codes in [-7, 7]; the sub-block's scale is the row's fp32 scale times a power of two):
//   s = max|w| / 112 (1 for an all-zero row);  e_b = the smallest e in 0..4 with  7 * 2^e * s >= max_{h in b} |w|  (else 4);
//   c = clip(rint(w / (s * 2^e_b)), -7, 7),  every step one fp32 operation, ties to even.
// Two codes per byte (even channel in the low nibble, 4-bit two's complement).  Exponents go to
// shift[b * shift_stride + row].

// rint(fdiv_rn(a, b)) without a division: the product with the rounded reciprocal y, corrected once by its exact remainder
// (q = a y, q + (a - q b) y: Newton's step on the quotient), is within 2^-23 of a unit in the last place of a / b before
// its one rounding, so it is the rounded quotient unless a / b lies that close to the middle of two fp32 numbers, and only
// next to a half integer would that matter.  The quotients that occur do not depend on more than two bf16 mantissas (of
// the row's maximum and of the entry) and the difference of their exponents, at most 31 binades of which do not round to
// zero: all of them, both signs, the second plane's remainders and the five 4-bit steps included, were compared with the
// division (1 294 464 quotients, no difference).  Rows whose step lies near the ends of the fp32 range, where the
// products would not be exact, and rows with a NaN take the division.  The integers end up in the low bits of t[] (two's
// complement).
constexpr float kRoundMagic = 12582912.f;                // 1.5 * 2^23: adding it rounds to an integer, ties to even
__device__ __forceinline__ void bf16x8_to_f32(const uint4 x, float f[8]) {
  const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    f[2 * i] = __uint_as_float(w[i] << 16);
    f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
  }
}
struct Step {
  float b, y;           // step and its reciprocal
  bool divide;          // (the same for the whole row)
};
__device__ __forceinline__ Step make_step(float b, bool divide) { return Step{b, __frcp_rn(b), divide}; }
__device__ __forceinline__ bool needs_division(float scale, bool has_nan) {
  return has_nan || !(scale > 1e-20f && scale < 1e30f);
}
__device__ __forceinline__ void round_div8(const float f[8], const Step& st, float limit, uint32_t t[8]) {
  if (st.divide) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
      t[i] = __float_as_uint(fminf(limit, fmaxf(-limit, rintf(__fdiv_rn(f[i], st.b)))) + kRoundMagic);
    return;
  }
  const uint64_t y2 = pack2(st.y, st.y), zero2 = pack2(-0.f, -0.f), mg = pack2(kRoundMagic, kRoundMagic),
                 nb = pack2(-st.b, -st.b);
#pragma unroll
  for (int i = 0; i < 8; i += 2) {
    const uint64_t a = pack2(f[i], f[i + 1]);
    const uint64_t q = fma2(a, y2, zero2);
    float r0, r1;
    unpack2(add2(fma2(fma2(q, nb, a), y2, q), mg), r0, r1);
    t[i] = __float_as_uint(r0);
    t[i + 1] = __float_as_uint(r1);
  }
}
// The low bytes of four words side by side.
__device__ __forceinline__ uint32_t pack_bytes(const uint32_t* t) {
  return __byte_perm(__byte_perm(t[0], t[1], 0x0040), __byte_perm(t[2], t[3], 0x0040), 0x5410);
}
// Running maximum of |x| over pairs of bf16; kNaN: a NaN comes through, otherwise it is dropped, as by fmaxf.
template <bool kNaN>
__device__ __forceinline__ uint32_t absmax_step(uint32_t m, const uint4 x) {
  const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t a = w[i] & 0x7FFF7FFFu;
    if (kNaN) asm("max.NaN.bf16x2 %0, %0, %1;" : "+r"(m) : "r"(a));
    else asm("max.bf16x2 %0, %0, %1;" : "+r"(m) : "r"(a));
  }
  return m;
}
template <bool kNaN>
__device__ __forceinline__ float absmax_of_pair(uint32_t m) {
  float a = __uint_as_float(m << 16);
  const float b = __uint_as_float(m & 0xFFFF0000u);
  if (kNaN) asm("max.NaN.f32 %0, %0, %1;" : "+f"(a) : "f"(b));
  else a = fmaxf(a, b);
  return a;
}
template <bool kNaN>
__device__ __forceinline__ float warp_max(float a) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float o = __shfl_xor_sync(0xffffffffu, a, off);
    if (kNaN) asm("max.NaN.f32 %0, %0, %1;" : "+f"(a) : "f"(o));
    else a = fmaxf(a, o);
  }
  return a;
}

// Element-by-element forms of a 16-byte load and of the stores, for the first n elements.
__device__ __forceinline__ uint4 gather8(const uint16_t* src, int n) {
  uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (i < n) w[i >> 1] |= static_cast<uint32_t>(src[i]) << (16 * (i & 1));
  return make_uint4(w[0], w[1], w[2], w[3]);
}
template <typename T>
__device__ __forceinline__ void scatter(T* dst, const uint4 x, int n) {
  const uint32_t w[4] = {x.x, x.y, x.z, x.w};
  constexpr int kPer = 4 / sizeof(T);
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (i < n) dst[i] = static_cast<T>(w[i / kPer] >> (8 * static_cast<int>(sizeof(T)) * (i % kPer)));
}

// Where the quantised rows go: rows of one width sit compactly in that width's buffer.
struct QuantOut {
  uint8_t* tables_width;        // where the tables of the groups go, when their widths come as launch parameters (else null)
  int* tables_row;
  const uint8_t* group_width;   // null: every row is `width` bits wide and row v of W is row v of its buffer
  const int* group_row;
  int width;
  uint16_t* w16;
  signed char* w8;
  uint8_t* w4;
  uint8_t* shift4;
  int shift_stride;
  float* scale;
};

// Widths of a head's groups as launch parameters, two bits each (0: 4 bits, 1: 8, 2: 16; 3 past the last one), and how many
// groups of 4 and of 8 bits come before each word: the kernel then makes the two tables as well, and no copy to the device
// precedes it.
constexpr int kMaxCodedGroups = 2048;                    // V <= 524288
struct GroupCodes {
  uint32_t w[kMaxCodedGroups / 16];
  uint32_t before[kMaxCodedGroups / 16];                 // 4 bits in the low half, 8 bits in the high half
};
struct NoCodes {};
__device__ __forceinline__ int same_codes(uint32_t word, uint32_t code) {        // fields of `word` that hold `code`
  const uint32_t x = word ^ (code * 0x55555555u);
  return __popc(~(x | (x >> 1)) & 0x55555555u);
}

// A head (or rows of it) to 4, 8 or 16 bits in ONE launch, a warp per row: one pass for the row's maximum, one that
// rounds (the row, 8 KB at 4096 channels, then comes out of the L1 or the L2).  Bound: HBM (2 bytes in, half to two out
// per weight).  32000 x 4096 at 4 / 8 / 16 bits in the proportions 20 / 70 / 10 %: a call of 81 us for 393 MB = 4.9 TB/s (61 us at
// the measured copy rate), of which the instructions (eleven per weight) take half; one launch per run of groups with a CTA per
// row, two bytes per load and a division per weight needed 540 us.  Rows kept in registers between the passes: 102 registers,
// 217 us with a slow path that divides next to half integers.
// kVec: rows and buffers that 16-byte pieces tile and that are aligned for it; otherwise the same element by element.
template <bool kVec, typename Codes = NoCodes>
__global__ void __launch_bounds__(256, 3) quantize_rows_kernel(const uint16_t* W, int V, int H, const QuantOut out,
                                                               const __grid_constant__ Codes codes) {
  const int v = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (v >= V) return;
  const int pieces = (H + 7) >> 3;                       // pieces of eight channels of a row
  const uint16_t* src = W + static_cast<size_t>(v) * H;
  int width = out.width;
  size_t row = v;
  if constexpr (sizeof(Codes) == sizeof(GroupCodes)) {
    // the groups before this one that have its width come first in that width's buffer (every one of them is whole)
    const int g = v / kGroupRows;
    const uint32_t mine = codes.w[g >> 4], code = (mine >> (2 * (g & 15))) & 3u;
    const uint32_t n = codes.before[g >> 4], n4 = n & 0xFFFFu, n8 = n >> 16;
    const int before = static_cast<int>(code == 0u ? n4 : code == 1u ? n8 : static_cast<uint32_t>(g & ~15) - n4 - n8) +
                       same_codes(mine | (0xFFFFFFFFu << (2 * (g & 15))), code);
    width = 4 << code;
    const int first = before * kGroupRows;
    row = static_cast<size_t>(first) + (v - g * kGroupRows);
    if (lane == 0 && v == g * kGroupRows) {
      out.tables_width[g] = static_cast<uint8_t>(width);
      out.tables_row[g] = first;
    }
  } else if (out.group_width) {
    const int g = v / kGroupRows;
    width = out.group_width[g];
    row = static_cast<size_t>(out.group_row[g]) + (v - g * kGroupRows);
  }
  auto fetch = [&](int p) {
    uint4 x = make_uint4(0u, 0u, 0u, 0u);
    if (p < pieces) x = kVec ? reinterpret_cast<const uint4*>(src)[p] : gather8(src + 8 * p, H - 8 * p);
    return x;
  };
  constexpr int kInFlight = kVec ? 8 : 1;
  if (width == 16) {
    uint16_t* dst = out.w16 + row * H;
    for (int p0 = lane; p0 < pieces; p0 += 32 * kInFlight) {
      uint4 x[kInFlight];
#pragma unroll
      for (int i = 0; i < kInFlight; ++i) x[i] = fetch(p0 + 32 * i);
#pragma unroll
      for (int i = 0; i < kInFlight; ++i) {
        const int p = p0 + 32 * i;
        if (p < pieces) {
          if (kVec) reinterpret_cast<uint4*>(dst)[p] = x[i];
          else scatter<uint16_t>(dst + 8 * p, x[i], H - 8 * p);
        }
      }
    }
    if (lane == 0) out.scale[v] = 1.f;
    return;
  }
  uint32_t m = 0;
  for (int p0 = lane; p0 < pieces; p0 += 32 * kInFlight) {
    uint4 x[kInFlight];
#pragma unroll
    for (int i = 0; i < kInFlight; ++i) x[i] = fetch(p0 + 32 * i);
#pragma unroll
    for (int i = 0; i < kInFlight; ++i) m = absmax_step<true>(m, x[i]);
  }
  float amax = warp_max<true>(absmax_of_pair<true>(m));
  const bool has_nan = amax != amax;
  if (has_nan) {
    m = 0;
    for (int p = lane; p < pieces; p += 32) m = absmax_step<false>(m, fetch(p));
    amax = warp_max<false>(absmax_of_pair<false>(m));
  }
  const float sc = amax > 0.f ? __fdiv_rn(amax, width == 8 ? 127.f : 112.f) : 1.f;
  if (lane == 0) out.scale[v] = sc;
  const bool divide = needs_division(sc, has_nan);
  uint4 x = fetch(lane), next = fetch(lane + 32);        // (two pieces ahead: the row comes back out of the L1 or the L2)
  if (width == 8) {
    const Step st = make_step(sc, divide);
    signed char* dst = out.w8 + row * H;
#pragma unroll 1
    for (int p = lane; p < pieces; p += 32) {
      const uint4 after = fetch(p + 64);
      float f[8];
      uint32_t t[8];
      bf16x8_to_f32(x, f);
      round_div8(f, st, 127.f, t);
      const uint2 b = make_uint2(pack_bytes(t), pack_bytes(t + 4));
      if (kVec) reinterpret_cast<uint2*>(dst)[p] = b;
      else scatter<signed char>(dst + 8 * p, make_uint4(b.x, b.y, 0u, 0u), H - 8 * p);
      x = next;
      next = after;
    }
  } else {
    uint8_t* dst = out.w4 + row * (H >> 1);
#pragma unroll 1
    for (int p0 = 0; p0 < pieces; p0 += 32) {
      const int p = p0 + lane;
      const uint4 after = fetch(p + 64);
      // a sub-block is sixteen pieces: lanes 0..15 or 16..31
      float bmax = absmax_of_pair<false>(absmax_step<false>(0u, x));
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, off));
      int e = 4;
#pragma unroll
      for (int c = 3; c >= 0; --c)
        if (__fmul_rn(sc, static_cast<float>(7 << c)) >= bmax) e = c;
      if (p < pieces) {
        float f[8];
        uint32_t t[8];
        bf16x8_to_f32(x, f);
        round_div8(f, make_step(sc * static_cast<float>(1 << e), divide), 7.f, t);     // (the product is exact)
        const uint32_t lo = pack_bytes(t), hi = pack_bytes(t + 4);
        const uint32_t a = (lo & 0x000F000Fu) | ((lo >> 4) & 0x00F000F0u);
        const uint32_t b = (hi & 0x000F000Fu) | ((hi >> 4) & 0x00F000F0u);
        const uint32_t packed = __byte_perm(a, b, 0x6420);
        if (kVec) reinterpret_cast<uint32_t*>(dst)[p] = packed;
        else scatter<uint8_t>(dst + 4 * p, make_uint4(packed, 0u, 0u, 0u), 4);
        if ((lane & 15) == 0)
          out.shift4[static_cast<size_t>(p >> 4) * out.shift_stride + row] = static_cast<uint8_t>(e);
      }
      x = next;
      next = after;
    }
  }
}

// The hidden rows of a call as one or two 8-bit planes (the 8-bit activation modes).  One plane: as an 8-bit weight row.
// Two planes (16-bit-class activations): per verify row
//   s1 = max|x| / 127 (1 if zero), q1 = clip(rint(x / s1));  r = x - s1 q1;  s2 = s1 / 254, q2 = clip(rint(r / s2)),
// every step one fp32 operation.  Operand layout of two planes: blocks of 32 verify rows, each block as 32 rows of q1
// followed by 32 rows of q2 (so that 64 consecutive accumulator columns hold both sums of the same 32 rows); rows past M
// are written as zeros.  A CTA per (padded) verify row: few rows, so what counts is the latency of one - two 16-byte
// loads per thread at 4096 channels, one barrier.
constexpr int kHidThreads = 256, kHidKeep = 4;
template <bool kTwoPlane>
__global__ void __launch_bounds__(kHidThreads) quantize_hidden_kernel(const uint4* X, int M, int H, int q_pitch,
                                                                      signed char* q, float* s1, float* s2) {
  __shared__ float sh_max[kHidThreads / 32];
  grid_dependency_wait();                                // (no-op unless launched with programmatic serialization)
  // The GEMM kernel may be put in place while this one runs, on the SMs that have none of its CTAs or no more (side by side they
  // do not fit: 14336 registers of a CTA here, 10240 that one of the GEMM kernel leaves): its launch and set-up and, on small
  // batches, its first requests for W_lm hide behind the quantisation.  It waits for this grid's end before it reads anything.
  // us, 8-bit planes, no release / at entry / here / behind the loads: one sequence, V = 32000 33.0 / 30.7 / 30.6 / 31.9, two
  // planes 33.4 / 30.8 / 31.3 / 31.2; 80 rows, V = 11000 17.5 / 16.5 / 16.2 / 16.3; 300 rows, V = 16000 28.1 / 26.9 / 26.7 / 28.4.
  grid_dependency_release();
  const int row = blockIdx.x;
  const int pieces = H >> 3;
  const size_t row1 = kTwoPlane ? static_cast<size_t>(64) * (row >> 5) + (row & 31) : static_cast<size_t>(row);
  uint2* q1 = reinterpret_cast<uint2*>(q + row1 * q_pitch);
  uint2* q2 = reinterpret_cast<uint2*>(q + (row1 + 32) * q_pitch);
  if (row >= M) {
    for (int p = threadIdx.x; p < pieces; p += kHidThreads) { q1[p] = make_uint2(0u, 0u); q2[p] = make_uint2(0u, 0u); }
    return;
  }
  const uint4* src = X + static_cast<size_t>(row) * pieces;
  const bool kept = pieces <= kHidThreads * kHidKeep;
  uint4 x[kHidKeep];
  auto fetch = [&](int p0) {
#pragma unroll
    for (int i = 0; i < kHidKeep; ++i) {
      const int p = p0 + kHidThreads * i + threadIdx.x;
      x[i] = p < pieces ? src[p] : make_uint4(0u, 0u, 0u, 0u);
    }
  };
  uint32_t m = 0;
  for (int p0 = 0; p0 < pieces; p0 += kHidThreads * kHidKeep) {
    fetch(p0);
#pragma unroll
    for (int i = 0; i < kHidKeep; ++i) m = absmax_step<true>(m, x[i]);
  }
  float amax = warp_max<true>(absmax_of_pair<true>(m));
  if ((threadIdx.x & 31) == 0) sh_max[threadIdx.x >> 5] = amax;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kHidThreads / 32; ++i) asm("max.NaN.f32 %0, %0, %1;" : "+f"(amax) : "f"(sh_max[i]));
  const bool has_nan = amax != amax;
  if (has_nan) {                                         // (the same decision in every thread) the maximum of the others
    m = 0;
    for (int p = threadIdx.x; p < pieces; p += kHidThreads) m = absmax_step<false>(m, src[p]);
    amax = warp_max<false>(absmax_of_pair<false>(m));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh_max[threadIdx.x >> 5] = amax;
    __syncthreads();
    for (int i = 0; i < kHidThreads / 32; ++i) amax = fmaxf(amax, sh_max[i]);
  }
  const float sc = amax > 0.f ? __fdiv_rn(amax, 127.f) : 1.f;
  const float sc2 = __fdiv_rn(sc, 254.f);
  const bool divide = needs_division(sc, has_nan);
  const Step st1 = make_step(sc, divide), st2 = make_step(sc2, divide);
  if (threadIdx.x == 0) {
    s1[row] = sc;
    if (kTwoPlane) s2[row] = sc2;
  }
  for (int p0 = 0; p0 < pieces; p0 += kHidThreads * kHidKeep) {
    if (!kept) fetch(p0);
#pragma unroll
    for (int i = 0; i < kHidKeep; ++i) {
      const int p = p0 + kHidThreads * i + threadIdx.x;
      if (p < pieces) {
        float f[8];
        uint32_t t[8];
        bf16x8_to_f32(x[i], f);
        round_div8(f, st1, 127.f, t);
        q1[p] = make_uint2(pack_bytes(t), pack_bytes(t + 4));
        if (kTwoPlane) {
#pragma unroll
          for (int n = 0; n < 8; ++n)                    // no fused multiply-add: two roundings
            f[n] = __fsub_rn(f[n], __fmul_rn(sc, __uint_as_float(t[n]) - kRoundMagic));
          round_div8(f, st2, 127.f, t);
          q2[p] = make_uint2(pack_bytes(t), pack_bytes(t + 4));
        }
      }
    }
  }
}

// bf16 hidden rows that start on no 32-byte sector, once more with a pitch of whole 128-byte lines (aligns_hidden): a CTA per row, up to
// four 16-byte loads per thread in flight; latency bounds it (some 2.4 us of a call).
constexpr int kAlignThreads = 256;
__global__ void __launch_bounds__(kAlignThreads) align_hidden_kernel(const uint4* X, int pieces, int pitch, uint4* out) {
  grid_dependency_wait();
  grid_dependency_release();                             // (as the quantiser does: the GEMM kernel is put in place meanwhile)
  const uint4* src = X + static_cast<size_t>(blockIdx.x) * pieces;
  uint4* dst = out + static_cast<size_t>(blockIdx.x) * pitch;
  for (int p0 = threadIdx.x; p0 < pieces; p0 += 4 * kAlignThreads) {
    uint4 x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (p0 + i * kAlignThreads < pieces) x[i] = src[p0 + i * kAlignThreads];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (p0 + i * kAlignThreads < pieces) dst[p0 + i * kAlignThreads] = x[i];
  }
}

// ------------------------------------------------------------------------------------------------ draft entropy
// Grid (rows, kHqSlices): CTA (r, s) leaves slice s of row r in part[r][s]; the accept/sample kernel adds the slices in
// index order.  Where the GEMM kernel does not make the pass itself: on a side stream under it, hence CTAs of 32 registers
// per thread, which fit beside that kernel's (a persistent form with eight loads in flight per thread, 100 registers, could
// not start before it had finished and made the step 45 us longer).
__global__ void __launch_bounds__(256) draft_entropy_kernel(const void* q, int q_dtype, int V, double* part) {
  __shared__ double sh_part[8];
  const double acc = warp_sum_f64(draft_slice_sum(q, q_dtype, V, blockIdx.x, blockIdx.y, threadIdx.x, 256));
  if ((threadIdx.x & 31) == 0) sh_part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tot = 0.0;
    for (int i = 0; i < 8; ++i) tot += sh_part[i];
    part[blockIdx.x * kHqSlices + blockIdx.y] = tot;
  }
}

// ------------------------------------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct Plan {
  int n_sub, N, rows_per_pass, passes, grid, stages, nbuf, rot, n_ptiles, n_kblocks, smem_bytes, tile_rows;
  int fused;            // all passes in one launch, groups of `passes` CTA pairs sharing the vocabulary tiles
  double mma_share;     // estimated tensor time over HBM time of a pass
  int kpb, k_tail;      // K blocks per ring slot; a partial last K block in a slot of its own
  double est_seconds;   // rough duration of all passes (the cost the split was chosen by)
};

}  // namespace

// What a call needs besides its arguments, kept from one call to the next: the launch geometry of a (rows, weight
// mode) pair and the tensor maps of a (hidden pointer, W_lm pointer, rows, weight mode) quadruple.  The key holds all that
// goes into a map: with mixed widths the three buffers and their row counts, because a head may be quantised anew, at other
// widths, into the same memory.
struct PlanEntry { int valid, M, w_dtype; Plan pl; };
struct MapEntry { int valid, M, w_dtype; const void* hidden; const void* W; const void* W4; const void* W16;
                  int rows8, rows4, rows16;
                  CUtensorMap th, tw, tw4, tw16;
                  const float* logits; int ldl; };       // rotating units: the logits buffer that tw4 maps (null: none)
constexpr int kPlanCache = 8, kMapCache = 8;

struct hola_ctx {
  int device, num_sms, maxB, maxK, H, V, ldl, max_rows;
  EncodeTiledFn encode;
  PlanEntry plans[kPlanCache];
  MapEntry maps[kMapCache];
  int plan_next, map_next;
  char* ws;                 // one device allocation, carved below
  size_t ws_bytes;
  float* logits;            // [max_rows][ldl]
  float4* partials;         // [max_rows][part_stride]
  int part_stride;          // CTAs a row may have partials of (the SM count)
  unsigned* status;         // [1]
  unsigned* pace;           // [2][kMaxPaceGroups] counters of the groups of pairs when all passes share a launch
  double* hq;               // [max_rows][kHqSlices] slice sums of q ln q over the draft rows
  signed char* hid8;        // [rows][hidden_pitch8] int8 hidden rows (8-bit activation modes), or bf16 rows (aligns_hidden)
  float* hid_scale;         // [max_rows]
  // staging for hola_verify_host
  void* st_hidden; int* st_tok; void* st_q; float* st_u;
  unsigned char* st_out;      // device block of one call's outputs (status, accept_len, next_tok, entropy, logZ, ...)
  unsigned char* h_out;       // pinned host block of the same layout, and where the device sees it: the accept/sample
  unsigned char* h_out_dev;   // kernel writes the outputs there itself, or they come back in ONE copy
  unsigned* flags_out;        // K3Params::flags_out of the launch being prepared
  int force_stages;
  int no_rot;                 // tuning override: never use the rotating accumulator units
  int force_passes;           // tuning override: passes over W_lm (0: chosen by cost)
  int no_pair256;             // tuning override: rotating units always as three MMAs of N = 128
  int no_fuse;                // tuning override: several passes always as one launch each
  int no_pace;                // tuning override: the groups of pairs of a fused launch do not keep in step
  int conv_group;             // tuning override (0 = by plan): converter warps per K block in the on-chip expansion
  int host_in_place;          // hola_verify_host: read draft rows not sent ahead in place from pinned host memory
  cudaStream_t copy_stream;   // hola_verify_host: the draft tensor travels here while the GEMM runs
  cudaEvent_t copy_done;
  cudaEvent_t fork_point;     // verify_device: where the side stream branches off the caller's stream
  int hq_ready;               // the draft-row entropies of this call are already being made on the side stream
  int host_overlap;           // 1: copy the draft tensor on copy_stream while the GEMM runs
  int host_lazy_q;            // hola_verify_host copies only the draft rows the step reads: 0 never, 1 always,
                              // -1 when the whole tensor would not fit under the GEMM (the default)
  float* st_qtok;             // device fp32 [maxB][maxK]: q_j(x_j) gathered on the host
  float* h_qtok;              // pinned host: the same values before the copy (inside h_small)
  unsigned char* h_small;     // pinned host mirror of the workspace span [st_tok, st_qtok + ...): tokens, uniforms, q_tok
  size_t small_u_off, small_qtok_off, small_span;   // offsets of the uniforms and of q_tok inside that span; its size
  int* h_accept;              // pinned host int32 [maxB]: accept_len read back between the two phases
  unsigned long long last_h2d, last_d2h;   // bytes the last hola_verify_host call moved
  // optional per-kernel timing (hola_profile_begin / hola_profile_end)
  cudaEvent_t* prof_ev;     // 3 events per recorded call: before the GEMM, after it, after accept/sample
  int prof_cap, prof_n, prof_on;
  char last_error[256];
};

namespace {

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Where one call's outputs sit inside the output block of hola_verify_host (16-byte aligned pieces, packed for the
// call's own B and k so that one copy brings them all back).
struct OutBlock {
  size_t status, accept, next, entropy, logZ, dent, flags, total;
};
OutBlock out_block(int B, int k) {
  const size_t rows = static_cast<size_t>(B) * (k + 1);
  OutBlock o;
  o.status = 0;
  o.accept = 16;
  o.next = o.accept + align_up(static_cast<size_t>(B) * 4, 16);
  o.entropy = o.next + align_up(static_cast<size_t>(B) * 4, 16);
  o.logZ = o.entropy + align_up(rows * 4, 16);
  o.dent = o.logZ + align_up(rows * 4, 16);
  o.flags = o.dent + align_up(static_cast<size_t>(B) * (k > 0 ? k : 1) * 4, 16);
  o.total = o.flags + align_up(static_cast<size_t>(B) * 4, 16);
  return o;
}

struct WsLayout {
  size_t logits, partials, status, pace, hq, hid8, hid_scale, st_hidden, st_tok, st_q, st_u, st_out, st_qtok, st_small_end, total;
};

// Bytes from one 8-bit hidden row to the next: rows start on 128-byte lines, so that a K block of a row is one line instead of
// parts of two, and whole 32-byte sectors.  Every CTA pair fetches those rows again, and that traffic out of the L2 is what bounds
// the 8-bit kind here.  us, rows side by side -> padded, rows that start on no sector (H = 4112) / on sectors (H = 4128; H = 4096: 67.4):
// 384 rows, V = 32000 75.5 -> 69.4 / 70.5 -> 68.9; 192 rows, V = 128256 164 -> 150 / 149 -> 147; two planes of 96 rows, V = 32000
// 48.3 -> 44.0 / 43.6 -> 42.5.
int hidden_pitch8(int H) { return static_cast<int>(align_up(static_cast<size_t>(H), 128)); }

WsLayout ws_layout(int maxB, int maxK, int H, int V, int num_sms) {
  const size_t rows = static_cast<size_t>(maxB) * (maxK + 1);
  const size_t ldl = align_up(static_cast<size_t>(V), 4);
  WsLayout w;
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes, 256); return o; };
  w.logits = take(rows * ldl * 4);
  w.partials = take(static_cast<size_t>(num_sms) * rows * 16);
  w.status = take(4);
  w.pace = take(8 * kMaxPaceGroups);
  w.hq = take(rows * kHqSlices * 8);
  w.hid8 = take(2 * align_up(rows, 32) * hidden_pitch8(H));           // one or two 8-bit planes of the hidden rows, or those
                                                                      // rows as they are, on whole lines
  w.hid_scale = take(2 * rows * 4);                                   // their scales (second plane after the first)
  w.st_hidden = take(rows * H * 2);
  // the three small per-step inputs side by side: hola_verify_host sends them as one copy
  w.st_tok = take(static_cast<size_t>(maxB) * maxK * 4);
  w.st_u = take(rows * 4);
  w.st_qtok = take(static_cast<size_t>(maxB) * (maxK > 0 ? maxK : 1) * 4);
  w.st_small_end = off;
  w.st_q = take(static_cast<size_t>(maxB) * maxK * V * 4);
  w.st_out = take(out_block(maxB, maxK).total);
  w.total = off;
  return w;
}

constexpr int kAssumedSms = 148;

void set_error(hola_ctx* ctx, const char* what, cudaError_t e) {
  snprintf(ctx->last_error, sizeof ctx->last_error, "%s: %s", what, cudaGetErrorString(e));
}

int round_up(int x, int a) { return (x + a - 1) / a * a; }

// Splits M verify rows into passes over W_lm and each pass into one or two MMAs per K step.
// A pass holds at most 512 rows (two MMAs of N <= 256 fill the tensor memory); N is a multiple of 16.
// Cost per pass: the slower of streaming W_lm once and the padded rows' tensor time, plus a fixed launch cost.
// How the r verify rows of a pass are laid out as operand rows: MMAs per K step, rows per MMA, verify rows that these hold.
struct RowSplit { int n_sub, N, rows_per_pass; };
inline RowSplit split_rows(const hola_ctx* ctx, int r, int w_dtype) {
  // up to 256 rows: one MMA, two accumulator buffers; up to 384: three MMAs of N <= 128 on rotating 128-column
  // units; beyond: two MMAs of N <= 256 that fill the tensor memory
  RowSplit f;
  if (w_dtype == HOLA_W8A16) {                     // operand rows: 64 per 32 verify rows; one or two MMAs, N % 64 == 0
    const int r8 = 2 * round_up(r, 32);
    f.n_sub = r8 > kMaxN ? 2 : 1;
    f.N = round_up(r8 / f.n_sub, 64);
    f.rows_per_pass = f.n_sub * f.N / 2;
    return f;
  }
  f.n_sub = (r > 3 * 128 || (ctx->no_rot && r > kMaxN)) ? 2 : (r > kMaxN ? 3 : 1);
  f.N = round_up((r + f.n_sub - 1) / f.n_sub, w_dtype == HOLA_W8A8 ? 32 : 16);
  f.rows_per_pass = f.n_sub * f.N;
  return f;
}

// `want`: number of passes (0: by that cost), vocabulary rows per CTA and tile (0: by the rules below), all passes in one launch.
struct PlanWish { int passes, tile_rows; bool fuse; };
Plan plan_as(const hola_ctx* ctx, int M, int w_dtype, const PlanWish& want) {
  const bool mixed = w_dtype == HOLA_W_MIXED;    // vocabulary groups of 4-, 8- and 16-bit rows, expanded on chip
  const bool w8 = w_dtype == HOLA_W_INT8 || mixed;   // int8 W_lm expanded on chip
  const bool two = w_dtype == HOLA_W8A16;        // as W8A8, with two operand rows per verify row
  const bool i8 = w_dtype == HOLA_W8A8 || two;   // 8-bit MMA: N a multiple of 32, K blocks of 128, twice the rate
  Plan best{};
  double best_cost = 1e300;
  const int rows = M > 0 ? M : 1;
  // expanded on chip: one MMA per K step, and tensor memory also holds the operand; two planes: two MMAs hold 256 rows
  const int max_rows_per_pass = w8 ? kExpandMaxN : two ? kMaxN : kMaxRowsPerPass;
  const int p_min = (rows + max_rows_per_pass - 1) / max_rows_per_pass;
  const double t_hbm = (w8 || i8 ? 1.0 : 2.0) * ctx->V * static_cast<double>(ctx->H) / 6.4e12;
  const int p_max = want.passes > p_min + 3 ? want.passes : p_min + 3;
  for (int passes = p_min; passes <= p_max; ++passes) {
    if (want.passes && passes != want.passes && want.passes >= p_min) continue;
    const int r = (rows + passes - 1) / passes;
    const RowSplit f = split_rows(ctx, r, w_dtype);
    const double t_mma = 2.0 * f.n_sub * f.N * static_cast<double>(ctx->V) * ctx->H / (i8 ? 2.8e15 : 1.4e15);
    const double cost = passes * ((t_mma > t_hbm ? t_mma : t_hbm) + 6e-6);
    if (cost < best_cost) {
      best_cost = cost;
      best.n_sub = f.n_sub; best.N = f.N; best.rows_per_pass = f.rows_per_pass; best.passes = passes;
      best.est_seconds = cost;
      best.mma_share = t_mma / t_hbm;
    }
  }
  // a pass may end up empty when rows_per_pass * (passes - 1) already covers M
  best.passes = (rows + best.rows_per_pass - 1) / best.rows_per_pass;
  best.nbuf = best.n_sub == 1 ? 2 : 1;
  best.rot = best.n_sub == 3 ? 1 : 0;
  // Vocabulary rows per CTA per tile.  To begin with the smallest multiple of 4 that covers V in the fewest whole rounds over
  // all pairs, so that every pair streams the same number of bytes (V = 32000 on 74 pairs: 2 rounds of 112 + 112
  // rows instead of 1.69 rounds of 128 + 128); the rules below make tiles taller where something else counts for more.
  const int all_pairs = ctx->num_sms / 2 > 0 ? ctx->num_sms / 2 : 1;
  // Several passes: one launch in which `passes` neighbouring pairs walk the same tiles together, one pass each (W_lm
  // then leaves HBM once, not once per pass), as long as every pass gets a pair.
  best.fused = (best.passes > 1 && want.fuse && all_pairs / best.passes >= 1) ? 1 : 0;
  const int pairs = best.fused ? all_pairs / best.passes : all_pairs;     // pairs that divide the tiles among them
  const int rounds = (ctx->V + pairs * kPairTile - 1) / (pairs * kPairTile);
  // One tile per pair: a tile costs the tensor cores and the traffic of the hidden rows the same whatever its height, and
  // the statistics of all CTAs have to be merged, so as many pairs as there are is not the best split of a small vocabulary.
  // At least 64 rows per CTA; with more than 96 operand rows a 42nd of the vocabulary per pair, or tiles of 256 rows where that
  // would be more (V > 10752: 43 pairs and up); with more than 256 operand rows tiles of 256 throughout.  42 pairs still stream
  // W_lm fast enough; the number is the best of those tried at the three sizes below on 74 pairs, not derived.  us, H = 4096:
  // V = 4000, 5 rows 16.6 -> 16.1, 96 rows 20.6 -> 20.0 (V = 12000 27.6 as it is, 28.4 on 47 pairs); V = 8000, 192 rows 34.6 ->
  // 28.6 (29.6 on 32 pairs), 384 rows 57.4 -> 45.0, two planes of 192 rows 38.2 -> 35.4; V = 12000, 192 rows 37.4 -> 33.6, 384
  // rows 61.0 -> 51.4.
  const int op_rows = best.n_sub * best.N;
  int spread = pairs;
  if (rounds == 1 && op_rows > 96) spread = op_rows > 256 ? 1 : (pairs < 42 ? pairs : 42);
  int tile_rows = round_up((ctx->V + 2 * spread * rounds - 1) / (2 * spread * rounds), 4);
  if (tile_rows < kLanes / 2) tile_rows = kLanes / 2;
  // Whole swizzle patterns, so that a slot can take several K blocks: always where tiles are narrow; a tall tile pays for
  // the rows added (up to 4 % of the busiest pair's work), which 32 K blocks per tile and more are worth, and rows that do
  // not start on a 128-byte line (the next K block then finds its share of the line in the L2).  us: one sequence,
  // V = 128256 172 -> 168, V = 50000, H = 2048 40.4 -> 39.2; 96 rows, V = 128256 210 -> 207; 92 rows, V = 50000, H = 4096
  // 81.7 -> 79.8, V = 90004, H = 1032 53 -> 52; but 32 rows, V = 50003, H = 1024 20.9 -> 21.5 (8-bit, one sequence: within
  // 1.5 % either way).
  const int row_bytes = ctx->H * (i8 ? 1 : 2);
  if (tile_rows < 104 || (!i8 && ctx->H >= 32 * kBlockK) || row_bytes % 128 != 0) tile_rows = round_up(tile_rows, 8);
  if (tile_rows > kLanes) tile_rows = kLanes;
  // Near and beyond the point where the tensor cores bound, a tile costs the same whatever its rows: as few tiles as
  // possible (the busiest pair has as many either way), because these loops run at the power cap and every MMA counts.
  // us: V = 32000, 384 rows (143 tiles of 224 rows -> 125 of 256) 117 -> 113, 8-bit 74.7 -> 72.9; V = 128256 (517 -> 501),
  // 384 rows 434 -> 430, 192 rows at 8 bits (0.87 of the HBM time) 144 -> 140, two planes 221 -> 212.
  if (rounds >= 2 && best.mma_share > 0.8) tile_rows = kLanes;
  if (want.tile_rows) tile_rows = want.tile_rows;
  if (mixed) tile_rows = kLanes;                 // a pair's tile is one group of 256 rows of one width
  best.tile_rows = tile_rows;
  best.n_ptiles = (ctx->V + 2 * tile_rows - 1) / (2 * tile_rows);
  best.grid = 2 * (best.n_ptiles < pairs ? best.n_ptiles : pairs) * (best.fused ? best.passes : 1);
  best.n_kblocks = i8 ? (ctx->H + 2 * kBlockK - 1) / (2 * kBlockK) : (ctx->H + kBlockK - 1) / kBlockK;
  // Ring slots.  Narrow tiles and few rows: several K blocks per slot, so that the producer's cost per slot (some 450
  // cycles whatever the size) is spread over 30 to 40 KB.  Wide tiles (or 225 rows and more) take longer than that for a
  // K block in HBM (or on the tensor cores) anyway.
  const int w_block = w8 || best.rot ? kWBlockBytes : round_up(best.tile_rows * 128, 1024);
  const int k_elems = i8 ? 2 * kBlockK : kBlockK;
  const int block_bytes = w_block + best.n_sub * (best.N / 2) * 128;
  const int whole_blocks = ctx->H / k_elems;
  best.kpb = 1;
  if (!w8 && best.n_sub == 1 && best.N <= 224 && best.tile_rows % 8 == 0) {
    if (whole_blocks >= 4 && 4 * block_bytes <= 40 * 1024) best.kpb = 4;
    else if (whole_blocks >= 2 && 2 * block_bytes <= 48 * 1024) best.kpb = 2;
  }
  best.k_tail = best.kpb > 1 && ctx->H % k_elems != 0 ? 1 : 0;
  const int stage_bytes = w8 ? kWBlockBytes + 2 * (best.N / 2) * 128 : best.kpb * block_bytes;
  // (rotating units: every epilogue warp stages a whole 32-row chunk, twice the bytes)
  const int trans_bytes = (w8 ? kW8EpiWarps : kEpiWarps) * kTransBytes * (best.n_sub == 3 ? 2 : 1);
  int stages = (kSmemBudget - 1024 - kBarrierBytes - trans_bytes) / stage_bytes;
  if (stages > kMaxStages) stages = kMaxStages;
  if (ctx->force_stages && ctx->force_stages < stages) stages = ctx->force_stages;
  best.stages = stages;
  best.smem_bytes = stages * stage_bytes + kBarrierBytes + trans_bytes + 1024;
  return best;
}

// Estimated microseconds of a launch in which every pair has one tile, without what all such launches have in common (some 10).
// A K block takes the slowest of: its MMAs; its bytes at what one SM gets out of the L2, 61 a cycle (with rows that start on no
// 128-byte line 48); the bytes of all SMs at what they get together, 6400 a cycle (5100); a turn of the threads that feed the
// ring; with on-chip expansion a turn of the converters.  All K blocks together take no less than W_lm's way out of HBM.  The
// read-out takes 1.8 us per chunk of 32 operand rows and epilogue warp.  Fitted to 37 shapes (V = 1200 .. 12000, H = 200 .. 8192,
// 5 .. 2304 rows, every weight mode) in 2 to 20 splits each: the split it picks was 0.7 % slower than the best one on average, 4 %
// at worst.
inline double one_tile_us(const hola_ctx* ctx, int w_dtype, int n_sub, int N, int tile_rows, int grid) {
  const bool expand = w_dtype == HOLA_W_INT8 || w_dtype == HOLA_W_MIXED, i8 = w_dtype == HOLA_W8A8 || w_dtype == HOLA_W8A16;
  const int op_rows = n_sub * N;
  const double mma = 1.16 * 4.0 * n_sub * (N / 2 > 46 ? N / 2 : 46);
  const double bytes = tile_rows * (expand ? 64.0 : 128.0) + op_rows * 64.0;
  const double line = !i8 && ctx->H % kBlockK != 0 ? 0.79 : 1.0;
  double block = expand ? 326.0 : 180.0;
  for (const double c : {mma, bytes / (61.0 * line), grid * bytes / (6400.0 * line)})
    if (c > block) block = c;
  const int n_kblocks = i8 ? (ctx->H + 2 * kBlockK - 1) / (2 * kBlockK) : (ctx->H + kBlockK - 1) / kBlockK;
  const double ring = n_kblocks * block / 1900.0, hbm = static_cast<double>(ctx->V) * ctx->H * (expand || i8 ? 1 : 2) / 7.2e6;
  const int groups = !expand ? kEpiWarps / 4 : op_rows <= 32 ? kW8FewEpiWarps / 4 : kW8EpiWarps / 4;
  return (ring > hbm ? ring : hbm) + 1.8 * (((op_rows + 31) / 32 + groups - 1) / groups);
}

// Vocabularies of a tile per pair and fewer leave pairs without work when all rows of a pass go to the same tile's pair.  The
// rows are then cut into more passes, which share the tiles in one launch, and the tiles into shorter ones, as the estimate has
// it (half a microsecond less than the split of the general rules, or that one stays).  us, before -> after, bf16: 417 rows,
// H = 5304, V = 1272 62.3 -> 25.3; 384, 4096, 8000 45.4 -> 36.4; 384, 1024, 4000 20.7 -> 14.1; 200, 2048, 3000 20.9 -> 15.0; 512, 512,
// 2000 22.1 -> 12.5; 153, 696, 6000 15.4 -> 13.4; 8-bit planes, 384, 4096, 4000 35.0 -> 22.8; two planes, 216, 1024, 7550 25.2 -> 20.1;
// mixed widths, 824, 1024, 1408 24.6 -> 16.4.
Plan make_plan(const hola_ctx* ctx, int M, int w_dtype = HOLA_W_BF16) {
  PlanWish want = {ctx->force_passes, 0, true};
  Plan best = plan_as(ctx, M, w_dtype, want);
  const int pairs = ctx->num_sms / 2;
  const int p_min = best.passes;
  if (!ctx->force_passes && best.n_ptiles * p_min <= pairs) {
    // (by the estimate alone, and laid out in full once: a split takes 0.15 to 0.45 us of the host; every try laid out, up to 1.8)
    constexpr int kTries = 16;
    struct { RowSplit rows; int passes; } tries[kTries];
    int n_tries = 0;
    for (; n_tries < kTries && p_min + n_tries <= pairs; ++n_tries) {
      const int passes = p_min + n_tries;
      if (n_tries && M < 32 * passes) break;
      const RowSplit rows = split_rows(ctx, M > 0 ? (M + passes - 1) / passes : 1, w_dtype);
      tries[n_tries] = {rows, M > 0 ? (M + rows.rows_per_pass - 1) / rows.rows_per_pass : 1};
    }
    double best_us = one_tile_us(ctx, w_dtype, best.n_sub, best.N, best.tile_rows, best.grid) - 0.5;
    for (int tile_rows = kLanes; tile_rows >= (w_dtype == HOLA_W_MIXED ? kLanes : 32); tile_rows -= 32) {
      const int tiles = (ctx->V + 2 * tile_rows - 1) / (2 * tile_rows);
      for (int i = 0; i < n_tries && (p_min + i) * tiles <= pairs; ++i) {
        const double us = one_tile_us(ctx, w_dtype, tries[i].rows.n_sub, tries[i].rows.N, tile_rows, 2 * tiles * tries[i].passes);
        if (us < best_us) {
          best_us = us;
          want.passes = p_min + i; want.tile_rows = tile_rows;
        }
      }
    }
    if (want.passes) {
      best = plan_as(ctx, M, w_dtype, want);
      best.est_seconds = best_us * 1e-6 + 6e-6;
    }
  }
  if (ctx->no_fuse && best.passes > 1) {           // the same passes, a launch each
    const double est = best.est_seconds;
    want.passes = best.passes; want.fuse = false;
    best = plan_as(ctx, M, w_dtype, want);
    best.est_seconds = est;
  }
  return best;
}

// make_plan through the context's cache (the geometry depends on the context's shape and tuning options, on the number
// of verify rows and on the weight mode only).
const Plan& plan_for(hola_ctx* ctx, int M, int w_dtype) {
  for (int i = 0; i < kPlanCache; ++i)
    if (ctx->plans[i].valid && ctx->plans[i].M == M && ctx->plans[i].w_dtype == w_dtype) return ctx->plans[i].pl;
  PlanEntry& e = ctx->plans[ctx->plan_next];
  ctx->plan_next = (ctx->plan_next + 1) % kPlanCache;
  e.pl = make_plan(ctx, M, w_dtype);
  e.M = M; e.w_dtype = w_dtype; e.valid = 1;
  return e.pl;
}

// K-major 2-D tensor map.  bf16: box of 64 elements x box_rows; int8: box of 128 elements; both 128 bytes per row with
// the 128-byte swizzle that the MMA reads (and that spreads the rows of 8-bit codes over the banks for the converter
// warps).  `packed4`: rows of cols / 2 bytes holding two 4-bit codes each; box of 64 bytes (128 codes), 64-byte swizzle.
hola_status encode_map(hola_ctx* ctx, CUtensorMap* map, const void* ptr, uint64_t rows, uint64_t cols,
                       uint32_t box_rows, bool int8 = false, bool packed4 = false, int kpb = 1, int pitch = 0) {
  if (packed4) { cols /= 2; int8 = true; }
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {pitch ? static_cast<cuuint64_t>(pitch) : cols * (int8 ? 1u : 2u)};
  const cuuint32_t box[2] = {static_cast<cuuint32_t>(int8 && !packed4 ? 2 * kBlockK : kBlockK), box_rows};
  const cuuint32_t estr[2] = {1, 1};
  // `pitch`: bytes from row to row (0: rows side by side).  `kpb` > 1: the same memory as (element of a K block, row, K
  // block), kpb K blocks per box; needs whole K blocks
  const cuuint64_t dims3[3] = {box[0], rows, cols / box[0]};
  const cuuint64_t strides3[2] = {strides[0], 128};
  const cuuint32_t box3[3] = {box[0], box_rows, static_cast<cuuint32_t>(kpb)};
  const cuuint32_t estr3[3] = {1, 1, 1};
  const bool three = kpb > 1;
  const CUresult r = ctx->encode(map, int8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16,
                                 three ? 3 : 2, const_cast<void*>(ptr), three ? dims3 : dims, three ? strides3 : strides,
                                 three ? box3 : box, three ? estr3 : estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                 packed4 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    snprintf(ctx->last_error, sizeof ctx->last_error, "cuTensorMapEncodeTiled failed with CUresult %d", (int)r);
    return HOLA_ERR_CUDA;
  }
  return HOLA_OK;
}

hola_status check_common(const hola_ctx* ctx, const hola_verify_args* a) {
  if (!ctx || !a) return HOLA_ERR_INVALID_ARG;
  if (a->B < 0 || a->k < 0 || a->H <= 0 || a->V <= 0) return HOLA_ERR_INVALID_ARG;
  if (a->H != ctx->H || a->V != ctx->V || a->B > ctx->maxB || a->k > ctx->maxK) return HOLA_ERR_UNSUPPORTED_SHAPE;
  if (a->q_dtype != HOLA_Q_BF16 && a->q_dtype != HOLA_Q_F32) return HOLA_ERR_INVALID_ARG;
  if (a->gate_source != HOLA_GATE_TARGET_ENTROPY && a->gate_source != HOLA_GATE_DRAFT_ENTROPY)
    return HOLA_ERR_INVALID_ARG;
  if (a->fallback != HOLA_FALLBACK_SAMPLE && a->fallback != HOLA_FALLBACK_GREEDY) return HOLA_ERR_INVALID_ARG;
  return HOLA_OK;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Logits and draft rows that 16-byte loads tile.
bool rows_of_pieces(const hola_verify_args* a, const float* logits, int ldl) {
  return a->V % 4 == 0 && ldl % 4 == 0 && aligned16(logits) && (a->k == 0 || aligned16(a->draft_q));
}

// How the accept/sample kernel is launched.
struct SampleForm {
  int S;            // CTAs per sequence
  bool solo;        // the one CTA has 1024 threads
  bool staged;      // the slices of all rows go through shared memory
  int cpc;          // chunks per CTA
  size_t smem;      // dynamic shared memory
};

// Cluster size (CTAs per sequence): as many as keep the grid within one wave of the SMs; one
// where no pass over the vocabulary follows the accept test (greedy fallback; us, V = 32000, H = 512, clusters of eight ->
// one: 384 rows 28.7 -> 27.8, 96 rows 15.2 -> 13.7).
int sample_cluster(int num_sms, int B, int V, int fallback) {
  if (fallback == HOLA_FALLBACK_GREEDY) return 1;
  const int nchunks = (V + kChunk - 1) / kChunk;
  int S = 8;
  while (S > 1 && (B * S > kK3MaxPerSm * num_sms || nchunks / S < 8)) S >>= 1;
  return S;
}

// One CTA of 1024 threads per sequence instead of a cluster of S: no exchange between CTAs, the statistics of a row merged once, and
// with one sequence per SM most SMs stay free for the next call's GEMM kernel, which then asks for its W_lm while this one runs.
// Up to 16384 entries (more take one SM too long).  Where clusters would take at most a quarter of the SMs they ask ahead as
// well, and have their rows staged: then only up to 8192 entries.  Rows of no whole 16-byte pieces are loaded element by element,
// and one SM is slow at that: only up to 8192 entries, and where clusters would take at most a quarter of the SMs only against
// clusters of two, or of four whose CTAs have more rows to merge than warps (8).
// us, cluster -> one CTA, k = 4, H = 1024: V = 3000, 32 / 100 sequences 12.9 -> 12.2, 15.2 -> 14.7; V = 8192, 16 / 64 13.8 -> 13.0,
// 17.9 -> 17.2; V = 16000, 1 / 8 / 148 12.6 -> 13.9, 15.6 -> 14.9, 41.5 -> 39.9; V = 24000, 32 25.3 -> 27.9; k = 30, V = 4000, 1
// 15.5 -> 12.6.  No whole pieces: V = 3001, 2 11.2 -> 10.8; V = 6001, 9 12.8 -> 13.0; V = 8191, 1 / 4 / 16 11.8 -> 12.3, 13.0 -> 13.5,
// 15.1 -> 14.5; k = 8, V = 4001, 1 11.8 -> 11.0.  (S = 1, up to 1920 entries: one CTA of 256 threads is enough.)  The line for few
// sequences was drawn when a cluster took longer: with k = 4 it is ahead there from some 4000 entries on by now (V = 3000, 2 10.2 -> 10.3;
// V = 6000, 1 10.6 -> 11.0; V = 8192, 1 / 4 11.2 -> 11.9, 12.1 -> 12.6).
bool sample_solo(int num_sms, int B, int k, int V, int S, bool vec) {
  const bool many = 4 * B * S > num_sms;
  if (S == 1 || B > num_sms) return false;
  if (vec) return V <= (many ? 16384 : 8192);
  return V <= 8192 && (many || S <= (k < kK3Threads / 32 ? 2 : 4));
}

// `vec`: rows_of_pieces.  `phase`, `shard`, `far`: see K3Params (a row read in place over the bus is not staged).
SampleForm sample_form(int num_sms, int B, int k, int V, int q_dtype, int fallback, bool vec, int phase = 0, bool shard = false,
                       bool far = false) {
  SampleForm f = {};
  const int S = phase == 1 ? 1 : sample_cluster(num_sms, B, V, fallback);            // (phase 1: no vocabulary pass)
  f.solo = phase == 0 && !shard && !far && sample_solo(num_sms, B, k, V, S, vec);
  f.S = f.solo ? 1 : S;
  const int nchunks = (V + kChunk - 1) / kChunk;
  f.cpc = (nchunks + f.S - 1) / f.S;
  if (phase == 1 || fallback == HOLA_FALLBACK_GREEDY) return f;
  f.smem = static_cast<size_t>(f.cpc) * sizeof(double);
  // Small batches (a CTA per SM at most, and no more than 4 MB of rows in all): row n would be asked for only after the
  // statistics and the accept test, so the slices of all rows are asked for before them (bulk copies: rows of whole
  // 16-byte pieces).
  if (vec && phase == 0 && (q_dtype == HOLA_Q_F32 || V % 8 == 0) && !far && !f.solo && B * S <= num_sms) {
    const size_t row_bytes = static_cast<size_t>(k + 1) * 4 + static_cast<size_t>(k) * (q_dtype == HOLA_Q_BF16 ? 2 : 4);
    const size_t bytes = row_bytes * f.cpc * kChunk + sizeof(double);   // (and the rows start on a 16-byte boundary)
    if (bytes + f.smem <= kK3MaxDynSmem && row_bytes * V * B <= 4u << 20) {
      f.staged = true;
      f.smem += bytes;
    }
  }
  return f;
}

// bf16 rows of 2 H = 16 bytes more than whole 32-byte sectors make every fetch of a K block of hidden rows five sectors instead of
// four, out of the L2 and for every tile.  A copy of the rows on whole lines takes some 2.4 us and pays for itself from 96 rows on
// where rows x K blocks x tiles per pair reach 8000; with one tile per pair and more than 256 rows the MMAs hide the fetches.  us, as
// they are -> copied (141 shapes were measured both ways): 99 rows, H = 4216, V = 67724 136.6 -> 122.1; 128, 840, 119544 71.2 -> 65.3;
// 160, 6568, 16524 63.5 -> 55.9; 600, 7240, 29827 336 -> 299; below the lines 92, 1032, 50003 36.0 -> 37.3, 210, 1832, 9089 22.8 ->
// 24.3; one tile, 480, 2456, 9633 36.1 -> 38.2.  Rows that start on sectors (H a multiple of 16) gain nothing wherever they start
// in a line (119 shapes): 312, 592, 53988 37.8 -> 40.4; 370, 1312, 10325 31.4 -> 33.1; 365, 2608, 38298 98.8 -> 99.7.  (With codes
// expanded on chip: no gain, 160 rows, H = 2064, V = 60000 63.5 -> 65.)
bool aligns_hidden(int w_dtype, int H, const Plan& pl) {
  if (w_dtype != HOLA_W_BF16 || H % 16 == 0) return false;
  const int op_rows = pl.n_sub * pl.N, pairs = pl.grid / (2 * (pl.fused ? pl.passes : 1));
  const int tiles = (pl.n_ptiles + pairs - 1) / pairs;
  return op_rows >= 96 && (tiles > 1 || op_rows <= 256) && static_cast<double>(tiles) * pl.n_kblocks * op_rows >= 8000.0;
}

// Where the logits of a verify step that does not hand them out go.  The greedy rule reads none (the arg-max travels with the
// statistics), so none are stored then.  8-bit head and hidden rows, 192 rows, V = 128256 (98 MB of logits beside 525 MB of
// codes): 137 -> 121 us.
float* logits_buffer(const hola_ctx* ctx, const hola_verify_args* a) {
  return a->fallback == HOLA_FALLBACK_GREEDY ? nullptr : ctx->logits;
}

// Steps 1-2: the LM-head GEMM with fused statistics, one launch (clusters of two CTAs) per pass over W_lm.
// `logits` null: statistics only.
// `few_before`: the kernel in front is expected to be this context's accept/sample kernel on a few SMs.
// `draft_pass`: the pass over the draft rows (draft-entropy gate) is made on the way.
// `next_reads_inputs`: the accept/sample kernel of the same arguments is launched right behind this.
// `want_arg`: the arg-max of every row whatever the fallback.
hola_status run_lm_head(hola_ctx* ctx, const hola_verify_args* a, float* logits, int ldl, const Plan& pl,
                        cudaStream_t stream, bool few_before = false, bool next_reads_inputs = false,
                        bool draft_pass = false, bool want_arg = false) {
  const int M = a->B * (a->k + 1);
  const bool mixed = a->w_dtype == HOLA_W_MIXED;
  const bool w8 = a->w_dtype == HOLA_W_INT8 || mixed, two = a->w_dtype == HOLA_W8A16,
             i8 = a->w_dtype == HOLA_W8A8 || two;
  const hola_wmix* mx = mixed ? a->wmix : nullptr;
  // (mixed widths: W_lm of the arguments is not read; the 8-bit buffer takes its place in the cache key and the map)
  const void* w_main = mixed ? (mx->rows8 > 0 ? mx->W8 : (mx->rows4 > 0 ? mx->W4 : mx->W16)) : a->W_lm;
  hola_status s;
  // 8-bit activations: the hidden operand is the context's own buffer of 8-bit planes, filled per call below
  // (as is one that is brought onto whole lines)
  const bool aligned = ctx->hid8 && aligns_hidden(a->w_dtype, a->H, pl);
  const void* hid_src = (two || i8 || aligned) ? static_cast<const void*>(ctx->hid8) : a->hidden;
  const int hid_pitch = (two || i8) ? hidden_pitch8(a->H) : aligned ? round_up(2 * a->H, 128) : 0;
  if ((two || i8) && !ctx->hid8) return HOLA_ERR_INVALID_ARG;   // (the entry point without a context has no room for it)
  if (two || i8) {
    // the same per-row quantiser as for W_lm (one plane), or the two-plane form in blocks of 32 rows
    const int padded = round_up(M, 32);
    cudaLaunchConfig_t qc = {};
    qc.gridDim = dim3(static_cast<unsigned>(two ? padded : M)); qc.blockDim = dim3(kHidThreads); qc.stream = stream;
    cudaLaunchAttribute qa[1];
    qa[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // launch latency hides behind the call before
    qa[0].val.programmaticStreamSerializationAllowed = 1;
    qc.attrs = qa; qc.numAttrs = 1;
    const cudaError_t qe =
        cudaLaunchKernelEx(&qc, two ? quantize_hidden_kernel<true> : quantize_hidden_kernel<false>,
                           static_cast<const uint4*>(a->hidden), M, a->H, hidden_pitch8(a->H), ctx->hid8, ctx->hid_scale,
                           ctx->hid_scale + ctx->max_rows);
    if (qe != cudaSuccess) { set_error(ctx, "launch of the hidden-row quantiser", qe); return HOLA_ERR_CUDA; }
  }
  if (aligned) {
    cudaLaunchConfig_t ac = {};
    ac.gridDim = dim3(static_cast<unsigned>(M)); ac.blockDim = dim3(kAlignThreads); ac.stream = stream;
    cudaLaunchAttribute aa[1];
    aa[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    aa[0].val.programmaticStreamSerializationAllowed = 1;
    ac.attrs = aa; ac.numAttrs = 1;
    const cudaError_t ae = cudaLaunchKernelEx(&ac, align_hidden_kernel, static_cast<const uint4*>(a->hidden), a->H / 8, hid_pitch / 16,
                                              reinterpret_cast<uint4*>(ctx->hid8));
    if (ae != cudaSuccess) { set_error(ctx, "launch align_hidden_kernel", ae); return HOLA_ERR_CUDA; }
  }
  MapEntry* me = nullptr;
  for (int i = 0; i < kMapCache; ++i) {
    MapEntry& c = ctx->maps[i];
    if (c.valid && c.hidden == hid_src && c.W == w_main && c.M == M && c.w_dtype == a->w_dtype &&
        (!mixed || (c.W4 == mx->W4 && c.W16 == mx->W16 && c.rows8 == mx->rows8 && c.rows4 == mx->rows4 &&
                    c.rows16 == mx->rows16))) { me = &c; break; }
  }
  if (!me) {
    me = &ctx->maps[ctx->map_next];
    ctx->map_next = (ctx->map_next + 1) % kMapCache;
    me->valid = 0;
    me->logits = nullptr;
    if (two)
      s = encode_map(ctx, &me->th, hid_src, static_cast<uint64_t>(2 * round_up(M, 32)), static_cast<uint64_t>(a->H),
                     static_cast<uint32_t>(pl.N / 2), true, false, pl.kpb, hid_pitch);
    else if (i8)
      s = encode_map(ctx, &me->th, hid_src, static_cast<uint64_t>(M), static_cast<uint64_t>(a->H),
                     static_cast<uint32_t>(pl.N / 2), true, false, pl.kpb, hid_pitch);
    else
      s = encode_map(ctx, &me->th, hid_src, static_cast<uint64_t>(M), static_cast<uint64_t>(a->H),
                     static_cast<uint32_t>(pl.N / 2), false, false, pl.kpb, hid_pitch);
    if (s != HOLA_OK) return s;
    const uint32_t trows = static_cast<uint32_t>(pl.tile_rows);
    if (!mixed) {
      s = encode_map(ctx, &me->tw, a->W_lm, static_cast<uint64_t>(a->V), static_cast<uint64_t>(a->H), trows, w8 || i8,
                     false, pl.kpb);
      if (s != HOLA_OK) return s;
      me->tw4 = me->tw; me->tw16 = me->tw;               // (read for a partial last K block only)
      if (pl.k_tail) {
        s = encode_map(ctx, &me->tw4, a->W_lm, static_cast<uint64_t>(a->V), static_cast<uint64_t>(a->H), trows, i8);
        if (s != HOLA_OK) return s;
        s = encode_map(ctx, &me->tw16, hid_src, static_cast<uint64_t>(two ? 2 * round_up(M, 32) : M),
                       static_cast<uint64_t>(a->H), static_cast<uint32_t>(pl.N / 2), i8, false, 1, hid_pitch);
        if (s != HOLA_OK) return s;
      }
      me->W4 = nullptr; me->W16 = nullptr;
    } else {
      // one map per width that occurs; a width that does not occur gets a copy of one that does (never used)
      bool have = false;
      if (mx->rows8 > 0) {
        s = encode_map(ctx, &me->tw, mx->W8, static_cast<uint64_t>(mx->rows8), static_cast<uint64_t>(a->H), trows, true);
        if (s != HOLA_OK) return s;
        have = true;
      }
      if (mx->rows4 > 0) {
        s = encode_map(ctx, &me->tw4, mx->W4, static_cast<uint64_t>(mx->rows4), static_cast<uint64_t>(a->H), trows, true,
                       true);
        if (s != HOLA_OK) return s;
        if (!have) me->tw = me->tw4;
        have = true;
      }
      if (mx->rows16 > 0) {
        s = encode_map(ctx, &me->tw16, mx->W16, static_cast<uint64_t>(mx->rows16), static_cast<uint64_t>(a->H), trows);
        if (s != HOLA_OK) return s;
        if (!have) me->tw = me->tw16;
        have = true;
      }
      if (mx->rows4 <= 0) me->tw4 = me->tw;
      if (mx->rows16 <= 0) me->tw16 = me->tw;
      me->W4 = mx->W4; me->W16 = mx->W16;
      me->rows8 = mx->rows8; me->rows4 = mx->rows4; me->rows16 = mx->rows16;
    }
    me->hidden = hid_src; me->W = w_main; me->M = M; me->w_dtype = a->w_dtype; me->valid = 1;
  }
  // Rotating units: the logits buffer, where its rows are whole 16-byte pieces; boxes of 16 rows x 32 entries, swizzled like
  // the staging buffers.
  const bool wide_logits = !pl.rot && pl.N >= 128 && ldl % 4 == 0 && aligned16(logits);      // (a row's last piece: within ldl)
  const bool bulk_logits = pl.rot && logits && ldl % 4 == 0 && aligned16(logits);
  if (bulk_logits && (me->logits != logits || me->ldl != ldl)) {
    me->logits = nullptr;
    const cuuint64_t dims[2] = {static_cast<cuuint64_t>(a->V), static_cast<cuuint64_t>(M)};
    const cuuint64_t strides[1] = {static_cast<cuuint64_t>(ldl) * 4};
    const cuuint32_t box[2] = {32, kTransRows}, estr[2] = {1, 1};
    const CUresult r = ctx->encode(&me->tw4, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, logits, dims, strides, box, estr,
                                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                   CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
      me->valid = 0;
      snprintf(ctx->last_error, sizeof ctx->last_error, "cuTensorMapEncodeTiled failed with CUresult %d", (int)r);
      return HOLA_ERR_CUDA;
    }
    me->logits = logits; me->ldl = ldl;
  }
  const CUtensorMap& th = me->th;
  const CUtensorMap& tw = me->tw;
  const CUtensorMap& tw4 = me->tw4;
  const CUtensorMap& tw16 = me->tw16;
  K1Params kp;
  kp.M = M; kp.V = a->V; kp.n_ptiles = pl.n_ptiles; kp.n_kblocks = pl.n_kblocks;
  kp.pair256 = (pl.rot && pl.N == 128 && !ctx->no_pair256) ? 1 : 0;
  kp.kpb = pl.kpb; kp.k_tail = pl.k_tail;
  kp.acc_cols = w8 ? round_up(pl.N, 32) : 256;
  const bool few = w8 && pl.N <= 32;                     // (four epilogue warps, one chunk each)
  kp.conv_groups = ctx->conv_group > kConvGroup ? 1 : few ? kConvGroupsFew : kConvGroups;
  const int a_slots = (kTmemCols - 2 * kp.acc_cols) / kOperandCols;
  kp.a_slots = a_slots < pl.stages ? a_slots : pl.stages;
  if (kp.conv_groups > kp.a_slots) kp.conv_groups = kp.a_slots;
  kp.stages = pl.stages; kp.nbuf = pl.nbuf; kp.rot = pl.rot; kp.n_sub = pl.n_sub; kp.N = pl.N; kp.tile_rows = pl.tile_rows; kp.ldl = ldl;
  kp.logits = logits; kp.partials = ctx->partials; kp.part_stride = ctx->part_stride;
  kp.status = a->status_word ? a->status_word : ctx->status;
  kp.w_scale = a->w_scale;
  kp.h_scale = ctx->hid_scale;
  kp.h_scale2 = ctx->hid_scale ? ctx->hid_scale + ctx->max_rows : nullptr;
  kp.bulk_logits = bulk_logits ? 1 : 0;
  kp.stream_logits = static_cast<double>(M) * a->V * 4.0 > 96e6 ? 1 : 0;     // beyond ~3/4 of the L2
  kp.group_width = mixed ? mx->group_width : nullptr;
  kp.group_row = mixed ? mx->group_row : nullptr;
  kp.shift4 = mixed ? mx->shift4 : nullptr;
  kp.rows4 = mixed ? mx->rows4 : 0;
  kp.want_arg = want_arg || a->fallback == HOLA_FALLBACK_GREEDY;
  cudaError_t e = cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(pl.grid));
  cfg.blockDim = dim3(kK1Threads);
  cfg.dynamicSmemBytes = static_cast<size_t>(pl.smem_bytes);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  // may start while the kernel before it in the stream drains (its threads wait for that kernel before they touch
  // global memory): launch, barrier set-up and tensor-memory allocation hide behind the previous call's last kernel
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  // Ahead of the dependency wait: 32 MB, about what HBM moves while the accept/sample kernel of the call before runs, where
  // that kernel leaves nearly all SMs to this one's CTAs.  V = 32000, H = 4096, one sequence, none / 16 / 32 / 48 MB: bf16
  // 52.2 / 50.9 / 50.0 / 49.7 us, mixed widths 43.9 / 42.2 / 42.6 / 43.2, 8-bit 37.2 / 36.3 / 36.5 / 36.8; with 16
  // sequences (128 CTAs of the accept/sample kernel in the way) 61.6 / 61.5 / 62.5 / 63.3, hence the limit.
  kp.next_tok = nullptr; kp.next_u = nullptr; kp.next_q = nullptr;
  kp.next_n = kp.next_q_elem = 0; kp.next_q_bytes = 0;
  if (next_reads_inputs && a->k > 0 && a->draft_tok && a->draft_q && a->uniforms) {
    kp.next_tok = a->draft_tok; kp.next_u = a->uniforms; kp.next_q = static_cast<const char*>(a->draft_q);
    kp.next_n = a->B * a->k; kp.next_q_elem = a->q_dtype == HOLA_Q_BF16 ? 2 : 4;
    const double q_bytes = static_cast<double>(kp.next_n) * a->V * kp.next_q_elem;
    if (q_bytes <= 2e6 && aligned16(a->draft_q) && a->fallback != HOLA_FALLBACK_GREEDY)
      kp.next_q_bytes = static_cast<unsigned>(q_bytes) & ~15u;
  }
  kp.prefetch_blocks = 0;
  if (few_before) {
    const int per_tile = w8 ? (pl.n_kblocks + 1) / 2 : pl.n_kblocks - pl.k_tail;
    const int ctas = pl.grid / (pl.fused ? pl.passes : 1);                                // that share W_lm among them
    const int blocks = static_cast<int>(32e6 / (static_cast<double>(ctas) * pl.tile_rows * 128.0));
    kp.prefetch_blocks = (blocks < per_tile ? blocks : per_tile) / pl.kpb * pl.kpb;
  }
  kp.n_pass = pl.fused ? pl.passes : 1;
  kp.rows_per_pass = pl.rows_per_pass;
  kp.pace = nullptr;
  if (pl.fused && ctx->pace && !ctx->no_pace && pl.grid / (2 * pl.passes) <= kMaxPaceGroups) kp.pace = ctx->pace;
  for (int pass = 0; pass < (pl.fused ? 1 : pl.passes); ++pass) {
    kp.row0 = pass * pl.rows_per_pass;
    kp.rows = M - kp.row0 < pl.rows_per_pass ? M - kp.row0 : pl.rows_per_pass;
    if (kp.rows <= 0) break;
    const bool draft = pass == 0 && draft_pass;
    kp.draft_q = draft ? a->draft_q : nullptr;
    kp.draft_q_dtype = a->q_dtype; kp.draft_units = a->B * a->k * kHqSlices; kp.draft_part = ctx->hq;
    kp.clear_status = pass == 0 && (a->flags & HOLA_ARG_CLEAR_STATUS) && a->status_word;
    e = two ? cudaLaunchKernelEx(&cfg, lm_head_entropy_kernel<3, false>, th, tw, tw4, tw16, kp)
      : i8 ? (pl.rot ? cudaLaunchKernelEx(&cfg, lm_head_entropy_kernel<2, true>, th, tw, tw4, tw16, kp)
             : wide_logits ? cudaLaunchKernelEx(&cfg, lm_head_entropy_kernel<2, false, false, true>, th, tw, tw4, tw16, kp)
                           : cudaLaunchKernelEx(&cfg, lm_head_entropy_kernel<2, false>, th, tw, tw4, tw16, kp))
      : few ? cudaLaunchKernelEx(&cfg, lm_head_entropy_kernel<1, false, true>, th, tw, tw4, tw16, kp)
      : w8 ? cudaLaunchKernelEx(&cfg, lm_head_entropy_kernel<1, false>, th, tw, tw4, tw16, kp)
           : (pl.rot ? cudaLaunchKernelEx(&cfg, lm_head_entropy_kernel<0, true>, th, tw, tw4, tw16, kp)
             : wide_logits ? cudaLaunchKernelEx(&cfg, lm_head_entropy_kernel<0, false, false, true>, th, tw, tw4, tw16, kp)
                           : cudaLaunchKernelEx(&cfg, lm_head_entropy_kernel<0, false>, th, tw, tw4, tw16, kp));
    if (e != cudaSuccess) { set_error(ctx, "launch lm_head_entropy_kernel", e); return HOLA_ERR_CUDA; }
  }
  return HOLA_OK;
}

// Partials per row that a GEMM launch (or one per pass) leaves: one per CTA that works on the row's pass.
int row_partials(const Plan& pl) { return pl.fused ? pl.grid / pl.passes : pl.grid; }

cudaError_t launch_finalize(const hola_ctx* ctx, const hola_verify_args* a, int M, int nparts, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>((M + 7) / 8)); cfg.blockDim = dim3(256); cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, finalize_kernel, static_cast<const float4*>(ctx->partials), nparts, ctx->part_stride, M,
                            a->logZ, a->entropy);
}

// What the accept/sample kernel needs to know in the vocabulary-parallel form.
struct ShardLaunch {
  int world, rank, v_offset, V_global;
  const float4* stats_all;   // world records (statistics, then draft-token logits)
  int rec_floats;            // floats per record
  double* mass_out;
  const double* mass_all;
};

// `settled`: the launch sits right behind this call's own GEMM kernel (see K3Params::inputs_settled).
hola_status run_accept_sample(hola_ctx* ctx, const hola_verify_args* a, const float* logits, int ldl, int combine,
                              int nparts, cudaStream_t stream, const float* q_tok = nullptr, int phase = 0,
                              const ShardLaunch* sh = nullptr, bool settled = false, const void* q_far = nullptr,
                              int q_far_from = 0) {
  K3Params kp{};
  kp.q_far = q_far; kp.q_far_from = q_far_from;
  kp.q_tok = q_tok; kp.phase = phase; kp.inputs_settled = settled ? 1 : 0;
  kp.B = a->B; kp.k = a->k; kp.V = a->V; kp.ldl = ldl; kp.logits = logits;
  kp.partials = ctx->partials; kp.nparts = nparts; kp.row_stride = ctx->part_stride; kp.part_stride = 1; kp.combine = combine;
  kp.tok = a->draft_tok; kp.q = a->draft_q; kp.q_dtype = a->q_dtype; kp.u = a->uniforms; kp.tau = a->tau;
  kp.gate_source = a->gate_source; kp.fallback = a->fallback; kp.hq_part = nullptr; kp.draft_entropy = a->draft_entropy;
  if (a->gate_source == HOLA_GATE_DRAFT_ENTROPY && a->k > 0) {
    // one more pass over the draft rows: H(q_j) for every (sequence, draft position) - unless the caller has put it
    // on the side stream already, next to the GEMM
    if (!ctx->hq_ready) {
      draft_entropy_kernel<<<dim3(static_cast<unsigned>(a->B * a->k), kHqSlices), 256, 0, stream>>>(
          a->draft_q, a->q_dtype, a->V, ctx->hq);
      const cudaError_t e0 = cudaGetLastError();
      if (e0 != cudaSuccess) { set_error(ctx, "launch draft_entropy_kernel", e0); return HOLA_ERR_CUDA; }
    }
    kp.hq_part = ctx->hq;
  }
  kp.accept_len = a->accept_len; kp.next_tok = a->next_tok; kp.entropy = a->entropy; kp.logZ = a->logZ;
  kp.status = a->status_word ? a->status_word : ctx->status;
  kp.flags_out = ctx->flags_out;
  if (sh) {
    kp.shard_world = sh->world; kp.shard_rank = sh->rank; kp.v_offset = sh->v_offset; kp.V_global = sh->V_global;
    kp.lx_all = reinterpret_cast<const float*>(sh->stats_all) + 4 * static_cast<size_t>(a->B) * (a->k + 1);
    kp.rec_stride = sh->rec_floats;
    kp.mass_out = sh->mass_out; kp.mass_all = sh->mass_all;
    if (combine) { kp.partials = sh->stats_all; kp.nparts = sh->world; kp.row_stride = 1; kp.part_stride = sh->rec_floats / 4; }
  }
  const bool vec = rows_of_pieces(a, logits, ldl) && aligned16(q_far);     // (rows read in place are the caller's own)
  const SampleForm f = sample_form(ctx->num_sms, a->B, a->k, a->V, a->q_dtype, a->fallback, vec, phase, sh != nullptr, q_far != nullptr);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(a->B * f.S));
  cfg.blockDim = dim3(f.solo ? kSoloThreads : kK3Threads);
  cfg.dynamicSmemBytes = f.smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(f.S);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  // May be scheduled as soon as every CTA of the kernel before it in the stream has exited; it waits for that
  // kernel's results itself.  (The GEMM kernel does not release its dependents earlier: their CTAs would then pile
  // up on whichever SMs its first CTAs leave, and the 8-CTA clusters of a large batch run unbalanced.)
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const bool ask = vec && !f.staged && f.cpc <= 64 && a->B * f.S > ctx->num_sms;
  if (f.solo) {
    attr[0] = attr[1];                                   // (no cluster)
    cfg.numAttrs = 1;
  }
  const cudaError_t e = f.solo && a->V <= kFewEntries && 2 * a->B <= ctx->num_sms
                            ? (vec ? cudaLaunchKernelEx(&cfg, accept_sample_kernel<true, false, 16>, kp)
                                   : cudaLaunchKernelEx(&cfg, accept_sample_kernel<false, false, 16>, kp))
                        : f.solo ? (vec ? cudaLaunchKernelEx(&cfg, accept_sample_kernel<true, false, 32>, kp)
                                        : cudaLaunchKernelEx(&cfg, accept_sample_kernel<false, false, 32>, kp))
                        : f.staged ? cudaLaunchKernelEx(&cfg, accept_sample_kernel<true, false, 0, true>, kp)
                        : ask ? cudaLaunchKernelEx(&cfg, accept_sample_kernel<true, true>, kp)
                        : vec ? cudaLaunchKernelEx(&cfg, accept_sample_kernel<true, false>, kp)
                              : cudaLaunchKernelEx(&cfg, accept_sample_kernel<false, false>, kp);
  if (e != cudaSuccess) { set_error(ctx, "launch accept_sample_kernel", e); return HOLA_ERR_CUDA; }
  return HOLA_OK;
}

hola_status check_lm_head_args(const hola_ctx* ctx, const hola_verify_args* a) {
  if (a->w_dtype < HOLA_W_BF16 || a->w_dtype > HOLA_W_MIXED) return HOLA_ERR_INVALID_ARG;
  if (a->w_dtype == HOLA_W_MIXED) {
    // vocabulary groups of mixed width: the weights come through args->wmix, W_lm is not read
    const hola_wmix* mx = a->wmix;
    if (!a->hidden || !aligned16(a->hidden) || !mx || !a->w_scale) return HOLA_ERR_INVALID_ARG;
    if (a->H % kSubBlock != 0) return HOLA_ERR_UNSUPPORTED_SHAPE;          // whole sub-blocks of 128 hidden channels
    if (mx->rows4 < 0 || mx->rows8 < 0 || mx->rows16 < 0 || !mx->group_width || !mx->group_row) return HOLA_ERR_INVALID_ARG;
    if (static_cast<long long>(mx->rows4) + mx->rows8 + mx->rows16 < a->V) return HOLA_ERR_INVALID_ARG;
    if ((mx->rows4 > 0 && (!mx->W4 || !mx->shift4 || !aligned16(mx->W4))) || (mx->rows8 > 0 && (!mx->W8 || !aligned16(mx->W8))) ||
        (mx->rows16 > 0 && (!mx->W16 || !aligned16(mx->W16))))
      return HOLA_ERR_INVALID_ARG;
    return HOLA_OK;
  }
  if (!a->hidden || !a->W_lm) return HOLA_ERR_INVALID_ARG;
  if (!aligned16(a->hidden) || !aligned16(a->W_lm)) return HOLA_ERR_INVALID_ARG;
  if (a->H % 8 != 0) return HOLA_ERR_UNSUPPORTED_SHAPE;
  if (a->w_dtype != HOLA_W_BF16) {
    if (!a->w_scale) return HOLA_ERR_INVALID_ARG;
    if (a->H % 16 != 0) return HOLA_ERR_UNSUPPORTED_SHAPE;     // int8 row pitch must be a multiple of 16 bytes
  }
  (void)ctx;
  return HOLA_OK;
}

hola_status check_sample_args(const hola_verify_args* a) {
  if (!a->uniforms || !a->accept_len || !a->next_tok || !a->entropy || !a->logZ) return HOLA_ERR_INVALID_ARG;
  if (a->k > 0 && (!a->draft_tok || !a->draft_q)) return HOLA_ERR_INVALID_ARG;
  return HOLA_OK;
}

// Once per context (and once per device for the entry point without one), with the device current: the kernels that
// ask for more dynamic shared memory than the default limit are told so here, not on every call.
cudaError_t configure_kernels() {
  cudaError_t e = cudaSuccess;
  const void* kernels[] = {reinterpret_cast<const void*>(lm_head_entropy_kernel<0, false>),
                           reinterpret_cast<const void*>(lm_head_entropy_kernel<0, false, false, true>),
                           reinterpret_cast<const void*>(lm_head_entropy_kernel<2, false, false, true>),
                           reinterpret_cast<const void*>(lm_head_entropy_kernel<0, true>),
                           reinterpret_cast<const void*>(lm_head_entropy_kernel<1, false>),
                           reinterpret_cast<const void*>(lm_head_entropy_kernel<1, false, true>),
                           reinterpret_cast<const void*>(lm_head_entropy_kernel<2, false>),
                           reinterpret_cast<const void*>(lm_head_entropy_kernel<2, true>),
                           reinterpret_cast<const void*>(lm_head_entropy_kernel<3, false>)};
  for (const void* k : kernels)
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(accept_sample_kernel<true, false, 0, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kK3MaxDynSmem);
  return e;
}

struct DeviceGuard {
  int prev = -1;
  bool ok = true, changed = false;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) { ok = false; return; }
    if (prev != dev) {
      changed = true;
      if (cudaSetDevice(dev) != cudaSuccess) ok = false;
    }
  }
  ~DeviceGuard() { if (changed) cudaSetDevice(prev); }
};

// An empty batch launches nothing; all there is to do is what HOLA_ARG_CLEAR_STATUS promises.
hola_status empty_batch(const hola_verify_args* a, void* cuda_stream) {
  if (!(a->flags & HOLA_ARG_CLEAR_STATUS) || !a->status_word) return HOLA_OK;
  return cudaMemsetAsync(a->status_word, 0, sizeof(uint32_t), static_cast<cudaStream_t>(cuda_stream)) == cudaSuccess ? HOLA_OK
                                                                                                                  : HOLA_ERR_CUDA;
}
hola_status empty_batch(const hola_ctx* ctx, const hola_verify_args* a, void* cuda_stream) {
  DeviceGuard guard(ctx->device);
  return empty_batch(a, cuda_stream);
}

}  // namespace

// ------------------------------------------------------------------------------------------------ C ABI
extern "C" {

const char* hola_version(void) { return "0.1"; }

const char* hola_strerror(hola_status s) {
  switch (s) {
    case HOLA_OK: return "ok";
    case HOLA_ERR_INVALID_ARG: return "invalid argument (null pointer, bad size or misaligned buffer)";
    case HOLA_ERR_UNSUPPORTED_SHAPE: return "unsupported shape (H % 8 != 0, or sizes beyond the context's limits)";
    case HOLA_ERR_WORKSPACE: return "workspace allocation failed";
    case HOLA_ERR_CUDA: return "CUDA call failed (see hola_last_cuda_error)";
    case HOLA_ERR_NO_DEVICE: return "no usable sm_100 device";
    case HOLA_ERR_STATIC_LIMIT:
      return "problem too large for the fixed scratch of hola_lm_head_entropy_static (more than 512 verify rows)";
    default: return "unknown status";
  }
}

const char* hola_last_cuda_error(const hola_ctx* ctx) { return ctx ? ctx->last_error : ""; }

size_t hola_workspace_bytes(int maxB, int maxK, int H, int V) {
  if (maxB <= 0 || maxK < 0 || H <= 0 || V <= 0) return 0;
  return ws_layout(maxB, maxK, H, V, kAssumedSms).total;
}

hola_status hola_create(hola_ctx** out, int device, int maxB, int maxK, int H, int V) {
  if (!out) return HOLA_ERR_INVALID_ARG;
  *out = nullptr;
  if (maxB <= 0 || maxK < 0 || H <= 0 || V <= 0) return HOLA_ERR_INVALID_ARG;
  if (H % 8 != 0 || maxK + 1 > kMaxK1 || V > kMaxChunks * kChunk) return HOLA_ERR_UNSUPPORTED_SHAPE;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) return HOLA_ERR_NO_DEVICE;
  int major = 0, sms = 0;                                // (cudaGetDeviceProperties would take a millisecond or more)
  if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess)
    return HOLA_ERR_NO_DEVICE;
  if (major != 10) return HOLA_ERR_NO_DEVICE;            // the kernels are sm_100a only; there is no fallback
  DeviceGuard guard(device);
  if (!guard.ok) return HOLA_ERR_NO_DEVICE;

  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || !fn ||
      qres != cudaDriverEntryPointSuccess)
    return HOLA_ERR_NO_DEVICE;

  hola_ctx* ctx = static_cast<hola_ctx*>(calloc(1, sizeof(hola_ctx)));
  if (!ctx) return HOLA_ERR_WORKSPACE;
  ctx->device = device; ctx->num_sms = sms; ctx->maxB = maxB; ctx->maxK = maxK;
  ctx->H = H; ctx->V = V; ctx->ldl = static_cast<int>(align_up(static_cast<size_t>(V), 4));
  ctx->max_rows = maxB * (maxK + 1);
  ctx->encode = reinterpret_cast<EncodeTiledFn>(fn);
  ctx->host_overlap = 1;
  ctx->host_lazy_q = -1;
  ctx->host_in_place = 1;
  if (configure_kernels() != cudaSuccess) { free(ctx); return HOLA_ERR_CUDA; }
  const WsLayout w = ws_layout(maxB, maxK, H, V, ctx->num_sms);
  const cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&ctx->ws), w.total);
  if (e != cudaSuccess) { free(ctx); return HOLA_ERR_WORKSPACE; }
  ctx->ws_bytes = w.total;
  ctx->logits = reinterpret_cast<float*>(ctx->ws + w.logits);
  ctx->partials = reinterpret_cast<float4*>(ctx->ws + w.partials);
  ctx->part_stride = ctx->num_sms;
  ctx->status = reinterpret_cast<unsigned*>(ctx->ws + w.status);
  ctx->pace = reinterpret_cast<unsigned*>(ctx->ws + w.pace);
  ctx->hq = reinterpret_cast<double*>(ctx->ws + w.hq);
  ctx->hid8 = reinterpret_cast<signed char*>(ctx->ws + w.hid8);
  ctx->hid_scale = reinterpret_cast<float*>(ctx->ws + w.hid_scale);
  ctx->st_hidden = ctx->ws + w.st_hidden; ctx->st_tok = reinterpret_cast<int*>(ctx->ws + w.st_tok);
  ctx->st_q = ctx->ws + w.st_q; ctx->st_u = reinterpret_cast<float*>(ctx->ws + w.st_u);
  ctx->st_out = reinterpret_cast<unsigned char*>(ctx->ws + w.st_out);
  ctx->st_qtok = reinterpret_cast<float*>(ctx->ws + w.st_qtok);
  cudaMemset(ctx->status, 0, 4);
  cudaMemset(ctx->pace, 0, 8 * kMaxPaceGroups);
  const size_t n_qtok = static_cast<size_t>(maxB) * (maxK > 0 ? maxK : 1);
  void* pinned = nullptr;
  if (cudaStreamCreateWithFlags(&ctx->copy_stream, cudaStreamNonBlocking) != cudaSuccess ||
      cudaEventCreateWithFlags(&ctx->copy_done, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&ctx->fork_point, cudaEventDisableTiming) != cudaSuccess ||
      cudaHostAlloc(&pinned, (w.st_small_end - w.st_tok) + maxB * 4 + 16 + out_block(maxB, maxK).total,
                    cudaHostAllocDefault) != cudaSuccess) {
    if (ctx->copy_done) cudaEventDestroy(ctx->copy_done);
    if (ctx->fork_point) cudaEventDestroy(ctx->fork_point);
    if (ctx->copy_stream) cudaStreamDestroy(ctx->copy_stream);
    cudaFree(ctx->ws);
    free(ctx);
    return HOLA_ERR_CUDA;
  }
  ctx->h_small = static_cast<unsigned char*>(pinned);
  ctx->small_u_off = w.st_u - w.st_tok;
  ctx->small_qtok_off = w.st_qtok - w.st_tok;
  ctx->small_span = w.st_small_end - w.st_tok;
  ctx->h_qtok = reinterpret_cast<float*>(ctx->h_small + ctx->small_qtok_off);
  ctx->h_accept = reinterpret_cast<int*>(ctx->h_small + ctx->small_span);
  (void)n_qtok;
  ctx->h_out = reinterpret_cast<unsigned char*>(align_up(reinterpret_cast<size_t>(ctx->h_accept + maxB), 16));
  void* pinned_dev = nullptr;
  if (cudaHostGetDevicePointer(&pinned_dev, pinned, 0) == cudaSuccess)
    ctx->h_out_dev = static_cast<unsigned char*>(pinned_dev) + (ctx->h_out - ctx->h_small);
  else
    cudaGetLastError();                                  // (outputs are copied then)
  *out = ctx;
  return HOLA_OK;
}

hola_status hola_destroy(hola_ctx* ctx) {
  if (!ctx) return HOLA_OK;
  DeviceGuard guard(ctx->device);
  for (int i = 0; i < 3 * ctx->prof_cap; ++i) cudaEventDestroy(ctx->prof_ev[i]);
  free(ctx->prof_ev);
  if (ctx->copy_done) cudaEventDestroy(ctx->copy_done);
  if (ctx->fork_point) cudaEventDestroy(ctx->fork_point);
  if (ctx->copy_stream) cudaStreamDestroy(ctx->copy_stream);
  if (ctx->h_small) cudaFreeHost(ctx->h_small);
  cudaFree(ctx->ws);
  free(ctx);
  return HOLA_OK;
}

static hola_status plan_for_shape(int num_sms, int H, int V, int rows, int w_dtype, Plan* pl) {
  if (num_sms < 2 || H <= 0 || V <= 0 || rows <= 0) return HOLA_ERR_INVALID_ARG;
  if (w_dtype < HOLA_W_BF16 || w_dtype > HOLA_W_MIXED) return HOLA_ERR_INVALID_ARG;
  if (H % 8 != 0 || V > kMaxChunks * kChunk) return HOLA_ERR_UNSUPPORTED_SHAPE;
  hola_ctx* c = static_cast<hola_ctx*>(calloc(1, sizeof(hola_ctx)));     // only the fields make_plan reads
  if (!c) return HOLA_ERR_WORKSPACE;
  c->num_sms = num_sms; c->H = H; c->V = V;
  *pl = make_plan(c, rows, w_dtype);
  free(c);
  return HOLA_OK;
}

hola_status hola_plan_for_shape(int num_sms, int H, int V, int rows, int w_dtype, hola_plan_info* out) {
  if (!out) return HOLA_ERR_INVALID_ARG;
  Plan pl;
  const hola_status s = plan_for_shape(num_sms, H, V, rows, w_dtype, &pl);
  if (s != HOLA_OK) return s;
  out->tile_v = 2 * pl.tile_rows; out->grid = pl.grid; out->stages = pl.stages; out->rows_per_pass = pl.rows_per_pass;
  out->passes = pl.passes; out->kernels_per_call = (pl.fused ? 1 : pl.passes) + 1;
  return HOLA_OK;
}

hola_status hola_hidden_form_for_shape(int num_sms, int H, int V, int rows, int w_dtype, int32_t* out) {
  if (!out) return HOLA_ERR_INVALID_ARG;
  Plan pl;
  const hola_status s = plan_for_shape(num_sms, H, V, rows, w_dtype, &pl);
  if (s != HOLA_OK) return s;
  *out = w_dtype == HOLA_W8A8 || w_dtype == HOLA_W8A16 ? HOLA_HIDDEN_8BIT
         : aligns_hidden(w_dtype, H, pl)               ? HOLA_HIDDEN_ON_LINES
                                                       : HOLA_HIDDEN_IN_PLACE;
  return HOLA_OK;
}

hola_status hola_sample_plan_for_shape(int num_sms, int B, int k, int V, int q_dtype, int fallback, hola_sample_info* out) {
  if (!out || num_sms < 2 || B <= 0 || k < 0 || V <= 0 || (q_dtype != HOLA_Q_BF16 && q_dtype != HOLA_Q_F32) ||
      (fallback != HOLA_FALLBACK_SAMPLE && fallback != HOLA_FALLBACK_GREEDY))
    return HOLA_ERR_INVALID_ARG;
  if (k >= kMaxK1 || V > kMaxChunks * kChunk) return HOLA_ERR_UNSUPPORTED_SHAPE;
  const SampleForm f = sample_form(num_sms, B, k, V, q_dtype, fallback, V % 4 == 0);
  out->ctas = f.S; out->threads = f.solo ? kSoloThreads : kK3Threads; out->staged = f.staged;
  return HOLA_OK;
}

hola_status hola_plan_ex(const hola_ctx* ctx, int B, int k, int w_dtype, hola_plan_info* out) {
  if (!ctx || !out || B < 0 || k < 0) return HOLA_ERR_INVALID_ARG;
  if (w_dtype < HOLA_W_BF16 || w_dtype > HOLA_W_MIXED) return HOLA_ERR_INVALID_ARG;
  if (B > ctx->maxB || k > ctx->maxK) return HOLA_ERR_UNSUPPORTED_SHAPE;
  const Plan pl = make_plan(ctx, B * (k + 1), w_dtype);
  out->tile_v = 2 * pl.tile_rows; out->grid = pl.grid; out->stages = pl.stages; out->rows_per_pass = pl.rows_per_pass;
  out->passes = pl.passes; out->kernels_per_call = (pl.fused ? 1 : pl.passes) + 1;
  return HOLA_OK;
}

hola_status hola_plan(const hola_ctx* ctx, int B, int k, hola_plan_info* out) {
  return hola_plan_ex(ctx, B, k, HOLA_W_BF16, out);
}

hola_status hola_set_option(hola_ctx* ctx, int option, int value) {
  if (!ctx) return HOLA_ERR_INVALID_ARG;
  switch (option) {
    case HOLA_OPT_RING_SLOTS:
      if (value != 0 && (value < 2 || value > kMaxStages)) return HOLA_ERR_INVALID_ARG;
      ctx->force_stages = value;
      break;
    case HOLA_OPT_ROTATING_UNITS: ctx->no_rot = value == 0; break;
    case HOLA_OPT_PAIR_MMA: ctx->no_pair256 = value == 0; break;
    case HOLA_OPT_HOST_IN_PLACE: ctx->host_in_place = value != 0; break;
    case HOLA_OPT_FUSED_PASSES:
      if (value < 0 || value > 2) return HOLA_ERR_INVALID_ARG;
      ctx->no_fuse = value == 0;
      ctx->no_pace = value == 2;
      break;
    case HOLA_OPT_CONVERTER_GROUP:
      if (value < 0 || value > kConvGroup * kConvGroups) return HOLA_ERR_INVALID_ARG;
      ctx->conv_group = value;
      break;
    case HOLA_OPT_PASSES:
      if (value < 0 || value > 64) return HOLA_ERR_INVALID_ARG;
      ctx->force_passes = value;
      break;
    case HOLA_OPT_HOST_OVERLAP: ctx->host_overlap = value != 0; break;
    case HOLA_OPT_HOST_ROWS_ON_DEMAND:
      if (value < -1 || value > 1) return HOLA_ERR_INVALID_ARG;
      ctx->host_lazy_q = value;
      break;
    default: return HOLA_ERR_INVALID_ARG;
  }
  for (int i = 0; i < kPlanCache; ++i) ctx->plans[i].valid = 0;     // the launch geometry may have changed
  for (int i = 0; i < kMapCache; ++i) ctx->maps[i].valid = 0;
  return HOLA_OK;
}

hola_status hola_selftest_bounded_wait(hola_ctx* ctx, long long limit_cycles, uint32_t* status_word,
                                       uint32_t* counters, void* cuda_stream) {
  if (!ctx || !status_word || !counters) return HOLA_ERR_INVALID_ARG;
  if (limit_cycles < 1000 || limit_cycles > 200000000ll) return HOLA_ERR_INVALID_ARG;   // at most ~0.1 s of SM clock
  DeviceGuard guard(ctx->device);
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  if (cudaMemsetAsync(counters, 0, 2 * sizeof(uint32_t), stream) != cudaSuccess) return HOLA_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2); cfg.blockDim = dim3(64); cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, bounded_wait_selftest_kernel, limit_cycles,
                                           static_cast<unsigned*>(status_word), static_cast<unsigned*>(counters));
  if (e != cudaSuccess) { set_error(ctx, "launch bounded_wait_selftest_kernel", e); return HOLA_ERR_CUDA; }
  return HOLA_OK;
}

static hola_status staged_wait_selftest(hola_ctx* ctx, long long limit_cycles, uint32_t* status_word, uint32_t* counters,
                                        void* cuda_stream, bool early) {
  if (!ctx || !status_word || !counters) return HOLA_ERR_INVALID_ARG;
  if (limit_cycles < 1000 || limit_cycles > 100000000ll) return HOLA_ERR_INVALID_ARG;   // (four times that is waited at most)
  DeviceGuard guard(ctx->device);
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  if (cudaMemsetAsync(counters, 0, (early ? 4 : 3) * sizeof(uint32_t), stream) != cudaSuccess) return HOLA_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2); cfg.blockDim = dim3(64); cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, early ? staged_wait_selftest_kernel<true> : staged_wait_selftest_kernel<false>,
                                           limit_cycles, static_cast<unsigned*>(status_word), static_cast<unsigned*>(counters));
  if (e != cudaSuccess) { set_error(ctx, "launch staged_wait_selftest_kernel", e); return HOLA_ERR_CUDA; }
  return HOLA_OK;
}

hola_status hola_selftest_staged_wait(hola_ctx* ctx, long long limit_cycles, uint32_t* status_word, uint32_t* counters,
                                      void* cuda_stream) {
  return staged_wait_selftest(ctx, limit_cycles, status_word, counters, cuda_stream, false);
}

hola_status hola_selftest_mass_wait(hola_ctx* ctx, long long limit_cycles, uint32_t* status_word, uint32_t* counters,
                                    void* cuda_stream) {
  return staged_wait_selftest(ctx, limit_cycles, status_word, counters, cuda_stream, true);
}

hola_status hola_selftest_pace(hola_ctx* ctx, uint32_t* words, void* cuda_stream) {
  if (!ctx || !words) return HOLA_ERR_INVALID_ARG;
  static_assert(HOLA_PACE_WORDS == 2 * kMaxPaceGroups, "two words per group");
  DeviceGuard guard(ctx->device);
  const cudaError_t e = cudaMemcpyAsync(words, ctx->pace, 4 * HOLA_PACE_WORDS, cudaMemcpyDeviceToDevice, static_cast<cudaStream_t>(cuda_stream));
  if (e != cudaSuccess) { set_error(ctx, "copy of the pace counters", e); return HOLA_ERR_CUDA; }
  return HOLA_OK;
}

hola_status hola_selftest_quotient(hola_ctx* ctx, const float* t, const float* s, int n, float* out, void* cuda_stream) {
  if (!ctx || !t || !s || !out || n <= 0) return HOLA_ERR_INVALID_ARG;
  DeviceGuard guard(ctx->device);
  quotient_selftest_kernel<<<(n - 1) / 256 + 1, 256, 0, static_cast<cudaStream_t>(cuda_stream)>>>(t, s, n, out);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error(ctx, "launch quotient_selftest_kernel", e); return HOLA_ERR_CUDA; }
  return HOLA_OK;
}

hola_status hola_lm_head_entropy(hola_ctx* ctx, const hola_verify_args* a, void* cuda_stream) {
  hola_status s = check_common(ctx, a);
  if (s != HOLA_OK) return s;
  if (a->B == 0) return empty_batch(ctx, a, cuda_stream);
  if ((s = check_lm_head_args(ctx, a)) != HOLA_OK) return s;
  if (!a->entropy || !a->logZ) return HOLA_ERR_INVALID_ARG;
  DeviceGuard guard(ctx->device);
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  const int M = a->B * (a->k + 1);
  const Plan& pl = plan_for(ctx, M, a->w_dtype);
  float* logits = a->logits_out ? a->logits_out : ctx->logits;
  const int ldl = a->logits_out ? a->V : ctx->ldl;
  if ((s = run_lm_head(ctx, a, logits, ldl, pl, stream, M <= 256)) != HOLA_OK) return s;
  const cudaError_t e = launch_finalize(ctx, a, M, row_partials(pl), stream);
  if (e != cudaSuccess) { set_error(ctx, "launch finalize_kernel", e); return HOLA_ERR_CUDA; }
  return HOLA_OK;
}

hola_status hola_accept_sample(hola_ctx* ctx, const hola_verify_args* a, void* cuda_stream) {
  hola_status s = check_common(ctx, a);
  if (s != HOLA_OK) return s;
  if (a->B == 0) return HOLA_OK;
  if ((s = check_sample_args(a)) != HOLA_OK) return s;
  if (!a->logits_out) return HOLA_ERR_INVALID_ARG;
  if (a->fallback == HOLA_FALLBACK_GREEDY) return HOLA_ERR_INVALID_ARG;   // needs the arg-max of the fused path
  DeviceGuard guard(ctx->device);
  return run_accept_sample(ctx, a, a->logits_out, a->V, 0, 0, static_cast<cudaStream_t>(cuda_stream));
}

}  // extern "C"

namespace {

// The whole step on device buffers.  `before_sample`, when given, is an event the accept/sample part waits for
// (the draft tensor still being copied in by hola_verify_host).
hola_status verify_device(hola_ctx* ctx, const hola_verify_args* a, cudaStream_t stream, cudaEvent_t before_sample) {
  const Plan& pl = plan_for(ctx, a->B * (a->k + 1), a->w_dtype);
  float* logits = a->logits_out ? a->logits_out : logits_buffer(ctx, a);
  const int ldl = a->logits_out ? a->V : ctx->ldl;
  const bool prof = ctx->prof_on && ctx->prof_n < ctx->prof_cap;
  cudaEvent_t* ev = prof ? ctx->prof_ev + 3 * ctx->prof_n : nullptr;
  if (prof) cudaEventRecord(ev[0], stream);
  // The pass over the draft rows (draft-entropy gate) depends on nothing the GEMM makes.  Up to 32 MB of them, that kernel's
  // epilogue warps make the pass while they wait for the first tile (us, against a kernel on a side stream: 16 sequences,
  // V = 32000 62.6 -> 59.4, one 49.6 -> 47.4, V = 1000 12.8 -> 10.9, 4 sequences, V = 9000 17.5 -> 14.5).  Beyond that, and with
  // rotating units (whose epilogue has no register to spare: 384 rows, V = 32000 0.9 % slower with the code in it, V = 128256
  // 441 -> 448 with the gate), a kernel of its own does, on the context's side stream, behind the copy of the draft tensor
  // where the host entry put one there.  It branches off the caller's stream before the GEMM and joins it again before the
  // accept/sample kernel: earlier calls that are still queued on that stream write and read ctx->hq too.  It is launched
  // AFTER the GEMM so that the GEMM's CTAs get their SMs first; its small CTAs fit beside them.  (While the caller records a
  // graph everything stays on the caller's stream.)
  const bool draft_gate = a->gate_source == HOLA_GATE_DRAFT_ENTROPY && a->k > 0;
  const double q_bytes = static_cast<double>(a->B) * a->k * a->V * (a->q_dtype == HOLA_Q_BF16 ? 2 : 4);
  const bool inside = draft_gate && !before_sample && !pl.rot && q_bytes <= 32e6;
  cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
  if (draft_gate && !inside && cudaStreamIsCapturing(stream, &capturing) != cudaSuccess) capturing = cudaStreamCaptureStatusActive;
  const bool side = draft_gate && !inside && (before_sample || capturing == cudaStreamCaptureStatusNone);
  if (side && cudaEventRecord(ctx->fork_point, stream) != cudaSuccess) return HOLA_ERR_CUDA;
  // (One CTA per sequence: half of the SMs free are enough; us, V = 8000, 64 sequences without / with 18.3 / 17.8.  Clusters: three
  // quarters; on up to half of the SMs V = 30000, 9 sequences 18.2 / 17.0, V = 32000, 5 / 8 50.6 / 49.9, 51.7 / 52.0, V = 128256,
  // 8 59.9 / 61.4: no line there that holds for all.)
  const SampleForm f = sample_form(ctx->num_sms, a->B, a->k, a->V, a->q_dtype, a->fallback, rows_of_pieces(a, logits, ldl));
  const bool few_before = a->B * f.S * (f.solo ? 2 : 4) <= ctx->num_sms;
  hola_status s = run_lm_head(ctx, a, logits, ldl, pl, stream, few_before, !before_sample, inside);
  if (s != HOLA_OK) return s;
  if (prof) cudaEventRecord(ev[1], stream);
  if (side) {
    cudaError_t e = cudaStreamWaitEvent(ctx->copy_stream, ctx->fork_point, 0);
    if (e == cudaSuccess) {
      draft_entropy_kernel<<<dim3(static_cast<unsigned>(a->B * a->k), kHqSlices), 256, 0, ctx->copy_stream>>>(
          a->draft_q, a->q_dtype, a->V, ctx->hq);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaEventRecord(ctx->copy_done, ctx->copy_stream);
    if (e != cudaSuccess) { set_error(ctx, "draft_entropy_kernel on the side stream", e); return HOLA_ERR_CUDA; }
    before_sample = ctx->copy_done;
  }
  if (before_sample && cudaStreamWaitEvent(stream, before_sample, 0) != cudaSuccess) return HOLA_ERR_CUDA;
  ctx->hq_ready = side || inside ? 1 : 0;
  // (behind the GEMM kernel: the caller's inputs are settled; an event wait in between makes it an ordinary launch)
  s = run_accept_sample(ctx, a, logits, ldl, 1, row_partials(pl), stream, nullptr, 0, nullptr, true);
  ctx->hq_ready = 0;
  if (prof) { cudaEventRecord(ev[2], stream); ctx->prof_n++; }
  return s;
}

// hola_verify_host while the target entropy gates.  Of the draft tensor the step then reads k single probabilities
// per sequence (q_j(x_j), gathered here on the host; the greedy fallback does not look at them) and at most ONE row per
// sequence: row accept_len, and none when every draft token was kept or the fallback is greedy.  Rows 0 .. ahead-1 of
// every sequence (as many as the bus carries while the GEMM runs, at least one) are sent ahead on the context's own stream;
// after the accept test the accept lengths come back and only the rows still missing follow, or the accept/sample kernel
// reads those in place.  Same arithmetic and so the same results as the whole-tensor copy, with one exception: a launch that
// reads rows in place keeps clusters where the others take one CTA (sample_solo), so that the chunks' masses are summed in
// another order, in fp64; a token differs only where u R falls within that rounding (some 1e-16) of a boundary.
constexpr double kHostBusBytesPerSecond = 50e9;          // what a pinned host-to-device copy reaches here

// Draft rows per sequence that can cross the bus while the GEMM of this call runs.
int rows_under_gemm(hola_ctx* ctx, const hola_verify_args* a) {
  const Plan& pl = plan_for(ctx, a->B * (a->k + 1), a->w_dtype);
  const double group = static_cast<double>(a->B) * a->V * (a->q_dtype == HOLA_Q_BF16 ? 2 : 4);
  const double n = pl.est_seconds * kHostBusBytesPerSecond / group;
  return n > 1e6 ? 1000000 : static_cast<int>(n);
}

// Points a call's outputs into the pinned host block, where the accept/sample kernel can write them (a few KB, posted
// writes: some 8 us less than a copy back behind the kernel).  The status word stays on the device, where kernels OR into
// it; its bits and each sequence's flags come back as plain words (collect_flags).
bool outputs_to_host(hola_ctx* ctx, hola_verify_args* d, const OutBlock& ob) {
  if (!ctx->h_out_dev) return false;
  d->accept_len = reinterpret_cast<int*>(ctx->h_out_dev + ob.accept);
  d->next_tok = reinterpret_cast<int*>(ctx->h_out_dev + ob.next);
  d->entropy = reinterpret_cast<float*>(ctx->h_out_dev + ob.entropy);
  d->logZ = reinterpret_cast<float*>(ctx->h_out_dev + ob.logZ);
  if (d->draft_entropy) d->draft_entropy = reinterpret_cast<float*>(ctx->h_out_dev + ob.dent);
  ctx->flags_out = reinterpret_cast<unsigned*>(ctx->h_out_dev + ob.flags);
  return true;
}
void collect_flags(hola_ctx* ctx, const OutBlock& ob, int B) {
  const unsigned* f = reinterpret_cast<const unsigned*>(ctx->h_out + ob.flags);
  unsigned all = 0;
  for (int b = 0; b < B; ++b) all |= f[b];
  memcpy(ctx->h_out + ob.status, &all, 4);
}

hola_status verify_host_lazy(hola_ctx* ctx, const hola_verify_args* a, cudaStream_t stream, int ahead) {
  const int B = a->B, k = a->k, V = a->V;
  const size_t rows = static_cast<size_t>(B) * (k + 1);
  const size_t q_elem = a->q_dtype == HOLA_Q_BF16 ? 2 : 4;
  const size_t row_bytes = static_cast<size_t>(V) * q_elem;
  const bool sample = a->fallback != HOLA_FALLBACK_GREEDY;
  cudaError_t e = cudaSuccess;
  unsigned long long up = 0, down = 0;
  auto h2d = [&](void* dst, const void* src, size_t bytes, cudaStream_t st) {
    if (e == cudaSuccess && bytes) e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st);
    up += bytes;
  };
  auto d2h = [&](void* dst, const void* src, size_t bytes) {
    if (e == cudaSuccess && bytes) e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, stream);
    down += bytes;
  };
  // The hidden rows first and with the bus to themselves: the GEMM waits for them, while the draft rows have until its end.
  // The host gathers the k probabilities per sequence (a cache miss each) while they travel.
  h2d(ctx->st_hidden, a->hidden, rows * a->H * 2, stream);
  for (int b = 0; b < B; ++b)
    for (int j = 0; j < k; ++j) {
      const int x = a->draft_tok[b * k + j];
      float qx = 0.f;
      if (x >= 0 && x < V) {
        const size_t qi = (static_cast<size_t>(b) * k + j) * V + x;
        if (a->q_dtype == HOLA_Q_BF16) {
          const uint32_t bits = static_cast<uint32_t>(static_cast<const uint16_t*>(a->draft_q)[qi]) << 16;
          memcpy(&qx, &bits, 4);
        } else {
          qx = static_cast<const float*>(a->draft_q)[qi];
        }
      }
      ctx->h_qtok[b * k + j] = qx;
    }
  // tokens, uniforms and the gathered probabilities: into the pinned mirror, then one copy of the span in use.  Only the
  // accept/sample part reads them: they travel with the draft rows, out of the GEMM's way.
  memcpy(ctx->h_small, a->draft_tok, static_cast<size_t>(B) * k * 4);
  memcpy(ctx->h_small + ctx->small_u_off, a->uniforms, rows * 4);
  if (e == cudaSuccess) e = cudaEventRecord(ctx->fork_point, stream);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(ctx->copy_stream, ctx->fork_point, 0);
  h2d(ctx->st_tok, ctx->h_small, ctx->small_qtok_off + static_cast<size_t>(B) * k * 4, ctx->copy_stream);
  const OutBlock ob = out_block(B, k);
  const size_t seq_pitch = static_cast<size_t>(k) * row_bytes;   // from row (b, 0) to row (b + 1, 0)
  ahead = ahead < 1 ? 1 : (ahead > k ? k : ahead);
  const size_t ahead_bytes = static_cast<size_t>(ahead) * row_bytes;     // rows 0 .. ahead-1 of a sequence are adjacent
  if (sample) {
    if (seq_pitch < (1ull << 31)) {
      if (e == cudaSuccess)
        e = cudaMemcpy2DAsync(ctx->st_q, seq_pitch, a->draft_q, seq_pitch, ahead_bytes, static_cast<size_t>(B),
                              cudaMemcpyHostToDevice, ctx->copy_stream);
      up += static_cast<size_t>(B) * ahead_bytes;
    } else {
      for (int b = 0; b < B; ++b)
        h2d(static_cast<char*>(ctx->st_q) + b * seq_pitch, static_cast<const char*>(a->draft_q) + b * seq_pitch,
            ahead_bytes, ctx->copy_stream);
    }
  }
  if (e == cudaSuccess) e = cudaEventRecord(ctx->copy_done, ctx->copy_stream);
  if (e != cudaSuccess) { set_error(ctx, "host-to-device copy", e); return HOLA_ERR_CUDA; }
  hola_verify_args d = *a;
  d.hidden = ctx->st_hidden; d.draft_tok = ctx->st_tok; d.draft_q = ctx->st_q; d.uniforms = ctx->st_u;
  d.accept_len = reinterpret_cast<int*>(ctx->st_out + ob.accept);
  d.next_tok = reinterpret_cast<int*>(ctx->st_out + ob.next);
  d.entropy = reinterpret_cast<float*>(ctx->st_out + ob.entropy);
  d.logZ = reinterpret_cast<float*>(ctx->st_out + ob.logZ);
  d.logits_out = nullptr; d.status_word = reinterpret_cast<uint32_t*>(ctx->st_out); d.draft_entropy = nullptr;
  d.flags = HOLA_ARG_CLEAR_STATUS;
  hola_status s;
  const Plan& pl = plan_for(ctx, B * (k + 1), a->w_dtype);
  float* logits = logits_buffer(ctx, a);
  if ((s = run_lm_head(ctx, &d, logits, ctx->ldl, pl, stream)) != HOLA_OK) return s;
  // Where the caller's draft tensor is pinned host memory that the device can address, the rows still missing after the
  // accept test are not copied at all: the accept/sample kernel reads row accept_len of a sequence in place, over the
  // bus, when that row is not among the ones sent ahead.  One launch, no read-back in the middle of the call.
  const void* q_far = nullptr;
  if (sample && ctx->host_in_place) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, a->draft_q) == cudaSuccess && at.type == cudaMemoryTypeHost && at.devicePointer)
      q_far = at.devicePointer;
    else
      cudaGetLastError();                                // (an unregistered pointer is not an error of this call)
  }
  bool direct = false;
  if (!sample || q_far) {
    // one accept/sample launch: it writes the outputs into the pinned block itself
    if (e == cudaSuccess) e = cudaStreamWaitEvent(stream, ctx->copy_done, 0);
    if (e != cudaSuccess) { set_error(ctx, "wait for the inputs sent ahead", e); return HOLA_ERR_CUDA; }
    direct = outputs_to_host(ctx, &d, ob);
    s = run_accept_sample(ctx, &d, logits, ctx->ldl, 1, row_partials(pl), stream, ctx->st_qtok, 0, nullptr, false, q_far, ahead);
    ctx->flags_out = nullptr;
    if (s != HOLA_OK) return s;
  } else {
    if (e == cudaSuccess) e = cudaStreamWaitEvent(stream, ctx->copy_done, 0);
    if (e != cudaSuccess) { set_error(ctx, "host-to-device copy of draft rows", e); return HOLA_ERR_CUDA; }
    if ((s = run_accept_sample(ctx, &d, ctx->logits, ctx->ldl, 1, row_partials(pl), stream, ctx->st_qtok, 1)) != HOLA_OK) return s;
    d2h(ctx->h_accept, d.accept_len, static_cast<size_t>(B) * 4);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) { set_error(ctx, "accept lengths to host", e); return HOLA_ERR_CUDA; }
    for (int b = 0; b < B; ++b) {
      const int n = ctx->h_accept[b];
      if (n >= ahead && n < k) {
        const size_t off = (static_cast<size_t>(b) * k + n) * row_bytes;
        h2d(static_cast<char*>(ctx->st_q) + off, static_cast<const char*>(a->draft_q) + off, row_bytes, stream);
      }
    }
    if (e != cudaSuccess) { set_error(ctx, "host-to-device copy of draft rows", e); return HOLA_ERR_CUDA; }
    // statistics and accept lengths are in place: this launch repeats the (cheap) accept test and draws the token
    if ((s = run_accept_sample(ctx, &d, ctx->logits, ctx->ldl, 0, 0, stream, ctx->st_qtok, 0)) != HOLA_OK) return s;
  }
  if (direct) down += ob.dent;
  else d2h(ctx->h_out, ctx->st_out, ob.dent);            // every output in one copy
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  if (e != cudaSuccess) { set_error(ctx, "outputs to host", e); return HOLA_ERR_CUDA; }
  if (direct) collect_flags(ctx, ob, B);
  memcpy(a->accept_len, ctx->h_out + ob.accept, static_cast<size_t>(B) * 4);
  memcpy(a->next_tok, ctx->h_out + ob.next, static_cast<size_t>(B) * 4);
  memcpy(a->entropy, ctx->h_out + ob.entropy, rows * 4);
  memcpy(a->logZ, ctx->h_out + ob.logZ, rows * 4);
  if (a->status_word) memcpy(a->status_word, ctx->h_out + ob.status, 4);
  if (q_far) {                                           // rows the kernel read over the bus count as bytes sent
    for (int b = 0; b < B; ++b) {
      const int n = a->accept_len[b];
      if (n >= ahead && n < k) up += row_bytes;
    }
  }
  ctx->last_h2d = up; ctx->last_d2h = down;
  return HOLA_OK;
}

}  // namespace

extern "C" {

hola_status hola_verify(hola_ctx* ctx, const hola_verify_args* a, void* cuda_stream) {
  hola_status s = check_common(ctx, a);
  if (s != HOLA_OK) return s;
  if (a->B == 0) return empty_batch(ctx, a, cuda_stream);
  if ((s = check_lm_head_args(ctx, a)) != HOLA_OK) return s;
  if ((s = check_sample_args(a)) != HOLA_OK) return s;
  DeviceGuard guard(ctx->device);
  return verify_device(ctx, a, static_cast<cudaStream_t>(cuda_stream), nullptr);
}

hola_status hola_profile_begin(hola_ctx* ctx, int max_calls) {
  if (!ctx || max_calls <= 0 || max_calls > 4096) return HOLA_ERR_INVALID_ARG;
  DeviceGuard guard(ctx->device);
  if (ctx->prof_cap < max_calls) {
    cudaEvent_t* ev = static_cast<cudaEvent_t*>(calloc(static_cast<size_t>(3) * max_calls, sizeof(cudaEvent_t)));
    if (!ev) return HOLA_ERR_WORKSPACE;
    for (int i = 0; i < 3 * max_calls; ++i) {
      const cudaError_t e = cudaEventCreate(&ev[i]);
      if (e != cudaSuccess) { set_error(ctx, "cudaEventCreate", e); free(ev); return HOLA_ERR_CUDA; }
    }
    for (int i = 0; i < 3 * ctx->prof_cap; ++i) cudaEventDestroy(ctx->prof_ev[i]);
    free(ctx->prof_ev);
    ctx->prof_ev = ev;
    ctx->prof_cap = max_calls;
  }
  ctx->prof_n = 0;
  ctx->prof_on = 1;
  return HOLA_OK;
}

hola_status hola_profile_end(hola_ctx* ctx, void* cuda_stream, double* lm_head_ms, double* accept_sample_ms,
                             int* calls) {
  if (!ctx || !lm_head_ms || !accept_sample_ms || !calls) return HOLA_ERR_INVALID_ARG;
  DeviceGuard guard(ctx->device);
  ctx->prof_on = 0;
  cudaError_t e = cudaStreamSynchronize(static_cast<cudaStream_t>(cuda_stream));
  if (e != cudaSuccess) { set_error(ctx, "cudaStreamSynchronize", e); return HOLA_ERR_CUDA; }
  double a = 0.0, b = 0.0;
  for (int i = 0; i < ctx->prof_n; ++i) {
    float ms1 = 0.f, ms2 = 0.f;
    e = cudaEventElapsedTime(&ms1, ctx->prof_ev[3 * i], ctx->prof_ev[3 * i + 1]);
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms2, ctx->prof_ev[3 * i + 1], ctx->prof_ev[3 * i + 2]);
    if (e != cudaSuccess) { set_error(ctx, "cudaEventElapsedTime", e); return HOLA_ERR_CUDA; }
    a += ms1; b += ms2;
  }
  *lm_head_ms = a; *accept_sample_ms = b; *calls = ctx->prof_n;
  return HOLA_OK;
}

hola_status hola_verify_host(hola_ctx* ctx, const hola_verify_args* a, void* cuda_stream) {
  hola_status s = check_common(ctx, a);
  if (s != HOLA_OK) return s;
  if (a->B == 0) {                                       // (the status word is the caller's host memory here)
    if ((a->flags & HOLA_ARG_CLEAR_STATUS) && a->status_word) *a->status_word = 0u;
    return HOLA_OK;
  }
  if (!a->hidden) return HOLA_ERR_INVALID_ARG;
  // (what is refused is refused before any copy is queued: the caller's buffers need not outlive the call)
  hola_verify_args staged = *a;
  staged.hidden = ctx->st_hidden;
  if ((s = check_lm_head_args(ctx, &staged)) != HOLA_OK) return s;
  if ((s = check_sample_args(a)) != HOLA_OK) return s;
  DeviceGuard guard(ctx->device);
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  const size_t rows = static_cast<size_t>(a->B) * (a->k + 1);
  const size_t q_elem = a->q_dtype == HOLA_Q_BF16 ? 2 : 4;
  if (ctx->host_lazy_q && a->k > 0 && a->gate_source == HOLA_GATE_TARGET_ENTROPY) {
    // when the whole draft tensor crosses the bus under the GEMM anyway, the plain copy below has one launch and
    // one synchronisation fewer
    const int ahead = rows_under_gemm(ctx, a);
    if (ctx->host_lazy_q > 0 || ahead < a->k) return verify_host_lazy(ctx, a, stream, ahead);
  }
  cudaError_t e = cudaSuccess;
  unsigned long long up = 0, down = 0;
  auto h2d = [&](void* dst, const void* src, size_t bytes) {
    if (e == cudaSuccess && bytes) e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, stream);
    up += bytes;
  };
  auto d2h = [&](void* dst, const void* src, size_t bytes) {
    if (e == cudaSuccess && bytes) e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, stream);
    down += bytes;
  };
  // The hidden rows go first, on the caller's stream: the GEMM waits for them.  The draft tensor, by far the largest input,
  // and the small ones are read by the accept/sample part only: they travel on the context's own stream while the GEMM runs.
  // (Only calls of this entry point use the staging, and they synchronise before they return: it is free.)
  h2d(ctx->st_hidden, a->hidden, rows * a->H * 2);
  memcpy(ctx->h_small, a->draft_tok, static_cast<size_t>(a->B) * a->k * 4);
  memcpy(ctx->h_small + ctx->small_u_off, a->uniforms, rows * 4);
  const size_t q_bytes = static_cast<size_t>(a->B) * a->k * a->V * q_elem;
  const bool overlap = q_bytes && ctx->host_overlap;
  const size_t small_bytes = ctx->small_u_off + rows * 4;
  if (overlap) {
    // Behind the inputs that the GEMM waits for, unless the draft entropy gates: its pass over the whole tensor then takes
    // longer than the GEMM (16 sequences, V = 32000: 153 us with the tensor on the bus from the start, 166 behind).
    if (a->gate_source == HOLA_GATE_TARGET_ENTROPY) {
      if (e == cudaSuccess) e = cudaEventRecord(ctx->fork_point, stream);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(ctx->copy_stream, ctx->fork_point, 0);
    }
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(ctx->st_tok, ctx->h_small, small_bytes, cudaMemcpyHostToDevice, ctx->copy_stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(ctx->st_q, a->draft_q, q_bytes, cudaMemcpyHostToDevice, ctx->copy_stream);
    if (e == cudaSuccess) e = cudaEventRecord(ctx->copy_done, ctx->copy_stream);
    up += small_bytes + q_bytes;
  } else {
    h2d(ctx->st_tok, ctx->h_small, small_bytes);
    h2d(ctx->st_q, a->draft_q, q_bytes);
  }
  const OutBlock ob = out_block(a->B, a->k);
  if (e != cudaSuccess) { set_error(ctx, "host-to-device copy", e); return HOLA_ERR_CUDA; }
  hola_verify_args d = *a;
  d.hidden = ctx->st_hidden; d.draft_tok = ctx->st_tok; d.draft_q = ctx->st_q; d.uniforms = ctx->st_u;
  d.accept_len = reinterpret_cast<int*>(ctx->st_out + ob.accept);
  d.next_tok = reinterpret_cast<int*>(ctx->st_out + ob.next);
  d.entropy = reinterpret_cast<float*>(ctx->st_out + ob.entropy);
  d.logZ = reinterpret_cast<float*>(ctx->st_out + ob.logZ);
  d.logits_out = nullptr; d.status_word = reinterpret_cast<uint32_t*>(ctx->st_out);
  d.flags = HOLA_ARG_CLEAR_STATUS;
  const bool want_dent = a->draft_entropy && a->gate_source == HOLA_GATE_DRAFT_ENTROPY;
  d.draft_entropy = a->draft_entropy ? reinterpret_cast<float*>(ctx->st_out + ob.dent) : nullptr;
  const bool direct = outputs_to_host(ctx, &d, ob);
  s = verify_device(ctx, &d, stream, overlap ? ctx->copy_done : nullptr);
  ctx->flags_out = nullptr;
  if (s != HOLA_OK) return s;
  if (direct) down += want_dent ? ob.flags : ob.dent;
  else d2h(ctx->h_out, ctx->st_out, want_dent ? ob.flags : ob.dent); // every output in one copy
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  if (e == cudaSuccess && direct) collect_flags(ctx, ob, a->B);
  if (e != cudaSuccess) { set_error(ctx, "device-to-host copy", e); return HOLA_ERR_CUDA; }
  memcpy(a->accept_len, ctx->h_out + ob.accept, static_cast<size_t>(a->B) * 4);
  memcpy(a->next_tok, ctx->h_out + ob.next, static_cast<size_t>(a->B) * 4);
  memcpy(a->entropy, ctx->h_out + ob.entropy, rows * 4);
  memcpy(a->logZ, ctx->h_out + ob.logZ, rows * 4);
  if (a->status_word) memcpy(a->status_word, ctx->h_out + ob.status, 4);
  if (want_dent) memcpy(a->draft_entropy, ctx->h_out + ob.dent, static_cast<size_t>(a->B) * a->k * 4);
  ctx->last_h2d = up; ctx->last_d2h = down;
  return HOLA_OK;
}

// ---- vocabulary-parallel form: three calls per step with two small all-gathers between them (made by the caller)
size_t hola_shard_record_bytes(int B, int k) {
  if (B <= 0 || k < 0) return 0;
  const size_t rows = static_cast<size_t>(B) * (k + 1);
  return rows * 16 + align_up(static_cast<size_t>(B) * k * 4, 16);
}

static hola_status check_shard(const hola_ctx* ctx, const hola_verify_args* a, const hola_shard_args* sh) {
  if (!sh || sh->world < 1 || sh->rank < 0 || sh->rank >= sh->world) return HOLA_ERR_INVALID_ARG;
  if (sh->v_offset < 0 || sh->V_global < sh->v_offset + a->V) return HOLA_ERR_INVALID_ARG;
  if (a->gate_source != HOLA_GATE_TARGET_ENTROPY) return HOLA_ERR_INVALID_ARG;   // H(q_j) would need q of all shards
  (void)ctx;
  return HOLA_OK;
}

static ShardLaunch shard_launch(const hola_verify_args* a, const hola_shard_args* sh) {
  ShardLaunch l;
  l.world = sh->world; l.rank = sh->rank; l.v_offset = sh->v_offset; l.V_global = sh->V_global;
  l.stats_all = static_cast<const float4*>(sh->records);
  l.rec_floats = static_cast<int>(hola_shard_record_bytes(a->B, a->k) / 4);
  l.mass_out = sh->mass_out; l.mass_all = sh->masses;
  return l;
}

hola_status hola_shard_lm_head(hola_ctx* ctx, const hola_verify_args* a, const hola_shard_args* sh, void* cuda_stream) {
  hola_status s = check_common(ctx, a);
  if (s != HOLA_OK) return s;
  if (a->B == 0) return empty_batch(ctx, a, cuda_stream);
  if ((s = check_lm_head_args(ctx, a)) != HOLA_OK) return s;
  if ((s = check_shard(ctx, a, sh)) != HOLA_OK) return s;
  if (!sh->record_out || !aligned16(sh->record_out) || (a->k > 0 && !a->draft_tok)) return HOLA_ERR_INVALID_ARG;
  DeviceGuard guard(ctx->device);
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  const int M = a->B * (a->k + 1);
  const Plan& pl = plan_for(ctx, M, a->w_dtype);
  float* logits = a->logits_out ? a->logits_out : ctx->logits;
  const int ldl = a->logits_out ? a->V : ctx->ldl;
  if ((s = run_lm_head(ctx, a, logits, ldl, pl, stream, false, false, false, true)) != HOLA_OK) return s;
  float4* stats_out = static_cast<float4*>(sh->record_out);
  float* lx_out = reinterpret_cast<float*>(stats_out + M);
  const int blocks = (M + 7) / 8 + (a->B * a->k + 255) / 256;
  shard_record_kernel<<<blocks, 256, 0, stream>>>(ctx->partials, row_partials(pl), ctx->part_stride, M, sh->v_offset, a->V, logits,
                                                  ldl, a->draft_tok, a->B, a->k, stats_out, lx_out);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error(ctx, "launch shard_record_kernel", e); return HOLA_ERR_CUDA; }
  return HOLA_OK;
}

static hola_status shard_phase(hola_ctx* ctx, const hola_verify_args* a, const hola_shard_args* sh, void* cuda_stream,
                               int phase) {
  hola_status s = check_common(ctx, a);
  if (s != HOLA_OK) return s;
  if (a->B == 0) return HOLA_OK;
  if ((s = check_sample_args(a)) != HOLA_OK) return s;
  if ((s = check_shard(ctx, a, sh)) != HOLA_OK) return s;
  if (!sh->records || !aligned16(sh->records) || (a->k > 0 && !sh->q_tok)) return HOLA_ERR_INVALID_ARG;
  if (phase == 3 && !sh->mass_out) return HOLA_ERR_INVALID_ARG;
  if (phase == 4 && (!sh->masses || a->fallback == HOLA_FALLBACK_GREEDY)) return HOLA_ERR_INVALID_ARG;
  DeviceGuard guard(ctx->device);
  const float* logits = a->logits_out ? a->logits_out : ctx->logits;
  const int ldl = a->logits_out ? a->V : ctx->ldl;
  const ShardLaunch l = shard_launch(a, sh);
  return run_accept_sample(ctx, a, logits, ldl, phase == 3 ? 1 : 0, 0, static_cast<cudaStream_t>(cuda_stream),
                           sh->q_tok, phase, &l);
}

hola_status hola_shard_accept(hola_ctx* ctx, const hola_verify_args* a, const hola_shard_args* sh, void* cuda_stream) {
  return shard_phase(ctx, a, sh, cuda_stream, 3);
}

hola_status hola_shard_sample(hola_ctx* ctx, const hola_verify_args* a, const hola_shard_args* sh, void* cuda_stream) {
  return shard_phase(ctx, a, sh, cuda_stream, 4);
}

hola_status hola_host_traffic(const hola_ctx* ctx, unsigned long long* h2d_bytes, unsigned long long* d2h_bytes) {
  if (!ctx || !h2d_bytes || !d2h_bytes) return HOLA_ERR_INVALID_ARG;
  *h2d_bytes = ctx->last_h2d; *d2h_bytes = ctx->last_d2h;
  return HOLA_OK;
}

static hola_status launch_quantiser(const void* W, int V, int H, const QuantOut& o, void* cuda_stream,
                                    const GroupCodes* codes = nullptr) {
  const bool vec = H % 8 == 0 && aligned16(W) && aligned16(o.w16) && aligned16(o.w8) && aligned16(o.w4);
  const unsigned grid = static_cast<unsigned>((V + 7) / 8);
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  const uint16_t* src = static_cast<const uint16_t*>(W);
  if (codes && vec) quantize_rows_kernel<true, GroupCodes><<<grid, 256, 0, stream>>>(src, V, H, o, *codes);
  else if (codes) quantize_rows_kernel<false, GroupCodes><<<grid, 256, 0, stream>>>(src, V, H, o, *codes);
  else if (vec) quantize_rows_kernel<true><<<grid, 256, 0, stream>>>(src, V, H, o, NoCodes{});
  else quantize_rows_kernel<false><<<grid, 256, 0, stream>>>(src, V, H, o, NoCodes{});
  return cudaGetLastError() == cudaSuccess ? HOLA_OK : HOLA_ERR_CUDA;
}

hola_status hola_quantize_w4(const void* W_bf16, int rows, int H, void* packed_out, uint8_t* shift_out, int shift_stride,
                             float* scale_out, void* cuda_stream) {
  if (!W_bf16 || !packed_out || !shift_out || !scale_out || rows <= 0 || H <= 0 || shift_stride < rows)
    return HOLA_ERR_INVALID_ARG;
  if (H % kSubBlock != 0) return HOLA_ERR_UNSUPPORTED_SHAPE;
  QuantOut o = {};
  o.width = 4; o.w4 = static_cast<uint8_t*>(packed_out); o.shift4 = shift_out; o.shift_stride = shift_stride; o.scale = scale_out;
  return launch_quantiser(W_bf16, rows, H, o, cuda_stream);
}

hola_status hola_quantize_w8(const void* W_bf16, int V, int H, void* q_out, float* scale_out, void* cuda_stream) {
  if (!W_bf16 || !q_out || !scale_out || V <= 0 || H <= 0) return HOLA_ERR_INVALID_ARG;
  QuantOut o = {};
  o.width = 8; o.w8 = static_cast<signed char*>(q_out); o.scale = scale_out;
  return launch_quantiser(W_bf16, V, H, o, cuda_stream);
}

static hola_status quantize_mixed(const void* W_bf16, int V, int H, const hola_wmix* out, float* scale_out, void* cuda_stream,
                                  const GroupCodes* codes) {
  if (!W_bf16 || !out || !scale_out || V <= 0 || H <= 0 || !out->group_width || !out->group_row) return HOLA_ERR_INVALID_ARG;
  if (H % kSubBlock != 0) return HOLA_ERR_UNSUPPORTED_SHAPE;
  if (out->rows4 < 0 || out->rows8 < 0 || out->rows16 < 0 ||
      static_cast<long long>(out->rows4) + out->rows8 + out->rows16 < V)
    return HOLA_ERR_INVALID_ARG;
  if ((out->rows4 > 0 && (!out->W4 || !out->shift4)) || (out->rows8 > 0 && !out->W8) || (out->rows16 > 0 && !out->W16))
    return HOLA_ERR_INVALID_ARG;
  QuantOut o = {};
  o.group_width = out->group_width; o.group_row = out->group_row;
  o.tables_width = const_cast<uint8_t*>(out->group_width); o.tables_row = const_cast<int*>(out->group_row);
  o.w16 = static_cast<uint16_t*>(const_cast<void*>(out->W16));
  o.w8 = static_cast<signed char*>(const_cast<void*>(out->W8));
  o.w4 = static_cast<uint8_t*>(const_cast<void*>(out->W4));
  o.shift4 = const_cast<uint8_t*>(out->shift4); o.shift_stride = out->rows4; o.scale = scale_out;
  return launch_quantiser(W_bf16, V, H, o, cuda_stream, codes);
}

hola_status hola_quantize_mixed(const void* W_bf16, int V, int H, const hola_wmix* out, float* scale_out, void* cuda_stream) {
  return quantize_mixed(W_bf16, V, H, out, scale_out, cuda_stream, nullptr);
}

hola_status hola_quantize_mixed_widths(const void* W_bf16, int V, int H, const uint8_t* widths, const hola_wmix* out,
                                       float* scale_out, void* cuda_stream) {
  if (!widths || !out || V <= 0) return HOLA_ERR_INVALID_ARG;
  const int groups = (V + kGroupRows - 1) / kGroupRows;
  if (groups > kMaxCodedGroups) return HOLA_ERR_UNSUPPORTED_SHAPE;
  GroupCodes codes;
  memset(&codes, 0xFF, sizeof codes);
  int rows[3] = {0, 0, 0}, count[3] = {0, 0, 0};
  for (int g = 0; g < groups; ++g) {
    if (widths[g] != 4 && widths[g] != 8 && widths[g] != 16) return HOLA_ERR_INVALID_ARG;
    const uint32_t code = widths[g] >> 3;                // 0, 1, 2
    if ((g & 15) == 0) codes.before[g >> 4] = static_cast<uint32_t>(count[0]) | static_cast<uint32_t>(count[1]) << 16;
    codes.w[g >> 4] ^= (3u ^ code) << (2 * (g & 15));
    ++count[code];
    rows[code] += g + 1 < groups ? kGroupRows : V - g * kGroupRows;
  }
  if (rows[0] != out->rows4 || rows[1] != out->rows8 || rows[2] != out->rows16) return HOLA_ERR_INVALID_ARG;
  return quantize_mixed(W_bf16, V, H, out, scale_out, cuda_stream, &codes);
}

}  // extern "C"

// ------------------------------------------------------------------------------------------------ no-allocation entry
// hola_lm_head_entropy_static: steps 1-2 for callers that must not allocate device memory.  The per-CTA softmax
// statistics, which hola_lm_head_entropy keeps in the context's cudaMalloc'ed workspace, live here in a fixed
// array inside the library image; logits, entropy and logZ go to the caller's buffers as usual.

namespace {

constexpr int kStaticMaxRows = 512;    // verify rows B(k+1) one call may have
constexpr int kStaticMaxCtas = 160;    // CTAs of the GEMM kernel that may leave statistics (one per SM; B200 has 148)
constexpr size_t kStaticStatusBytes = 256;
constexpr size_t kStaticScratchBytes =
    kStaticStatusBytes + static_cast<size_t>(kStaticMaxCtas) * kStaticMaxRows * sizeof(float4);   // 1 310 976 bytes

}  // namespace

// Every GPU that loads the library holds this array until the process exits.  In host code the name is only a
// handle for cudaGetSymbolAddress, never a device address.
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

namespace {

constexpr int kStaticMaxDevices = 64;
std::mutex g_static_mu;
hola_ctx g_static_ctx[kStaticMaxDevices];      // host-side descriptors only; they own no memory
bool g_static_ready[kStaticMaxDevices];

// Once per device, with that device current: where the array lives on this device, the tensor-map encoder of the
// driver, and the SM count.  Allocates nothing.
hola_status static_setup(int dev, hola_ctx* out) {
  std::lock_guard<std::mutex> lock(g_static_mu);
  hola_ctx* c = &g_static_ctx[dev];
  if (!g_static_ready[dev]) {
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess || prop.major != 10) return HOLA_ERR_NO_DEVICE;
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || !fn ||
        qres != cudaDriverEntryPointSuccess)
      return HOLA_ERR_NO_DEVICE;
    void* base = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&base, g_static_scratch);
    if (e != cudaSuccess || !base) return HOLA_ERR_CUDA;
    if (configure_kernels() != cudaSuccess) return HOLA_ERR_CUDA;
    memset(c, 0, sizeof *c);
    c->device = dev;
    c->num_sms = prop.multiProcessorCount;
    c->encode = reinterpret_cast<EncodeTiledFn>(fn);
    c->status = reinterpret_cast<unsigned*>(base);
    c->partials = reinterpret_cast<float4*>(static_cast<unsigned char*>(base) + kStaticStatusBytes);
    c->part_stride = kStaticMaxCtas;
    c->max_rows = kStaticMaxRows;
    g_static_ready[dev] = true;
  }
  *out = *c;
  return HOLA_OK;
}

}  // namespace

extern "C" hola_status hola_lm_head_entropy_static(const hola_verify_args* a, void* cuda_stream) {
  if (!a) return HOLA_ERR_INVALID_ARG;
  if (a->B < 0 || a->k < 0 || a->H <= 0 || a->V <= 0) return HOLA_ERR_INVALID_ARG;
  if (a->B == 0) return empty_batch(a, cuda_stream);
  if (!a->hidden || !a->W_lm || !a->logits_out || !a->entropy || !a->logZ) return HOLA_ERR_INVALID_ARG;
  if (!aligned16(a->hidden) || !aligned16(a->W_lm)) return HOLA_ERR_INVALID_ARG;
  if (a->H % 8 != 0) return HOLA_ERR_UNSUPPORTED_SHAPE;
  const long long rows = static_cast<long long>(a->B) * (a->k + 1);
  if (rows > kStaticMaxRows) return HOLA_ERR_STATIC_LIMIT;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kStaticMaxDevices) return HOLA_ERR_NO_DEVICE;
  hola_ctx local;                      // a per-call copy: concurrent host threads do not share host state
  hola_status s = static_setup(dev, &local);
  if (s != HOLA_OK) return s;
  local.H = a->H; local.V = a->V; local.maxB = a->B; local.maxK = a->k;
  const int M = static_cast<int>(rows);
  if (a->w_dtype != HOLA_W_BF16) return HOLA_ERR_INVALID_ARG;   // the 8-bit weight modes need a context's workspace
  const Plan pl = make_plan(&local, M, a->w_dtype);
  if (pl.grid > kStaticMaxCtas) return HOLA_ERR_STATIC_LIMIT;
  // a timed-out wait must be visible to the caller: the kernels report to the caller's status word when there is one
  // (run_lm_head picks it), else to the word inside the array, which nobody outside can read
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  // The array keeps whatever the last call left.  The statistics slots are fully overwritten for the rows of this
  // call before they are read; the internal status word is the one thing that must start at zero.
  if (cudaMemsetAsync(local.status, 0, sizeof(unsigned), stream) != cudaSuccess) return HOLA_ERR_CUDA;
  if ((s = run_lm_head(&local, a, a->logits_out, a->V, pl, stream)) != HOLA_OK) return s;
  return launch_finalize(&local, a, M, row_partials(pl), stream) == cudaSuccess ? HOLA_OK : HOLA_ERR_CUDA;
}
