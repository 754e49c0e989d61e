// Inference over all N neurons on the tensor pipe (dslide_predict_topk with dense = 1).
//
// The logits of a batch against every output neuron are one contraction, Z[B][N] = h[B][H] . W2[N][H]^T + b2
// (Section 3.6: "layer sparsity is 1"), so this path runs it on the fifth-generation tensor cores: tiles of W2
// arrive in shared memory by TMA (cp.async.bulk.tensor, 128-byte swizzle), the 128 samples' hidden activations of a
// block sit in tensor memory beside the accumulators, a single thread of one or two blocks issues tcgen05.mma (kind::tf32), and the
// read-back warps fetch the accumulators (tcgen05.ld) and keep, per sample, the candidates of the block's slice of
// neurons; four more warps take the largest row norm of W2 from the tiles while they are in shared memory.  W2 is
// streamed once per 128 samples (the groups of samples walk the same tiles together, so HBM sees it once per call).
//
// TF32 rounds both operands to 10 mantissa bits, far from the 1e-4 the scores must meet.  The tensor pass is
// therefore a FILTER, in two launches of the same kernel.  The first scores every TC_SUBSET-th tile of neurons and
// writes the scores (or the largest of neighbours) out; k_tc_tau takes, per sample, about the (k + TC_RANK_OVER)-th best of them as the
// sample's threshold -- about TC_TARGET times as many neurons reach it over all N.  The second launch scores all tiles and a
// thread appends the few scores of its sample that reach the threshold to the sample's candidate buffer.
// k_tc_refine recomputes the cap = 2k + TC_EXTRA or so best candidates exactly in fp32 and orders them (logit descending, id
// ascending).  The filter is exact when the k-th exact score clears every discarded neuron's approximate score by
// more than the approximation's error bound, 2^-9 |h| |w|_max (plus accumulation); a sample for which that cannot
// be shown (or whose buffers ran over) is listed, and k_scan_all scores all N neurons for the listed samples in fp32.
// Results are therefore those of the exact path.  The kernels of a call follow one another by programmatic dependent launch.
#include <cuda.h>

#include "common.cuh"
#include "waits.cuh"

namespace dslide {

constexpr int TC_M = 128;          // samples per block = lanes of the accumulator
constexpr int TC_N = 128;          // neurons per tile = columns of the accumulator
constexpr int TC_KB = 32;          // hidden units per 128-byte swizzled row
constexpr int TC_STAGES = 6;       // tiles of W2 in flight at most (as many as fit in shared memory)
constexpr int TC_NACC = 3;         // tensor memory: up to three accumulators of TC_N columns (two when H > TC_N), then the activations (H columns)
constexpr int TC_TMEM_COLS = 512;
constexpr int TC_SPLIT = 4;        // read-back warps per quarter of tensor memory (each takes 1 / TC_SPLIT of a tile's columns)
constexpr int TC_EPI = 128 * TC_SPLIT;                 // read-back threads
constexpr int TC_THREADS = 64 + TC_EPI;                // warp 0: TMA producer; warp 1: tensor memory + MMA issue; then the read-back warps (tc_threads: further ones)
constexpr int TC_NORM_WARPS = 4;   // that take the row norms.  One held a tile's stage for 2,050 cycles of 2,280 (128 units, two groups of samples); us for one,
                                   // two and four: 256 x 670,091 x 128 139, 134, 129; 512 x 600,011 x 32 to 96 no more than one; 100 x 100,003 x 512 95, 88, 83
constexpr int TC_EXTRA = 16;       // candidates kept beyond 2k (the wider the margin, the rarer the exact fall-back)
constexpr int TC_H_TMEM = 256;     // hidden layers up to this width sit in tensor memory beside two accumulators; wider ones are
                                   // streamed through shared memory with the tiles (WIDE)
constexpr int TC_H_SINGLE = 192;   // up to this width two tiles fit a block's shared memory
constexpr int TC_WIDE_STAGES = TC_STAGES;      // WIDE: pairs of slabs (32 units of the samples, 32 units of the neurons) in flight
constexpr int TC_RANK_MIN = 8, TC_RANK_OVER = 5, TC_RANK_CAP = 24;      // the threshold's rank in the subset: k + TC_RANK_OVER, within these
constexpr int TC_GBUF_MIN = 2;     // candidate slots per (buffer, sample) at least, in neighbouring neurons that the buffer takes of a tile (32, or 64 of
                                   // a wide pair's): many times the expected fill, but a trained model may favour neighbours together, and a buffer
                                   // that runs over sends the sample to the exact scan (512 x 100,003 neurons x 512 units all undecided: 3,300 us for 137)
constexpr int TC_TARGET = 64;      // candidates aimed at per sample: so many times that rank
constexpr int TC_SUBSET = 64;      // the threshold pass scores every TC_SUBSET-th tile
constexpr int TC_SUB_BYTES = TC_M * 128;               // one 32-unit slab of 128 rows
constexpr float TC_ERR = 2.2e-3f;  // |approximate - exact| <= TC_ERR * |h| * |w|: two operands cut to 10 mantissa bits, fp32 sums

constexpr int TC_BT = 8;           // tiles whose biases are in shared memory or on their way there
// Neurons of a tile: 256 where the activations do not stand beside the accumulators in tensor memory and two blocks share a tile
__host__ __device__ constexpr int tc_cols(bool wide, bool pair) { return wide && pair ? 2 * TC_N : TC_N; }

// Warps after the read-back's: one for the biases, those for the row norms, and, in pairs whose second block learns from the first of
// the rows that it sums, one for that
__host__ __device__ constexpr int tc_threads(bool wide, bool pair) { return TC_THREADS + 32 * (1 + (wide && pair ? 0 : TC_NORM_WARPS) + (pair && !wide ? 1 : 0)); }

struct TcParams {
  const RowHdr* hdr2;
  const float* h;                  // [>= B][H] hidden activations of the batch
  const float* W2;
  int2* cand;                      // [TC_SPLIT * slices][Bpad][gbuf] (score bits, id), cand_cnt of them valid, no order
  int* cand_cnt;                   // [TC_SPLIT * slices][Bpad]
  float* dump;                     // DUMP launch: [Bpad][dump_cols] scores of the subset's tiles
  const float* tau;                // filter launch: [Bpad] thresholds
  int* need_fix;                   // [B] set when a sample's buffer ran over
  int* n_fix;                      // cleared for k_tc_refine
  unsigned int* norm2max;          // filter launch: largest squared norm of a row of W2, as the bits of a non-negative float
  DevState* st;
  int B, Bpad, H, N, nslices, ntiles;          // ntiles: tiles this launch walks
  int tile_stride;                 // tile i of the launch is tile i * tile_stride of W2
  int stages;                      // tiles of W2 in flight, 1 .. TC_STAGES
  int dump_cols, dump_max;         // per sample: largest scores of dump_max neighbours each
  int gbuf;                        // slots per candidate buffer
};

__device__ __forceinline__ void tc_bar_init(uint64_t* bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tc_smem(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void tc_bar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc_smem(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void tc_bar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc_smem(bar)) : "memory");
}
// The address, in the cluster's shared memory, of a barrier of the block of rank `rank`; an arrival there.  Most arrivals and
// waits order what the block itself needs (default scope): the operands and accumulators are ordered by the copies' and the tensor
// unit's own completion and by tcgen05.fence.  With release and acquire at cluster scope every one of them cost about 1,000 cycles.
// The second block's ordinary loads of rows whose copies the first block counts are ordered by none of these: the first block's
// wait for the copies, the arrival that passes them on (tc_bar_pass_on) and the second block's wait are at cluster scope.
__device__ __forceinline__ uint32_t tc_at_rank(const void* p, uint32_t rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(tc_smem(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void tc_bar_arrive_at(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_bar_pass_on(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_cluster_sync() {
  __syncthreads();
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// Into this block's shared memory, counted by a barrier of either block of the pair
__device__ __forceinline__ void tc_tma_2d_pair(void* dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%2, %3}], [%4];"
               ::"r"(tc_smem(dst)), "l"(map), "r"(x), "r"(y), "r"(bar) : "memory");
}
__device__ __forceinline__ void tc_tma_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
               ::"r"(tc_smem(dst)), "l"(map), "r"(x), "r"(y), "r"(tc_smem(bar)) : "memory");
}
// Shared-memory operand descriptor: K-major tile of 128-byte rows, 128-byte swizzle, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);            // start address
  d |= (uint64_t)1 << 16;                              // leading-dimension offset: unused with swizzled K-major rows
  d |= (uint64_t)(1024 >> 4) << 32;                    // stride between groups of eight rows
  d |= (uint64_t)1 << 46;                              // descriptor version of this architecture
  d |= (uint64_t)2 << 61;                              // 128-byte swizzle
  return d;
}
// Instruction descriptor: fp32 accumulator, tf32 x tf32, both operands K-major, N x M tile.
__host__ __device__ constexpr uint32_t tc_idesc(int M, int N) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// D[tmem] (+)= A[tmem] . B[smem]^T: the first operand is read from tensor memory, so shared memory serves one operand only.
// A pair's instruction takes the accumulators and first operands of both blocks and half of the second operand from each.
template <bool PAIR>
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  if (PAIR) asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::2.kind::tf32 [%0], [%1], %2, %3, p;\n\t}"
                      ::"r"(d_tmem), "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
  else asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n\t}"
                      ::"r"(d_tmem), "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
// The same with both operands in shared memory (hidden layers too wide for tensor memory)
template <bool PAIR>
__device__ __forceinline__ void tc_mma_ss(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  if (PAIR) asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
                      ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
  else asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
                      ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tc_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, "
      "%19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
        "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
        "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
// Arrives on the barrier -- of the blocks of a pair that `ranks` names, both by default -- once the instructions issued before have completed
template <bool PAIR>
__device__ __forceinline__ void tc_commit(uint64_t* bar, int ranks = 3) {
  if (PAIR)
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(tc_smem(bar)), "h"((uint16_t)ranks) : "memory");
  else
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tc_smem(bar)) : "memory");
}
__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, "
      "%19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// (z0, z1) = (a0, a1) + the two floats of b
__device__ __forceinline__ void tc_add2(float& z0, float& z1, uint32_t a0, uint32_t a1, unsigned long long b) {
  asm("{\n\t.reg .b64 a;\n\tmov.b64 a, {%2, %3};\n\tadd.rn.f32x2 a, a, %4;\n\tmov.b64 {%0, %1}, a;\n\t}" : "=f"(z0), "=f"(z1) : "r"(a0), "r"(a1), "l"(b));
}
__device__ __forceinline__ float tc_max32(const float (&z)[32]) {
  float m[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    m[i] = fmaxf(z[8 * i], z[8 * i + 1]);
#pragma unroll
    for (int c = 2; c < 8; c += 2) m[i] = fmaxf(fmaxf(m[i], z[8 * i + c]), z[8 * i + c + 1]);
  }
  return fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
}
__device__ __forceinline__ bool tc_better(float za, int ia, float zb, int ib) { return za > zb || (za == zb && ia < ib); }

// Adds the squares of C of the eight 16-byte pieces of a 128-byte swizzled row, from piece c0 on
template <int C>
__device__ __forceinline__ void tc_squares(const unsigned char* row, int c0, int key, unsigned long long (&n)[2]) {
  ulonglong2 w[C];
#pragma unroll
  for (int c = 0; c < C; ++c) w[c] = *reinterpret_cast<const ulonglong2*>(row + (size_t)(((c0 + c) ^ key) * 16));
#pragma unroll
  for (int c = 0; c < C; ++c) {
    asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(n[0]) : "l"(w[c].x));
    asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(n[1]) : "l"(w[c].y));
  }
}
// One lane of a converged warp, the same at every call: the copies, multiplications and commits are its own, while the whole warp
// walks the tiles and waits, so that their operands are the warp's.  Issued by one lane of a diverged warp an instruction took 84 to 134
// cycles where the tensor pipe takes 64, which bounded the filter at every width (a tile of 256 units in pairs 2,970 cycles, so 2,080;
// 1,024 samples x 253,855 neurons x 200 units 246 us, so 218).
__device__ __forceinline__ bool tc_elect() {
  uint32_t one;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(one));
  return one != 0u;
}

// Grid: (slices of the neurons, groups of 128 samples).  Dynamic shared memory (1024-byte aligned):
// TC_STAGES tiles of W2 as [ceil(H/32)][128 rows][128 B], then
// the tiles' biases, the barriers.  (The samples' candidate buffers are in global memory.)
// Every width and every k takes this kernel; a scan on the ALUs (one bulk copy per row of W2, 8 to 32 samples against a
// staged row) took 11,700 us where the filter takes 389 us (H 200, N 253,855, 1,024 samples, k 5).
// A hidden width that is no multiple of 32 ends in a slab whose missing units the tensor copy fills with zeros.
// WIDE (H > TC_H_TMEM): the activations do not fit tensor memory, so a stage is one slab of the tile and the same 32
// units of the block's samples, both by tensor copies; the samples' slabs come from L2 once per tile, which doubles
// the copies of a tile but keeps the multiplications on the tensor pipe.
// PAIR: two multiprocessors (a cluster of two blocks) share a tile, half of its rows in the shared memory of each, and take
// 128 samples each; the first block issues instructions of 256 samples for both (use_pairs says when).  WIDE tiles are
// then 256 neurons, so that the samples' slabs serve twice as many.
// What a tile took besides the multiplications, 1,000 to 2,000 cycles: the issue of the multiplications (tc_elect), read-back warps that
// waited for one another, the row norms (TC_NORM_WARPS).  Now 2,080 cycles at 256 units in pairs, of which the multiplications are
// 2,050; 1,850 and 1,650 at 200 units in pairs; 1,740 and 1,060 at 128 units, where shared memory bounds it (the copies 64 KB,
// the multiplications 64, the norms 32 to 64 per tile, at 128 bytes per cycle).
// The rows' norms in pairs: the second block reads its half of a tile once the first block, which counts the copies, has passed
// that on; at cluster scope this takes 1,000 cycles, which a warp of its own spends (by the norm warps themselves 1,024 samples x
// 253,855 neurons x 200 units took 262 us where a warp of its own took 256).  That warp's pace is the least time of a tile, 1,500 cycles.  A slab has not that much time (512 samples x 100,003 neurons x 512 units 229 us):
// WIDE pairs take the norms from global memory, where L2 has the rows (135 us; at 200 units it would be 283): the read-back warps,
// before they wait for the tile's scores.
template <bool DUMP, bool WIDE, bool PAIR>      // DUMP: write every score out (threshold pass); else append the scores that reach the sample's threshold
__global__ void __launch_bounds__(tc_threads(WIDE, PAIR), 1)
k_dense_tc(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmH, const TcParams p) {
  extern __shared__ __align__(1024) unsigned char tc_smem_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(tc_smem_raw) + 1023) & ~(uintptr_t)1023);
  const int ksub = (p.H + TC_KB - 1) / TC_KB;
  const int kfull = p.H / TC_KB;
  const int klast = (p.H - (ksub - 1) * TC_KB + 7) >> 3;      // instructions (eight units each) of the last slab
  constexpr int NT = tc_cols(WIDE, PAIR);                      // neurons of a tile
  constexpr int ROWS = PAIR ? NT / 2 : NT;                     // of which this block holds so many rows
  constexpr uint32_t SLAB = ROWS * 128;                        // 32 units of them
  const uint32_t tile_bytes = WIDE ? SLAB + TC_SUB_BYTES : (uint32_t)ksub * SLAB;      // of a stage
  unsigned char* smB = sm;
  const int nst = p.stages;
  float* sb = reinterpret_cast<float*>(smB + (size_t)nst * tile_bytes);                         // [TC_BT][NT] biases of the tiles
  uint64_t* bars = reinterpret_cast<uint64_t*>(sb + TC_BT * NT);
  uint64_t* bar_a = bars;                      // activations are in tensor memory
  constexpr int NST = WIDE ? TC_WIDE_STAGES : TC_STAGES;
  uint64_t* bar_full = bars + 1;               // [NST] the stage has arrived
  uint64_t* bar_empty = bars + 1 + NST;        // [NST] the stage has been consumed
  uint64_t* bar_accfull = bars + 1 + 2 * NST;              // [TC_NACC] accumulator written
  uint64_t* bar_accempty = bars + 1 + 2 * NST + TC_NACC;   // [TC_NACC] accumulator read back
  uint64_t* bar_landed = bars + 1 + 2 * NST + 2 * TC_NACC; // [NST] second block of a pair: the stage has arrived (the pair's bytes are counted in the first)
  uint64_t* bar_drain = bars + 1 + 3 * NST + 2 * TC_NACC;  // after a wait has run out: the multiplications issued before have completed
  uint64_t* bar_bfull = bar_drain + 1;         // [TC_BT] the biases of a tile have arrived
  uint64_t* bar_bempty = bar_bfull + TC_BT;    // [TC_BT] and have been read
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_bempty + TC_BT);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  unsigned* best_slot = tmem_slot + 2;         // OWN_ROWS: the block's largest squared norm, as bits

  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const uint32_t rank = PAIR ? blockIdx.x & 1u : 0u;       // in the pair: the first block counts arrivals and issues the multiplications
  const int slice = PAIR ? blockIdx.x >> 1 : blockIdx.x, s0 = PAIR ? (2 * (int)blockIdx.y + (int)rank) * TC_M : (int)blockIdx.y * TC_M;
  // tiles of this slice: slice, slice + nslices, ... (both sample groups walk the same tiles at the same time: the
  // second read of a tile is served by L2)
  const int my_tiles = slice < p.ntiles ? (p.ntiles - slice + p.nslices - 1) / p.nslices : 0;
  // The filter launch also takes the largest squared row norm of W2 (the error bound needs it) from the tiles as
  // they pass through shared memory; up to four sample groups share a tile's rows (they all see the same tiles).
  const int nshare = (int)gridDim.y >= 4 ? 4 : ((int)gridDim.y >= 2 ? 2 : 1);
  constexpr bool OWN_ROWS = WIDE && PAIR;                          // norms by the read-back warps
  const bool norms = !DUMP && !OWN_ROWS && (int)blockIdx.y < nshare;
  const int nacc = WIDE ? (PAIR ? 2 : TC_NACC) : (p.H <= TC_N ? TC_NACC : 2);      // accumulators in use; the activations follow them
  const uint32_t acol = (uint32_t)(nacc * NT);

  if (tid == 0) {
    tc_bar_init(bar_a, PAIR ? 8 : 4);            // a warp each
    tc_bar_init(bar_drain, 1);
    for (int i = 0; i < NST; ++i) { tc_bar_init(bar_full + i, 1); tc_bar_init(bar_landed + i, 1); tc_bar_init(bar_empty + i, norms ? 1 + TC_NORM_WARPS : 1); }
    for (int i = 0; i < TC_NACC; ++i) { tc_bar_init(bar_accfull + i, 1); tc_bar_init(bar_accempty + i, (PAIR ? 2 : 1) * TC_EPI / 32); }
    for (int i = 0; i < TC_BT; ++i) { tc_bar_init(bar_bfull + i, 32); tc_bar_init(bar_bempty + i, TC_EPI / 32); }
    *abort_flag = 0;
    *best_slot = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {      // tensor memory: all of it (one block per SM)
    if (PAIR) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem(tmem_slot)), "r"(TC_TMEM_COLS) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem(tmem_slot)), "r"(TC_TMEM_COLS) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (PAIR) tc_cluster_sync();       // the other block's barriers are ready
  else __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = *tmem_slot;
  griddep_launch_dependents();       // the next kernel of the call may be placed as blocks of this one leave
  griddep_wait();                    // the filter launch reads the thresholds of the kernel before it

  // Copies, multiplications and commits stop where a wait has run out; the other roles run through to their ends.  Each lane of the
  // warps that issue them has a wait of its own.  All take part in the election whatever it has answered, the elected one issues by
  // its own answer, and then they agree whether to go on, while what has been issued is under way.  (us for a call of 256 samples x
  // 1,024 neurons x 1,024 units: 54.1 so, 54.8 with the vote before the election, 53.0 with none.)
  auto agreed = [](bool ok) { return __all_sync(0xffffffffu, ok) != 0; };
  int fills = 0;                     // stages that this block has asked for, or would have when a wait ran out
  if (warp == 0) {
    // ---------------- producer: one thread feeds the TMA ----------------
    int st = 0, stround = 0;
    bool on = true;
    for (int i = 0; on && i < my_tiles; ++i) {
      const int row0 = (slice + i * p.nslices) * p.tile_stride * NT + (int)rank * ROWS;
      if (WIDE) {
        for (int ks = 0; on && ks < ksub; ++ks, ++fills) {
          const bool ok = stround == 0 || tc_bar_wait<PAIR>(bar_empty + st, (stround - 1) & 1, abort_flag);
          unsigned char* to = smB + (size_t)st * tile_bytes;
          if (tc_elect() && ok) {
            if (PAIR) {
              if (rank == 0) tc_bar_expect(bar_full + st, 2u * tile_bytes);
              const uint32_t full = tc_at_rank(bar_full + st, 0u);
              tc_tma_2d_pair(to, &tmW, ks * TC_KB, row0, full);
              tc_tma_2d_pair(to + SLAB, &tmH, ks * TC_KB, s0, full);
            } else {
              tc_bar_expect(bar_full + st, tile_bytes);
              tc_tma_2d(to, &tmW, ks * TC_KB, row0, bar_full + st);
              tc_tma_2d(to + SLAB, &tmH, ks * TC_KB, s0, bar_full + st);
            }
          }
          on = agreed(ok);
          if (++st == nst) { st = 0; ++stround; }
        }
        continue;
      }
      const bool ok = stround == 0 || tc_bar_wait<PAIR>(bar_empty + st, (stround - 1) & 1, abort_flag);
      if (tc_elect() && ok) {
        if (rank == 0) tc_bar_expect(bar_full + st, (PAIR ? 2u : 1u) * tile_bytes);
        const uint32_t full = PAIR ? tc_at_rank(bar_full + st, 0u) : 0u;
        for (int ks = 0; ks < ksub; ++ks) {
          unsigned char* to = smB + (size_t)st * tile_bytes + (size_t)ks * SLAB;
          if (PAIR) tc_tma_2d_pair(to, &tmW, ks * TC_KB, row0, full);
          else tc_tma_2d(to, &tmW, ks * TC_KB, row0, bar_full + st);
        }
      }
      on = agreed(ok);
      ++fills;
      if (++st == nst) { st = 0; ++stround; }
    }
    // the last fill of every stage has been consumed: no copy and no arrival at this block's barriers is on its way any more
    for (int f = max(0, fills - nst); on && f < fills; ++f) on = tc_bar_wait_warp<PAIR>(bar_empty + f % nst, (f / nst) & 1, abort_flag);
  } else if (warp == 1) {
    // ---------------- MMA issue: one thread (of a pair's first block) ----------------
    if (rank == 0) {
      const uint32_t idesc = tc_idesc(PAIR ? 2 * TC_M : TC_M, NT);
      bool on = WIDE || tc_bar_wait_warp<PAIR>(bar_a, 0, abort_flag);
      const uint64_t b_base = tc_desc(tc_smem(smB));      // a descriptor's address field counts 16-byte units
      int st = 0, stround = 0, acc = 0, accround = 0;
      for (int i = 0; on && i < my_tiles; ++i) {
        bool ok = WIDE || tc_bar_wait<PAIR>(bar_full + st, stround & 1, abort_flag);
        ok = (accround == 0 || tc_bar_wait<PAIR>(bar_accempty + acc, (accround - 1) & 1, abort_flag)) && ok;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t d = tmem_base + (uint32_t)(acc * NT);
        if (WIDE) {
          for (int ks = 0; on && ks < ksub; ++ks) {
            ok = tc_bar_wait<PAIR>(bar_full + st, stround & 1, abort_flag) && ok;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (tc_elect() && ok) {
              const uint64_t b = b_base + (uint64_t)(((uint32_t)st * tile_bytes) >> 4);
              const uint64_t a = b + (uint64_t)(SLAB >> 4);
              const int kn = ks == ksub - 1 ? klast : TC_KB / 8;
              for (int kk = 0; kk < kn; ++kk)
                tc_mma_ss<PAIR>(d, a + (uint64_t)(kk * 2), b + (uint64_t)(kk * 2), idesc, (ks | kk) != 0 ? 1u : 0u);
              tc_commit<PAIR>(bar_empty + st);
            }
            on = agreed(ok);
            if (++st == nst) { st = 0; ++stround; }
          }
          if (!on) break;
          if (tc_elect()) tc_commit<PAIR>(bar_accfull + acc);
          __syncwarp();
          if (++acc == nacc) { acc = 0; ++accround; }
          continue;
        }
        if (tc_elect() && ok) {
          const uint64_t b_tile = b_base + (uint64_t)(((uint32_t)st * tile_bytes) >> 4);
          for (int ks = 0; ks < kfull; ++ks) {
            const uint32_t a = tmem_base + acol + (uint32_t)(ks * TC_KB);      // lanes = samples, columns = hidden units
            const uint64_t b = b_tile + (uint64_t)((ks * SLAB) >> 4);
#pragma unroll
            for (int kk = 0; kk < TC_KB / 8; ++kk)              // eight tf32 = 32 bytes per instruction
              tc_mma<PAIR>(d, a + (uint32_t)(kk * 8), b + (uint64_t)(kk * 2), idesc, (ks | kk) != 0 ? 1u : 0u);
          }
          if (kfull < ksub)                                     // a last slab of fewer units
            for (int kk = 0; kk < klast; ++kk)
              tc_mma<PAIR>(d, tmem_base + acol + (uint32_t)(kfull * TC_KB + kk * 8), b_tile + (uint64_t)((kfull * SLAB) >> 4) + (uint64_t)(kk * 2),
                     idesc, (kfull | kk) != 0 ? 1u : 0u);
          tc_commit<PAIR>(bar_empty + st);          // the tile's shared memory is free once these instructions have read it
          tc_commit<PAIR>(bar_accfull + acc);       // and the accumulator is complete
        }
        on = agreed(ok);
        if (++st == nst) { st = 0; ++stround; }
        if (++acc == nacc) { acc = 0; ++accround; }
      }
    }
  } else if (warp == TC_THREADS / 32) {
    // ---------------- biases: a tile's, TC_BT tiles ahead of the read-back (zero past the last neuron) ----------------
    bool on = true;
    for (int i = 0; on && i < my_tiles; ++i) {
      const int slot = i & (TC_BT - 1), round = i / TC_BT;
      if (round > 0 && !(on = tc_bar_wait<PAIR>(bar_bempty + slot, (round - 1) & 1, abort_flag))) break;
      const int j0 = (slice + i * p.nslices) * p.tile_stride * NT + lane;
#pragma unroll
      for (int c = 0; c < NT; c += 32) {
        const int j = j0 + c;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;"
                     ::"r"(tc_smem(sb + slot * NT + c + lane)), "l"(&p.hdr2[j < p.N ? j : 0].b), "r"(j < p.N ? 4 : 0) : "memory");
      }
      asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(tc_smem(bar_bfull + slot)) : "memory");
    }
    asm volatile("cp.async.wait_all;" ::: "memory");      // nothing is on its way into shared memory when the block ends
  } else if (!OWN_ROWS && warp > TC_THREADS / 32 && warp <= TC_THREADS / 32 + TC_NORM_WARPS) {
    // ---------------- row norms: the lanes of the warps share the block's rows, one or more rows to a lane or 2, 4 or 8 lanes to a
    // row (8 in pairs whose tiles are shared by four groups of samples).  Sums of squares do not care about the swizzle, but the lanes of a quarter-warp read different 16-byte pieces so
    // that all banks are busy ----------------
    if (norms) {
      constexpr int LANES = 32 * TC_NORM_WARPS, RMAX = ROWS / LANES > 1 ? ROWS / LANES : 1;
      constexpr int LPR_MAX = LANES / (ROWS / 4);      // lanes of a row at most
      static_assert(LPR_MAX <= 8 && (ROWS % LANES == 0 || LANES % ROWS == 0), "no more lanes to a row than it has pieces");
      const int nrows = ROWS / nshare;                 // rows of this block
      const int lpr = nrows < LANES ? LANES / nrows : 1, nrr = nrows < LANES ? 1 : nrows / LANES;
      const int idx = (warp - TC_THREADS / 32 - 1) * 32 + lane, cn = 8 / lpr, c0 = idx % lpr * cn;
      const int row0 = nrows * (int)blockIdx.y + idx / lpr;      // the lane's first row; the others LANES apart (multiples of eight)
      float best = 0.f;
      int st = 0, stround = 0;
      for (int i = 0; i < my_tiles; ++i) {
        unsigned long long n[RMAX][2];                 // sums of a row's squares, in pairs
#pragma unroll
        for (int rr = 0; rr < RMAX; ++rr) n[rr][0] = n[rr][1] = 0ull;
        for (int k0 = 0; k0 < ksub; k0 += WIDE ? 1 : ksub) {      // the slabs of a stage
          // the bytes of a pair are counted in its first block, which tells the second
          if (PAIR && rank == 1) tc_bar_wait<PAIR, true>(bar_landed + st, stround & 1, abort_flag);
          else tc_bar_wait<PAIR>(bar_full + st, stround & 1, abort_flag);
          const unsigned char* tile = smB + (size_t)st * tile_bytes + (size_t)row0 * 128;
#pragma unroll
          for (int rr = 0; rr < RMAX; ++rr)
            if (rr < nrr)
              for (int ks = 0; ks < (WIDE ? 1 : ksub); ++ks) {
                const unsigned char* rowp = tile + (size_t)ks * SLAB + (size_t)rr * LANES * 128;
                if (cn == 8) tc_squares<8>(rowp, c0, row0 & 7, n[rr]);
                else if (cn == 4) tc_squares<4>(rowp, c0, row0 & 7, n[rr]);
                else if (LPR_MAX < 8 || cn == 2) tc_squares<2>(rowp, c0, row0 & 7, n[rr]);
                else tc_squares<1>(rowp, c0, row0 & 7, n[rr]);
              }
          __syncwarp();
          if (lane == 0) tc_bar_arrive(bar_empty + st);
          if (++st == nst) { st = 0; ++stround; }
        }
#pragma unroll
        for (int rr = 0; rr < RMAX; ++rr) {
          float sq = (__uint_as_float((unsigned)n[rr][0]) + __uint_as_float((unsigned)(n[rr][0] >> 32))) +
                     (__uint_as_float((unsigned)n[rr][1]) + __uint_as_float((unsigned)(n[rr][1] >> 32)));
          if (lpr >= 2) sq += __shfl_xor_sync(0xffffffffu, sq, 1);
          if (lpr >= 4) sq += __shfl_xor_sync(0xffffffffu, sq, 2);
          if (LPR_MAX == 8 && lpr == 8) sq += __shfl_xor_sync(0xffffffffu, sq, 4);
          best = fmaxf(best, sq);
        }
      }
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, d));
      if (lane == 0) atomicMax(p.norm2max, __float_as_uint(best));
    }
  } else if (PAIR && !WIDE && warp == TC_THREADS / 32 + 1 + TC_NORM_WARPS) {
    // ---------------- first block of a pair: what has landed is passed on to the second block's row norms ----------------
    if (norms && rank == 0 && lane == 0) {
      int st = 0, stround = 0;
      for (int i = 0; i < my_tiles; ++i) {
        if (!tc_bar_wait<PAIR, true>(bar_full + st, stround & 1, abort_flag)) break;
        tc_bar_pass_on(tc_at_rank(bar_landed + st, 1u));
        if (++st == nst) { st = 0; ++stround; }
      }
    }
  } else {
    // ---------------- read-back: thread = (sample, share of a tile's columns) ----------------
    // Per 32 columns the bias is added; then, threshold pass: the scores are written out; filter pass: which of them
    // reach the sample's threshold (32 independent comparisons, a bit each), then the appends of those that do.
    const int q = warp & 3;                 // a warp reaches the 32 lanes of tensor memory of its number modulo four
    const int half = (warp - 2) >> 2;       // which share of a tile's columns
    const int row = 32 * q + lane;          // sample inside the block
    const int vslice = slice * TC_SPLIT + half;    // buffers are kept per (slice, share of the columns)
    int2* mybuf = p.cand + ((size_t)vslice * p.Bpad + s0 + row) * p.gbuf;
    const float tau = DUMP ? 0.f : (s0 + row < p.B ? p.tau[s0 + row] : INFINITY);      // rows past the batch keep nothing
    int cnt = 0;
    if (DUMP && slice == 0 && half == 0) {      // the threshold pass also clears what the filter pass accumulates into
      if (s0 + row < p.B) p.need_fix[s0 + row] = 0;
      if (tid == 64 && blockIdx.y == 0) { *p.norm2max = 0u; *p.n_fix = 0; }
    }
    if (!WIDE && half == 0) {
      // the block's activations -> tensor memory: lane = sample, column = hidden unit (samples past the batch: zeros)
      const float4* hrow = reinterpret_cast<const float4*>(p.h + (size_t)(s0 + row) * p.H);
      const bool live = s0 + row < p.B;
      for (int c0 = 0; c0 < p.H; c0 += 32) {
        uint32_t r[32];
#pragma unroll
        for (int c4 = 0; c4 < 8; ++c4) {
          const float4 v = live && c0 + 4 * c4 < p.H ? hrow[(c0 >> 2) + c4] : make_float4(0.f, 0.f, 0.f, 0.f);
          r[4 * c4] = __float_as_uint(v.x); r[4 * c4 + 1] = __float_as_uint(v.y);
          r[4 * c4 + 2] = __float_as_uint(v.z); r[4 * c4 + 3] = __float_as_uint(v.w);
        }
        tc_st32(tmem_base + ((uint32_t)(32 * q) << 16) + acol + (uint32_t)c0, r);
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) {
        if (PAIR) tc_bar_arrive_at(tc_at_rank(bar_a, 0u));
        else tc_bar_arrive(bar_a);
      }
    }
    float best = 0.f;                              // OWN_ROWS: the largest squared norm of the thread's rows
    int acc = 0, accround = 0;
    for (int i = 0; i < my_tiles; ++i) {
      const int tile = slice + i * p.nslices;
      const int j0 = tile * p.tile_stride * NT;
      const float* tb = sb + (i & (TC_BT - 1)) * NT;
      if (OWN_ROWS && !DUMP) {
        // up to four groups share the tile's rows, and so do their blocks and a block's warps: 4, 8 or 16 lanes to a row
        const int shares = (int)gridDim.y >= 4 ? 8 : ((int)gridDim.y >= 2 ? 4 : 2), share = 2 * (int)blockIdx.y + (int)rank;
        const int lanes = 2 * shares, j = j0 + share * (NT / shares) + (warp - 2) * (32 / lanes) + lane / lanes;
        if (share < shares) {
          unsigned long long n0 = 0ull, n1 = 0ull;
          if (j < p.N) {
            const ulonglong2* r = reinterpret_cast<const ulonglong2*>(p.W2 + (size_t)j * p.H);
#pragma unroll 8
            for (int c = lane & (lanes - 1); c < p.H >> 2; c += lanes) {
              const ulonglong2 w = r[c];
              asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(n0) : "l"(w.x));
              asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(n1) : "l"(w.y));
            }
          }
          float n = (__uint_as_float((unsigned)n0) + __uint_as_float((unsigned)(n0 >> 32))) +
                    (__uint_as_float((unsigned)n1) + __uint_as_float((unsigned)(n1 >> 32)));
          for (int o = lanes / 2; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
          best = fmaxf(best, n);
        }
      }
      // A warp waits for itself, takes its columns into registers and gives the accumulator back before it looks at them: the
      // next tiles are multiplied meanwhile, and a warp with candidates to append holds up no other (300 samples x 600,011 neurons x
      // 64 units 138 us, so 122).
      tc_bar_wait<PAIR>(bar_bfull + (i & (TC_BT - 1)), (i / TC_BT) & 1, abort_flag);
      tc_bar_wait<PAIR>(bar_accfull + acc, accround & 1, abort_flag);
      __syncwarp();                          // lanes may leave a wait one by one; tensor memory is read by whole warps
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
      for (int c0 = (NT / TC_SPLIT) * half; c0 < (NT / TC_SPLIT) * (half + 1); c0 += 32) {
        uint32_t r[32];
        tc_ld32(tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)(acc * NT + c0), r);
        if (c0 + 32 == (NT / TC_SPLIT) * (half + 1)) {      // the warp's last columns
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) {
            if (PAIR) tc_bar_arrive_at(tc_at_rank(bar_accempty + acc, 0u));
            else tc_bar_arrive(bar_accempty + acc);
          }
        }
        const int jb = j0 + c0;
        float z[32];
#pragma unroll
        for (int c = 0; c < 32; c += 4) {    // two sums in one instruction
          const ulonglong2 bq = *reinterpret_cast<const ulonglong2*>(tb + c0 + c);
          tc_add2(z[c], z[c + 1], r[c], r[c + 1], bq.x);
          tc_add2(z[c + 2], z[c + 3], r[c + 2], r[c + 3], bq.y);
        }
        if (DUMP) {
          // neurons past the end score -infinity
#pragma unroll
          for (int c = 0; c < 32; ++c)
            if (jb + c >= p.N) z[c] = -INFINITY;
          if (p.dump_max == 32) {            // the largest of the thread's 32 (none of them a number: minus infinity)
            __stcg(p.dump + (size_t)(s0 + row) * p.dump_cols + (tile * NT + c0) / 32, tc_max32(z));
          } else if (p.dump_max == 4) {
            float4* out = reinterpret_cast<float4*>(p.dump + (size_t)(s0 + row) * p.dump_cols + (tile * NT + c0) / 4);
#pragma unroll
            for (int c = 0; c < 32; c += 16)
              __stcg(out + c / 16, make_float4(fmaxf(fmaxf(z[c], z[c + 1]), fmaxf(z[c + 2], z[c + 3])), fmaxf(fmaxf(z[c + 4], z[c + 5]), fmaxf(z[c + 6], z[c + 7])),
                                               fmaxf(fmaxf(z[c + 8], z[c + 9]), fmaxf(z[c + 10], z[c + 11])), fmaxf(fmaxf(z[c + 12], z[c + 13]), fmaxf(z[c + 14], z[c + 15]))));
          } else {                           // all of them: 128 contiguous bytes
            float4* out = reinterpret_cast<float4*>(p.dump + (size_t)(s0 + row) * p.dump_cols + (size_t)tile * NT + c0);
#pragma unroll
            for (int c4 = 0; c4 < 8; ++c4) __stcg(out + c4, make_float4(z[4 * c4], z[4 * c4 + 1], z[4 * c4 + 2], z[4 * c4 + 3]));
          }
        } else {
          const float most = tc_max32(z);    // a score that is not a number is none of them
          if (__any_sync(0xffffffffu, most >= tau)) {
            unsigned hm = 0u;
#pragma unroll
            for (int c = 0; c < 32; ++c)
              if (z[c] >= tau) hm |= 1u << c;
            if (p.N - jb < 32) hm &= p.N > jb ? (1u << (p.N - jb)) - 1u : 0u;      // neurons past the end (last tile only)
            // every sample of the warp appends its next one; halving picks its score from the registers
            while (__any_sync(0xffffffffu, hm != 0u)) {
              const int c = (__ffs(hm) - 1) & 31;
              float w[16];
#pragma unroll
              for (int e = 0; e < 16; ++e) w[e] = (c & 16) ? z[e + 16] : z[e];
#pragma unroll
              for (int e = 0; e < 8; ++e) w[e] = (c & 8) ? w[e + 8] : w[e];
#pragma unroll
              for (int e = 0; e < 4; ++e) w[e] = (c & 4) ? w[e + 4] : w[e];
#pragma unroll
              for (int e = 0; e < 2; ++e) w[e] = (c & 2) ? w[e + 2] : w[e];
              const float zc = (c & 1) ? w[1] : w[0];
              if (hm != 0u) {
                if (cnt < p.gbuf) __stcg(mybuf + cnt, make_int2(__float_as_int(zc), jb + c));
                ++cnt;
              }
              hm &= hm - 1u;
            }
          }
        }
      }
      __syncwarp();
      if (lane == 0) tc_bar_arrive(bar_bempty + (i & (TC_BT - 1)));
      if (++acc == nacc) { acc = 0; ++accround; }
    }
    if (OWN_ROWS && !DUMP) {
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, d));
      if (lane == 0) atomicMax(best_slot, __float_as_uint(best));
    }
    if (!DUMP && s0 + row < p.B) {
      p.cand_cnt[(size_t)vslice * p.Bpad + s0 + row] = cnt < p.gbuf ? cnt : p.gbuf;
      if (cnt > p.gbuf) p.need_fix[s0 + row] = 1;          // candidates were dropped: the sample is scored exactly
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (PAIR) tc_cluster_sync();       // nothing of the other block's reaches this one's shared memory any more
  else __syncthreads();
  if (*abort_flag) {                 // of both blocks, or of neither: what has been issued still comes to its end, but not for ever
    const long long until = clock64() + DRAIN_CYCLES;
    if (tid == 0) {
      if (rank == 0)
        for (int f = max(0, fills - nst); f < fills; ++f) tc_bar_drain(bar_full + f % nst, (f / nst) & 1, until);
      else
        while (clock64() < until) __nanosleep(1000);      // its copies are counted in the first block, which may not have asked for the same stages
    }
    if (warp == 1 && rank == 0) {
      __syncwarp();
      if (tc_elect()) tc_commit<PAIR>(bar_drain, 1);      // of the lane that has issued them
      __syncwarp();
      tc_bar_drain(bar_drain, 0, until);
    }
    if (PAIR) tc_cluster_sync();
    else __syncthreads();
  }
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (PAIR) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TC_TMEM_COLS) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TC_TMEM_COLS) : "memory");
  }
  if (OWN_ROWS && !DUMP && tid == 0) atomicMax(p.norm2max, *best_slot);
  if (tid == 0 && *abort_flag) atomicCAS(&p.st->status, 0, (int)DSLIDE_ERR_TIMEOUT);
}

// Floats as keys that order like them (unsigned); no real score has key 0.
__device__ __forceinline__ uint32_t tc_key(float z) {
  const uint32_t b = __float_as_uint(z);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float tc_unkey(uint32_t k) { return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k); }
// The rank-th largest of the keys in the warp's registers, V per lane, found bit by bit down to bit `last` (lower bits zero); 0
// when fewer than rank of them are set.
template <int V>
__device__ __forceinline__ uint32_t tc_select(const uint32_t (&v)[V], int rank, int last) {
  uint32_t K = 0u;
  for (int bit = 31; bit >= last; --bit) {
    const uint32_t trial = K | (1u << bit);
    int n = 0;
#pragma unroll
    for (int i = 0; i < V; ++i) n += v[i] >= trial ? 1 : 0;
    if (__reduce_add_sync(0xffffffffu, n) >= rank) K = trial;
  }
  return K;
}

// A warp per sample.  The sample's scores of the subset (or the largest of 32 neighbours each) are shared out to 512 places
// of the warp's registers, each keeping the largest; the rank-th largest of these maxima, cut to 20 bits, is the sample's
// threshold.  At least rank neurons of the subset reach it (about as many where the best fell to different places); -infinity when
// the subset is smaller than that.  Any threshold gives the same results: it only decides how many candidates the filter pass hands on.
constexpr int TAU_WARPS = 4, TAU_V = 16;
__global__ void __launch_bounds__(32 * TAU_WARPS) k_tc_tau(const float* dump, int cols, int rank, float* tau) {
  const int s = blockIdx.x * TAU_WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  griddep_launch_dependents();
  griddep_wait();                    // the threshold pass has completed
  uint32_t v[TAU_V];
#pragma unroll
  for (int i = 0; i < TAU_V; ++i) v[i] = 0u;
  const float* mine = dump + (size_t)s * cols;
  for (int e0 = lane; e0 < cols; e0 += 32 * TAU_V) {
    float z[TAU_V];
#pragma unroll
    for (int i = 0; i < TAU_V; ++i) z[i] = e0 + 32 * i < cols ? __ldcg(mine + e0 + 32 * i) : 0.f;
#pragma unroll
    for (int i = 0; i < TAU_V; ++i) v[i] = e0 + 32 * i < cols ? max(v[i], tc_key(z[i])) : v[i];
  }
  const uint32_t K = tc_select(v, rank, 12);
  if (lane == 0) {
    float t = tc_unkey(K);
    if (K == 0u || !(t == t)) t = -INFINITY;      // everything passes
    tau[s] = t;
  }
}

// One block per sample: the slices' candidates -> those whose approximate score reaches the cap-th largest of the
// threads' maxima (cap of them, or a few more) -> their exact fp32 logits -> the k best by (logit descending, id
// ascending).  A sample for which the filter cannot be shown to be exact is listed for k_scan_all.
// A chain of memory rounds, each of which asks for all it can: a thread reads the fill of its buffers and their first entries
// together (most hold no more), a warp the rows of four candidates.  With the buffers' fills summed up, a search for every
// entry, a count over the block for every bit of the cut and a row at a time it took 18.9 us for 256 samples x 670,091 neurons x
// 128 units, now 12.4 (1,024 samples: 35 and 20).
constexpr int RF_THREADS = 256, RF_WARPS = RF_THREADS / 32;
constexpr int RF_MAXV = 512;       // buffers per sample at most
constexpr int RF_SLOTS = 384;      // candidates scored exactly at most (k = 64: about 190 reach the cut)
static_assert(RF_MAXV == 2 * RF_THREADS, "two places to a thread");
constexpr int RF_ROWS = 4;         // candidates of a warp side by side
__global__ void __launch_bounds__(RF_THREADS, 4)      // 512 samples in one wave
k_tc_refine(const float* W2, const RowHdr* hdr2, const float* h, const int2* cand, const int* cand_cnt, int gbuf, const float* tau, int Bpad,
            const unsigned int* norm2max, int B, int H, int N, int cap, int nvs, int k, int32_t* out_ids, float* out_scores,
            const int* need_fix, int* n_fix, int* fix_list) {
  __shared__ uint32_t most[RF_THREADS];          // the threads' largest keys
  __shared__ uint32_t sh_K;
  __shared__ float ez[RF_SLOTS], sz[RF_SLOTS];
  __shared__ int ei[RF_SLOTS], si[RF_SLOTS];
  __shared__ float red[RF_WARPS];
  __shared__ int sh_n, sh_fix, sh_total;
  const int s = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) { sh_n = 0; sh_total = 0; }
  griddep_launch_dependents();
  griddep_wait();                                // the filter pass has completed
  if (tid == 0) sh_fix = need_fix[s];            // a buffer of the sample ran over in the filter pass
  const float4* h4 = reinterpret_cast<const float4*>(h + (size_t)s * H);
  const int H4 = H >> 2;
  // A buffer's entries are shared out to 2^lg places, which makes more places than threads: a thread has two at most.  (Where
  // candidates are many in most buffers nearly every thread has a largest key to go by; with 64 results the cut is at the 144th.)
  const int lg = 31 - __clz(RF_MAXV / nvs), g = 1 << lg;
  const int p1 = tid + RF_THREADS, s0 = tid & (g - 1), s1 = p1 & (g - 1);
  const bool two = (p1 >> lg) < nvs;
  const int c0 = (tid >> lg) < nvs ? __ldcg(cand_cnt + (size_t)(tid >> lg) * Bpad + s) : 0;
  const int c1 = two ? __ldcg(cand_cnt + (size_t)(p1 >> lg) * Bpad + s) : 0;
  const int2* buf0 = cand + ((size_t)(tid >> lg) * Bpad + s) * gbuf;
  const int2* buf1 = cand + ((size_t)(p1 >> lg) * Bpad + s) * gbuf;
  int2 first[4];                                 // two entries of each place
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int e = (u < 2 ? s0 : s1) + (u & 1) * g;
    first[u] = e < (u < 2 ? c0 : c1) ? __ldcg((u < 2 ? buf0 : buf1) + e) : make_int2(0, 0);
  }
  // the thread's entries: f(score bits, id)
  auto entries = [&](auto f) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if ((u < 2 ? s0 : s1) + (u & 1) * g < (u < 2 ? c0 : c1)) f(first[u].x, first[u].y);
#pragma unroll 1
    for (int i = 0; i < 2; ++i) {
      const int2* buf = i ? buf1 : buf0;
      const int c = i ? c1 : c0;
#pragma unroll 1
      for (int e0 = (i ? s1 : s0) + 2 * g; e0 < c; e0 += 4 * g) {
        int2 x[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) x[e] = e0 + e * g < c ? __ldcg(buf + e0 + e * g) : make_int2(0, 0);
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (e0 + e * g < c) f(x[e].x, x[e].y);
      }
    }
  };
  int total = 0;
  uint32_t mine = 0u;
  entries([&](int z, int) { const uint32_t key = tc_key(__int_as_float(z)); mine = key > mine ? key : mine; });
  total = __reduce_add_sync(0xffffffffu, (s0 == 0 ? c0 : 0) + (s1 == 0 ? c1 : 0));
  most[tid] = mine;
  if (lane == 0) atomicAdd(&sh_total, total);
  auto find_cut = [&]() {                        // the cap-th of the maxima
    __syncthreads();
    if (warp == 0) {
      uint32_t v[RF_WARPS];
#pragma unroll
      for (int i = 0; i < RF_WARPS; ++i) v[i] = most[32 * i + lane];
      const uint32_t cut = tc_select(v, cap, 12);
      if (lane == 0) sh_K = cut;
    }
    __syncthreads();
  };
  find_cut();
  total = sh_total;
  // The candidates that reach the cap-th largest of the threads' maxima, cut to 20 bits, go on; all of them when there are no more than
  // cap, or when fewer threads than that have any (the cut is 0 then)
  uint32_t K = total <= cap ? 0u : sh_K;
  auto collect = [&]() {
    entries([&](int z, int id) {
      if (tc_key(__int_as_float(z)) >= K) { const int slot = atomicAdd(&sh_n, 1); if (slot < RF_SLOTS) ei[slot] = id; }
    });
  };
  collect();
  __syncthreads();
  if (sh_n > RF_SLOTS) {
    // More than are scored exactly: the best are neighbours, in few buffers and so with few threads, and a cut that the other
    // threads' maxima make up for lets all of them pass.  Shared out anew, by their ids, neighbours have a maximum each
    // (512 of them favoured by 256 samples of 670,091 neurons x 128 units: 162 us, by k_scan_all 2,954; of one sample of 100,003 neurons 62 and 96).
    __syncthreads();
    most[tid] = 0u;
    if (tid == 0) sh_n = 0;
    __syncthreads();
    entries([&](int z, int id) {
      const uint32_t key = tc_key(__int_as_float(z));
      if (key >= K) atomicMax(&most[((unsigned)id * 2654435761u) >> 24], key);
    });
    find_cut();
    if (sh_K > K) K = sh_K;
    collect();
    __syncthreads();
  }
  const int nc = sh_n;
  const bool fix = nc > RF_SLOTS;                // many equal scores at the cut: the sample is scored exactly
  if (!fix) {
  // exact logits of the kept candidates, RF_ROWS of a warp side by side
  for (int e0 = warp; e0 < nc; e0 += RF_ROWS * RF_WARPS) {
    int j[RF_ROWS];
    float4 q[RF_ROWS];                           // four partial sums per lane as in the exact path
#pragma unroll
    for (int u = 0; u < RF_ROWS; ++u) {
      j[u] = ei[e0 + u * RF_WARPS < nc ? e0 + u * RF_WARPS : e0];
      q[u] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const int mine = e0 + (lane < RF_ROWS ? lane : 0) * RF_WARPS;
    const float bias = hdr2[ei[mine < nc ? mine : e0]].b;
#pragma unroll 1
    for (int i = lane; i < H4; i += 32) {
      const float4 x = h4[i];
      float4 a[RF_ROWS];
#pragma unroll
      for (int u = 0; u < RF_ROWS; ++u) a[u] = reinterpret_cast<const float4*>(W2 + (size_t)j[u] * H)[i];
#pragma unroll
      for (int u = 0; u < RF_ROWS; ++u) {
        q[u].x = fmaf(a[u].x, x.x, q[u].x); q[u].y = fmaf(a[u].y, x.y, q[u].y);
        q[u].z = fmaf(a[u].z, x.z, q[u].z); q[u].w = fmaf(a[u].w, x.w, q[u].w);
      }
    }
    float d[RF_ROWS];
#pragma unroll
    for (int u = 0; u < RF_ROWS; ++u) d[u] = (q[u].x + q[u].y) + (q[u].z + q[u].w);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int u = 0; u < RF_ROWS; ++u) d[u] += __shfl_xor_sync(0xffffffffu, d[u], o);
#pragma unroll
    for (int u = 0; u < RF_ROWS; ++u)
      if (lane == u && mine < nc) ez[mine] = bias + d[u];
  }
  // |h|^2 of the sample
  float hs = 0.f;
  for (int c = tid; c < H; c += RF_THREADS) { const float x = h[(size_t)s * H + c]; hs += x * x; }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) hs += __shfl_xor_sync(0xffffffffu, hs, o);
  if (lane == 0) red[warp] = hs;
  __syncthreads();
  // order the exact scores: an entry's place is the number of better ones ((score, id) pairs are all different)
  for (int e = tid; e < nc; e += RF_THREADS) {
    const float z = ez[e]; const int j = ei[e];
    int rank = 0;
    for (int u = 0; u < nc; ++u) rank += tc_better(ez[u], ei[u], z, j) ? 1 : 0;
    sz[rank] = z; si[rank] = j;
  }
  __syncthreads();
  if (tid < k) {
    out_ids[(size_t)s * k + tid] = tid < nc ? si[tid] : -1;
    out_scores[(size_t)s * k + tid] = tid < nc ? sz[tid] : -INFINITY;
  }
  if (tid == 0) {
    float hn = 0.f;
    for (int w = 0; w < RF_WARPS; ++w) hn += red[w];
    // Every neuron that did not go on to the exact pass has an approximate score below T: the cut when there was one
    // here, else the sample's threshold (a neuron below it was never a candidate; the cut is no lower, both are cut to 20 bits).
    // Its exact score is at most T plus the error bound; the k best are certain when the k-th exact score lies above.
    const float T = K != 0u ? tc_unkey(K) : tau[s];
    if (nc < k && nc < N) sh_fix = 1;            // scores that are not numbers never become candidates
    if (T > -INFINITY) {
      const float bound = T + TC_ERR * sqrtf(hn) * sqrtf(__uint_as_float(*norm2max)) + 1e-30f;
      const int kth = (k < nc ? k : nc) - 1;
      if (nc < k || !(sz[kth] > bound)) sh_fix = 1;
    }
  }
  }
  if (tid == 0 && (fix || sh_fix)) fix_list[atomicAdd(n_fix, 1)] = s;      // k_scan_all takes it (in any order: a sample's result is its own)
}

// ---------------------------------------------------------------------------
// Every neuron scored in fp32: for the samples that k_tc_refine lists, or (no list) for all samples of the batch --
// fewer neurons than a tile, or no room for the filter's work space
// ---------------------------------------------------------------------------
// Groups of XS_SG samples x slices of the neurons, as many slices as the grid has blocks for (one listed sample: every
// multiprocessor takes a share of W2; a whole batch: the groups of a slice read its rows at the same time, from L2).  A
// warp takes XS_ROWS rows against the group's activations in shared memory: a lane reads 16 bytes of every row and keeps
// the XS_ROWS x XS_SG partial sums in registers; exchanging what they give up, the lanes end with one total each.  Every
// warp keeps the best k per sample in order in shared memory; the block's lists are merged by a warp per sample, the
// slices' lists by the block that finishes last.  Bound by the rows' bytes for a few samples, by shared memory and the
// multiply-adds for a batch.
constexpr int XS_THREADS = 256, XS_WARPS = XS_THREADS / 32;
constexpr int XS_SG = 8, XS_ROWS = 4;
constexpr int XS_MIN_ROWS = 64;        // of a slice
constexpr int XS_GROUPS = 4096;        // of the largest batch, at one sample each
constexpr int XS_FEW = 512;            // of fewer neurons a group is one sample: there is little to read, and many blocks share the lists' upkeep
static_assert(XS_SG * XS_ROWS == 32 && XS_SG == XS_WARPS, "a lane per (row, sample), a warp per sample when lists are merged");

struct ScanParams {
  const float *W2, *h;
  const RowHdr* hdr2;
  const int *n_list, *list;        // the samples to score; null: all B
  int* done;                       // [XS_GROUPS] finished slices of a group (returns to 0)
  float* pz;                       // [blocks][XS_SG][k] the slices' lists; null: one slice
  int* pi;
  int B, H, N, k, sg;              // sg: samples of a group, XS_SG at most
  int32_t* out_ids;
  float* out_scores;
};

// Whether entry a goes before entry b in a merge (id -1: none).  Scores that are not numbers keep to the order of ids.
__device__ __forceinline__ bool xs_before(float za, int ia, float zb, int ib) {
  if (ia < 0 || ib < 0) return ia >= 0;
  return tc_better(za, ia, zb, ib) || (!tc_better(zb, ib, za, ia) && ia < ib);
}

__global__ void __launch_bounds__(XS_THREADS, 2) k_scan_all(const ScanParams p) {
  extern __shared__ __align__(16) unsigned char xs_smem[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int H = p.H, H4 = H >> 2, k = p.k, N = p.N, G = (int)gridDim.x;
  float* hs = reinterpret_cast<float*>(xs_smem);                             // [XS_SG][H]
  float* lz = hs + XS_SG * H;                                                // [XS_WARPS][XS_SG][k]
  int* li = reinterpret_cast<int*>(lz + XS_WARPS * XS_SG * k);
  int* cnts = li + XS_WARPS * XS_SG * k;                                     // [XS_WARPS][XS_SG]
  uint8_t* heads = reinterpret_cast<uint8_t*>(cnts + XS_WARPS * XS_SG);      // [XS_SG][slices]
  __shared__ int sh_last;
  griddep_launch_dependents();
  griddep_wait();
  const int n = p.n_list ? __ldcg(p.n_list) : p.B;
  const int ngroups = (n + p.sg - 1) / p.sg;
  if (ngroups == 0) return;
  int slices = G / ngroups;
  if (slices > (N + XS_MIN_ROWS - 1) / XS_MIN_ROWS) slices = (N + XS_MIN_ROWS - 1) / XS_MIN_ROWS;
  if (slices < 1 || p.pz == nullptr) slices = 1;
  const int per = (N + slices - 1) / slices;
  const int ms = lane & (XS_SG - 1), mr = lane / XS_SG;                      // the (sample, row) whose total this lane gets
  for (int item = blockIdx.x; item < ngroups * slices; item += G) {
    const int g = item % ngroups, slice = item / ngroups;
    const int ns = min(p.sg, n - g * p.sg);
    const int jb = min(N, slice * per), je = min(N, jb + per);
    auto sample = [&](int s) { return p.n_list ? __ldcg(p.list + g * p.sg + s) : g * p.sg + s; };
    __syncthreads();                           // readers of the item before are done
    for (int s = 0; s < XS_SG; ++s) {
      const float* from = p.h + (size_t)(s < ns ? sample(s) : 0) * H;
      for (int c = tid; c < H; c += XS_THREADS) hs[s * H + c] = s < ns ? __ldcg(from + c) : 0.f;
    }
    __syncthreads();
    const float4* hs4 = reinterpret_cast<const float4*>(hs);
    float* wz = lz + (size_t)warp * XS_SG * k;
    int* wi = li + (size_t)warp * XS_SG * k;
    int cnt = 0, last_i = 0;                   // of sample ms: the list's length, and its last entry once it is full
    float last_z = 0.f;
    for (int j0 = jb + XS_ROWS * warp; j0 < je; j0 += XS_ROWS * XS_WARPS) {
      const float4* row[XS_ROWS];
#pragma unroll
      for (int r = 0; r < XS_ROWS; ++r) row[r] = reinterpret_cast<const float4*>(p.W2 + (size_t)min(j0 + r, je - 1) * H);
      const int j = j0 + mr;
      const float bias = j < je ? p.hdr2[j].b : 0.f;
      float v[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = 0.f;
      for (int c = lane; c < H4; c += 32) {
        float4 w[XS_ROWS];
#pragma unroll
        for (int r = 0; r < XS_ROWS; ++r) w[r] = row[r][c];
#pragma unroll
        for (int s = 0; s < XS_SG; ++s) {
          const float4 x = hs4[s * H4 + c];
#pragma unroll
          for (int r = 0; r < XS_ROWS; ++r) {
            float& a = v[r * XS_SG + s];
            a = fmaf(w[r].x, x.x, a); a = fmaf(w[r].y, x.y, a); a = fmaf(w[r].z, x.z, a); a = fmaf(w[r].w, x.w, a);
          }
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < o; ++i) {
          const float got = __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + o], o);
          v[i] = (up ? v[i + o] : v[i]) + got;
        }
      }
      const float z = bias + v[0];
      unsigned todo = __ballot_sync(0xffffffffu, j < je && ms < ns && (cnt < k || tc_better(z, j, last_z, last_i)));
      while (todo) {                           // rare once the lists have filled
        const int l = __ffs(todo) - 1;
        todo &= todo - 1;
        const int s = l & (XS_SG - 1);
        const float zn = __shfl_sync(0xffffffffu, z, l);
        const int jn = __shfl_sync(0xffffffffu, j, l), have = __shfl_sync(0xffffffffu, cnt, l);
        float *z0 = wz + s * k + lane, *z1 = z0 + 32;
        int *i0 = wi + s * k + lane, *i1 = i0 + 32;
        const bool in0 = lane < have, in1 = lane + 32 < have;
        const float az = in0 ? *z0 : 0.f, bz = in1 ? *z1 : 0.f;
        const int ai = in0 ? *i0 : 0, bi = in1 ? *i1 : 0;
        // the entries that stay before the new one
        const unsigned lo = __ballot_sync(0xffffffffu, in0 && !tc_better(zn, jn, az, ai)), hi = __ballot_sync(0xffffffffu, in1 && !tc_better(zn, jn, bz, bi));
        const int pos = hi ? 64 - __clz(hi) : 32 - __clz(lo);
        if (pos >= k) continue;                // a better one of the same rows has filled the list
        if (in0 && lane >= pos && lane + 1 < k) { z0[1] = az; i0[1] = ai; }
        if (in1 && lane + 32 >= pos && lane + 33 < k) { z1[1] = bz; i1[1] = bi; }
        if (lane == 0) { wz[s * k + pos] = zn; wi[s * k + pos] = jn; }
        __syncwarp();
        if (ms == s) {
          cnt = min(have + 1, k);
          if (cnt == k) { last_z = wz[s * k + k - 1]; last_i = wi[s * k + k - 1]; }
        }
        __syncwarp();
      }
    }
    if (mr == 0) cnts[warp * XS_SG + ms] = cnt;
    __syncthreads();
    // the warps' lists: warp = sample, lane = list
    const int s = warp;
    if (s < ns) {
      const int mine = lane < XS_WARPS ? cnts[lane * XS_SG + s] : 0;
      int head = 0;
      for (int q = 0; q < k; ++q) {
        const int at = (lane * XS_SG + s) * k + head;
        float z = head < mine ? lz[at] : -INFINITY;
        int id = head < mine ? li[at] : -1, who = lane;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const float oz = __shfl_xor_sync(0xffffffffu, z, o);
          const int oi = __shfl_xor_sync(0xffffffffu, id, o), ow = __shfl_xor_sync(0xffffffffu, who, o);
          if (xs_before(oz, oi, z, id)) { z = oz; id = oi; who = ow; }
        }
        who = __shfl_sync(0xffffffffu, who, 0);
        if (lane == who) ++head;
        if (lane == 0) {
          const size_t to = slices == 1 ? (size_t)sample(s) * k + q : ((size_t)item * XS_SG + s) * k + q;
          (slices == 1 ? p.out_ids : p.pi)[to] = id;
          (slices == 1 ? p.out_scores : p.pz)[to] = z;
        }
      }
    }
    if (slices == 1) continue;
    __threadfence();
    __syncthreads();
    if (tid == 0) sh_last = atomicAdd(p.done + g, 1) == slices - 1 ? 1 : 0;
    __syncthreads();
    if (!sh_last) continue;
    __threadfence();                           // the other slices' lists are visible
    if (tid == 0) p.done[g] = 0;
    if (s < ns) {                              // warp = sample, a lane walks the lists lane, lane + 32, ...
      for (int t = lane; t < slices; t += 32) heads[s * slices + t] = 0;
      float z = -INFINITY;
      int id = -1, list = -1;
      bool stale = true;
      for (int q = 0; q < k; ++q) {
        if (stale) {                           // this lane's best entry
          z = -INFINITY; id = -1; list = -1;
          for (int t = lane; t < slices; t += 32) {
            const int hd = heads[s * slices + t];
            if (hd >= k) continue;
            const size_t at = ((size_t)(t * ngroups + g) * XS_SG + s) * k + hd;
            const float tz = __ldcg(p.pz + at);
            const int ti = __ldcg(p.pi + at);
            if (xs_before(tz, ti, z, id)) { z = tz; id = ti; list = t; }
          }
        }
        float bz = z;
        int bi = id, who = lane;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const float oz = __shfl_xor_sync(0xffffffffu, bz, o);
          const int oi = __shfl_xor_sync(0xffffffffu, bi, o), ow = __shfl_xor_sync(0xffffffffu, who, o);
          if (xs_before(oz, oi, bz, bi)) { bz = oz; bi = oi; who = ow; }
        }
        who = __shfl_sync(0xffffffffu, who, 0);
        stale = lane == who && list >= 0;
        if (stale) ++heads[s * slices + list];
        if (lane == 0) {
          p.out_ids[(size_t)sample(s) * k + q] = bi;
          p.out_scores[(size_t)sample(s) * k + q] = bz;
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// rows x H fp32, row-major; boxes of box_rows rows x 32 units, 128-byte swizzle; rows past the end read as zero
static bool make_map(CUtensorMap* m, const float* base, int rows, int H, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)H, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)H * 4};
  const cuuint32_t box[2] = {(cuuint32_t)TC_KB, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Work space of at least `need` bytes; its head (flags, k_scan_all's counters) starts out as zeros.
constexpr size_t WS_DONE = 256, WS_HEAD = WS_DONE + (size_t)XS_GROUPS * 4;
static cudaError_t grow(Ctx* c, size_t need) {
  if (need <= c->pd_cap) return cudaSuccess;
  cudaError_t e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) return e;
  if (c->pd_part) cudaFree(c->pd_part);
  c->pd_part = nullptr; c->pd_cap = 0;
  if ((e = cudaMalloc(&c->pd_part, need)) != cudaSuccess) {
    c->pd_part = nullptr;
    cudaGetLastError();
    return e;
  }
  c->pd_cap = need;
  return cudaMemsetAsync(c->pd_part, 0, WS_HEAD, c->stream);
}

static size_t scan_part_bytes(const Ctx* c, int k) { return (size_t)2 * c->num_sms * XS_SG * k * 8; }

// The lists of the slices are at off_part of the work space (0: none, a group's neurons are not shared out).
static cudaError_t launch_scan_all(Ctx* c, int batch, int k, const int* n_list, const int* list, size_t off_part, int32_t* out_ids, float* out_scores) {
  ScanParams q;
  q.W2 = c->W2; q.h = c->h; q.hdr2 = c->hdr2; q.n_list = n_list; q.list = list;
  unsigned char* ws = reinterpret_cast<unsigned char*>(c->pd_part);
  const int blocks = 2 * c->num_sms;
  q.done = reinterpret_cast<int*>(ws + WS_DONE);
  q.pz = off_part ? reinterpret_cast<float*>(ws + off_part) : nullptr;
  q.pi = reinterpret_cast<int*>(ws + off_part + (size_t)blocks * XS_SG * k * 4);
  q.B = batch; q.H = c->H; q.N = c->N; q.k = k; q.sg = c->N < XS_FEW ? 1 : XS_SG; q.out_ids = out_ids; q.out_scores = out_scores;
  const int smem = XS_SG * c->H * 4 + XS_WARPS * XS_SG * (k * 8 + 4) + XS_SG * blocks;
  const cudaError_t e = cudaFuncSetAttribute(k_scan_all, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
  if (e != cudaSuccess) return e;
  return launch_dependent(k_scan_all, dim3(blocks), dim3(XS_THREADS), (size_t)smem, c->stream, q);
}

static cudaError_t launch_exact_scan(Ctx* c, int batch, int k, int32_t* out_ids, float* out_scores) {
  // few neurons need no slices, and where even their lists find no room the scan does without
  const cudaError_t e = c->N < TC_N ? cudaErrorMemoryAllocation : grow(c, WS_HEAD + scan_part_bytes(c, k));
  if (e != cudaSuccess && e != cudaErrorMemoryAllocation) return e;
  LaunchScope ls(c, KID_PREDICT);
  return launch_scan_all(c, batch, k, nullptr, nullptr, e == cudaSuccess ? WS_HEAD : 0, out_ids, out_scores);
}

// As launch_dependent; the two blocks of a pair are a cluster.
static cudaError_t launch_tc(void (*kernel)(const CUtensorMap, const CUtensorMap, const TcParams), bool wide, bool pair, int slices, int groups, size_t smem,
                             cudaStream_t stream, const CUtensorMap& tmW, const CUtensorMap& tmH, const TcParams& p) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((pair ? 2 : 1) * slices, groups); cfg.blockDim = dim3(tc_threads(wide, pair)); cfg.dynamicSmemBytes = smem; cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = pair ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, tmW, tmH, p);
}

// Whether two multiprocessors share a tile of W2 and 256 samples.  The tile then crosses from L2 once instead of twice, and a
// stage takes half the shared memory; the multiplications take as long as in two blocks (63 to 68 cycles for 256 samples x
// 128 neurons x 8 units, as for 128 x 128 x 8 in a block; of the 2,840 cycles of a tile of 200 units they are 1,650).  It pays
// where a block has room for one tile only (more than 192 units), or streams the activations with the tiles (more than 256):
// us for a call of 1,024 samples x 253,855 neurons x 200 units 371 by single blocks and 256 by pairs, 512 x 4,000,000 x 256
// 2,600 and 1,980, 512 x 100,003 x 512 206 and 135; not at 160 units (300 x 100,003: 69 and 80) or 128 (147.9 and 148.8 for 670,091).  And where the tiles
// keep the pairs busy: a round of tiles takes a pair 0.7 of a block's time, at more than 256 units 1.2 for twice the tile.
static bool use_pairs(const Ctx* c, int batch) {
  if (batch <= TC_M || c->H <= TC_H_SINGLE) return false;
  const bool wide = c->H > TC_H_TMEM;
  auto rounds = [&](bool pair) {
    const int per = (pair ? 2 : 1) * TC_M, groups = (batch + per - 1) / per;
    const int slices = max(1, (pair ? c->num_sms / 2 : c->num_sms) / groups), nt = tc_cols(wide, pair);
    return ((c->N + nt - 1) / nt + slices - 1) / slices;
  };
  return wide ? 6 * rounds(true) < 5 * rounds(false) : 7 * rounds(true) < 10 * rounds(false);
}

// The hidden activations of the batch are in c->h (left there by the forward kernel in predict mode).
cudaError_t launch_dense_tc(Ctx* c, int batch, int k, int32_t* out_ids, float* out_scores) {
  if (c->N < TC_N || encode_fn() == nullptr) return launch_exact_scan(c, batch, k, out_ids, out_scores);
  const int cap = 2 * k + TC_EXTRA;
  const bool wide = c->H > TC_H_TMEM;
  const bool pair = use_pairs(c, batch);
  const int NT = tc_cols(wide, pair);
  const int groups = pair ? (batch + 2 * TC_M - 1) / (2 * TC_M) : (batch + TC_M - 1) / TC_M;      // of 256 samples, or of 128
  const int ntiles = (c->N + NT - 1) / NT;
  int nslices = (pair ? c->num_sms / 2 : c->num_sms) / groups;
  if (nslices < 1) nslices = 1;
  if (nslices > ntiles) nslices = ntiles;
  if (TC_SPLIT * nslices > RF_MAXV) nslices = RF_MAXV / TC_SPLIT;      // k_tc_refine's table of buffer offsets
  // threshold pass: every `stride`-th tile, at most TAU_MAX_TILES of them
  const int TAU_MAX_TILES = 128 * TC_N / NT;
  int stride = TC_SUBSET;
  if ((ntiles + stride - 1) / stride > TAU_MAX_TILES) stride = (ntiles + TAU_MAX_TILES - 1) / TAU_MAX_TILES;
  const int nsub = (ntiles + stride - 1) / stride;
  int nslices_sub = nslices < nsub ? nslices : nsub;
  // work space: the norm bound, the flags, the thresholds, the candidate buffers of every slice and their fill, the
  // threshold pass's scores
  const int Bpad = groups * (pair ? 2 : 1) * TC_M;
  const int nvs = TC_SPLIT * nslices;
  auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
  const size_t off_part = WS_HEAD, off_fix = off_part + up(scan_part_bytes(c, k)), off_list = off_fix + up((size_t)Bpad * 4);
  const size_t off_tau = off_list + up((size_t)Bpad * 4), off_cnt = off_tau + up((size_t)Bpad * 4);
  const size_t off_cand = off_cnt + up((size_t)nvs * Bpad * 4);
  // The threshold is the rank-th best of the subset's maxima, the rank chosen so that about TC_TARGET times as many neurons
  // reach it over all N whatever the subset's share; a buffer has room for four times its expected fill.  A rank of TC_RANK_MIN,
  // for k up to 3, leaves fewer candidates than the cap once in 10^9 samples or less, that of k = 5, 10, once in 10^11 (such a sample
  // is still decided by its threshold, mostly), and one above k keeps that so where the best neighbours are all in the subset.  With a
  // few tiles the subset is one of them: of 129 neurons x 1,024 units 1 in 80 samples is undecided with k = 5, and with k = 64 all of 129
  // neurons and up to 80 % of 384 are, for fewer than k reach rank 24 of 128.
  const int want = min(TC_RANK_CAP, max(TC_RANK_MIN, k + TC_RANK_OVER));
  int rank = (want * TC_TARGET + stride - 1) / stride;
  if (rank > want) rank = want;
  if (rank < 5) rank = 5;
  // Where the subset has enough groups of 32 or 4 neighbours, their largest scores stand for it.
  const int dump_max = nsub * NT / 32 >= 8 * rank ? 32 : (nsub * NT / 4 >= 8 * rank ? 4 : 1);
  const int dump_cols = nsub * NT / dump_max;
  int gbuf = TC_GBUF_MIN * NT / TC_SPLIT;
  while (gbuf * nvs < 4 * rank * stride) gbuf <<= 1;
  const size_t off_dump = off_cand + up((size_t)nvs * Bpad * gbuf * sizeof(int2));
  const size_t need = off_dump + (size_t)Bpad * dump_cols * 4;
  cudaError_t e;
  if ((e = grow(c, need)) != cudaSuccess)       // no room for the filter: scored without it (slower, same results)
    return e == cudaErrorMemoryAllocation ? launch_exact_scan(c, batch, k, out_ids, out_scores) : e;
  unsigned char* ws = reinterpret_cast<unsigned char*>(c->pd_part);
  unsigned int* norm2 = reinterpret_cast<unsigned int*>(ws);
  int* n_fix = reinterpret_cast<int*>(ws) + 1;
  int* need_fix = reinterpret_cast<int*>(ws + off_fix);
  int* fix_list = reinterpret_cast<int*>(ws + off_list);
  float* tau = reinterpret_cast<float*>(ws + off_tau);
  int* cand_cnt = reinterpret_cast<int*>(ws + off_cnt);
  int2* cand = reinterpret_cast<int2*>(ws + off_cand);
  float* dump = reinterpret_cast<float*>(ws + off_dump);

  const int rows = pair ? NT / 2 : NT;               // of a tile, in a block
  CUtensorMap tmW, tmH;
  if (!make_map(&tmW, c->W2, c->N, c->H, rows) || !make_map(&tmH, c->h, batch, c->H, TC_M)) return cudaErrorInvalidValue;

  TcParams p;
  p.hdr2 = c->hdr2; p.h = c->h; p.W2 = c->W2; p.cand = cand; p.cand_cnt = cand_cnt; p.dump = dump; p.tau = tau; p.need_fix = need_fix; p.norm2max = norm2; p.n_fix = n_fix; p.st = c->dstate;
  p.B = batch; p.Bpad = Bpad; p.H = c->H; p.N = c->N; p.dump_cols = dump_cols; p.dump_max = dump_max; p.gbuf = gbuf;
  const size_t tile_bytes = wide ? (size_t)rows * 128 + TC_SUB_BYTES : (size_t)((c->H + TC_KB - 1) / TC_KB) * rows * 128;
  auto smem_of = [&](int st) { return 1024 + tile_bytes * st + (size_t)TC_BT * NT * 4 + (2 + 3 * TC_STAGES + 2 * TC_NACC + 2 * TC_BT) * 8 + 64; };
  // Tiles in flight: six of a narrow model, but beyond three only what 144 KB hold (300 samples x 600,011 neurons x 64 units: 143 us
  // with three or six, 139 with four), and in the threshold pass no more than a block has tiles, mostly one: its blocks and those of
  // the kernels that follow then find room side by side (1 x 5,003 x 64: 28.3 us, with six stages 29.6; 1 x 5,003 x 128 29.1 and 30.4).
  // Pairs keep to one block per multiprocessor: two that wait for tensor memory of the same two could each hold what the other needs.
  const int fit = (int)(((size_t)200 << 10) / tile_bytes), lean = (int)(((size_t)144 << 10) / tile_bytes);
  const int stages = wide ? min(TC_WIDE_STAGES, fit) : min(fit, max(3, min(lean, TC_STAGES)));
  const int sub_tiles = (nsub + nslices_sub - 1) / nslices_sub;
  const int stages_sub = wide || pair ? stages : min(stages, sub_tiles);
  auto k_sub = pair ? (wide ? k_dense_tc<true, true, true> : k_dense_tc<true, false, true>) : (wide ? k_dense_tc<true, true, false> : k_dense_tc<true, false, false>);
  auto k_all = pair ? (wide ? k_dense_tc<false, true, true> : k_dense_tc<false, false, true>) : (wide ? k_dense_tc<false, true, false> : k_dense_tc<false, false, false>);
  if ((e = cudaFuncSetAttribute(k_sub, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_of(stages_sub))) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(k_all, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_of(stages))) != cudaSuccess) return e;
  {
    LaunchScope ls(c, KID_PREDICT);
    p.nslices = nslices_sub; p.ntiles = nsub; p.tile_stride = stride; p.stages = stages_sub;
    // each kernel of the call may be placed while the kernel before it drains (they wait for it before they read or
    // write anything); the first follows the hidden-layer kernel in the same way
    if ((e = launch_tc(k_sub, wide, pair, nslices_sub, groups, smem_of(stages_sub), c->stream, tmW, tmH, p)) != cudaSuccess) return e;
    if ((e = launch_dependent(k_tc_tau, dim3(Bpad / TAU_WARPS), dim3(32 * TAU_WARPS), 0, c->stream, (const float*)dump, dump_cols, rank, tau)) != cudaSuccess)
      return e;
    p.nslices = nslices; p.ntiles = ntiles; p.tile_stride = 1; p.stages = stages;
    if ((e = launch_tc(k_all, wide, pair, nslices, groups, smem_of(stages), c->stream, tmW, tmH, p)) != cudaSuccess) return e;
    if ((e = launch_dependent(k_tc_refine, dim3(batch), dim3(RF_THREADS), 0, c->stream, (const float*)c->W2, (const RowHdr*)c->hdr2,
                              (const float*)c->h, (const int2*)cand, (const int*)cand_cnt, gbuf, (const float*)tau, Bpad,
                              (const unsigned int*)norm2, batch, c->H, c->N, cap, nvs, k, out_ids, out_scores, (const int*)need_fix, n_fix, fix_list)) !=
        cudaSuccess)
      return e;
    if ((e = launch_scan_all(c, batch, k, n_fix, fix_list, off_part, out_ids, out_scores)) != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace dslide
