// Per-sample forward kernel of the SLIDE step: one thread block per sample runs
//   hidden layer (Section 3.6, feed forward of the first type: sparse input)
//   -> L bucket codes of the hidden activation (SimHash or DWTA, Section 4.1)
//   -> bucket lookup, union over the tables plus the labels (Section 2.1, Fig. 1)
//   -> logits over the active set only (feed forward of the second type)
//   -> softmax, loss and errors over that ragged set (Algorithm 1 "Compute Errors")
//   -> error back-propagated to the hidden layer (Section 2.1, back-propagation stage)
// and hands the touched rows of W2 and W1 to the update kernel.
// The same kernel in predict mode stops after the logits and selects the top k.
//
// Every phase is a short chain of memory rounds, so each round puts as much in flight as it can:
// the rows of W1 of a chunk of nonzeros arrive together by 16-byte asynchronous copies and are summed in the stored order
// (beyond 512 units a thread copies and adds its own piece of every row); the L bucket offsets are fetched in one round and
// all bucket entries in a second; the active rows of W2 are staged in the shared memory the dedup work space no longer needs and
// serve logits, sums and the back-propagated error, or, in wide layers and sets larger than that space, pass through a ring of
// every warp, which takes all of these in one pass.  Optional steps of the selection: densification
// of all-zero DWTA bins of the query (Section 4.1) and the sampling budget of Section 3.7.
// A block's eight warps issue an instruction every four cycles or so: code that is run once costs more than the loads it waits for.
#include "common.cuh"
#include "waits.cuh"

namespace dslide {

constexpr int FWD_THREADS = 256;
constexpr int FWD_WARPS = FWD_THREADS / 32;
constexpr int ACT_SM = 1024;      // active ids and logits are mirrored in shared memory when the set is this small
constexpr int HID_MIN_BYTES = 64 * 1024;   // staging space for the hidden layer's rows of W1
constexpr int RANK_MAX = 1024;    // candidate sets up to this size are put in order by counting, larger ones by a bitonic sort
constexpr int SORT_SMALL = 1024;  // candidate sets up to this size are sorted rather than run through the bitmap
constexpr int SORT_FEW = 160, BITMAP_CHEAP = 32768;      // ... and up to this size when all neurons are few
constexpr unsigned FULLM = 0xffffffffu;

struct FwdParams {
  const float *W1, *b1, *W2;
  const int32_t *hash_idx, *hash_sign, *bucket_off, *bucket_ids;
  const uint16_t* hash_pk;     // SimHash: [fn_len][KL] coordinate, top bit = minus
  const int32_t *row_ptr, *col_idx;
  const float* vals;
  const int32_t *label_ptr, *labels;
  float *h, *dh, *loss;
  uint32_t* codes;
  int32_t *act_cnt, *act_ids;
  float *act_z, *act_p, *act_g;
  uint32_t *mask1, *mask2;
  uint32_t* touch2;         // MODE 2: a bit per row of W2 that some sample touches
  int2 *ovf1, *ovf2;
  const int32_t* hotmap1;   // rows of W1 with a line of the coefficient table
  float* hotcoef1;
  int bstride;              // samples per line of that table
  RowHdr *hdr1, *hdr2;
  int2 *own1, *own2;
  int32_t *hot_rows, *med_rows;
  DevState* st;
  int32_t* out_ids;
  float* out_scores;
  long long nb;
  int B, D, H, N, K, L, KL, family, lg_bin, fn_len, cap;
  int act_stride, Wd, dense, dedup_mode, max_labels, sort_cap, topk, parity;
  int stage_bytes;     // bytes of the staging region (it starts at off_dedup and overlays the dedup work space)
  int hid_rows;        // rows of W1 staged per chunk of the hidden layer
  int budget;          // Section 3.7: active neurons kept per sample, labels included (0 = no budget)
  int budget_fill;     // Section 3.7: a set below the budget is topped up with uniform draws
  unsigned long long tcount;   // steps taken so far (the reservoir's draws are numbered by step, sample and candidate)
  int densify;         // DWTA: all-zero bins of the query borrow another bin's position
  unsigned long long seed, rcount;   // for the probe sequence of the densification: the model's seed, rebuilds so far
  int hash_sm_off;     // where in the staging region the hash functions' index tables are mirrored (-1: read from global memory)
  int hash_sm_bytes;
  int hash_sm_late;    // of which the first ones lie where the hidden layer's rows are staged
  int sort_small;      // candidate sets up to this size are deduplicated by sorting even when a bitmap is available
  // LSH-sampled hidden layer (L1 > 0): projections over the input coordinates, tables over the hidden neurons
  const int8_t* proj1;
  const int32_t *bucket1_off, *bucket1_ids;
  uint32_t *codes1, *hmask, *cmask1;
  int K1, L1, KL1, cap1, Hw, off_h1;
  int inputs_ready;    // the batch arrays were complete before the launch: they may be read before griddep_wait()
  int off_dh, off_code, off_part, off_misc, off_lab, off_tbase, off_tbeg, off_topk, off_ids, off_z, off_col, off_val,
      off_dedup;
};

__device__ __forceinline__ void set_status(DevState* st, int code) { atomicCAS(&st->status, 0, code); }

// ---- bulk copy (global -> shared) with completion on an mbarrier ------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// 16-byte asynchronous copy global -> shared (through L2 only), and the wait for all of a thread's copies
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// Until at most n of the thread's groups of copies are in flight, n <= 7
__device__ __forceinline__ void cp_async_wait_pending(int n) {
  switch (n) {
    case 0: asm volatile("cp.async.wait_group 0;" ::: "memory"); break;
    case 1: asm volatile("cp.async.wait_group 1;" ::: "memory"); break;
    case 2: asm volatile("cp.async.wait_group 2;" ::: "memory"); break;
    case 3: asm volatile("cp.async.wait_group 3;" ::: "memory"); break;
    case 4: asm volatile("cp.async.wait_group 4;" ::: "memory"); break;
    case 5: asm volatile("cp.async.wait_group 5;" ::: "memory"); break;
    case 6: asm volatile("cp.async.wait_group 6;" ::: "memory"); break;
    default: asm volatile("cp.async.wait_group 7;" ::: "memory");
  }
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
// The touch that takes a row past ROW_SLOTS touching samples enters the row in the list of rows that a warp of
// the update kernel sums from slots and mask; the touch that takes it past HOT_T enters it in the list of rows
// summed in slices.  The row's count word is marked so that the update kernel knows where the row is listed.
__device__ __forceinline__ void list_row(const FwdParams& p, uint32_t* cnt, int code, unsigned nth) {
  if (nth == (unsigned)ROW_SLOTS) {
    const unsigned at = atomicAdd(&p.st->n_med[p.parity], 1u);
    if (at < (unsigned)MED_CAP) {
      p.med_rows[at] = code;
      atomicOr(cnt, CNT_MED);
    }
  }
  if (nth == (unsigned)HOT_T) {
    const unsigned at = atomicAdd(&p.st->n_hot[p.parity], 1u);
    if (at < (unsigned)HOT_CAP) {
      p.hot_rows[at] = code;
      atomicOr(cnt, CNT_HOT);
    }
  }
}

// Handing a touched row to the update kernel, once the row's touch counter has answered (nth = touches before this
// one).  touch_mark: the (sample, coefficient) pair goes into the row's slot nth, or, past the slots, the sample's bit
// into the row's mask (and, up to PAIR_T touches, the pair into the side array); the touch that fills the slots or
// reaches HOT_T lists the row (list_row: an atomic whose answer is needed, so callers on the critical path put it
// off to the end of the kernel).  own_reserve / own_store: the first toucher enters (row, its own sample) in the list
// of distinct rows, so that the update kernel can fetch that sample's row at once; positions are handed out per
// warp by one atomic, asked for by own_reserve and used by own_store (callers put other work in between, so that
// no warp waits for the answer).  All three are called by whole warps; `live` tells whether this thread has a touch.
template <bool LIST = true>      // LIST = false: the caller lists the row (list_row) itself, later
__device__ __forceinline__ void touch_mark(const FwdParams& p, bool live, RowHdr* hd, uint32_t* maskrow, int2* ovfrow, int code,
                                           unsigned nth, int s, float coef) {
  if (!live) return;
  if (nth < (unsigned)ROW_SLOTS) hd->slot[nth] = make_int2(s, __float_as_int(coef));
  else {
    atomicOr(maskrow + (s >> 5), 1u << (s & 31));
    // up to PAIR_T touches keep their pair as well, so that a row with that many is summed without any search
    if (nth < (unsigned)PAIR_T) ovfrow[nth] = make_int2(s, __float_as_int(coef));
  }
  if (LIST) list_row(p, &hd->cnt, code, nth);
}
__device__ __forceinline__ unsigned own_reserve(bool first, unsigned int* n_own) {
  const unsigned fm = __ballot_sync(FULLM, first);
  unsigned base = 0;
  if (fm && (threadIdx.x & 31) == 0) base = atomicAdd(n_own, (unsigned)__popc(fm));
  return base;                                   // valid in lane 0
}
__device__ __forceinline__ void own_store(bool first, unsigned base, int2* own, int row, int s) {
  const int lane = threadIdx.x & 31;
  const unsigned fm = __ballot_sync(FULLM, first);
  if (!fm) return;
  base = __shfl_sync(FULLM, base, 0);
  if (first) own[base + __popc(fm & ((1u << lane) - 1u))] = make_int2(row, s);
}
__device__ __forceinline__ void finish_touch(const FwdParams& p, bool live, RowHdr* hd, uint32_t* maskrow, int2* ovfrow, int2* own,
                                             unsigned int* n_own, int row, int code, unsigned nth, int s, float coef) {
  touch_mark(p, live, hd, maskrow, ovfrow, code, nth, s, coef);
  const bool first = live && nth == 0u;
  const unsigned base = own_reserve(first, n_own);
  own_store(first, base, own, row, s);
}

// The whole hand-off of one nonzero (entry e of the batch's columns) of sample s, by a whole warp.
__device__ __forceinline__ void touch_w1(const FwdParams& p, bool live, int e, int s) {
  int c = 0;
  unsigned nth = 0u;
  float x = 0.f;
  if (live) {
    c = __ldg(p.col_idx + e);
    x = __ldg(p.vals + e);
    nth = atomicAdd(&p.hdr1[c].cnt, 1u) & CNT_MASK;
    const int line = __ldcg(p.hotmap1 + c);
    if (line >= 0) p.hotcoef1[(size_t)line * p.bstride + s] = x;
  }
  finish_touch(p, live, p.hdr1 + c, p.mask1 + (size_t)c * p.Wd, p.ovf1 + (size_t)c * PAIR_T, p.own1, &p.st->n_own[p.parity][1], c, ~c, nth, s, x);
}

// Maximum / sum over the lanes of a warp in a fixed order (same value in every lane).
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v = fmaxf(v, __shfl_xor_sync(FULLM, v, d));
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(FULLM, v, d);
  return v;
}

// Exclusive prefix sum of one int per thread over the block; *total gets the block sum.
// sh needs FWD_WARPS + 1 ints.  Ends with a barrier, so sh may be reused afterwards.
__device__ __forceinline__ int block_excl_scan(int v, int* sh, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    int n = __shfl_up_sync(FULLM, incl, d);
    if (lane >= d) incl += n;
  }
  if (lane == 31) sh[warp] = incl;
  __syncthreads();
  if (threadIdx.x == 0) {
    int run = 0;
    for (int w = 0; w < FWD_WARPS; ++w) { int c = sh[w]; sh[w] = run; run += c; }
    sh[FWD_WARPS] = run;
  }
  __syncthreads();
  int res = incl - v + sh[warp];
  *total = sh[FWD_WARPS];
  __syncthreads();
  return res;
}

// Block-wide max / sum in a fixed order (same value in every thread).  sh: FWD_WARPS floats.
__device__ __forceinline__ float block_max(float v, float* sh) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v = fmaxf(v, __shfl_xor_sync(FULLM, v, d));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = sh[0];
  for (int w = 1; w < FWD_WARPS; ++w) r = fmaxf(r, sh[w]);
  __syncthreads();
  return r;
}
__device__ __forceinline__ float block_sum(float v, float* sh) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(FULLM, v, d);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = sh[0];
  for (int w = 1; w < FWD_WARPS; ++w) r += sh[w];
  __syncthreads();
  return r;
}

// Floats as keys that order like them (unsigned; both zeros are one), those that are no numbers last; no number has key 0.
__device__ __forceinline__ uint32_t score_key(float z) {
  const uint32_t b = __float_as_uint(z + 0.f);      // minus zero plus zero is zero
  return z != z ? 1u : (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
// A score and its position as a word: the larger is the better, of equal scores the earlier
__device__ __forceinline__ unsigned long long place_of(float z, int a) { return ((unsigned long long)score_key(z) << 32) | (uint32_t)~a; }
// Inference: the k best of the scores zp[0 .. na) by (score descending, id ascending); ids ascend with the position (ids
// null: they are the positions).  The scores that reach the k-th largest of the threads' maxima (about k of them) are counted
// against one another: a score's place is the number of better ones.  Where too many are equal there, the best is taken k times.
// Lists of k per warp, fed one score at a time by lane 0, took 11,000 to 14,600 of the 35,000 to 45,000 cycles of a block (154 to
// 238 scores, 1 and 5 results), and their merge 1,400 to 5,700: 256 samples x 670,091 neurons, 5 results, 29.4 us, now 20.0;
// 64 samples with 6,000 scores of 128 units, 64 results, 620 us, now 108.
// mine: the best of the thread's own scores (any sharing out; place_of: zero when it has none).  work: [512].  Called by the whole
// block.  With k = 1 the scores are not read again (zp need not hold them).
constexpr int BEST_N = 384;
__device__ __noinline__ void best_of(int32_t* out_i, float* out_z, int k, const int* ids, const float* zp, int na, unsigned long long mine,
                                     unsigned long long* work, int* sh_n) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  auto most = [&](unsigned long long best) {         // over the block
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      const unsigned long long o = __shfl_xor_sync(FULLM, best, d);
      best = o > best ? o : best;
    }
    if (lane == 0) work[warp] = best;
    __syncthreads();
    for (int w = 0; w < FWD_WARPS; ++w) best = work[w] > best ? work[w] : best;
    return best;
  };
  if (k == 1) {
    const unsigned long long best = most(mine);
    if (tid == 0) {
      const uint32_t key = (uint32_t)(best >> 32);
      const int a = (int)~(uint32_t)best;
      out_i[0] = na == 0 ? -1 : ids ? ids[a] : a;
      out_z[0] = na == 0 ? -INFINITY : key == 1u ? NAN : __uint_as_float((key & 0x80000000u) ? (key & 0x7fffffffu) : ~key);
    }
    return;
  }
  uint32_t* sh_max = reinterpret_cast<uint32_t*>(work + BEST_N);      // [FWD_THREADS]
  sh_max[tid] = (uint32_t)(mine >> 32);
  if (tid == 0) *sh_n = 0;
  __syncthreads();                     // the scores are visible to the block, too
  // every warp finds the cut by itself, bit by bit; the last bits are left out: a few more scores reach it
  uint32_t v[FWD_WARPS], K = 0u;
#pragma unroll
  for (int i = 0; i < FWD_WARPS; ++i) v[i] = sh_max[32 * i + lane];
  for (int bit = 31; bit >= 12; --bit) {
    const uint32_t trial = K | (1u << bit);
    int c = 0;
#pragma unroll
    for (int i = 0; i < FWD_WARPS; ++i) c += v[i] >= trial ? 1 : 0;
    if (__reduce_add_sync(FULLM, c) >= k) K = trial;
  }
  constexpr int U = 8;
  for (int a0 = tid; a0 < na; a0 += U * FWD_THREADS) {
    uint32_t key[U];
#pragma unroll
    for (int u = 0; u < U; ++u) key[u] = a0 + u * FWD_THREADS < na ? score_key(zp[a0 + u * FWD_THREADS]) : 0u;
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (a0 + u * FWD_THREADS < na && key[u] >= K) {
        const int at = atomicAdd(sh_n, 1);
        if (at < BEST_N) work[at] = ((unsigned long long)key[u] << 32) | (uint32_t)~(a0 + u * FWD_THREADS);
      }
  }
  __syncthreads();
  const int n = *sh_n;
  auto put = [&](int place, unsigned long long x) {
    const int a = (int)~(uint32_t)x;
    out_i[place] = ids ? ids[a] : a;
    out_z[place] = zp[a];
  };
  for (int q = na + tid; q < k; q += FWD_THREADS) { out_i[q] = -1; out_z[q] = -INFINITY; }      // fewer scores than results
  if (n <= BEST_N) {
    for (int e = tid; e < n; e += FWD_THREADS) {
      const unsigned long long x = work[e];
      int place = 0;
#pragma unroll 4
      for (int u = 0; u < n; ++u) place += work[u] > x ? 1 : 0;
      if (place < k) put(place, x);
    }
    return;
  }
  __syncthreads();
  unsigned long long last = ~0ull;     // (na > BEST_N >= k)
  for (int q = 0; q < k; ++q) {
    unsigned long long best = 0ull;
    for (int a = tid; a < na; a += FWD_THREADS) {
      const unsigned long long x = place_of(zp[a], a);
      if (x < last && x > best) best = x;
    }
    best = most(best);
    __syncthreads();
    last = best;
    if (tid == 0) put(q, best);
  }
}

// Puts n <= PER * FWD_THREADS values in ascending order by counting: the place of a value is the number of values
// before it (by value, then by position).  src and dst are in shared memory; thread t owns the values t, t +
// FWD_THREADS, ...; threads without a value skip the counting loop.
// PACKED: src holds (value << RANK_BITS | position), padded with 0xffffffff to a multiple of four -- all distinct,
// so one comparison per pair decides; dst receives the values alone.
constexpr int RANK_BITS = 10;
template <int PER, bool PACKED>
__device__ __forceinline__ void rank_sort(const uint32_t* src, uint32_t* dst, int n) {
  const int tid = threadIdx.x;
  if (tid >= n) return;
  uint32_t v[PER];
  int pos[PER];
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int i = tid + u * FWD_THREADS;
    v[u] = i < n ? src[i] : 0xffffffffu;
    pos[u] = 0;
  }
  if (PACKED) {
    const uint4* src4 = reinterpret_cast<const uint4*>(src);
    const int n4 = (n + 3) >> 2;
#pragma unroll 2
    for (int k = 0; k < n4; ++k) {
      const uint4 a = src4[k];
#pragma unroll
      for (int u = 0; u < PER; ++u)
        pos[u] += (a.x < v[u] ? 1 : 0) + (a.y < v[u] ? 1 : 0) + (a.z < v[u] ? 1 : 0) + (a.w < v[u] ? 1 : 0);
    }
#pragma unroll
    for (int u = 0; u < PER; ++u)
      if (tid + u * FWD_THREADS < n) dst[pos[u]] = v[u] >> RANK_BITS;
  } else {
#pragma unroll 4
    for (int k = 0; k < n; ++k) {
      const uint32_t a = src[k];
#pragma unroll
      for (int u = 0; u < PER; ++u) pos[u] += (a < v[u] || (a == v[u] && k < tid + u * FWD_THREADS)) ? 1 : 0;
    }
#pragma unroll
    for (int u = 0; u < PER; ++u)
      if (tid + u * FWD_THREADS < n) dst[pos[u]] = v[u];
  }
}

// Section 3.7, the fill option: a set below the budget is topped up with neurons drawn one after the other,
// id_k = rng(seed, RNG_FILL, steps taken, sample * 2^32 + k) mod N; a draw already in the set (retrieved, label, or
// drawn before) is passed over; drawing stops when the set has min(budget, N) members or after 2 * missing + 64
// draws.  All draws are evaluated at once: a shared-memory hash set records the first draw of every id, a search in
// the (ascending) set tells which ids are new, and the running count in draw order says which of them still fit.
// The accepted ids are put in order and merged with the set.  Returns the new count.
__device__ __forceinline__ int fill_work_bytes(int need) {
  const int D = 2 * need + 64;
  int ts = 64;
  while (ts < 2 * D) ts <<= 1;
  return 4 * D + ((D + 3) & ~3) + 8 * ts + 8 * need;       // draws, flags, hash set (ids, first draws), accepted ids twice
}
__device__ __noinline__ int budget_fill(int budget, int N, uint64_t seed, uint64_t tcount, int s, int32_t* ids, int* sh_ids,
                                        int na, unsigned char* work, int work_bytes, int* sh_scan, DevState* st) {
  const int tid = threadIdx.x;
  const int target = min(budget, N);
  if (na >= target) return na;
  const int need = target - na;
  const int D = 2 * need + 64;
  int ts = 64;
  while (ts < 2 * D) ts <<= 1;
  if (fill_work_bytes(need) + 4 * target > work_bytes) {     // cannot happen with the sizes checked at start-up
    if (tid == 0) set_status(st, DSLIDE_ERR_OVERFLOW);
    return na;
  }
  int* draw = reinterpret_cast<int*>(work);                 // [D]
  unsigned char* okf = reinterpret_cast<unsigned char*>(draw + D);       // [D]
  int* keys = reinterpret_cast<int*>(okf + ((D + 3) & ~3)); // [ts] ids seen, -1 = empty
  int* mink = keys + ts;                                    // [ts] the first draw of that id
  int* F = mink + ts;                                       // [need] accepted ids in draw order
  int* Fs = F + need;                                       // [need] ascending
  int* out = Fs + need;                                     // [target]
  const int lg = 31 - __clz(ts);
  for (int h = tid; h < ts; h += FWD_THREADS) { keys[h] = -1; mink[h] = 0x7fffffff; }
  for (int k = tid; k < D; k += FWD_THREADS)
    draw[k] = (int)(ctr_rng(seed, RNG_FILL, tcount, ((uint64_t)(uint32_t)s << 32) + (uint64_t)k) % (uint64_t)N);
  __syncthreads();
  for (int k = tid; k < D; k += FWD_THREADS) {
    const int id = draw[k];
    unsigned h = ((unsigned)id * 2654435761u) >> (32 - lg);
    for (int it = 0; it < ts; ++it) {
      const int prev = atomicCAS(&keys[h], -1, id);
      if (prev == -1 || prev == id) { atomicMin(&mink[h], k); break; }
      h = (h + 1) & (unsigned)(ts - 1);
    }
  }
  __syncthreads();
  for (int k = tid; k < D; k += FWD_THREADS) {
    const int id = draw[k];
    unsigned h = ((unsigned)id * 2654435761u) >> (32 - lg);
    bool first = false;
    for (int it = 0; it < ts; ++it) {
      if (keys[h] == id) { first = mink[h] == k; break; }
      h = (h + 1) & (unsigned)(ts - 1);
    }
    int lo = 0, hi = na;                                    // is the id in the set already?
    while (lo < hi) { const int mid = (lo + hi) >> 1; const int v = mid < ACT_SM ? sh_ids[mid] : ids[mid]; if (v < id) lo = mid + 1; else hi = mid; }
    const bool in_set = lo < na && (lo < ACT_SM ? sh_ids[lo] : ids[lo]) == id;
    okf[k] = (first && !in_set) ? 1 : 0;
  }
  __syncthreads();
  // running count in draw order: the first `need` new ids are accepted
  const int chunk = (D + FWD_THREADS - 1) / FWD_THREADS;
  const int k0 = min(D, tid * chunk), k1 = min(D, k0 + chunk);
  int cnt = 0;
  for (int k = k0; k < k1; ++k) cnt += okf[k];
  int total_ok = 0;
  int at = block_excl_scan(cnt, sh_scan, &total_ok);
  for (int k = k0; k < k1; ++k)
    if (okf[k]) { if (at < need) F[at] = draw[k]; ++at; }
  const int got = min(total_ok, need);
  __syncthreads();
  for (int j = tid; j < got; j += FWD_THREADS) {            // ascending order by counting (the ids are distinct)
    const int v = F[j];
    int r = 0;
    for (int q = 0; q < got; ++q) r += F[q] < v ? 1 : 0;
    Fs[r] = v;
  }
  __syncthreads();
  for (int i = tid; i < na; i += FWD_THREADS) {             // merge: each element lands after the smaller ones of both lists
    const int v = i < ACT_SM ? sh_ids[i] : ids[i];
    int lo = 0, hi = got;
    while (lo < hi) { const int mid = (lo + hi) >> 1; if (Fs[mid] < v) lo = mid + 1; else hi = mid; }
    out[i + lo] = v;
  }
  for (int j = tid; j < got; j += FWD_THREADS) {
    const int v = Fs[j];
    int lo = 0, hi = na;
    while (lo < hi) { const int mid = (lo + hi) >> 1; const int w = mid < ACT_SM ? sh_ids[mid] : ids[mid]; if (w < v) lo = mid + 1; else hi = mid; }
    out[j + lo] = v;
  }
  __syncthreads();
  const int total = na + got;
  for (int a = tid; a < total; a += FWD_THREADS) {
    ids[a] = out[a];
    if (a < ACT_SM) sh_ids[a] = out[a];
  }
  __syncthreads();
  return total;
}

// Section 3.7: the sample's retrieved neurons exceed the sampling budget -> reservoir sampling keeps
// m = max(0, budget - labels) of those that are not labels.  The textbook algorithm runs over the candidates in
// ascending id order: the first m fill the reservoir, candidate i >= m draws j uniform in [0, i] and replaces slot j
// when j < m.  Its outcome is fixed by the draws alone -- slot j ends with the LAST candidate that drew j, or with
// candidate j itself -- so the block evaluates all draws at once and settles every slot with a shared-memory max.
// ids[0 .. na) (ascending, mirrored in sh_ids up to ACT_SM) is rewritten with the labels and the reservoir,
// ascending; returns the new count.  work: 4 * na + 4 * m + nc + 4 * (m + labels) bytes of shared memory.
// Called by the whole block; kept out of line because most configurations never run it.
__device__ __noinline__ int budget_select(int budget, int fill, int N, uint64_t seed, uint64_t tcount, int s, int32_t* ids,
                                          int* sh_ids, int na, const int32_t* lab, int nlab, unsigned char* work,
                                          int work_bytes, int* sh_scan, DevState* st) {
  const int tid = threadIdx.x;
  int* cidx = reinterpret_cast<int*>(work);                 // [na] index among the candidates, -1 for a label
  const int chunk = (na + FWD_THREADS - 1) / FWD_THREADS;
  const int a0 = min(na, tid * chunk), a1 = min(na, a0 + chunk);
  int cnt = 0;
  for (int a = a0; a < a1; ++a) {
    const int id = a < ACT_SM ? sh_ids[a] : ids[a];
    bool isl = false;
    for (int i = 0; i < nlab; ++i) isl = isl || lab[i] == id;
    cidx[a] = isl ? -1 : 0;
    cnt += isl ? 0 : 1;
  }
  int nc = 0;
  int at = block_excl_scan(cnt, sh_scan, &nc);
  const int ny = na - nc;
  const int m = max(0, budget - ny);
  if (nc <= m)                                               // uniform over the block
    return fill ? budget_fill(budget, N, seed, tcount, s, ids, sh_ids, na, work, work_bytes, sh_scan, st) : na;
  for (int a = a0; a < a1; ++a)
    if (cidx[a] == 0) cidx[a] = at++;
  int* win = cidx + na;                                      // [m] the last candidate that drew the slot
  unsigned char* sel = reinterpret_cast<unsigned char*>(win + m);        // [nc]
  int* out = reinterpret_cast<int*>(work + (((size_t)4 * na + (size_t)4 * m + nc + 15) & ~(size_t)15));  // [m + ny]
  for (int j = tid; j < m; j += FWD_THREADS) win[j] = -1;
  for (int i = tid; i < nc; i += FWD_THREADS) sel[i] = 0;
  __syncthreads();
  for (int a = a0; a < a1; ++a) {
    const int i = cidx[a];
    if (i >= m) {
      const uint64_t u = ctr_rng(seed, RNG_SAMPLE, tcount, ((uint64_t)(uint32_t)s << 32) + (uint64_t)i);
      const int j = (int)(u % (uint64_t)(i + 1));
      if (j < m) atomicMax(&win[j], i);
    }
  }
  __syncthreads();
  for (int j = tid; j < m; j += FWD_THREADS) sel[win[j] >= 0 ? win[j] : j] = 1;
  __syncthreads();
  cnt = 0;
  for (int a = a0; a < a1; ++a) cnt += (cidx[a] < 0 || sel[cidx[a]]) ? 1 : 0;
  int total = 0;
  at = block_excl_scan(cnt, sh_scan, &total);
  for (int a = a0; a < a1; ++a)
    if (cidx[a] < 0 || sel[cidx[a]]) out[at++] = a < ACT_SM ? sh_ids[a] : ids[a];
  __syncthreads();
  for (int a = tid; a < total; a += FWD_THREADS) {
    ids[a] = out[a];
    if (a < ACT_SM) sh_ids[a] = out[a];
  }
  __syncthreads();
  return total;
}

// SimHash sums of the hidden activation, carried on over n rows (coordinates) of the packed table: a warp reads 32 functions'
// i-th coordinates (top bit = minus) side by side; their places in h are close together (a function's coordinates ascend), so
// few of the reads conflict.  A thread has the functions f and f + FWD_THREADS: each a chain of additions in stored order.
__device__ __forceinline__ void simhash_rows(const float* h, const uint16_t* pk, int f, int KL, int n, float& sum0, float& sum1) {
  auto term = [&](unsigned e) { return __uint_as_float(__float_as_uint(h[e & 0x7fffu]) ^ (e & 0x8000u) << 16); };
  const uint16_t* q = pk + f;
  if (f + FWD_THREADS < KL) {
#pragma unroll 4
    for (int i = 0; i < n; ++i, q += KL) {
      const unsigned e0 = q[0], e1 = q[FWD_THREADS];
      sum0 = __fadd_rn(sum0, term(e0));
      sum1 = __fadd_rn(sum1, term(e1));
    }
  } else if (f < KL) {
#pragma unroll 4
    for (int i = 0; i < n; ++i, q += KL) sum0 = __fadd_rn(sum0, term(q[0]));
  }
}
// A packed table larger than the staging space passes through its two halves, a piece on its way while the other is read (700
// functions of 171 coordinates: 20,500 cycles of a block, 55,000 from global memory; a step of 16 samples x 512 units 147 us, now
// 79).  Up to SIM_SUMS functions per thread.  The number of pieces (bar0 has completed half of them, rounded up, bar1 the others);
// 0 when one did not come in time, with nothing left in flight.  Called by the whole block; out of line, so that the other
// families' blocks stay short (in line a step of 256 samples of the 670,091-neuron shape took 65.0 us for 64.3).
constexpr int SIM_SUMS = 4;
__device__ __noinline__ int simhash_in_pieces(const float* h, const uint16_t* table, int KL, int n_all, unsigned char* space, int space_bytes, uint64_t* bar0,
                                              uint64_t* bar1, unsigned char* bits) {
  const int tid = threadIdx.x;
  const int half = (space_bytes / 2) & ~127, per = max(8, (half / (2 * KL)) & ~7), pieces = (n_all + per - 1) / per;
  float sum[SIM_SUMS] = {0.f, 0.f, 0.f, 0.f};
  auto fetch = [&](int c) {
    const uint32_t bytes = (uint32_t)((min(per, n_all - c * per) * KL * 2 + 15) & ~15);
    uint64_t* bar = (c & 1) ? bar1 : bar0;
    mbar_expect_tx(bar, bytes);
    bulk_g2s(space + (c & 1) * half, table + (size_t)c * per * KL, bytes, bar);
  };
  fence_proxy_async();
  __syncthreads();
  if (tid == 0) {
    fetch(0);
    if (pieces > 1) fetch(1);
  }
  for (int c = 0; c < pieces; ++c) {
    const bool ok = bar_wait_limited((c & 1) ? bar1 : bar0, (uint32_t)(c >> 1) & 1u);
    if (__syncthreads_or(ok ? 0 : 1)) {
      bar_wait_limited((c & 1) ? bar1 : bar0, (uint32_t)(c >> 1) & 1u);
      if (c + 1 < pieces) bar_wait_limited((c & 1) ? bar0 : bar1, (uint32_t)((c + 1) >> 1) & 1u);
      __syncthreads();
      return 0;
    }
    const uint16_t* pk = reinterpret_cast<const uint16_t*>(space + (c & 1) * half);
    const int n = min(per, n_all - c * per);
    simhash_rows(h, pk, tid, KL, n, sum[0], sum[1]);
    simhash_rows(h, pk, tid + 2 * FWD_THREADS, KL, n, sum[2], sum[3]);
    fence_proxy_async();
    __syncthreads();
    if (tid == 0 && c + 2 < pieces) fetch(c + 2);
  }
#pragma unroll
  for (int u = 0; u < SIM_SUMS; ++u)
    if (tid + u * FWD_THREADS < KL) bits[tid + u * FWD_THREADS] = sum[u] >= 0.f ? 1 : 0;
  return pieces;
}

// The sample is skipped: no loss, no gradient, nothing touched (predict: no candidates).
template <int MODE>
__device__ __forceinline__ void skip_sample(const FwdParams& p, int s, int code) {
  const int tid = threadIdx.x;
  if (MODE != 1) {
    for (int k = tid; k < p.H; k += FWD_THREADS) { p.h[(size_t)s * p.H + k] = 0.f; p.dh[(size_t)s * p.H + k] = 0.f; }
    if (tid == 0) { p.act_cnt[s] = 0; p.loss[s] = 0.f; }
  } else {
    for (int q = tid; q < p.topk; q += FWD_THREADS) {
      p.out_ids[(size_t)s * p.topk + q] = -1;
      p.out_scores[(size_t)s * p.topk + q] = -INFINITY;
    }
  }
  if (tid == 0) set_status(p.st, code);
}

// Rows of a group in the pass over the active rows: eight 16-byte pieces of them in a lane's registers, four rows at most (a reduction,
// an exponential and a look at the maximum for all of them)
template <int NP> struct RowPass { static constexpr int ROWS = NP <= 2 ? 4 : 8 / NP; };
constexpr int RING_DEPTH = 8;      // groups of a warp's ring at most
constexpr int RING_HEAD = FWD_WARPS * RING_DEPTH * 8 + 16;      // the rings' barriers, and 16 bytes of zeros

// MODE 0 = training step, 1 = predict top-k, 2 = the part of a training step up to the active sets (tiles.cu goes on from
// there: sets of many neurons that the batch's samples share); NP = 16-byte pieces of a row that a lane holds (H <= 128 * NP);
// BULK, of NP = 1: active sets of many chunks are expected (the host's estimate from the tables' shape) and their rows come by bulk copies
template <int MODE, int NP, bool BULK = false>
__global__ void __launch_bounds__(FWD_THREADS, 2) k_forward(const FwdParams p) {
  constexpr int KPT = NP <= 2 ? 1 : NP / 2;      // hidden units per thread
  extern __shared__ __align__(128) unsigned char smem[];
  float* sh_h = reinterpret_cast<float*>(smem);
  float* sh_dh = reinterpret_cast<float*>(smem + p.off_dh);          // [FWD_WARPS][H]
  uint32_t* sh_code = reinterpret_cast<uint32_t*>(smem + p.off_code);
  unsigned char* sh_part = smem + p.off_part;
  int* sh_misc = reinterpret_cast<int*>(smem + p.off_misc);          // 32 ints
  float* sh_red = reinterpret_cast<float*>(sh_misc + 16);
  uint64_t* sh_bar = reinterpret_cast<uint64_t*>(sh_misc + 26);      // 8-byte aligned: off_misc is 16-byte aligned
  uint64_t* sh_bar2 = reinterpret_cast<uint64_t*>(sh_misc + 28);     // completion of the hash functions' mirror 
  int* sh_lab = reinterpret_cast<int*>(smem + p.off_lab);            // [max_labels]
  int* sh_tbase = reinterpret_cast<int*>(smem + p.off_tbase);        // [L + 1]
  int* sh_tbeg = reinterpret_cast<int*>(smem + p.off_tbeg);          // [L]
  int* sh_ids = reinterpret_cast<int*>(smem + p.off_ids);            // [ACT_SM]
  float* sh_z = reinterpret_cast<float*>(smem + p.off_z);            // [ACT_SM]
  float* sh_g = reinterpret_cast<float*>(smem + p.off_topk);         // [ACT_SM] training: errors of a small set (predict: work space of best_of)
  int* sh_col = reinterpret_cast<int*>(smem + p.off_col);            // [hid_rows]
  float* sh_val = reinterpret_cast<float*>(smem + p.off_val);        // [hid_rows]
  unsigned char* sh_b1 = smem + p.off_h1;                            // [256] bits of the hidden layer's projections
  int* sh_c1beg = reinterpret_cast<int*>(smem + p.off_h1 + 256);     // [64] start of the slice of every hidden-layer table
  int* sh_c1cnt = sh_c1beg + 64;                                     // [64] and its length
  uint32_t* sh_hmask = reinterpret_cast<uint32_t*>(sh_c1cnt + 64);   // [32] active hidden neurons of the sample
  uint32_t* sh_dd = reinterpret_cast<uint32_t*>(smem + p.off_dedup);
  float* stage = reinterpret_cast<float*>(smem + p.off_dedup);       // overlays the dedup work space

  const int s = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int H = p.H, H4 = H >> 2, N = p.N;
  // Unless the caller has promised that the batch arrays were complete before the launch, they may still be being
  // written by the kernel before this one in the stream: wait for it before the first read.
  bool waited = false;
  if (!p.inputs_ready) {
    griddep_wait();
    waited = true;
  }
  const int rbeg = p.row_ptr[s], rend = p.row_ptr[s + 1];
  const int nnz = rend - rbeg;
  int lbeg = 0, nlab = 0;
  if (MODE != 1) { lbeg = p.label_ptr[s]; nlab = p.label_ptr[s + 1] - lbeg; }

  griddep_launch_dependents();       // the update kernel may be placed as blocks of this one leave
  const void* hash_tab = p.family == DSLIDE_SIMHASH ? static_cast<const void*>(p.hash_pk) : static_cast<const void*>(p.hash_idx);
  if (tid == 0) {
    sh_misc[24] = 0;                 // bucket entries fetched by this sample
    mbar_init(sh_bar, 1);
    mbar_init(sh_bar2, p.hash_sm_late > 0 ? 2 : 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    // the hash functions' tables (constant between rebuilds) come into the upper part of the staging region, which
    // is free until the candidates are collected; what reaches down into the rows of W1 comes after the hidden layer
    if (p.hash_sm_off >= 0 && !p.dense) {
      const int now = p.hash_sm_bytes - p.hash_sm_late;
      mbar_expect_tx(sh_bar2, (uint32_t)now);
      if (now > 0) bulk_g2s(smem + p.off_dedup + p.hash_sm_off + p.hash_sm_late, static_cast<const unsigned char*>(hash_tab) + p.hash_sm_late, (uint32_t)now, sh_bar2);
    }
  }

  // ---- label checks: ids in range, list within the maximum (merged with the column checks by the first barrier) ----
  int bad = 0;
  if (nnz < 0 || nlab < 0) bad = DSLIDE_ERR_BAD_INDEX;
  else if (MODE != 1) {
    for (int i = tid; i < nlab; i += FWD_THREADS) {
      int y = p.labels[lbeg + i];
      if (y < 0 || y >= N) bad = DSLIDE_ERR_BAD_INDEX;
    }
  }
  const bool too_many_labels = MODE != 1 && nnz >= 0 && nlab > p.max_labels;

  // ---- hidden layer: bias, then one fused multiply-add per nonzero in stored order, ReLU.  The rows of W1 of a
  //      chunk of nonzeros are copied into shared memory together, 16 bytes per thread and copy (cp.async: all of
  //      them in flight at once, no registers held), and then summed per hidden unit in the stored order; the
  //      column ids are checked on the way (in range, ascending) ----
  //      Up to here, and through the first chunk's column ids and values, only the caller's batch is read: with
  //      inputs_ready the kernel runs that far while the previous step's update kernel is still finishing.
  float acc[KPT];
  float s1 = 0.f;                    // sampled hidden layer: the input's sum under projection `tid`
  int c1 = 0, line1 = -1;            // this thread's nonzero (tid-th of the sample), kept for the hand-off to the update kernel
  float x1 = 0.f;
  const int R = p.hid_rows;
  // a thread's place in the copy pattern: 16-byte piece c4 of row r, advancing FWD_THREADS pieces per round
  const int cp_dr = FWD_THREADS / H4, cp_dc = FWD_THREADS - cp_dr * H4;
  const int cp_r0 = tid / H4, cp_c0 = tid - cp_r0 * H4;
  bool pieced = false;
  if constexpr (NP == 8) {
  if (p.L1 == 0 && H > 512 && nnz > R && nnz <= ACT_SM) {
    // More rows than a chunk (more than 512 units): a thread owns a 16-byte piece of every row, copies it and adds it up, HID_G rows to a
    // group of copies, as many groups ahead as fit -- no barriers.  (In chunks, a barrier before and after each, 76 rows of 1,024
    // units took 33,000 cycles of a block: a step of 1,024 samples 498 us, so 472; of one sample 48.6 and 43.7.  Of up to 512 units,
    // half of the threads or fewer, it is the slower: 64 x 512 units 72.0 and 73.2; steps by tiles, which take this instance from 257 units
    // on, of 64 samples x 200 nonzeros x 260 units 197.9 and 206.3, 256 x 76 x 384 340.9 and 344.0.)
    pieced = true;
    constexpr int HID_G = 4;
    for (int i = tid; i < nnz; i += FWD_THREADS) {
      const int c = __ldg(p.col_idx + rbeg + i);
      const int prev = i > 0 ? __ldg(p.col_idx + rbeg + i - 1) : -1;
      const bool okc = c >= 0 && c < p.D && prev < c;
      if (!okc) bad = DSLIDE_ERR_BAD_INDEX;
      const float xv = __ldg(p.vals + rbeg + i);
      sh_ids[i] = okc ? c : 0;
      sh_z[i] = xv;
      if (i == tid) { c1 = okc ? c : 0; x1 = xv; }
    }
    bad = __syncthreads_or(bad);
    if (!bad) {
      if (!waited) {
        griddep_wait();
        waited = true;
      }
      if (MODE == 0 && tid < R) line1 = __ldcg(p.hotmap1 + c1);      // (nnz > R)
      if (tid < H4) {
        float4 a = reinterpret_cast<const float4*>(p.b1)[tid];
        const int depth = min(8, R / HID_G), ngroups = (nnz + HID_G - 1) / HID_G;
        int asked = 0, to = 0, from = 0;
        auto ask = [&]() {
#pragma unroll
          for (int q = 0; q < HID_G; ++q) {
            const int i = asked * HID_G + q;
            if (i < nnz) cp_async16(stage + (size_t)(to * HID_G + q) * H + 4 * tid, p.W1 + (size_t)sh_ids[i] * H + 4 * tid);
          }
          cp_async_commit();
          ++asked;
          to = to + 1 == depth ? 0 : to + 1;
        };
        for (int g = 0; g < depth - 1; ++g) ask();
#pragma unroll 1
        for (int g = 0; g < ngroups; ++g) {
          ask();
          cp_async_wait_pending(depth - 1);
#pragma unroll
          for (int q = 0; q < HID_G; ++q) {
            const int i = g * HID_G + q;
            if (i < nnz) {
              const float4 w = *reinterpret_cast<const float4*>(stage + (size_t)(from * HID_G + q) * H + 4 * tid);
              const float xv = sh_z[i];
              a.x = __fmaf_rn(xv, w.x, a.x); a.y = __fmaf_rn(xv, w.y, a.y); a.z = __fmaf_rn(xv, w.z, a.z); a.w = __fmaf_rn(xv, w.w, a.w);
            }
          }
          from = from + 1 == depth ? 0 : from + 1;
        }
        reinterpret_cast<float4*>(sh_h)[tid] = a;
      }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < KPT; ++u) acc[u] = tid + u * FWD_THREADS < H ? sh_h[tid + u * FWD_THREADS] : 0.f;
  }
  }
  for (int c0 = 0; c0 < nnz && !pieced; c0 += R) {
    const int nr = min(R, nnz - c0);
    for (int i = tid; i < nr; i += FWD_THREADS) {
      const int c = __ldg(p.col_idx + rbeg + c0 + i);
      const int prev = c0 + i > 0 ? __ldg(p.col_idx + rbeg + c0 + i - 1) : -1;
      const bool okc = c >= 0 && c < p.D && prev < c;
      if (!okc) bad = DSLIDE_ERR_BAD_INDEX;
      sh_col[i] = okc ? c : 0;
      const float xv = __ldg(p.vals + rbeg + c0 + i);
      sh_val[i] = xv;
      if (c0 + i == tid) { c1 = okc ? c : 0; x1 = xv; }
    }
    bad = __syncthreads_or(bad);     // also: the previous chunk's readers of the staging space are done
    if (bad) break;                  // nothing was copied
    if (!waited) {
      griddep_wait();
      waited = true;
    }
    // a feature that has been hot before has a line of the coefficient table (written by the update kernel)
    if (MODE == 0 && c0 == 0 && tid < nr) line1 = __ldcg(p.hotmap1 + c1);
    for (int r = cp_r0, c4 = cp_c0; r < nr;) {
      cp_async16(stage + (size_t)r * H + 4 * c4, p.W1 + (size_t)sh_col[r] * H + 4 * c4);
      c4 += cp_dc; r += cp_dr;
      if (c4 >= H4) { c4 -= H4; ++r; }
    }
    if (c0 == 0) {
#pragma unroll
      for (int u = 0; u < KPT; ++u) {
        const int k = tid + u * FWD_THREADS;
        acc[u] = k < H ? p.b1[k] : 0.f;
      }
    }
    if (p.L1 > 0 && tid < p.KL1) {
      // sampled hidden layer: the input's sum under projection `tid`, nonzeros in stored order (coordinates that the
      // projection does not select add nothing)
      const int8_t* pj = p.proj1 + tid;
      for (int i0 = 0; i0 < nr; i0 += 16) {
        int e[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) e[j] = i0 + j < nr ? (int)__ldg(pj + (size_t)sh_col[i0 + j] * p.KL1) : 0;
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (e[j] != 0) s1 = __fadd_rn(s1, e[j] > 0 ? sh_val[i0 + j] : -sh_val[i0 + j]);
      }
    }
    cp_async_wait_all();
    __syncthreads();
#pragma unroll
    for (int u = 0; u < KPT; ++u) {
      const int k = tid + u * FWD_THREADS;
      if (k < H) {
        float a = acc[u];
#pragma unroll 8
        for (int i = 0; i < nr; ++i) a = __fmaf_rn(sh_val[i], stage[(size_t)i * H + k], a);
        acc[u] = a;
      }
    }
    if (c0 + R < nnz) __syncthreads();       // the next chunk overwrites the column ids and values
  }
  if (nnz <= 0) bad = __syncthreads_or(bad);       // no chunk, no barrier yet: the label checks are merged here
  if (!waited) {                     // no nonzeros, or a bad column id: nothing of the model has been read yet
    griddep_wait();
#pragma unroll
    for (int u = 0; u < KPT; ++u) {
      const int k = tid + u * FWD_THREADS;
      acc[u] = k < H ? p.b1[k] : 0.f;
    }
  }
  if (bad || too_many_labels) {
    if (p.hash_sm_off >= 0 && !p.dense) {          // no copy into this block may be left in flight
      if (p.hash_sm_late > 0 && tid == 0) mbar_expect_tx(sh_bar2, 0u);
      bar_wait_limited(sh_bar2, 0u);
    }
    skip_sample<MODE>(p, s, (!bad && too_many_labels) ? DSLIDE_ERR_OVERFLOW : DSLIDE_ERR_BAD_INDEX);
    return;
  }
  if (p.L1 > 0) {
    // ---- sampled hidden layer (Algorithm 1: retrieve the layer's active neurons with the layer's input): codes of
    //      the input, one bucket slice per table, union as a bit mask over the hidden neurons.  A neuron that is
    //      not retrieved is a NoOp: activation 0 (Section 2.1) ----
    if (tid < p.KL1) sh_b1[tid] = s1 >= 0.f ? 1 : 0;
    if (tid < 32) sh_hmask[tid] = 0u;
    __syncthreads();
    if (tid < p.L1) {
      uint32_t code = 0;
      for (int k = 0; k < p.K1; ++k) code |= (uint32_t)sh_b1[tid * p.K1 + k] << k;
      if (MODE != 1) p.codes1[(size_t)s * p.L1 + tid] = code;
      const int32_t* off = p.bucket1_off + (size_t)tid * ((1 << p.K1) + 1) + code;
      const int beg = __ldg(off);
      int cnt = __ldg(off + 1) - beg;
      sh_c1beg[tid] = beg;
      sh_c1cnt[tid] = cnt < p.cap1 ? cnt : p.cap1;
    }
    __syncthreads();
    for (int t = warp; t < p.L1; t += FWD_WARPS)
      for (int i = lane; i < sh_c1cnt[t]; i += 32) {
        const int k = __ldg(p.bucket1_ids + (size_t)t * H + sh_c1beg[t] + i);
        atomicOr(&sh_hmask[k >> 5], 1u << (k & 31));
      }
    __syncthreads();
    if (MODE != 1 && tid < p.Hw) p.hmask[(size_t)s * p.Hw + tid] = sh_hmask[tid];
  }
#pragma unroll
  for (int u = 0; u < KPT; ++u) {
    const int k = tid + u * FWD_THREADS;
    if (k < H) {
      const bool on = p.L1 == 0 || ((sh_hmask[k >> 5] >> (k & 31)) & 1u);
      const float hv = (on && acc[u] > 0.f) ? acc[u] : 0.f;
      sh_h[k] = hv;
      if (MODE != 1 || p.dense) p.h[(size_t)s * H + k] = hv;
    }
  }
  if (MODE == 1 && p.dense) return;        // inference over all neurons: the logits are taken by the kernels of dense_tc.cu
  if (p.hash_sm_late > 0) fence_proxy_async();
  __syncthreads();
  if (p.hash_sm_late > 0 && !p.dense && tid == 0) {
    mbar_expect_tx(sh_bar2, (uint32_t)p.hash_sm_late);
    bulk_g2s(smem + p.off_dedup + p.hash_sm_off, hash_tab, (uint32_t)p.hash_sm_late, sh_bar2);
  }

  const bool dense = p.dense != 0;
  uint32_t w2phase = 0u;             // of sh_bar
  bool marked = false;               // MODE 2: the rows' bits have been set from the sample's bitmap
  int na = N;
  int32_t* ids = p.act_ids + (size_t)s * p.act_stride;

  if (!dense) {
    // ---- bucket codes of the hidden activation ----
    const int32_t* hidx = p.hash_idx;
    const uint16_t* hpk = p.hash_pk;
    if (p.hash_sm_off >= 0) {
      const bool ok = bar_wait_limited(sh_bar2, 0u);
      if (__syncthreads_or(ok ? 0 : 1)) {          // the mirror did not arrive in time: the sample is given up
        bar_wait_limited(sh_bar2, 0u);
        __syncthreads();
        skip_sample<MODE>(p, s, DSLIDE_ERR_TIMEOUT);
        return;
      }
      hidx = reinterpret_cast<const int32_t*>(smem + p.off_dedup + p.hash_sm_off);
      hpk = reinterpret_cast<const uint16_t*>(hidx);
    }
    if (p.family == DSLIDE_SIMHASH) {
      if (p.hash_sm_off >= 0 || p.KL > SIM_SUMS * FWD_THREADS) {      // mirrored, or from global memory: thousands of functions
        for (int f = tid; f < p.KL; f += 2 * FWD_THREADS) {
          float sum0 = 0.f, sum1 = 0.f;
          simhash_rows(sh_h, hpk, f, p.KL, p.fn_len, sum0, sum1);
          sh_part[f] = sum0 >= 0.f ? 1 : 0;
          if (f + FWD_THREADS < p.KL) sh_part[f + FWD_THREADS] = sum1 >= 0.f ? 1 : 0;
        }
      } else {
        const int pieces = simhash_in_pieces(sh_h, p.hash_pk, p.KL, p.fn_len, smem + p.off_dedup, p.stage_bytes, sh_bar2, sh_bar, sh_part);
        if (pieces == 0) {                           // not in time: the sample is given up
          skip_sample<MODE>(p, s, DSLIDE_ERR_TIMEOUT);
          return;
        }
        w2phase = (uint32_t)(pieces >> 1) & 1u;      // of sh_bar
      }
    } else
    for (int f = tid; f < p.KL; f += FWD_THREADS) {
      const int32_t* ix = hidx + (size_t)f * p.fn_len;
      if (p.fn_len == 8 && (reinterpret_cast<uintptr_t>(hidx) & 15) == 0) {
        // bins of eight: both halves of the index list in one load each, the eight values fetched side by side
        const int4 ia = reinterpret_cast<const int4*>(ix)[0], ib = reinterpret_cast<const int4*>(ix)[1];
        const float v0 = sh_h[ia.x], v1 = sh_h[ia.y], v2 = sh_h[ia.z], v3 = sh_h[ia.w];
        const float v4 = sh_h[ib.x], v5 = sh_h[ib.y], v6 = sh_h[ib.z], v7 = sh_h[ib.w];
        int best = 0;
        float bv = v0;
        if (v1 > bv) { bv = v1; best = 1; }       // strict: the lowest position wins ties
        if (v2 > bv) { bv = v2; best = 2; }
        if (v3 > bv) { bv = v3; best = 3; }
        if (v4 > bv) { bv = v4; best = 4; }
        if (v5 > bv) { bv = v5; best = 5; }
        if (v6 > bv) { bv = v6; best = 6; }
        if (v7 > bv) { bv = v7; best = 7; }
        sh_part[f] = (unsigned char)best;
        sh_part[p.KL + f] = bv == 0.f ? 1 : 0;     // activations are not negative: a maximum of zero is a bin of zeros
      } else {
        int best = 0;
        float bv = sh_h[ix[0]];
        for (int i = 1; i < p.fn_len; ++i) {
          float v = sh_h[ix[i]];
          if (v > bv) { bv = v; best = i; }       // strict: the lowest position wins ties
        }
        sh_part[f] = (unsigned char)best;
        sh_part[p.KL + f] = bv == 0.f ? 1 : 0;
      }
    }
    __syncthreads();
    // ---- codes, and the slice of every table's bucket the sample reads: all offsets in one round ----
    const int shift = p.family == DSLIDE_SIMHASH ? 1 : p.lg_bin;
    auto table_code = [&](int t) -> uint32_t {
      uint32_t code = 0;
      for (int k = 0; k < p.K; ++k) {
        const int f = t * p.K + k;
        uint32_t pos = sh_part[f];
        if (p.densify && p.family == DSLIDE_DWTA && sh_part[p.KL + f] && p.KL > 1) {
          // a bin of zeros: the position of the first probed function whose own bin is not all zero, else 0
          pos = 0;
          for (int a = 0; a < DENSIFY_ATTEMPTS; ++a) {
            const uint64_t u = ctr_rng(p.seed, RNG_PROBE, p.rcount, (uint64_t)f * DENSIFY_ATTEMPTS + (uint64_t)a);
            const int g = (int)(((uint64_t)f + 1u + u % (uint64_t)(p.KL - 1)) % (uint64_t)p.KL);
            if (!sh_part[p.KL + g]) { pos = sh_part[g]; break; }
          }
        }
        code |= pos << (k * shift);
      }
      return code;
    };
    if (p.L <= 64) {
      // up to 64 tables: one warp fetches all the offsets (two tables per lane) and takes the running sum of the
      // slice lengths in registers -- one barrier instead of two
      if (warp == 0) {
        int beg[2], cnt[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int t = lane + 32 * u;
          beg[u] = 0; cnt[u] = 0;
          if (t < p.L) {
            const uint32_t code = table_code(t);
            sh_code[t] = code;
            if (MODE != 1) p.codes[(size_t)s * p.L + t] = code;
            const int32_t* off = p.bucket_off + (size_t)t * (size_t)(p.nb + 1) + code;
            beg[u] = __ldg(off);
            cnt[u] = __ldg(off + 1);
          }
        }
        int run = 0;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int t = lane + 32 * u;
          int c = cnt[u] - beg[u];
          c = c < p.cap ? c : p.cap;
          int incl = c;
#pragma unroll
          for (int d = 1; d < 32; d <<= 1) {
            int n = __shfl_up_sync(FULLM, incl, d);
            if (lane >= d) incl += n;
          }
          if (t < p.L) { sh_tbeg[t] = beg[u]; sh_tbase[t + 1] = run + incl; }
          run += __shfl_sync(FULLM, incl, 31);
        }
        if (lane == 0) { sh_tbase[0] = 0; sh_misc[24] = run; }
      }
      __syncthreads();
    } else {
      for (int t = tid; t < p.L; t += FWD_THREADS) {
        const uint32_t code = table_code(t);
        sh_code[t] = code;
        if (MODE != 1) p.codes[(size_t)s * p.L + t] = code;
        const int32_t* off = p.bucket_off + (size_t)t * (size_t)(p.nb + 1) + code;
        const int beg = __ldg(off);
        int cnt = __ldg(off + 1) - beg;
        cnt = cnt < p.cap ? cnt : p.cap;
        sh_tbeg[t] = beg;
        sh_tbase[t + 1] = cnt;
      }
      __syncthreads();
      if (warp == 0) {            // running sum of the slice lengths: where each table's candidates start
        int run = 0;
        for (int b = 0; b < p.L; b += 32) {
          const int t = b + lane;
          const int v = t < p.L ? sh_tbase[t + 1] : 0;
          int incl = v;
#pragma unroll
          for (int d = 1; d < 32; d <<= 1) {
            int n = __shfl_up_sync(FULLM, incl, d);
            if (lane >= d) incl += n;
          }
          if (t < p.L) sh_tbase[t + 1] = run + incl;
          run += __shfl_sync(FULLM, incl, 31);
        }
        if (lane == 0) { sh_tbase[0] = 0; sh_misc[24] = run; }
      }
      __syncthreads();
    }

    // ---- all bucket entries in one round; union over the tables, labels, duplicates removed, ascending ids.
    //      A small candidate set is cheaper to sort than a bitmap over all N neurons is to clear and scan. ----
    const int ncand = sh_tbase[p.L];
    int total = 0;
    const bool bitmap = p.dedup_mode == 1 && ncand + nlab > p.sort_small;
    int n2 = 1;
    if (!bitmap) while (n2 < ncand + nlab) n2 <<= 1;
    // ids short enough to share a word with their position are sorted as such words
    const bool packed = !bitmap && ncand + nlab <= RANK_MAX && N <= (1 << (32 - RANK_BITS));
    if (bitmap) {
      uint4* dd4 = reinterpret_cast<uint4*>(sh_dd);
      const int n4 = (((N + 31) >> 5) + 3) >> 2;
      for (int w = tid; w < n4; w += FWD_THREADS) dd4[w] = make_uint4(0u, 0u, 0u, 0u);
      __syncthreads();
    }
    if (bitmap && ncand >= 16 * p.L) {
      // long slices: a warp takes two tables at a time, their entries side by side and four rounds in flight (a thread per
      // candidate searched for its table first: 27,000 cycles for 50 slices of 128, so 7,000)
      for (int t = warp; t < p.L; t += 2 * FWD_WARPS) {
        const int t1 = t + FWD_WARPS < p.L ? t + FWD_WARPS : t;
        const int n0 = sh_tbase[t + 1] - sh_tbase[t], n1 = t1 != t ? sh_tbase[t1 + 1] - sh_tbase[t1] : 0;
        const int32_t *s0 = p.bucket_ids + (size_t)t * N + sh_tbeg[t], *s1 = p.bucket_ids + (size_t)t1 * N + sh_tbeg[t1];
        for (int i0 = lane; i0 - lane < max(n0, n1); i0 += 128) {
          int j0[4], j1[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            j0[u] = i0 + 32 * u < n0 ? __ldg(s0 + i0 + 32 * u) : -1;
            j1[u] = i0 + 32 * u < n1 ? __ldg(s1 + i0 + 32 * u) : -1;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if (j0[u] >= 0) atomicOr(&sh_dd[j0[u] >> 5], 1u << (j0[u] & 31));
            if (j1[u] >= 0) atomicOr(&sh_dd[j1[u] >> 5], 1u << (j1[u] & 31));
          }
        }
      }
    } else {
      for (int c = tid; c < ncand; c += FWD_THREADS) {
        int lo = 0, hi = p.L - 1;          // last table whose candidates start at or before c
        while (lo < hi) { int mid = (lo + hi + 1) >> 1; if (sh_tbase[mid] <= c) lo = mid; else hi = mid - 1; }
        const int j = __ldg(p.bucket_ids + (size_t)lo * N + sh_tbeg[lo] + (c - sh_tbase[lo]));
        if (bitmap) atomicOr(&sh_dd[j >> 5], 1u << (j & 31));
        else sh_dd[c] = packed ? ((uint32_t)j << RANK_BITS) | (uint32_t)c : (uint32_t)j;
      }
    }
    if (MODE != 1)
      for (int i = tid; i < nlab; i += FWD_THREADS) {
        const int y = p.labels[lbeg + i];
        if (bitmap) atomicOr(&sh_dd[y >> 5], 1u << (y & 31));
        else sh_dd[ncand + i] = packed ? ((uint32_t)y << RANK_BITS) | (uint32_t)(ncand + i) : (uint32_t)y;
      }
    if (bitmap) {
      __syncthreads();
      // every warp takes a contiguous share of the words, WU times 32 at a time; a lane writes out the ids of its words, one of
      // each in turn (one word at a time 31,000 cycles for 6,000 ids of 253,855, so 20,000)
      constexpr int WU = 4;
      const int nwords = (N + 31) >> 5;
      const int share = ((nwords + FWD_WARPS - 1) / FWD_WARPS + 31) & ~31;
      const int wbeg = min(nwords, warp * share), wend = min(nwords, wbeg + share);
      int cnt = 0;
#pragma unroll 4
      for (int w = wbeg + lane; w < wend; w += 32) cnt += __popc(sh_dd[w]);
      cnt = __reduce_add_sync(FULLM, cnt);
      if (lane == 0) sh_misc[warp] = cnt;
      __syncthreads();
      int pos = 0;
      for (int q = 0; q < FWD_WARPS; ++q) {
        const int cq = sh_misc[q];
        if (q < warp) pos += cq;
        total += cq;
      }
      if (total <= p.act_stride && cnt > 0 && share == 32) {       // few words: all of the warp's at once
        const uint32_t mine = wbeg + lane < wend ? sh_dd[wbeg + lane] : 0u;
        int at = __popc(mine);
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const int n = __shfl_up_sync(FULLM, at, d);
          if (lane >= d) at += n;
        }
        at += pos - __popc(mine);
        for (uint32_t bits = mine; bits; bits &= bits - 1) {
          const int j = ((wbeg + lane) << 5) + __ffs(bits) - 1;
          ids[at] = j;
          if (MODE != 2 && at < ACT_SM) sh_ids[at] = j;
          ++at;
        }
      } else if (total <= p.act_stride && cnt > 0)
#pragma unroll 1
        for (int w0 = wbeg; w0 < wend; w0 += 32 * WU) {
          uint32_t bits[WU];
          int at[WU];
#pragma unroll
          for (int u = 0; u < WU; ++u) {
            bits[u] = w0 + 32 * u + lane < wend ? sh_dd[w0 + 32 * u + lane] : 0u;
            at[u] = __popc(bits[u]);
          }
#pragma unroll
          for (int d = 1; d < 32; d <<= 1)
#pragma unroll
            for (int u = 0; u < WU; ++u) {
              const int n = __shfl_up_sync(FULLM, at[u], d);
              if (lane >= d) at[u] += n;
            }
#pragma unroll
          for (int u = 0; u < WU; ++u) {
            const int all = __shfl_sync(FULLM, at[u], 31);
            at[u] += pos - __popc(bits[u]);
            pos += all;
          }
          while (bits[0] | bits[1] | bits[2] | bits[3]) {
#pragma unroll
            for (int u = 0; u < WU; ++u)
              if (bits[u]) {
                const int j = ((w0 + 32 * u + lane) << 5) + __ffs(bits[u]) - 1;
                ids[at[u]] = j;
                if (MODE != 2 && at[u] < ACT_SM) sh_ids[at[u]] = j;
                ++at[u];
                bits[u] &= bits[u] - 1;
              }
          }
        }
      if (MODE == 2 && p.budget > 0) {                       // the budget reads the mirror
        __syncthreads();
        for (int a = tid; a < min(total, ACT_SM) && total <= p.act_stride; a += FWD_THREADS) sh_ids[a] = ids[a];
      }
      if (MODE == 2 && total <= p.act_stride && p.budget == 0) {
        // The rows of W2 that the batch touches, as a bit per row: the words of the sample's own bitmap, those already marked passed
        // over; blocks begin at different words, so that most of their bits have been marked by others when they come to them
        // (bit by bit from the list of ids it took 30,000 cycles in the first wave of blocks; a step of 256 samples x 325,056 neurons
        // 365 us, by long slices, this and the words above 339).
        marked = true;
        const int nw = (N + 31) >> 5, rounds = (nw + FWD_THREADS - 1) / FWD_THREADS;
        int r = (int)(blockIdx.x % (unsigned)rounds);
        constexpr int TU = 4;
        for (int i = 0; i < rounds; i += TU) {
          uint32_t have[TU], bits[TU];
          int w[TU];
#pragma unroll
          for (int u = 0; u < TU; ++u) {
            w[u] = r * FWD_THREADS + tid;
            bits[u] = i + u < rounds && w[u] < nw ? sh_dd[w[u]] : 0u;
            have[u] = bits[u] ? __ldcg(p.touch2 + w[u]) : 0u;
            if (++r == rounds) r = 0;
          }
#pragma unroll
          for (int u = 0; u < TU; ++u)
            if (bits[u] & ~have[u]) atomicOr(p.touch2 + w[u], bits[u]);
        }
      }
    } else if (ncand + nlab <= RANK_MAX) {
      const int n = ncand + nlab;
      if (packed && tid < 4 && n + tid < ((n + 3) & ~3)) sh_dd[n + tid] = 0xffffffffu;
      __syncthreads();
      uint32_t* srt = sh_dd + RANK_MAX;
      const int per = (n + FWD_THREADS - 1) / FWD_THREADS;
      if (MODE != 2 && packed && n <= FWD_THREADS - 64) {
        // the warps the counting below leaves idle ask L2 for the candidates' rows of W2 meanwhile (the staging after
        // the dedup then finds most of them there); a hint only: duplicates are asked twice, nothing waits for it
        const int idle0 = (n + 31) & ~31;                          // first thread without a value to rank
        const int lines = (H * 4 + 127) >> 7;
        for (int e = tid - idle0; e >= 0 && e < n * (lines + 1); e += FWD_THREADS - idle0) {
          const int c = e / (lines + 1), q = e - c * (lines + 1);
          const int j = (int)(sh_dd[c] >> RANK_BITS);
          prefetch_l2(q < lines ? static_cast<const void*>(p.W2 + (size_t)j * H + 32 * q) : static_cast<const void*>(p.hdr2 + j));
        }
      }
      if (packed) {
        if (per <= 1) rank_sort<1, true>(sh_dd, srt, n);
        else if (per == 2) rank_sort<2, true>(sh_dd, srt, n);
        else rank_sort<RANK_MAX / FWD_THREADS, true>(sh_dd, srt, n);
      } else {
        if (per <= 1) rank_sort<1, false>(sh_dd, srt, n);
        else if (per == 2) rank_sort<2, false>(sh_dd, srt, n);
        else rank_sort<RANK_MAX / FWD_THREADS, false>(sh_dd, srt, n);
      }
      __syncthreads();
      // element i = u * FWD_THREADS + tid of the sorted list is kept when it is the first of its run; its place is
      // the number of kept elements before it: whole rounds and warps (counts exchanged through shared memory) plus
      // the warp's own ballot
      constexpr int PER = RANK_MAX / FWD_THREADS;
      int* sh_cntw = reinterpret_cast<int*>(sh_dh);      // [PER][FWD_WARPS]; the space is not used before the back-propagation
      const unsigned lt = (1u << lane) - 1u;
      const int rounds = (n + FWD_THREADS - 1) / FWD_THREADS;
      unsigned keep[PER];
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        keep[u] = 0u;
        if (u < rounds) {
          const int i = u * FWD_THREADS + tid;
          keep[u] = __ballot_sync(FULLM, i < n && (i == 0 || srt[i - 1] != srt[i]));
          if (lane == 0) sh_cntw[u * FWD_WARPS + warp] = __popc(keep[u]);
        }
      }
      __syncthreads();
      {
        int before = 0;
        for (int q = 0; q < rounds * FWD_WARPS; ++q) {
          const int cq = sh_cntw[q];
          total += cq;
          if (q < warp) before += cq;           // round 0; later rounds add their offset below
        }
        if (total <= p.act_stride) {
          int base = before;
#pragma unroll
          for (int u = 0; u < PER; ++u) {
            if (u < rounds) {
              if (u > 0) {
                base = 0;
                for (int q = 0; q < u * FWD_WARPS + warp; ++q) base += sh_cntw[q];
              }
              const int i = u * FWD_THREADS + tid;
              if ((keep[u] >> lane) & 1u) {
                const int at = base + __popc(keep[u] & lt);
                ids[at] = (int)srt[i];
                if (at < ACT_SM) sh_ids[at] = (int)srt[i];
              }
            }
          }
        }
      }
    } else {
      // sort path: bitonic sort of the candidates, keep the first of each run
      for (int i = ncand + nlab + tid; i < n2; i += FWD_THREADS) sh_dd[i] = 0x7fffffffu;
      __syncthreads();
      for (int k = 2; k <= n2; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
          for (int i = tid; i < n2; i += FWD_THREADS) {
            int x = i ^ j;
            if (x > i) {
              uint32_t a = sh_dd[i], b = sh_dd[x];
              bool asc = (i & k) == 0;
              if ((a > b) == asc) { sh_dd[i] = b; sh_dd[x] = a; }
            }
          }
          __syncthreads();
        }
      const int chunk = (n2 + FWD_THREADS - 1) / FWD_THREADS;
      const int ebeg = tid * chunk, eend = min(n2, ebeg + chunk);
      int cnt = 0;
      for (int i = ebeg; i < eend; ++i) {
        uint32_t a = sh_dd[i];
        cnt += (a != 0x7fffffffu && (i == 0 || sh_dd[i - 1] != a)) ? 1 : 0;
      }
      int pos = block_excl_scan(cnt, sh_misc, &total);
      if (total <= p.act_stride) {
        for (int i = ebeg; i < eend; ++i) {
          uint32_t a = sh_dd[i];
          if (a != 0x7fffffffu && (i == 0 || sh_dd[i - 1] != a)) {
            ids[pos] = (int)a;
            if (pos < ACT_SM) sh_ids[pos] = (int)a;
            ++pos;
          }
        }
      }
    }
    if (total > p.act_stride) {      // uniform over the block
      skip_sample<MODE>(p, s, DSLIDE_ERR_OVERFLOW);
      return;
    }
    na = total;
    __syncthreads();                 // ids visible to the block; the dedup work space is free from here on
    if (p.budget > 0)
      na = budget_select(p.budget, p.budget_fill, N, p.seed, p.tcount, s, ids, sh_ids, na, MODE != 1 ? p.labels + lbeg : nullptr,
                         nlab, smem + p.off_dedup, p.stage_bytes, sh_misc, p.st);
  }
  if (MODE != 1 && tid == 0) p.act_cnt[s] = na;
  if (MODE == 2) {
    // ---- the rows of W2 that the batch touches (most are marked already: a read is enough), unless the bitmap has told, and
    //      the hand-off of the sample's rows of W1 ----
    constexpr int TU = 4;
    for (int a0 = tid; a0 < na && !marked; a0 += TU * FWD_THREADS) {
      int j[TU];
      uint32_t have[TU];
#pragma unroll
      for (int u = 0; u < TU; ++u) j[u] = a0 + u * FWD_THREADS < na ? ids[a0 + u * FWD_THREADS] : -1;
#pragma unroll
      for (int u = 0; u < TU; ++u) have[u] = j[u] >= 0 ? __ldcg(p.touch2 + (j[u] >> 5)) : 0xffffffffu;
#pragma unroll
      for (int u = 0; u < TU; ++u)
        if (j[u] >= 0 && !((have[u] >> (j[u] & 31)) & 1u)) atomicOr(p.touch2 + (j[u] >> 5), 1u << (j[u] & 31));
    }
    if (p.L1 > 0)
      for (int i = tid; i < nnz; i += FWD_THREADS) {
        const int c = __ldg(p.col_idx + rbeg + i);
        for (int w = 0; w < p.Hw; ++w)
          if (sh_hmask[w]) atomicOr(&p.cmask1[(size_t)c * p.Hw + w], sh_hmask[w]);
      }
    for (int i0 = 0; i0 < nnz; i0 += FWD_THREADS) touch_w1(p, i0 + tid < nnz, rbeg + i0 + tid, s);
    if (tid == 0) {
      atomicAdd(&p.st->acc[p.parity][0], (unsigned long long)na);
      atomicAdd(&p.st->acc[p.parity][1], (unsigned long long)nnz);
      atomicAdd(&p.st->acc[p.parity][2], (unsigned long long)sh_misc[24]);
    }
    return;
  }
  const bool small = !dense && na <= ACT_SM;      // ids and logits mirrored in shared memory
  // one pointer per array, to shared or to global memory (a conditional expression over two loads would issue both)
  const int* idp = small ? sh_ids : ids;
  const float* zp = small ? sh_z : p.act_z + (size_t)s * p.act_stride;
  const float* gp = small ? sh_g : p.act_g + (size_t)s * p.act_stride;

  // ---- positions of the sample's distinct labels inside the active set (needed while the rows are staged) ----
  if (MODE == 0) {
    for (int i = tid; i < nlab; i += FWD_THREADS) {
      int y = p.labels[lbeg + i];
      bool first = true;
      for (int q = 0; q < i; ++q) first = first && (p.labels[lbeg + q] != y);
      int pos = y;
      if (!dense) {
        int lo = 0, hi = na;
        while (lo < hi) { int mid = (lo + hi) >> 1; if (idp[mid] < y) lo = mid + 1; else hi = mid; }
        pos = lo;
      }
      sh_lab[i] = first ? pos : -1;
    }
    __syncthreads();
    if (tid == 0) {
      int ny = 0;
      for (int i = 0; i < nlab; ++i) ny += sh_lab[i] >= 0 ? 1 : 0;
      sh_misc[8] = ny;
    }
  }

  float* z = p.act_z + (size_t)s * p.act_stride;
  unsigned long long mine = 0ull;                  // predict: the thread's best score
  const bool keep_z = MODE == 0 || (!small && p.topk > 1);
  // hand-off to the update kernel: the touch counters of the sample's rows of W1 (one per thread) and of HO_PER of its active
  // rows per thread (act0: which) are asked while the first rows of W2 are on their way, the list places after the
  // first logits, and everything is written at the end -- no warp waits for an answer
  constexpr int HO_PER = 2;
  int jj0[HO_PER], act0[HO_PER], ho_rows = HO_PER * FWD_THREADS;
  unsigned nth1 = 0u, nth0[HO_PER], base1 = 0u, base0[HO_PER];
#pragma unroll
  for (int u = 0; u < HO_PER; ++u) { jj0[u] = 0; act0[u] = -1; nth0[u] = 0u; base0[u] = 0u; }
  if constexpr (NP == 1) {
  // ---- logits over the active set.  The active rows of W2 are copied into shared memory, as many as fit at a
  //      time.  When the whole set fits, the rows stay there for the back-propagation below.  When it does not, the
  //      back-propagated error is accumulated in the same pass, chunk by chunk, with a running maximum M and sums
  //      rescaled whenever M grows: S = sum_a exp(z_a - M) W2[j_a,:], E = sum_a exp(z_a - M), and T = the sum of the
  //      label rows; then dh = (S / E - T / |Y|) / B, and every row is fetched once. ----
  const float4* sh_h4 = reinterpret_cast<const float4*>(sh_h);
  const int ldr = H + 4;                           // staged rows are padded by 16 bytes: a thread per row reads without bank conflicts
  const int stage_rows = p.stage_bytes / (ldr * 4 + 4);      // a row and one float of the chunk's exp(z - M)
  float* sh_ce = stage + (size_t)stage_rows * ldr;           // [stage_rows]
  const bool streaming = MODE == 0 && na > stage_rows;
  float Mrun = -INFINITY, Erun = 0.f;
  // The sums of a warp's rows of a chunk, or of all that is staged: a lane holds four consecutive units of every 128, and of up to 64
  // units 8 or 16 lanes have a row each.  (A thread per unit, with rows shared out to groups of threads, read four times as
  // often: 64 samples of SimHash sets of 400 rows x 128 units, a step 68.8 us, so 67.5; the 670,091-neuron shape, whose sets are
  // one chunk or a little more, 64.5 and 63.1.)
  constexpr int NCH = 2;                           // H <= 128 * NCH
  float4 av[NCH];
#pragma unroll
  for (int q = 0; q < NCH; ++q) av[q] = make_float4(0.f, 0.f, 0.f, 0.f);
  const int rl = H4 <= 8 ? 8 : H4 <= 16 ? 16 : 32, lg_rl = H4 <= 8 ? 3 : H4 <= 16 ? 4 : 5;      // lanes of a row
  auto add_rows = [&](const float* coef, int n) {
#pragma unroll 4
    for (int a = (tid >> lg_rl); a < n; a += FWD_THREADS >> lg_rl) {
      const float ga = coef[a];
      const float4* row = reinterpret_cast<const float4*>(stage + (size_t)a * ldr);
#pragma unroll
      for (int q = 0; q < NCH; ++q) {
        const int c = (lane & (rl - 1)) + 32 * q;
        if (c < H4) {
          const float4 w = row[c];
          av[q].x = fmaf(ga, w.x, av[q].x); av[q].y = fmaf(ga, w.y, av[q].y);
          av[q].z = fmaf(ga, w.z, av[q].z); av[q].w = fmaf(ga, w.w, av[q].w);
        }
      }
    }
  };
  // a thread's place in the copy pattern of the padded rows: H4 + 1 pieces per row
  const int rp_dr = FWD_THREADS / (H4 + 1), rp_dc = FWD_THREADS - rp_dr * (H4 + 1);
  const int rp_r0 = tid / (H4 + 1), rp_c0 = tid - rp_r0 * (H4 + 1);
  bool timed_out = false;                          // block-uniform
  const bool bulk = BULK && streaming && na >= 4 * stage_rows;      // many chunks: the batch's samples share most rows (see below)
  // (a training sample with nothing active still goes through once: its rows of W1 are counted in here)
  for (int c0 = 0; c0 < na || (MODE == 0 && c0 == 0); c0 += stage_rows) {
    const int nr = min(stage_rows, na - c0);
    __syncthreads();                               // earlier readers and writers of the staging space are done
    if (bulk) {
      // A set streamed in many chunks re-reads rows that other samples of the batch have brought into L2; there the
      // bulk-copy engine moves about twice what 16-byte copies do per multiprocessor: one copy per row and one for
      // the head of its record (count, bias, bias moments), which lands in the row's padding; completion on an mbarrier
      if (tid == 0) mbar_expect_tx(sh_bar, (uint32_t)nr * ((uint32_t)H * 4u + 16u));
      fence_proxy_async();
      for (int r = tid; r < nr; r += FWD_THREADS) {
        const int j = dense ? c0 + r : idp[c0 + r];
        bulk_g2s(stage + (size_t)r * ldr, p.W2 + (size_t)j * H, (uint32_t)H * 4u, sh_bar);
        bulk_g2s(stage + (size_t)r * ldr + H, p.hdr2 + j, 16u, sh_bar);
      }
    } else {
      // 16 bytes per thread and copy, all in flight at once: the H4 pieces of the row, and as piece H4 the head of
      // the row's record, which lands in the row's padding
      for (int r = rp_r0, c4 = rp_c0; r < nr;) {
        const int j = dense ? c0 + r : idp[c0 + r];
        const void* src = c4 < H4 ? static_cast<const void*>(p.W2 + (size_t)j * H + 4 * c4) : static_cast<const void*>(p.hdr2 + j);
        cp_async16(stage + (size_t)r * ldr + 4 * c4, src);
        c4 += rp_dc; r += rp_dr;
        if (c4 > H4) { c4 -= H4 + 1; ++r; }
      }
    }
    if (c0 == 0 && MODE == 0) {
      // the touch counters: this thread's nonzero of the sample, and its first HO_PER active rows
      if (tid < nnz) {
        if (tid >= R) {                              // beyond the first chunk: not kept in registers above
          c1 = __ldg(p.col_idx + rbeg + tid);
          x1 = __ldg(p.vals + rbeg + tid);
          line1 = __ldcg(p.hotmap1 + c1);
        }
        nth1 = atomicAdd(&p.hdr1[c1].cnt, 1u) & CNT_MASK;
        if (line1 >= 0) p.hotcoef1[(size_t)line1 * p.bstride + s] = x1;
      }
      if (!dense) {
#pragma unroll
        for (int u = 0; u < HO_PER; ++u) {
          const int a = tid + u * FWD_THREADS;
          if (a < na) {
            jj0[u] = idp[a];
            act0[u] = a;
            nth0[u] = atomicAdd(&p.hdr2[jj0[u]].cnt, 1u) & CNT_MASK;
          }
        }
      }
    }
    if (bulk) {
      const bool ok = bar_wait_limited(sh_bar, w2phase);
      w2phase ^= 1u;
      if (__syncthreads_or(ok ? 0 : 1)) { timed_out = true; break; }
    } else {
      cp_async_wait_all();
      __syncthreads();
    }
    // one thread per staged row
    for (int ab = 0; ab < nr; ab += FWD_THREADS) {
      const int a = ab + tid;
      const bool live = a < nr;
      float dot = 0.f;
      if (live) {
        const float4* row = reinterpret_cast<const float4*>(stage + (size_t)a * ldr);
        float d0 = 0.f, d1 = 0.f, d2 = 0.f, d3 = 0.f;
#pragma unroll 4
        for (int c = 0; c < H4; ++c) {
          const float4 w = row[c], x = sh_h4[c];
          d0 = fmaf(w.x, x.x, d0);
          d1 = fmaf(w.y, x.y, d1);
          d2 = fmaf(w.z, x.z, d2);
          d3 = fmaf(w.w, x.w, d3);
        }
        dot = (d0 + d1) + (d2 + d3);
      }
      if (live) {
        const float zv = stage[(size_t)a * ldr + H + 1] + dot;      // the bias came with the row
        if (small) sh_z[c0 + a] = zv;
        if (keep_z) z[c0 + a] = zv;
        if (streaming) sh_ce[a] = zv;
        if (MODE == 1) mine = max(mine, place_of(zv, c0 + a));
      }
    }
    if (MODE == 0 && c0 == 0) {
      // the touch counters have answered by now.  W1 side: slot / mask entries (the coefficient is the input value);
      // both sides: places in the lists of distinct rows asked for, used at the end of the kernel
      touch_mark<false>(p, tid < nnz, p.hdr1 + c1, p.mask1 + (size_t)c1 * p.Wd, p.ovf1 + (size_t)c1 * PAIR_T, ~c1, nth1, s, x1);
      base1 = own_reserve(tid < nnz && nth1 == 0u, &p.st->n_own[p.parity][1]);
      if (!dense) {
#pragma unroll
        for (int u = 0; u < HO_PER; ++u)
          if (u * FWD_THREADS < na)          // uniform over the block
            base0[u] = own_reserve(tid + u * FWD_THREADS < na && nth0[u] == 0u, &p.st->n_own[p.parity][0]);
      }
    }
    if (streaming) {
      __syncthreads();
      float cm = -INFINITY;
      for (int a = tid; a < nr; a += FWD_THREADS) cm = fmaxf(cm, sh_ce[a]);
      const float Mnew = fmaxf(Mrun, block_max(cm, sh_red));
      const float base = Mnew > -INFINITY ? Mnew : 0.f; // masked neurons only so far (biases of minus infinity): they weigh nothing
      const float scale = expf(Mrun - base);            // 0 for the first chunk
      float es = 0.f;
      for (int a = tid; a < nr; a += FWD_THREADS) {
        const float ea = expf(sh_ce[a] - base);
        sh_ce[a] = ea;
        es += ea;
      }
      Erun = Erun * scale + block_sum(es, sh_red);      // its barriers make the chunk's exp values visible
      Mrun = Mnew;
#pragma unroll
      for (int q = 0; q < NCH; ++q) { av[q].x *= scale; av[q].y *= scale; av[q].z *= scale; av[q].w *= scale; }
      add_rows(sh_ce, nr);
    }
  }
  if (BULK && timed_out) {
    // a copy did not complete in time: the copies in flight get one more bounded wait, then the sample is given up.
    // Its touches are already counted, so the hand-off below still runs, with every coefficient zero.
    bar_wait_limited(sh_bar, w2phase ^ 1u);
    __syncthreads();
    if (tid == 0) set_status(p.st, DSLIDE_ERR_TIMEOUT);
  }
  if (MODE == 1) {
    unsigned long long* work = reinterpret_cast<unsigned long long*>(smem + p.off_topk);
    best_of(p.out_ids + (size_t)s * p.topk, p.out_scores + (size_t)s * p.topk, p.topk, dense ? nullptr : idp, zp, na, mine, work,
            sh_misc);
    return;
  }
  __syncthreads();           // logits visible to the block

  // ---- softmax over the ragged active set, loss, errors.  A small set's logits sit in shared memory: every warp
  //      takes the maximum and the sum over all of them by itself (same order, same result in every warp), which
  //      spares the block-wide reductions and their barriers ----
  float* pr = p.act_p + (size_t)s * p.act_stride;
  float* g = p.act_g + (size_t)s * p.act_stride;
  float M = Mrun, E = Erun;                        // known already when the rows were streamed
  if (!streaming) {
    if (small) {
      float m = -INFINITY;
#pragma unroll 4
      for (int a = lane; a < na; a += 32) m = fmaxf(m, sh_z[a]);
      M = warp_max(m);
      float e = 0.f;
#pragma unroll 4
      for (int a = lane; a < na; a += 32) e += expf(sh_z[a] - M);
      E = warp_sum(e);
    } else {
      float m = -INFINITY;
      for (int a = tid; a < na; a += FWD_THREADS) m = fmaxf(m, zp[a]);
      M = block_max(m, sh_red);
      float e = 0.f;
      for (int a = tid; a < na; a += FWD_THREADS) e += expf(zp[a] - M);
      E = block_sum(e, sh_red);
    }
  }
  const float fB = (float)p.B;
  const int ny = sh_misc[8];
  if (tid == FWD_THREADS - 1) {                    // the last thread has the fewest rows below
    float sum = 0.f;
    const float logE = logf(E);
    for (int i = 0; i < nlab; ++i)
      if (sh_lab[i] >= 0) sum += zp[sh_lab[i]] - M - logE;
    p.loss[s] = ny > 0 && !(BULK && timed_out) ? -sum / (float)ny : 0.f;
  }
  // the errors of a small set go to shared memory as well (beside the logits: no barrier before they are written)
  for (int a = tid; a < na; a += FWD_THREADS) {
    const float pa = expf(zp[a] - M) / E;
    pr[a] = pa;
    float ga = pa / fB;
    for (int i = 0; i < nlab; ++i)
      if (sh_lab[i] == a) ga = (pa - 1.f / (float)ny) / fB;
    if (BULK && timed_out) ga = 0.f;
    g[a] = ga;
    if (small) sh_g[a] = ga;
  }
  __syncthreads();

  // ---- error at the hidden layer: dh = [h > 0] * sum_a g_a W2[j_a, :] (weights before the update).  Every warp has
  //      its staged rows; the warps' sums are then added in warp order.  When the rows were streamed the sums
  //      exist already ----
  {
    if (!streaming) add_rows(gp, na);
    for (int o = rl; o < 32; o <<= 1) {            // the rows side by side
      av[0].x += __shfl_xor_sync(FULLM, av[0].x, o); av[0].y += __shfl_xor_sync(FULLM, av[0].y, o);
      av[0].z += __shfl_xor_sync(FULLM, av[0].z, o); av[0].w += __shfl_xor_sync(FULLM, av[0].w, o);
    }
#pragma unroll
    for (int q = 0; q < NCH; ++q) {
      const int c = lane + 32 * q;
      if (c < H4) reinterpret_cast<float4*>(sh_dh + (size_t)warp * H)[c] = av[q];
    }
    __syncthreads();
    for (int k = tid; k < H; k += FWD_THREADS) {
      float y[FWD_WARPS];
#pragma unroll
      for (int w = 0; w < FWD_WARPS; ++w) y[w] = sh_dh[(size_t)w * H + k];
      float v = ((y[0] + y[1]) + (y[2] + y[3])) + ((y[4] + y[5]) + (y[6] + y[7]));      // in pairs, so that no sum is long
      if (streaming) {                             // (the label rows are in L2)
        float T = 0.f;
        for (int i = 0; i < nlab; ++i)
          if (sh_lab[i] >= 0) T += p.W2[(size_t)(dense ? sh_lab[i] : idp[sh_lab[i]]) * H + k];
        v = (v / E - (ny > 0 ? T / (float)ny : 0.f)) / fB;
      }
      p.dh[(size_t)s * H + k] = sh_h[k] > 0.f && !(BULK && timed_out) ? v : 0.f;
    }
  }
  } else {
  // ---- one pass over the active rows of W2: logits and, with a running maximum M, the sums S = sum_a exp(z_a - M) W2[j_a,:]
  //      and E = sum_a exp(z_a - M); then dh = (S / E - T / |Y|) / B with T the sum of the label rows.  Warp w takes the groups
  //      w, w + 8, ... of ROWS rows through its own ring in shared memory: a bulk copy per row, completion on an mbarrier per
  //      group; the groups ahead are in flight while a group is read, once, for both sums.  No warp waits for another, and
  //      whatever the set's size the rings are full until its end.  Bound by the instructions of a warp (about 400 a group at
  //      four cycles), by what a multiprocessor keeps in flight (2 x 90 KB) for few rows.  In chunks of the whole space, with
  //      barriers around each and a thread per staged row, logits and copies took 57,000 cycles of a block's 96,000 at 512 units and
  //      160 rows.  At up to 128 units that is the better way still: a thread per row takes a fortieth of the instructions
  //      for a logit, and most sets are one chunk (256 x 670,091 x 128: a step 64.1 us, by rings 64.9; 32 x 2,000 x 32: 31.1 and 39.8) ----
  float M = -INFINITY, E = 0.f;
  float accT[KPT];
#pragma unroll
  for (int u = 0; u < KPT; ++u) accT[u] = 0.f;
  {
    constexpr int R = RowPass<NP>::ROWS, Q = 32 / R;         // rows of a group; lanes that end with the same row's sum
    const int row_b = H * 4, nw = min(FWD_WARPS, (p.stage_bytes - RING_HEAD) / (R * row_b));      // warps that have a ring (all but in tight layouts)
    const int depth = min(RING_DEPTH, (p.stage_bytes - RING_HEAD) / nw / (R * row_b));            // groups of a ring
    uint64_t* bars = reinterpret_cast<uint64_t*>(stage) + warp * RING_DEPTH;
    float* zeros = stage + RING_HEAD / 4 - 4;
    float* ring = stage + RING_HEAD / 4 + (size_t)warp * depth * R * H;
    const int ngroups = (na + R - 1) / R, mygroups = warp < nw && warp < ngroups ? (ngroups - warp + nw - 1) / nw : 0;
    fence_proxy_async();
    __syncthreads();                               // the readers of the space before this are done
    if (lane < RING_DEPTH) mbar_init(bars + lane, 1);
    if (tid == 0) { zeros[0] = zeros[1] = zeros[2] = zeros[3] = 0.f; sh_misc[9] = 0; }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_proxy_async();
    __syncthreads();
    // Rows of the warp, 32 at a time: lane l has row l % R of group l / R -- its id, its bias and, of the first two rounds, the
    // touch counter's answer
    auto row_of = [&](int l) { const int a = (warp + (l / R) * nw) * R + l % R; return l / R < mygroups && a < na ? a : -1; };
    auto id_of = [&](int a) { return a < 0 ? 0 : (dense ? a : idp[a]); };
    int ac = row_of(lane), idc = id_of(ac), an = row_of(32 + lane), idn = id_of(an);
    float bc = ac < 0 ? 0.f : p.hdr2[idc].b, bn = 0.f;      // of the batch that is summed; of the one that is asked for
    int gi = 0, gslot = 0;                                   // group to ask for, and its place in the ring
    static_assert(HO_PER == 2, "the counters of a warp's first 64 rows");
    auto count_in = [&](int u) {                             // training: the touch counters of the rows
      if (MODE != 0 || dense || u >= HO_PER) return;
      const unsigned nth = ac >= 0 ? atomicAdd(&p.hdr2[idc].cnt, 1u) & CNT_MASK : 0u;
      if (u == 0) { act0[0] = ac; jj0[0] = idc; nth0[0] = nth; }
      else { act0[1] = ac; jj0[1] = idc; nth0[1] = nth; }
    };
    auto ask = [&]() {
      if (gi < mygroups) {
        const int l0 = (gi * R) & 31, l = lane - l0, m = min(R, na - (warp + gi * nw) * R);
        if (l0 == 0 && gi > 0) {                             // the next 32 rows
          ac = an; idc = idn;
          bn = ac < 0 ? 0.f : p.hdr2[idc].b;
          count_in(gi * R / 32);
          an = row_of(gi * R + 32 + lane);
          idn = id_of(an);
        }
        if (lane == 0) mbar_expect_tx(bars + gslot, (uint32_t)(m * row_b));
        __syncwarp();
        if (l >= 0 && l < m) bulk_g2s(ring + (gslot * R + l) * H, p.W2 + (size_t)idc * H, (uint32_t)row_b, bars + gslot);
        ++gi;
        gslot = gslot + 1 == depth ? 0 : gslot + 1;
      }
    };
    for (int i = 0; i < depth - 1; ++i) ask();
    if (MODE == 0) {
      // the touch counter of this thread's nonzero of the sample
      if (tid < nnz) {
        if (tid >= p.hid_rows) {                     // beyond the first chunk: not kept in registers above
          c1 = __ldg(p.col_idx + rbeg + tid);
          x1 = __ldg(p.vals + rbeg + tid);
          line1 = __ldcg(p.hotmap1 + c1);
        }
        nth1 = atomicAdd(&p.hdr1[c1].cnt, 1u) & CNT_MASK;
        if (line1 >= 0) p.hotcoef1[(size_t)line1 * p.bstride + s] = x1;
      }
      count_in(0);
      ho_rows = HO_PER * 32 * nw;
    }
    constexpr bool HREG = NP <= 4;                 // the sample's activations in registers, else read again for every row
    constexpr int SURE = NP / 2;                   // pieces that every lane has; past the row's end it reads zeros (not a piece of the
    ulonglong2 hx[HREG ? NP : 1], S[NP];           // row: a weight of minus infinity times an activation of zero is no number)
    const ulonglong2* sh_h2 = reinterpret_cast<const ulonglong2*>(sh_h);
    const float* base[NP - SURE];
    int mul[NP - SURE];
#pragma unroll
    for (int u = 0; u < NP; ++u) {
      const bool in = lane + 32 * u < H4;
      if (HREG) hx[HREG ? u : 0] = in ? sh_h2[lane + 32 * u] : make_ulonglong2(0ull, 0ull);
      S[u] = make_ulonglong2(0ull, 0ull);            // pairs of floats: two multiply-adds per instruction
      if (u >= SURE) {
        base[u < SURE ? 0 : u - SURE] = in ? ring + 4 * (lane + 32 * u) : zeros;
        mul[u < SURE ? 0 : u - SURE] = in ? H : 0;
      }
    }
    int slot = 0;
    uint32_t phase = 0u;
#pragma unroll 1
    for (int i = 0; i < mygroups; ++i) {
      ask();
      if (!bar_wait_limited_warp(bars + slot, phase)) {
        if (lane == 0) sh_misc[9] = 1;
        for (int q = i; q < gi; ++q) {             // what is still in flight gets one more bounded wait
          bar_wait_limited(bars + slot, phase);
          if (++slot == depth) { slot = 0; phase ^= 1u; }
        }
        break;
      }
      const int a0 = (warp + i * nw) * R, m = min(R, na - a0), at0 = slot * R, l0 = (i * R) & 31;
      if (++slot == depth) { slot = 0; phase ^= 1u; }
      if (l0 == 0 && i > 0) bc = bn;
      ulonglong2 x[R][NP];
      float d[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        unsigned long long d0 = 0ull, d1 = 0ull;
        if (r < m) {
#pragma unroll
          for (int u = 0; u < NP; ++u) {
            x[r][u] = *reinterpret_cast<const ulonglong2*>(u < SURE ? ring + (at0 + r) * H + 4 * (lane + 32 * u)
                                                                    : base[u < SURE ? 0 : u - SURE] + (at0 + r) * mul[u < SURE ? 0 : u - SURE]);
            const ulonglong2 hv = HREG ? hx[HREG ? u : 0] : *(u < SURE || lane + 32 * u < H4 ? sh_h2 + lane + 32 * u : reinterpret_cast<const ulonglong2*>(zeros));
            fma2(d0, x[r][u].x, hv.x);
            fma2(d1, x[r][u].y, hv.y);
          }
        }
        d[r] = (lo2(d0) + hi2(d0)) + (lo2(d1) + hi2(d1));
      }
      // every exchange halves the rows a lane has part of
#pragma unroll
      for (int n2 = R / 2, o = 16; n2 > 0; n2 >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int r = 0; r < n2; ++r) d[r] = (up ? d[r + n2] : d[r]) + __shfl_xor_sync(FULLM, up ? d[r] : d[r + n2], o);
      }
      float y = d[0];
#pragma unroll
      for (int o = Q / 2; o > 0; o >>= 1) y += __shfl_xor_sync(FULLM, y, o);
      const int q = lane / Q, at = a0 + q;         // the row whose sum this lane has
      const float bias = __shfl_sync(FULLM, bc, l0 + q);
      const float zv = q < m ? bias + y : -INFINITY;
      if (q < m && (lane & (Q - 1)) == (i & (Q - 1))) {      // a lane of the row's, in turn (predict: the threads' maxima)
        if (small) sh_z[at] = zv;
        if (keep_z) z[at] = zv;
        if (MODE == 1) mine = max(mine, place_of(zv, at));
      }
      if (MODE == 0) {
        if (__any_sync(FULLM, zv > M)) {
          float zm = fmaxf(zv, M);
#pragma unroll
          for (int o = Q; o < 32; o <<= 1) zm = fmaxf(zm, __shfl_xor_sync(FULLM, zm, o));
          const float scale = expf(M - zm);
          const unsigned long long sc = pair2(scale, scale);
          M = zm;
          E *= scale;
#pragma unroll
          for (int u = 0; u < NP; ++u) {
            mul2(S[u].x, sc);
            mul2(S[u].y, sc);
          }
        }
        // a masked neuron (bias of minus infinity) weighs nothing, also while nothing else has been met and M is minus infinity
        const float e = zv != -INFINITY ? expf(zv - M) : 0.f;
        E += e;                                    // this lane's rows only, until the end
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const float g = __shfl_sync(FULLM, e, Q * r);
          const unsigned long long gg = pair2(g, g);
          if (r < m) {
#pragma unroll
            for (int u = 0; u < NP; ++u) {
              fma2(S[u].x, gg, x[r][u].x);
              fma2(S[u].y, gg, x[r][u].y);
            }
          }
        }
      }
      __syncwarp();                                // the rows have been read: their places may be filled again
    }
    if (MODE == 0) {
#pragma unroll
      for (int o = Q; o < 32; o <<= 1) E += __shfl_xor_sync(FULLM, E, o);      // lanes hold different rows
#pragma unroll
      for (int u = 0; u < NP; ++u)
        if (lane + 32 * u < H4) reinterpret_cast<ulonglong2*>(sh_dh + (size_t)warp * H)[lane + 32 * u] = S[u];
      if (lane == 0) { sh_misc[warp] = __float_as_int(M); sh_red[warp] = E; }
    }
  }
  if (MODE == 1) {
    __syncthreads();
    if (sh_misc[9] != 0) {                         // a copy did not complete in time
      skip_sample<MODE>(p, s, DSLIDE_ERR_TIMEOUT);
      return;
    }
    unsigned long long* work = reinterpret_cast<unsigned long long*>(smem + p.off_topk);
    best_of(p.out_ids + (size_t)s * p.topk, p.out_scores + (size_t)s * p.topk, p.topk, dense ? nullptr : idp, zp, na, mine, work,
            sh_misc);
    return;
  }
  // the label rows (they are in L2 by now)
  for (int i = 0; i < nlab; ++i)
    if (sh_lab[i] >= 0) {
      const float* row = p.W2 + (size_t)p.labels[lbeg + i] * H;
#pragma unroll
      for (int u = 0; u < KPT; ++u)
        if (tid + u * FWD_THREADS < H) accT[u] += row[tid + u * FWD_THREADS];
    }
  // the touch counters have answered by now.  W1 side: slot / mask entries (the coefficient is the input value);
  // both sides: places in the lists of distinct rows asked for, used at the end of the kernel
  touch_mark<false>(p, tid < nnz, p.hdr1 + c1, p.mask1 + (size_t)c1 * p.Wd, p.ovf1 + (size_t)c1 * PAIR_T, ~c1, nth1, s, x1);
  base1 = own_reserve(tid < nnz && nth1 == 0u, &p.st->n_own[p.parity][1]);
#pragma unroll
  for (int u = 0; u < HO_PER; ++u) base0[u] = own_reserve(act0[u] >= 0 && nth0[u] == 0u, &p.st->n_own[p.parity][0]);
  __syncthreads();           // logits and the warps' sums visible to the block
  // A copy did not complete in time: the sample is given up.  Its touches are already counted, so the hand-off below still
  // runs, with every coefficient zero.
  const bool timed_out = sh_misc[9] != 0;
  if (timed_out && tid == 0) set_status(p.st, DSLIDE_ERR_TIMEOUT);

  // ---- the warps' maxima and sums put together; loss, errors, error at the hidden layer ----
  float* pr = p.act_p + (size_t)s * p.act_stride;
  float* g = p.act_g + (size_t)s * p.act_stride;
  float fac[FWD_WARPS];
  M = __int_as_float(sh_misc[0]);
#pragma unroll
  for (int w = 1; w < FWD_WARPS; ++w) M = fmaxf(M, __int_as_float(sh_misc[w]));
#pragma unroll
  for (int w = 0; w < FWD_WARPS; ++w) fac[w] = sh_red[w] == 0.f ? 0.f : expf(__int_as_float(sh_misc[w]) - M);
  // (in pairs, so that no sum is long)
  auto of_warps = [&](const float* x, int stride) {
    float y[FWD_WARPS / 2];
#pragma unroll
    for (int w = 0; w < FWD_WARPS / 2; ++w) y[w] = fmaf(fac[2 * w], x[(size_t)(2 * w) * stride], fac[2 * w + 1] * x[(size_t)(2 * w + 1) * stride]);
    return (y[0] + y[1]) + (y[2] + y[3]);
  };
  E = of_warps(sh_red, 1);
  const float fB = (float)p.B;
  const int ny = sh_misc[8];
#pragma unroll
  for (int u = 0; u < KPT; ++u) {
    const int k = tid + u * FWD_THREADS;
    if (k < H) {
      float v = of_warps(sh_dh + k, H);
      v = na > 0 ? (v / E - (ny > 0 ? accT[u] / (float)ny : 0.f)) / fB : 0.f;
      p.dh[(size_t)s * H + k] = sh_h[k] > 0.f && !timed_out ? v : 0.f;
    }
  }
  if (tid == FWD_THREADS - 1) {                    // the last thread has the fewest rows below
    float sum = 0.f;
    const float logE = logf(E);
    for (int i = 0; i < nlab; ++i)
      if (sh_lab[i] >= 0) sum += zp[sh_lab[i]] - M - logE;
    p.loss[s] = ny > 0 && !timed_out ? -sum / (float)ny : 0.f;
  }
  // the errors of a small set go to shared memory as well (beside the logits: no barrier before they are written)
  for (int a = tid; a < na; a += FWD_THREADS) {
    const float pa = expf(zp[a] - M) / E;
    pr[a] = pa;
    float ga = pa / fB;
    for (int i = 0; i < nlab; ++i)
      if (sh_lab[i] == a) ga = (pa - 1.f / (float)ny) / fB;
    if (timed_out) ga = 0.f;
    g[a] = ga;
    if (small) sh_g[a] = ga;
  }
  __syncthreads();
  }

  // ---- the rest of the hand-off: slot / mask entries of the rows of W2 (their coefficient is the error), the
  //      entries of both lists of distinct rows, and whatever did not fit the registers above ----
  own_store(tid < nnz && nth1 == 0u, base1, p.own1, c1, s);
  if (tid < nnz) list_row(p, &p.hdr1[c1].cnt, ~c1, nth1);
  if (p.L1 > 0)          // sampled hidden layer: of the rows of W1 the sample touches, only its active neurons' weights
    for (int i = tid; i < nnz; i += FWD_THREADS) {
      const int c = i == tid ? c1 : __ldg(p.col_idx + rbeg + i);
      for (int w = 0; w < p.Hw; ++w)
        if (sh_hmask[w]) atomicOr(&p.cmask1[(size_t)c * p.Hw + w], sh_hmask[w]);
    }
  for (int i0 = FWD_THREADS; i0 < nnz; i0 += FWD_THREADS) touch_w1(p, i0 + tid < nnz, rbeg + i0 + tid, s);
  if (!dense) {
#pragma unroll
    for (int u = 0; u < HO_PER; ++u)
      if (u * (ho_rows / HO_PER) < na) {   // uniform over the block; the rows counted in above, of fewer rings than warps not one per thread
        const int a = act0[u];
        const bool live = a >= 0;
        touch_mark(p, live, p.hdr2 + jj0[u], p.mask2 + (size_t)jj0[u] * p.Wd, p.ovf2 + (size_t)jj0[u] * PAIR_T, jj0[u], nth0[u], s,
                   live ? gp[a] : 0.f);
        own_store(live && nth0[u] == 0u, base0[u], p.own2, jj0[u], s);
      }
    for (int a0 = ho_rows; a0 < na; a0 += FWD_THREADS) {
      const int a = a0 + tid;
      const bool live = a < na;
      int jj = 0;
      unsigned nth = 0u;
      float ga = 0.f;
      if (live) {
        jj = idp[a];
        ga = gp[a];
        nth = atomicAdd(&p.hdr2[jj].cnt, 1u) & CNT_MASK;
      }
      finish_touch(p, live, p.hdr2 + jj, p.mask2 + (size_t)jj * p.Wd, p.ovf2 + (size_t)jj * PAIR_T, p.own2, &p.st->n_own[p.parity][0], jj, jj, nth, s, ga);
    }
  }
  if (tid == 0) {
    atomicAdd(&p.st->acc[p.parity][0], (unsigned long long)na);
    atomicAdd(&p.st->acc[p.parity][1], (unsigned long long)nnz);
    atomicAdd(&p.st->acc[p.parity][2], (unsigned long long)sh_misc[24]);
  }
}


// ---------------------------------------------------------------------------
// Host side: shared-memory layout and launches
// ---------------------------------------------------------------------------
static int align16(int x) { return (x + 15) & ~15; }
static int align128(int x) { return (x + 127) & ~127; }

constexpr int TWO_PER_SM = (227 * 1024) / 2 - 1024;      // shared memory of a block of which two are resident

struct FwdLayout {
  int off_dh, off_code, off_part, off_misc, off_lab, off_tbase, off_tbeg, off_topk, off_ids, off_z, off_col, off_val,
      off_h1, off_dedup, fixed_bytes, hid_rows;
};

static FwdLayout fwd_layout(const Ctx* c) {
  FwdLayout l;
  // rows of W1 staged per chunk of the hidden layer: HID_MIN_BYTES worth, between 8 and 128
  int hid_rows = HID_MIN_BYTES / (c->H * 4);
  if (hid_rows > 128) hid_rows = 128;
  if (hid_rows < 8) hid_rows = 8;
  // wide hidden layers: two rows less rather than one block per multiprocessor less
  const int around = align16(c->H * 4) * (1 + FWD_WARPS) + c->L * 12 + 2 * c->KL + c->cfg.max_labels * 4 + FWD_WARPS * 64 * 8 + 2 * ACT_SM * 4 + 2048;
  while (hid_rows > 8 && around + hid_rows * (c->H * 4 + 8) > TWO_PER_SM) --hid_rows;
  l.hid_rows = hid_rows;
  int o = align16(c->H * 4);
  l.off_dh = o;      o = align16(o + FWD_WARPS * c->H * 4);
  l.off_code = o;    o = align16(o + c->L * 4);
  l.off_part = o;    o = align16(o + 2 * c->KL);     // position and all-zero flag of every function's bin
  l.off_misc = o;    o = align16(o + 32 * 4);
  l.off_lab = o;     o = align16(o + (c->cfg.max_labels > 0 ? c->cfg.max_labels : 1) * 4);
  l.off_tbase = o;   o = align16(o + (c->L + 1) * 4);
  l.off_tbeg = o;    o = align16(o + c->L * 4);
  l.off_topk = o;    o = align16(o + FWD_WARPS * 64 * 8);
  l.off_ids = o;     o = align16(o + ACT_SM * 4);
  l.off_z = o;       o = align16(o + ACT_SM * 4);
  l.off_col = o;     o = align16(o + hid_rows * 4);
  l.off_val = o;     o = align16(o + hid_rows * 4);
  l.off_h1 = o;      o = align16(o + 256 + 64 * 4 * 2 + 32 * 4);     // sampled hidden layer: bits, slice starts and lengths, active mask
  o = align128(o);
  l.off_dedup = o;
  l.fixed_bytes = o;
  return l;
}

cudaError_t setup_forward(Ctx* c) {
  FwdLayout l = fwd_layout(c);
  const int budget = 227 * 1024 - l.fixed_bytes;
  const int bitmap_bytes = align16(((c->N + 31) / 32) * 4);
  int64_t worst = (int64_t)c->L * c->cap + c->cfg.max_labels;
  int64_t pow2 = 1;
  while (pow2 < worst) pow2 <<= 1;
  const int64_t sort_bytes = pow2 * 4;
  // the staging space holds the hidden layer's chunk of W1 rows and, later, active rows of W2
  const int stage_min = l.hid_rows * c->H * 4;
  int mode = c->cfg.dedup_mode;
  int dd_bytes = 0;
  if (c->dense) { mode = 1; c->sort_cap = 0; }
  else {
    if (mode == 0) mode = (bitmap_bytes <= 100 * 1024 || sort_bytes > budget) ? 1 : 2;
    if (mode == 1 && bitmap_bytes > budget) return cudaErrorInvalidValue;
    if (mode == 2 && sort_bytes > budget) return cudaErrorInvalidValue;
    c->sort_cap = (int)pow2;
    dd_bytes = mode == 1 ? bitmap_bytes : (int)sort_bytes;
  }
  c->dedup_mode = mode;
  int stage = dd_bytes > stage_min ? dd_bytes : stage_min;
  // when the dedup work space leaves room for two blocks per multiprocessor, staging gets the rest of a half
  const int two_per_sm = TWO_PER_SM - l.fixed_bytes;
  if (stage < two_per_sm) stage = two_per_sm;
  if (stage > budget) stage = budget;
  if (stage < stage_min || stage < c->H * 4) return cudaErrorInvalidValue;
  c->fwd_stage_bytes = stage & ~15;
  // dedup by sorting for small candidate sets: mode 0 picks per sample, mode 1 always uses the bitmap, mode 2 always sorts
  c->fwd_sort_small = 0;
  if (mode == 1 && c->cfg.dedup_mode == 0 && !c->dense) {
    int cap_small = c->fwd_stage_bytes / 8;      // the sort pads to a power of two
    // A bitmap of a few words per thread is cleared and read out faster than more than a few hundred pairs are ranked.
    // Ranked / bitmap in us, 256 samples, 64 units: 200 candidates 36.3 / 36.0 (32,768 neurons, training), 36.3 / 35.0
    // (12,007), 20.6 / 19.6 (inference); 800 candidates 59.5 / 29.4 (32,768, inference), 59.5 / 28.8 (1,000).
    const int most = c->N <= BITMAP_CHEAP ? SORT_FEW : SORT_SMALL;
    c->fwd_sort_small = cap_small < most ? cap_small : most;
  }
  // the hash functions' tables are mirrored at the end of the staging space: SimHash's packed ones wherever they fit (from global
  // memory the 450 functions of 67 coordinates of a block took 20,000 to 29,000 cycles, from the mirror 5,000 to 6,800), DWTA's above the hidden layer's chunk
  {
    const long long one = (long long)c->KL * c->fn_len * 4;
    const bool sim = c->cfg.hash_family == DSLIDE_SIMHASH;
    const long long hb = sim ? (one / 2 + 15) & ~15ll : one;
    c->fwd_hash_sm_off = -1;
    c->fwd_hash_sm_bytes = c->fwd_hash_sm_late = 0;
    if (!c->dense && (sim ? hb <= (long long)c->fwd_stage_bytes : one % 16 == 0 && hb <= 32 * 1024 && stage_min + hb <= (long long)c->fwd_stage_bytes)) {
      c->fwd_hash_sm_bytes = (int)hb;
      c->fwd_hash_sm_off = (c->fwd_stage_bytes - (int)hb) & ~15;
      c->fwd_hash_sm_late = c->fwd_hash_sm_off < stage_min ? (stage_min - c->fwd_hash_sm_off + 15) & ~15 : 0;
      if (c->fwd_hash_sm_late > c->fwd_hash_sm_bytes) c->fwd_hash_sm_late = c->fwd_hash_sm_bytes;
    }
  }
  if (c->cfg.sample_budget > 0 && !c->dense) {
    // the reservoir's work space (an index per retrieved id, a slot per kept one, flags, the kept ids) overlays the staging region
    const long long a = c->act_stride, m = c->cfg.sample_budget < c->act_stride ? c->cfg.sample_budget : c->act_stride;
    if (4 * a + 4 * m + a + 16 + 4 * (m + c->cfg.max_labels) > (long long)c->fwd_stage_bytes) return cudaErrorInvalidValue;
    if (c->cfg.budget_fill) {
      // the fill's work space for the largest number of missing ids (the whole budget): draws, flags, hash set, ids
      const long long b = c->cfg.sample_budget < c->N ? c->cfg.sample_budget : c->N, D = 2 * b + 64;
      long long ts = 64;
      while (ts < 2 * D) ts <<= 1;
      if (4 * D + D + 4 + 8 * ts + 8 * b + 4 * b > (long long)c->fwd_stage_bytes) return cudaErrorInvalidValue;
    }
  }
  c->fwd_smem = l.fixed_bytes + c->fwd_stage_bytes;
  cudaError_t e = cudaSuccess;
  for (void (*k)(const FwdParams) : {k_forward<0, 1>, k_forward<0, 1, true>, k_forward<0, 2>, k_forward<0, 4>, k_forward<0, 8>, k_forward<1, 1>, k_forward<1, 2>, k_forward<1, 4>,
                                     k_forward<1, 8>, k_forward<2, 2>, k_forward<2, 8>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  return e;
}

static FwdParams make_params(Ctx* c, int batch, const int32_t* row_ptr, const int32_t* col_idx, const float* vals,
                             const int32_t* label_ptr, const int32_t* labels) {
  FwdParams p;
  p.W1 = c->W1; p.b1 = c->b1; p.W2 = c->W2;
  p.hash_idx = c->hash_idx; p.hash_sign = c->hash_sign; p.hash_pk = c->hash_pk; p.bucket_off = c->bucket_off; p.bucket_ids = c->bucket_ids;
  p.row_ptr = row_ptr; p.col_idx = col_idx; p.vals = vals; p.label_ptr = label_ptr; p.labels = labels;
  p.h = c->h; p.dh = c->dh; p.loss = c->loss; p.codes = c->codes;
  p.act_cnt = c->act_cnt; p.act_ids = c->act_ids; p.act_z = c->act_z; p.act_p = c->act_p; p.act_g = c->act_g;
  p.mask1 = c->mask1; p.mask2 = c->mask2; p.touch2 = c->touch2; p.ovf1 = c->ovf1; p.ovf2 = c->ovf2;
  p.hotmap1 = c->hotmap1; p.hotcoef1 = c->hotcoef1; p.bstride = c->cfg.max_batch; p.hdr1 = c->hdr1; p.hdr2 = c->hdr2;
  p.own1 = c->own1; p.own2 = c->own2; p.hot_rows = c->hot_rows; p.med_rows = c->med_rows; p.parity = (int)(c->t_host & 1);
  p.st = c->dstate; p.out_ids = nullptr; p.out_scores = nullptr;
  p.nb = c->nb;
  p.B = batch; p.D = c->D; p.H = c->H; p.N = c->N; p.K = c->K; p.L = c->L; p.KL = c->KL;
  p.family = c->cfg.hash_family; p.lg_bin = c->lg_bin; p.fn_len = c->fn_len; p.cap = c->cap;
  p.act_stride = c->act_stride; p.Wd = c->Wd; p.dense = c->dense; p.dedup_mode = c->dedup_mode;
  p.max_labels = c->cfg.max_labels; p.sort_cap = c->sort_cap; p.topk = 1;
  FwdLayout l = fwd_layout(c);
  p.stage_bytes = c->fwd_stage_bytes; p.hid_rows = l.hid_rows; p.sort_small = c->fwd_sort_small;
  p.densify = c->cfg.dwta_densify; p.seed = c->cfg.seed; p.rcount = (unsigned long long)c->r_host;
  p.budget = c->cfg.sample_budget; p.budget_fill = c->cfg.budget_fill; p.tcount = (unsigned long long)c->t_host;
  p.hash_sm_off = c->fwd_hash_sm_off; p.hash_sm_bytes = c->fwd_hash_sm_bytes; p.hash_sm_late = c->fwd_hash_sm_late; p.inputs_ready = 1;
  p.off_dh = l.off_dh; p.off_code = l.off_code; p.off_part = l.off_part; p.off_misc = l.off_misc;
  p.off_lab = l.off_lab; p.off_tbase = l.off_tbase; p.off_tbeg = l.off_tbeg; p.off_topk = l.off_topk;
  p.off_ids = l.off_ids; p.off_z = l.off_z; p.off_col = l.off_col; p.off_val = l.off_val; p.off_dedup = l.off_dedup;
  p.off_h1 = l.off_h1;
  p.proj1 = c->proj1; p.bucket1_off = c->bucket1_off; p.bucket1_ids = c->bucket1_ids;
  p.codes1 = c->codes1; p.hmask = c->hmask; p.cmask1 = c->cmask1;
  p.K1 = c->K1; p.L1 = c->L1; p.KL1 = c->KL1; p.cap1 = c->cap1; p.Hw = c->Hw;
  return p;
}

// Expected size of an active set from the tables' shape: L buckets of about N / 2^bits ids, cut at the cap (and at the sampling budget)
static double expected_set(const Ctx* c) {
  const double per_bucket = (double)c->N / (double)(1ll << c->bits);
  double expect = c->cfg.force_dense ? (double)c->N : (double)c->L * (per_bucket < c->cfg.bucket_cap ? per_bucket : (double)c->cfg.bucket_cap);
  if (c->cfg.sample_budget > 0 && expect > c->cfg.sample_budget) expect = c->cfg.sample_budget;
  return expect;
}
// Whether the active rows go through the warps' rings (k_forward<., 2 ...>) or are staged in chunks of the block's space.  us, staged /
// by rings: a step of 256 samples x 256 units x 200 rows 84.7 / 79.6, 16 x 200 units x 200 rows 36.7 / 34.8, one sample x 512 units
// 54.9 / 36.9, 1,024 x 1,024 units 615 / 498; but 1,024 x 200 units x 100 rows, which are one chunk, 167 / 171, one sample x 136
// units x 200 rows (a chunk and a quarter) 26.0 / 27.0.  Both ways over 136, 200 and 256 units, 1 to 1,024 samples and sets of 48 to 694
// rows, 168 shapes, by the set's size in chunks: steps staged / by rings 0.94 to 1.04 below one chunk, 0.97 to 1.05 from 1.25 to 1.6,
// 0.99 to 1.19 above; inference 0.90 to 1.03, 0.89 to 1.03 and 0.89 to 1.14.  What loses by the rule: inference at 136 units, where
// two lanes of 32 have a second piece (up to 12 %), and steps of 256 units at 1.15 chunks, which are staged (up to 11 %).
// (A DWTA bucket that is met holds a row more than the mean.)
static bool by_rings(const Ctx* c) {
  if (c->H <= 128 || c->H > 256) return c->H > 256;
  return expected_set(c) + c->L > 1.25 * (double)(c->fwd_stage_bytes / ((c->H + 4) * 4 + 4));
}

cudaError_t launch_forward_train(Ctx* c, int batch, const int32_t* row_ptr, const int32_t* col_idx, const float* vals,
                                 const int32_t* label_ptr, const int32_t* labels, int inputs_ready) {
  FwdParams p = make_params(c, batch, row_ptr, col_idx, vals, label_ptr, labels);
  p.inputs_ready = inputs_ready;
  if (use_tiles(c, batch)) {
    LaunchScope ls(c, KID_FORWARD);
    const cudaError_t e = launch_dependent(c->H <= FWD_THREADS ? k_forward<2, 2> : k_forward<2, 8>, dim3(batch), dim3(FWD_THREADS), (size_t)c->fwd_smem, c->stream, p);
    return e != cudaSuccess ? e : launch_tiles_forward(c, batch, label_ptr, labels);
  }
  {
    LaunchScope ls(c, KID_FORWARD);
    // Sets of many chunks of the staging space take the variant that fetches rows by bulk copies.
    const double expect = expected_set(c);
    const bool bulk = expect >= 4.0 * (double)(p.stage_bytes / ((c->H + 4) * 4 + 4));
    const cudaError_t e = launch_dependent(!by_rings(c) ? (bulk ? k_forward<0, 1, true> : k_forward<0, 1>) : c->H <= 256 ? k_forward<0, 2> : c->H <= 512 ? k_forward<0, 4> : k_forward<0, 8>,
                                           dim3(batch), dim3(FWD_THREADS), (size_t)c->fwd_smem, c->stream, p);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

cudaError_t launch_predict(Ctx* c, int batch, const int32_t* row_ptr, const int32_t* col_idx, const float* vals,
                           int k, int dense, int32_t* out_ids, float* out_scores) {
  FwdParams p = make_params(c, batch, row_ptr, col_idx, vals, nullptr, nullptr);
  p.topk = k;
  p.out_ids = out_ids;
  p.out_scores = out_scores;
  if (dense) p.dense = 1;
  p.inputs_ready = 0;            // the batch may come from the kernel before this one in the stream: nothing is read before it has completed
  LaunchScope ls(c, KID_PREDICT);
  // placed while the kernel before it drains (the call before this one, in a serving loop)
  cudaError_t e = launch_dependent(!by_rings(c) ? k_forward<1, 1> : c->H <= 256 ? k_forward<1, 2> : c->H <= 512 ? k_forward<1, 4> : k_forward<1, 8>,
                                   dim3(batch), dim3(FWD_THREADS), (size_t)c->fwd_smem, c->stream, p);
  if (e != cudaSuccess || !dense) return e;
  return launch_dense_tc(c, batch, k, out_ids, out_scores);      // over all neurons: the kernel above has left the hidden activations
}

}  // namespace dslide
