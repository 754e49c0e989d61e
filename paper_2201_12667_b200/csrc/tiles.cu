// Training steps whose active sets hold thousands of neurons that the batch's samples share: logits and the
// back-propagated error by tiles of rows of W2 instead of sample by sample.
//
// A block per sample fetches every active row once per sample that has it active (14 to 60 times over a batch: 5 GB
// per step where the rows are 82 MB), and counts every touch with an atomic.  Here the rows that the batch touches
// are numbered in id order and cut into tiles that fit shared memory; a tile's rows are fetched once and serve all
// samples (once per group of samples where the chunks' sums would not fit TILE_PART_BYTES: tile_grid).  A sample's active ids are ascending, so its entries of a tile are one run of its list.
//
//   k_forward<2>    : hidden layer, codes, active sets; marks the touched rows in a bitmap (forward.cu)
//   k_tile_scan     : touched rows before every word of the bitmap, and where the tiles start
//   k_tile_index    : the list of touched rows; per active neuron its place in its tile; per (tile, sample) the run
//   k_tile_forward  : a block holds a tile; a warp takes a sample's run: rows are read into registers several at a time,
//                     their logits taken, and the sums S = sum_a exp(z_a - M) W2[a], E = sum_a exp(z_a - M) carried
//                     along with a running maximum M (so a row is read from shared memory once for both).
//   k_tile_combine  : per sample: the row chunks' S, E, M put together, loss, errors, error at the hidden layer
//   k_tile_lists    : per touched row the list of (sample, error), ascending samples
//   k_rows_update   : gradients and Adam of the touched rows of W2 (update.cu)
// The order of every sum follows from the touched rows alone: results are the same from run to run.
#include <math.h>

#include "common.cuh"
#include "waits.cuh"

namespace dslide {

constexpr unsigned TFULL = 0xffffffffu;
// x / step for 0 <= x <= TILE_N_MAX and step <= TILE_ROWS_MAX, by a multiplication with ceil(2^32 / step)
__host__ __device__ __forceinline__ unsigned tile_magic(int step) { return (unsigned)(((1ull << 32) + (unsigned)step - 1) / (unsigned)step); }
__device__ __forceinline__ int tile_of(int x, unsigned magic, int step) { return step == 1 ? x : (int)__umulhi((unsigned)x, magic); }
constexpr int TS_THREADS = 1024;
constexpr int TS_WORDS = 16;
constexpr int TI_THREADS = 512;
constexpr int TF_THREADS = 512;
constexpr int TF_WARPS = TF_THREADS / 32;
constexpr int TC3_THREADS = 512;
constexpr int TL_THREADS = 512;
constexpr int TL_WARPS = TL_THREADS / 32;
constexpr int TL_CHUNK = 1024;                         // samples listed at a time
constexpr int TILE_BYTES = 196 * 1024;                 // shared memory for a tile's rows
constexpr int TILE_N_MAX = 8 << 20;
constexpr int TILE_STEP_MIN = 32;
constexpr int TILE_ROWS_MAX = 512;                     // a thread of k_tile_lists each
constexpr size_t TILE_PART_BYTES = (size_t)32 << 20;   // the row chunks' sums stay in L2
constexpr size_t TILE_SEG_BYTES = (size_t)512 << 20, TILE_LIST_BYTES = (size_t)2 << 30;      // beyond these the work space is not worth it
// Which steps go by tiles: from TILE_MIN_SET neurons per sample on, when a sample has at least TILE_MIN_RUN of them in a
// tile on average (below that, walking the (tile, sample) pairs costs more than the shared rows save).
// A touched row must serve several samples: at three (81,000 pairs over 28,600 rows of 64 units) the eight launches took
// 138 us against 95 of the block per sample, at twenty (36,000 pairs over 1,741 rows of 252 units) 102 against 186.
// And a block per sample must have enough to fetch: what the tiles save is its rows, set x width floats for every 296
// samples (two blocks per multiprocessor), while the six more launches and the lists cost the same at any width.
// Measured over 219 random shapes that pass the other conditions (4 to 1,024 units, 4 to 2,048 samples): with
// TILE_MIN_ROWS 152 of them go by tiles, 124 of those faster by 3 % and more (up to 4x) and 13 slower by 10 % and more
// (their sets are smaller than the tables' shape lets expect), nine that gained are refused (7 of them 10 % and more);
// without it 73 were slower, down to 0.34x.  On the line's two sides, by tiles / sample by sample in us: 1,406 neurons x
// 32 units, 64 samples 93 / 88, 1,024 samples 465 / 618; x 64 units, 64 samples 96 / 105; 1,169 x 32, 256 samples 196 / 142.
constexpr double TILE_MIN_SET = 512.0, TILE_MIN_RUN = 1.5, TILE_MIN_SHARE = 6.0, TILE_MIN_ROWS = 64000.0;

// Expected size of an active set and of the pool of rows the tables hand out, from the tables' shape: L buckets of
// about N / 2^bits ids; where the cap cuts them, the lowest ids of every bucket are what all samples share.
static void expect_sets(Ctx* c) {
  const double mean = (double)c->N / (double)c->nb;
  const double per = mean < c->cap ? mean : (double)c->cap;
  double pool = (double)c->N;
  if (mean > c->cap && 1.6 * c->cap * (double)c->nb < pool) pool = 1.6 * c->cap * (double)c->nb;
  double got = pool * -expm1(-(double)c->L * per / pool);
  if (c->cfg.sample_budget > 0 && got > c->cfg.sample_budget) got = c->cfg.sample_budget;
  c->tile_got = got;
  c->tile_pool = pool;
}

// floats that a multiprocessor's blocks fetch from W2, in sets of a sample
static bool enough_rows(const Ctx* c, int batch) {
  const double waves = (double)batch / (2.0 * c->num_sms);
  return c->tile_got * c->H * (waves > 1.0 ? waves : 1.0) >= TILE_MIN_ROWS;
}

bool use_tiles(const Ctx* c, int batch) {
  if (c->tile_rows == 0 || !enough_rows(c, batch)) return false;
  const double touched = c->tile_pool * -expm1(-(double)batch * c->tile_got / c->tile_pool);
  return c->tile_got * (double)c->tile_step >= TILE_MIN_RUN * touched && (double)batch * c->tile_got >= TILE_MIN_SHARE * touched;
}

// Rows of a tile for this batch (a tile may hold up to 31 more): as many as fit, or so few that every multiprocessor has
// two tiles -- small batches -- while a sample still has a dozen entries in a tile on average.
static int call_step(const Ctx* c, int batch) {
  const double touched = c->tile_pool * -expm1(-(double)batch * c->tile_got / c->tile_pool);
  double want = touched / (2.0 * c->num_sms);
  if (want < 12.0 * touched / c->tile_got) want = 12.0 * touched / c->tile_got;
  if (want < TILE_STEP_MIN) want = TILE_STEP_MIN;
  return want < c->tile_step ? (int)want : c->tile_step;
}
// Tiles at most (k_tile_scan makes them smaller, so that the row chunks get the same number: up to one more each)
static int call_tiles(const Ctx* c, int batch) { return c->N / call_step(c, batch) + 2 + c->num_sms; }

// Row chunks (blocks that walk the tiles side by side) and groups of samples of k_tile_forward.
static void tile_grid(const Ctx* c, int batch, int* chunks, int* groups) {
  const size_t one = (size_t)batch * (c->H + 4) * sizeof(float);
  int most = (int)(TILE_PART_BYTES / one);
  if (most < 1) most = 1;
  int q = (c->num_sms + most - 1) / most;
  const int qmax = (batch + TF_WARPS - 1) / TF_WARPS;
  if (q > qmax) q = qmax;
  if (q < 1) q = 1;
  int p = c->num_sms / q;
  if (p < 1) p = 1;
  const int tiles = c->N / call_step(c, batch) + 2;
  if (p > tiles) p = tiles;
  *chunks = p;
  *groups = q;
}

cudaError_t setup_tiles(Ctx* c) {
  c->tile_rows = 0;
  if (c->dense) return cudaSuccess;
  expect_sets(c);
  const double most_shared = c->cfg.max_batch * c->tile_got / (c->tile_pool * -expm1(-c->cfg.max_batch * c->tile_got / c->tile_pool));
  if (c->tile_got < TILE_MIN_SET || most_shared < TILE_MIN_SHARE || !enough_rows(c, c->cfg.max_batch)) return cudaSuccess;      // no batch would take them
  int rows = TILE_BYTES / ((c->H + 4) * 4);
  if (rows > TILE_ROWS_MAX) rows = TILE_ROWS_MAX;
  const int step = rows - 31;                // a tile takes whole words of the bitmap
  if (step < 1 || c->N > TILE_N_MAX) return cudaSuccess;
  c->tile_step = step;
  const size_t B = c->cfg.max_batch;
  size_t most = 0, runs = 0, tiles = 0;
  for (int b = 1; b <= c->cfg.max_batch; ++b) {
    int p, q;
    tile_grid(c, b, &p, &q);
    const size_t n = (size_t)p * b * (c->H + 4), t = (size_t)call_tiles(c, b) + 1;
    if (n > most) most = n;
    if (t * b > runs) runs = t * b;
    if (t > tiles) tiles = t;
  }
  if (runs * 4 > TILE_SEG_BYTES || B * (size_t)c->act_stride * 8 > TILE_LIST_BYTES) return cudaSuccess;
  const size_t nw = ((size_t)c->N + 31) / 32;
  struct Part { void** p; size_t bytes; };
  const Part parts[] = {{(void**)&c->touch2, nw * 4}, {(void**)&c->wpre, (nw + 1) * 4}, {(void**)&c->trows, (size_t)c->N * 4},
                        {(void**)&c->tstart, tiles * 4}, {(void**)&c->tinfo, 32}, {(void**)&c->act_loc, B * (size_t)c->act_stride * 2},
                        {(void**)&c->seg, runs * 4}, {(void**)&c->tpart, most * 4}, {(void**)&c->rinfo, (size_t)c->N * 8},
                        {(void**)&c->tlist, B * (size_t)c->act_stride * 8}, {(void**)&c->tlab, B * (size_t)c->cfg.max_labels * 4}};
  // The context works without (every step sample by sample), so the work space never stands in its way: it takes at most
  // half of what the model has left free on the device, and what cannot be had is given back.
  size_t sum = 0, left = 0, all = 0;
  for (const Part& q : parts) sum += q.bytes;
  cudaError_t e = cudaMemGetInfo(&left, &all);
  if (e != cudaSuccess) return e;
  if (sum > left / 2) return cudaSuccess;
  for (const Part& q : parts)
    if (e == cudaSuccess && (e = cudaMalloc(q.p, q.bytes)) != cudaSuccess) *q.p = nullptr;
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    for (const Part& q : parts) {
      if (*q.p) cudaFree(*q.p);
      *q.p = nullptr;
    }
    return cudaSuccess;
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(c->touch2, 0, nw * 4, c->stream);
  if (e == cudaSuccess) c->tile_rows = rows;
  return e;
}

// One block: touched rows before every word (exclusive running sum of the words' bit counts), and the first row of
// every tile: word w belongs to tile wpre[w] / step.  The step is `most`, or, where the row chunks would take two to four rounds of
// tiles, so much less that the last round is a whole one (a step of 256 samples x 325,056 neurons x 128 units 340 us, so 333; 512
// x 200,003 x 64 471 and 459; not tiles of few words of the bitmap, whose sizes jump: 512 x 50,021 x 128, 32 rows, 259 and 272).  Both
// ways over 60 shapes, 32 to 256 units, 20,011 to 325,056 neurons, 64 to 1,024 samples: at worst 0.4 % slower, at best 3 % faster.
__global__ void __launch_bounds__(TS_THREADS)
k_tile_scan(const uint32_t* touch, int nw, int most, int chunks, int* wpre, int* tstart, int* tinfo, unsigned int* n_touched) {
  __shared__ int sh[TS_THREADS / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  griddep_launch_dependents();
  griddep_wait();
  const int per = ((nw + TS_THREADS - 1) / TS_THREADS + 3) & ~3;
  const int w0 = min(nw, tid * per), w1 = min(nw, w0 + per);
  // a thread's words stay in registers between the count and the walk (more of them than that are read again)
  uint32_t word[TS_WORDS];
#pragma unroll
  for (int i = 0; i < TS_WORDS; ++i) word[i] = i < w1 - w0 ? __ldcg(touch + w0 + i) : 0u;
  int mine = 0;
#pragma unroll
  for (int i = 0; i < TS_WORDS; ++i) mine += __popc(word[i]);
  for (int w = w0 + TS_WORDS; w < w1; ++w) mine += __popc(__ldcg(touch + w));
  int incl = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int o = __shfl_up_sync(TFULL, incl, d);
    if (lane >= d) incl += o;
  }
  if (lane == 31) sh[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    int v = sh[lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int o = __shfl_up_sync(TFULL, v, d);
      if (lane >= d) v += o;
    }
    sh[lane] = v;
  }
  __syncthreads();
  const int total = sh[TS_THREADS / 32 - 1];
  int run = incl - mine + (warp > 0 ? sh[warp - 1] : 0);
  // (a tile starts at a word, so up to one more tile than rows / step)
  const int rounds = (total / most + chunks) / chunks;
  const int even = (total + rounds * chunks - 1) / (rounds * chunks);
  const int step = rounds < 2 || rounds > 4 || even < 96 ? most : min(most, even);
  // the tile of the word before this thread's first one: its start, or that of a tile further back, covers `run`
  const unsigned magic = tile_magic(step);
  int tile = -1;
  if (w0 > 0 && w0 < w1) {
    const int before = run - __popc(__ldcg(touch + w0 - 1));
    tile = tile_of(before, magic, step);
  }
  auto walk = [&](int w, uint32_t bits) {
    wpre[w] = run;
    const int t = tile_of(run, magic, step);
    for (; tile < t;) tstart[++tile] = run;
    run += __popc(bits);
  };
#pragma unroll
  for (int i = 0; i < TS_WORDS; ++i)
    if (i < w1 - w0) walk(w0 + i, word[i]);
  for (int w = w0 + TS_WORDS; w < w1; ++w) walk(w, __ldcg(touch + w));
  if (w0 < w1 && w1 == nw) {                 // the thread with the last word
    wpre[nw] = total;
    tstart[tile + 1] = total;
    tinfo[0] = tile + 1;
    tinfo[1] = 0;
    tinfo[2] = 0;
    tinfo[3] = step;
    tinfo[4] = (int)magic;
    *n_touched = (unsigned)total;
  }
}

// Blocks [0, B): a sample's entries -- place in the tile, and where the runs of the tiles start (a tile without
// entries has an empty run).  The blocks after them write the list of touched rows.
__global__ void __launch_bounds__(TI_THREADS + 32)
k_tile_index(const uint32_t* touch, const int* wpre, const int* tstart, const int* tinfo, int nw, int B, int bstride,
             const int* act_cnt, const int32_t* act_ids, int act_stride, const int32_t* label_ptr, const int32_t* labels,
             int max_labels, uint16_t* act_loc, int* seg, int* trows, int* tlab) {
  const int tid = threadIdx.x;
  griddep_launch_dependents();
  griddep_wait();
  if ((int)blockIdx.x >= B) {
    if (tid >= TI_THREADS) return;
    const int nb = (int)gridDim.x - B;
    for (int w = ((int)blockIdx.x - B) * TI_THREADS + tid; w < nw; w += nb * TI_THREADS) {
      uint32_t bits = __ldcg(touch + w);
      int at = __ldcg(wpre + w);
      while (bits) {
        trows[at++] = (w << 5) + __ffs(bits) - 1;
        bits &= bits - 1;
      }
    }
    return;
  }
  const int s = blockIdx.x;
  const int na = __ldcg(act_cnt + s), nt = __ldcg(tinfo);
  const int32_t* ids = act_ids + (size_t)s * act_stride;
  uint16_t* loc = act_loc + (size_t)s * act_stride;
  if (tid >= TI_THREADS) {                    // the last warp: the labels' places in the active set (a repeated label counts once)
    const int lbeg = label_ptr[s], nlab = na > 0 ? label_ptr[s + 1] - lbeg : 0;
    for (int i = tid - TI_THREADS; i < nlab; i += 32) {
      const int y = labels[lbeg + i];
      bool first = true;
      for (int q = 0; q < i; ++q) first = first && labels[lbeg + q] != y;
      int lo = 0, hi = na;
      while (lo < hi) { const int mid = (lo + hi) >> 1; if (__ldcg(ids + mid) < y) lo = mid + 1; else hi = mid; }
      tlab[(size_t)s * max_labels + i] = first ? lo : -1;
    }
    return;
  }
  if (na == 0) {
    for (int t = tid; t <= nt; t += TI_THREADS) seg[(size_t)t * bstride + s] = 0;
    return;
  }
  constexpr int U = 4;                       // entries per thread and round: their chains of loads run side by side
  const int step = __ldcg(tinfo + 3);
  const unsigned magic = (unsigned)__ldcg(tinfo + 4);
  for (int a0 = 0; a0 < na; a0 += U * TI_THREADS) {
    int j[U], pre[U], prev[U], ts[U];
    uint32_t bits[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int a = a0 + u * TI_THREADS + tid;
      j[u] = a < na ? __ldcg(ids + a) : 0;
      prev[u] = a < na && a > 0 && (tid & 31) == 0 ? __ldcg(ids + a - 1) : -1;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      pre[u] = __ldcg(wpre + (j[u] >> 5));
      bits[u] = __ldcg(touch + (j[u] >> 5));
      if (prev[u] >= 0) prev[u] = __ldcg(wpre + (prev[u] >> 5));
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      bits[u] = (uint32_t)__popc(bits[u] & ((1u << (j[u] & 31)) - 1u));      // touched rows of the word before this one
      ts[u] = __ldcg(tstart + tile_of(pre[u], magic, step));
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int a = a0 + u * TI_THREADS + tid;
      const int t = tile_of(pre[u], magic, step);
      const int up = __shfl_up_sync(TFULL, t, 1);
      const int before = (tid & 31) == 0 ? (prev[u] >= 0 ? tile_of(prev[u], magic, step) : -1) : up;
      if (a >= na) continue;
      loc[a] = (uint16_t)(pre[u] + (int)bits[u] - ts[u]);
      for (int q = before + 1; q <= t; ++q) seg[(size_t)q * bstride + s] = a;
      if (a == na - 1)
        for (int q = t + 1; q <= nt; ++q) seg[(size_t)q * bstride + s] = na;
    }
  }
}

struct TileParams {
  const float* W2;
  const RowHdr* hdr2;
  const float* h;
  const int *trows, *tstart, *seg;
  int* tinfo;            // number of tiles; whether a tile's rows did not come in time
  const uint16_t* act_loc;
  float *act_z, *part;
  DevState* st;
  int B, H, act_stride, bstride, chunks, gs;      // gs: samples of a group
};

__device__ __forceinline__ uint32_t t_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void t_bulk(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(t_smem(dst)), "l"(src), "r"(bytes), "r"(t_smem(bar)) : "memory");
}
// Brings tile t into shared memory, all threads: the rows one after the other, each followed by the head of its record
// (count, bias, bias moments).  False when they did not come in time (block-uniform; nothing is left in flight).
__device__ __forceinline__ bool load_tile(const TileParams& p, int t, float* tile, uint64_t* bar, uint32_t phase) {
  const int H = p.H, ld = H + 4;
  const int r0 = __ldcg(p.tstart + t), nr = __ldcg(p.tstart + t + 1) - r0;
  __syncthreads();                             // readers of the tile before are done
  if (threadIdx.x == 0)
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(t_smem(bar)), "r"((uint32_t)nr * ((uint32_t)H * 4u + 16u)) : "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  for (int r = threadIdx.x; r < nr; r += TF_THREADS) {
    const int j = __ldcg(p.trows + r0 + r);
    t_bulk(tile + (size_t)r * ld, p.W2 + (size_t)j * H, (uint32_t)H * 4u, bar);
    t_bulk(tile + (size_t)r * ld + H, p.hdr2 + j, 16u, bar);
  }
  const bool ok = bar_wait_limited(bar, phase);
  if (!__syncthreads_or(ok ? 0 : 1)) return true;
  bar_wait_limited(bar, phase);                          // one more bounded wait for the copies in flight, then out
  if (threadIdx.x == 0) { p.tinfo[1] = 1; atomicCAS(&p.st->status, 0, (int)DSLIDE_ERR_TIMEOUT); }
  return false;
}
// Grid (row chunks, groups of samples).  A group of G lanes takes a row: lane g of it holds the 16-byte pieces g, g + G,
// ... (NP of them).  R rows per group at a time: their dot products with the sample's activations are reduced
// together (lanes exchange the values they give up, so that Q lanes of the group end with each row's sum).  Rows of
// up to 128 units are taken by half warps, four rows each (G = 16); wider ones by whole warps (G = 32: with half warps the
// eight rows of 200 units do not fit the registers and the one-hot word shape took 1,614 us a step instead of 1,531), eight
// rows up to 256 units -- one reduction, one exponential and one look at the maximum for eight rows: 563 us instead of 587 for
// 1,024 samples x 6,100 neurons x 200 units -- and four beyond.  At more than 512 units the rows' places and weights pass
// through shared memory, as with eight rows: by shuffles they cost 700 bytes of spills (512 samples x 60,013 neurons x 1,024
// units, a step 7,180 us, now 4,240); at 257 to 512 shuffles are the faster (463 us against 535 for 400 samples x 332 units).
// Rows of up to 256 units stay in registers between the logits and the sums, others are read a second time.
template <int G, int NP, int R>
__global__ void __launch_bounds__(TF_THREADS, 1) k_tile_forward(const TileParams p) {
  constexpr bool KEEP = G == 16 || NP <= 2;
  constexpr bool STAGED = R == 8 || NP == 8;   // places and weights of rows by way of shared memory: one load for a shuffle per row, fewer registers
  constexpr int Q = G / R;                     // lanes that end with the same row's sum
  constexpr int RPI = R * 32 / G;              // rows per iteration
  extern __shared__ __align__(128) unsigned char t_sm[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ __align__(16) float zeros[4];
  __shared__ __align__(16) uint16_t places[STAGED ? TF_WARPS : 1][32];       // of 32 entries of the run a warp is at
  __shared__ __align__(16) float weights[STAGED ? TF_WARPS : 1][RPI];        // of the rows of an iteration
  float* tile = reinterpret_cast<float*>(t_sm);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int H = p.H, H4 = H >> 2, ld = H + 4;
  const int gl = lane & (G - 1), first = lane / G * R;      // place in the group; the group's first row of an iteration
  if (tid < 4) zeros[tid] = 0.f;
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(t_smem(&bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // the pieces of a row this lane reads: every lane has the first SURE ones; past the row's end it reads zeros (not a
  // piece of the row: a weight of minus infinity, which masks the neuron, times an activation of zero is no number)
  constexpr int SURE = NP / 2;
  int off[NP - SURE], mul[NP - SURE];
#pragma unroll
  for (int u = SURE; u < NP; ++u) {
    const bool in = gl + G * u < H4;
    off[u - SURE] = in ? 4 * (gl + G * u) : (int)(zeros - tile);
    mul[u - SURE] = in ? ld : 0;
  }
  auto piece = [&](int u, int l) {             // of the row at place l
    return *reinterpret_cast<const ulonglong2*>(u < SURE ? tile + (l * ld + 4 * (gl + G * u)) : tile + (l * mul[u < SURE ? 0 : u - SURE] + off[u < SURE ? 0 : u - SURE]));
  };
  griddep_launch_dependents();
  griddep_wait();
  const int nt = __ldcg(p.tinfo);
  const int q0 = (int)blockIdx.y * p.gs, q1 = min(p.B, q0 + p.gs);
  uint32_t phase = 0u;
  for (int t = blockIdx.x; t < nt; t += p.chunks, phase ^= 1u) {
    if (!load_tile(p, t, tile, &bar, phase)) return;
    const bool fresh = t == (int)blockIdx.x;   // the chunk's first tile: nothing to carry on from
    // a warp's samples: q0 + warp, + TF_WARPS, ...; lane i holds the run of the i-th of 32 of them
    for (int sb = q0 + warp; sb < q1; sb += 32 * TF_WARPS) {
      const int ms = sb + lane * TF_WARPS;
      int ra = 0, rn = 0;
      if (ms < q1) {
        ra = __ldcg(p.seg + (size_t)t * p.bstride + ms);
        rn = __ldcg(p.seg + (size_t)(t + 1) * p.bstride + ms) - ra;
      }
      unsigned todo = __ballot_sync(TFULL, ms < q1 && (rn > 0 || fresh));
      while (todo) {
        const int i = __ffs(todo) - 1;
        todo &= todo - 1;
        const int s = sb + i * TF_WARPS;
        const int a0 = __shfl_sync(TFULL, ra, i), n = __shfl_sync(TFULL, rn, i);
        float* part = p.part + ((size_t)blockIdx.x * p.B + s) * ld;
        if (n == 0) {
          if (lane == 0) { part[H] = -INFINITY; part[H + 1] = 0.f; }
          continue;
        }
        const uint16_t* locp = p.act_loc + (size_t)s * p.act_stride + a0;
        float* zp = p.act_z + (size_t)s * p.act_stride + a0;
        int loc = lane < n ? (int)__ldcg(locp + lane) : 0;
        ulonglong2 hx[NP], S[NP];                // pairs of floats: two multiply-adds per instruction
        float M = -INFINITY, E = 0.f, E0 = 0.f;  // E: this lane's rows only, until the end of the run; E0: the tiles before
#pragma unroll
        for (int u = 0; u < NP; ++u) {
          const int c = gl + G * u;
          hx[u] = c < H4 ? reinterpret_cast<const ulonglong2*>(p.h + (size_t)s * H)[c] : make_ulonglong2(0ull, 0ull);
          S[u] = make_ulonglong2(0ull, 0ull);
        }
        if (!fresh) {
          const float2 me = *reinterpret_cast<const float2*>(part + H);
          ulonglong2 sv[NP];
#pragma unroll
          for (int u = 0; u < NP; ++u) {
            const int c = gl + G * u;
            sv[u] = c < H4 && lane < G ? reinterpret_cast<const ulonglong2*>(part)[c] : make_ulonglong2(0ull, 0ull);
          }
          if (me.y > 0.f || me.y != me.y) {       // something was summed before: the first group carries it on
            M = me.x;
            E0 = me.y;
#pragma unroll
            for (int u = 0; u < NP; ++u) S[u] = sv[u];
          }
        }
        for (int c0 = 0; c0 < n; c0 += 32) {
          if (c0 > 0) loc = c0 + lane < n ? (int)__ldcg(locp + c0 + lane) : 0;
          const int m = min(32, n - c0);
          {
            const int some = __shfl_sync(TFULL, loc, 0);      // past the run: a row of the run, with weight zero below
            if (lane >= m) loc = some;
          }
          if (STAGED) {
            __syncwarp();
            places[warp][lane] = (uint16_t)loc;
            __syncwarp();
          }
          for (int k = 0; k < m; k += RPI) {
            int rl[R];                           // places of the group's rows
            if (STAGED) {
#pragma unroll
              for (int r = 0; r < R; r += 4) {
                const uint2 w = *reinterpret_cast<const uint2*>(&places[warp][k + r]);
                rl[r] = (int)(w.x & 0xffffu); rl[r + 1] = (int)(w.x >> 16); rl[r + 2] = (int)(w.y & 0xffffu); rl[r + 3] = (int)(w.y >> 16);
              }
            } else {
#pragma unroll
              for (int r = 0; r < R; ++r) rl[r] = __shfl_sync(TFULL, loc, k + first + r);
            }
            ulonglong2 x[R][KEEP ? NP : 1];
            float d[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
              unsigned long long d0 = 0ull, d1 = 0ull;
#pragma unroll
              for (int u = 0; u < NP; ++u) {
                const ulonglong2 v = piece(u, rl[r]);
                if (KEEP) x[r][KEEP ? u : 0] = v;
                fma2(d0, v.x, hx[u].x);
                fma2(d1, v.y, hx[u].y);
              }
              d[r] = (lo2(d0) + hi2(d0)) + (lo2(d1) + hi2(d1));
            }
            // every exchange halves the rows a lane has part of
#pragma unroll
            for (int n2 = R / 2, o = G / 2; n2 > 0; n2 >>= 1, o >>= 1) {
              const bool up = (lane & o) != 0;
#pragma unroll
              for (int r = 0; r < n2; ++r) d[r] = (up ? d[r + n2] : d[r]) + __shfl_xor_sync(TFULL, up ? d[r] : d[r + n2], o);
            }
            float y = d[0];
#pragma unroll
            for (int o = Q / 2; o > 0; o >>= 1) y += __shfl_xor_sync(TFULL, y, o);
            int ml;                              // the row whose sum this lane has
            if (STAGED) {
              ml = places[warp][k + lane / Q];
            } else {
              const bool hi = (lane & (2 * Q)) != 0, od = (lane & Q) != 0;
              ml = hi ? (od ? rl[3] : rl[2]) : (od ? rl[1] : rl[0]);
            }
            float z = tile[ml * ld + H + 1] + y;                     // the bias came with the row
            const int mine = k + lane / Q;
            if (mine >= m) z = -INFINITY;
            else if ((lane & (Q - 1)) == 0) zp[c0 + mine] = z;
            if (__any_sync(TFULL, z > M)) {
              float zm = fmaxf(z, M);
#pragma unroll
              for (int o = Q; o < 32; o <<= 1) zm = fmaxf(zm, __shfl_xor_sync(TFULL, zm, o));
              const float scale = expf(M - zm);
              const unsigned long long sc = pair2(scale, scale);
              M = zm;
              E *= scale;
              E0 *= scale;
#pragma unroll
              for (int u = 0; u < NP; ++u) { mul2(S[u].x, sc); mul2(S[u].y, sc); }
            }
            // a masked neuron (bias of minus infinity) weighs nothing, also while nothing else has been met and M is minus infinity
            const float e = z != -INFINITY ? expf(z - M) : 0.f;
            E += e;
            float4 four[STAGED ? R / 4 : 1];
            if (STAGED) {
              __syncwarp();                      // the weights before have been read
              if ((lane & (Q - 1)) == 0) weights[warp][lane / Q] = e;
              __syncwarp();
#pragma unroll
              for (int r = 0; r < R; r += 4) four[STAGED ? r / 4 : 0] = *reinterpret_cast<const float4*>(&weights[warp][r]);
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
              const float4& f4 = four[STAGED ? r / 4 : 0];
              const float g = !STAGED ? __shfl_sync(TFULL, e, (lane & ~(G - 1)) + Q * r) : (r & 3) == 0 ? f4.x : (r & 3) == 1 ? f4.y : (r & 3) == 2 ? f4.z : f4.w;
              const unsigned long long gg = pair2(g, g);
#pragma unroll
              for (int u = 0; u < NP; ++u) {
                const ulonglong2 v = KEEP ? x[r][KEEP ? u : 0] : piece(u, rl[r]);
                fma2(S[u].x, gg, v.x);
                fma2(S[u].y, gg, v.y);
              }
            }
          }
        }
#pragma unroll
        for (int o = Q; o < 32; o <<= 1) E += __shfl_xor_sync(TFULL, E, o);      // lanes hold different rows
#pragma unroll
        for (int u = 0; u < NP; ++u) {
          const int c = gl + G * u;
          if (G == 16) {                         // the two halves' sums
            const unsigned long long ox = __shfl_xor_sync(TFULL, S[u].x, 16), oy = __shfl_xor_sync(TFULL, S[u].y, 16);
            const unsigned long long one = pair2(1.f, 1.f);
            fma2(S[u].x, ox, one);
            fma2(S[u].y, oy, one);
          }
          if (c < H4 && lane < G) reinterpret_cast<ulonglong2*>(part)[c] = S[u];
        }
        if (lane == 0) *reinterpret_cast<float2*>(part + H) = make_float2(M, E0 + E);
      }
    }
  }
}

// One block per sample: softmax, loss and errors over the active set, and the error at the hidden layer,
// dh = [h > 0] (S / E - T / |Y|) / B with T the sum of the label rows.  Also clears the bitmap for the next step.
struct CombineParams {
  const float *W2, *h, *part, *act_z;
  const int32_t *label_ptr, *act_ids;
  const int *act_cnt, *tinfo, *tlab;
  float *act_p, *act_g, *dh, *loss;
  uint32_t* touch;
  int B, H, act_stride, chunks, nw, max_labels;
};

__global__ void __launch_bounds__(TC3_THREADS) k_tile_combine(const CombineParams p) {
  extern __shared__ __align__(16) unsigned char tc3_sm[];      // [chunks] factors, [parts][H] partial sums, [max_labels] places of the labels
  __shared__ float sh_M, sh_E;
  __shared__ int sh_ny;
  const int s = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int H = p.H, ld = H + 4;
  const int parts = H >= TC3_THREADS ? 1 : TC3_THREADS / H;    // threads that share a hidden unit's sum over the chunks
  float* fac = reinterpret_cast<float*>(tc3_sm);
  float* ps = fac + ((p.chunks + 3) & ~3);
  int* lab = reinterpret_cast<int*>(ps + parts * H);
  griddep_launch_dependents();
  griddep_wait();
  {
    const int per = (p.nw + p.B - 1) / p.B;
    for (int w = s * per + tid; w < min(p.nw, (s + 1) * per); w += TC3_THREADS) p.touch[w] = 0u;
  }
  const int na = p.act_cnt[s];
  if (na == 0) {                               // a skipped sample, or one without labels whose buckets are all empty
    for (int k = tid; k < H; k += TC3_THREADS) p.dh[(size_t)s * H + k] = 0.f;
    if (tid == 0) p.loss[s] = 0.f;
    return;
  }
  const int np = min(p.chunks, __ldcg(p.tinfo));
  const int nlab = p.label_ptr[s + 1] - p.label_ptr[s];
  if (warp == 0) {
    // maximum and sum over the chunks (lane i takes the chunks i, i + 32, ...; then the lanes, in a fixed order)
    float M = -INFINITY;
    for (int b = lane; b < np; b += 32) M = fmaxf(M, __ldcg(p.part + ((size_t)b * p.B + s) * ld + H));
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) M = fmaxf(M, __shfl_xor_sync(TFULL, M, d));
    float E = 0.f;
    for (int b = lane; b < np; b += 32) {
      const float2 me = __ldcg(reinterpret_cast<const float2*>(p.part + ((size_t)b * p.B + s) * ld + H));
      const float f = me.y == 0.f ? 0.f : expf(me.x - M);
      fac[b] = f;
      E += me.y * f;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) E += __shfl_xor_sync(TFULL, E, d);
    if (lane == 0) { sh_M = M; sh_E = E; }
  } else if (warp == 1) {
    int ny = 0;
    for (int i = lane; i < nlab; i += 32) {
      const int at = __ldcg(p.tlab + (size_t)s * p.max_labels + i);
      lab[i] = at;
      ny += at >= 0 ? 1 : 0;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) ny += __shfl_xor_sync(TFULL, ny, d);
    if (lane == 0) sh_ny = ny;
  }
  const int32_t* ids = p.act_ids + (size_t)s * p.act_stride;
  const float* z = p.act_z + (size_t)s * p.act_stride;
  float* g = p.act_g + (size_t)s * p.act_stride;
  float* pr = p.act_p + (size_t)s * p.act_stride;
  __syncthreads();
  if (__ldcg(p.tinfo + 1) != 0) {              // rows missing: the step's samples are given up, every coefficient zero
    if (tid == 0) p.loss[s] = 0.f;
    for (int a = tid; a < na; a += TC3_THREADS) { pr[a] = 0.f; g[a] = 0.f; }
    for (int k = tid; k < H; k += TC3_THREADS) p.dh[(size_t)s * H + k] = 0.f;
    return;
  }
  const float M = sh_M, E = sh_E, fB = (float)p.B;
  const int ny = sh_ny;
  if (tid == TC3_THREADS - 1) {
    float sum = 0.f;
    const float logE = logf(E);
    for (int i = 0; i < nlab; ++i)
      if (lab[i] >= 0) sum += z[lab[i]] - M - logE;
    p.loss[s] = ny > 0 ? -sum / (float)ny : 0.f;
  }
  constexpr int U = 4;
  for (int a0 = tid; a0 < na; a0 += U * TC3_THREADS) {
    float zv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) zv[u] = a0 + u * TC3_THREADS < na ? __ldcg(z + a0 + u * TC3_THREADS) : 0.f;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int a = a0 + u * TC3_THREADS;
      if (a < na) {
        const float pa = expf(zv[u] - M) / E;
        pr[a] = pa;
        g[a] = pa / fB;
      }
    }
  }
  // sums over the chunks: `parts` threads per hidden unit, each a contiguous share of the chunks, added in order below
  for (int e = tid; e < parts * H; e += TC3_THREADS) {
    const int part = e / H, k = e - part * H;
    const int per = (np + parts - 1) / parts;
    const int b1 = min(np, (part + 1) * per);
    float S = 0.f;
#pragma unroll 8
    for (int b = part * per; b < b1; ++b) {
      const float f = fac[b];
      const float v = f != 0.f ? __ldcg(p.part + ((size_t)b * p.B + s) * ld + k) : 0.f;
      S = fmaf(f, v, S);
    }
    ps[e] = S;
  }
  __syncthreads();
  for (int k = tid; k < H; k += TC3_THREADS) {
    float S = 0.f, T = 0.f;
    for (int q = 0; q < parts; ++q) S += ps[q * H + k];
#pragma unroll 4
    for (int i = 0; i < nlab; ++i)
      if (lab[i] >= 0) T += p.W2[(size_t)ids[lab[i]] * H + k];
    const float v = (S / E - (ny > 0 ? T / (float)ny : 0.f)) / fB;
    p.dh[(size_t)s * H + k] = p.h[(size_t)s * H + k] > 0.f ? v : 0.f;
  }
  for (int i = tid; i < nlab; i += TC3_THREADS)
    if (lab[i] >= 0) g[lab[i]] = (pr[lab[i]] - 1.f / (float)ny) / fB;
}

// The touches of a tile's rows, row by row, in ascending sample order.  Per chunk of TL_CHUNK samples a bit per (row,
// sample) is set in shared memory; a row's words are then counted up, so that the place of an entry is known from the
// bits before its own whatever the order the entries are met in.  The tile's share of the list comes from a counter
// (where a tile's entries lie does not matter).
struct ListParams {
  const int *tstart, *seg;
  int* tinfo;
  const uint16_t* act_loc;
  const float* act_g;
  int2 *rinfo, *list;
  int B, act_stride, bstride, rows;      // rows: of a tile at most
};

__global__ void __launch_bounds__(TL_THREADS) k_tile_lists(const ListParams p) {
  extern __shared__ __align__(16) unsigned char tl_sm[];
  constexpr int NWD = TL_CHUNK / 32, LD = NWD + 1;
  uint32_t* mask = reinterpret_cast<uint32_t*>(tl_sm);                             // [rows][LD]
  int* start = reinterpret_cast<int*>(mask + (size_t)p.rows * LD);                 // [rows] where the row's next entries go
  int* cnt = start + p.rows;                                                       // [rows]
  uint16_t* pre = reinterpret_cast<uint16_t*>(cnt + p.rows);                       // [rows][LD]
  __shared__ int wsum[TL_WARPS];
  __shared__ int sh_base;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  griddep_launch_dependents();
  griddep_wait();
  const int nt = __ldcg(p.tinfo);
  const int nchunks = (p.B + TL_CHUNK - 1) / TL_CHUNK;
  for (int t = blockIdx.x; t < nt; t += gridDim.x) {
    const int r0 = __ldcg(p.tstart + t), nr = __ldcg(p.tstart + t + 1) - r0;
    // every entry of the samples [s0, s0 + TL_CHUNK) by some thread: f(sample, place, index); four runs side by side
    auto runs = [&](int s0, auto f) {
      const int s1 = min(p.B, s0 + TL_CHUNK);
      for (int sb = s0 + warp; sb < s1; sb += 32 * TL_WARPS) {
        const int ms = sb + lane * TL_WARPS;
        int ra = 0, rn = 0;
        if (ms < s1) {
          ra = __ldcg(p.seg + (size_t)t * p.bstride + ms);
          rn = __ldcg(p.seg + (size_t)(t + 1) * p.bstride + ms) - ra;
        }
        const int most = min(32, (s1 - sb + TL_WARPS - 1) / TL_WARPS);
        for (int i0 = 0; i0 < most; i0 += 4) {
          int loc[4], n[4];
          size_t at[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            n[u] = __shfl_sync(TFULL, rn, i0 + u);
            at[u] = (size_t)(sb + (i0 + u) * TL_WARPS) * p.act_stride + __shfl_sync(TFULL, ra, i0 + u);
            loc[u] = lane < n[u] ? (int)p.act_loc[at[u] + lane] : -1;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (loc[u] >= 0) f(sb + (i0 + u) * TL_WARPS, loc[u], at[u] + lane);
#pragma unroll
          for (int u = 0; u < 4; ++u)
            for (int c = 32 + lane; c < n[u]; c += 32) f(sb + (i0 + u) * TL_WARPS, (int)p.act_loc[at[u] + c], at[u] + c);
        }
      }
    };
    __syncthreads();                           // readers of the tile before are done
    for (int r = tid; r < nr; r += TL_THREADS) cnt[r] = 0;
    __syncthreads();
    if (nchunks > 1) {
      for (int ch = 0; ch < nchunks; ++ch) runs(ch * TL_CHUNK, [&](int, int loc, size_t) { atomicAdd(&cnt[loc], 1); });
      __syncthreads();
    }
    for (int ch = 0; ch < nchunks; ++ch) {
      for (int e = tid; e < nr * LD; e += TL_THREADS) mask[e] = 0u;
      __syncthreads();
      runs(ch * TL_CHUNK, [&](int s, int loc, size_t) { const int b = s - ch * TL_CHUNK; atomicOr(&mask[loc * LD + (b >> 5)], 1u << (b & 31)); });
      __syncthreads();
      int here = 0;                            // the row's entries in this chunk
      if (tid < nr) {
#pragma unroll 8
        for (int w = 0; w < NWD; ++w) {
          pre[tid * LD + w] = (uint16_t)here;
          here += __popc(mask[tid * LD + w]);
        }
      }
      if (ch == 0) {
        // the rows' places in the list: running sum of their counts from the tile's base
        const int mine = tid < nr ? (nchunks > 1 ? cnt[tid] : here) : 0;
        int incl = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const int o = __shfl_up_sync(TFULL, incl, d);
          if (lane >= d) incl += o;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        int before = 0, total = 0;
        for (int w = 0; w < TL_WARPS; ++w) {
          if (w < warp) before += wsum[w];
          total += wsum[w];
        }
        if (tid == 0) sh_base = atomicAdd(p.tinfo + 2, total);
        __syncthreads();
        if (tid < nr) {
          start[tid] = sh_base + before + incl - mine;
          p.rinfo[r0 + tid] = make_int2(start[tid], mine);
        }
      }
      __syncthreads();
      runs(ch * TL_CHUNK, [&](int s, int loc, size_t at) {
        const int b = s - ch * TL_CHUNK, w = b >> 5;
        const int to = start[loc] + pre[loc * LD + w] + __popc(mask[loc * LD + w] & ((1u << (b & 31)) - 1u));
        p.list[to] = make_int2(s, __float_as_int(__ldcg(p.act_g + at)));
      });
      __syncthreads();
      if (tid < nr) start[tid] += here;
    }
  }
}

cudaError_t launch_tiles_forward(Ctx* c, int batch, const int32_t* label_ptr, const int32_t* labels) {
  const int nw = (c->N + 31) / 32;
  int chunks, groups;
  tile_grid(c, batch, &chunks, &groups);
  const int step = call_step(c, batch);
  c->launches += 5;          // with the kernel before them they make one entry of the profile
  cudaError_t e = launch_dependent(k_tile_scan, dim3(1), dim3(TS_THREADS), 0, c->stream, (const uint32_t*)c->touch2, nw, step, chunks,
                                   c->wpre, c->tstart, c->tinfo, &c->dstate->n_own[c->t_host & 1][0]);
  if (e != cudaSuccess) return e;
  const int extra = (nw + 4 * TI_THREADS - 1) / (4 * TI_THREADS);
  e = launch_dependent(k_tile_index, dim3(batch + extra), dim3(TI_THREADS + 32), 0, c->stream, (const uint32_t*)c->touch2, (const int*)c->wpre,
                       (const int*)c->tstart, (const int*)c->tinfo, nw, batch, batch, (const int*)c->act_cnt,
                       (const int32_t*)c->act_ids, c->act_stride, label_ptr, labels, c->cfg.max_labels, c->act_loc, c->seg, c->trows, c->tlab);
  if (e != cudaSuccess) return e;
  TileParams p;
  p.W2 = c->W2; p.hdr2 = c->hdr2; p.h = c->h; p.trows = c->trows; p.tstart = c->tstart; p.tinfo = c->tinfo; p.seg = c->seg;
  p.act_loc = c->act_loc; p.act_z = c->act_z; p.part = c->tpart; p.st = c->dstate;
  p.B = batch; p.H = c->H; p.act_stride = c->act_stride; p.bstride = batch; p.chunks = chunks; p.gs = (batch + groups - 1) / groups;
  const int smem = (step + 31) * (c->H + 4) * 4;
  auto k = c->H <= 64 ? k_tile_forward<16, 1, 4> : c->H <= 128 ? k_tile_forward<16, 2, 4> : c->H <= 256 ? k_tile_forward<32, 2, 8>
           : c->H <= 512 ? k_tile_forward<32, 4, 4> : k_tile_forward<32, 8, 4>;
  if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024)) != cudaSuccess) return e;
  if ((e = launch_dependent(k, dim3(chunks, groups), dim3(TF_THREADS), (size_t)smem, c->stream, p)) != cudaSuccess) return e;
  CombineParams q;
  q.W2 = c->W2; q.h = c->h; q.part = c->tpart; q.act_z = c->act_z; q.label_ptr = label_ptr; q.act_ids = c->act_ids;
  q.act_cnt = c->act_cnt; q.tinfo = c->tinfo; q.tlab = c->tlab; q.act_p = c->act_p; q.act_g = c->act_g; q.dh = c->dh; q.loss = c->loss;
  q.touch = c->touch2; q.B = batch; q.H = c->H; q.act_stride = c->act_stride; q.chunks = chunks; q.nw = nw; q.max_labels = c->cfg.max_labels;
  const int parts = c->H >= TC3_THREADS ? 1 : TC3_THREADS / c->H;
  const size_t csm = (size_t)(((chunks + 3) & ~3) + parts * c->H + c->cfg.max_labels) * 4;
  if ((e = launch_dependent(k_tile_combine, dim3(batch), dim3(TC3_THREADS), csm, c->stream, q)) != cudaSuccess) return e;
  ListParams l;
  l.tstart = c->tstart; l.seg = c->seg; l.tinfo = c->tinfo; l.act_loc = c->act_loc; l.act_g = c->act_g; l.rinfo = c->rinfo; l.list = c->tlist;
  l.B = batch; l.act_stride = c->act_stride; l.bstride = batch; l.rows = step + 31;
  const size_t lsm = (size_t)(step + 31) * ((TL_CHUNK / 32 + 1) * 6 + 8);
  if ((e = cudaFuncSetAttribute(k_tile_lists, cudaFuncAttributeMaxDynamicSharedMemorySize, 112 * 1024)) != cudaSuccess) return e;
  return launch_dependent(k_tile_lists, dim3(2 * c->num_sms), dim3(TL_THREADS), lsm, c->stream, l);
}

}  // namespace dslide
