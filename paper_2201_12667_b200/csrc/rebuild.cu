// Initialisation and table (re)build (Algorithm 1: "Initialize layers with randomly generated
// weights", "Hash weights to hash tables", "Rebuild hash tables and hash functions"; Section 2.1
// phase 1; Section 3.1 "locally updated with a frequency schedule").
//
//   k_init_gauss   : weights ~ N(0, std^2) from the counter-based generator (Box-Muller).
//   k_draw_simhash / k_draw_dwta : the hash functions of rebuild count r.
//   k_hash_neurons* : the L bucket codes of every row of W2 (same functions as the queries) and
//                    the size of every bucket.
//   k_bucket_scan  : bucket sizes -> bucket offsets (one block per table).
//   k_sort_hist / k_sort_scan / k_sort_scatter : a stable least-significant-digit radix sort of the
//                    neuron ids of each table by bucket code, so that every bucket lists its
//                    neurons in ascending id (the first `cap` of them are what a query reads).
#include "common.cuh"

namespace dslide {

// ------------------------------------------------------------------ weights
__global__ void k_init_gauss(float* w, long long n, uint64_t seed, uint64_t stream_id, double std) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long step = (long long)gridDim.x * blockDim.x;
  for (; i < n; i += step) {
    uint64_t a = ctr_rng(seed, stream_id, 0, 2ull * (uint64_t)i);
    uint64_t b = ctr_rng(seed, stream_id, 0, 2ull * (uint64_t)i + 1ull);
    double u1 = ((double)(a >> 11) + 0.5) * (1.0 / 9007199254740992.0);
    double u2 = ((double)(b >> 11) + 0.5) * (1.0 / 9007199254740992.0);
    w[i] = (float)(std * sqrt(-2.0 * log(u1)) * cos(6.283185307179586476925 * u2));
  }
}

cudaError_t launch_init_gauss(Ctx* c, float* w, int64_t n, uint64_t stream_id) {
  if (n <= 0) return cudaSuccess;
  {
    LaunchScope ls(c, KID_INIT);
    k_init_gauss<<<c->num_sms * 8, 256, 0, c->stream>>>(w, n, c->cfg.seed, stream_id, (double)c->cfg.init_std);
  }
  return cudaGetLastError();
}

// ------------------------------------------------------------------ hash functions
// SimHash: projection f has fn_len distinct coordinates (partial Fisher-Yates over 0..H-1, then
// sorted ascending) and a sign per coordinate.  One thread per projection; H <= 1024.
__global__ void k_draw_simhash(int32_t* idx, int32_t* sign, int KL, int H, int m, uint64_t seed, uint64_t r) {
  int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= KL) return;
  short perm[1024];
  for (int i = 0; i < H; ++i) perm[i] = (short)i;
  for (int i = 0; i < m; ++i) {
    uint64_t u = ctr_rng(seed, RNG_HASH, r, (uint64_t)f * 2ull * (uint64_t)m + (uint64_t)i);
    int j = i + (int)(u % (uint64_t)(H - i));
    short tmp = perm[i]; perm[i] = perm[j]; perm[j] = tmp;
  }
  for (int i = 1; i < m; ++i) {      // insertion sort of the chosen coordinates
    short v = perm[i];
    int q = i;
    while (q > 0 && perm[q - 1] > v) { perm[q] = perm[q - 1]; --q; }
    perm[q] = v;
  }
  for (int i = 0; i < m; ++i) {
    uint64_t u = ctr_rng(seed, RNG_HASH, r, (uint64_t)f * 2ull * (uint64_t)m + (uint64_t)m + (uint64_t)i);
    idx[(size_t)f * m + i] = perm[i];
    sign[(size_t)f * m + i] = (u & 1ull) ? 1 : -1;
  }
}

// DWTA: ceil(K*L*bin / H) random permutations of the coordinates, concatenated; hash function f
// reads entries [f*bin, (f+1)*bin).  One block per permutation: the swap partner of every position is drawn by
// its own thread (the generator is counter-based), then one thread applies the swaps from the last position down.
constexpr int DRAW_THREADS = 128;
__global__ void __launch_bounds__(DRAW_THREADS) k_draw_dwta(int32_t* idx, long long total, int H, uint64_t seed, uint64_t r) {
  extern __shared__ int draw_sm[];          // [H] permutation, [H] swap partners
  int* perm = draw_sm;
  int* partner = draw_sm + H;
  const int q = blockIdx.x;
  for (int i = threadIdx.x; i < H; i += DRAW_THREADS) {
    perm[i] = i;
    const uint64_t u = ctr_rng(seed, RNG_HASH, r, (uint64_t)q * (uint64_t)H + (uint64_t)i);
    partner[i] = i >= 1 ? (int)(u % (uint64_t)(i + 1)) : 0;
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int i = H - 1; i >= 1; --i) {
      const int j = partner[i];
      const int tmp = perm[i]; perm[i] = perm[j]; perm[j] = tmp;
    }
  __syncthreads();
  for (int i = threadIdx.x; i < H; i += DRAW_THREADS) {
    const long long e = (long long)q * H + i;
    if (e < total) idx[e] = perm[i];
  }
}

// SimHash functions as the forward kernel reads them: [coordinate of the function][function], 16 bits each, top bit =
// minus, so that the threads of a warp (one function each) read side by side.
__global__ void k_pack_simhash(const int32_t* idx, const int32_t* sign, uint16_t* pk, int KL, int m) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= KL * m) return;
  const int i = e / KL, f = e - i * KL;
  pk[e] = (uint16_t)((idx[(size_t)f * m + i] & 0x7fff) | (sign[(size_t)f * m + i] > 0 ? 0 : 0x8000));
}

cudaError_t launch_pack_hash(Ctx* c) {
  if (c->cfg.hash_family != DSLIDE_SIMHASH || c->dense) return cudaSuccess;
  LaunchScope ls(c, KID_DRAW_HASH);
  const int n = c->KL * c->fn_len;
  k_pack_simhash<<<(n + 255) / 256, 256, 0, c->stream>>>(c->hash_idx, c->hash_sign, c->hash_pk, c->KL, c->fn_len);
  return cudaGetLastError();
}

cudaError_t launch_draw_hash(Ctx* c, int64_t r) {
  {
    LaunchScope ls(c, KID_DRAW_HASH);
    if (c->cfg.hash_family == DSLIDE_SIMHASH) {
      k_draw_simhash<<<(c->KL + 63) / 64, 64, 0, c->stream>>>(c->hash_idx, c->hash_sign, c->KL, c->H, c->fn_len,
                                                             c->cfg.seed, (uint64_t)r);
    } else {
      long long total = (long long)c->KL * c->fn_len;
      int nperm = (int)((total + c->H - 1) / c->H);
      k_draw_dwta<<<nperm, DRAW_THREADS, 2 * c->H * sizeof(int), c->stream>>>(c->hash_idx, total, c->H, c->cfg.seed, (uint64_t)r);
    }
  }
  const cudaError_t e = cudaGetLastError();
  return e != cudaSuccess ? e : launch_pack_hash(c);
}

// ------------------------------------------------------------------ LSH-sampled hidden layer
// Projections over the D input coordinates (Section 3.6: the hidden layer as a sparse layer; Algorithm 1 retrieves
// active neurons for every layer): entry (c, p) is +1, -1 or 0 with probability 1/6, 1/6, 2/3, drawn by itself from
// the counter-based generator.
__global__ void k_draw_proj1(int8_t* proj, long long n, uint64_t seed, uint64_t r) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long step = (long long)gridDim.x * blockDim.x;
  for (; i < n; i += step) {
    const uint64_t u = ctr_rng(seed, RNG_HASH1, r, (uint64_t)i) % 6ull;
    proj[i] = u == 0 ? 1 : (u == 1 ? -1 : 0);
  }
}

cudaError_t launch_draw_proj1(Ctx* c, int64_t r) {
  if (c->L1 <= 0) return cudaSuccess;
  LaunchScope ls(c, KID_DRAW_HASH);
  k_draw_proj1<<<c->num_sms * 8, 256, 0, c->stream>>>(c->proj1, (long long)c->D * c->KL1, c->cfg.seed, (uint64_t)r);
  return cudaGetLastError();
}

// Codes of the hidden neurons: neuron k's weight vector is column k of W1.  A block owns 32 neurons (the lanes) and
// 16 projections (four per warp) and walks the input coordinates in ascending order, because the sums are sequential
// like the oracle's.  Tiles of H1_CT coordinates pass through shared memory: the 128-byte pieces of the rows of W1
// by cp.async, two tiles deep; the projections' entries as floats (+1, -1, 0), so that one fused multiply-add per
// (coordinate, projection) adds +w, -w or nothing -- fma(+-1, w, s) rounds like s +- w, and fma(0, w, s) is s.
constexpr int H1_THREADS = 128;
constexpr int H1_CT = 128;        // coordinates per tile
constexpr int H1_PB = 16;         // projections per block
__global__ void __launch_bounds__(H1_THREADS)
k_hash_hidden(const float* __restrict__ W1, const int8_t* __restrict__ proj, unsigned char* bits, int D, int H, int KL1) {
  __shared__ __align__(16) float tw[2][H1_CT][32];
  __shared__ __align__(16) float tf[2][H1_CT][H1_PB];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k0 = blockIdx.x * 32, p0 = blockIdx.y * H1_PB;
  const int ntiles = (D + H1_CT - 1) / H1_CT;
  auto load_w = [&](int stage, int t) {        // 128 rows x 8 pieces of 16 bytes
    const int c0 = t * H1_CT;
    for (int e = tid; e < H1_CT * 8; e += H1_THREADS) {
      const int row = e >> 3, piece = e & 7;
      if (c0 + row < D && k0 + 4 * piece < H)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(&tw[stage][row][4 * piece])),
                     "l"(W1 + (size_t)(c0 + row) * H + k0 + 4 * piece) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // the projections' entries of a tile: thread = coordinate, 16 bytes each, held in registers until the tile's turn
  signed char pe[H1_PB];
  auto load_p = [&](int t) {
    const int c = t * H1_CT + tid;
#pragma unroll
    for (int q = 0; q < H1_PB; ++q) pe[q] = (c < D && p0 + q < KL1) ? (signed char)__ldg(proj + (size_t)c * KL1 + p0 + q) : (signed char)0;
  };
  float s[4] = {0.f, 0.f, 0.f, 0.f};
  load_w(0, 0);
  load_p(0);
  for (int t = 0; t < ntiles; ++t) {
    const int st = t & 1;
#pragma unroll
    for (int q = 0; q < H1_PB; ++q) tf[st][tid][q] = (float)pe[q];
    if (t + 1 < ntiles) {
      load_w(st ^ 1, t + 1);
      load_p(t + 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const int nc = min(H1_CT, D - t * H1_CT);
#pragma unroll 8
    for (int c = 0; c < nc; ++c) {
      const float w = tw[st][c][lane];
      const float4 e = *reinterpret_cast<const float4*>(&tf[st][c][4 * warp]);
      s[0] = __fmaf_rn(e.x, w, s[0]);
      s[1] = __fmaf_rn(e.y, w, s[1]);
      s[2] = __fmaf_rn(e.z, w, s[2]);
      s[3] = __fmaf_rn(e.w, w, s[3]);
    }
    __syncthreads();
  }
  const int k = k0 + lane;
  if (k < H)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int p = p0 + 4 * warp + q;
      if (p < KL1) bits[(size_t)p * H + k] = s[q] >= 0.f ? 1 : 0;
    }
}

// One block per table: codes from the bits, bucket sizes, offsets, and every neuron to its bucket's start plus the
// number of lower-numbered neurons with the same code (ascending ids inside a bucket).  H <= 1024.
__global__ void __launch_bounds__(1024)
k_tables1(const unsigned char* bits, uint32_t* codes, int32_t* off, int32_t* ids, int H, int K1) {
  extern __shared__ int t1_smem[];          // [H] codes, [2^K1 + 1] offsets
  int* scode = t1_smem;
  int* soff = t1_smem + H;
  const int t = blockIdx.x, nb = 1 << K1, tid = threadIdx.x;
  for (int b = tid; b <= nb; b += blockDim.x) soff[b] = 0;
  __syncthreads();
  for (int k = tid; k < H; k += blockDim.x) {
    int code = 0;
    for (int q = 0; q < K1; ++q) code |= (int)bits[(size_t)(t * K1 + q) * H + k] << q;
    scode[k] = code;
    codes[(size_t)t * H + k] = (uint32_t)code;
    atomicAdd(&soff[code + 1], 1);
  }
  __syncthreads();
  if (tid == 0) {
    int run = 0;
    for (int b = 0; b <= nb; ++b) { run += soff[b]; soff[b] = run; }
  }
  __syncthreads();
  int32_t* o = off + (size_t)t * (nb + 1);
  for (int b = tid; b <= nb; b += blockDim.x) o[b] = soff[b];
  for (int k = tid; k < H; k += blockDim.x) {
    const int code = scode[k];
    int before = 0;
    for (int j = 0; j < k; ++j) before += scode[j] == code ? 1 : 0;
    ids[(size_t)t * H + soff[code] + before] = k;
  }
}

cudaError_t launch_build_tables1(Ctx* c) {
  if (c->L1 <= 0) return cudaSuccess;
  unsigned char* bits = reinterpret_cast<unsigned char*>(c->codes1n + (size_t)c->L1 * c->H);     // [KL1][H] after the codes
  {
    LaunchScope ls(c, KID_HASH_NEURONS);
    dim3 grid((c->H + 31) / 32, (c->KL1 + H1_PB - 1) / H1_PB);
    k_hash_hidden<<<grid, H1_THREADS, 0, c->stream>>>(c->W1, c->proj1, bits, c->D, c->H, c->KL1);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int smem = (c->H + (1 << c->K1) + 1) * (int)sizeof(int);
  if (smem > 48 * 1024) {
    e = cudaFuncSetAttribute(k_tables1, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
  }
  LaunchScope ls(c, KID_BUCKET_SCAN);
  k_tables1<<<c->L1, 1024, smem, c->stream>>>(bits, c->codes1n, c->bucket1_off, c->bucket1_ids, c->H, c->K1);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ codes of all neurons
constexpr int HN_ROWS = 32;
constexpr int HN_THREADS = 256;
constexpr int HN_WARPS = HN_THREADS / 32;
constexpr int HN_FN_SMEM_MAX = 96 * 1024;    // hash-function tables larger than this stay in global memory

// A block stages HN_ROWS rows of W2 in shared memory (padded, so that 32 threads reading the same
// column of 32 different rows hit 32 banks) and evaluates the L DWTA codes of each row: lane = row, the
// warps share out the tables.  The hash functions sit in shared memory too, 16 bits per coordinate,
// read as warp-wide broadcasts.
// keys[t][j] = code of neuron j in table t.
template <bool FN_SMEM>
__global__ void __launch_bounds__(HN_THREADS)
k_hash_neurons(const float* __restrict__ W2, const int32_t* __restrict__ hidx, uint32_t* keys, int N, int H, int K, int L, int lg_bin, int fn_len) {
  extern __shared__ __align__(16) unsigned char hn_smem[];
  float* tile = reinterpret_cast<float*>(hn_smem);                    // [HN_ROWS][H + 1]
  const int ld = H + 1;
  unsigned short* fn = reinterpret_cast<unsigned short*>(hn_smem + (((size_t)HN_ROWS * ld * 4 + 15) & ~(size_t)15));
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nfn = K * L * fn_len;
  if (FN_SMEM) {
    for (int e = threadIdx.x; e < nfn; e += HN_THREADS) fn[e] = (unsigned short)hidx[e];
  }
  const int ntiles = (N + HN_ROWS - 1) / HN_ROWS;
  for (int tl = blockIdx.x; tl < ntiles; tl += gridDim.x) {
    const int j0 = tl * HN_ROWS;
    const int rows = min(HN_ROWS, N - j0);
    __syncthreads();
    {
      const int H4 = H >> 2, total4 = rows * H4;
      const float4* src = reinterpret_cast<const float4*>(W2 + (size_t)j0 * H);
      for (int e = threadIdx.x; e < total4; e += HN_THREADS) {
        const float4 x = __ldg(src + e);
        const int r = e / H4, k = (e - r * H4) << 2;
        float* d = tile + r * ld + k;
        d[0] = x.x; d[1] = x.y; d[2] = x.z; d[3] = x.w;
      }
    }
    __syncthreads();
    if (lane < rows) {
      const float* v = tile + lane * ld;
      for (int t = warp; t < L; t += HN_WARPS) {
        uint32_t code = 0;
#pragma unroll 2
        for (int k = 0; k < K; ++k) {
          const int f = t * K + k;
          int best = 0;
          float bv;
          if (FN_SMEM && fn_len == 8) {
            // bin of eight: the eight coordinates come in one 16-byte broadcast load
            const uint4 q = *reinterpret_cast<const uint4*>(fn + (size_t)f * 8);
            const float x0 = v[q.x & 0xffffu], x1 = v[q.x >> 16], x2 = v[q.y & 0xffffu], x3 = v[q.y >> 16];
            const float x4 = v[q.z & 0xffffu], x5 = v[q.z >> 16], x6 = v[q.w & 0xffffu], x7 = v[q.w >> 16];
            bv = x0;
            if (x1 > bv) { bv = x1; best = 1; }
            if (x2 > bv) { bv = x2; best = 2; }
            if (x3 > bv) { bv = x3; best = 3; }
            if (x4 > bv) { bv = x4; best = 4; }
            if (x5 > bv) { bv = x5; best = 5; }
            if (x6 > bv) { bv = x6; best = 6; }
            if (x7 > bv) { bv = x7; best = 7; }
          } else if (FN_SMEM) {
            const unsigned short* ix = fn + (size_t)f * fn_len;
            bv = v[ix[0]];
            for (int i = 1; i < fn_len; ++i) {
              const float x = v[ix[i]];
              if (x > bv) { bv = x; best = i; }
            }
          } else {
            const int32_t* ix = hidx + (size_t)f * fn_len;
            bv = v[__ldg(ix)];
            for (int i = 1; i < fn_len; ++i) {
              const float x = v[__ldg(ix + i)];
              if (x > bv) { bv = x; best = i; }
            }
          }
          code |= (uint32_t)best << (k * lg_bin);
        }
        keys[(size_t)t * N + j0 + lane] = code;
      }
    }
  }
}

// SimHash: R rows per lane (rows lane, lane + 32, ... of a tile of 32 R), interleaved per coordinate, so that one load of
// 4 R bytes fetches a coordinate of all of them, and its address and sign are worked out once for them.  A projection's sum
// is the sequential one of the definition: a fused multiply-add by plus or minus one per coordinate, two rows per
// instruction.  The tables' functions sit in shared memory, 16 bits per coordinate (top bit: minus), filled up to whole
// 16-byte words with a coordinate that is zero; blocks of another y take other tables, as many at a time as find room.
// Bound by the loads from shared memory (4 bytes per row, function and coordinate: 30 GB at 253,855 rows of 200 units and 450
// functions).  With one row per lane, as before, the instructions around the loads bound it: a rebuild of those rows took
// 2,814 us and now takes 1,506; 128 units 1,818 and 968; 20,011 rows of 1,024 units 6,757 and 3,839 (one row per lane
// here too, but 13 warps for one tile instead of eight).  Where a block that fills a multiprocessor has fewer tables at a time
// than it could have warps, the functions of a table are shared out between warps, and the code's bits meet in shared memory:
// 6 tables of 24 functions, 20,011 rows of 256 units 670 us with one row per lane, 723 with a warp per table, 630 so.
constexpr int HNS_SMEM = 224 * 1024;
constexpr int HNS_WARPS = 24;              // of a block that has a multiprocessor to itself
constexpr int HNS_MIN_TABLES = 8;          // more rows per lane only while the functions of so many tables fit beside the tile
template <int R, bool SPLIT>      // SPLIT: `parts` warps share a table's functions
__global__ void __launch_bounds__(1024)
k_hash_neurons_sim(const float* __restrict__ W2, const int32_t* __restrict__ hidx, const int32_t* __restrict__ hsign, uint32_t* keys, int N, int H, int K,
                   int L, int m, int per, int parts) {
  constexpr int ROWS = 32 * R, ES = 4 * R;
  extern __shared__ __align__(16) unsigned char hn_smem[];
  const int ld = H + 1;                                               // odd: a warp's loads of one coordinate spread over the banks
  const int mp = (m + 7) & ~7;
  unsigned short* fn = reinterpret_cast<unsigned short*>(hn_smem + (((size_t)32 * ld * ES + 15) & ~(size_t)15));
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int t0 = blockIdx.y * per, nt = min(L - t0, per);
  for (int e = threadIdx.x; e < nt * K * mp; e += blockDim.x) {
    const int f = e / mp, i = e - f * mp;
    const size_t at = (size_t)(t0 * K + f) * m + i;
    fn[e] = i < m ? (unsigned short)(hidx[at] | (hsign[at] > 0 ? 0 : 0x8000)) : (unsigned short)H;
  }
  if (threadIdx.x < 32)
    for (int u = 0; u < R; ++u) reinterpret_cast<float*>(hn_smem)[(threadIdx.x * ld + H) * R + u] = 0.f;
  uint32_t* codes = reinterpret_cast<uint32_t*>(fn + (size_t)per * K * mp);      // SPLIT: [table][row], put together from the warps' bits
  if (SPLIT)
    for (int e = threadIdx.x; e < nt * ROWS; e += blockDim.x) codes[e] = 0u;
  const unsigned char* v = hn_smem + (size_t)lane * ld * ES;
  const int ntiles = (N + ROWS - 1) / ROWS;
  for (int tl = blockIdx.x; tl < ntiles; tl += gridDim.x) {
    const int j0 = tl * ROWS;
    const int rows = min(ROWS, N - j0);
    __syncthreads();
    // a thread takes one coordinate of one lane's rows: reads run along a row, one vector store places them
    for (int g = warp; g < 32; g += nwarps)
      for (int k = lane; k < H; k += 32) {
        float x[R];
#pragma unroll
        for (int u = 0; u < R; ++u) x[u] = g + 32 * u < rows ? __ldg(W2 + (size_t)(j0 + g + 32 * u) * H + k) : 0.f;
        float* to = reinterpret_cast<float*>(hn_smem) + ((size_t)g * ld + k) * R;
        if (R == 4) *reinterpret_cast<float4*>(to) = make_float4(x[0], x[1 % R], x[2 % R], x[3 % R]);
        else if (R == 2) *reinterpret_cast<float2*>(to) = make_float2(x[0], x[1 % R]);
        else *to = x[0];
      }
    __syncthreads();
    for (int it = warp; it < (SPLIT ? nt * parts : nt); it += nwarps) {
      const int t = SPLIT ? it / parts : it, part = it - t * parts, k1 = SPLIT ? (part + 1) * K / parts : K;
      uint32_t code[R];
#pragma unroll
      for (int u = 0; u < R; ++u) code[u] = 0u;
      for (int k = SPLIT ? part * K / parts : 0; k < k1; ++k) {
        const uint4* q4 = reinterpret_cast<const uint4*>(fn + (size_t)(t * K + k) * mp);
        unsigned long long s0 = 0ull, s1 = 0ull;
        float s = 0.f;
        for (int i0 = 0; i0 < mp / 8; ++i0) {
          const uint4 q = q4[i0];
          const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const uint32_t e = i & 1 ? w[i >> 1] >> 16 : w[i >> 1];
            const uint32_t sg = ((i & 1 ? w[i >> 1] : w[i >> 1] << 16) & 0x80000000u) | 0x3f800000u;
            const unsigned char* at = v + (e & 0x7fffu) * ES;
            const unsigned long long pm = ((unsigned long long)sg << 32) | sg;
            if (R == 4) {
              const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(at);
              asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(s0) : "l"(x.x), "l"(pm));
              asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(s1) : "l"(x.y), "l"(pm));
            } else if (R == 2) {
              asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(s0) : "l"(*reinterpret_cast<const unsigned long long*>(at)), "l"(pm));
            } else {
              s = fmaf(*reinterpret_cast<const float*>(at), __uint_as_float(sg), s);
            }
          }
        }
        const float sum[4] = {R == 1 ? s : __uint_as_float((unsigned)s0), __uint_as_float((unsigned)(s0 >> 32)), __uint_as_float((unsigned)s1),
                              __uint_as_float((unsigned)(s1 >> 32))};
#pragma unroll
        for (int u = 0; u < R; ++u) code[u] |= (sum[u] >= 0.f ? 1u : 0u) << k;
      }
      if (SPLIT) {
#pragma unroll
        for (int u = 0; u < R; ++u) atomicOr(codes + t * ROWS + 32 * u + lane, code[u]);
        continue;
      }
#pragma unroll
      for (int u = 0; u < R; ++u)
        if (lane + 32 * u < rows) keys[(size_t)(t0 + t) * N + j0 + 32 * u + lane] = code[u];
    }
    if (SPLIT) {
      __syncthreads();
      for (int e = threadIdx.x; e < nt * ROWS; e += blockDim.x) {
        const int t = e / ROWS, r = e - t * ROWS;
        if (r < rows) keys[(size_t)(t0 + t) * N + j0 + r] = codes[e];
        codes[e] = 0u;
      }
    }
  }
}

// DWTA with bins of eight, hash functions in shared memory: 2 * RP rows per lane (rows lane, lane + 32, ... of a tile of
// 64 * RP), interleaved per coordinate, so that one 8- or 16-byte load fetches a coordinate of all of them and the
// address arithmetic is shared; the function table holds byte offsets.
//
// The winner of a bin is found without a chain of compare-and-select (three instructions per value on the half-rate
// pipe, which bounded the kernel): m = the maximum of the eight (three-input maxima); d_i = (x_i - m) 2^40 by one
// multiply-add, exactly zero where x_i equals m and at most -2^-109 elsewhere; t_i = d_i 2^120 - i, which is -i at the
// winners and below -2^11 elsewhere; so the maximum of the t_i is minus the lowest winning position.  The multiply-adds
// take two rows per instruction.  A winner's t lies in [-7, 0].  Where a value is not a number, infinite or beyond 2^87 a
// bin's maximum may be below -7 or not a number, and where all eight are below -2^87 it may be plus infinity (the code is
// then minus infinity): such a row's table is done again by the chain.  Bound now by the loads from shared memory (a value is read
// K L 8 / H times: 6.4 GB for 670,091 rows of 128 units and 300 functions).
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
  float d;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ float max8_nan(float a, float b, float c, float d, float e, float f, float g, float h) {
  float r = max3_nan(max3_nan(a, b, c), d, e);
  r = max3_nan(r, f, g);
  asm("max.NaN.f32 %0, %0, %1;" : "+f"(r) : "f"(h));
  return r;
}
__device__ __forceinline__ unsigned long long fma_pair(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ unsigned long long pair_of(float lo, float hi) {
  return ((unsigned long long)__float_as_uint(hi) << 32) | __float_as_uint(lo);
}
__device__ __forceinline__ float pair_lo(unsigned long long v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float pair_hi(unsigned long long v) { return __uint_as_float((unsigned)(v >> 32)); }

constexpr int HN8_WARPS_MAX = 16;

template <int RP>
__global__ void __launch_bounds__(32 * HN8_WARPS_MAX)
k_hash_neurons_dwta8(const float* __restrict__ W2, const int32_t* __restrict__ hidx, uint32_t* keys, int N, int H, int K, int L) {
  constexpr int ROWS = 64 * RP, ES = 8 * RP;                          // rows of a tile, bytes of a coordinate of a lane's rows
  extern __shared__ __align__(16) unsigned char hn_smem[];
  const int ld = H + 1;                                               // odd: a warp's loads of one coordinate spread over the banks
  uint32_t* fn = reinterpret_cast<uint32_t*>(hn_smem + (((size_t)32 * ld * ES + 15) & ~(size_t)15));
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  for (int e = threadIdx.x; e < K * L * 8; e += blockDim.x) fn[e] = (uint32_t)hidx[e] * ES;
  const unsigned char* v = hn_smem + (size_t)lane * ld * ES;
  const unsigned long long S = pair_of(0x1p40f, 0x1p40f), BIG = pair_of(0x1p120f, 0x1p120f);
  const int ntiles = (N + ROWS - 1) / ROWS;
  for (int tl = blockIdx.x; tl < ntiles; tl += gridDim.x) {
    const int j0 = tl * ROWS;
    const int rows = min(ROWS, N - j0);
    __syncthreads();
    // a thread takes one coordinate of one lane's rows: reads run along a row, one vector store places them
    for (int g = warp; g < 32; g += nwarps)
      for (int k = lane; k < H; k += 32) {
        float x[2 * RP];
#pragma unroll
        for (int u = 0; u < 2 * RP; ++u) x[u] = g + 32 * u < rows ? __ldg(W2 + (size_t)(j0 + g + 32 * u) * H + k) : 0.f;
        unsigned char* to = hn_smem + ((size_t)g * ld + k) * ES;
        if (RP == 2) *reinterpret_cast<float4*>(to) = make_float4(x[0], x[1], x[2 * RP - 2], x[2 * RP - 1]);
        else *reinterpret_cast<float2*>(to) = make_float2(x[0], x[1]);
      }
    __syncthreads();
    for (int t = warp; t < L; t += nwarps) {
      unsigned long long code[RP];
      float worst = 0.f;
      float scale = -1.f;
#pragma unroll
      for (int r = 0; r < RP; ++r) code[r] = 0ull;
      for (int k = 0; k < K; ++k) {
        const uint4 qa = *reinterpret_cast<const uint4*>(fn + (size_t)(t * K + k) * 8);
        const uint4 qb = *reinterpret_cast<const uint4*>(fn + (size_t)(t * K + k) * 8 + 4);
        const uint32_t q[8] = {qa.x, qa.y, qa.z, qa.w, qb.x, qb.y, qb.z, qb.w};
        unsigned long long x[8][RP];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if (RP == 2) {
            const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(v + q[i]);
            x[i][0] = w.x; x[i][RP - 1] = w.y;
          } else {
            x[i][0] = *reinterpret_cast<const unsigned long long*>(v + q[i]);
          }
        }
        const unsigned long long sc = pair_of(scale, scale);
#pragma unroll
        for (int r = 0; r < RP; ++r) {
          const float ma = max8_nan(pair_lo(x[0][r]), pair_lo(x[1][r]), pair_lo(x[2][r]), pair_lo(x[3][r]), pair_lo(x[4][r]),
                                    pair_lo(x[5][r]), pair_lo(x[6][r]), pair_lo(x[7][r]));
          const float mb = max8_nan(pair_hi(x[0][r]), pair_hi(x[1][r]), pair_hi(x[2][r]), pair_hi(x[3][r]), pair_hi(x[4][r]),
                                    pair_hi(x[5][r]), pair_hi(x[6][r]), pair_hi(x[7][r]));
          const unsigned long long nm = pair_of((0.f - ma) * 0x1p40f, (0.f - mb) * 0x1p40f);      // 0 - m: a zero of either sign gives +0
          unsigned long long d[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) d[i] = fma_pair(fma_pair(x[i][r], S, nm), BIG, pair_of(-(float)i, -(float)i));
          const float ta = max8_nan(pair_lo(d[0]), pair_lo(d[1]), pair_lo(d[2]), pair_lo(d[3]), pair_lo(d[4]), pair_lo(d[5]), pair_lo(d[6]), pair_lo(d[7]));
          const float tb = max8_nan(pair_hi(d[0]), pair_hi(d[1]), pair_hi(d[2]), pair_hi(d[3]), pair_hi(d[4]), pair_hi(d[5]), pair_hi(d[6]), pair_hi(d[7]));
          asm("min.NaN.f32 %0, %0, %1, %2;" : "+f"(worst) : "f"(ta), "f"(tb));
          code[r] = fma_pair(pair_of(ta, tb), sc, code[r]);          // minus position times minus 8^k: exact below 2^24
        }
        scale *= 8.f;
      }
      uint32_t c[2 * RP];
#pragma unroll
      for (int r = 0; r < RP; ++r) { c[2 * r] = __float2uint_rn(pair_lo(code[r])); c[2 * r + 1] = __float2uint_rn(pair_hi(code[r])); }
      bool sure = worst >= -7.f;
#pragma unroll
      for (int r = 0; r < RP; ++r) sure = sure && pair_lo(code[r]) >= 0.f && pair_hi(code[r]) >= 0.f;
      if (!sure) {                                                     // rare: see above
        for (int u = 0; u < 2 * RP; ++u) {
          uint32_t cc = 0;
          for (int k = 0; k < K; ++k) {
            const uint32_t* q = fn + (size_t)(t * K + k) * 8;
            int best = 0;
            float bv = reinterpret_cast<const float*>(v + q[0])[u];
            for (int i = 1; i < 8; ++i) {
              const float y = reinterpret_cast<const float*>(v + q[i])[u];
              if (y > bv) { bv = y; best = i; }
            }
            cc |= (uint32_t)best << (3 * k);
          }
          c[u] = cc;
        }
      }
#pragma unroll
      for (int u = 0; u < 2 * RP; ++u)
        if (lane + 32 * u < rows) keys[(size_t)t * N + j0 + 32 * u + lane] = c[u];
    }
  }
}

// Counting as a pass of its own (the counters of 2^21 buckets x 64 tables are half a gigabyte): the blocks walk table
// after table, so that the counters being incremented at any moment are those of one or two tables and the atomics stay
// in L2.  ranks[t][j] = arrivals before j in its bucket.
__global__ void __launch_bounds__(256) k_count_ranks(const uint32_t* keys, uint32_t* ranks, int32_t* counts, int N, long long nb) {
  const int t = blockIdx.y;
  const uint32_t* k = keys + (size_t)t * N;
  uint32_t* r = ranks + (size_t)t * N;
  int32_t* cnt = counts + (size_t)t * (size_t)(nb + 1) + 1;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < N; j += gridDim.x * blockDim.x) {
    r[j] = (uint32_t)atomicAdd(cnt + k[j], 1);
  }
}

// counts[t][0] = 0, counts[t][c + 1] = size of bucket c  ->  inclusive running sum = bucket offsets.
// Two kernels over chunks of BS_CHUNK counters: the sum of every chunk, then per chunk the sum of the
// table's earlier chunks plus a scan inside the chunk.
constexpr int ORD_SMALL = 16;     // buckets up to this size are put in order in registers
constexpr int ORD_BLOCK = 4096;   // up to this size by one block in shared memory
constexpr int BS_THREADS = 256;
constexpr int BS_PER = 16;
constexpr int BS_CHUNK = BS_THREADS * BS_PER;

__global__ void __launch_bounds__(BS_THREADS) k_bucket_sums(const int32_t* off, long long nb, int32_t* part, int nchunks) {
  __shared__ int sh[BS_THREADS / 32];
  const int32_t* o = off + (size_t)blockIdx.y * (size_t)(nb + 1);
  const long long n = nb + 1, base = (long long)blockIdx.x * BS_CHUNK;
  int sum = 0;
#pragma unroll
  for (int u = 0; u < BS_PER; ++u) {
    const long long i = base + threadIdx.x + (long long)u * BS_THREADS;
    sum += i < n ? o[i] : 0;
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    int tot = 0;
    for (int w = 0; w < BS_THREADS / 32; ++w) tot += sh[w];
    part[(size_t)blockIdx.y * nchunks + blockIdx.x] = tot;
  }
}

// With cnt != null the buckets of more than min_n (>= ORD_SMALL) ids are entered in the lists of the block-wide and
// the ordered-pass ordering kernels on the way (cnt[0] / cnt[1] are the lists' lengths).
__global__ void __launch_bounds__(BS_THREADS) k_bucket_scan(int32_t* off, long long nb, const int32_t* part, int nchunks,
                                                            int min_n, int2* mid, int2* big, int* cnt) {
  __shared__ int sh[BS_THREADS / 32 + 1];
  int32_t* o = off + (size_t)blockIdx.y * (size_t)(nb + 1);
  const long long n = nb + 1, base = (long long)blockIdx.x * BS_CHUNK;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // everything before this chunk
  int before = 0;
  for (int c = threadIdx.x; c < (int)blockIdx.x; c += BS_THREADS) before += part[(size_t)blockIdx.y * nchunks + c];
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) before += __shfl_xor_sync(0xffffffffu, before, d);
  if (lane == 0) sh[warp] = before;
  __syncthreads();
  before = 0;
  for (int w = 0; w < BS_THREADS / 32; ++w) before += sh[w];
  __syncthreads();
  // the chunk itself: every warp owns BS_PER * 32 consecutive counters and walks them 32 at a time
  const long long wbase = base + (long long)warp * (BS_PER * 32);
  int v[BS_PER];
  int wsum = 0;
#pragma unroll
  for (int u = 0; u < BS_PER; ++u) {
    const long long i = wbase + u * 32 + lane;
    v[u] = i < n ? o[i] : 0;
    wsum += v[u];
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) wsum += __shfl_xor_sync(0xffffffffu, wsum, d);
  if (lane == 0) sh[warp] = wsum;
  __syncthreads();
  int run = before;
  for (int w = 0; w < warp; ++w) run += sh[w];
#pragma unroll
  for (int u = 0; u < BS_PER; ++u) {
    int incl = v[u];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      int x = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += x;
    }
    const long long i = wbase + u * 32 + lane;
    if (i < n) o[i] = run + incl;
    if (cnt && i >= 1 && i < n && v[u] > min_n) {          // word i counts bucket i - 1
      if (v[u] <= ORD_BLOCK) mid[atomicAdd(cnt, 1)] = make_int2((int)blockIdx.y, (int)(i - 1));
      else big[atomicAdd(cnt + 1, 1)] = make_int2((int)blockIdx.y, (int)(i - 1));
    }
    run += __shfl_sync(0xffffffffu, incl, 31);
  }
}

// ------------------------------------------------------------------ stable LSD radix sort, per table
constexpr int SORT_THREADS = 512;
constexpr int SORT_WARPS = SORT_THREADS / 32;
constexpr int SORT_TILE = 8192;                      // elements per block
constexpr int SORT_SUB = SORT_TILE / SORT_WARPS;     // contiguous elements per warp
constexpr int SORT_ITERS = SORT_SUB / 32;            // groups of 32 keys a warp walks, all fetched up front
constexpr int SORT_MAX_WIDTH = 9;                    // bits per pass

// hist[t][digit][tile] = number of keys of that digit in the tile.
__global__ void __launch_bounds__(SORT_THREADS)
k_sort_hist(const uint32_t* keys, int32_t* hist, int N, int tiles, int shift, int width) {
  __shared__ int cnt[1 << SORT_MAX_WIDTH];
  const int radix = 1 << width, t = blockIdx.y, tl = blockIdx.x;
  for (int d = threadIdx.x; d < radix; d += SORT_THREADS) cnt[d] = 0;
  __syncthreads();
  const uint32_t* k = keys + (size_t)t * N;
  const int beg = tl * SORT_TILE, end = min(N, beg + SORT_TILE);
  for (int i = beg + threadIdx.x; i < end; i += SORT_THREADS) atomicAdd(&cnt[(k[i] >> shift) & (radix - 1)], 1);
  __syncthreads();
  for (int d = threadIdx.x; d < radix; d += SORT_THREADS) hist[((size_t)t * radix + d) * tiles + tl] = cnt[d];
}

// Exclusive scan of hist[t][*][*] in (digit, tile) order: where each tile's run of each digit starts.
__global__ void __launch_bounds__(1024) k_sort_scan(int32_t* hist, int n) {
  __shared__ int sh[33];
  int32_t* o = hist + (size_t)blockIdx.x * n;
  const int chunk = (n + 1023) / 1024;
  const int beg = min(n, (int)threadIdx.x * chunk), end = min(n, beg + chunk);
  int sum = 0;
  for (int i = beg; i < end; ++i) sum += o[i];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = sum;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    int v = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += v;
  }
  if (lane == 31) sh[warp] = incl;
  __syncthreads();
  if (threadIdx.x == 0) {
    int run = 0;
    for (int w = 0; w < 32; ++w) { int c = sh[w]; sh[w] = run; run += c; }
  }
  __syncthreads();
  int run = incl - sum + sh[warp];
  for (int i = beg; i < end; ++i) { int c = o[i]; o[i] = run; run += c; }
}

// Each warp owns a contiguous part of the tile and walks it in order, 32 keys at a time; equal
// digits inside a group of 32 are ranked by lane with a match mask, so the order of equal digits is
// kept.  All of a warp's keys (and values) are fetched before the walk.  The walk places the elements
// in shared memory in digit order; they are then written out in that order, so that a warp's stores
// cover a few contiguous runs instead of 32 scattered words.
// vals_in == nullptr means the value of element i is i (first pass).  keys_out may be nullptr
// (last pass).
constexpr int SORT_RADIX_MAX = 1 << SORT_MAX_WIDTH;
constexpr int SORT_SMEM = (2 * SORT_TILE + SORT_WARPS * SORT_RADIX_MAX + 2 * SORT_RADIX_MAX + 64) * 4;

__global__ void __launch_bounds__(SORT_THREADS, 2)
k_sort_scatter(const uint32_t* keys_in, const int32_t* vals_in, uint32_t* keys_out, int32_t* vals_out,
               const int32_t* hist, int N, int tiles, int shift, int width) {
  extern __shared__ __align__(16) int ss_smem[];
  uint32_t* skey = reinterpret_cast<uint32_t*>(ss_smem);                 // [SORT_TILE] the tile in digit order
  int* sval = ss_smem + SORT_TILE;                                       // [SORT_TILE]
  int* offs = ss_smem + 2 * SORT_TILE;                                   // [SORT_WARPS][radix] cursor of (warp, digit) in the tile
  int* gbase = offs + SORT_WARPS * SORT_RADIX_MAX;                       // [radix] where the tile's run of a digit starts globally
  int* tbase = gbase + SORT_RADIX_MAX;                                   // [radix] where it starts inside the tile
  int* sh = tbase + SORT_RADIX_MAX;                                      // [33] scan scratch
  const int radix = 1 << width, t = blockIdx.y, tl = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t* kin = keys_in + (size_t)t * N;
  const int32_t* vin = vals_in ? vals_in + (size_t)t * N : nullptr;
  uint32_t* kout = keys_out ? keys_out + (size_t)t * N : nullptr;
  int32_t* vout = vals_out + (size_t)t * N;
  const int tbeg = tl * SORT_TILE, tn = min(SORT_TILE, N - tbeg);
  const int wbeg = min(N, tbeg + warp * SORT_SUB), wend = min(N, wbeg + SORT_SUB);

  uint32_t key[SORT_ITERS];
#pragma unroll
  for (int it = 0; it < SORT_ITERS; ++it) {
    const int i = wbeg + it * 32 + lane;
    key[it] = i < wend ? kin[i] : 0u;
  }
  int* myoffs = offs + warp * SORT_RADIX_MAX;
  for (int d = lane; d < radix; d += 32) myoffs[d] = 0;
  __syncwarp();
  // walk 1: rank of every element among the warp's elements of the same digit (counts fall out at the end)
  unsigned short lrank[SORT_ITERS];
#pragma unroll
  for (int it = 0; it < SORT_ITERS; ++it) {
    const bool live = wbeg + it * 32 + lane < wend;
    const int digit = live ? (int)((key[it] >> shift) & (radix - 1)) : radix + lane;   // dead lanes match nobody
    const unsigned peers = __match_any_sync(0xffffffffu, digit);
    const int rank = __popc(peers & ((1u << lane) - 1u));
    int base = 0;
    if (live) base = myoffs[digit];
    __syncwarp();
    if (live && rank == 0) myoffs[digit] = base + __popc(peers);
    __syncwarp();
    lrank[it] = (unsigned short)(base + rank);
  }
  __syncthreads();
  // per digit: the tile's count, the warps' starts relative to the digit's run, the global start of the run
  int cnt[(SORT_RADIX_MAX + SORT_THREADS - 1) / SORT_THREADS];
#pragma unroll
  for (int u = 0; u < (SORT_RADIX_MAX + SORT_THREADS - 1) / SORT_THREADS; ++u) {
    const int d = threadIdx.x + u * SORT_THREADS;
    cnt[u] = 0;
    if (d < radix) {
      int run = 0;
      for (int w = 0; w < SORT_WARPS; ++w) { int c = offs[w * SORT_RADIX_MAX + d]; offs[w * SORT_RADIX_MAX + d] = run; run += c; }
      cnt[u] = run;
      gbase[d] = hist[((size_t)t * radix + d) * tiles + tl];
    }
  }
  // exclusive scan of the counts over the digits (digit d lives in thread d % SORT_THREADS, round d / SORT_THREADS)
  int carry = 0;
#pragma unroll
  for (int u = 0; u < (SORT_RADIX_MAX + SORT_THREADS - 1) / SORT_THREADS; ++u) {
    int incl = cnt[u];
#pragma unroll
    for (int dd = 1; dd < 32; dd <<= 1) {
      int x = __shfl_up_sync(0xffffffffu, incl, dd);
      if (lane >= dd) incl += x;
    }
    __syncthreads();
    if (lane == 31) sh[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      int w = lane < SORT_WARPS ? sh[lane] : 0, wi = w;
#pragma unroll
      for (int dd = 1; dd < 32; dd <<= 1) {
        int x = __shfl_up_sync(0xffffffffu, wi, dd);
        if (lane >= dd) wi += x;
      }
      if (lane < SORT_WARPS) sh[lane] = wi - w;
      if (lane == 31) sh[32] = wi;
    }
    __syncthreads();
    const int d = threadIdx.x + u * SORT_THREADS;
    if (d < radix) tbase[d] = carry + sh[warp] + incl - cnt[u];
    carry += sh[32];
  }
  __syncthreads();
  // walk 2: place the elements in digit order in shared memory
#pragma unroll
  for (int it = 0; it < SORT_ITERS; ++it) {
    const int i = wbeg + it * 32 + lane;
    if (i < wend) {
      const int digit = (int)((key[it] >> shift) & (radix - 1));
      const int lpos = tbase[digit] + myoffs[digit] + (int)lrank[it];
      skey[lpos] = key[it];
      sval[lpos] = vin ? vin[i] : i;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < tn; i += SORT_THREADS) {
    const uint32_t k = skey[i];
    const int d = (int)((k >> shift) & (radix - 1));
    const int g = gbase[d] + (i - tbase[d]);
    if (kout) kout[g] = k;
    vout[g] = sval[i];
  }
}

// ------------------------------------------------------------------ wide codes: partition, then place in shared memory
// Codes wider than one radix digit: the ids of a table are first partitioned by the upper bits of their codes (about a
// thousand ids per part; order inside a part does not matter), as words that hold the lower bits of the code and the
// id.  A block then takes a part: counts its buckets, writes their offsets, places the ids in shared memory and writes
// them out in one run.  So neither a counter nor an id goes to memory as a scattered 4-byte access (33.5 M of each at
// 670,091 neurons x 50 tables were what the placement by rank of arrival cost), and the offsets come out with it.
// Buckets larger than the cap are put in ascending order afterwards (k_order_*), as on the other path.
constexpr int PT_THREADS = 512;
constexpr int PT_TILE = 6144;
constexpr int PT_PER = PT_TILE / PT_THREADS;
constexpr int PT_HIST = 32768;                      // ids that a block counts
constexpr int PT_MAX_UP = 10, PT_MAX_LOW = 11;      // upper and lower bits of a code at most
constexpr int PP_THREADS = 256, PP_CAP = 4096;      // ids of a part that fit shared memory

__global__ void __launch_bounds__(PT_THREADS) k_part_hist(const uint32_t* keys, int* total, int N, int low, int up) {
  __shared__ int cnt[1 << PT_MAX_UP];
  const int t = blockIdx.y, P = 1 << up;
  griddep_launch_dependents();
  for (int d = threadIdx.x; d < P; d += PT_THREADS) cnt[d] = 0;
  __syncthreads();
  griddep_wait();
  const uint32_t* k = keys + (size_t)t * N;
  const int beg = blockIdx.x * PT_HIST, end = min(N, beg + PT_HIST);
  for (int i0 = beg + threadIdx.x; i0 < end; i0 += 8 * PT_THREADS) {
    uint32_t c[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) c[u] = i0 + u * PT_THREADS < end ? k[i0 + u * PT_THREADS] : 0u;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (i0 + u * PT_THREADS < end) atomicAdd(&cnt[c[u] >> low], 1);
  }
  __syncthreads();
  for (int d = threadIdx.x; d < P; d += PT_THREADS)
    if (cnt[d]) atomicAdd(&total[t * P + d], cnt[d]);
}

// One block per table: where the parts start (base[t][P + 1]) and the cursors that hand out their space.
__global__ void __launch_bounds__(1 << PT_MAX_UP) k_part_scan(int* total, int* base, int up) {
  __shared__ int sh[32];
  const int P = 1 << up, t = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  griddep_launch_dependents();
  griddep_wait();
  const int mine = tid < P ? total[t * P + tid] : 0;
  int incl = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += o;
  }
  if (lane == 31) sh[warp] = incl;
  __syncthreads();
  int before = 0;
  for (int w = 0; w < warp; ++w) before += sh[w];
  if (tid < P) {
    base[t * (P + 1) + tid] = before + incl - mine;
    total[t * P + tid] = before + incl - mine;
    if (tid == P - 1) base[t * (P + 1) + P] = before + incl;
  }
}

__global__ void __launch_bounds__(PT_THREADS, 4) k_part_scatter(const uint32_t* keys, int* cursor, uint32_t* out, int N, int low, int up, int id_bits) {
  __shared__ int cnt[1 << PT_MAX_UP], at[1 << PT_MAX_UP];      // of a part: the tile's ids; where they go globally minus where they are in the tile
  __shared__ uint32_t word[PT_TILE];
  __shared__ uint16_t part[PT_TILE];
  __shared__ int sh[PT_THREADS / 32];
  const int t = blockIdx.y, P = 1 << up, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  griddep_launch_dependents();
  for (int d = tid; d < P; d += PT_THREADS) cnt[d] = 0;
  __syncthreads();
  griddep_wait();
  const uint32_t* k = keys + (size_t)t * N;
  const int beg = blockIdx.x * PT_TILE, n = min(PT_TILE, N - beg);
  uint32_t key[PT_PER];
#pragma unroll
  for (int u = 0; u < PT_PER; ++u) {
    const int i = u * PT_THREADS + tid;
    key[u] = i < n ? k[beg + i] : 0u;
  }
#pragma unroll
  for (int u = 0; u < PT_PER; ++u)
    if (u * PT_THREADS + tid < n) atomicAdd(&cnt[key[u] >> low], 1);
  __syncthreads();
  // running sum over the parts (two per thread at most), and the tile's space in every part
  int c0 = 2 * tid < P ? cnt[2 * tid] : 0, c1 = 2 * tid + 1 < P ? cnt[2 * tid + 1] : 0;
  int incl = c0 + c1;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += o;
  }
  if (lane == 31) sh[warp] = incl;
  __syncthreads();
  int run = incl - c0 - c1;
  for (int w = 0; w < warp; ++w) run += sh[w];
  if (2 * tid < P) {
    cnt[2 * tid] = run;
    at[2 * tid] = (c0 ? atomicAdd(&cursor[t * P + 2 * tid], c0) : 0) - run;
  }
  if (2 * tid + 1 < P) {
    cnt[2 * tid + 1] = run + c0;
    at[2 * tid + 1] = (c1 ? atomicAdd(&cursor[t * P + 2 * tid + 1], c1) : 0) - (run + c0);
  }
  __syncthreads();
  const uint32_t lmask = (1u << low) - 1u;
#pragma unroll
  for (int u = 0; u < PT_PER; ++u) {
    const int i = u * PT_THREADS + tid;
    if (i < n) {
      const int d = (int)(key[u] >> low), to = atomicAdd(&cnt[d], 1);
      word[to] = ((key[u] & lmask) << id_bits) | (uint32_t)(beg + i);
      part[to] = (uint16_t)d;
    }
  }
  __syncthreads();
  uint32_t* o = out + (size_t)t * N;
#pragma unroll
  for (int u = 0; u < PT_PER; ++u) {
    const int i = u * PT_THREADS + tid;
    if (i < n) o[at[part[i]] + i] = word[i];
  }
}

// Grid (parts, tables).  Also enters the buckets of more than min_n ids in the lists of the ordering kernels.  The words
// are read twice (the second time from the caches) and nothing of them is kept in registers, so that eight blocks are
// resident: a block is a chain of short phases.
// A crowded part (equal rows, or zero rows, all hash alike) is one block's work too.  With every row alike (670,091 rows,
// 50 tables) a rebuild takes 3.2 to 3.5 ms, 1.2 to 1.5 of them here, where the build by counted ranks takes 3.0; with a
// tenth of the rows alike 2.25 against 2.6.  Adding up a warp's lanes before the counter, 16-byte loads of the words and
// four ids in flight per thread were measured on it and changed nothing.
__global__ void __launch_bounds__(PP_THREADS, 8)
k_part_place(const uint32_t* words, const int* base, int32_t* off, int32_t* ids, int N, long long nb, int low, int up, int id_bits,
             int min_n, int2* mid, int2* big, int* ord_cnt) {
  __shared__ int cnt[1 << PT_MAX_LOW];
  __shared__ int out[PP_CAP];
  __shared__ int sh[PP_THREADS / 32];
  const int t = blockIdx.y, d = blockIdx.x, P = 1 << up, R = 1 << low, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  griddep_wait();
  const int b0 = base[t * (P + 1) + d], n = base[t * (P + 1) + d + 1] - b0;
  const uint32_t* w = words + (size_t)t * N + b0;
  int32_t* to = ids + (size_t)t * N + b0;
  const uint32_t imask = (1u << id_bits) - 1u;
  for (int c = tid; c < R; c += PP_THREADS) cnt[c] = 0;
  __syncthreads();
  for (int i0 = tid; i0 < n; i0 += 4 * PP_THREADS) {
    uint32_t e[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) e[u] = i0 + u * PP_THREADS < n ? w[i0 + u * PP_THREADS] : 0u;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i0 + u * PP_THREADS < n) atomicAdd(&cnt[e[u] >> id_bits], 1);
  }
  __syncthreads();
  // running sum over the part's buckets; a thread owns R / PP_THREADS consecutive ones (at least one)
  const int per = (R + PP_THREADS - 1) / PP_THREADS;
  const int c0 = min(R, tid * per), c1 = min(R, c0 + per);
  int mine = 0;
  for (int c = c0; c < c1; ++c) mine += cnt[c];
  int incl = mine;
#pragma unroll
  for (int q = 1; q < 32; q <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, incl, q);
    if (lane >= q) incl += o;
  }
  if (lane == 31) sh[warp] = incl;
  __syncthreads();
  int run = incl - mine;
  for (int q = 0; q < warp; ++q) run += sh[q];
  for (int c = c0; c < c1; ++c) {
    const int m = cnt[c];
    cnt[c] = run;
    if (ord_cnt && m > min_n) {
      const int2 tc = make_int2(t, (d << low) + c);
      if (m <= ORD_BLOCK) mid[atomicAdd(ord_cnt, 1)] = tc;
      else big[atomicAdd(ord_cnt + 1, 1)] = tc;
    }
    run += m;
  }
  __syncthreads();
  int32_t* o = off + (size_t)t * (size_t)(nb + 1) + ((size_t)d << low);
  for (int c = tid; c < R; c += PP_THREADS) o[c] = b0 + cnt[c];
  if (d == P - 1 && tid == 0) o[R] = N;
  __syncthreads();                      // the offsets have been read out of cnt
  const bool fits = n <= PP_CAP;        // a crowded part (codes far from evenly spread) is placed straight in memory
  for (int i0 = tid; i0 < n; i0 += 4 * PP_THREADS) {
    uint32_t e[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) e[u] = i0 + u * PP_THREADS < n ? w[i0 + u * PP_THREADS] : 0u;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i0 + u * PP_THREADS < n) {
        const int at = atomicAdd(&cnt[e[u] >> id_bits], 1), id = (int)(e[u] & imask);
        if (fits) out[at] = id;
        else to[at] = id;
      }
  }
  if (!fits) return;
  __syncthreads();
  for (int i = tid; i < n; i += PP_THREADS) to[i] = out[i];
}

// Upper and lower bits of the partition, or false when a word cannot hold the lower bits and an id.
static bool part_shape(const Ctx* c, int* low, int* up, int* id_bits) {
  int ib = 1;
  while (((int64_t)1 << ib) < c->N) ++ib;
  int u = 0;
  while (u < PT_MAX_UP && (c->N >> u) > 1536) ++u;              // about a thousand ids per part
  if (u > c->bits - 1) u = c->bits - 1;
  if (c->bits - u > PT_MAX_LOW) u = c->bits - PT_MAX_LOW;
  if (c->bits - u + ib > 32) u = c->bits + ib - 32;
  if (u < 1) u = 1;
  *up = u; *low = c->bits - u; *id_bits = ib;
  return c->place_path && u <= PT_MAX_UP && u < c->bits;
}
size_t part_ints(int L) { return (size_t)L * (2 * (1 << PT_MAX_UP) + 1); }

// ------------------------------------------------------------------ wide codes: place, then order inside buckets
// What is left when the lower bits and an id do not fit a word (2^21 buckets x 4 M neurons): a counting pass hands every
// id its rank of arrival inside its bucket, the id goes to the bucket's start plus that rank, and the ids of each bucket are then put in ascending
// order where they stand: in registers for
// buckets of up to ORD_SMALL ids, by a block-wide sort in shared memory up to ORD_BLOCK, and for a larger bucket by
// one ordered pass over the table's codes that writes the matching ids out again.
constexpr int ORD_THREADS = 256;

__global__ void __launch_bounds__(256) k_place_ids(const uint32_t* keys, const uint32_t* ranks, const int32_t* off, int32_t* ids,
                                                   int N, long long nb) {
  const int t = blockIdx.y;
  const uint32_t* k = keys + (size_t)t * N;
  const uint32_t* r = ranks + (size_t)t * N;
  const int32_t* o = off + (size_t)t * (size_t)(nb + 1);
  int32_t* out = ids + (size_t)t * N;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < N; j += gridDim.x * blockDim.x)
    out[__ldg(o + k[j]) + (int)r[j]] = j;
}

// Sorts n <= M ids in place with an odd-even transposition network (fully unrolled: the ids stay in registers).
template <int M>
__device__ __forceinline__ void order_in_registers(int32_t* p, int n) {
  int a[M];
#pragma unroll
  for (int i = 0; i < M; ++i) a[i] = i < n ? p[i] : 0x7fffffff;
#pragma unroll
  for (int round = 0; round < M; ++round) {
#pragma unroll
    for (int i = round & 1; i + 1 < M; i += 2) {
      const int lo = min(a[i], a[i + 1]), hi = max(a[i], a[i + 1]);
      a[i] = lo; a[i + 1] = hi;
    }
  }
#pragma unroll
  for (int i = 0; i < M; ++i)
    if (i < n) p[i] = a[i];
}

// One thread per bucket.  cnt[0] / cnt[1]: lengths of the lists of buckets left to the block-wide and to the ordered-
// pass kernels.
// Only buckets of more than min_n ids are touched.
__global__ void __launch_bounds__(256) k_order_small(const int32_t* off, int32_t* ids, int N, long long nb, int2* mid,
                                                     int2* big, int* cnt, int min_n) {
  const int t = blockIdx.y;
  const int32_t* o = off + (size_t)t * (size_t)(nb + 1);
  int32_t* out = ids + (size_t)t * N;
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < nb; c += (long long)gridDim.x * blockDim.x) {
    const int beg = o[c], n = o[c + 1] - beg;
    if (n <= min_n) continue;
    if (n <= 4) order_in_registers<4>(out + beg, n);
    else if (n <= 8) order_in_registers<8>(out + beg, n);
    else if (n <= ORD_SMALL) order_in_registers<ORD_SMALL>(out + beg, n);
    else if (n <= ORD_BLOCK) {
      mid[atomicAdd(cnt, 1)] = make_int2(t, (int)c);
    } else {
      big[atomicAdd(cnt + 1, 1)] = make_int2(t, (int)c);
    }
  }
}

// Buckets of ORD_SMALL + 1 .. ORD_BLOCK ids: a block loads one, sorts it in shared memory (bitonic) and writes it back.
__global__ void __launch_bounds__(ORD_THREADS) k_order_mid(const int32_t* off, int32_t* ids, int N, long long nb, const int2* mid,
                                                           const int* cnt) {
  __shared__ int sm[ORD_BLOCK];
  const int nmid = cnt[0];
  for (int q = blockIdx.x; q < nmid; q += gridDim.x) {
    const int2 tc = mid[q];
    const int32_t* o = off + (size_t)tc.x * (size_t)(nb + 1);
    int32_t* out = ids + (size_t)tc.x * N;
    const int beg = o[tc.y], n = o[tc.y + 1] - beg;
    int n2 = 1;
    while (n2 < n) n2 <<= 1;
    __syncthreads();
    for (int i = threadIdx.x; i < n2; i += ORD_THREADS) sm[i] = i < n ? out[beg + i] : 0x7fffffff;
    __syncthreads();
    for (int k = 2; k <= n2; k <<= 1)
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int i = threadIdx.x; i < n2; i += ORD_THREADS) {
          const int x = i ^ j;
          if (x > i) {
            const int a = sm[i], b = sm[x];
            const bool asc = (i & k) == 0;
            if ((a > b) == asc) { sm[i] = b; sm[x] = a; }
          }
        }
        __syncthreads();
      }
    for (int i = threadIdx.x; i < n; i += ORD_THREADS) out[beg + i] = sm[i];
  }
}

// Larger buckets: the ids of bucket c in ascending order are the j, ascending, whose code is c.
__global__ void __launch_bounds__(ORD_THREADS) k_order_big(const uint32_t* keys, const int32_t* off, int32_t* ids, int N,
                                                           long long nb, const int2* big, const int* cnt) {
  __shared__ int sh[ORD_THREADS / 32 + 1];
  const int nbig = cnt[1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int q = blockIdx.x; q < nbig; q += gridDim.x) {
    const int2 tc = big[q];
    const uint32_t* k = keys + (size_t)tc.x * N;
    int32_t* out = ids + (size_t)tc.x * N + off[(size_t)tc.x * (size_t)(nb + 1) + tc.y];
    int run = 0;
    for (int base = 0; base < N; base += ORD_THREADS) {
      const int j = base + threadIdx.x;
      const bool hit = j < N && k[j] == (uint32_t)tc.y;
      const unsigned m = __ballot_sync(0xffffffffu, hit);
      __syncthreads();
      if (lane == 0) sh[warp] = __popc(m);
      __syncthreads();
      int before = 0, total = 0;
      for (int w = 0; w < ORD_THREADS / 32; ++w) { const int x = sh[w]; if (w < warp) before += x; total += x; }
      if (hit) out[run + before + __popc(m & ((1u << lane) - 1u))] = j;
      run += total;
    }
  }
}

// Puts the ids of every bucket with more than min_n ids in ascending order (place path only).  With `listed`, the
// offset scan has already entered those buckets in the lists (all of them larger than ORD_SMALL).
static cudaError_t order_buckets(Ctx* c, int min_n, bool listed) {
  if (min_n < 1) min_n = 1;
  LaunchScope ls(c, KID_ORDER_BUCKETS);
  if (!listed) {
    cudaError_t e = cudaMemsetAsync(c->ord_cnt, 0, 2 * sizeof(int), c->stream);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)min((long long)((c->nb + 255) / 256), 2048LL), c->L);
    k_order_small<<<grid, 256, 0, c->stream>>>(c->bucket_off, c->bucket_ids, c->N, c->nb, c->ord_mid, c->ord_big, c->ord_cnt, min_n);
  }
  k_order_mid<<<c->num_sms * 4, ORD_THREADS, 0, c->stream>>>(c->bucket_off, c->bucket_ids, c->N, c->nb, c->ord_mid, c->ord_cnt);
  k_order_big<<<c->num_sms, ORD_THREADS, 0, c->stream>>>(c->keysA, c->bucket_off, c->bucket_ids, c->N, c->nb, c->ord_big,
                                                          c->ord_cnt);
  return cudaGetLastError();
}

cudaError_t launch_order_buckets(Ctx* c, int min_n) { return order_buckets(c, min_n, false); }

// Warps of a block of the bins-of-eight kernel: the tables go round the warps, so as many as leave the fewest idle.
static int dwta8_warps(int L) {
  int best = 8;
  double eff = 0.0;
  for (int w = 8; w <= HN8_WARPS_MAX; ++w) {
    const double now = (double)L / (double)(w * ((L + w - 1) / w));
    if (now > eff + 1e-9) { eff = now; best = w; }
  }
  return best;
}

template <int RP>
static cudaError_t launch_dwta8(Ctx* c, int smem) {
  cudaError_t e = cudaFuncSetAttribute(k_hash_neurons_dwta8<RP>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const int threads = 32 * dwta8_warps(c->L);
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_hash_neurons_dwta8<RP>, threads, smem);
  if (e != cudaSuccess) return e;
  LaunchScope ls(c, KID_HASH_NEURONS);
  k_hash_neurons_dwta8<RP><<<c->num_sms * (per_sm > 0 ? per_sm : 1), threads, smem, c->stream>>>(c->W2, c->hash_idx, c->keysA, c->N, c->H, c->K, c->L);
  return cudaGetLastError();
}

template <int R>
static cudaError_t launch_sim(Ctx* c, int tile_bytes, int table_bytes) {
  // as many tables at a time as find room; more shares than that where the tiles leave multiprocessors idle
  const int ntiles = (c->N + 32 * R - 1) / (32 * R);
  int per = (HNS_SMEM - tile_bytes) / table_bytes;
  if (per > c->L) per = c->L;
  int shares = (c->L + per - 1) / per;
  if (ntiles * shares < 2 * c->num_sms) shares = (2 * c->num_sms + ntiles - 1) / ntiles;
  if (shares > c->L) shares = c->L;
  per = (c->L + shares - 1) / shares;
  shares = (c->L + per - 1) / per;
  // Few tables at a time are few warps: the functions of a table are then shared out too, where the block has a multiprocessor
  // to itself (smaller blocks fill it by their number)
  const int code_bytes = per * 32 * R * 4;
  int parts = 1;
  if (tile_bytes + per * table_bytes > 113 * 1024 && per < HNS_WARPS && tile_bytes + per * table_bytes + code_bytes <= HNS_SMEM)
    parts = min(c->K, HNS_WARPS / per);
  int warps = 8;                              // the rounds that the tables take decide, then the warps' number
  const int items = per * parts;
  for (int w = 9; w <= 32; ++w)
    if ((items + w - 1) / w * w <= (items + warps - 1) / warps * warps) warps = w;
  const int smem = tile_bytes + per * table_bytes + (parts > 1 ? code_bytes : 0);
  auto kern = parts > 1 ? k_hash_neurons_sim<R, true> : k_hash_neurons_sim<R, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * warps, smem);
  if (e != cudaSuccess) return e;
  int nb = c->num_sms * (per_sm > 0 ? per_sm : 1) / shares;
  if (nb < 1) nb = 1;
  if (nb > ntiles) nb = ntiles;
  LaunchScope ls(c, KID_HASH_NEURONS);
  kern<<<dim3(nb, shares), 32 * warps, smem, c->stream>>>(c->W2, c->hash_idx, c->hash_sign, c->keysA, c->N, c->H, c->K, c->L, c->fn_len, per, parts);
  return cudaGetLastError();
}

cudaError_t launch_build_tables(Ctx* c) {
  const size_t off_bytes = (size_t)c->L * (size_t)(c->nb + 1) * sizeof(int32_t);
  int low = 0, up = 0, id_bits = 0;
  const bool parts = part_shape(c, &low, &up, &id_bits);
  cudaError_t e = cudaSuccess;
  // What the kernels below count into is cleared first, so that nothing stands between them: the partition's kernels follow
  // the hashing and one another by dependent launch (a small table is a chain of launches: 20,011 rows, K 6, L 12 61.5 us in stream order, 54.3 so).
  if (c->place_path && !parts && (e = cudaMemsetAsync(c->bucket_off, 0, off_bytes, c->stream)) != cudaSuccess) return e;
  const bool list_in_scan = c->place_path && c->cap >= ORD_SMALL;
  // on the wide-code paths, with a cap of at least ORD_SMALL, the buckets that must be in order for the step (those
  // above the cap) are listed on the way: no separate pass over all bucket sizes
  if (list_in_scan && (e = cudaMemsetAsync(c->ord_cnt, 0, 2 * sizeof(int), c->stream)) != cudaSuccess) return e;
  const size_t counted = parts ? (size_t)c->L << up : (c->place_path ? 0 : (size_t)c->L * (size_t)c->nb);
  if (counted && (e = cudaMemsetAsync(c->part_work, 0, counted * sizeof(int), c->stream)) != cudaSuccess) return e;
  const int tile_bytes = (HN_ROWS * (c->H + 1) * (int)sizeof(float) + 15) & ~15;
  const long long fn_bytes = (long long)c->KL * c->fn_len * 2;
  const bool fn_smem = fn_bytes <= HN_FN_SMEM_MAX && c->H <= 0x7fff;
  const int smem = tile_bytes + (fn_smem ? (int)fn_bytes : 0);
  // bins of eight: four rows per lane while two blocks fit a multiprocessor, else two rows while two blocks fit, else the
  // general kernel.  With one block the tile's loads and the bins take turns: 66,656 rows of 488 units, a rebuild in us by
  // one block of two rows per lane / the general kernel: K 2, L 9 162 / 94; K 4, L 20 175 / 108; K 6, L 50 267 / 191;
  // 760 units 211 / 135, 223 / 149, 316 / 233; at 392 units (two blocks) 99, 111, 193 against 117, 132, 230 by the kernel
  // before, which the general one equals.
  const long long smem4 = ((32LL * (c->H + 1) * 16 + 15) & ~15LL) + 2 * fn_bytes, smem2 = ((32LL * (c->H + 1) * 8 + 15) & ~15LL) + 2 * fn_bytes;
  if (c->cfg.hash_family == DSLIDE_SIMHASH) {
    const int table = c->K * ((c->fn_len + 7) & ~7) * 2;
    auto tile = [&](int r) { return (32 * (c->H + 1) * 4 * r + 15) & ~15; };
    if (tile(4) + HNS_MIN_TABLES * table <= HNS_SMEM) e = launch_sim<4>(c, tile(4), table);
    else if (tile(2) + HNS_MIN_TABLES * table <= HNS_SMEM) e = launch_sim<2>(c, tile(2), table);
    else e = launch_sim<1>(c, tile(1), table);
    if (e != cudaSuccess) return e;
  } else if (fn_smem && c->fn_len == 8 && smem2 <= 112 * 1024) {
    e = smem4 <= 112 * 1024 ? launch_dwta8<2>(c, (int)smem4) : launch_dwta8<1>(c, (int)smem2);
    if (e != cudaSuccess) return e;
  } else {
    auto kern = fn_smem ? k_hash_neurons<true> : k_hash_neurons<false>;
    if (smem > 48 * 1024) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      if (e != cudaSuccess) return e;
    }
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, HN_THREADS, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    LaunchScope ls(c, KID_HASH_NEURONS);
    kern<<<c->num_sms * per_sm, HN_THREADS, smem, c->stream>>>(c->W2, c->hash_idx, c->keysA, c->N, c->H, c->K, c->L, c->lg_bin, c->fn_len);
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (parts) {
    int* total = c->part_work;
    int* base = total + (size_t)c->L * ((size_t)1 << up);
    const dim3 grid((c->N + PT_TILE - 1) / PT_TILE, c->L);
    {
      LaunchScope ls(c, KID_SORT_HIST);
      e = launch_dependent(k_part_hist, dim3((c->N + PT_HIST - 1) / PT_HIST, c->L), dim3(PT_THREADS), 0, c->stream, (const uint32_t*)c->keysA, total, c->N, low, up);
      if (e != cudaSuccess) return e;
    }
    {
      LaunchScope ls(c, KID_SORT_SCAN);
      if ((e = launch_dependent(k_part_scan, dim3(c->L), dim3(1 << (up < 5 ? 5 : up)), 0, c->stream, total, base, up)) != cudaSuccess) return e;
    }
    {
      LaunchScope ls(c, KID_SORT_SCATTER);
      e = launch_dependent(k_part_scatter, grid, dim3(PT_THREADS), 0, c->stream, (const uint32_t*)c->keysA, total, c->keysB, c->N, low, up, id_bits);
      if (e != cudaSuccess) return e;
    }
    {
      LaunchScope ls(c, KID_PLACE_IDS);
      e = launch_dependent(k_part_place, dim3(1 << up, c->L), dim3(PP_THREADS), 0, c->stream, (const uint32_t*)c->keysB, (const int*)base, c->bucket_off,
                           c->bucket_ids, c->N, (long long)c->nb, low, up, id_bits, c->cap, c->ord_mid, c->ord_big, list_in_scan ? c->ord_cnt : (int*)nullptr);
      if (e != cudaSuccess) return e;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // A query reads a whole bucket unless it holds more than `cap` ids, and the union of the buckets is put in
    // order afterwards anyway: only buckets larger than the cap must be in ascending order for the step.  The
    // smaller ones are ordered when the table is read back (launch_order_buckets(c, 1)).
    c->ids_ordered_above = c->cap;
    return order_buckets(c, c->cap, list_in_scan);
  }
  if (!c->place_path) {
    // codes of at most one radix digit: the buckets are counted tile by tile in shared memory, and the running sum over
    // a table's counts is its offsets
    LaunchScope ls(c, KID_BUCKET_SCAN);
    c->launches += 1;
    e = launch_dependent(k_part_hist, dim3((c->N + PT_HIST - 1) / PT_HIST, c->L), dim3(PT_THREADS), 0, c->stream, (const uint32_t*)c->keysA, c->part_work, c->N, 0, c->bits);
    if (e != cudaSuccess) return e;
    e = launch_dependent(k_part_scan, dim3(c->L), dim3(1 << (c->bits < 5 ? 5 : c->bits)), 0, c->stream, c->part_work, c->bucket_off, c->bits);
    if (e != cudaSuccess) return e;
  } else {
    LaunchScope ls(c, KID_HASH_NEURONS);
    dim3 grid((unsigned)min((long long)(c->N + 255) / 256, 2048LL), c->L);
    k_count_ranks<<<grid, 256, 0, c->stream>>>(c->keysA, c->keysB, c->bucket_off, c->N, c->nb);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if (c->place_path) {
    const int nchunks = (int)((c->nb + 1 + BS_CHUNK - 1) / BS_CHUNK);
    dim3 grid(nchunks, c->L);
    LaunchScope ls(c, KID_BUCKET_SCAN);
    k_bucket_sums<<<grid, BS_THREADS, 0, c->stream>>>(c->bucket_off, c->nb, c->bucket_part, nchunks);
    k_bucket_scan<<<grid, BS_THREADS, 0, c->stream>>>(c->bucket_off, c->nb, c->bucket_part, nchunks, c->cap, c->ord_mid,
                                                      c->ord_big, list_in_scan ? c->ord_cnt : nullptr);
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;

  if (c->place_path) {
    {
      LaunchScope ls(c, KID_PLACE_IDS);
      dim3 grid((unsigned)min((long long)(c->N + 255) / 256, 1024LL), c->L);
      k_place_ids<<<grid, 256, 0, c->stream>>>(c->keysA, c->keysB, c->bucket_off, c->bucket_ids, c->N, c->nb);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    c->ids_ordered_above = c->cap;      // as above
    return order_buckets(c, c->cap, list_in_scan);
  }

  if ((e = cudaFuncSetAttribute(k_sort_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, SORT_SMEM)) != cudaSuccess) return e;
  const uint32_t* kin = c->keysA;
  const int32_t* vin = nullptr;
  for (int pass = 0; pass < c->sort_passes; ++pass) {
    const bool last = pass == c->sort_passes - 1;
    const int shift = pass * c->sort_width;
    const int width = min(c->sort_width, c->bits - shift);
    const int radix = 1 << width;
    uint32_t* kout = last ? nullptr : (kin == c->keysA ? c->keysB : c->keysA);
    int32_t* vout = last ? c->bucket_ids : (vin == c->valsA ? c->valsB : c->valsA);
    dim3 grid(c->sort_tiles, c->L);
    {
      LaunchScope ls(c, KID_SORT_HIST);
      k_sort_hist<<<grid, SORT_THREADS, 0, c->stream>>>(kin, c->tile_hist, c->N, c->sort_tiles, shift, width);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    {
      LaunchScope ls(c, KID_SORT_SCAN);
      k_sort_scan<<<c->L, 1024, 0, c->stream>>>(c->tile_hist, radix * c->sort_tiles);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    {
      LaunchScope ls(c, KID_SORT_SCATTER);
      k_sort_scatter<<<grid, SORT_THREADS, SORT_SMEM, c->stream>>>(kin, vin, kout, vout, c->tile_hist, c->N, c->sort_tiles,
                                                          shift, width);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    kin = kout;
    vin = vout;
  }
  return cudaSuccess;
}

int sort_tile_elems() { return SORT_TILE; }
int order_small_max() { return ORD_SMALL; }
int order_block_max() { return ORD_BLOCK; }
int bucket_scan_chunk() { return BS_CHUNK; }
int sort_max_width() { return SORT_MAX_WIDTH; }

}  // namespace dslide
