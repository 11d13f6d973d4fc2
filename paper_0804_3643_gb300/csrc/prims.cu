// prims.cu -- scoring tables, a device-wide exclusive scan and a stable LSD
// radix sort of (uint64 key, uint32 value) pairs.  The sort gives stage 0 its
// CSR order (positions stay increasing within a key because the sort is
// stable) and stage 2 its canonical record order.
#include <algorithm>
#include <atomic>
#include <mutex>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include "common.cuh"

namespace plast {

std::atomic<long long> g_launches{0};
void note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }
long long launch_total() { return g_launches.load(); }

__constant__ int8_t c_score[NCODE * NCODE];
__constant__ int8_t c_cls2[NAA];
__constant__ int8_t c_cls3[NAA];

static int code_of(char c) {
  const char* p = strchr(ALPHABET, c);
  return p ? (int)(p - ALPHABET) : -1;
}

void build_tables(Tables* t) {
  for (int a = 0; a < NCODE; a++)
    for (int b = 0; b < NCODE; b++) {
      int v;
      if (a == SENTINEL || b == SENTINEL) v = SENT_SCORE;
      else if (a == STOP && b == STOP) v = 1;
      else if (a == STOP || b == STOP) v = -4;
      else v = 0;  // filled from the transcription below
      t->score[a * NCODE + b] = (int8_t)v;
    }
  for (int a = 0; a < NAA; a++) {
    const char* s = B62_UPPER[a];
    for (int b = a; b < NAA; b++) {
      char* end;
      long v = strtol(s, &end, 10);
      s = end;
      t->score[a * NCODE + b] = t->score[b * NCODE + a] = (int8_t)v;
    }
  }
  for (int k = 0; k < 2; k++)
    for (const char* p = SEED_POS2[k]; *p; p++) {
      int c = code_of(*p);
      if (c >= 0) t->cls2[c] = (int8_t)k;
    }
  for (int k = 0; k < 11; k++)
    for (const char* p = SEED_POS3[k]; *p; p++) {
      int c = code_of(*p);
      if (c >= 0) t->cls3[c] = (int8_t)k;
    }
}

cudaError_t upload_tables_once() {
  static std::mutex mu;
  static bool done[64] = {false};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> g(mu);
  if (dev < 64 && done[dev]) return cudaSuccess;
  // keep freed stream-ordered memory in the pool: scratch and banks are
  // re-allocated on every call
  cudaMemPool_t pool;
  if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
    uint64_t thr = ~0ull;
    cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
  }
  Tables t;
  build_tables(&t);
  if ((e = cudaMemcpyToSymbol(c_score, t.score, sizeof(t.score))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_cls2, t.cls2, sizeof(t.cls2))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_cls3, t.cls3, sizeof(t.cls3))) != cudaSuccess) return e;
  if (dev < 64) done[dev] = true;
  return cudaSuccess;
}

// ---------------------------------------------------------------------------
// Exclusive scan, int32 in -> int64 out, over tiles of SCAN_TILE elements: tile
// sums, a one-CTA scan of the sums, tile scans.  Up to SCAN_FEW_TILES tiles (two
// million elements, 8 KB of sums for the last CTA to read) the second launch,
// 2 to 3 us of a few microseconds' work, goes: the tile scans add up the sums.
// ---------------------------------------------------------------------------
constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;
constexpr int64_t SCAN_FEW_TILES = 1024;

__device__ __forceinline__ int64_t block_exclusive_scan(int64_t v, int64_t* total) {
  __shared__ int64_t s_warp[SCAN_THREADS / 32];
  int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int64_t w = lane < SCAN_THREADS / 32 ? s_warp[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int64_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < SCAN_THREADS / 32) s_warp[lane] = w;
  }
  __syncthreads();
  int64_t before = warp ? s_warp[warp - 1] : 0;
  if (total) *total = s_warp[SCAN_THREADS / 32 - 1];
  int64_t r = before + x - v;
  __syncthreads();
  return r;
}

// n_dev (optional): the element count lives in device memory, at most n.
__device__ __forceinline__ int64_t count_of(int64_t n, const int64_t* n_dev) {
  return n_dev ? min(n, max(*n_dev, (int64_t)0)) : n;
}

__global__ void k_scan_tile_sums(const int32_t* in, int64_t n, int64_t* sums, const int64_t* n_dev) {
  n = count_of(n, n_dev);
  int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
  int64_t acc = 0;
#pragma unroll
  for (int r = 0; r < SCAN_ITEMS; r++) {
    int64_t i = base + r * SCAN_THREADS + threadIdx.x;
    if (i < n) acc += in[i];
  }
  int64_t tot;
  block_exclusive_scan(acc, &tot);
  if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

__global__ void k_scan_sums(int64_t* sums, int64_t nt, int64_t* d_total) {
  int64_t carry = 0;
  for (int64_t b = 0; b < nt; b += SCAN_THREADS) {
    int64_t i = b + threadIdx.x;
    int64_t v = i < nt ? sums[i] : 0;
    int64_t tot;
    int64_t ex = block_exclusive_scan(v, &tot);
    if (i < nt) sums[i] = carry + ex;
    carry += tot;
  }
  if (threadIdx.x == 0 && d_total) *d_total = carry;
}

// FEW: the sums are the tiles' own, and each CTA adds up those before its tile.
template <bool FEW>
__global__ void k_scan_tiles(const int32_t* in, int64_t n, const int64_t* sums, int64_t* out, int64_t* d_total,
                             const int64_t* n_dev) {
  n = count_of(n, n_dev);
  int64_t before = 0;
  if (FEW) {
    int64_t x = 0;
    for (int64_t i = threadIdx.x; i < blockIdx.x; i += SCAN_THREADS) x += sums[i];
    block_exclusive_scan(x, &before);
    if (threadIdx.x == 0 && d_total && blockIdx.x == gridDim.x - 1) *d_total = before + sums[blockIdx.x];
  } else {
    before = sums[blockIdx.x];
  }
  // thread t owns the contiguous items [t*ITEMS, t*ITEMS + ITEMS) of the tile
  int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
  int32_t v[SCAN_ITEMS];
  int64_t acc = 0;
#pragma unroll
  for (int r = 0; r < SCAN_ITEMS; r++) {
    int64_t i = base + r;
    v[r] = i < n ? in[i] : 0;
    acc += v[r];
  }
  int64_t ex = block_exclusive_scan(acc, nullptr) + before;
#pragma unroll
  for (int r = 0; r < SCAN_ITEMS; r++) {
    int64_t i = base + r;
    if (i < n) out[i] = ex;
    ex += v[r];
  }
}

size_t scan_tmp_bytes(int64_t n) {
  int64_t nt = (n + SCAN_TILE - 1) / SCAN_TILE;
  return (size_t)(nt + 1) * sizeof(int64_t);
}

cudaError_t scan_exclusive(const int32_t* in, int64_t* out, int64_t n, int64_t* d_total, void* tmp,
                           size_t tmp_bytes, cudaStream_t st, const int64_t* n_dev) {
  if (n <= 0) {
    if (d_total) return cudaMemsetAsync(d_total, 0, sizeof(int64_t), st);
    return cudaSuccess;
  }
  int64_t nt = (n + SCAN_TILE - 1) / SCAN_TILE;
  if (tmp_bytes < scan_tmp_bytes(n)) return cudaErrorInvalidValue;
  int64_t* sums = (int64_t*)tmp;
  note_launch();
  k_scan_tile_sums<<<(unsigned)nt, SCAN_THREADS, 0, st>>>(in, n, sums, n_dev);
  if (nt <= SCAN_FEW_TILES) {
    note_launch();
    k_scan_tiles<true><<<(unsigned)nt, SCAN_THREADS, 0, st>>>(in, n, sums, out, d_total, n_dev);
    return cudaGetLastError();
  }
  note_launch();
  k_scan_sums<<<1, SCAN_THREADS, 0, st>>>(sums, nt, d_total);
  note_launch();
  k_scan_tiles<false><<<(unsigned)nt, SCAN_THREADS, 0, st>>>(in, n, sums, out, nullptr, n_dev);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Stable LSD radix sort, 8-bit digits, a counting pass per digit over tiles of
// RS_THREADS * PER elements.  Where a tile's run of each digit starts comes
// from the digit counts of all tiles, in one of two ways:
//  - up to RS_FEW_TILES tiles of 1,024 (the lists that a search of a few
//    queries leaves): every CTA adds the counts up itself, and each pass counts
//    the next one's digits as it writes, so a pass is one launch.  Bound by its
//    launches: 16,000 records of 44 bits take 6 and a memset, 37 us on the
//    device; with a histogram and a scan a pass they took 25 and 152 us.
//  - beyond, where a CTA would read more than 256 KB of counts: a histogram
//    kernel, the scan above and the pass, tiles of 2,048 (3,072: 1.48 ms where
//    these take 1.35).  40.3 M records of 46 bits: passes 1.35 ms (4.3 TB/s),
//    histograms 0.55, scans 0.29; ranking a round of 256 elements at a time,
//    with match.any and four barriers each, the passes took 2.63.
// ---------------------------------------------------------------------------
constexpr int RS_THREADS = 256;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_COL = RS_WARPS + 2;  // counters of a digit: the warps', spread over the banks
constexpr int RS_PER_FEW = 4, RS_PER_MANY = 8;
constexpr int64_t RS_TILE_FEW = RS_THREADS * RS_PER_FEW, RS_TILE_MANY = RS_THREADS * RS_PER_MANY;
constexpr int64_t RS_FEW_TILES = 256;

__device__ __forceinline__ int radix_digit(uint64_t key, int shift) { return (int)(key >> shift) & 255; }

// Digit counts of a tile: hist[tile * row + digit * col].
template <int PER>
__global__ void k_radix_hist(const uint64_t* keys, int64_t n, int shift, int32_t* hist, int64_t row, int64_t col,
                             const int64_t* n_dev) {
  __shared__ int h[256];
  n = count_of(n, n_dev);
  h[threadIdx.x] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * (RS_THREADS * PER);
#pragma unroll
  for (int r = 0; r < PER; r++) {
    const int64_t i = base + r * RS_THREADS + threadIdx.x;
    if (i < n) atomicAdd(&h[radix_digit(keys[i], shift)], 1);
  }
  __syncthreads();
  hist[blockIdx.x * row + threadIdx.x * col] = h[threadIdx.x];
}

// One pass over a tile.  The warps own consecutive elements; a lane finds the
// lanes of its digit by ballots and the warp's earlier ones by its counter,
// the counters' scan gives every element its place in the tile, and the tile
// leaves digit by digit, consecutive threads to consecutive addresses.
// FEW: `counts` is this pass's table of all tiles' counts ([tile][digit]) and
// `next` the next pass's, zeroed, to be counted here (nullptr: the last);
// else `off` holds the scanned counts ([digit][tile], nt tiles).
template <int PER, bool FEW>
__global__ void __launch_bounds__(RS_THREADS, 4) k_radix_pass(const uint64_t* kin, const uint32_t* vin, uint64_t* kout,
                                                           uint32_t* vout, int64_t n, int shift, const int64_t* off,
                                                           int64_t nt, const int32_t* counts, int32_t* next,
                                                           const int64_t* n_dev) {
  constexpr int TILE = RS_THREADS * PER;
  __shared__ uint64_t s_key[TILE];
  __shared__ uint32_t s_val[TILE];
  __shared__ int64_t s_base[256];  // where digit d's run starts, less its place in the tile
  __shared__ uint16_t s_cnt[256 * RS_COL];
  __shared__ int s_wsum[2][RS_WARPS];
  n = count_of(n, n_dev);
  const int64_t base = (int64_t)blockIdx.x * TILE;
  if (base >= n) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int in_tile = (int)min((int64_t)TILE, n - base);
  const int at0 = warp * (32 * PER) + lane;
  uint64_t k[PER];
  uint32_t v[PER];
#pragma unroll
  for (int j = 0; j < PER; j++) {
    const bool ok = at0 + 32 * j < in_tile;
    k[j] = ok ? kin[base + at0 + 32 * j] : 0;
    v[j] = ok ? vin[base + at0 + 32 * j] : 0;
  }
  // thread = digit: the elements of the digit before this tile, and in all
  int before = 0, all = 0;
  if (FEW) {
    const int tiles = (int)((n + TILE - 1) / TILE);
#pragma unroll 8
    for (int x = 0; x < tiles; x++) {
      const int c = counts[x * 256 + tid];
      all += c;
      if (x < (int)blockIdx.x) before += c;
    }
  }
  for (int x = tid; x < 256 * RS_COL / 2; x += RS_THREADS) reinterpret_cast<uint32_t*>(s_cnt)[x] = 0;
  __syncthreads();
  uint16_t rank[PER];
#pragma unroll
  for (int j = 0; j < PER; j++) {
    const bool ok = at0 + 32 * j < in_tile;
    const int d = radix_digit(k[j], shift);
    unsigned peers = __ballot_sync(0xffffffffu, ok);
#pragma unroll
    for (int b = 0; b < 8; b++) {
      const bool bit = d >> b & 1;
      const unsigned m = __ballot_sync(0xffffffffu, bit);
      peers &= bit ? m : ~m;
    }
    uint16_t* c = s_cnt + d * RS_COL + warp;
    const int have = ok ? *c : 0;
    __syncwarp();
    if (ok && lane == __ffs(peers) - 1) *c = (uint16_t)(have + __popc(peers));
    __syncwarp();
    rank[j] = (uint16_t)(have + __popc(peers & ((1u << lane) - 1u)));
  }
  __syncthreads();
  {
    uint16_t* c = s_cnt + tid * RS_COL;
    int cw[RS_WARPS], mine = 0;
#pragma unroll
    for (int w = 0; w < RS_WARPS; w++) {
      cw[w] = mine;
      mine += c[w];
    }
    // exclusive scans over the digits of the tile's counts and, FEW, of all
    int x = mine, y = all;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int p = __shfl_up_sync(0xffffffffu, x, o), q = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) x += p, y += q;
    }
    if (lane == 31) s_wsum[0][warp] = x, s_wsum[1][warp] = y;
    __syncthreads();
    int start = x - mine, first = y - all;
    for (int w = 0; w < warp; w++) start += s_wsum[0][w], first += s_wsum[1][w];
#pragma unroll
    for (int w = 0; w < RS_WARPS; w++) c[w] = (uint16_t)(start + cw[w]);
    s_base[tid] = (FEW ? (int64_t)first + before : off[(int64_t)tid * nt + blockIdx.x]) - start;
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < PER; j++)
    if (at0 + 32 * j < in_tile) {
      const int at = s_cnt[radix_digit(k[j], shift) * RS_COL + warp] + rank[j];
      s_key[at] = k[j];
      s_val[at] = v[j];
    }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < PER; r++) {
    const int j = tid + r * RS_THREADS;
    if (j < in_tile) {
      const uint64_t key = s_key[j];
      const int64_t dst = s_base[radix_digit(key, shift)] + j;
      kout[dst] = key;
      vout[dst] = s_val[j];
      if (FEW && next) atomicAdd(&next[dst / TILE * 256 + radix_digit(key, shift + 8)], 1);
    }
  }
}

static bool radix_few(int64_t n) { return n <= RS_FEW_TILES * RS_TILE_FEW; }

size_t radix_tmp_bytes(int64_t n) {
  if (radix_few(n)) return (size_t)(8 * ((n + RS_TILE_FEW - 1) / RS_TILE_FEW) * 256) * sizeof(int32_t);
  const int64_t nt = (n + RS_TILE_MANY - 1) / RS_TILE_MANY;
  const size_t h = (size_t)256 * nt;
  return h * sizeof(int32_t) + h * sizeof(int64_t) + scan_tmp_bytes((int64_t)h) + 64;
}

cudaError_t radix_sort_pairs(uint64_t* keys, uint32_t* vals, uint64_t* keys_alt, uint32_t* vals_alt, int64_t n,
                             int bits, void* tmp, size_t tmp_bytes, cudaStream_t st, bool* result_in_alt,
                             const int64_t* n_dev) {
  *result_in_alt = false;
  if ((n <= 1 && !n_dev) || n <= 0 || bits <= 0) return cudaSuccess;
  if (tmp_bytes < radix_tmp_bytes(n)) return cudaErrorInvalidValue;
  uint64_t *ki = keys, *ko = keys_alt;
  uint32_t *vi = vals, *vo = vals_alt;
  cudaError_t e;
  if (radix_few(n)) {
    const int64_t nt = (n + RS_TILE_FEW - 1) / RS_TILE_FEW;
    const int passes = (bits + 7) / 8;
    int32_t* counts = (int32_t*)tmp;
    if (passes > 1 &&
        (e = cudaMemsetAsync(counts + nt * 256, 0, (size_t)((passes - 1) * nt * 256) * sizeof(int32_t), st)) !=
            cudaSuccess)
      return e;
    note_launch();
    k_radix_hist<RS_PER_FEW><<<(unsigned)nt, RS_THREADS, 0, st>>>(ki, n, 0, counts, 256, 1, n_dev);
    for (int p = 0; p < passes; p++) {
      note_launch();
      k_radix_pass<RS_PER_FEW, true><<<(unsigned)nt, RS_THREADS, 0, st>>>(
          ki, vi, ko, vo, n, 8 * p, nullptr, nt, counts + p * nt * 256,
          p + 1 < passes ? counts + (p + 1) * nt * 256 : nullptr, n_dev);
      std::swap(ki, ko);
      std::swap(vi, vo);
    }
    *result_in_alt = passes & 1;
    return cudaGetLastError();
  }
  const int64_t nt = (n + RS_TILE_MANY - 1) / RS_TILE_MANY;
  const size_t h = (size_t)256 * nt;
  int32_t* hist = (int32_t*)tmp;
  int64_t* off = (int64_t*)((char*)tmp + ((h * sizeof(int32_t) + 15) & ~(size_t)15));
  void* stmp = (char*)off + h * sizeof(int64_t);
  const size_t stmp_bytes = scan_tmp_bytes((int64_t)h);
  for (int shift = 0; shift < bits; shift += 8) {
    note_launch();
    k_radix_hist<RS_PER_MANY><<<(unsigned)nt, RS_THREADS, 0, st>>>(ki, n, shift, hist, 1, nt, n_dev);
    e = scan_exclusive(hist, off, (int64_t)h, nullptr, stmp, stmp_bytes, st);
    if (e != cudaSuccess) return e;
    note_launch();
    k_radix_pass<RS_PER_MANY, false><<<(unsigned)nt, RS_THREADS, 0, st>>>(ki, vi, ko, vo, n, shift, off, nt, nullptr,
                                                                         nullptr, n_dev);
    std::swap(ki, ko);
    std::swap(vi, vo);
    *result_in_alt = !*result_in_alt;
  }
  return cudaGetLastError();
}

}  // namespace plast
