// index.cu -- stage 0 (Section 3.3.1) and the six-frame translation of
// Section 6, as device kernels.
//
// A bank lives on the device as
//   pad      codes with GAP sentinel bytes before, between and after the
//            sequences: sequence s starts at pad_off[s] = seq_off[s] + GAP*(s+1)
//   pos      padded start of every indexed word, grouped by key (CSR by
//            key_off[8801]), increasing within a key
//   nb       the 48-residue neighbourhood of every indexed word, in the
//            order stage 2 consumes it: the 26 residues from the seed start
//            rightwards, then the 22 residues left of it walking leftwards
//            (Section 3.3.2's neighbourhood blocks, built once per bank).
#include <algorithm>
#include <atomic>

#include "common.cuh"
#include "gapped.cuh"
#include "index.cuh"

namespace plast {

// last s in [0, n) with off[s] <= p (off non-decreasing, off[0] <= p)
__device__ __forceinline__ int32_t find_seq(const int64_t* off, int32_t n, int64_t p) {
  int32_t lo = 0, hi = n - 1;
  while (lo < hi) {
    int32_t mid = (lo + hi + 1) >> 1;
    if (off[mid] <= p) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// True in every byte lane of w whose byte, read unsigned, is above hi
// (0 <= hi < 127): adding 127 - hi to the low seven bits carries into bit 7
// exactly when the byte exceeds hi, and bytes of 128 or more have bit 7 set.
__device__ __forceinline__ uint32_t bytes_above(uint32_t w, uint32_t hi) {
  return (((w & 0x7f7f7f7fu) + 0x01010101u * (127u - hi)) | w) & 0x80808080u;
}

// *bad is raised if a code lies outside [0, hi]: 16 bytes a thread, single ones
// before the first 16-byte boundary and after the last.
__global__ void k_check_codes(const int8_t* codes, int64_t n, int hi, int* bad) {
  const int64_t head = min(n, (int64_t)(-reinterpret_cast<uintptr_t>(codes) & 15)), chunks = (n - head) >> 4;
  const int64_t tail = head + (chunks << 4);
  const uint4* body = reinterpret_cast<const uint4*>(codes + head);
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t b = 0;
  for (int64_t c = t; c < chunks; c += (int64_t)gridDim.x * blockDim.x) {
    const uint4 v = body[c];
    b |= bytes_above(v.x, hi) | bytes_above(v.y, hi) | bytes_above(v.z, hi) | bytes_above(v.w, hi);
  }
  if (t < head) b |= bytes_above((uint8_t)codes[t], hi);
  if (t < n - tail) b |= bytes_above((uint8_t)codes[tail + t], hi);
  if (b) atomicOr(bad, 1);
}

// Padded bank, one thread per 16-byte chunk of codes: the chunk's sequence by
// one binary search; a chunk inside one sequence moves with one 16-byte load
// and store (sequence s moves by GAP * (s + 1), a multiple of 16, into a
// 16-byte aligned pad), the others byte by byte.  Every code is checked
// against [0, hi]; *bad is raised if one is outside.
static_assert(GAP % 16 == 0, "sequences move by whole 16-byte chunks");
__global__ void k_build_pad(const int8_t* codes, const int64_t* seq_off, int32_t n_seqs, int64_t n_res, int hi,
                            int8_t* pad, int* bad) {
  const bool vec = (reinterpret_cast<uintptr_t>(codes) & 15) == 0;
  const int64_t n_chunks = (n_res + 15) >> 4;
  uint32_t b = 0;
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n_chunks; c += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p0 = c << 4, p1 = min(p0 + 16, n_res);
    int32_t s = find_seq(seq_off, n_seqs, p0);
    if (vec && p1 - p0 == 16 && seq_off[s + 1] >= p1) {
      const uint4 v = *reinterpret_cast<const uint4*>(codes + p0);
      b |= bytes_above(v.x, hi) | bytes_above(v.y, hi) | bytes_above(v.z, hi) | bytes_above(v.w, hi);
      *reinterpret_cast<uint4*>(pad + p0 + (int64_t)GAP * (s + 1)) = v;
    } else {
      for (int64_t p = p0; p < p1; p++) {
        while (seq_off[s + 1] <= p) s++;  // seq_off[n_seqs] = n_res > p ends the walk
        const int8_t x = codes[p];
        if (x < 0 || x > hi) b = 1;
        pad[p + (int64_t)GAP * (s + 1)] = x;
      }
    }
  }
  if (b) atomicOr(bad, 1);
}

// Stage 0's lookup table and lists (Section 3.3.1) as a stable counting sort
// of the padded positions by key, high digit first.  A word is indexed when
// its four letters are residues (codes below 20: no stop, no sentinel, so no
// word crosses a sequence end).  The key's high digit (key / 128) names its
// bucket, of 69.  The padded bank is cut into chunks of 8192 positions and
// these into groups (IndexShape):
//   k_index_hist   counts each chunk's words per bucket and each group's per
//                  key; an exclusive scan of the two tables, bucket-major and
//                  key-major, gives every (bucket, chunk) and every (key,
//                  group) its first slot, and with it the CSR offsets;
//   k_index_split  sorts each chunk by bucket in shared memory: positions and
//                  low digits move to their buckets, in position order;
//   k_index_fill   takes a bucket's words of one group, sorts them by the low
//                  digit and writes each key's run of positions and windows.
// Why two digits: with 8,800 destinations at once a word's 4-byte position and
// 48-byte window go to places that no other word of the same few microseconds
// touches, and every store is a partial line.  Split first, the runs are some
// 90 words (split) and 47 words (fill) long, and the words a CTA of k_index_fill
// holds come from a stretch of 1 MB or so of the bank, in L2 for all buckets.
// For 166 M words in 206 M padded positions: hist 0.43 ms, split 0.98, fill
// 2.96; one scatter over all keys took 3.69 and the windows, gathered in key
// order over the whole bank, 4.09 (sorting both digits of a chunk in one CTA
// and storing the windows from there: 8.5).
constexpr int IX_THREADS = 512;
constexpr int IX_WARPS = IX_THREADS / 32;
constexpr int IX_PER = 16;                      // positions per thread and chunk
constexpr int IX_CHUNK = IX_THREADS * IX_PER;   // 8192
constexpr int IX_LO = 128;                      // keys per bucket
constexpr int IX_LO_BITS = 7;
constexpr int IX_BUCKETS = (NKEYS + IX_LO - 1) / IX_LO;
static_assert(1 << IX_LO_BITS == IX_LO, "the low digit");

// Keys of the 16 words at p0 .. p0 + 15 from five aligned words of pad (p0 is
// a multiple of 16; a thread at or past n_pad reads nothing, the others at
// most 19 bytes past p0, inside the bank's trailing slack); bit j of the
// result says whether word p0 + j is indexed.
__device__ __forceinline__ uint32_t keys16_from(const uint32_t w[5], const int8_t* cls2, const int8_t* cls3,
                                                int32_t key[IX_PER]) {
  uint32_t by[IX_PER + 3];
#pragma unroll
  for (int j = 0; j < IX_PER + 3; j++) by[j] = (w[j >> 2] >> (8 * (j & 3))) & 0xffu;
  uint32_t valid = 0;
#pragma unroll
  for (int j = 0; j < IX_PER; j++) {
    const uint32_t a0 = by[j], a1 = by[j + 1], a2 = by[j + 2], a3 = by[j + 3];
    const bool ok = a0 < NAA && a1 < NAA && a2 < NAA && a3 < NAA;
    key[j] = ok ? (((int)(a0 * 2) + cls2[ok ? a1 : 0]) * 11 + cls3[ok ? a2 : 0]) * 20 + (int)a3 : -1;
    valid |= (uint32_t)ok << j;
  }
  return valid;
}

// The 20 bytes pad[p0 .. p0 + 20) as five words (p0 a multiple of 16); all
// sentinels at or past n_pad (nothing is read there; below it at most 19
// bytes past p0 are read, inside the bank's trailing slack).
__device__ __forceinline__ void load20(const int8_t* pad, int64_t p0, int64_t n_pad, uint32_t w[5]) {
  if (p0 < n_pad) {
    const uint4 v = *reinterpret_cast<const uint4*>(pad + p0);
    w[0] = v.x;
    w[1] = v.y;
    w[2] = v.z;
    w[3] = v.w;
    w[4] = *reinterpret_cast<const uint32_t*>(pad + p0 + 16);
  } else {
#pragma unroll
    for (int k = 0; k < 5; k++) w[k] = 0x01010101u * SENTINEL;
  }
}

// Keys of the 16 words at p0 .. p0 + 15; bit j of the result says whether
// word p0 + j is indexed.
__device__ __forceinline__ uint32_t word_keys16(const int8_t* pad, int64_t p0, int64_t n_pad, const int8_t* cls2,
                                                const int8_t* cls3, int32_t key[IX_PER]) {
  uint32_t w[5];
  load20(pad, p0, n_pad, w);
  return keys16_from(w, cls2, cls3, key);
}

__device__ __forceinline__ void load_classes(int8_t* cls2, int8_t* cls3) {
  if (threadIdx.x < NAA) {
    cls2[threadIdx.x] = c_cls2[threadIdx.x];
    cls3[threadIdx.x] = c_cls3[threadIdx.x];
  }
}

// hist[b * n_chunks + c] = words of bucket b in chunk c; behind those,
// hist_key[k * n_groups + g] += words of key k in the CTA's chunks, `per`
// consecutive ones of group g (several CTAs a group: added up in memory).
__global__ void __launch_bounds__(IX_THREADS) k_index_hist(const int8_t* pad, int64_t n_pad, IndexShape sh,
                                                           int32_t* hist) {
  __shared__ int32_t cnt[NKEYS];
  __shared__ int32_t bucket[IX_BUCKETS];
  __shared__ int8_t cls2[NAA], cls3[NAA];
  for (int k = threadIdx.x; k < NKEYS; k += IX_THREADS) cnt[k] = 0;
  if (threadIdx.x < IX_BUCKETS) bucket[threadIdx.x] = 0;
  load_classes(cls2, cls3);
  __syncthreads();
  const int64_t c0 = (int64_t)blockIdx.x * sh.per, c1 = min(c0 + sh.per, sh.n_chunks);
  for (int64_t c = c0; c < c1; c++) {
    int32_t key[IX_PER];
    const uint32_t valid = word_keys16(pad, c * IX_CHUNK + threadIdx.x * IX_PER, n_pad, cls2, cls3, key);
#pragma unroll
    for (int j = 0; j < IX_PER; j++)
      if (valid >> j & 1) {
        atomicAdd(&cnt[key[j]], 1);
        atomicAdd(&bucket[key[j] >> IX_LO_BITS], 1);
      }
    __syncthreads();
    if (threadIdx.x < IX_BUCKETS) {
      hist[threadIdx.x * sh.n_chunks + c] = bucket[threadIdx.x];
      bucket[threadIdx.x] = 0;
    }
    __syncthreads();
  }
  int32_t* hist_key = hist + IX_BUCKETS * sh.n_chunks + c0 / sh.group;
  for (int k = threadIdx.x; k < NKEYS; k += IX_THREADS)
    if (cnt[k]) atomicAdd(&hist_key[k * sh.n_groups], cnt[k]);
}

// key_off[k] = first slot of key k (off: the scanned tables; the key table's
// slots start after the bucket table's total, which is the number of words).
__global__ void k_index_key_off(const int64_t* off, IndexShape sh, int64_t* key_off) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t* off_key = off + IX_BUCKETS * sh.n_chunks;
  if (k < NKEYS) key_off[k] = off_key[k * sh.n_groups] - off_key[0];
  if (k == NKEYS) key_off[k] = off_key[0];
}

// Four bytes from any offset of a 4-byte aligned array.
__device__ __forceinline__ uint32_t word_at(const uint8_t* bytes, int at) {
  const uint32_t* w = reinterpret_cast<const uint32_t*>(bytes + (at & ~3));
  return __funnelshift_r(w[0], w[1], 8 * (at & 3));
}

// Counters of a stable counting pass over up to 128 digits: one column per
// warp, the columns WARPS + 2 apart so that a warp's digits spread over the
// banks.
template <int WARPS>
struct RankSmem {
  static constexpr int COL = WARPS + 2;
  uint16_t cnt[IX_LO * COL];
  int32_t wsum[WARPS];

  __device__ void clear() {
    for (int k = threadIdx.x; k < IX_LO * COL / 2; k += 32 * WARPS) reinterpret_cast<uint32_t*>(cnt)[k] = 0;
  }
  // Rank of this lane's word among those of its digit that its warp has met.
  // (Seven ballots find the lanes of the same digit faster than one
  // match.any: the pass over 205 M positions 0.98 ms against 1.23.)
  __device__ int rank(int warp, int lane, int digit, bool ok) {
    unsigned peers = __ballot_sync(0xffffffffu, ok);
#pragma unroll
    for (int k = 0; k < IX_LO_BITS; k++) {
      const bool bit = digit >> k & 1;
      const unsigned m = __ballot_sync(0xffffffffu, bit);
      peers &= bit ? m : ~m;
    }
    uint16_t* c = cnt + digit * COL + warp;
    const int have = ok ? *c : 0;
    __syncwarp();
    if (ok && lane == __ffs(peers) - 1) *c = (uint16_t)(have + __popc(peers));
    __syncwarp();
    return have + __popc(peers & ((1u << lane) - 1u));
  }
  // Counts to first places, digit by digit, the warps in order within one;
  // the total.  Between barriers of its own.
  __device__ int scan() {
    constexpr int PER = IX_LO * WARPS / (32 * WARPS);  // 4 counters a thread
    constexpr int PER_DIGIT = WARPS / PER;             // threads a digit
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    __syncthreads();
    uint16_t* c = cnt + (t / PER_DIGIT) * COL + (t % PER_DIGIT) * PER;
    const int c0 = c[0], c1 = c[1], c2 = c[2], c3 = c[3];
    int x = c0 + c1 + c2 + c3;
    const int mine = x;
#pragma unroll
    for (int d = 1; d < 32; d *= 2) {
      const int y = __shfl_up_sync(0xffffffffu, x, d);
      if (lane >= d) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    int before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < WARPS; w++) {
      const int v = wsum[w];
      if (w < warp) before += v;
      total += v;
    }
    const int e = before + x - mine;
    c[0] = (uint16_t)e;
    c[1] = (uint16_t)(e + c0);
    c[2] = (uint16_t)(e + c0 + c1);
    c[3] = (uint16_t)(e + c0 + c1 + c2);
    __syncthreads();
    return total;
  }
  __device__ int place(int warp, int digit, int rank) const { return cnt[digit * COL + warp] + rank; }
};

struct SplitSmem {
  uint32_t el[IX_CHUNK];                        // key << 14 | offset in the chunk, by bucket
  alignas(16) uint8_t code[IX_CHUNK + 16];
  int32_t slot[IX_BUCKETS];                     // first slot of each bucket less the index of its first word
  RankSmem<IX_WARPS> rank;
  int8_t cls2[NAA], cls3[NAA];
};
static_assert(IX_CHUNK <= 1 << 14 && NKEYS <= 1 << 14, "packing");
static_assert(sizeof(SplitSmem) <= 48 * 1024, "static shared memory");

// Bound by the ALU pipe (89 % busy, the ballots' selects; issue 65 %), one chunk
// a CTA and three CTAs an SM (four: 1.00 ms for 0.98 at 206 M positions, their
// 32 registers spill).
__global__ void __launch_bounds__(IX_THREADS, 3) k_index_split(const int8_t* pad, int64_t n_pad, IndexShape sh,
                                                               const int64_t* off, uint32_t* by_pos,
                                                               uint8_t* by_lo) {
  __shared__ SplitSmem sm;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int64_t c = blockIdx.x, q0 = c * IX_CHUNK;
  const uint4 gap = make_uint4(0x01010101u * SENTINEL, 0x01010101u * SENTINEL, 0x01010101u * SENTINEL,
                               0x01010101u * SENTINEL);
  // from n_pad on the words hold a sentinel; the bank's trailing slack covers the reads
  const int64_t p = q0 + 16 * t;
  *reinterpret_cast<uint4*>(sm.code + 16 * t) = p < n_pad ? *reinterpret_cast<const uint4*>(pad + p) : gap;
  if (t == 0)
    *reinterpret_cast<uint4*>(sm.code + IX_CHUNK) =
        q0 + IX_CHUNK < n_pad ? *reinterpret_cast<const uint4*>(pad + q0 + IX_CHUNK) : gap;
  if (t < IX_BUCKETS) sm.slot[t] = (int32_t)off[t * sh.n_chunks + c];
  load_classes(sm.cls2, sm.cls3);
  sm.rank.clear();
  __syncthreads();
  const int at0 = warp * (32 * IX_PER) + lane;
  uint32_t w[IX_PER];  // key << 16 | rank
#pragma unroll
  for (int j = 0; j < IX_PER; j++) {
    const uint32_t b = word_at(sm.code, at0 + 32 * j);
    const uint32_t a0 = b & 0xff, a1 = b >> 8 & 0xff, a2 = b >> 16 & 0xff, a3 = b >> 24;
    const bool ok = a0 < NAA && a1 < NAA && a2 < NAA && a3 < NAA;
    const int key = ok ? (((int)(a0 * 2) + sm.cls2[a1]) * 11 + sm.cls3[a2]) * 20 + (int)a3 : 0;
    const int r = sm.rank.rank(warp, lane, key >> IX_LO_BITS, ok);
    w[j] = ok ? (uint32_t)key << 16 | (uint32_t)r : 0xffffffffu;
  }
  const int n = sm.rank.scan();
#pragma unroll
  for (int j = 0; j < IX_PER; j++)
    if (w[j] != 0xffffffffu)
      sm.el[sm.rank.place(warp, (int)(w[j] >> (16 + IX_LO_BITS)), (int)(w[j] & 0xffff))] =
          w[j] >> 16 << 14 | (uint32_t)(at0 + 32 * j);
  if (t < IX_BUCKETS) sm.slot[t] -= sm.rank.place(0, t, 0);
  __syncthreads();
  for (int i = t; i < n; i += IX_THREADS) {
    const uint32_t e = sm.el[i];
    const int slot = sm.slot[e >> (14 + IX_LO_BITS)] + i;
    by_pos[slot] = (uint32_t)q0 + (e & 0x3fff);
    by_lo[slot] = (uint8_t)(e >> 14 & (IX_LO - 1));
  }
}

// Bound by the shared-memory pipe (84 % of its wavefronts in use; DRAM 35 %,
// writing 2.9 TB/s): each window passes it twice.  Cutting thirds of windows
// out of shared memory with three lanes each cost 5.9 wavefronts a word and
// 3.71 ms where this costs 3.11 (with match.any ranks; 2.96 with ballots).
//
// One bucket's words of one group, FILL_CHUNK at a time: sorted by the low
// digit, a key's words leave as one run of consecutive slots.  The window of
// a word at p is cells 0..25 = pad[p .. p+25] and 26..47 = pad[p-1], pad[p-2],
// .., pad[p-22]; with S[j] = pad[p - 22 + j] that is S[22..47] and S[21] ..
// S[0].  Four lanes fetch the 64 aligned bytes around S (pad is 16-byte
// aligned with slack on both sides, so they stay inside it) into the warp's
// corner of shared memory, one lane shifts the window out of them, and the
// warp's 32 windows leave as 16-byte stores, consecutive within a key's run.
constexpr int FILL_THREADS = 256;
constexpr int FILL_WARPS = FILL_THREADS / 32;
constexpr int FILL_PER = 8;
constexpr int FILL_CHUNK = FILL_THREADS * FILL_PER;  // 2048
// 32-bit words a window's bytes take in the corner: 16 and 4, so that rows
// four apart differ by 16 banks (a quarter warp stores two such rows at once)
// and the rows a quarter warp reads, one a lane, lie in different banks
constexpr int FILL_ROW = 20;
struct FillSmem {
  uint32_t pos[FILL_CHUNK];
  uint8_t lo[FILL_CHUNK];
  alignas(16) uint32_t corner[FILL_WARPS][32 * FILL_ROW];
  int32_t slot[IX_LO];                               // next slot of each key, less the index of its first word
  RankSmem<FILL_WARPS> rank;
};
static_assert(sizeof(FillSmem) <= 48 * 1024, "static shared memory");

__global__ void __launch_bounds__(FILL_THREADS, 4) k_index_fill(const int8_t* pad, IndexShape sh, const int64_t* off,
                                                                const uint32_t* by_pos, const uint8_t* by_lo,
                                                                uint32_t* pos, int8_t* nb) {
  __shared__ FillSmem sm;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int64_t g = blockIdx.x / IX_BUCKETS;
  const int b = (int)(blockIdx.x - g * IX_BUCKETS);
  // the next group's first slot ends this one's (the last group's: the next
  // bucket's first slot, or the total, which is where the key table starts)
  const int64_t cell = b * sh.n_chunks + g * sh.group, cell_end = b * sh.n_chunks + min((g + 1) * sh.group, sh.n_chunks);
  const int64_t i0 = off[cell], i1 = off[cell_end];
  if (i0 == i1) return;
  const int64_t* off_key = off + IX_BUCKETS * sh.n_chunks;
  if (t < IX_LO) {
    const int64_t k = b * IX_LO + t;
    sm.slot[t] = k < NKEYS ? (int32_t)(off_key[k * sh.n_groups + g] - off_key[0]) : 0;
  }
  for (int64_t c0 = i0; c0 < i1; c0 += FILL_CHUNK) {
    const int n = (int)min((int64_t)FILL_CHUNK, i1 - c0);
    const int steps = (n + FILL_THREADS - 1) / FILL_THREADS;  // each warp's share of the words, in 32s
    const int at0 = warp * 32 * steps + lane;
    sm.rank.clear();
    uint32_t p[FILL_PER], w[FILL_PER];  // position; rank << 8 | low digit
#pragma unroll
    for (int j = 0; j < FILL_PER; j++) {
      const bool ok = j < steps && at0 + 32 * j < n;
      p[j] = ok ? by_pos[c0 + at0 + 32 * j] : 0;
      w[j] = ok ? by_lo[c0 + at0 + 32 * j] : IX_LO;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < FILL_PER; j++)
      if (j < steps) w[j] |= (uint32_t)sm.rank.rank(warp, lane, (int)w[j] & (IX_LO - 1), w[j] < IX_LO) << 8;
    sm.rank.scan();
#pragma unroll
    for (int j = 0; j < FILL_PER; j++)
      if (!(w[j] & IX_LO)) {
        const int at = sm.rank.place(warp, (int)(w[j] & 0xff), (int)(w[j] >> 8));
        sm.pos[at] = p[j];
        sm.lo[at] = (uint8_t)w[j];
      }
    if (t < IX_LO) sm.slot[t] -= sm.rank.place(0, t, 0);
    __syncthreads();
    for (int i = t; i < n; i += FILL_THREADS) pos[sm.slot[sm.lo[i]] + i] = sm.pos[i];
    uint32_t* corner = sm.corner[warp];
    // the row and quarter of this lane's fetches, and where they are kept
    const int frow = (lane >> 3) + (lane & 4), quarter = lane & 3;
    for (int i = 32 * warp; i < n; i += FILL_THREADS) {
      uint4 v[4];
#pragma unroll
      for (int r = 0; r < 4; r++) {
        const int x = min(i + 8 * r + frow, n - 1);
        v[r] = __ldg(reinterpret_cast<const uint4*>(pad + (((int64_t)sm.pos[x] - 22) & ~(int64_t)15)) + quarter);
      }
#pragma unroll
      for (int r = 0; r < 4; r++)
        *reinterpret_cast<uint4*>(corner + (8 * r + frow) * FILL_ROW + 4 * quarter) = v[r];
      __syncwarp();
      const int x = min(i + lane, n - 1);
      const uint32_t o = (sm.pos[x] - 22) & 15;
      uint32_t raw[16], W[13], S[12], cell[12];
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const uint4 r = *reinterpret_cast<const uint4*>(corner + lane * FILL_ROW + 4 * k);
        raw[4 * k] = r.x, raw[4 * k + 1] = r.y, raw[4 * k + 2] = r.z, raw[4 * k + 3] = r.w;
      }
      const bool two = o & 8, one = o & 4;
#pragma unroll
      for (int k = 0; k < 14; k++) raw[k] = two ? raw[k + 2] : raw[k];
#pragma unroll
      for (int k = 0; k < 13; k++) W[k] = one ? raw[k + 1] : raw[k];
#pragma unroll
      for (int k = 0; k < 12; k++) S[k] = __funnelshift_r(W[k], W[k + 1], 8 * (o & 3));  // S[4k ..]
#pragma unroll
      for (int k = 0; k < 6; k++) cell[k] = __funnelshift_r(S[5 + k], S[6 + k], 16);     // S[22 + 4k ..]
      cell[6] = __byte_perm(S[11], S[5], 0x4532);                                        // S46 S47 S21 S20
#pragma unroll
      for (int k = 7; k < 12; k++) cell[k] = __byte_perm(S[11 - k], 0, 0x0123);          // S[4(11-k)+3] .. S[4(11-k)]
      __syncwarp();
      uint4* out = reinterpret_cast<uint4*>(corner);
      out[3 * lane] = make_uint4(cell[0], cell[1], cell[2], cell[3]);
      out[3 * lane + 1] = make_uint4(cell[4], cell[5], cell[6], cell[7]);
      out[3 * lane + 2] = make_uint4(cell[8], cell[9], cell[10], cell[11]);
      const int slot = sm.slot[sm.lo[x]] + x;
      __syncwarp();
#pragma unroll
      for (int r = 0; r < 3; r++) {
        const int e = 32 * r + lane, row = e / 3;
        const int64_t to = __shfl_sync(0xffffffffu, slot, row);
        if (i + row < n) *reinterpret_cast<uint4*>(nb + to * WIN + 16 * (e - 3 * row)) = out[e];
      }
      __syncwarp();
    }
    __syncthreads();
    // a key's next word follows this chunk's last: its first word's index
    // back on, and the count (the next digit's first place less its own)
    if (t < IX_LO) sm.slot[t] += t + 1 < IX_LO ? sm.rank.place(0, t + 1, 0) : n;
    __syncthreads();
  }
}

__global__ void k_block_seq(const int64_t* pad_off, int32_t n_seqs, int64_t n_blk, int32_t* blk) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_blk; i += (int64_t)gridDim.x * blockDim.x)
    blk[i] = n_seqs > 0 ? find_seq(pad_off, n_seqs, i * SEQ_BLK) : 0;
}

__global__ void k_export_pos(const uint32_t* pos, int64_t n, const int64_t* pad_off, int32_t n_seqs, int32_t* out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    int64_t p = pos[i];
    int32_t s = find_seq(pad_off, n_seqs, p);
    out[i] = (int32_t)(p - (int64_t)GAP * (s + 1));
  }
}

// ---------------------------------------------------------------------------
// Six-frame translation.  Standard genetic code, codons indexed by
// n1*16 + n2*4 + n3 with A C G T = 0 1 2 3.
// ---------------------------------------------------------------------------
__constant__ char c_code[65] = "KNKNTTTTRSRSIIMIQHQHPPPPRRRRLLLLEDEDAAAAGGGGVVVV*Y*YSSSS*CWCLFLF";
__constant__ int8_t c_aa_of_letter[26];

// One thread per 16 consecutive translated residues: one binary search for
// the sequence (contig, frame) of the first.  Where all 16 lie in it, their 48
// nucleotides are 13 aligned words, a codon's index one dot product of three
// of its bytes (read backwards and complemented in the reverse frames: 63 less
// the mirrored sum) and the residues one 16-byte store; the others walk
// forward byte by byte.  40 M residues of 20 M bases: 52 us, byte by byte 141
// (k_check_codes of the bases, 16 a load instead of one: 10 us and 37).
constexpr int TR_PER = 16;
__global__ void k_translate6(const uint8_t* dna, const int64_t* contig_off, int32_t n_contigs, const int64_t* seq_off,
                             int64_t n_aa, int8_t* aa) {
  // codon -> residue code, in shared memory (lanes read different entries,
  // which constant memory would serialise)
  __shared__ int8_t code_of[64];
  if (threadIdx.x < 64) {
    const char letter = c_code[threadIdx.x];
    code_of[threadIdx.x] = letter == '*' ? (int8_t)STOP : c_aa_of_letter[letter - 'A'];
  }
  __syncthreads();
  const int32_t n_seqs = 6 * n_contigs;
  const int64_t n_chunks = (n_aa + TR_PER - 1) / TR_PER;
  const bool vec = (reinterpret_cast<uintptr_t>(aa) & 15) == 0;
  const uintptr_t dna0 = reinterpret_cast<uintptr_t>(dna), dna1 = dna0 + (uintptr_t)contig_off[n_contigs];
  for (int64_t ch = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; ch < n_chunks;
       ch += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t0 = ch * TR_PER, t1 = min(t0 + TR_PER, n_aa);
    // the last sequence with seq_off[s] <= t that is not empty holds t
    int32_t s = find_seq(seq_off, n_seqs, t0);
    if (vec && t1 - t0 == TR_PER && seq_off[s + 1] >= t1) {
      const int32_t c = s / 6, f = s % 6;
      const bool rev = f >= 3;
      const int64_t q = (f % 3) + 3 * (t0 - seq_off[s]);
      // the 48 nucleotides from `lo` on, inside the contig
      const uintptr_t lo = dna0 + (uintptr_t)(rev ? contig_off[c + 1] - q - 48 : contig_off[c] + q);
      const uintptr_t first = lo & ~(uintptr_t)3;
      if (first >= dna0 && first + 52 <= dna1) {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(first);
        const uint32_t sh = 8 * (uint32_t)(lo & 3), weights = rev ? 0x00100401u : 0x00010410u;
        uint32_t w[13], S[13], r[4];
#pragma unroll
        for (int k = 0; k < 13; k++) w[k] = __ldg(src + k);
#pragma unroll
        for (int k = 0; k < 12; k++) S[k] = __funnelshift_r(w[k], w[k + 1], sh);
        S[12] = 0;
#pragma unroll
        for (int j = 0; j < 4; j++) {
          r[j] = 0;
#pragma unroll
          for (int k = 4 * j; k < 4 * j + 4; k++) {  // the codon of bytes 3k .. 3k + 2
            const uint32_t x = __funnelshift_r(S[3 * k >> 2], S[(3 * k >> 2) + 1], 8 * (3 * k & 3));
            const uint32_t v = __dp4a(x, weights, 0u);
            r[j] |= (uint32_t)(uint8_t)code_of[rev ? 63 - v : v] << (8 * (k & 3));
          }
        }
        *reinterpret_cast<uint4*>(aa + t0) =
            rev ? make_uint4(__byte_perm(r[3], 0, 0x0123), __byte_perm(r[2], 0, 0x0123), __byte_perm(r[1], 0, 0x0123),
                             __byte_perm(r[0], 0, 0x0123))
                : make_uint4(r[0], r[1], r[2], r[3]);
        continue;
      }
    }
    for (int64_t t = t0; t < t1; t++) {
      while (s + 1 < n_seqs && seq_off[s + 1] <= t) s++;
      const int32_t c = s / 6, f = s % 6;
      const int64_t i = t - seq_off[s];
      const int64_t c0 = contig_off[c], L = contig_off[c + 1] - c0;
      const int64_t q = (f % 3) + 3 * i;
      int n1, n2, n3;
      if (f < 3) {
        n1 = dna[c0 + q];
        n2 = dna[c0 + q + 1];
        n3 = dna[c0 + q + 2];
      } else {
        n1 = 3 - dna[c0 + L - 1 - q];
        n2 = 3 - dna[c0 + L - 2 - q];
        n3 = 3 - dna[c0 + L - 3 - q];
      }
      aa[t] = code_of[n1 * 16 + n2 * 4 + n3];
    }
  }
}

cudaError_t upload_code_letters_once() {
  static std::atomic<bool> done[64];  // per device; calls may come from several threads
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 64 && done[dev]) return cudaSuccess;
  int8_t m[26];
  for (int i = 0; i < 26; i++) m[i] = -1;
  for (int i = 0; i < NAA; i++) m[ALPHABET[i] - 'A'] = (int8_t)i;
  cudaError_t e = cudaMemcpyToSymbol(c_aa_of_letter, m, sizeof(m));
  if (e == cudaSuccess && dev < 64) done[dev] = true;
  return e;
}

static unsigned grid_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  if (b > 152 * 64) b = 152 * 64;
  if (b < 1) b = 1;
  return (unsigned)b;
}

cudaError_t launch_check_codes(const int8_t* codes, int64_t n, int hi, int* bad, cudaStream_t st) {
  if (n > 0) {
    note_launch();
    k_check_codes<<<grid_for((n + 15) / 16, 256), 256, 0, st>>>(codes, n, hi, bad);
  }
  return cudaGetLastError();
}

cudaError_t launch_build_pad(const int8_t* codes, const int64_t* seq_off, int32_t n_seqs, int64_t n_res, int hi,
                             int8_t* pad, int* bad, cudaStream_t st) {
  if (n_res > 0) {
    note_launch();
    k_build_pad<<<grid_for((n_res + 15) / 16, 256), 256, 0, st>>>(codes, seq_off, n_seqs, n_res, hi, pad, bad);
  }
  return cudaGetLastError();
}

IndexShape index_shape(int64_t n_pad) {
  IndexShape sh;
  sh.n_chunks = (n_pad + IX_CHUNK - 1) / IX_CHUNK;
  // four CTAs of k_index_hist an SM before one takes more than one chunk
  sh.per = 1;
  while (sh.per < 8 && sh.n_chunks / (2 * sh.per) >= 608) sh.per *= 2;
  // 18 groups or more keep 152 SMs busy with a bucket each; a group of 64
  // chunks gives each of its 69 buckets some 6,000 words
  sh.group = std::min<int64_t>(64, std::max<int64_t>(1, sh.n_chunks / 18));
  sh.group = (sh.group + sh.per - 1) / sh.per * sh.per;
  sh.n_groups = (sh.n_chunks + sh.group - 1) / sh.group;
  return sh;
}

int64_t index_cells(const IndexShape& sh) { return IX_BUCKETS * sh.n_chunks + (int64_t)NKEYS * sh.n_groups; }

cudaError_t launch_index_hist(const int8_t* pad, int64_t n_pad, const IndexShape& sh, int32_t* hist,
                              cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(hist + IX_BUCKETS * sh.n_chunks, 0, (size_t)NKEYS * sh.n_groups * sizeof(int32_t), st);
  if (e != cudaSuccess) return e;
  note_launch();
  k_index_hist<<<(unsigned)((sh.n_chunks + sh.per - 1) / sh.per), IX_THREADS, 0, st>>>(pad, n_pad, sh, hist);
  return cudaGetLastError();
}

cudaError_t launch_index_key_off(const int64_t* off, const IndexShape& sh, int64_t* key_off, cudaStream_t st) {
  note_launch();
  k_index_key_off<<<(NKEYS + 1 + 255) / 256, 256, 0, st>>>(off, sh, key_off);
  return cudaGetLastError();
}

cudaError_t launch_index_split(const int8_t* pad, int64_t n_pad, const IndexShape& sh, const int64_t* off,
                               uint32_t* by_pos, uint8_t* by_lo, cudaStream_t st) {
  note_launch();
  k_index_split<<<(unsigned)sh.n_chunks, IX_THREADS, 0, st>>>(pad, n_pad, sh, off, by_pos, by_lo);
  return cudaGetLastError();
}

cudaError_t launch_index_fill(const int8_t* pad, const IndexShape& sh, const int64_t* off, const uint32_t* by_pos,
                              const uint8_t* by_lo, uint32_t* pos, int8_t* nb, cudaStream_t st) {
  note_launch();
  k_index_fill<<<(unsigned)(sh.n_groups * IX_BUCKETS), FILL_THREADS, 0, st>>>(pad, sh, off, by_pos, by_lo, pos, nb);
  return cudaGetLastError();
}

cudaError_t launch_block_seq(const int64_t* pad_off, int32_t n_seqs, int64_t n_pad, int32_t* blk, cudaStream_t st) {
  const int64_t n_blk = n_pad / SEQ_BLK + 1;
  note_launch();
  k_block_seq<<<grid_for(n_blk, 256), 256, 0, st>>>(pad_off, n_seqs, n_blk, blk);
  return cudaGetLastError();
}

cudaError_t launch_export_pos(const uint32_t* pos, int64_t n, const int64_t* pad_off, int32_t n_seqs, int32_t* out,
                              cudaStream_t st) {
  if (n > 0) {
    note_launch();
    k_export_pos<<<grid_for(n, 256), 256, 0, st>>>(pos, n, pad_off, n_seqs, out);
  }
  return cudaGetLastError();
}

cudaError_t launch_translate6(const uint8_t* dna, const int64_t* contig_off, int32_t n_contigs, const int64_t* seq_off,
                              int64_t n_aa, int8_t* aa, cudaStream_t st) {
  cudaError_t e = upload_code_letters_once();
  if (e != cudaSuccess) return e;
  if (n_aa > 0) {
    note_launch();
    k_translate6<<<grid_for((n_aa + TR_PER - 1) / TR_PER, 256), 256, 0, st>>>(dna, contig_off, n_contigs, seq_off,
                                                                              n_aa, aa);
  }
  return cudaGetLastError();
}

}  // namespace plast
