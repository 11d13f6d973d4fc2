// ungapped_mma.cu -- stage 2 (Section 3.3.3, the loop of Annex 4) with an
// exact filter on the fp4 tensor cores of sm_103a.
//
// Of the pairs of an ordinary protein bank one in some 570 reaches S1, so
// most of the work of the direct form (ungapped.cu: every running sum and
// maximum of every pair) goes to pairs that are dropped.  Here the tensor
// cores compute an upper bound of every pair's score, and only the pairs
// whose bound reaches S1 (about 1.6 % at S1 = 38) get the exact extension.
// The bound never lies below the score, so the hits are the same.
//
// The bound.  Let P be the positive part of the substitution score, rounded
// up to a value e2m1 can hold (times 2: 1 2 3 4 6 8 12; only the diagonal
// entries 5, 7, 9 and 11 are moved), and N = score - P <= 0 (all of its values
// are e2m1 values too, and it takes the rounding back).  Cut each side of the
// window into segments; the largest prefix sum ending inside a segment is at
// most (sum of P + N before the segment) + (sum of P in it).  With V the
// maximum of that over the segments of a side, the ungapped score is at most
// V_right + V_left (the seed cells 0-3 are taken exactly: their sum is their
// largest prefix).  Three segments a side: right 7, 6 and 9 cells after the
// seed, left 6, 6 and 10.
//
// As a contraction.  A window of bank 2 is a one-hot vector over (cell,
// residue code), a row of bank 1 the scores of its residues: the sum over
// a run of cells is a product of the two.  Three cells of 20 codes make one
// K = 64 step of tcgen05.mma kind::mxf4; a pair's accumulator adds the P step
// of the segment (read: the segment's bound), then the N steps of the same
// cells, then the next segment.  A first step with a block scale of 2^23 sets
// every accumulator to 1.5 * 2^23: the sums are whole numbers, so from there
// on the low half of the fp32 word is the sum as int16, and tcgen05.ld
// .pack::16b delivers two rows a register, ready for int16x2 maxima (half the
// ALU work and registers of fp32 maxima).  M = 128 windows, N = 16 to 64 rows;
// the right and the left side are two accumulators, and the rows go in two
// halves: four chains of MMA and read, so that each one's latency is behind
// the others' work.  The one-hot operand lives in tensor memory (it is used
// once for P and once for N; from shared memory it would double the operand
// traffic); the rows' profile, 25 steps of 32 bytes a row, in shared memory.
//
// Roles of a CTA (one per SM):
//   8 epilogue warps   read the accumulators (32 windows x half of the rows a
//                      warp), keep the maxima, test the bound, leave the
//                      candidates as masks
//   8 expand warps     one side of a bank-2 window per lane: residue codes to
//                      one-hot words from a table with a private bank per
//                      lane (no conflicts), stored to tensor memory
//   8 extend warps     take an epilogue warp's masks, extend the candidates 32
//                      at a time exactly (one per lane), emit the hits
//   4 MMA warps        issue a chain's MMAs each
//   1 tile warp        fetches the tiles, ahead of the others
// They meet at two mbarriers per segment and half.  Every wait has a limit
// (struct Waits); a wait that runs out raises the launch's error flag and ends
// the CTA's work.
// The roles' loops are kept short: straight-line code of this many roles
// does not stay in the instruction caches.
//
// What bounds it: instruction issue and the latency of the chains (a pass of
// 128 windows x 128 rows takes 2.3 us on an SM: issue 66 %, shared memory
// wavefronts 71 %, tensor pipe 33 %, ALU 48 %).  Stage 2 of 10,000 x 100,000
// proteins (2.15e10 pairs): 20.6 ms, with the plain wide kernel 45.5 ms; of
// 10,000 x 10,000: 3.1 ms against 4.5.  Measured on the way: fp32 maxima of
// the accumulators (no base of 2^23) 33.8 ms; the one-hot steps by one warp
// a quadrant instead of two 24.8; candidates queued by the epilogue warps
// instead of masks decoded by the extend warps 22.4; tiles fetched by an
// extend warp instead of one that runs ahead 22.7 (10,000 x 10,000: 4.0).
#define PLAST_WHOLE_PROGRAM  // see build.py
#include <atomic>

#include "common.cuh"
#include "ungapped.cuh"

namespace plast {

namespace {

constexpr int EPI_WARPS = 8;
constexpr int EXP_WARPS = 8;  // four a side
constexpr int EXT_WARPS = EPI_WARPS;
constexpr int EXP_WARP = EPI_WARPS;
constexpr int EXT_WARP = EXP_WARP + EXP_WARPS;
constexpr int MMA_WARP = EXT_WARP + EXT_WARPS;
constexpr int TILE_WARP = MMA_WARP + 4;
constexpr int TC_THREADS = (TILE_WARP + 4) * 32;  // 1024: eight warpgroups (the last: the tile warp)
// registers a thread: launched with 64, the warpgroups then take 104
// (epilogue, two), 56 (expand, two), 64 (extend, two), 32 (MMA) and 32 (tile):
// 8 x 64 in all
constexpr int TC_REGS_EPI = 104, TC_REGS_EXP = 56, TC_REGS_EXT = 64, TC_REGS_MMA = 32;
constexpr int TC_M = UNG_TC_PASS;                // windows per pass
constexpr int TC_N = UNG_T1;                     // rows of a full tile
static_assert(TC_M == 128 && TC_N == 128, "one accumulator lane per window, 128 columns");

// K steps of three cells: 0-7 the right side (cells 1, 2, 4 and on), 8-15 the
// left side (the last holds one cell).
constexpr int KSTEPS = 16;
constexpr int NSEG = 3;
// first K step and K steps of segment `seg` of a side (0: right, 1: left)
__host__ __device__ constexpr int seg_first(int side, int seg) {
  return side == 0 ? (seg == 0 ? 0 : seg == 1 ? 3 : 5) : (seg == 0 ? 8 : seg == 1 ? 10 : 12);
}
__host__ __device__ constexpr int seg_steps(int side, int seg) {
  return side == 0 ? (seg == 1 ? 2 : 3) : (seg == 2 ? 4 : 2);
}
constexpr int NGROUP = 2 * NSEG;  // one-hot groups: one per segment, in the order of use (side = g & 1)
// Profile slots: P of the 16 steps, then N of the steps of the first two
// segments of each side.
constexpr int SLOT_N0 = KSTEPS;           // N of steps 0-4
constexpr int SLOT_N8 = KSTEPS + 5;       // N of steps 8-11
constexpr int SLOT_BASE = KSTEPS + 5 + 4;  // the accumulators' base: 1.5 in the first dimension of every row
constexpr int NSLOT = SLOT_BASE + 1;       // 26
constexpr int SLOT_BYTES = TC_N * 32;     // [2 chunks of 16 bytes][128 rows]
constexpr int CHUNK_BYTES = TC_N * 16;

// Profile slot of a step's N plane (the P plane's slot is the step).
__host__ __device__ constexpr int slot_n(int step) { return step < 8 ? SLOT_N0 + step : SLOT_N8 + (step - 8); }
// Cell t (0-2) of a K step: 1, 2 and 4 for step 0, 3 step + 2 + t for the
// others; 48 and above: none (the last two of step 15).
__host__ __device__ constexpr int cell_of(int step, int t) { return 3 * step + 2 + t - (step == 0 && t < 2); }

// A row's residue codes as the extend warps use them: their part of a score's
// address, (code >> 2) * 128 + (code & 3); and back.
__device__ __forceinline__ uint32_t row_entries(uint32_t two_codes) {
  return ((two_codes << 5) & 0x03800380u) | (two_codes & 0x00030003u);
}
__device__ __forceinline__ uint32_t row_code(uint32_t entry) { return (entry >> 7) * 4 + (entry & 3); }

// tensor memory columns
constexpr uint32_t TM_ACC = 64;    // accumulator 2 * side + half of the rows at 64 times that
constexpr uint32_t TM_A = 256;     // one-hot steps, 8 columns each
constexpr uint32_t TM_BASE = 384;  // the base's step: 1 in the first dimension
constexpr uint32_t TM_SF1 = 392;   // block scales: 1, 2 (the scores are held halved), 2^23 (the base)
constexpr uint32_t TM_SF2 = 400;
constexpr uint32_t TM_SFB = 408;
constexpr uint32_t TM_COLS = 512;

// shared memory
constexpr int LUT_STRIDE = 32 * 16;                        // one code: three words (and one of padding) of 32 lanes
constexpr int LUT_CODES = NCODE + 1;                       // the last: no cell, all zero
constexpr int LUT_BYTES = LUT_CODES * LUT_STRIDE;          // per shift (0 and 16 bits)
constexpr int ROW_STRIDE = 112;                            // 48 uint16 (row_entries), an odd number of 16-byte banks
constexpr int ROWS_BYTES = TC_N * ROW_STRIDE;              // the rows of one tile
constexpr int WIN_STRIDE = 36;                             // an expand lane's part of a window: 9 words, conflict-free bytes
constexpr int LEFT_BYTE = 16;                              // first byte of the left side's part
constexpr int RING = 8;                                    // passes of an epilogue warp whose masks are on their way
constexpr int QCAP = 64;                                   // candidates of an extend warp
constexpr int HBUF = 32;
constexpr int TILES = 4;                                   // tile slots
constexpr int TILE_ROWS = 3;                               // row buffers
constexpr int OFF_PROF = 0;
constexpr int OFF_LUT = OFF_PROF + NSLOT * SLOT_BYTES;     // 106496
constexpr int OFF_ROWS = OFF_LUT + 2 * LUT_BYTES;
constexpr int OFF_PLUT = OFF_ROWS + TILE_ROWS * ROWS_BYTES;        // P, N, seed and seed correction words per code
constexpr int PLUT_BYTES = 4 * NCODE * 16;
// Scores for the exact extension, a bank per lane: row code a, window code b
// of lane l at b * TAB_B + (a >> 2) * 128 + 4 l + (a & 3).  (One table for the
// warp: 3.4 wavefronts a look-up, and shared memory bound the kernel.)
constexpr int OFF_TAB = OFF_PLUT + PLUT_BYTES;
constexpr int TAB_B = (NCODE + 3) / 4 * 128;
constexpr int TAB_BYTES = NCODE * TAB_B;                   // 16896
constexpr int OFF_WIN = OFF_TAB + TAB_BYTES;
constexpr int OFF_RING = (OFF_WIN + 2 * TC_M * WIN_STRIDE + 15) & ~15;
constexpr int OFF_QUEUE = OFF_RING + EPI_WARPS * RING * 32 * 8;
constexpr int OFF_HKEY = OFF_QUEUE + EXT_WARPS * QCAP * 8;
constexpr int OFF_HVAL = OFF_HKEY + EXT_WARPS * HBUF * 8;
constexpr int OFF_BAR = OFF_HVAL + EXT_WARPS * HBUF * 4;
constexpr int OFF_WAITS = OFF_BAR + (4 * NGROUP + 3) * 8;  // abort flag and wait limit
constexpr int OFF_MISC = OFF_WAITS + 8;                    // tensor memory address, tiles fetched
// per epilogue warp: passes written, passes taken; per extend warp: tiles ended
constexpr int OFF_RPOS = (OFF_MISC + 8 + 15) & ~15;
constexpr int RP_TAKEN = EPI_WARPS, RP_EXT = 2 * EPI_WARPS;
constexpr int RP_WORDS = 2 * EPI_WARPS + EXT_WARPS;
constexpr int OFF_SLOTS = (OFF_RPOS + RP_WORDS * 4 + 15) & ~15;
constexpr int SLOT_INFO = 48;
constexpr int TC_SMEM = OFF_SLOTS + TILES * SLOT_INFO;
static_assert(OFF_LUT % 128 == 0 && OFF_HKEY % 8 == 0 && OFF_BAR % 8 == 0 && OFF_ROWS % 16 == 0, "alignment");
static_assert(OFF_PLUT % 16 == 0, "alignment");
static_assert(TC_SMEM <= 232448, "shared memory per CTA");

// barriers, per segment g (in the order of use) and half of the rows; each
// completes once a pass.
// GO: the MMAs of the segment may run: its one-hot steps are written (the
//     expand warps) and the accumulator's previous use is read (the half's
//     epilogue warps)
// DONE: its MMAs have ended (the accumulator can be read, the one-hot steps
//     that no later segment uses written again)
// and per tile
// READ: the epilogue warps have read the last tile's accumulators (its MMAs
//     have ended: the profile may be rebuilt)
// PROF: the tile's profile is built
enum { BAR_GO = 0, BAR_DONE = 2 * NGROUP, BAR_READ = 4 * NGROUP, BAR_PROF, BAR_DRAIN };

__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// A CTA's waits: each ends after `limit` clocks, UNG_WAIT_CLOCKS (two seconds; a
// pass takes microseconds) unless a caller has set fewer; one that runs out
// raises `abort`, and a raised `abort` ends every later wait.  The tile warp,
// which waits for whole tiles, counts from the last pass that ended.  (Both
// in one word of shared memory and 32-bit clocks: the limit in two registers
// and 64 bits cost the stage 2 of ordinary banks 3 %.)
struct Waits {
  int abort;
  uint32_t limit;
};
__device__ __forceinline__ uint32_t now() { return (uint32_t)clock(); }
__device__ __forceinline__ bool over(Waits* waits, uint32_t t0) {  // (the whole warp)
  int abort;
  uint32_t limit;
  asm volatile("ld.volatile.shared.v2.u32 {%0, %1}, [%2];" : "=r"(abort), "=r"(limit) : "r"(saddr(waits)) : "memory");
  if (!__any_sync(0xffffffffu, abort || now() - t0 > limit)) return false;
  *(volatile int*)&waits->abort = 1;
  return true;
}

__device__ __forceinline__ bool bar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0u;
}
// Waits for the phase of the given parity.  (The votes keep the warp's lanes
// together: loops that each lane leaves by itself cost more than the votes.)
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity, Waits* waits) {
  if (__any_sync(0xffffffffu, bar_try(bar, parity))) return true;
  const uint32_t t0 = now();
  for (;;) {
    if (__any_sync(0xffffffffu, bar_try(bar, parity))) return true;
    if (over(waits, t0)) return false;
  }
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// One thread of the warp, as a predicate the compiler knows to be one thread
// (a lane test costs 90 clocks an MMA in moves to uniform registers, this 12).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0u;
}

// One K = 64 step: 128 windows (tensor memory) x N rows (shared memory); ACC:
// added to the accumulator, else the accumulator is set.
template <int ACC>
__device__ __forceinline__ void tc_mma(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t sfa) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], [%1], %2, %3, [%5], [%6], p;\n\t}" ::"r"(d),
      "r"(a), "l"(b), "r"(idesc), "n"(ACC), "r"(sfa), "r"(TM_SF1)
      : "memory");
}

// Shared-memory operand: 8-row x 16-byte core matrices, no swizzle, the two
// 16-byte chunks of a step CHUNK_BYTES apart, 8-row groups 128 bytes apart.
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3fff) | ((uint64_t)(CHUNK_BYTES >> 4) << 16) | ((uint64_t)(128 >> 4) << 32) |
         ((uint64_t)1 << 46);
}

__device__ __forceinline__ void tm_store8(uint32_t addr, const uint32_t (&w)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(addr), "r"(w[0]),
               "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}

// 2 NW accumulator columns of the warp's 32 lanes, the low halves of two
// columns a register.
template <int NW>
__device__ __forceinline__ void tm_load_pack(uint32_t addr, uint32_t* v) {
  static_assert(NW == 8 || NW == 16 || NW == 24 || NW == 32, "words");
  if constexpr (NW == 8) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.pack::16b.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(addr)
                 : "memory");
  } else if constexpr (NW == 16) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.pack::16b.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(addr)
        : "memory");
  } else if constexpr (NW == 24) {
    tm_load_pack<16>(addr, v);
    tm_load_pack<8>(addr + 32, v + 16);
  } else {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.pack::16b.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,"
        "%29,%30,%31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
          "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(addr)
        : "memory");
  }
}
// Waits for the loads above; the values pass through it, so that no use of
// them moves ahead of the wait.
template <int N>
__device__ __forceinline__ void tm_wait_load(uint32_t* v) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < N; i++) asm volatile("" : "+r"(v[i]));
}

// e2m1 code of v / 2 for v in {0, +-1, 2, 3, 4, 6, 8, 12}
__device__ __forceinline__ uint32_t e2m1(int v) {
  const int a = v < 0 ? -v : v;
  const uint32_t m = a <= 4 ? (uint32_t)a : a == 6 ? 5u : a == 8 ? 6u : 7u;
  return m | (v < 0 ? 8u : 0u);
}
// the smallest e2m1 value (times 2) at or above v, -12 <= v <= 12
__device__ __forceinline__ int round_up_e2m1(int v) {
  if (v > 8) return 12;
  if (v > 6) return 8;
  if (v > 4) return 6;
  if (v >= -4) return v;
  return v >= -6 ? (v == -6 ? -6 : -4) : v >= -8 ? (v == -8 ? -8 : -6) : v >= -12 ? (v == -12 ? -12 : -8) : -12;
}

// The score the bound uses for row code a against window code b < 20: the
// window codes 20 (stop) and 21 (sentinel) are taken as WILD, which no row
// scores below them; the stop row's entry there covers stop against stop.
constexpr int WILD = 17;  // W
__device__ __forceinline__ int bound_score(const int8_t* score, int a, int b) {
  int v = score[a * NCODE + b];
  if (b == WILD) v = max(v, max((int)score[a * NCODE + STOP], (int)score[a * NCODE + SENTINEL]));
  return max(v, -12);
}

// The substitution scores as a kernel parameter: this file is compiled as a
// whole program (setmaxnreg is ignored in relocatable device code), so it
// does not see the other files' constant memory.
struct ScoreTable {
  int8_t score[NCODE * NCODE];
};

// A tile as the roles use it.
struct TileInfo {
  int64_t u0, v0;    // first bank-1 and bank-2 CSR index
  int rows, n2;      // rows of the tile (0: no more tiles), windows of its range
  int half;          // rows of a half: the rows rounded up to 32, over 2
  uint32_t thr4;     // (the scores of cells 0 and 3, less S1) / 2 as the sum of four e2m1 values
};
static_assert(sizeof(TileInfo) <= SLOT_INFO, "tile slot size");

// Tile k of this CTA, once it has been fetched; false when there is
// none or the launch has failed.
__device__ __forceinline__ bool wait_tile(const unsigned char* smem, uint32_t k, TileInfo& t, Waits* waits) {
  volatile const uint32_t* fetched = reinterpret_cast<volatile const uint32_t*>(smem + OFF_MISC + 4);
  if (__any_sync(0xffffffffu, *fetched <= k)) {
    const uint32_t t0 = now();
    while (__any_sync(0xffffffffu, *fetched <= k)) {
      if (over(waits, t0)) return false;
      __nanosleep(64);
    }
  }
  __threadfence_block();
  t = *reinterpret_cast<const TileInfo*>(smem + OFF_SLOTS + (k % TILES) * SLOT_INFO);
  return t.rows > 0;
}

// ---------------------------------------------------------------------------
// expand warps
// ---------------------------------------------------------------------------
// One K step: its cells are bytes of the lane's window in shared memory.
__device__ __forceinline__ void expand_step(int step, uint32_t win, uint32_t lut, uint32_t tm) {
  uint32_t w[3][3];
#pragma unroll
  for (int t = 0; t < 3; t++) {
    uint32_t code;
    [[maybe_unused]] uint32_t pad;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(code) : "r"(win + cell_of(step, t)));
    const uint32_t at = lut + (t == 1 ? LUT_BYTES : 0) + code * LUT_STRIDE;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(w[t][0]), "=r"(w[t][1]), "=r"(w[t][2]), "=r"(pad)
                 : "r"(at));
  }
  // cell 0: bits 0-79, cell 1: bits 80-159 (its table is 16 bits up, from word
  // 2), cell 2: bits 160-239; bits 240-255, four dimensions that are always 1
  // (used by step 0: the bound's constant)
  const uint32_t o[8] = {w[0][0], w[0][1], w[0][2] | w[1][0], w[1][1], w[1][2], w[2][0], w[2][1], w[2][2] | 0x22220000u};
  tm_store8(tm + 8 * step, o);
}

// One pass: one side of the lane's window to one-hot steps, segment by segment
// as their last use has ended.
__device__ __forceinline__ bool expand_pass(int side, uint32_t win, uint32_t lut, uint32_t tm, uint32_t bars,
                                            uint32_t pass, Waits* waits, int lane) {
#pragma unroll 1
  for (int g = side; g < NGROUP; g += 2) {
    // the steps' last use: N in the side's next segment (none after the last)
    const int last = g + 2 < NGROUP ? g + 2 : g;
    for (int h = 0; h < 2; h++)
      if (!bar_wait(bars + 8 * (BAR_DONE + 2 * last + h), (pass + 1) & 1, waits)) return false;
    tc_fence_after();
    const int first = seg_first(side, g >> 1), end = first + seg_steps(side, g >> 1);
#pragma unroll 2
    for (int step = first; step < end; step++) expand_step(step, win, lut, tm);
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    tc_fence_before();
    __syncwarp();
    if (lane < 2) bar_arrive(bars + 8 * (BAR_GO + 2 * g + lane));
  }
  return true;
}

// ---------------------------------------------------------------------------
// extend warps
// ---------------------------------------------------------------------------
// The exact score (the loop of Annex 4) of one row against one window.
// row: the row's 48 entries; x, y, z: its window's codes; tab: the scores;
// lane4: 4 times the lane, in both halves.  A loop over thirds of the window:
// straight-line code would not stay in the instruction cache beside the other
// roles'.
__device__ __forceinline__ int exact_score(const uint4* row, uint4 x, uint4 y, uint4 z, const int8_t* tab,
                                           uint32_t lane4) {
  int s = 0, m = 0;
#pragma unroll 1
  for (int c = 0; c < 3; c++) {
    const uint4 ra = row[2 * c], rb = row[2 * c + 1];
    const uint32_t a2[8] = {ra.x, ra.y, ra.z, ra.w, rb.x, rb.y, rb.z, rb.w};
    const uint32_t b4[4] = {x.x, x.y, x.z, x.w};
    int v[16];
#pragma unroll
    for (int j = 0; j < 8; j++) {
      // two cells' addresses
      const uint32_t at = __byte_perm(b4[j >> 1], 0u, (j & 1) ? 0x4342u : 0x4140u) * TAB_B + a2[j] + lane4;
      v[2 * j] = tab[at & 0xffffu];
      v[2 * j + 1] = tab[at >> 16];
    }
#pragma unroll
    for (int j = 0; j < 8; j++) {
      if (2 * j == RIGHT - 16) s = c == 1 ? m : s;  // the reset of Annex 4 before cell 26
      const int u = s + v[2 * j];
      s = u + v[2 * j + 1];
      m = __vimax3_s32(m, u, s);
    }
    x = y;
    y = z;
  }
  return m;
}

// A warp's hits on their way out.
struct HitBuf {
  uint64_t* key;
  uint32_t* val;
  int n;  // warp-uniform
};

__device__ __forceinline__ void flush_hits(HitBuf& h, const UngArgs& a, int lane) {
  __syncwarp();
  unsigned long long at = 0;
  if (lane == 0) at = atomicAdd(a.out_count, (unsigned long long)h.n);
  at = __shfl_sync(0xffffffffu, at, 0) + lane;
  if (lane < h.n && (int64_t)at < a.cap) {
    a.out_key[at] = h.key[lane];
    a.out_val[at] = h.val[lane];
  }
  __syncwarp();
  h.n = 0;
}

struct ExtState {
  uint64_t* queue;  // QCAP candidates: row << 32 | window (offset in the tile's range)
  int n;            // warp-uniform
  HitBuf hits;
};

// Extends the queue's last min(32, n) candidates.
__device__ __forceinline__ void extend_queue(ExtState& e, const TileInfo& t, const UngArgs& a,
                                             const unsigned char* rows, const int8_t* tab, int lane) {
  const int n = min(32, e.n);
  __syncwarp();
  int score = -(1 << 20), row = 0;
  int64_t v = 0;
  if (lane < n) {
    const uint64_t c = e.queue[e.n - n + lane];
    row = (int)(c >> 32);
    v = t.v0 + (int64_t)(uint32_t)c;
    const uint4* src = reinterpret_cast<const uint4*>(a.nb2 + v * WIN);
    const uint4 x = __ldg(src), y = __ldg(src + 1), z = __ldg(src + 2);
    score = exact_score(reinterpret_cast<const uint4*>(rows + row * ROW_STRIDE), x, y, z, tab,
                        (uint32_t)lane * 0x00040004u);
  }
  __syncwarp();
  e.n -= n;
  const bool hit = score >= a.s1;
  const unsigned hits = __ballot_sync(0xffffffffu, hit);
  if (hits == 0u) return;
  const int total = __popc(hits);
  if (e.hits.n + total > HBUF) flush_hits(e.hits, a, lane);
  if (hit) {
    const int at = e.hits.n + __popc(hits & ((1u << lane) - 1u));
    e.hits.key[at] = ((uint64_t)a.pos1[t.u0 + row] << a.sh) | (uint64_t)a.pos2[v];
    e.hits.val[at] = (uint32_t)(uint16_t)score;
  }
  __syncwarp();
  e.hits.n += total;
}

// The tile's candidates of one epilogue warp, from the masks it leaves per
// pass (ring; rp: passes written and taken), extended 32 at a time.  row0,
// window0: the first row and, of a pass, window of the epilogue warp; pass:
// passes so far.
__device__ __forceinline__ bool extend_tile(ExtState& e, const TileInfo& t, const UngArgs& a, const unsigned char* rows,
                                            const int8_t* tab, const uint2* ring, volatile uint32_t* rp, int row0,
                                            int window0, uint32_t& pass, Waits* waits, int lane) {
  const int n_pass = (t.n2 + TC_M - 1) / TC_M;
  for (int p = 0; p < n_pass; p++, pass++) {
    for (const uint32_t t0 = now(); __shfl_sync(0xffffffffu, rp[0], 0) == pass;) {
      if (over(waits, t0)) return false;
      __nanosleep(100);
    }
    __threadfence_block();
    uint2 c = ring[(pass % RING) * 32 + lane];
    __syncwarp();
    if (lane == 0) rp[RP_TAKEN] = pass + 1;
    const uint32_t w = (uint32_t)(p * TC_M + window0 + lane);
    for (;;) {
      const unsigned with = __ballot_sync(0xffffffffu, (c.x | c.y) != 0u);
      if (with == 0u) break;
      if (c.x | c.y) {
        // row 4 j + b of a mask's 32 at bit 8 b + j
        const bool lo = c.x != 0u;
        const uint32_t m = lo ? c.x : c.y;
        const int bit = __ffs(m) - 1;
        if (lo) c.x = m & (m - 1u);
        else c.y = m & (m - 1u);
        e.queue[e.n + __popc(with & ((1u << lane) - 1u))] =
            ((uint64_t)(uint32_t)(row0 + (lo ? 0 : 32) + 4 * (bit & 7) + (bit >> 3)) << 32) | w;
      }
      e.n += __popc(with);
      if (e.n >= 32) extend_queue(e, t, a, rows, tab, lane);
    }
  }
  while (e.n > 0) extend_queue(e, t, a, rows, tab, lane);  // (the rows change with the tile)
  return true;
}

// ---------------------------------------------------------------------------
// epilogue warps
// ---------------------------------------------------------------------------
// Segment g of a pass: the half's 2 NW rows into m (a side's first segment) or
// maximised with it; then the accumulator may take the side's next segment.
template <int NW, bool FIRST>
__device__ __forceinline__ bool read_segment(uint32_t (&m)[NW], int g, uint32_t bars, int half, uint32_t pass,
                                             uint32_t tm, Waits* waits, int lane) {
  if (!bar_wait(bars + 8 * (BAR_DONE + 2 * g + half), pass & 1, waits)) return false;
  tc_fence_after();
  uint32_t v[NW];
  tm_load_pack<NW>(tm, v);
  tm_wait_load<NW>(v);
  // (in registers: the next segment's MMAs run while the maxima are taken)
  tc_fence_before();
  __syncwarp();
  if (lane == 0) bar_arrive(bars + 8 * (BAR_GO + 2 * (g + 2 < NGROUP ? g + 2 : g + 2 - NGROUP) + half));
#pragma unroll
  for (int j = 0; j < NW; j++) m[j] = FIRST ? v[j] : __vmaxs2(m[j], v[j]);
  return true;
}

// The tile's passes for the epilogue warp of one quadrant of windows and one
// half of the rows: the rows whose bound reaches S1, as two masks a window,
// go to the ring.  tm: the half's right-side accumulator; rp: the ring's
// passes written and taken; pass: passes so far.
template <int NW>
__device__ __forceinline__ bool epilogue_tile(const TileInfo& t, uint2* ring, volatile uint32_t* rp, uint32_t bars,
                                              uint32_t tm, int half, int lane_window, uint32_t& pass,
                                              Waits* waits, int lane) {
  constexpr int NMASK = (NW + 15) / 16;  // masks of 32 rows: row 4 j + b of a mask's rows at bit 8 b + j
  const int n_pass = (t.n2 + TC_M - 1) / TC_M;
  const int row0 = half * 2 * NW;
  uint32_t seen = __shfl_sync(0xffffffffu, rp[RP_TAKEN], 0);  // passes taken, as last seen
  uint32_t valid[NMASK];
#pragma unroll
  for (int i = 0; i < NMASK; i++) {
    valid[i] = 0;
    for (int b = 0; b < 32; b++)
      if (4 * (b & 7) + (b >> 3) + 32 * i < 2 * NW && row0 + 32 * i + 4 * (b & 7) + (b >> 3) < t.rows) valid[i] |= 1u << b;
  }
  for (int p = 0; p < n_pass; p++) {
    uint32_t r[NW], l[NW];
    const uint32_t tl = tm + 2 * TM_ACC;
    if (!read_segment<NW, true>(r, 0, bars, half, pass, tm, waits, lane)) return false;
    if (!read_segment<NW, true>(l, 1, bars, half, pass, tl, waits, lane)) return false;
#pragma unroll 1
    for (int g = 2; g < NGROUP; g += 2) {
      if (!read_segment<NW, false>(r, g, bars, half, pass, tm, waits, lane)) return false;
      if (!read_segment<NW, false>(l, g + 1, bars, half, pass, tl, waits, lane)) return false;
    }
    // the sign bits of bound - S1, gathered eight words (16 rows) at a time
    // into bit 7 of the mask's bytes, which move down
    uint32_t cand[2] = {0u, 0u};
    if (p * TC_M + lane_window < t.n2) {
#pragma unroll
      for (int i = 0; i < NMASK; i++) {
        uint32_t neg = 0;
#pragma unroll
        for (int j = 0; j < 8; j++) {
          neg >>= 1;
          const int k = 16 * i + 2 * j;
          if (k < NW)
            neg |= __byte_perm(__vadd2(r[k < NW ? k : 0], l[k < NW ? k : 0]),
                               __vadd2(r[k + 1 < NW ? k + 1 : 0], l[k + 1 < NW ? k + 1 : 0]), 0x7531u) & 0x80808080u;
        }
        cand[i] = ~neg & valid[i];
      }
    }
    // a free place of the ring
    if (pass - seen >= RING) {
      const uint32_t t0 = now();
      while (pass - (seen = __shfl_sync(0xffffffffu, rp[RP_TAKEN], 0)) >= RING) {
        if (over(waits, t0)) return false;
        __nanosleep(100);
      }
    }
    ring[(pass % RING) * 32 + lane] = make_uint2(cand[0], cand[1]);
    __threadfence_block();
    __syncwarp();
    pass++;
    if (lane == 0) rp[0] = pass;
  }
  return true;
}

// ---------------------------------------------------------------------------
// MMA warp
// ---------------------------------------------------------------------------
// One segment of a chain (a side of a half of the rows): N of the side's
// segment before it, or the accumulator's base, then P of its own.  The tensor
// memory addresses are constants (the CTA holds all of it): an operand that
// the compiler does not know to be uniform costs its move at each MMA.
template <int SIDE, int HALF, int SEG>
__device__ __forceinline__ bool mma_segments(uint64_t prof, uint32_t idesc, uint32_t bars, uint32_t pass,
                                             Waits* waits) {
  if constexpr (SEG < NSEG) {
    constexpr int G = 2 * SEG + SIDE;
    constexpr uint32_t d = (2 * SIDE + HALF) * TM_ACC;
    if (!bar_wait(bars + 8 * (BAR_GO + 2 * G + HALF), pass & 1, waits)) return false;
    tc_fence_after();
    if (elect_one()) {
      if constexpr (SEG == 0) {
        tc_mma<0>(d, TM_BASE, prof + (uint64_t)(SLOT_BASE * (SLOT_BYTES >> 4)), idesc, TM_SFB);
      } else {
#pragma unroll
        for (int i = 0; i < seg_steps(SIDE, SEG - 1); i++) {
          const int step = seg_first(SIDE, SEG - 1) + i;
          tc_mma<1>(d, TM_A + 8 * step, prof + (uint64_t)(slot_n(step) * (SLOT_BYTES >> 4)), idesc, TM_SF2);
        }
      }
#pragma unroll
      for (int i = 0; i < seg_steps(SIDE, SEG); i++) {
        const int step = seg_first(SIDE, SEG) + i;
        tc_mma<1>(d, TM_A + 8 * step, prof + (uint64_t)(step * (SLOT_BYTES >> 4)), idesc, TM_SF2);
      }
      tc_commit(bars + 8 * (BAR_DONE + 2 * G + HALF));
    }
    __syncwarp();
    return mma_segments<SIDE, HALF, SEG + 1>(prof, idesc, bars, pass, waits);
  }
  return true;
}

// The tile's passes of a chain.
template <int SIDE, int HALF>
__device__ __forceinline__ void mma_tile(uint64_t prof, uint32_t idesc, uint32_t bars, int n_pass, uint32_t& pass,
                                         Waits* waits) {
  for (int p = 0; p < n_pass; p++, pass++)
    if (!mma_segments<SIDE, HALF, 0>(prof, idesc, bars, pass, waits)) return;
}

// ---------------------------------------------------------------------------
// tiles
// ---------------------------------------------------------------------------
// Fetches tile k of the CTA (the tile warp): the descriptor, the bound's
// constant, the rows; false when there is none.
__device__ __forceinline__ bool fetch_tile(const UngArgs& a, const ScoreTable& c, unsigned char* smem, uint32_t k,
                                           int lane) {
  int i = 0;
  if (lane == 0) i = !a.persistent ? (k == 0 ? (int)blockIdx.x : a.n_tiles) : atomicAdd(a.tile_counter, 1);
  i = __shfl_sync(0xffffffffu, i, 0);
  TileInfo t;
  t.rows = 0;
  t.u0 = t.v0 = 0;
  t.n2 = t.half = 0;
  t.thr4 = 0;
  if (i < a.n_tiles) {
    const int4 tile = a.tiles[a.tile_base + i];
    const int key = tile_key(tile), a0 = key / (2 * 11 * 20), a3 = key % 20;
    t.rows = tile_rows(tile);
    t.half = (t.rows + 31) / 32 * 16;
    t.u0 = (int64_t)(uint32_t)tile.y;
    t.v0 = a.key_off2[key] + tile.z;
    t.n2 = tile.w - tile.z;
    // cells 0 and 3 pair a residue with itself (the subset seed's positions
    // 1 and 4 have one class per residue); the constant (negative: S1 is at
    // least UNG_TC_MIN_S1) is rounded up where four e2m1 values cannot give it
    int rest = c.score[a0 * NCODE + a0] + c.score[a3 * NCODE + a3] - a.s1;
    for (int j = 0; j < 4; j++) {
      const int part = round_up_e2m1(max(rest, -12));
      t.thr4 |= e2m1(part) << (4 * j);
      rest -= part;
    }
    unsigned char* rows = smem + OFF_ROWS + (k % TILE_ROWS) * ROWS_BYTES;
    for (int e = lane; e < 2 * t.half * 3; e += 32) {
      const int r = e / 3, q = e - 3 * r;
      uint4 x = make_uint4(0x15151515u, 0x15151515u, 0x15151515u, 0x15151515u);
      if (r < t.rows) x = __ldg(reinterpret_cast<const uint4*>(a.nb1 + (t.u0 + r) * WIN) + q);
      const uint32_t xs[4] = {x.x, x.y, x.z, x.w};
      uint32_t e2[8];
#pragma unroll
      for (int j = 0; j < 8; j++) e2[j] = row_entries(__byte_perm(xs[j >> 1], 0u, (j & 1) ? 0x4342u : 0x4140u));
      uint4* d = reinterpret_cast<uint4*>(rows + r * ROW_STRIDE + 32 * q);
      d[0] = make_uint4(e2[0], e2[1], e2[2], e2[3]);
      d[1] = make_uint4(e2[4], e2[5], e2[6], e2[7]);
    }
  }
  if (lane == 0) *reinterpret_cast<TileInfo*>(smem + OFF_SLOTS + (k % TILES) * SLOT_INFO) = t;
  __threadfence_block();
  __syncwarp();
  if (lane == 0) *reinterpret_cast<volatile uint32_t*>(smem + OFF_MISC + 4) = k + 1;
  return t.rows > 0;
}

// The profile of a tile's rows (the epilogue warps): a thread takes one row
// and every other K step.
__device__ __forceinline__ void build_profile(unsigned char* smem, const unsigned char* rows, const TileInfo& t,
                                              int tid) {
  static_assert(EPI_WARPS * 32 == 2 * TC_N, "two threads a row");
  const int r = tid % TC_N;
  if (r >= 2 * t.half) return;
  const uint4* lut = reinterpret_cast<const uint4*>(smem + OFF_PLUT);
  const uint16_t* codes = reinterpret_cast<const uint16_t*>(rows + r * ROW_STRIDE);
  for (int step = tid / TC_N; step < KSTEPS; step += 2) {
    int code[3];
#pragma unroll
    for (int c = 0; c < 3; c++) code[c] = cell_of(step, c) < WIN ? (int)row_code(codes[cell_of(step, c)]) : -1;
    const bool has_n = step < 5 || (step >= 8 && step < 12);
    for (int plane = 0; plane < (has_n ? 2 : 1); plane++) {
      uint4 x[3];
#pragma unroll
      for (int c = 0; c < 3; c++) {
        const int pp = step == 0 && c < 2 ? plane + 2 : plane;  // cells 1 and 2: the seed planes
        x[c] = code[c] >= 0 ? lut[pp * NCODE + code[c]] : make_uint4(0u, 0u, 0u, 0u);
      }
      if (step == 0 && plane == 0) x[2].z |= t.thr4 << 16;
      unsigned char* d = smem + OFF_PROF + (plane ? slot_n(step) : step) * SLOT_BYTES + r * 16;
      *reinterpret_cast<uint4*>(d) =
          make_uint4(x[0].x, x[0].y, x[0].z | (x[1].x << 16), __funnelshift_l(x[1].x, x[1].y, 16));
      *reinterpret_cast<uint4*>(d + CHUNK_BYTES) = make_uint4(__funnelshift_l(x[1].y, x[1].z, 16), x[2].x, x[2].y, x[2].z);
    }
  }
}

__global__ void __launch_bounds__(TC_THREADS, 1) k_ungapped_mma(UngArgs a, const __grid_constant__ ScoreTable c,
                                                                const uint32_t wait_limit) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t sb = saddr(smem);
  const uint32_t bars = sb + OFF_BAR;
  Waits* waits = reinterpret_cast<Waits*>(smem + OFF_WAITS);

  // one-time set-up: tables, barriers, tensor memory, block scales
  int8_t* tab = reinterpret_cast<int8_t*>(smem + OFF_TAB);
  for (int i = tid; i < TAB_BYTES; i += TC_THREADS) {
    const int b = i / TAB_B, aa = i % TAB_B / 128 * 4 + (i & 3);
    tab[i] = aa < NCODE ? c.score[aa * NCODE + b] : (int8_t)0;
  }
  for (int i = tid; i < 2 * LUT_CODES * 32 * 4; i += TC_THREADS) {
    const int sh = i / (LUT_CODES * 128), b = i / 128 % LUT_CODES, w = i % 4;
    const int bit = 4 * (b < NAA ? b : WILD) + 1 + 16 * sh - 32 * w;  // e2m1 1.0 = 0b0010
    reinterpret_cast<uint32_t*>(smem + OFF_LUT)[i] = b < NCODE && w < 3 && bit >= 0 && bit < 32 ? 1u << bit : 0u;
  }
  for (int i = tid; i < 4 * NCODE * 4; i += TC_THREADS) {
    // plane 0: P, 1: N = score - P, 2: the seed cells' score rounded up, 3: its correction
    const int plane = i / (NCODE * 4), aa = i / 4 % NCODE, w = i % 4;
    uint32_t x = 0;
    for (int j = 0; j < 8; j++) {
      const int b = 8 * w + j;
      if (b >= NAA) break;
      const int s = bound_score(c.score, aa, b), p = round_up_e2m1(max(s, 0)), g = round_up_e2m1(s);
      x |= e2m1(plane == 0 ? p : plane == 1 ? s - p : plane == 2 ? g : s - g) << (4 * j);
    }
    reinterpret_cast<uint32_t*>(smem + OFF_PLUT)[i] = x;
  }
  if (tid < RP_WORDS) reinterpret_cast<uint32_t*>(smem + OFF_RPOS)[tid] = 0;
  for (int i = tid; i < SLOT_BYTES / 4; i += TC_THREADS)  // 1.5 in each row's first dimension
    reinterpret_cast<uint32_t*>(smem + OFF_PROF + SLOT_BASE * SLOT_BYTES)[i] =
        i < CHUNK_BYTES / 4 && i % 4 == 0 ? 3u : 0u;
  for (int i = tid; i < TC_M; i += TC_THREADS)  // no cell: past the window
    *reinterpret_cast<uint32_t*>(smem + OFF_WIN + (TC_M + i) * WIN_STRIDE + WIN - LEFT_BYTE) = 0x01010101u * NCODE;
  if (tid == 0) {
    waits->abort = 0;
    waits->limit = wait_limit;
    *reinterpret_cast<uint32_t*>(smem + OFF_MISC + 4) = 0;
    for (int g = 0; g < 2 * NGROUP; g++) {
      bar_init(bars + 8 * (BAR_GO + g), EXP_WARPS / 2 + EPI_WARPS / 2);
      bar_init(bars + 8 * (BAR_DONE + g), 1);
    }
    bar_init(bars + 8 * BAR_READ, EPI_WARPS);
    bar_init(bars + 8 * BAR_PROF, EPI_WARPS);
    bar_init(bars + 8 * BAR_DRAIN, 4);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == MMA_WARP) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sb + OFF_MISC), "r"(TM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // (all columns are allocated, so the base is column 0)
  const uint32_t tm_base = *reinterpret_cast<uint32_t*>(smem + OFF_MISC);
  if (tm_base != 0u) {
    *(volatile int*)&waits->abort = 1;
    if (tid == 0) atomicOr(a.err, UNG_ERR_TMEM);
  }
  if (warp < 4) {
    const uint32_t tml = (uint32_t)(warp * 32) << 16;
    const uint32_t s1[8] = {0x7f7f7f7fu, 0x7f7f7f7fu, 0x7f7f7f7fu, 0x7f7f7f7fu,
                            0x7f7f7f7fu, 0x7f7f7f7fu, 0x7f7f7f7fu, 0x7f7f7f7fu};  // UE8M0 2^0
    const uint32_t s2[8] = {0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u,
                            0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u};  // 2^1
    const uint32_t sb23[8] = {0x96969696u, 0x96969696u, 0x96969696u, 0x96969696u,
                              0x96969696u, 0x96969696u, 0x96969696u, 0x96969696u};  // 2^23
    const uint32_t one[8] = {2u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    tm_store8(tml + TM_SF1, s1);
    tm_store8(tml + TM_SF2, s2);
    tm_store8(tml + TM_SFB, sb23);
    tm_store8(tml + TM_BASE, one);
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // (the base's slot)
  tc_fence_before();
  __syncthreads();
  tc_fence_after();

  // every role walks the same tiles
  TileInfo t;
  uint32_t pass = 0;
  if (warp < EPI_WARPS) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(TC_REGS_EPI));
    uint2* ring = reinterpret_cast<uint2*>(smem + OFF_RING) + warp * RING * 32;
    volatile uint32_t* rp = reinterpret_cast<volatile uint32_t*>(smem + OFF_RPOS) + warp;
    const int q = warp & 3, half = warp >> 2;
    // the accumulators are free: the first pass's first segments wait for the expand warps only
    if (lane == 0) {
      bar_arrive(bars + 8 * (BAR_GO + half));
      bar_arrive(bars + 8 * (BAR_GO + 2 + half));
    }
    for (uint32_t k = 0; wait_tile(smem, k, t, waits); k++) {
      __syncwarp();
      if (lane == 0) bar_arrive(bars + 8 * BAR_READ);
      if (!bar_wait(bars + 8 * BAR_READ, k & 1, waits)) break;
      build_profile(smem, smem + OFF_ROWS + (k % TILE_ROWS) * ROWS_BYTES, t, tid);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      if (lane == 0) bar_arrive(bars + 8 * BAR_PROF);
      const uint32_t tml = ((uint32_t)(q * 32) << 16) + half * TM_ACC;
      const int lw = q * 32 + lane;
      bool ok;
      if (t.half == 64) ok = epilogue_tile<32>(t, ring, rp, bars, tml, half, lw, pass, waits, lane);
      else if (t.half == 48) ok = epilogue_tile<24>(t, ring, rp, bars, tml, half, lw, pass, waits, lane);
      else if (t.half == 32) ok = epilogue_tile<16>(t, ring, rp, bars, tml, half, lw, pass, waits, lane);
      else ok = epilogue_tile<8>(t, ring, rp, bars, tml, half, lw, pass, waits, lane);
      if (!ok) break;
    }
  } else if (warp < EXT_WARP) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(TC_REGS_EXP));
    const int q = warp & 3, side = (warp - EXP_WARP) >> 2;  // tensor memory lanes 32 q ..
    const uint32_t tml = ((uint32_t)(q * 32) << 16) + TM_A;
    const uint32_t lut = sb + OFF_LUT + 16 * lane;
    // the right side is bytes 0-25 of a window, the left side 26-47: two 16-byte words each
    uint32_t* win = reinterpret_cast<uint32_t*>(smem + OFF_WIN + (side * TC_M + q * 32 + lane) * WIN_STRIDE);
    const uint32_t win_s = saddr(win) - side * LEFT_BYTE;
    const uint4 sent = make_uint4(0x15151515u, 0x15151515u, 0x15151515u, 0x15151515u);
    for (uint32_t k = 0; wait_tile(smem, k, t, waits); k++) {
      const uint4* src = reinterpret_cast<const uint4*>(a.nb2 + t.v0 * WIN) + side;
      uint4 x = sent, y = sent;
      if (q * 32 + lane < t.n2) {
        x = __ldg(src + (int64_t)(q * 32 + lane) * 3);
        y = __ldg(src + (int64_t)(q * 32 + lane) * 3 + 1);
      }
      const int n_pass = (t.n2 + TC_M - 1) / TC_M;
      bool ok = true;
      for (int p = 0; p < n_pass && ok; p++, pass++) {
        win[0] = x.x;
        win[1] = x.y;
        win[2] = x.z;
        win[3] = x.w;
        win[4] = y.x;
        win[5] = y.y;
        win[6] = y.z;
        win[7] = y.w;
        const int w = (p + 1) * TC_M + q * 32 + lane;
        x = y = sent;
        if (w < t.n2) {
          x = __ldg(src + (int64_t)w * 3);
          y = __ldg(src + (int64_t)w * 3 + 1);
        }
        ok = expand_pass(side, win_s, lut, tml, bars, pass, waits, lane);
      }
      if (!ok) break;
    }
  } else if (warp < MMA_WARP) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(TC_REGS_EXT));
    const int x = warp - EXT_WARP;  // the epilogue warp whose candidates it takes
    ExtState e;
    e.queue = reinterpret_cast<uint64_t*>(smem + OFF_QUEUE) + x * QCAP;
    e.n = 0;
    e.hits.key = reinterpret_cast<uint64_t*>(smem + OFF_HKEY) + x * HBUF;
    e.hits.val = reinterpret_cast<uint32_t*>(smem + OFF_HVAL) + x * HBUF;
    e.hits.n = 0;
    const uint2* ring = reinterpret_cast<const uint2*>(smem + OFF_RING) + x * RING * 32;
    volatile uint32_t* rp = reinterpret_cast<volatile uint32_t*>(smem + OFF_RPOS) + x;
    volatile uint32_t* ended = reinterpret_cast<volatile uint32_t*>(smem + OFF_RPOS) + RP_EXT;
    for (uint32_t k = 0; wait_tile(smem, k, t, waits); k++) {
      if (!extend_tile(e, t, a, smem + OFF_ROWS + (k % TILE_ROWS) * ROWS_BYTES, reinterpret_cast<const int8_t*>(smem + OFF_TAB),
                       ring, rp, (x >> 2) * t.half, (x & 3) * 32, pass, waits, lane))
        break;
      __syncwarp();
      if (lane == 0) ended[x] = k + 1;
    }
    if (e.hits.n > 0) flush_hits(e.hits, a, lane);
  } else if (warp < TILE_WARP) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(TC_REGS_MMA));
    const uint64_t prof = tc_desc(sb + OFF_PROF);
    for (uint32_t k = 0; wait_tile(smem, k, t, waits); k++) {
      if (!bar_wait(bars + 8 * BAR_PROF, k & 1, waits)) break;
      tc_fence_after();
      const uint32_t n = __shfl_sync(0xffffffffu, (uint32_t)t.half, 0);
      const uint32_t idesc = (1u << 7) | (1u << 10) | ((n >> 3) << 17) | (1u << 23) | (8u << 24);
      const int n_pass = (t.n2 + TC_M - 1) / TC_M;
      if (warp == MMA_WARP) mma_tile<0, 0>(prof, idesc, bars, n_pass, pass, waits);
      else if (warp == MMA_WARP + 1) mma_tile<1, 0>(prof, idesc, bars, n_pass, pass, waits);
      else if (warp == MMA_WARP + 2) mma_tile<0, 1>(prof + n, idesc, bars, n_pass, pass, waits);
      else mma_tile<1, 1>(prof + n, idesc, bars, n_pass, pass, waits);
    }
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(TC_REGS_MMA));
    if (warp == TILE_WARP) {
      // ahead of the others, once every extend warp has ended the tile that
      // used the row buffer last (a tile can take long: the limit counts from
      // the last pass that an extend warp took)
      volatile uint32_t* taken = reinterpret_cast<volatile uint32_t*>(smem + OFF_RPOS) + RP_TAKEN + lane % EXT_WARPS;
      volatile uint32_t* ended = reinterpret_cast<volatile uint32_t*>(smem + OFF_RPOS) + RP_EXT + lane % EXT_WARPS;
      for (uint32_t k = 0;; k++) {
        bool ok = true;
        uint32_t t0 = now(), last = *taken;
        for (uint32_t polls = 1; ok && __any_sync(0xffffffffu, *ended + TILE_ROWS <= k); polls++) {
          if (polls % 64 == 0) {  // (at every poll the longer loop cost the other roles 1 %)
            const uint32_t at = *taken;
            if (__any_sync(0xffffffffu, at != last)) t0 = now();
            last = at;
            ok = !over(waits, t0);
          }
          __nanosleep(400);
        }
        if (!ok || !fetch_tile(a, c, smem, k, lane)) break;
      }
    }
  }
  __syncwarp();
  if (warp >= MMA_WARP && warp < TILE_WARP) {
    // the MMAs in flight (there are some only when a wait ran out) end before
    // shared and tensor memory go
    if (elect_one()) tc_commit(bars + 8 * BAR_DRAIN);
    __syncwarp();
    const uint32_t t0 = now();
    while (!bar_try(bars + 8 * BAR_DRAIN, 0) && now() - t0 < UNG_WAIT_CLOCKS) {
    }
  }
  tc_fence_before();
  __syncthreads();
  if (tid == 0 && *(volatile int*)&waits->abort) atomicOr(a.err, UNG_ERR_WAIT);
  if (warp == MMA_WARP)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm_base), "r"(TM_COLS));
}

}  // namespace

static std::atomic<uint32_t> g_wait_limit{UNG_WAIT_CLOCKS};
void set_ungapped_wait_limit(int64_t clocks) {
  g_wait_limit.store(clocks > 0 && clocks < UNG_WAIT_CLOCKS ? (uint32_t)clocks : UNG_WAIT_CLOCKS);
}

cudaError_t launch_ungapped_mma(const UngArgs& a, int grid, cudaStream_t st) {
  static std::atomic<bool> attr_set[64];  // per device; calls may come from several threads
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 64 && !attr_set[dev]) {
    cudaError_t e = cudaFuncSetAttribute(k_ungapped_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
    if (e != cudaSuccess) return e;
    attr_set[dev] = true;
  }
  if (grid <= 0) return cudaSuccess;
  static const ScoreTable table = [] {
    Tables t;
    build_tables(&t);
    ScoreTable s;
    for (int i = 0; i < NCODE * NCODE; i++) s.score[i] = t.score[i];
    return s;
  }();
  note_launch();
  k_ungapped_mma<<<grid, TC_THREADS, TC_SMEM, st>>>(a, table, g_wait_limit.load());
  return cudaGetLastError();
}

}  // namespace plast
