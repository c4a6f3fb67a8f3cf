// Split-precision (emulated FP64) GEMMs on the tcgen05 tensor cores.
//
// An FP64 operand is scaled per row (A) or per column (B) by a power of two 2^e with
// max|x| < 2^e, rounded to 47 fractional bits and cut into NDIG = 6 balanced base-256 digits,
//     x = 2^e * 2^-7 * sum_s d_s 2^-8s ,   |d_s| <= 128,
// each stored exactly as a BF16 "digit plane" value d_s * 2^-8s.  The product keeps the digit pairs
// with s + t <= 5 (21 of 36):
//   * groups q = s + t = 0..3 are accumulated EXACTLY: every partial sum is an integer multiple
//     of 2^-8q of magnitude at most 2^24 * 2^-8q when a group is flushed every 256 values of k,
//     so the FP32 tensor-core accumulator loses nothing; each flush is added, as an integer, into
//     an int64 fixed-point accumulator;
//   * groups q = 4, 5 (weights 2^-32 and 2^-40) each have one FP32 accumulator over the whole
//     K range of a tile.  (The tensor core's FP32 accumulation of products of very different
//     weights is measurably less accurate than IEEE rounding, which is why weight 2^-24 is kept
//     in the exact part and every accumulator holds one weight only.)
// The recombination uses integer arithmetic only (FP64 arithmetic is slow on this part): the
// fixed-point sum and the two rounded FP32 tails are merged into one int64 and turned into an
// FP64 value by building its bit pattern.  The chosen digit count and pair set follow the split-product
// ("Ozaki") scheme for emulating a higher precision with low-precision products.
#include <cuda.h>
#include <cuda_bf16.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "digit_planes.h"
#include "las_split.cuh"
#include "sm100_ptx.cuh"

namespace lasdf_split {

constexpr int NEXACT = 4;        // exact weight groups q = 0..3
constexpr int NGROUP = 6;        // weight groups q = s + t = 0..5 kept (21 digit pairs)

constexpr int CHUNK = 16;        // stages per exact chunk (256 values of k)
constexpr int A_PLANE = BM * BK * 2;                 // 4096 B
constexpr int A_BYTES = NDIG * A_PLANE;              // 24576
constexpr int TMEM_COLS = 512;
constexpr int HEAD = 4;          // stages of a chunk's first turn (issue_turns)
constexpr int EPI_WARPS = 16;    // epilogue warps: 4 column groups x 4 TMEM lane quarters
constexpr int EPI_WARP0 = 3;     // warp 0 TMA, warps 1 and 2 MMA, then the epilogue warps
constexpr int NTHREADS = 32 * (EPI_WARP0 + EPI_WARPS);

// Tile width bn (columns of the output per CTA tile, a product's parameter: 48, 64, 80 or 96) and the
// stage layout, sized for the widest tile BN.  The exact weight groups q = 0..3 each own one
// FP32 accumulator of bn TMEM columns, at column q*bn, and the tail groups 4 and 5 share one
// more, at the fixed column TAIL_COL = 4*BN whatever the tile width, so that consecutive tiles
// of different widths in one launch never put one tile's tail where the previous tile's exact
// accumulators are still being drained (every accumulator starts at a multiple of 16).  The
// six B digit planes of a stage lie back to back in shared memory (plane t at t*bn rows), so
// that one MMA of A_s against planes t0..t1 of B (N = (t1-t0+1)*bn <= 256) lands every product
// A_s B_t in the accumulator of its own exact group s + t: the ten exact products of a
// stage take six MMAs at bn = 96 (four of N = 192) and four at bn = 64 (N = 256, 192, 128, 64).
// (Tiles with a second tail accumulator, so that the tail products could be merged the same way,
// measured slower: a shorter stage carries the same waits for data and for the exact drains.)
template <int BN_>
struct OzTile {
  static constexpr int BN = BN_;   // the widest tile the stage layout holds
  static_assert(BN % 32 == 0 && (NEXACT + 1) * BN <= TMEM_COLS, "tile width");
  static constexpr int B_PLANE = BN * BK * 2;    // bytes per B plane at the widest tile
  static constexpr int TAIL_COL = NEXACT * BN;   // TMEM column of the tail accumulator
  static constexpr int B_BYTES = NDIG * B_PLANE;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int NSTAGE = (220 * 1024) / STAGE_BYTES < 6 ? (220 * 1024) / STAGE_BYTES : 6;
  static constexpr int SMEM_BYTES = NSTAGE * STAGE_BYTES + 1024 + 256;
  static_assert(STAGE_BYTES % 1024 == 0, "stages stay 1024-byte aligned");
};

struct OzParams {
  int M, N;                // output rows / columns
  int a_rpad, b_rpad;      // padded rows of the A / B plane layouts
  int a_row0, b_row0;      // first row of A / B used: multiples of ROWGRAN (box coordinates)
  int row_skip;            // rows between a_row0 and the product's first row (computed, not stored)
  int kb_total;            // K blocks of BK
  int kb_per_split;
  int ksplit;
  const int* ea;           // row exponents [M] (nullptr: 0)
  const int* eb;           // column exponents [N]
  double* out;
  int mode;                // 0: out[z*zstride + r*ldc + c]; 1: Ht layout out[z*zstride +
                           // (L*ht_op + c)*ht_n + mu] (rows (L,mu))
  int vec;                 // mode 0: rows of out are 32-byte aligned at multiples of 4 columns
  long ldc, zstride;
  int ht_n, ht_op;
  int lower;               // symmetric product: only tiles that touch the lower triangle
  long tiles_z;            // tiles per K split (the lower-triangle ones only when lower != 0)
  int sh;                  // fractional bits kept when merging the tail
  int bn;                  // tile width: 48, 64, 80 or 96 columns
  int a_mn;                // A read MN-major: rows of the stored planes are K, their K is M
  // A = the Cholesky vectors in packed-triangle digit form (a_pack != 0; see BPacked): the
  // product's row tiles are the full 128-row blocks R of each b^L (tile m = L * pk_nb1 + R of the
  // chunk), and each 16-wide K block is read from the stored lower tile (R, J) as is (J <= R),
  // from the stored tile (J, R) MN-major (R < J < pk_nb1), or from the ragged rows nu >= n1 of
  // b^L MN-major (tensor maps tmA, tmA2 and tmA3)
  int a_pack;
  int pk_nb1, pk_T, pk_rp; // full row blocks per L, stored tiles per L, stored ragged rows per L
  int pk_L0;               // first auxiliary index of the chunk
  int ht_rows, ht_mu0;     // mode 1: rows of the product per L, and mu of its first row
  int ht_live;             // mode 1: rows per L that are stored (the others are padding)
  int ea_perL;             // the row exponents are per auxiliary index: ea[L], not ea[row]
  int* status;
};

// W * 2^E (|W| < 2^63) rounded once to FP64 (round to nearest even), built from the integer: the
// leading one moved to bit 62, half a unit of bit 10 added (ties to even), the exponent field
// put in front.  Results outside the normal range (rare) go through ldexp.
// The 64-bit conversions run on the FP64 path of this part, a few per clock and SM: with
// __ll2double_rn here and __float2ll_rn in the tail, a 128 x 96 tile's conversions took about
// 12000 clocks, half of them before the next tile could start.
__device__ __forceinline__ double make_double(long long W, int E) {
  const unsigned long long a = (unsigned long long)(W < 0 ? -W : W);
  const int n = __clzll((long long)a);            // 1..63 for a != 0
  unsigned long long m = a << (n - 1);
  m += 511 + ((m >> 10) & 1);
  const int ex = 1086 - n + E;                    // biased exponent: 63 - n + E + 1023
  if (a == 0) return 0.0;
  if (ex <= 0 || ex >= 2046) return ldexp(__ll2double_rn(W), E);
  const unsigned long long b = ((unsigned long long)(ex - 1) << 52) + (m >> 10);
  return __longlong_as_double((long long)(b | ((unsigned long long)W & (1ull << 63))));
}

// rint(f) as int64 for |f| < 2^46, without a 64-bit conversion: the part above 2^16 first, then
// the exact rest (the first part is even, so ties round as in one step).
__device__ __forceinline__ long long rint_ll(float f) {
  const int hi = __float2int_rn(f * 0x1p-16f);
  const int lo = __float2int_rn(fmaf((float)hi, -65536.0f, f));
  return (long long)hi * 65536 + lo;
}

// Column tiles of row tile i that touch the lower triangle (column tile j with j*bn < (i+1)*BM).
__host__ __device__ __forceinline__ int lower_tiles_in_row(int i, int ntn, int bn) {
  const int c = ((i + 1) * BM + bn - 1) / bn;
  return c < ntn ? c : ntn;
}

__device__ __forceinline__ void tile_coords(const OzParams& p, long t, int& m0, int& n0,
                                            int& kb0, int& nkb) {
  const int bn = p.bn;
  const int ntn = (p.N + bn - 1) / bn;
  const int z = (int)(t / p.tiles_z);
  long rem = t - (long)z * p.tiles_z;
  // the column tiles of one row tile are adjacent in tile order so that concurrently running
  // CTAs share that row tile's digit planes through L2
  if (!p.lower) {
    m0 = (int)(rem / ntn) * BM;
    n0 = (int)(rem % ntn) * bn;
  } else {
    // only the tiles that touch the lower triangle are enumerated, so that the persistent CTAs
    // share out the work evenly
    int i = 0;
    for (int c = lower_tiles_in_row(0, ntn, bn); rem >= c; c = lower_tiles_in_row(++i, ntn, bn))
      rem -= c;
    m0 = i * BM;
    n0 = (int)rem * bn;
  }
  kb0 = z * p.kb_per_split;
  nkb = min(p.kb_total, kb0 + p.kb_per_split) - kb0;
}

// One product of a grouped launch: its tensor maps, parameters and first tile in the launch's
// tile order (problems are concatenated; tile0 of problem g+1 = tile0 + tiles of problem g).
struct OzProblem {   // aligned as its tensor maps
  CUtensorMap tmA, tmB, tmA2, tmA3;   // tmA2, tmA3: packed-triangle A only
  OzParams p;
  long tile0;
};

// The tile a role works on: its product (parameters and maps) and coordinates.  A role's tiles
// only ever increase, so the product index moves forward only.
template <bool GROUPED>
struct OzCursor {
  int g = 0;
  const OzParams* P = nullptr;
  const CUtensorMap* ma = nullptr;
  const CUtensorMap* mb = nullptr;
  const CUtensorMap* ma2 = nullptr;
  const CUtensorMap* ma3 = nullptr;
  int m0 = 0, n0 = 0, kb0 = 0, nkb = 0;
  __device__ __forceinline__ bool seek(long t, const OzParams& p1, const CUtensorMap* a1,
                                       const CUtensorMap* b1, const CUtensorMap* a2,
                                       const CUtensorMap* a3, const OzProblem* probs,
                                       int nprob) {
    long tl = t;
    bool moved = P == nullptr;
    if constexpr (GROUPED) {
      while (g + 1 < nprob && probs[g + 1].tile0 <= t) {
        ++g;
        moved = true;
      }
      P = &probs[g].p;
      ma = &probs[g].tmA;
      mb = &probs[g].tmB;
      ma2 = &probs[g].tmA2;
      ma3 = &probs[g].tmA3;
      tl = t - probs[g].tile0;
    } else {
      P = &p1;
      ma = a1;
      mb = b1;
      ma2 = a2;
      ma3 = a3;
    }
    tile_coords(*P, tl, m0, n0, kb0, nkb);
    return moved;
  }
};

// Descriptor of plane `plane` of an operand whose planes lie `bytes` apart: formed for each MMA, or
// (BASE) as the first plane's plus an offset, which is faster where addresses stay in uniform
// registers (issue_in_turn; 800-orbital autograd 11.2 -> 11.0 ms).
template <bool BASE>
__device__ __forceinline__ uint64_t plane_desc(uint32_t addr, int plane, int bytes, bool mn) {
  if constexpr (BASE)
    return (mn ? sm100::smem_desc_sw32_mn(addr) : sm100::smem_desc_sw32(addr)) +
           (uint64_t)(plane * (bytes >> 4));
  else
    return mn ? sm100::smem_desc_sw32_mn(addr + plane * bytes)
              : sm100::smem_desc_sw32(addr + plane * bytes);
}

// One stage's products, A plane by A plane.  EXACT: groups 0..3, A_s against planes 0 .. 3-s of B as
// few MMAs of balanced width (N = np * BNV <= 256) that land in the accumulators of groups s .. 3;
// s = 0 spans all four and starts them when start_exact.  TAIL: groups 4 and 5 (eleven MMAs into the
// tail accumulator), started when start_tail.  KEEP: the MMAs of one A plane, which follow one
// another, read it from shared memory once, the first keeping it in the collector buffer; only
// where no other thread's MMAs come between them.  amn: the stage holds the transposed access of
// planes stored with rows along K (A MN-major).  Everything is a compile-time constant once
// inlined: the issuing thread must not spend its time on address arithmetic.
template <int BNV, bool EXACT, bool TAIL, bool KEEP>
__device__ __forceinline__ void mma_stage(uint32_t tmem, uint32_t tmem_tail, uint32_t sa,
                                          uint32_t sb, bool start_exact, bool start_tail, bool amn) {
  constexpr int maxp = 256 / BNV;
  const uint32_t ia = amn ? sm100::IDESC_A_MN : 0u;
#pragma unroll
  for (int s = 0; s < NDIG; ++s) {
    const int nt = EXACT && s < NEXACT ? NEXACT - s : 0, nm = (nt + maxp - 1) / maxp;
    const int t_tail = s < NEXACT ? NEXACT - s : 0;
    const int all = nm + (TAIL ? NGROUP - s - t_tail : 0);
    int t = 0;
#pragma unroll
    for (int m = 0; m < all; ++m) {
      const uint64_t a = plane_desc<KEEP>(sa, s, A_PLANE, amn);
      uint32_t d, id, acc;
      uint64_t b;
      if (m < nm) {
        const int np = (nt - t) / (nm - m);
        d = tmem + (uint32_t)((s + t) * BNV);
        b = plane_desc<KEEP>(sb, t, BNV * BK * 2, false);
        id = sm100::idesc_bf16(BM, np * BNV) | ia;
        acc = s > 0 || !start_exact ? 1u : 0u;
        t += np;
      } else {
        d = tmem_tail;
        b = plane_desc<KEEP>(sb, t_tail + m - nm, BNV * BK * 2, false);
        id = sm100::idesc_bf16(BM, BNV) | ia;
        acc = s > 0 || m > nm || !start_tail ? 1u : 0u;
      }
      if (!KEEP || all == 1) sm100::mma_bf16(d, a, b, id, acc);
      else if (m == 0) sm100::mma_bf16<sm100::FILL>(d, a, b, id, acc);
      else if (m < all - 1) sm100::mma_bf16<sm100::USE>(d, a, b, id, acc);
      else sm100::mma_bf16<sm100::LAST_USE>(d, a, b, id, acc);
    }
  }
}

// How a launch's two issuers share the work.  In turn: each issues all 21 products of every other
// stage, as a converged warp that elects the issuing thread (its addresses stay in uniform registers:
// an MMA in 48 clocks instead of 56), so that an A plane is read from shared memory once for its
// two to four MMAs.  By group: one issues the exact products, the other the tail's, each as a single
// thread.  In turn a stage at 64
// columns takes about 990 clocks, by group 1130 to 1170 (800-orbital autograd 12.2 -> 11.0 ms, JK 7.2 ->
// 6.7 ms; with the MMAs and copies alone 750 and 950).  At 96 and 80 columns the exact drains (4900 clocks each) set the pace and
// in turn they leave fewer products to run meanwhile (1200-orbital half 23.7 ms by group, 24.0 in
// turn; 400 orbitals 1.39 and 1.44); grouped launches hold several widths' code and spill (batch of 8:
// 3.6 and 4.7 ms).
__host__ __device__ constexpr bool issue_in_turn(bool grouped, int fixbn) {
  return !grouped && (fixbn == 64 || fixbn == 48);
}

// f(tile width as a compile-time constant): the launch's fixed width, or the one of this tile.
template <int FIXBN, class F>
__device__ __forceinline__ bool with_width(int bn, F f) {
  if constexpr (FIXBN != 0) {
    return f(std::integral_constant<int, FIXBN>());
  } else {
    if (bn == 48) return f(std::integral_constant<int, 48>());
    if (bn == 64) return f(std::integral_constant<int, 64>());
    if (bn == 80) return f(std::integral_constant<int, 80>());
    return f(std::integral_constant<int, 96>());
  }
}

// Persistent CTAs (one per SM) walk the tiles (row tile, column tile, K split).  Roles:
// warp 0 streams digit-plane stages with TMA, warps 1 and 2 issue the tcgen05.mma (by group, or a
// stage each in turn: issue_in_turn), warps 3.. drain the TMEM accumulators.  Stage, chunk and tile
// counters run on across tiles so that the loads of the next tile overlap the last MMAs of the current
// one, and its MMAs overlap the current tile's conversion and stores.
// Two issuers, because one thread issues an MMA in 56 clocks at best (descriptors and all; 65 in
// this loop), so a single issuer's 17 MMAs took as long at 64 columns as at 96: the issue, not the
// tensor pipe, set the stage time.
// By group, the issuers write disjoint accumulators and each waits only for what it overwrites: the
// exact issuer for the drain of the previous chunk, the tail issuer for the read-out of the previous
// tile's tail, so that tail products of up to NSTAGE stages run during a drain.  Shared memory is
// the bound: the MMAs' reads of A and B and the stage's own bytes are 173 KB at 96 columns, 1352
// clocks at 128 bytes a clock.
// In turn, both write all accumulators, one after the other: a turn is handed on through an
// mbarrier between tcgen05 fences.  A chunk's first turn takes up to HEAD stages, whose tail
// products run while the last chunk is drained; the others take one.  accf counts one commit by the
// issuer of each of the chunk's last two turns (both by the first when there is only one), since a
// commit covers the MMAs of its own thread; the earlier of the two comes before its turn is handed
// on, so that no arrival of the next chunk can precede it.
// GROUPED: the launch walks the concatenated tiles of nprob products described in global
// memory (probs); otherwise the one product of the kernel parameters.  FIXBN: the tile width of
// every product of the launch as a compile-time constant, or 0 when a grouped launch holds other
// widths than 64 or 96 alone (each tile then reads its product's width).  PACK: the launch
// may hold products whose A is the packed-triangle form of the Cholesky vectors (a_pack); the
// other instantiations leave that logic out of the issuing and loading threads entirely.  AMN:
// the A orientation of the launch's products as a compile-time constant (0: K-major, 1:
// MN-major), or 2 when each tile reads its product's; the issuing thread runs measurably faster
// with a constant.
template <int BN, bool GROUPED, int FIXBN, bool PACK, int AMN = 2>
__global__ void __launch_bounds__(NTHREADS, 1)
k_ozaki(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
        const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmA3,
        const __grid_constant__ OzParams p1, const OzProblem* __restrict__ probs, int nprob,
        long ntiles) {
  using T = OzTile<BN>;
  constexpr int NSTAGE = T::NSTAGE;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = (uint64_t*)(smem + NSTAGE * T::STAGE_BYTES);
  uint64_t* full = bars;              // [NSTAGE]
  uint64_t* empty = bars + NSTAGE;    // [NSTAGE]
  uint64_t* accf = bars + 2 * NSTAGE;
  uint64_t* acce = bars + 2 * NSTAGE + 1;
  uint64_t* drain = bars + 2 * NSTAGE + 2;  // [2] teardown of the two issuers
  uint64_t* accT = bars + 2 * NSTAGE + 4;   // tail accumulator read out (once per tile)
  uint64_t* tailf = bars + 2 * NSTAGE + 5;  // by group: tail accumulator complete (once per tile)
  uint64_t* turn = bars + 2 * NSTAGE + 6;   // [2] in turn: the issuer's go
  uint32_t* tmem_slot = (uint32_t*)(bars + 2 * NSTAGE + 8);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);

  pdl_trigger();
  constexpr bool IN_TURN = issue_in_turn(GROUPED, FIXBN);
  const int warp = IN_TURN ? __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0)
                           : (int)threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  // status word for waits outside any tile (the first product's)
  int* const status0 = GROUPED ? probs[0].p.status : p1.status;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NSTAGE; ++s) {
      sm100::mbar_init(&full[s], 1);
      sm100::mbar_init(&empty[s], IN_TURN ? 1 : 2);
    }
    sm100::mbar_init(accf, IN_TURN ? 2 : 1);
    sm100::mbar_init(acce, EPI_WARPS);
    sm100::mbar_init(accT, EPI_WARPS);
    for (int w = 0; w < 2; ++w) {
      sm100::mbar_init(&drain[w], 1);
      sm100::mbar_init(&turn[w], 1);
    }
    sm100::mbar_init(tailf, 1);
    *abort_flag = 0;
    sm100::fence_mbar_init();
    if (!GROUPED) {
      sm100::tma_prefetch_desc(&tmA);
      sm100::tma_prefetch_desc(&tmB);
      if (PACK && p1.a_pack) {
        sm100::tma_prefetch_desc(&tmA2);
        sm100::tma_prefetch_desc(&tmA3);
      }
    }
  }
  if (warp == 1) {
    sm100::tmem_alloc(tmem_slot, TMEM_COLS);
    sm100::tmem_relinquish();
  }
  sm100::tc_fence_before();
  __syncthreads();
  sm100::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();   // nothing before this reads what an earlier launch wrote

  // ---------------- MMA issuers by group: exact (warp 1) or tail (warp 2) ----------------
  [[maybe_unused]] auto issue_group = [&](auto exact_c) {
    constexpr bool exact = decltype(exact_c)::value;
    auto wait = [&](uint64_t* bar, uint32_t parity, int* status) -> bool {
      return sm100::mbar_wait(bar, parity, abort_flag, status, LAS_ERR_TIMEOUT);
    };
    int st = 0;
    uint32_t phase = 0;
    uint32_t nstart = 0;   // accumulations started so far (exact: chunks; tail: tiles)
    bool ok = true;
    OzCursor<GROUPED> cur;
    for (long t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
      cur.seek(t, p1, &tmA, &tmB, &tmA2, &tmA3, probs, nprob);
      const OzParams& p = *cur.P;
      const int nkb = cur.nkb;
      [[maybe_unused]] const bool amn_tile = p.a_mn != 0;
      // packed-triangle A: K blocks of column blocks J > R (above the diagonal) are read MN-major
      const bool pack = PACK && p.a_pack != 0;
      [[maybe_unused]] const int kb_mn = pack ? 8 * ((cur.m0 / BM) % p.pk_nb1 + 1) : 0;
      // Stages [i0, i1) of the tile with one A orientation (a compile-time constant where the
      // launch fixes it) and one width; false when a wait ran out.
      auto stages_of = [&](auto bn_c, auto amn, int i0, int i1) -> bool {
        constexpr int bn = decltype(bn_c)::value;
        for (int i = i0; i < i1; ++i) {
          if (!wait(&full[st], phase, p.status)) return false;
          const bool first = exact ? (i % CHUNK) == 0 : i == 0;
          if (first) {   // the accumulators this stage starts must have been read out
            if (nstart > 0 && !wait(exact ? acce : accT, (nstart - 1) & 1, p.status)) return false;
            ++nstart;
          }
          sm100::tc_fence_after();
          const uint32_t sa = sm100::smem_u32(smem + st * T::STAGE_BYTES);
          mma_stage<bn, exact, !exact, false>(tmem, tmem + T::TAIL_COL, sa, sa + A_BYTES, first,
                                              first, amn);
          sm100::mma_commit(&empty[st]);
          if (exact && ((i % CHUNK) == CHUNK - 1 || i == nkb - 1)) sm100::mma_commit(accf);
          if (++st == NSTAGE) {
            st = 0;
            phase ^= 1;
          }
        }
        return true;
      };
      auto stages = [&](auto amn, int i0, int i1) -> bool {
        return with_width<FIXBN>(p.bn, [&](auto bn_c) { return stages_of(bn_c, amn, i0, i1); });
      };
      using K_MAJOR = std::integral_constant<bool, false>;
      using MN_MAJOR = std::integral_constant<bool, true>;
      if constexpr (PACK) {
        // packed-triangle A: the K-major stages (up to the diagonal block), then the MN-major ones
        const int isplit = pack ? min(nkb, max(0, kb_mn - cur.kb0)) : amn_tile ? 0 : nkb;
        ok = stages(K_MAJOR(), 0, isplit) && stages(MN_MAJOR(), isplit, nkb);
      } else if constexpr (AMN == 2) {
        ok = stages(amn_tile, 0, nkb);
      } else {
        ok = stages(std::integral_constant<bool, AMN == 1>(), 0, nkb);
      }
      if (ok && !exact) sm100::mma_commit(tailf);
    }
    // make sure no MMA is still writing TMEM when the CTA tears down
    sm100::mma_commit(&drain[exact]);
    sm100::mbar_wait(&drain[exact], 0, abort_flag, status0, LAS_ERR_TIMEOUT);
  };

  // ---------------- MMA issuers in turn (warps 1 and 2) ----------------
  [[maybe_unused]] auto issue_turns = [&](const int who) {
    auto wait = [&](uint64_t* bar, uint32_t parity, int* status) -> bool {
      return __all_sync(0xffffffffu,
                        sm100::mbar_wait(bar, parity, abort_flag, status, LAS_ERR_TIMEOUT));
    };
    int st = 0;
    uint32_t phase = 0;
    uint32_t turns = 0, chunks = 0, tiles = 0;   // turns, exact chunks and tiles so far
    bool ok = true;
    OzCursor<GROUPED> cur;
    for (long t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
      cur.seek(t, p1, &tmA, &tmB, &tmA2, &tmA3, probs, nprob);
      const OzParams& p = *cur.P;
      const int nkb = cur.nkb;
      [[maybe_unused]] const bool amn_tile = p.a_mn != 0;
      // packed-triangle A: K blocks of column blocks J > R (above the diagonal) are read MN-major
      const bool pack = PACK && p.a_pack != 0;
      [[maybe_unused]] const int kb_mn = pack ? 8 * ((cur.m0 / BM) % p.pk_nb1 + 1) : 0;
      // Stages [i0, i1) of the tile with one A orientation (a compile-time constant where the
      // launch fixes it) and one width; false when a wait ran out.
      auto stages_of = [&](auto bn_c, auto amn, int i0, int i1) -> bool {
        constexpr int bn = decltype(bn_c)::value;
        const uint32_t tail = tmem + T::TAIL_COL, ring = sm100::smem_u32(smem);
        auto my_turn = [&]() -> bool {
          return turns == 0 || wait(&turn[who], ((turns - 1) >> 1) & 1, p.status);
        };
        // after the last MMA of a turn that ends at stage e: the other issuer's go, the chunk's
        // commits before it (one by each issuer of the chunk's last two turns)
        auto pass_turn = [&](int i, int e) {
          const int ce = min(nkb, (i & ~(CHUNK - 1)) + CHUNK);
          if (e + 1 >= ce) {
            sm100::mma_commit(accf);
            if (e == ce && (i & (CHUNK - 1)) == 0) sm100::mma_commit(accf);
          }
          sm100::tc_fence_before();
          sm100::mbar_arrive(&turn[who ^ 1]);
        };
#pragma unroll 1
        for (int i = i0; i < i1; ++turns) {
          const bool head = (i & (CHUNK - 1)) == 0;
          const int len = head ? min(HEAD, i1 - i) : 1;
          const bool mine = (turns & 1) == (uint32_t)who;
          if (mine && head) {
            // A chunk's first stages: tail products while the last chunk is drained, then the exact
            // products (which start the accumulators)
            int slot = st;
            uint32_t ph = phase;
#pragma unroll 1
            for (int j = 0; j < len; ++j) {
              if (!wait(&full[slot], ph, p.status) || (j == 0 && !my_turn()) ||
                  (i + j == 0 && tiles > 0 && !wait(accT, (tiles - 1) & 1, p.status)))
                return false;
              sm100::tc_fence_after();
              const uint32_t sa = ring + slot * T::STAGE_BYTES;
              if (sm100::elect_one())
                mma_stage<bn, false, true, true>(tmem, tail, sa, sa + A_BYTES, false, i + j == 0, amn);
              __syncwarp();
              if (++slot == NSTAGE) {
                slot = 0;
                ph ^= 1;
              }
            }
            if (chunks > 0 && !wait(acce, (chunks - 1) & 1, p.status)) return false;
            sm100::tc_fence_after();
            slot = st;
#pragma unroll 1
            for (int j = 0; j < len; ++j) {
              const uint32_t sa = ring + slot * T::STAGE_BYTES;
              if (sm100::elect_one()) {
                mma_stage<bn, true, false, true>(tmem, tail, sa, sa + A_BYTES, j == 0, false, amn);
                sm100::mma_commit(&empty[slot]);
                if (j == len - 1) pass_turn(i, i + len);
              }
              __syncwarp();
              if (++slot == NSTAGE) slot = 0;
            }
          } else if (mine) {
            if (!wait(&full[st], phase, p.status) || !my_turn()) return false;
            sm100::tc_fence_after();
            const uint32_t sa = ring + st * T::STAGE_BYTES;
            if (sm100::elect_one()) {
              mma_stage<bn, true, true, true>(tmem, tail, sa, sa + A_BYTES, false, false, amn);
              pass_turn(i, i + 1);
              sm100::mma_commit(&empty[st]);
            }
            __syncwarp();
          }
          if (head) ++chunks;
          i += len;
          st += len;
          if (st >= NSTAGE) {
            st -= NSTAGE;
            phase ^= 1;
          }
        }
        return true;
      };
      auto stages = [&](auto amn, int i0, int i1) -> bool {
        return with_width<FIXBN>(p.bn, [&](auto bn_c) { return stages_of(bn_c, amn, i0, i1); });
      };
      using K_MAJOR = std::integral_constant<bool, false>;
      using MN_MAJOR = std::integral_constant<bool, true>;
      if constexpr (PACK) {
        // packed-triangle A: the K-major stages (up to the diagonal block), then the MN-major ones
        const int isplit = pack ? min(nkb, max(0, kb_mn - cur.kb0)) : amn_tile ? 0 : nkb;
        ok = stages(K_MAJOR(), 0, isplit) && stages(MN_MAJOR(), isplit, nkb);
      } else if constexpr (AMN == 2) {
        ok = stages(amn_tile, 0, nkb);
      } else {
        ok = stages(std::integral_constant<bool, AMN == 1>(), 0, nkb);
      }
      ++tiles;
    }
    // make sure no MMA is still writing TMEM when the CTA tears down
    if (sm100::elect_one()) sm100::mma_commit(&drain[who]);
    sm100::mbar_wait(&drain[who], 0, abort_flag, status0, LAS_ERR_TIMEOUT);
  };

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer ----------------
    int st = 0, filled = 0;     // ring slot; slots filled so far (at most NSTAGE)
    uint32_t phase = 0;         // completed rounds of the ring, modulo 2
    bool ok = true;
    OzCursor<GROUPED> cur;
    for (long t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
      if (cur.seek(t, p1, &tmA, &tmB, &tmA2, &tmA3, probs, nprob) && GROUPED) {
        sm100::tma_prefetch_desc(cur.ma);
        sm100::tma_prefetch_desc(cur.mb);
        if (PACK && cur.P->a_pack) {
          sm100::tma_prefetch_desc(cur.ma2);
          sm100::tma_prefetch_desc(cur.ma3);
        }
      }
      const OzParams& p = *cur.P;
      PackedBoxes pk = {};
      if (PACK && p.a_pack) pk = packed_boxes(p.pk_L0, cur.m0 / BM, p.pk_nb1, p.pk_T, p.pk_rp);
      for (int i = 0; i < cur.nkb; ++i) {
        if (filled == NSTAGE && !sm100::mbar_wait(&empty[st], phase ^ 1, abort_flag, p.status,
                                                  LAS_ERR_TIMEOUT)) {
          ok = false;
          break;
        }
        uint8_t* sa = smem + st * T::STAGE_BYTES;
        sm100::mbar_arrive_expect_tx(&full[st], A_BYTES + NDIG * (FIXBN ? FIXBN : p.bn) * BK * 2);
        const int kb = cur.kb0 + i;
        if (PACK && p.a_pack) {   // K block kb = 8 J + kk lies in column block J of b^L
          const int J = kb >> 3;
          if (J <= pk.R)           // stored lower tile (R, J): rows mu, K = nu
            sm100::tma_load_3d(sa, cur.ma, &full[st], 0, pk.lower(kb), 0);
          else if (J < p.pk_nb1)   // stored tile (J, R) read MN-major: its rows are this K
            sm100::tma_load_4d(sa, cur.ma2, &full[st], 0, kb & 7, pk.mirror(J), 0);
          else                     // ragged rows nu >= n1 of b^L, MN-major
            sm100::tma_load_4d(sa, cur.ma3, &full[st], 0, pk.ragged(kb), pk.R * (BM / BK), 0);
        } else if (p.a_mn) {   // rows of the stored planes are this product's K, their K blocks its M
          sm100::tma_load_4d(sa, cur.ma, &full[st], 0, p.a_row0 / ROWGRAN + kb, cur.m0 / BK, 0);
        } else {
          sm100::tma_load_3d(sa, cur.ma, &full[st], 0, box_row(kb, p.a_rpad, p.a_row0, cur.m0), 0);
        }
        sm100::tma_load_3d(sa + A_BYTES, cur.mb, &full[st], 0,
                           box_row(kb, p.b_rpad, p.b_row0, cur.n0), 0);
        if (filled < NSTAGE) ++filled;
        if (++st == NSTAGE) {
          st = 0;
          phase ^= 1;
        }
      }
    }
    // never leave the CTA with a bulk copy still writing its shared memory: wait for the last
    // copy into every slot (slots before st in this round of the ring, the others in the last one)
    for (int k = 0; k < filled; ++k)
      sm100::mbar_wait(&full[k], k < st ? phase : phase ^ 1, abort_flag, status0,
                       LAS_ERR_TIMEOUT);
  } else if (warp == 1 || warp == 2) {
    if constexpr (IN_TURN) issue_turns(warp - 1);
    else if (lane == 0 && warp == 1) issue_group(std::true_type());
    else if (lane == 0) issue_group(std::false_type());
  } else if (warp >= EPI_WARP0) {
    // ---------------- epilogue (16 warps) ----------------
    const int lq = warp & 3;                 // TMEM lane quarter this warp may access
    const int cg = (warp - EPI_WARP0) >> 2;          // column blocks cg, cg + 4, cg + 8, ... of 8
    const uint32_t tl = tmem + ((uint32_t)(lq * 32) << 16);
    uint32_t gc = 0, tcount = 0;
    bool ok = true;
    OzCursor<GROUPED> cur;
    // One tile of a width: drains, then results; false when a wait ran out.
    auto finish_tile = [&](auto bn_c) -> bool {
      constexpr int bn = decltype(bn_c)::value;
      // the tile's 8-column blocks are dealt round-robin to the 4 column groups (every TMEM load is
      // 8 columns at an 8-aligned column): at most MAXB per thread
      constexpr int MAXB = (bn / 8 + 3) / 4;
      const OzParams& p = *cur.P;
      const int m0 = cur.m0, n0 = cur.n0, kb0 = cur.kb0, nkb = cur.nkb;
      const int nb = (bn / 8 - cg + 3) / 4;   // this warp's column blocks (warp-uniform)
      const float tscale = __int_as_float((127 + 8 * (NEXACT - 1) + p.sh) << 23);  // 2^(24+sh)
      const int nchunks = (nkb + CHUNK - 1) / CHUNK;
      unsigned long long acc[MAXB * 8];
#pragma unroll
      for (int j = 0; j < MAXB * 8; ++j) acc[j] = 0;
      for (int c = 0; c < nchunks; ++c, ++gc) {
        const bool fin = (c == nchunks - 1);
        if (!sm100::mbar_wait(accf, gc & 1, abort_flag, p.status, LAS_ERR_TIMEOUT, 256) ||
            (!IN_TURN && fin && !sm100::mbar_wait(tailf, tcount & 1, abort_flag, p.status, LAS_ERR_TIMEOUT,
                                      64)))
          return false;
        sm100::tc_fence_after();
        int extra = 0;
        if (fin) {
          // tail first, so that the next tile's tail MMAs can start:
          // acc <- acc * 2^sh + rint(tail * 2^(24+sh))  (int64, modulo 2^64)
          uint32_t r[MAXB][8];
#pragma unroll
          for (int b = 0; b < MAXB; ++b)
            if (b < nb) sm100::tmem_ld8(tl + T::TAIL_COL + (uint32_t)((cg + 4 * b) * 8), r[b]);
          sm100::tmem_wait_ld();
          sm100::tc_fence_before();
          __syncwarp();
          if (lane == 0) sm100::mbar_arrive(accT);
#pragma unroll
          for (int b = 0; b < MAXB; ++b)
            if (b < nb)
#pragma unroll
              for (int e = 0; e < 8; ++e)
                acc[b * 8 + e] = (acc[b * 8 + e] << p.sh) +
                                 (unsigned long long)rint_ll(__uint_as_float(r[b][e]) * tscale);
          extra = p.sh;
        }
        // exact groups: integers g_q (|g_q| <= 2^24) in units of 2^-8q, merged as
        // V = ((g_0 2^8 + g_1) 2^8 + g_2) 2^8 + g_3 (the first step fits 32 bits)
        static_assert(NEXACT == 4, "the merge below is written for four exact groups");
#pragma unroll
        for (int b = 0; b < MAXB; ++b) {
          if (b < nb) {
            const uint32_t col = (uint32_t)((cg + 4 * b) * 8);
            uint32_t r[NEXACT][8];
#pragma unroll
            for (int q = 0; q < NEXACT; ++q) sm100::tmem_ld8(tl + q * bn + col, r[q]);
            sm100::tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const int g0 = __float2int_rn(__uint_as_float(r[0][e]));
              const int g1 = __float2int_rn(__uint_as_float(r[1][e]) * 256.0f);
              const int g2 = __float2int_rn(__uint_as_float(r[2][e]) * 65536.0f);
              const int g3 = __float2int_rn(__uint_as_float(r[3][e]) * 16777216.0f);
              const long long v = (long long)(g0 * 256 + g1) * 65536 + (long long)g2 * 256 + g3;
              acc[b * 8 + e] += (unsigned long long)v << extra;
            }
          }
        }
        sm100::tc_fence_before();
        __syncwarp();
        if (lane == 0) sm100::mbar_arrive(acce);   // exact accumulators free from here on
      }
      // FP64 results (overlaps the next tile's MMAs)
      const int row = m0 + lq * 32 + lane - p.row_skip;
      bool live = row >= 0 && row < p.M;
      long L = 0, mu = 0;
      int ea;
      if constexpr (PACK) {
        if (p.mode == 1) {   // row (L, mu) of the Ht layout
          L = row / p.ht_rows;
          const int j = (int)(row - L * p.ht_rows);
          mu = p.ht_mu0 + j;
          live = live && j < p.ht_live;
        }
        ea = (p.ea && live) ? p.ea[p.ea_perL ? L : row] : 0;
      } else {
        ea = (p.ea && live) ? p.ea[row] : 0;
        if (p.mode == 1) {
          L = row / p.ht_n;
          mu = row - L * p.ht_n;
        }
      }
      const int z = kb0 / p.kb_per_split;
      const int e0 = ea - 14 - 8 * (NEXACT - 1) - p.sh;
      double* const orow = p.mode == 0 ? p.out + (long)z * p.zstride + (long)row * p.ldc
                                       : p.out + (long)z * p.zstride +
                                             L * p.ht_op * (long)p.ht_n + mu;
#pragma unroll
      for (int b = 0; b < MAXB; ++b) {
        const int c0 = n0 + (cg + 4 * b) * 8;
        if (b >= nb || !live || c0 >= p.N) continue;
        if (p.vec && c0 + 8 <= p.N) {
          // a thread's 8 columns are 64 bytes of its row: two 32-byte stores (8-byte ones of a warp
          // are 32 partial sectors each, and a tile's took 18000 clocks)
#pragma unroll
          for (int h = 0; h < 8; h += 4) {
            double v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
              v[e] = make_double((long long)acc[b * 8 + h + e], e0 + p.eb[c0 + h + e]);
            sm100::st_global_32b(orow + c0 + h, v);
          }
        } else {
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const int col = c0 + e;
            if (col < p.N) {
              const double v = make_double((long long)acc[b * 8 + e], e0 + p.eb[col]);
              orow[p.mode == 0 ? (long)col : col * (long)p.ht_n] = v;
            }
          }
        }
      }
      return true;
    };
    for (long t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++tcount) {
      cur.seek(t, p1, &tmA, &tmB, &tmA2, &tmA3, probs, nprob);
      ok = with_width<FIXBN>(cur.P->bn, finish_tile);
    }
    sm100::tc_fence_before();
  }
  __syncthreads();
  if (warp == 1) {
    sm100::tc_fence_after();
    sm100::tmem_dealloc(tmem, TMEM_COLS);
  }
}

// ------------------------------------------------------------------------------------------
// Digit extraction (integer operations on the FP64 bit patterns)
// ------------------------------------------------------------------------------------------
struct RowsStrided {  // element (r, k) = base[r*sr + k*sk]
  const double* base;
  long sr, sk;
  __device__ __forceinline__ double operator()(long r, long k) const {
    return base[r * sr + k * sk];
  }
};

// Rows that are contiguous in K: row r starts at base + r*sr.
struct RowsContig {
  const double* base;
  long sr;
  __host__ __device__ __forceinline__ const double* row(long r) const { return base + r * sr; }
  bool aligned() const { return ((uintptr_t)base & 15) == 0 && (sr & 1) == 0; }
  __device__ __forceinline__ double operator()(long r, long k) const { return row(r)[k]; }
};

struct RowsPacked {   // element (r = L*n + mu, k = nu) of the packed symmetric b^L
  const double* Bp;
  long npair;
  int n;
  __device__ __forceinline__ double operator()(long r, long k) const {
    long L = r / n, mu = r - L * n;
    long hi = mu > k ? mu : k, lo = mu > k ? k : mu;
    return Bp[L * npair + hi * (hi + 1) / 2 + lo];
  }
};

// Six balanced base-256 digits of x * 2^-e rounded at 2^-47 (|x| < 2^e), returned as the floats
// d_s * 2^-8s (exact in BF16: the upper halves of their bit patterns).  About 35 integer and FP32
// instructions; a recurrence digit by digit with conversions took 100, and the slicers were bound
// by them (3.3 to 4.4 ps per value over the chip).  With y = x 2^(47-e) rounded to an integer,
// half a unit of every digit is added at once, Y = y + sum_k 128 * 256^k, so that the bytes of Y are
// d_s + 128; a byte put under the exponent of 2^(23-8s) is the float 2^(23-8s) + (d_s + 128) 2^-8s.
__device__ __forceinline__ void digits_of(double xv, int e, uint32_t (&f)[NDIG]) {
  const uint32_t hi = (uint32_t)__double2hiint(xv), lo = (uint32_t)__double2loint(xv);
  int ee = (int)(hi >> 20) & 0x7FF;
  const uint32_t mh = (hi & 0xFFFFF) | (ee != 0 ? 0x100000u : 0u);
  ee = max(ee, 1);
  // |x| 2^(47-e) = m 2^(ee-1028-e); |x| < 2^e, so the shift is to the right.  Half up: shift by
  // one less, add 1, halve.
  const int sh = min(1027 + e - ee, 63);
  const unsigned long long m = ((unsigned long long)mh << 32) | lo;
  const unsigned long long y = ((m >> sh) + 1) >> 1;
  const unsigned long long Y = ((int)hi < 0 ? 0ull - y : y) + 0x808080808080ull;
  const uint32_t yl = (uint32_t)Y, yh = (uint32_t)(Y >> 32);
  auto digit = [](uint32_t biased, int s) {   // bits of 2^(23-8s) + (d + 128) 2^-8s -> d 2^-8s
    const float w = __int_as_float((127 - 8 * s) << 23);
    return __float_as_uint(__uint_as_float(biased) - (8388608.0f + 128.0f) * w);
  };
  auto under = [](uint32_t word, int byte, int s) {
    return __byte_perm(word, (uint32_t)(150 - 8 * s) << 23, 0x7540 | byte);
  };
  f[0] = digit(0x4B000000u | (yh >> 8), 0);   // d_0 + 128 in 0..256
  f[1] = digit(under(yh, 0, 1), 1);
  f[2] = digit(under(yl, 3, 2), 2);
  f[3] = digit(under(yl, 2, 3), 3);
  f[4] = digit(under(yl, 1, 4), 4);
  f[5] = digit(under(yl, 0, 5), 5);
}
__device__ __forceinline__ __nv_bfloat16 digit_bf16(uint32_t f) {
  return __ushort_as_bfloat16((unsigned short)(f >> 16));
}

// Digits of 8 values of one row (k0 a multiple of 8), one 16-byte store per plane.
__device__ __forceinline__ void store_digits8(const Planes& P, long r, long k0,
                                              const double (&x)[8], int e) {
  uint32_t w[NDIG][4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    uint32_t a[NDIG], b[NDIG];
    digits_of(x[2 * j], e, a);
    digits_of(x[2 * j + 1], e, b);
#pragma unroll
    for (int s = 0; s < NDIG; ++s) w[s][j] = __byte_perm(a[s], b[s], 0x7632);   // upper halves
  }
  __nv_bfloat16* p = P.p + P.idx(0, r, k0);
#pragma unroll
  for (int s = 0; s < NDIG; ++s)
    *(uint4*)(p + s * P.plane) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
}

__device__ __forceinline__ int exp_of_maxbits(unsigned long long mx) {
  return mx ? (int)((mx >> 52) & 0x7FF) - 1022 : 0;   // max|x| < 2^e
}

__device__ __forceinline__ unsigned long long absbits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}

// Rows contiguous in K, read once: rb rows (a power of two) go through shared memory (row stride S
// doubles), their maxima taken on the way in, and are cut from there, 8 values and one 16-byte
// store per plane at a time.  Rows >= R are written as zeros, and every k in [K, kb*BK).  The bytes
// are the bound: 8 read and 12 written per value; reading the row a second time from memory took
// 28 (2400 x 192 rows of 1200 values: 2.02 ms, 5.5 TB/s, against 2.34).  Few rows per block leave room for
// five or more blocks per SM, whose loads and stores overlap.  S = 2 modulo 16: the 16-byte reads of
// 8 neighbouring threads (rows, or 4 rows and two halves) fall into different banks.
// Blocks of 256 threads.
__device__ __forceinline__ void slice_kmajor_block(const RowsContig& src, int vec, const Planes& P,
                                                   long rows, long kb, int lg, int S, int* ex,
                                                   long block) {
  extern __shared__ __align__(16) double rowbuf[];
  __shared__ unsigned long long mxs[32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rb = 1 << lg;
  const long r0 = block << lg;
  const int n = (int)P.K, kend = (int)(kb * BK);
  if (tid < rb) mxs[tid] = 0;
  __syncthreads();
  const int parts = rb < 8 ? 8 >> lg : 1, seg = ((kend + parts - 1) / parts + 63) / 64 * 64;
  for (int i = warp; i < rb * parts; i += 8) {
    const int row = i & (rb - 1), k0 = (i >> lg) * seg, k1 = min(kend, k0 + seg);
    const long r = r0 + row;
    const bool live = r < P.R;
    const double* p = live ? src.row(r) : nullptr;
    double* q = rowbuf + row * S;
    unsigned long long m = 0;
    auto take = [&](int k, double2 v) {
      *(double2*)(q + k) = v;
      const unsigned long long a = absbits(v.x), b = absbits(v.y), c = a > b ? a : b;
      m = c > m ? c : m;
    };
    int k = k0 + 2 * lane;
    const int kv = live && vec ? min(k1, n & ~1) : k0;
#pragma unroll 5
    for (; k < kv; k += 64) take(k, __ldg((const double2*)(p + k)));
    for (; k < k1; k += 64)
      take(k, make_double2(live && k < n ? p[k] : 0.0, live && k + 1 < n ? p[k + 1] : 0.0));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long v = __shfl_xor_sync(0xffffffffu, m, o);
      m = v > m ? v : m;
    }
    if (lane == 0) atomicMax(&mxs[row], m);
  }
  __syncthreads();
  if (tid < rb && r0 + tid < P.R) ex[r0 + tid] = exp_of_maxbits(mxs[tid]);
  const int row = tid & (rb - 1);
  const long r = r0 + row;
  if (r >= rows) return;
  const int e = exp_of_maxbits(mxs[row]);
  const double* q = rowbuf + row * S;
  for (int k = (tid >> lg) * 8; k < kend; k += (256 >> lg) * 8) {
    double x[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const double2 t = *(const double2*)(q + k + 2 * j);
      x[2 * j] = t.x;
      x[2 * j + 1] = t.y;
    }
    store_digits8(P, r, k, x, e);
  }
}

// Sources read along the rows r (neighbouring r are neighbours in memory, or nearly), 16 rows per
// block over all of K: maxima first, then a warp cuts 16 rows x 16 values of K per step, whose
// stores are 512 contiguous bytes per plane.  For products small enough to stay in L2 between the
// two passes.  Rows >= R are written as zeros.  Blocks of NT threads.
template <int NT, class Acc>
__device__ __forceinline__ void slice_cols_block(const Acc& acc, const Planes& P, long rows,
                                                 long kb, int* ex, long block) {
  constexpr int NW = NT / 32;
  __shared__ unsigned long long red[NW][16];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rl = lane & 15;
  const long r = block * 16 + rl;
  const bool live = r < P.R;
  unsigned long long m = 0;
  if (live) {
#pragma unroll 4
    for (long k = tid >> 4; k < P.K; k += NT / 16) {
      const unsigned long long b = absbits(acc(r, k));
      m = b > m ? b : m;
    }
  }
  const unsigned long long o = __shfl_xor_sync(0xffffffffu, m, 16);
  m = o > m ? o : m;
  if (lane < 16) red[warp][rl] = m;
  __syncthreads();
  for (int w = 0; w < NW; ++w) m = red[w][rl] > m ? red[w][rl] : m;
  const int e = exp_of_maxbits(m);
  if (tid < 16 && live) ex[r] = e;
  if (r >= rows) return;
  for (long b = warp; b < kb; b += NW) {
    const long k0 = b * BK + (lane >> 4) * 8;
    double x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = (live && k0 + j < P.K) ? acc(r, k0 + j) : 0.0;
    store_digits8(P, r, k0, x, e);
  }
}

__global__ void __launch_bounds__(256)
k_slice_kmajor(RowsContig src, int vec, Planes P, long rows, long kb, int lg, int S, int* ex) {
  pdl_begin();
  slice_kmajor_block(src, vec, P, rows, kb, lg, S, ex, blockIdx.x);
}

template <class Acc>
__global__ void __launch_bounds__(512)
k_slice_cols(Acc acc, Planes P, long rows, long kb, int* ex) {
  pdl_begin();
  slice_cols_block<512>(acc, P, rows, kb, ex, blockIdx.x);
}

// Both operands of a product A B, A contiguous in K, B along its columns, in one launch: the first
// ncols blocks cut B (each of them takes longest), the others A; and the status word is cleared.
__global__ void __launch_bounds__(256)
k_slice_operands(RowsContig a, int vec, Planes Pa, long kb, int lg, int S, int* ea, RowsStrided b,
                 Planes Pb, int* eb, int ncols, int* status) {
  pdl_begin();
  if (blockIdx.x == 0 && threadIdx.x == 0) *status = 0;
  if ((int)blockIdx.x < ncols)
    slice_cols_block<256>(b, Pb, Pb.R, kb, eb, blockIdx.x);
  else
    slice_kmajor_block(a, vec, Pa, Pa.R, kb, lg, S, ea, (long)blockIdx.x - ncols);
}

// The second pass of such sources with the maxima given (mx): one warp per 16 rows x 16 values of
// K, live rows only.
__global__ void __launch_bounds__(256)
k_digits_cols(RowsStrided acc, Planes P, long kb, const unsigned long long* __restrict__ mx, int* ex) {
  pdl_begin();
  const long groups = (P.R + 15) / 16;
  const long w = blockIdx.x * 8L + (threadIdx.x >> 5);
  if (w >= groups * kb) return;
  const long b = w / groups;
  const int lane = threadIdx.x & 31;
  const long r = (w - b * groups) * 16 + (lane & 15);
  if (r >= P.R) return;
  const int e = exp_of_maxbits(mx[r]);
  const long k0 = b * BK + (lane >> 4) * 8;
  if (k0 == 0) ex[r] = e;
  double x[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) x[j] = k0 + j < P.K ? acc(r, k0 + j) : 0.0;
  store_digits8(P, r, k0, x, e);
}

// Rows too long for k_slice_kmajor, and sources contiguous in neither index: one warp per row
// r < rows (rows >= R are written as zeros); exponent e_r with max|x| < 2^e_r for r < R, digit
// planes for every k < kb*BK (zero beyond K).
template <class Acc>
__global__ void __launch_bounds__(256)
k_slice_rows(Acc acc, Planes P, long rows, long kb, int* ex) {
  pdl_begin();
  const long r = (blockIdx.x * (long)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (r >= rows) return;
  const bool live = r < P.R;
  unsigned long long mx = 0;
  if (live)
    for (long k = lane; k < P.K; k += 32) {
      const unsigned long long b = absbits(acc(r, k));
      mx = b > mx ? b : mx;
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long v = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = v > mx ? v : mx;
  }
  const int e = exp_of_maxbits(mx);
  if (lane == 0 && live) ex[r] = e;
  const long kend = kb * BK;
  for (long k = lane; k < kend; k += 32) {
    uint32_t d[NDIG];
    digits_of((live && k < P.K) ? acc(r, k) : 0.0, e, d);
#pragma unroll
    for (int s = 0; s < NDIG; ++s) P.p[P.idx(s, r, k)] = digit_bf16(d[s]);
  }
}

// Long rows, pass 1: mx[r] = max_k |x(r,k)| as ordered bit patterns (grid: segments x rows).
__global__ void __launch_bounds__(256)
k_rowmax_long(RowsContig acc, long K, long seg, unsigned long long* mx) {
  pdl_begin();
  __shared__ unsigned long long red[8];
  const long r = blockIdx.y;
  const long k0 = (long)blockIdx.x * seg, k1 = min(K, k0 + seg);
  unsigned long long m = 0;
  for (long k = k0 + threadIdx.x; k < k1; k += blockDim.x) {
    const unsigned long long b = absbits(acc(r, k));
    m = b > m ? b : m;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long v = __shfl_xor_sync(0xffffffffu, m, o);
    m = v > m ? v : m;
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = red[w] > m ? red[w] : m;
    if (m) atomicMax(&mx[r], m);
  }
}

// Long rows, pass 2: 8 values per thread over rows x kb*BK (zeros outside R x K); the source is
// contiguous in K.  Neighbouring threads write neighbouring 16 bytes of a K block.
__global__ void __launch_bounds__(256)
k_digits_long(RowsContig acc, Planes P, long rows, long kbc, const unsigned long long* mx, int* ex) {
  pdl_begin();
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i >= rows * kbc * 2) return;
  const long kb = i / (rows * 2), rem = i - kb * (rows * 2);
  const long r = rem >> 1, k0 = kb * BK + (rem & 1) * 8;
  const bool live = r < P.R;
  const int e = live ? exp_of_maxbits(mx[r]) : 0;
  if (k0 == 0 && live) ex[r] = e;
  double x[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) x[j] = (live && k0 + j < P.K) ? acc(r, k0 + j) : 0.0;
  store_digits8(P, r, k0, x, e);
}

// Packed-triangle digit planes of B (see BPacked).  Pass 1: max |b^L| over the packed triangle
// of each L (one block per L) and its exponent.
__global__ void __launch_bounds__(256)
k_bpacked_max(const double* __restrict__ Bp, long npair, unsigned long long* __restrict__ mx,
              int* __restrict__ ex) {
  __shared__ unsigned long long red[8];
  const long L = blockIdx.x;
  const double* b = Bp + L * npair;
  unsigned long long m = 0;
  for (long k = threadIdx.x; k < npair; k += blockDim.x) {
    const unsigned long long v = absbits(b[k]);
    m = v > m ? v : m;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long v = __shfl_xor_sync(0xffffffffu, m, o);
    m = v > m ? v : m;
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = red[w] > m ? red[w] : m;
    mx[L] = m;
    ex[L] = exp_of_maxbits(m);
  }
}

// Pass 2: the stored tiles, one thread per element in storage order (plane by plane: tile, K
// block of 16, row, column), digits relative to 2^e(L).
__global__ void __launch_bounds__(256)
k_bpacked_tiles(const double* __restrict__ Bp, long npair, int T, const int* __restrict__ ex,
                Planes P, long total) {
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i >= total) return;
  const int c = (int)(i & 15), row = (int)((i >> 4) & 127), kk = (int)((i >> 11) & 7);
  const long tt = i >> 14;              // tile index L T + t
  const long L = tt / T;
  const int t = (int)(tt - L * T);
  int I = (int)((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);   // t = I (I + 1) / 2 + J, J <= I
  while ((I + 1) * (I + 2) / 2 <= t) ++I;
  while (I * (I + 1) / 2 > t) --I;
  const int J = t - I * (I + 1) / 2;
  const long mu = 128L * I + row, nu = 128L * J + 16 * kk + c;
  const long hi = mu > nu ? mu : nu, lo = mu > nu ? nu : mu;
  uint32_t d[NDIG];
  digits_of(Bp[L * npair + hi * (hi + 1) / 2 + lo], ex[L], d);
  const long o = (tt * 8 + kk) * (128L * BK) + Planes::swz(row, c);
#pragma unroll
  for (int s = 0; s < NDIG; ++s) P.p[s * P.plane + o] = digit_bf16(d[s]);
}

// Pass 3: the ragged rows mu = n1 + j (rows (L, j), j < rp, of all X rp, zeros for j >= r; then
// zero padding rows), every K block of the layout (zero digits for nu >= n), in the K-blocked
// storage order.
__global__ void __launch_bounds__(256)
k_bpacked_ragged(const double* __restrict__ Bp, long npair, int n, int n1, int r, int rp,
                 const int* __restrict__ ex, Planes P, long live_rows) {
  const long kend = P.nkb * BK;
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i >= P.Rpad * kend) return;
  const long kb = i / (P.Rpad * BK), rem = i - kb * (P.Rpad * BK);
  const long row = rem / BK, k = kb * BK + (rem - row * BK);
  double x = 0.0;
  int e = 0;
  if (row < live_rows) {
    const long L = row / rp, j = row - L * rp, mu = n1 + j;
    e = ex[L];
    if (k < n && j < r) {
      const long hi = mu > k ? mu : k, lo = mu > k ? k : mu;
      x = Bp[L * npair + hi * (hi + 1) / 2 + lo];
    }
  }
  uint32_t d[NDIG];
  digits_of(x, e, d);
#pragma unroll
  for (int s = 0; s < NDIG; ++s) P.p[P.idx(s, row, k)] = digit_bf16(d[s]);
}

// Column maxima of Ht [R][n] over its rows (coalesced along the columns): mx[mu] (atomic max of
// |x| bit patterns).  Grid: (ceil(n/256), row segments).
__global__ void __launch_bounds__(256)
k_colmax(const double* __restrict__ Ht, long R, int n, long seg, unsigned long long* mx) {
  pdl_begin();
  const int mu = blockIdx.x * 256 + threadIdx.x;
  if (mu >= n) return;
  const long r0 = (long)blockIdx.y * seg, r1 = min(R, r0 + seg);
  unsigned long long m = 0;
  for (long r = r0; r < r1; ++r) {
    const unsigned long long b = absbits(Ht[r * n + mu]);
    m = b > m ? b : m;
  }
  if (m) atomicMax(&mx[mu], m);
}

}  // namespace lasdf_split

using namespace lasdf_split;

// ------------------------------------------------------------------------------------------
// Host side
// ------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  }
  return fn;
}

// 3D map over K-blocked digit planes: dims {256, nkb*Rpad/16, NDIG} (rows of 16 stored rows), box
// {256, box_rows/16, NDIG}: box_rows * 32 contiguous bytes per plane, copied as they are.
static las_status make_plane_map(CUtensorMap* m, const Planes& P, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return LAS_ERR_CUDA;
  const long rows = P.nkb * P.Rpad / ROWGRAN;
  if (((uintptr_t)P.p & 15) || P.Rpad % ROWGRAN || box_rows % ROWGRAN || rows <= 0 ||
      rows > 0x7FFFFFFFL / ROWGRAN)
    return LAS_ERR_INTERNAL;
  cuuint64_t dims[3] = {(cuuint64_t)ROWGRAN * BK, (cuuint64_t)rows, (cuuint64_t)NDIG};
  cuuint64_t strides[2] = {(cuuint64_t)ROWGRAN * BK * 2, (cuuint64_t)P.plane * 2};
  cuuint32_t box[3] = {(cuuint32_t)(ROWGRAN * BK), (cuuint32_t)(box_rows / ROWGRAN),
                       (cuuint32_t)NDIG};
  cuuint32_t es[3] = {1, 1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, (void*)P.p, dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? LAS_OK : LAS_ERR_INTERNAL;
}

// 4D map for reading planes MN-major (as the A operand of a product whose K runs along the
// stored rows): dims {256, Rpad/16, nkb, NDIG}; a box is 16 stored rows (16 values of K, 512
// bytes) of BM / BK consecutive K blocks of the stored layout (BM values of M), every plane:
// BM * 32 bytes per plane, as in the K-major case.  Boxes past the last stored K block read the
// TMA's zero fill.
static las_status make_plane_map_mn(CUtensorMap* m, const Planes& P) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return LAS_ERR_CUDA;
  static_assert(ROWGRAN == BK, "a 512-byte row holds the 16 values of K of one stage");
  if (((uintptr_t)P.p & 15) || P.Rpad <= 0 || P.Rpad % ROWGRAN || P.Rpad > 0x7FFFFFFFL ||
      P.nkb <= 0)
    return LAS_ERR_INTERNAL;
  cuuint64_t dims[4] = {(cuuint64_t)ROWGRAN * BK, (cuuint64_t)(P.Rpad / ROWGRAN),
                        (cuuint64_t)P.nkb, (cuuint64_t)NDIG};
  cuuint64_t strides[3] = {(cuuint64_t)ROWGRAN * BK * 2, (cuuint64_t)P.Rpad * BK * 2,
                           (cuuint64_t)P.plane * 2};
  cuuint32_t box[4] = {(cuuint32_t)(ROWGRAN * BK), 1, (cuuint32_t)(BM / BK), (cuuint32_t)NDIG};
  cuuint32_t es[4] = {1, 1, 1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (void*)P.p, dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? LAS_OK : LAS_ERR_INTERNAL;
}

// Widest tile (the stage layout's B region): 96 columns, so that the four exact accumulators and the
// tail take 480 of the 512 TMEM columns.  A product runs with tiles of 48, 64, 80 or 96 columns.
constexpr int OZ_BN = 96;
constexpr int TILE_WIDTHS[] = {48, 64, 80, 96};
// Time of a stage (16 values of K) of each width in launches of 50 to 75 stages a tile, in clocks of
// 2070 MHz; only the ratios are used.  (The SMs run this kernel at 1.95 to 2.0 GHz: 503 ns at 64
// columns, 679 in the half transform and 699 in the full transform at 96, the half transform's being
// 1340 clocks by the SM's own counter.)  What a narrow tile saves is its B planes and, at 48 and 64
// columns, the issue in turn, so the width that wins is mostly the one that fits.  op = 128 (800
// orbitals): 2 x 64 columns 2040, 96 + 64 2450 and B read twice.  Grouped launches, which issue by
// group, take 1130 to 1170 at 64 columns; the rule is the same there, and for 241 to 256 columns takes
// 4 x 64 although 3 x 96 would end about 7 % sooner.
constexpr int STAGE_TIME[] = {1000, 1020, 1310, 1430};
static bool valid_bn(int bn) { return bn == 48 || bn == 64 || bn == 80 || bn == 96; }
static int stage_time(int bn) { return STAGE_TIME[(bn - 48) / 16]; }
static long cols_time(long N, int bn) { return (N + bn - 1) / bn * stage_time(bn); }
static int pick_bn(long N) {
  int best = 96;
  for (int w : TILE_WIDTHS)
    if (cols_time(N, w) < cols_time(N, best)) best = w;
  return best;
}

template <bool GROUPED, int FIXBN>
static cudaError_t ozaki_attr() {
  auto set = [](auto kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                OzTile<OZ_BN>::SMEM_BYTES);
  };
  cudaError_t e;
  if constexpr (GROUPED) {
    e = set(k_ozaki<OZ_BN, true, FIXBN, false>);
  } else {
    e = set(k_ozaki<OZ_BN, false, FIXBN, false, 0>);
    if (e == cudaSuccess) e = set(k_ozaki<OZ_BN, false, FIXBN, false, 1>);
  }
  return e != cudaSuccess ? e : set(k_ozaki<OZ_BN, GROUPED, FIXBN, true>);
}

// Dynamic shared memory that a row-slicing launch may ask for: one row of 383 K blocks.  Beside it
// stands the kernels' static part of 1 and 2 KB (the launch would be refused at the default limit,
// which counts both), so ozaki_prepare raises the limit.
constexpr int SLICE_SMEM = 48 * 1024;
static cudaError_t slice_attr() {
  auto set = [](auto kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SLICE_SMEM);
  };
  const cudaError_t e = set(k_slice_kmajor);
  return e != cudaSuccess ? e : set(k_slice_operands);
}

// Does the product need the instantiation with the packed-triangle logic (its A is the packed
// form, or its rows are the ragged rows of that form, with one exponent per auxiliary index)?
static inline bool needs_pack(const OzParams& p) { return p.a_pack || p.ea_perL; }

static las_status ozaki_prepare() {
  static volatile int done[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return LAS_ERR_CUDA;
  if (done[dev]) return LAS_OK;
  cudaError_t e = ozaki_attr<false, 96>();
  if (e == cudaSuccess) e = ozaki_attr<false, 80>();
  if (e == cudaSuccess) e = ozaki_attr<false, 64>();
  if (e == cudaSuccess) e = ozaki_attr<false, 48>();
  if (e == cudaSuccess) e = ozaki_attr<true, 96>();
  if (e == cudaSuccess) e = ozaki_attr<true, 64>();
  if (e == cudaSuccess) e = ozaki_attr<true, 0>();
  if (e == cudaSuccess) e = slice_attr();
  if (e != cudaSuccess) {
    las_record_cuda_error(e, "cudaFuncSetAttribute(split products)", __FILE__, __LINE__);
    return LAS_ERR_CUDA;
  }
  done[dev] = 1;
  return LAS_OK;
}

static inline long rup(long x, long m) { return (x + m - 1) / m * m; }

static int num_sms() {
  static int nsm = 0;
  if (!nsm) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm <= 0)
      nsm = 148;
  }
  return nsm;
}


// out = A * B^T over K: rows [a_row0, a_row0 + M) of A (row exponents ea, or 0 when null),
// rows [b_row0, b_row0 + N) of B (row exponents eb: the column exponents of the product).
// mode 0: out[z*zstride + r*ldc + c] (z = K split); mode 1: Ht layout (rows (L, mu)).
// Output tiles of an M x N product per K split (lower: only those touching the lower triangle).
static long ozaki_tiles(long M, long N, int lower, int bn = OZ_BN) {
  const long ntm = (M + BM - 1) / BM, ntn = (N + bn - 1) / bn;
  if (!lower) return ntm * ntn;
  long t = 0;
  for (long i = 0; i < ntm; ++i) t += lower_tiles_in_row((int)i, (int)ntn, bn);
  return t;
}

// K-split factor in [lo, cap] that shares `tiles` output tiles of a product with kb K blocks out
// most evenly over the persistent CTAs: ceil(tiles*ks / SMs) rounds, each of ceil(kb/ks) blocks
// plus about a chunk of pipeline fill and drain.
static int balanced_ksplit(long tiles, long kb, long cap, long lo = 1) {
  const long sms = num_sms();
  int best = (int)lo;
  double best_t = 1e300;
  for (long ks = lo; ks <= cap; ++ks) {
    const double t = (double)((tiles * ks + sms - 1) / sms) * (double)((kb + ks - 1) / ks + CHUNK);
    if (t < best_t * (1.0 - 1e-9)) {
      best_t = t;
      best = (int)ks;
    }
  }
  return best;
}

// Shortest K of a split: one chunk.  (At 2048 the projection of the 48-orbital problem, K = 2560,
// was one tile on one SM: 120 us.)
constexpr long KSPLIT_MIN = CHUNK * BK;

// Products recorded instead of launched while a group is being recorded on this host thread.
struct OzGroup {
  std::vector<OzProblem> probs;
  long tiles = 0;
};
static thread_local OzGroup* g_record = nullptr;

OzGroup* ozgroup_new() { return new OzGroup(); }
void ozgroup_free(OzGroup* g) { delete g; }
void ozgroup_record(OzGroup* g) { g_record = g; }
size_t ozgroup_count(const OzGroup* g) { return g ? g->probs.size() : 0; }
size_t ozgroup_bytes(size_t nprob) { return nprob * sizeof(OzProblem); }

// One persistent launch over every recorded product (tiles concatenated in recording order);
// `dev` is device memory for the product descriptions, filled by ozgroup_upload before the
// launch runs (the launch may be captured into a graph first).
las_status ozgroup_launch(const OzGroup* g, void* dev, cudaStream_t st) {
  if (!g || g->probs.empty()) return LAS_OK;
  if (!dev || ((uintptr_t)dev % alignof(OzProblem))) return LAS_ERR_INTERNAL;
  OzParams dummy;
  memset(&dummy, 0, sizeof(dummy));
  CUtensorMap m0;
  memset(&m0, 0, sizeof(m0));
  dim3 grid((unsigned)std::min<long>(g->tiles, num_sms()), 1, 1);
  int bn = g->probs[0].p.bn;   // one width for the whole launch, or 0: read per product
  for (const OzProblem& pr : g->probs)
    if (pr.p.bn != bn) bn = 0;
  bool pack = false;
  for (const OzProblem& pr : g->probs) pack |= needs_pack(pr.p);
  const OzProblem* probs = (const OzProblem*)dev;
  const int np = (int)g->probs.size();
  constexpr int SM = OzTile<OZ_BN>::SMEM_BYTES;
  auto go = [&](auto kern) {
    launch_chained(kern, grid, NTHREADS, SM, st, m0, m0, m0, m0, dummy, probs, np, g->tiles);
  };
  if (bn == 96) pack ? go(k_ozaki<OZ_BN, true, 96, true>) : go(k_ozaki<OZ_BN, true, 96, false>);
  else if (bn == 64) pack ? go(k_ozaki<OZ_BN, true, 64, true>) : go(k_ozaki<OZ_BN, true, 64, false>);
  else pack ? go(k_ozaki<OZ_BN, true, 0, true>) : go(k_ozaki<OZ_BN, true, 0, false>);
  las_count_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    las_record_cuda_error(e, "k_ozaki grouped launch", __FILE__, __LINE__);
    return LAS_ERR_CUDA;
  }
  return LAS_OK;
}

las_status ozgroup_upload(const OzGroup* g, void* dev) {
  if (!g || g->probs.empty()) return LAS_OK;
  LAS_CUDA_TRY(cudaMemcpy(dev, g->probs.data(), g->probs.size() * sizeof(OzProblem),
                          cudaMemcpyHostToDevice));
  return LAS_OK;
}

// Launch one product (persistent: one CTA per SM), or record it into the group being recorded.
static las_status ozaki_submit(OzProblem& pr, cudaStream_t st) {
  const OzParams& p = pr.p;
  const long tiles = p.tiles_z * p.ksplit;
  if (g_record) {   // part of a grouped launch
    pr.tile0 = g_record->tiles;
    g_record->tiles += tiles;
    g_record->probs.push_back(pr);
    return LAS_OK;
  }
  dim3 grid((unsigned)std::min<long>(tiles, num_sms()), 1, 1);
  constexpr int SM = OzTile<OZ_BN>::SMEM_BYTES;
  auto go = [&](auto kern) {
    launch_chained(kern, grid, NTHREADS, SM, st, pr.tmA, pr.tmB, pr.tmA2, pr.tmA3, p, nullptr, 0, tiles);
  };
  const bool pack = needs_pack(p);
  // full-row products take an instantiation with their A orientation as a compile-time constant
  auto width = [&](auto bn_c) {
    constexpr int bn = decltype(bn_c)::value;
    if (pack) go(k_ozaki<OZ_BN, false, bn, true>);
    else if (p.a_mn) go(k_ozaki<OZ_BN, false, bn, false, 1>);
    else go(k_ozaki<OZ_BN, false, bn, false, 0>);
  };
  switch (p.bn) {
    case 48: width(std::integral_constant<int, 48>()); break;
    case 64: width(std::integral_constant<int, 64>()); break;
    case 80: width(std::integral_constant<int, 80>()); break;
    default: width(std::integral_constant<int, 96>()); break;
  }
  las_count_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    las_record_cuda_error(e, "k_ozaki launch", __FILE__, __LINE__);
    return LAS_ERR_CUDA;
  }
  return LAS_OK;
}

// Fractional bits kept for the tail: |fixed-point sum| < 2^38 * (k per CTA) must fit 62 bits.
static int tail_shift(int kb_per_split) {
  int lgk = 0;
  while ((1L << lgk) < (long)kb_per_split * BK) ++lgk;
  return std::max(0, std::min(20, 61 - 14 - 8 * (NEXACT - 1) - lgk));
}

// The product's description (tensor maps and parameters), ready to be launched or recorded.
static las_status ozaki_setup(OzProblem& pr, const Planes& A, long a_row0, const int* ea, long M,
                              const Planes& B, long b_row0, const int* eb, long N, long K,
                              int ksplit, int mode, double* out, long ldc, long zstride, int ht_n,
                              int ht_op, int* status, int lower, int bn, int a_mn) {
  // a_mn: A's stored rows [a_row0, a_row0 + K) are the product's K, its stored K the rows M
  const bool a_ok = a_mn ? (a_row0 + K <= A.Rpad && M <= A.nkb * BK)
                         : (a_row0 + M <= A.Rpad && K <= A.nkb * BK);
  if (!a_ok || b_row0 + N > B.Rpad || K > B.nkb * BK || !valid_bn(bn) || (a_mn && lower))
    return LAS_ERR_INTERNAL;
  // box coordinates are multiples of ROWGRAN rows: the product starts up to 15 rows early and
  // drops what it computes there
  const int skip = box_skip(a_row0);
  if (b_row0 % ROWGRAN || (skip && (a_mn || lower)) || M + skip > 0x7FFFFFFFL)
    return LAS_ERR_INTERNAL;
  las_status s = ozaki_prepare();
  if (s != LAS_OK) return s;
  memset(&pr, 0, sizeof(pr));
  if ((s = a_mn ? make_plane_map_mn(&pr.tmA, A) : make_plane_map(&pr.tmA, A, BM)) != LAS_OK)
    return s;
  if ((s = make_plane_map(&pr.tmB, B, bn)) != LAS_OK) return s;
  OzParams& p = pr.p;
  p.M = (int)M;
  p.N = (int)N;
  p.a_rpad = (int)A.Rpad;
  p.b_rpad = (int)B.Rpad;
  p.a_row0 = (int)(a_row0 - skip);
  p.row_skip = skip;
  p.b_row0 = (int)b_row0;
  p.kb_total = (int)((K + BK - 1) / BK);
  if (p.kb_total < 1) p.kb_total = 1;
  if (ksplit < 1) ksplit = 1;
  p.kb_per_split = (p.kb_total + ksplit - 1) / ksplit;
  ksplit = (p.kb_total + p.kb_per_split - 1) / p.kb_per_split;
  p.ksplit = ksplit;
  p.ea = ea;
  p.eb = eb;
  p.out = out;
  p.mode = mode;
  p.vec = mode == 0 && ((uintptr_t)out & 31) == 0 && ldc % 4 == 0 && zstride % 4 == 0;
  p.ldc = ldc;
  p.zstride = zstride;
  p.ht_n = ht_n;
  p.ht_op = ht_op;
  p.ht_rows = p.ht_live = ht_n;
  p.ht_mu0 = 0;
  p.lower = lower;
  p.tiles_z = ozaki_tiles(M + skip, N, lower, bn);
  p.sh = tail_shift(p.kb_per_split);
  p.bn = bn;
  p.a_mn = a_mn;
  p.status = status;
  return LAS_OK;
}

las_status ozaki_gemm(const Planes& A, long a_row0, const int* ea, long M, const Planes& B,
                      long b_row0, const int* eb, long N, long K, int ksplit, int mode,
                      double* out, long ldc, long zstride, int ht_n, int ht_op, int* status,
                      cudaStream_t st, int lower = 0, int bn = 0, int a_mn = 0) {
  if (M <= 0 || N <= 0) return LAS_OK;
  if (bn == 0) bn = lower && N > 64 ? OZ_BN : pick_bn(N);   // 0: the rule's width
  OzProblem pr;
  las_status s = ozaki_setup(pr, A, a_row0, ea, M, B, b_row0, eb, N, K, ksplit, mode, out, ldc,
                             zstride, ht_n, ht_op, status, lower, bn, a_mn);
  return s == LAS_OK ? ozaki_submit(pr, st) : s;
}

// out[L][p][mu] (the Ht layout, ht_op columns per L) = sum_nu b^L(mu, nu) X(nu, p) for the
// auxiliary rows [l0, l0 + nL) of packed-triangle B and the N columns p of X whose digit planes
// (rows p, K = nu) start at row x_row0 of Xd (column exponents xexp).  Two products: the full
// 128-row blocks of every b^L from the stored tiles, and the ragged rows mu >= n1.
static las_status bpacked_half(const BPacked& b, int l0, int nL, const Planes& Xd, long x_row0,
                               const int* xexp, long N, double* out, int ht_op, int* status,
                               cudaStream_t st, int bn) {
  if (nL <= 0 || N <= 0) return LAS_OK;
  if (l0 < 0 || l0 + nL > b.X || x_row0 + N > Xd.Rpad || x_row0 % ROWGRAN ||
      b.n > Xd.nkb * BK || !valid_bn(bn))
    return LAS_ERR_INTERNAL;
  las_status rc = ozaki_prepare();
  if (rc != LAS_OK) return rc;
  if (b.nb1 > 0) {
    const long M = (long)nL * b.n1;
    if (M > 0x7FFFFFFFL) return LAS_ERR_UNSUPPORTED;
    OzProblem pr;
    memset(&pr, 0, sizeof(pr));
    if ((rc = make_plane_map(&pr.tmA, b.tiles, BM)) != LAS_OK) return rc;
    if ((rc = make_plane_map_mn(&pr.tmA2, b.tiles)) != LAS_OK) return rc;
    if (b.r > 0 && (rc = make_plane_map_mn(&pr.tmA3, b.rag)) != LAS_OK) return rc;
    if ((rc = make_plane_map(&pr.tmB, Xd, bn)) != LAS_OK) return rc;
    OzParams& p = pr.p;
    p.M = (int)M;
    p.N = (int)N;
    p.a_rpad = BM;
    p.b_rpad = (int)Xd.Rpad;
    p.b_row0 = (int)x_row0;
    p.kb_total = (b.n + BK - 1) / BK;
    p.kb_per_split = p.kb_total;
    p.ksplit = 1;
    p.ea = b.exp + l0;
    p.eb = xexp;
    p.out = out;
    p.mode = 1;
    p.ht_n = b.n;
    p.ht_op = ht_op;
    p.ht_rows = p.ht_live = b.n1;
    p.ht_mu0 = 0;
    p.ea_perL = 1;
    p.tiles_z = ozaki_tiles(M, N, 0, bn);
    p.sh = tail_shift(p.kb_per_split);
    p.bn = bn;
    p.a_pack = 1;
    p.pk_nb1 = b.nb1;
    p.pk_T = b.T;
    p.pk_rp = b.rp;
    p.pk_L0 = l0;
    p.status = status;
    if ((rc = ozaki_submit(pr, st)) != LAS_OK) return rc;
  }
  if (b.r > 0) {
    OzProblem pr;
    rc = ozaki_setup(pr, b.rag, (long)l0 * b.rp, b.exp + l0, (long)nL * b.rp, Xd, x_row0, xexp,
                     N, b.n, 1, 1, out, 0, 0, b.n, ht_op, status, 0, bn, 0);
    if (rc != LAS_OK) return rc;
    pr.p.ht_rows = b.rp;
    pr.p.ht_live = b.r;
    pr.p.ht_mu0 = b.n1;
    pr.p.ea_perL = 1;
    rc = ozaki_submit(pr, st);
  }
  return rc;
}

// Digit planes P and row exponents ex of a source.  live_only: only rows < R and the K blocks that
// hold K are written (planes whose padding rows were zeroed at set-up); otherwise every padded row
// and K block of the layout is written.
static las_status slice_done(const char* what) {
  las_count_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    las_record_cuda_error(e, what, __FILE__, __LINE__);
    return LAS_ERR_CUDA;
  }
  return LAS_OK;
}
static long slice_extent(const Planes& P, bool live_only, long* kb) {
  *kb = live_only ? std::min(P.nkb, planes_nkb(P.K)) : P.nkb;
  return live_only ? P.R : P.Rpad;
}

// Any source: one warp per row.
template <class Acc>
static las_status slice_rows(Acc acc, const Planes& P, int* ex, cudaStream_t st,
                             bool live_only = false) {
  if (P.R <= 0) return LAS_OK;
  long kb;
  const long rows = slice_extent(P, live_only, &kb);
  launch_chained(k_slice_rows<Acc>, (unsigned)((rows * 32 + 255) / 256), 256, 0, st, acc, P, rows, kb, ex);
  return slice_done("k_slice_rows launch");
}

static bool slice_fits(long kb) { return (kb * BK + 2) * 8 <= SLICE_SMEM; }
static int slice_lg(long S, long rows) {
  int lg = 0;
  while (lg < 5 && (S * 8 << (lg + 1)) <= 40 * 1024 && (rows >> (lg + 1)) >= 2 * num_sms()) ++lg;
  return lg;
}

// Rows contiguous in K.  Rows per block: up to 40 KB of shared memory, and
// no more than leaves two blocks per SM; a single row has to fit 48 KB (K <= 6128).
static las_status slice_contig(RowsContig src, const Planes& P, int* ex, cudaStream_t st,
                               bool live_only = false) {
  if (P.R <= 0) return LAS_OK;
  long kb;
  const long rows = slice_extent(P, live_only, &kb);
  const long S = kb * BK + 2;
  if (!slice_fits(kb)) return slice_rows(src, P, ex, st, live_only);
  const int lg = slice_lg(S, rows);
  launch_chained(k_slice_kmajor, (unsigned)((rows + (1 << lg) - 1) >> lg), 256, (size_t)(S * 8) << lg, st, src, src.aligned(), P, rows, kb, lg, (int)S, ex);
  return slice_done("k_slice_kmajor launch");
}

// Sources read along the rows, small enough that both passes of a block of 16 rows find them in L2.
template <class Acc>
static las_status slice_cols(Acc acc, const Planes& P, int* ex, cudaStream_t st,
                             bool live_only = false) {
  if (P.R <= 0) return LAS_OK;
  long kb;
  const long rows = slice_extent(P, live_only, &kb);
  launch_chained(k_slice_cols<Acc>, (unsigned)((rows + 15) / 16), 512, 0, st, acc, P, rows, kb, ex);
  return slice_done("k_slice_cols launch");
}

// Few long rows contiguous in K (the projection's W): a block per row while a row fits shared
// memory (one launch); else block-parallel maxima in mx, then the digits of the live rows.
static las_status slice_long(RowsContig src, const Planes& P, int* ex, unsigned long long* mx,
                             cudaStream_t st) {
  if (P.R <= 0) return LAS_OK;
  if (slice_fits(planes_nkb(P.K))) return slice_contig(src, P, ex, st, true);
  LAS_CUDA_TRY(cudaMemsetAsync(mx, 0, P.R * sizeof(unsigned long long), st));
  const long seg = 8192;
  dim3 g1((unsigned)((P.K + seg - 1) / seg), (unsigned)P.R);
  launch_chained(k_rowmax_long, g1, 256, 0, st, src, P.K, seg, mx);
  las_count_launch();
  const long kb = std::min(P.nkb, planes_nkb(P.K)), tot = P.R * kb * 2;
  launch_chained(k_digits_long, (unsigned)((tot + 255) / 256), 256, 0, st, src, P, P.R, kb, mx, ex);
  return slice_done("k_digits_long launch");
}

// Large sources read along the rows ([K][R] in memory, rows of the planes = columns of the source):
// column maxima in mx (have_max: already there), then the digits of the live rows.
static las_status slice_transposed(const double* src, const Planes& P, int* ex,
                                   unsigned long long* mx, bool have_max, cudaStream_t st) {
  if (P.R <= 0) return LAS_OK;
  if (!have_max) {
    LAS_CUDA_TRY(cudaMemsetAsync(mx, 0, P.R * sizeof(unsigned long long), st));
    const long seg = 512;
    dim3 g1((unsigned)((P.R + 255) / 256), (unsigned)((P.K + seg - 1) / seg));
    launch_chained(k_colmax, g1, 256, 0, st, src, P.K, (int)P.R, seg, mx);
    las_count_launch();
  }
  const long kb = planes_nkb(P.K), warps = (P.R + 15) / 16 * kb;
  launch_chained(k_digits_cols, (unsigned)((warps + 7) / 8), 256, 0, st, 
      RowsStrided{src, 1, P.R}, P, kb, mx, ex);
  return slice_done("k_digits_cols launch");
}

struct SplitState {
  int n, X, op, Lc;
  int packed;            // layout of the Cholesky vectors' digit planes:
  Planes Bdig;           //   0: full rows (L, mu) of all X*n, K = nu, exponent per row
  int* Bexp;             //      [X*n]
  BPacked Bpk;           //   1: packed-triangle tiles, exponent per L
  Planes Cdig;           // rows p of C_occ^T, K = nu
  int* Cexp;             // [op]
  Planes Hdig;           // rows (L, p) of a chunk, K = mu
  int* Hexp;             // [Lc*op]
  Planes HdigT;          // rows mu, K = (L, p)
  Planes Wdig;           // rows q, K = (L, p)
  int* Wexp;             // [op]
  double* part;          // split_part_elems(n, op): [ks][n][op], or [ks][n][n] of the exchange
  unsigned long long* mx;  // [op + n] row maxima for long-row slicing
  Planes Mpd;            // rows p of C[:, p0:p1]^T (K = mu) for the (L|pu) transform (lazy)
  int* Mpexp;
  void* Mpblob;
  Planes hdig;           // rows mu of h, K = nu
  int* hexp;             // [n]
  int ksplit6;           // the projection's partials fit `part` for this many K splits
  int ks;                // split-K factor of the projection GEMM (autotunable)
  int bn[SPLIT_NKIND];   // tile width of each product kind (64 or 96) as chosen by the caller or the
                         // autotuner, or 0: by the rule of its columns
  // tangent (Hessian-vector) scratch, allocated by the first split_tangent_prepare: digit planes
  // of dC_occ^T (rows p, K = nu) and of the chunk's dH (rows (L, p), K = mu)
  Planes dCdig;
  int* dCexp;
  Planes dHdig;
  int* dHexp;
  void* tblob;
  int* status;
};

static void split_free(SplitState* s) {
  if (s->Mpblob) cudaFree(s->Mpblob);
  if (s->tblob) cudaFree(s->tblob);
  void* ptrs[] = {s->Bdig.p, s->Bexp, s->Bpk.tiles.p, s->Bpk.rag.p, s->Bpk.exp, s->Bpk.mx,
                  s->Cdig.p, s->Cexp,
                  s->Hdig.p, s->Hexp, s->HdigT.p,
                  s->Wdig.p, s->Wexp, s->part, s->mx, s->hdig.p, s->hexp};
  for (void* q : ptrs)
    if (q) cudaFree(q);
}

size_t split_bytes_per_aux(int n, int op) {
  // Hdig + HdigT + Wdig per auxiliary index (K-blocked, padded), plus exponents
  return (size_t)NDIG * op * rup(n, BK) * 2 * 2 + (size_t)NDIG * ROWPAD * op * 2 + (size_t)op * 4;
}

// Doubles of the partial buffer: 64 K splits of an n x op projection, and at least one n x n partial
// of the exchange product (more when n > 64 op: few occupied orbitals in a large basis).
constexpr int PART_KSPLIT = 64;
size_t split_part_elems(int n, int op) {
  return (size_t)n * std::max((long)PART_KSPLIT * op, (long)n);
}

las_status split_create(SplitState** out, int n, int X, int op, int Lc, const double* Bp,
                        int packed, int* status, cudaStream_t st, size_t* bytes) {
  *out = nullptr;
  if (!encode_fn()) return LAS_ERR_UNSUPPORTED;
  SplitState* s = (SplitState*)calloc(1, sizeof(SplitState));
  if (!s) return LAS_ERR_INTERNAL;
  s->n = n;
  s->X = X;
  s->op = op;
  s->Lc = Lc;
  s->status = status;
  s->ksplit6 = PART_KSPLIT;
  // one-time launch attributes, so that later calls can be captured into CUDA graphs
  if (ozaki_prepare() != LAS_OK || num_sms() <= 0) {
    free(s);
    return LAS_ERR_CUDA;
  }
  // projection split-K (autotunable): output n x op, K = the (L, p) rows of one chunk
  s->ks = split_balanced_ksplit(s, Lc);
  size_t total = 0;
  las_status rc = LAS_OK;
  auto A = [&](void** p, size_t b) {
    if (rc != LAS_OK) return;
    if (cudaMalloc(p, b) != cudaSuccess) {
      *p = nullptr;
      rc = LAS_ERR_CUDA;
      las_record_cuda_error(cudaErrorMemoryAllocation, "cudaMalloc(split)", __FILE__, __LINE__);
      return;
    }
    total += b;
  };
  const long R = (long)Lc * op;
  void* q = nullptr;
  s->packed = packed != 0;
  BPacked& bp = s->Bpk;
  bp = bpacked_geometry(n, X);
  if (!s->packed) {
    A(&q, planes_bytes((long)X * n, n));
    s->Bdig = make_planes(q, (long)X * n, n);
    q = nullptr;
    A((void**)&s->Bexp, (size_t)X * n * 4);
  } else {
  if (bp.nb1 > 0) {
    A(&q, bpacked_tile_bytes(bp));
    bp.tiles.p = (__nv_bfloat16*)q;
    bp.tiles.R = bp.tiles.Rpad = 128;
    bp.tiles.nkb = 8L * X * bp.T;
    bp.tiles.K = bp.tiles.nkb * BK;
    bp.tiles.plane = bp.tiles.nkb * 128 * BK;
    q = nullptr;
  }
  if (bp.r > 0) {
    A(&q, planes_bytes((long)X * bp.rp, n));
    bp.rag = make_planes(q, (long)X * bp.rp, n);
    q = nullptr;
  }
  A((void**)&bp.exp, (size_t)X * 4);
  A((void**)&bp.mx, (size_t)X * 8);
  }
  A(&q, planes_bytes(op, n));        s->Cdig = make_planes(q, op, n);   q = nullptr;
  A((void**)&s->Cexp, (size_t)op * 4);
  A(&q, planes_bytes(R, n));         s->Hdig = make_planes(q, R, n);    q = nullptr;
  A((void**)&s->Hexp, (size_t)R * 4);
  A(&q, planes_bytes(n, R));         s->HdigT = make_planes(q, n, R);   q = nullptr;
  A(&q, planes_bytes(op, R));        s->Wdig = make_planes(q, op, R);   q = nullptr;
  A((void**)&s->Wexp, (size_t)op * 4);
  A((void**)&s->part, split_part_elems(n, op) * 8);
  A((void**)&s->mx, (size_t)(op + n) * 8);
  A(&q, planes_bytes(n, n));         s->hdig = make_planes(q, n, n);    q = nullptr;
  A((void**)&s->hexp, (size_t)n * 4);
  // rows mu >= n of the transposed planes and the padding rows of C, W and h are never written by the
  // per-evaluation slicers: make them zero once
  const struct { void* p; size_t b; } zero[] = {
      {s->HdigT.p, planes_bytes(n, R)}, {s->Wdig.p, planes_bytes(op, R)},
      {s->Cdig.p, planes_bytes(op, n)}, {s->hdig.p, planes_bytes(n, n)}};
  for (const auto& z : zero) {
    if (rc != LAS_OK) break;
    cudaError_t e = cudaMemsetAsync(z.p, 0, z.b, st);
    if (e != cudaSuccess) {
      las_record_cuda_error(e, "cudaMemsetAsync(split planes)", __FILE__, __LINE__);
      rc = LAS_ERR_CUDA;
    }
  }
  if (rc == LAS_OK && !s->packed) {
    // one-time digit planes of the Cholesky vectors: rows (L, mu), K = nu
    RowsPacked acc{Bp, (long)n * (n + 1) / 2, n};
    rc = slice_rows(acc, s->Bdig, s->Bexp, st);
  } else if (rc == LAS_OK) {
    // one-time packed-triangle digit planes of the Cholesky vectors, one exponent per L
    const long npair = (long)n * (n + 1) / 2;
    k_bpacked_max<<<(unsigned)X, 256, 0, st>>>(Bp, npair, bp.mx, bp.exp);
    las_count_launch();
    if (bp.nb1 > 0) {
      const long total = 8L * X * bp.T * 128 * BK;
      k_bpacked_tiles<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(Bp, npair, bp.T, bp.exp,
                                                                        bp.tiles, total);
      las_count_launch();
    }
    if (bp.r > 0) {
      const long total = bp.rag.Rpad * bp.rag.nkb * BK;
      k_bpacked_ragged<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(
          Bp, npair, n, bp.n1, bp.r, bp.rp, bp.exp, bp.rag, (long)X * bp.rp);
      las_count_launch();
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
      las_record_cuda_error(e, "packed digit planes of B", __FILE__, __LINE__);
      rc = LAS_ERR_CUDA;
    }
  }
  if (rc != LAS_OK) {
    split_free(s);
    free(s);
    return rc;
  }
  *bytes += total;
  *out = s;
  return LAS_OK;
}

void split_destroy(SplitState* s) {
  if (!s) return;
  split_free(s);
  free(s);
}

const int* split_hexp(SplitState* s) { return s->Hexp; }

int split_get_ksplit(SplitState* s) { return s->ks; }
int split_balanced_ksplit(SplitState* s, int nL) {
  const int bn = s->bn[SPLIT_PROJECT] ? s->bn[SPLIT_PROJECT] : pick_bn(s->op);
  return balanced_ksplit(ozaki_tiles(s->n, s->op, 0, bn),
                         ((long)nL * s->op + BK - 1) / BK,
                         std::min<long>(s->ksplit6, std::max(1L, ((long)nL * s->op) / KSPLIT_MIN)));
}
// The one-electron products are fewer tiles than SMs: the shorter tile ends first.
static int one_electron_bn(const SplitState* s) {
  return s->bn[SPLIT_ONE_ELECTRON] ? s->bn[SPLIT_ONE_ELECTRON] : s->op <= 48 ? 48 : 64;
}

// K splits of a projection over R rows (L, p): at most s->ks of at least KSPLIT_MIN each, counted
// as ozaki_setup forms them (equal numbers of K blocks, none empty), so that every partial summed
// afterwards has been written.
static int project_ksplit(const SplitState* s, long R) {
  const long kb = (R + BK - 1) / BK, ks = std::max(1L, std::min((long)s->ks, R / KSPLIT_MIN));
  const long per = (kb + ks - 1) / ks;
  return (int)((kb + per - 1) / per);
}
int split_get_tile(SplitState* s, int kind) { return s->bn[kind]; }
las_status split_set_tile(SplitState* s, int kind, int bn) {
  if (kind < 0 || kind >= SPLIT_NKIND || (bn != 0 && bn != 64 && bn != 96)) return LAS_ERR_ARG;
  s->bn[kind] = bn;
  return LAS_OK;
}
void split_set_ksplit(SplitState* s, int ks) { s->ks = std::max(1, std::min(ks, s->ksplit6)); }

// The half-transform-shaped products of the Cholesky vectors, in either digit layout:
// out[L][p][mu] (ht_op columns per L) = sum_nu b^L(mu, nu) X(nu, p) for L in [l0, l0 + nL), X
// given by the digit planes of its transpose (rows p from x_row0, K = nu; exponents xexp).
static las_status b_half(const SplitState* s, int l0, int nL, const Planes& Xd, long x_row0,
                         const int* xexp, long N, double* out, int ht_op, cudaStream_t st,
                         int bn) {
  if (s->packed)
    return bpacked_half(s->Bpk, l0, nL, Xd, x_row0, xexp, N, out, ht_op, s->status, st, bn);
  return ozaki_gemm(s->Bdig, (long)l0 * s->n, s->Bexp + (long)l0 * s->n, (long)nL * s->n, Xd,
                    x_row0, xexp, N, s->n, 1, 1, out, 0, 0, s->n, ht_op, s->status, st, 0, bn);
}

// The same with the widths of its column tiles chosen here.  The columns beyond the last whole
// 96-column tile may form a second product of a narrower tile (150 columns as 96 + 54: 160 computed
// instead of 192); not while products are recorded for a grouped launch, which would then hold
// more of them.  bn: 0 = by stage times, or the width asked for.
static las_status b_half_cols(const SplitState* s, int l0, int nL, const Planes& Xd,
                              const int* xexp, long N, double* out, int ht_op, cudaStream_t st,
                              int bn) {
  const long whole = N / 96 * 96, rest = N - whole;
  const bool ends = whole > 0 && rest > 0 && rest <= 64 && !g_record;   // 96s and a narrower one
  int last = 64;
  bool two = bn == 96 && ends;
  if (bn == 0) {
    bn = pick_bn(N);
    last = pick_bn(rest);
    // a second launch reads B once more: it has to save a twentieth
    two = ends && (cols_time(whole, 96) + stage_time(last)) * 20 < cols_time(N, bn) * 19;
  }
  if (two) {
    las_status rc = b_half(s, l0, nL, Xd, 0, xexp, whole, out, ht_op, st, 96);
    if (rc != LAS_OK) return rc;
    return b_half(s, l0, nL, Xd, whole, xexp + whole, rest, out + whole * s->n, ht_op, st, last);
  }
  return b_half(s, l0, nL, Xd, 0, xexp, N, out, ht_op, st, bn);
}

las_status split_prepare_C(SplitState* s, const double* Cocc, cudaStream_t st) {
  // rows p of C_occ^T (K = nu): element (p, nu) = Cocc[nu*op + p]
  return slice_cols(RowsStrided{Cocc, 1, s->op}, s->Cdig, s->Cexp, st, true);
}

// ------------------------------------------------------------------------------------------
// Tangent of the evaluation along dC (the orbital Hessian-vector product): the same products
// with dC_occ in place of C_occ where the chain rule puts it
// ------------------------------------------------------------------------------------------
las_status split_tangent_prepare(SplitState* s, const double* dCocc, cudaStream_t st,
                                 size_t* bytes) {
  if (!s->tblob) {
    const long R = (long)s->Lc * s->op;
    const size_t b0 = rup(planes_bytes(s->op, s->n), 256), b1 = rup((size_t)s->op * 4, 256);
    const size_t b2 = rup(planes_bytes(R, s->n), 256), b3 = rup((size_t)R * 4, 256);
    if (cudaMalloc(&s->tblob, b0 + b1 + b2 + b3) != cudaSuccess) {
      s->tblob = nullptr;
      las_record_cuda_error(cudaErrorMemoryAllocation, "cudaMalloc(tangent)", __FILE__, __LINE__);
      return LAS_ERR_CUDA;
    }
    // padding rows are never written by the slicers: zero once
    cudaError_t e = cudaMemsetAsync(s->tblob, 0, b0 + b1 + b2 + b3, st);
    if (e != cudaSuccess) {
      las_record_cuda_error(e, "cudaMemsetAsync(tangent)", __FILE__, __LINE__);
      return LAS_ERR_CUDA;
    }
    uint8_t* w = (uint8_t*)s->tblob;
    s->dCdig = make_planes(w, s->op, s->n);
    s->dCexp = (int*)(w + b0);
    s->dHdig = make_planes(w + b0 + b1, R, s->n);
    s->dHexp = (int*)(w + b0 + b1 + b2);
    *bytes += b0 + b1 + b2 + b3;
  }
  return slice_cols(RowsStrided{dCocc, 1, s->op}, s->dCdig, s->dCexp, st, true);
}

// dH = b^L dC_occ for the chunk's aux rows (Ht layout [nL][op][n])
las_status split_tangent_half(SplitState* s, int l0, int nL, double* dHt, cudaStream_t st) {
  return b_half_cols(s, l0, nL, s->dCdig, s->dCexp, s->op, dHt, s->op, st, s->bn[SPLIT_HALF]);
}

// After split_full of the chunk: X[(L,p)][q] = sum_mu H_L(mu,p) dC(mu,q) (so that dT_L = X_L +
// X_L^T), and the digits of dH (rows (L,p), K = mu) with their row exponents.
las_status split_tangent_full(SplitState* s, int nL, const double* dHt, double* X,
                              cudaStream_t st) {
  const long R = (long)nL * s->op;
  las_status rc = ozaki_gemm(s->Hdig, 0, s->Hexp, R, s->dCdig, 0, s->dCexp, s->op, s->n, 1, 0, X,
                             s->op, 0, 0, 0, s->status, st, 0, s->bn[SPLIT_FULL]);
  if (rc != LAS_OK) return rc;
  Planes dH = s->dHdig;
  dH.R = R;
  return slice_contig(RowsContig{dHt, s->n}, dH, s->dHexp, st, true);
}

const int* split_tangent_dhexp(SplitState* s) { return s->dHexp; }

// Out (+)= sum_{(L,p)} A(mu,(L,p)) W((L,p),q): A = H (which = 0) or dH (which = 1), read
// MN-major from its digit planes; Wt[q][(L,p)] holds W scaled by that operand's row exponents.
las_status split_tangent_project(SplitState* s, int nL, int which, const double* Wt, double* Out,
                                 int accumulate, cudaStream_t st) {
  const long R = (long)nL * s->op;
  Planes W = s->Wdig;
  W.K = R;
  las_status rc = slice_long(RowsContig{Wt, R}, W, s->Wexp, s->mx, st);
  if (rc != LAS_OK) return rc;
  const int ks = project_ksplit(s, R);
  rc = ozaki_gemm(which ? s->dHdig : s->Hdig, 0, nullptr, s->n, W, 0, s->Wexp, s->op, R, ks, 0,
                  s->part, s->op, (long)s->n * s->op, 0, 0, s->status, st, 0,
                  s->bn[SPLIT_PROJECT], 1);
  if (rc != LAS_OK) return rc;
  launch_reduce_partials(s->part, ks, (long)s->n * s->op, Out, accumulate, st);
  return LAS_OK;
}

// hdC = h dC_occ (the digits of h from split_one_electron_hc of the same h)
las_status split_tangent_one_electron(SplitState* s, double* hdC, cudaStream_t st) {
  return ozaki_gemm(s->hdig, 0, s->hexp, s->n, s->dCdig, 0, s->dCexp, s->op, s->n, 1, 0, hdC,
                    s->op, 0, 0, 0, s->status, st, 0, one_electron_bn(s));
}

las_status split_lpu(SplitState* s, int nL, const double* Ht, int a, const double* C, int nmo,
                     int p0, int np, double* Lpu, cudaStream_t st, size_t* bytes) {
  // Lpu[L][p][u] = sum_mu C[mu][p0+p] Ht[L][u][mu]: rows (L,u) of the half transform times the
  // rows p of C[:, p0:p1]^T, written in the (L, p, u) layout by the half-transform epilogue mode
  const int n = s->n;
  if (a < 1 || np < 1) return LAS_OK;
  if (np > nmo) return LAS_ERR_INTERNAL;
  if (!s->Mpblob) {   // planes for all nmo rows of C^T: allocated once per context
    const size_t pb = planes_bytes(nmo, n), eb = rup((size_t)nmo * 4, 256);
    if (cudaMalloc(&s->Mpblob, rup(pb, 256) + eb) != cudaSuccess) {
      s->Mpblob = nullptr;
      las_record_cuda_error(cudaErrorMemoryAllocation, "cudaMalloc(lpu)", __FILE__, __LINE__);
      return LAS_ERR_CUDA;
    }
    *bytes += rup(pb, 256) + eb;
    cudaError_t e = cudaMemsetAsync(s->Mpblob, 0, rup(pb, 256) + eb, st);
    if (e != cudaSuccess) {
      las_record_cuda_error(e, "cudaMemsetAsync(lpu)", __FILE__, __LINE__);
      return LAS_ERR_CUDA;
    }
    s->Mpd = make_planes(s->Mpblob, nmo, n);
    s->Mpexp = (int*)((uint8_t*)s->Mpblob + rup(pb, 256));
  }
  Planes Mp = s->Mpd;
  Mp.R = np;
  las_status rc = slice_cols(RowsStrided{C + p0, 1, nmo}, Mp, s->Mpexp, st, true);
  // the active rows (L,u) of this chunk, sliced into the H digit planes (capacity Lc*op rows)
  Planes Hd = s->Hdig;
  Hd.R = (long)nL * a;
  if (rc == LAS_OK) rc = slice_contig(RowsContig{Ht, n}, Hd, s->Hexp, st, true);
  if (rc == LAS_OK)
    rc = ozaki_gemm(Hd, 0, s->Hexp, (long)nL * a, Mp, 0, s->Mpexp, np, n, 1, 1, Lpu, 0, 0, a, np,
                    s->status, st);
  return rc;
}

las_status split_half(SplitState* s, int l0, int nL, int oc, double* Ht, cudaStream_t st) {
  if (oc < 1 || oc > s->op) return LAS_ERR_INTERNAL;
  return b_half_cols(s, l0, nL, s->Cdig, s->Cexp, oc, Ht, oc, st, s->bn[SPLIT_HALF]);
}

las_status split_full(SplitState* s, int nL, const double* Ht, double* T, cudaStream_t st) {
  const long R = (long)nL * s->op;
  Planes Hd = s->Hdig;
  Hd.R = R;
  las_status rc = slice_contig(RowsContig{Ht, s->n}, Hd, s->Hexp, st, true);
  if (rc != LAS_OK) return rc;
  return ozaki_gemm(s->Hdig, 0, s->Hexp, R, s->Cdig, 0, s->Cexp, s->op, s->n, 1, 0, T, s->op, 0,
                    0, 0, s->status, st, 0, s->bn[SPLIT_FULL]);
}

las_status split_project_gemm(SplitState* s, int nL, const double* Wt, int* ks_used,
                              cudaStream_t st) {
  const long R = (long)nL * s->op;      // K of the projection: (L, p); a multiple of 16
  // A: the digit planes of H written by split_full (rows (L,p), K = mu), read MN-major: rows mu,
  // K = (L,p); their per-(L,p) exponents are folded into W.
  // W rows q (K = (L,p)), already scaled by 2^Hexp[(L,p)] and stored transposed: Wt[q][R]
  Planes W = s->Wdig;
  W.K = R;
  las_status rc = slice_long(RowsContig{Wt, R}, W, s->Wexp, s->mx, st);
  if (rc != LAS_OK) return rc;
  const int ks = project_ksplit(s, R);
  *ks_used = ks;
  return ozaki_gemm(s->Hdig, 0, nullptr, s->n, W, 0, s->Wexp, s->op, R, ks, 0, s->part, s->op,
                    (long)s->n * s->op, 0, 0, s->status, st, 0, s->bn[SPLIT_PROJECT], 1);
}

void split_project_reduce(SplitState* s, int ks, double* Out, int accumulate, cudaStream_t st) {
  launch_reduce_partials(s->part, ks, (long)s->n * s->op, Out, accumulate, st);
}

las_status split_project(SplitState* s, int nL, const double* Wt, double* Out, int accumulate,
                         cudaStream_t st) {
  int ks = 1;
  las_status rc = split_project_gemm(s, nL, Wt, &ks, st);
  if (rc != LAS_OK) return rc;
  split_project_reduce(s, ks, Out, accumulate, st);
  return LAS_OK;
}

las_status split_exchange_max(SplitState* s, unsigned long long** mx, cudaStream_t st) {
  LAS_CUDA_TRY(cudaMemsetAsync(s->mx, 0, s->n * sizeof(unsigned long long), st));
  *mx = s->mx;
  return LAS_OK;
}

las_status split_exchange(SplitState* s, int nL, int oc, const double* Ht, double* K, int accumulate,
                          double sgn, cudaStream_t st) {
  // K(mu,nu) (+)= sum_{(L,p)} Ht[(L,p)][mu] Ht[(L,p)][nu]: rows mu of H^T, scaled per row over
  // the long index (L,p), serve as both operands
  const long R = (long)nL * oc, n = s->n;
  if (oc < 1 || oc > s->op) return LAS_ERR_INTERNAL;
  Planes HT = s->HdigT;
  HT.K = R;
  las_status rc = slice_transposed(Ht, HT, s->hexp, s->mx, true, st);
  if (rc != LAS_OK) return rc;
  // Partials live in the projection's partial buffer (room rows of n doubles).  Only tiles that touch
  // the lower triangle are computed; the caller mirrors the result.  When the rows past the last
  // whole 128-row tile are few, their row tile is mostly padding: they then go as the columns of a
  // second product instead, stored transposed, if that ends sooner (800 orbitals: 30 row-column
  // tiles and 7 narrow ones instead of 39).
  const long kb = (R + BK - 1) / BK, n1 = n / BM * BM, r = n - n1,
             room = (long)(split_part_elems(s->n, s->op) / n);
  auto rounds = [&](long tiles, long ks) {
    return (tiles * ks + num_sms() - 1) / num_sms() * ((kb + ks - 1) / ks + CHUNK);
  };
  auto cap = [&](long rows) { return std::max(1L, std::min(rows, R / KSPLIT_MIN)); };
  long n0 = n, tiles = ozaki_tiles(n, n, 1);
  int ks = balanced_ksplit(tiles, kb, cap(room / n)), ksr = 0;
  if (n1 > 0 && r > 0) {
    const int bn = pick_bn(r);
    const long t1 = ozaki_tiles(n1, n1, 1), t2 = ozaki_tiles(n, r, 0, bn);
    const int k2 = balanced_ksplit(t2, kb, cap(std::min(64L, room / 4 / r)));
    // no fewer splits than the one product has: the tail's FP32 sums run over a split's K
    const int k1 = balanced_ksplit(t1, kb, cap((room - k2 * r) / n1), ks);
    if (k2 >= ks && k2 * r + k1 * n1 <= room && (kb + k1 - 1) / k1 * (k1 - 1) < kb &&
        (kb + k2 - 1) / k2 * (k2 - 1) < kb &&
        rounds(t1, k1) * stage_time(OZ_BN) + rounds(t2, k2) * stage_time(bn) <
            rounds(tiles, ks) * stage_time(OZ_BN)) {
      n0 = n1;
      ks = k1;
      ksr = k2;
    }
  }
  if (ks * n0 + ksr * r > room) return LAS_ERR_INTERNAL;
  rc = ozaki_gemm(HT, 0, s->hexp, n0, HT, 0, s->hexp, n0, R, ks, 0, s->part, n, n0 * n, 0, 0,
                  s->status, st, 1, OZ_BN);
  if (rc != LAS_OK) return rc;
  launch_reduce_partials(s->part, ks, n0 * n, K, accumulate, st, 0, 0, sgn);
  if (ksr > 0) {
    // rows n1.. of K: element (n1 + c, mu) = sum over (mu, c) of the product, written along mu
    double* part = s->part + (size_t)ks * n1 * n;
    rc = ozaki_gemm(HT, 0, s->hexp, n, HT, n1, s->hexp + n1, r, R, ksr, 1, part, 0, r * n, (int)n,
                    (int)r, s->status, st);
    if (rc != LAS_OK) return rc;
    launch_reduce_partials(part, ksr, r * n, K + n1 * n, accumulate, st, 0, 0, sgn);
  }
  return LAS_OK;
}

las_status split_one_electron_hc(SplitState* s, const double* h, double* hC, cudaStream_t st) {
  // hC = h C_occ  (rows mu of h, columns p of C_occ: the digits of C_occ are already sliced)
  las_status rc = slice_contig(RowsContig{h, s->n}, s->hdig, s->hexp, st, true);
  if (rc == LAS_OK)
    rc = ozaki_gemm(s->hdig, 0, s->hexp, s->n, s->Cdig, 0, s->Cexp, s->op, s->n, 1, 0, hC, s->op,
                    0, 0, 0, s->status, st, 0, one_electron_bn(s));
  return rc;
}

// ------------------------------------------------------------------------------------------
// Standalone emulated-FP64 GEMM through the same kernels (C ABI)
// ------------------------------------------------------------------------------------------
static size_t sgemm_ws(long M, long N, long K) {
  return rup(planes_bytes(M, K), 256) + rup(planes_bytes(N, K), 256) + rup(M * 4, 256) +
         rup(N * 4, 256) + 256;
}

// K splits of the product: few tiles leave SMs idle, and a split costs the sum of its partials: 6 K
// blocks' time at 2999 x 1201 x 187 (48 tiles in 3 parts), taken for all sizes, although the sum grows
// with M N ks.  (us without and with the split: 116 and 81 at 3000 x 1500 x 96, 127 and 56 at 40 x 2000
// x 96, 104 and 84 at 2999 x 1201 x 187, 177 and 107 at 2000 x 3000 x 64.)
static int sgemm_ksplit(long M, long N, long K, size_t room) {
  const long tiles = ozaki_tiles(M, N, 0, pick_bn(N)), kb = planes_nkb(K), sms = num_sms();
  const long cap = std::min<long>({16, kb / 4, (long)(room / ((size_t)M * N * 8))});
  int best = 1;
  long best_t = (tiles + sms - 1) / sms * (kb + CHUNK);
  for (long ks = 2; ks <= cap; ++ks) {
    const long per = (kb + ks - 1) / ks;
    const long t = (tiles * ks + sms - 1) / sms * (per + CHUNK) + 6;
    if (t < best_t && (kb + per - 1) / per == ks) {
      best_t = t;
      best = (int)ks;
    }
  }
  return best;
}

extern "C" size_t las_split_gemm_workspace(long M, long N, long K) {
  if (M <= 0 || N <= 0 || K <= 0) return 0;
  const int ks = sgemm_ksplit(M, N, K, ~(size_t)0 >> 1);
  return sgemm_ws(M, N, K) + (ks > 1 ? (size_t)ks * M * N * 8 : 0);
}

extern "C" las_status las_split_gemm(long M, long N, long K, const double* A, long lda,
                                     const double* B, long ldb, double* C, long ldc,
                                     void* workspace, size_t workspace_bytes, void* stream) {
  if (M < 0 || N < 0 || K < 0) return LAS_ERR_ARG;
  if (M == 0 || N == 0) return LAS_OK;
  if (!A || !B || !C) return LAS_ERR_ARG;
  if (lda < K || ldb < N || ldc < N) return LAS_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (K == 0) {
    for (long r = 0; r < M; ++r)
      LAS_CUDA_TRY(cudaMemsetAsync(C + r * ldc, 0, N * 8, st));
    return LAS_OK;
  }
  if (!workspace) return LAS_ERR_ARG;
  if (workspace_bytes < sgemm_ws(M, N, K) || ((uintptr_t)workspace & 255)) return LAS_ERR_WORKSPACE;
  uint8_t* w = (uint8_t*)workspace;
  Planes Ad = make_planes(w, M, K);
  w += rup(planes_bytes(M, K), 256);
  Planes Bd = make_planes(w, N, K);
  w += rup(planes_bytes(N, K), 256);
  int* ea = (int*)w;
  w += rup(M * 4, 256);
  int* eb = (int*)w;
  w += rup(N * 4, 256);
  int* status = (int*)w;
  w += 256;
  las_status rc = ozaki_prepare();
  if (rc != LAS_OK) return rc;
  ChainScope chain(st);
  // the planes' padding rows stay unwritten: they only feed rows and columns that are not stored
  const RowsContig ra{A, lda};
  const RowsStrided rb{B, 1, ldb};
  if (slice_fits(Ad.nkb)) {
    const long S = Ad.nkb * BK + 2;
    const int lg = slice_lg(S, M), ncols = (int)((N + 15) / 16);
    launch_chained(k_slice_operands, (unsigned)(ncols + ((M + (1 << lg) - 1) >> lg)), 256,
                   (size_t)(S * 8) << lg, st, ra, (int)ra.aligned(), Ad, Ad.nkb, lg, (int)S, ea, rb,
                   Bd, eb, ncols, status);
    rc = slice_done("k_slice_operands launch");
  } else {
    LAS_CUDA_TRY(cudaMemsetAsync(status, 0, 4, st));
    rc = slice_rows(ra, Ad, ea, st, true);
    if (rc == LAS_OK) rc = slice_cols(rb, Bd, eb, st, true);
  }
  if (rc != LAS_OK) return rc;
  const int ks = sgemm_ksplit(M, N, K, workspace_bytes - sgemm_ws(M, N, K));
  double* part = (double*)w;
  if (ks == 1) {
    rc = ozaki_gemm(Ad, 0, ea, M, Bd, 0, eb, N, K, 1, 0, C, ldc, 0, 0, 0, status, st);
  } else {
    rc = ozaki_gemm(Ad, 0, ea, M, Bd, 0, eb, N, K, ks, 0, part, N, M * N, 0, 0, status, st);
    if (rc == LAS_OK) launch_reduce_partials(part, ks, M * N, C, 0, st, N, ldc);
  }
  if (rc != LAS_OK) return rc;
  int h = 0;
  LAS_CUDA_TRY(cudaMemcpyAsync(&h, status, 4, cudaMemcpyDeviceToHost, st));
  LAS_CUDA_TRY(cudaStreamSynchronize(st));
  return h ? (las_status)h : LAS_OK;
}

// ------------------------------------------------------------------------------------------
// Fragment-embedding AO2MO in split precision (Eqs. ao2mo_1, ao2mo_2, ppaa, papa)
// ------------------------------------------------------------------------------------------
namespace lasdf_split {
// Row (u, v) of the active block of T (rows (L, p), columns q), K = the auxiliary row L:
// T[L][a0+u][a0+v]
struct RowsAA {
  const double* T;
  long n2;
  int nmo, a0, ma;
  __device__ __forceinline__ double operator()(long r, long k) const {
    const int u = (int)(r / ma), v = (int)(r - (long)u * ma);
    return T[k * n2 + (long)(a0 + u) * nmo + a0 + v];
  }
};
// Row (p, u) of the MO-active columns of T, K = L: T[L][p][a0+u]
struct RowsPA {
  const double* T;
  long n2;
  int nmo, a0, ma;
  __device__ __forceinline__ double operator()(long r, long k) const {
    const long p = r / ma, u = r - p * ma;
    return T[k * n2 + p * nmo + a0 + u];
  }
};
}  // namespace lasdf_split

struct FragSplit {
  int n, nmo, ma, Lc;
  Planes Mdig;   int* Mexp;     // rows p of M^T, K = e
  Planes Hd;     int* Hexp;     // rows (L, p) of the half transform, K = e
  Planes Tpl;    int* Texp;     // rows (p, q) of T, K = L
  Planes Taa;    int* Taaexp;   // rows (u, v) of the active block, K = L
  Planes Tpa;    int* Tpaexp;   // rows (p, u), K = L
  unsigned long long* mx;       // [nmo^2] column maxima of T
  void* blob;
};

las_status frag_split_create(FragSplit** out, int n, int nmo, int ma, int Lc, cudaStream_t st,
                             size_t* bytes) {
  *out = nullptr;
  if (!encode_fn()) return LAS_ERR_UNSUPPORTED;
  if (ozaki_prepare() != LAS_OK) return LAS_ERR_CUDA;
  FragSplit* f = (FragSplit*)calloc(1, sizeof(FragSplit));
  if (!f) return LAS_ERR_INTERNAL;
  f->n = n;
  f->nmo = nmo;
  f->ma = ma;
  f->Lc = Lc;
  const long n2 = (long)nmo * nmo, R1 = (long)Lc * nmo;
  const size_t parts[] = {planes_bytes(nmo, n),             (size_t)nmo * 4,
                          planes_bytes(R1, n),              (size_t)R1 * 4,
                          planes_bytes(n2, Lc),             (size_t)n2 * 4,
                          planes_bytes((long)ma * ma, Lc),  (size_t)ma * ma * 4,
                          planes_bytes((long)nmo * ma, Lc), (size_t)nmo * ma * 4,
                          (size_t)n2 * 8};   // each part is rounded up to 256 bytes below
  size_t total = 0;
  for (size_t b : parts) total += rup(b, 256);
  if (cudaMalloc(&f->blob, total) != cudaSuccess) {
    las_record_cuda_error(cudaErrorMemoryAllocation, "cudaMalloc(frag ao2mo)", __FILE__, __LINE__);
    free(f);
    return LAS_ERR_CUDA;
  }
  // padding rows and K blocks are never written by the live-row slicers: zero them once
  cudaError_t e = cudaMemsetAsync(f->blob, 0, total, st);
  if (e != cudaSuccess) {
    las_record_cuda_error(e, "cudaMemsetAsync(frag ao2mo)", __FILE__, __LINE__);
    cudaFree(f->blob);
    free(f);
    return LAS_ERR_CUDA;
  }
  uint8_t* w = (uint8_t*)f->blob;
  auto take = [&](size_t b) { void* q = w; w += rup(b, 256); return q; };
  f->Mdig = make_planes(take(parts[0]), nmo, n);
  f->Mexp = (int*)take(parts[1]);
  f->Hd = make_planes(take(parts[2]), R1, n);
  f->Hexp = (int*)take(parts[3]);
  f->Tpl = make_planes(take(parts[4]), n2, Lc);
  f->Texp = (int*)take(parts[5]);
  f->Taa = make_planes(take(parts[6]), (long)ma * ma, Lc);
  f->Taaexp = (int*)take(parts[7]);
  f->Tpa = make_planes(take(parts[8]), (long)nmo * ma, Lc);
  f->Tpaexp = (int*)take(parts[9]);
  f->mx = (unsigned long long*)take(parts[10]);
  *bytes += total;
  *out = f;
  return LAS_OK;
}

void frag_split_destroy(FragSplit* f) {
  if (!f) return;
  if (f->blob) cudaFree(f->blob);
  free(f);
}

int frag_split_fits(const FragSplit* f, int n, int nmo, int ma, int Lc) {
  return f && f->n == n && f->nmo == nmo && f->ma >= ma && f->Lc >= Lc;
}

las_status frag_split_prepare_M(FragSplit* f, const double* M, cudaStream_t st) {
  // rows p of M^T (K = e): element (p, e) = M[e][p]
  return slice_cols(RowsStrided{M, 1, f->nmo}, f->Mdig, f->Mexp, st, true);
}

las_status frag_split_chunk(SplitState* s, FragSplit* f, int l0, int nL, double* H, double* T,
                            int a0, int ma, double* ppaa, double* papa, double* part,
                            long part_elems, int accumulate, cudaStream_t st) {
  const int n = f->n, nmo = f->nmo;
  const long n2 = (long)nmo * nmo, R1 = (long)nL * nmo;
  if (nL < 1 || nL > f->Lc || ma > f->ma) return LAS_ERR_INTERNAL;
  // Eq. ao2mo_1: H[L][p][e2] = sum_e1 b^L(e2, e1) M[e1][p]
  las_status rc = b_half_cols(s, l0, nL, f->Mdig, f->Mexp, nmo, H, nmo, st, 0);
  // Eq. ao2mo_2: T[L][p][q] = sum_e H[L][p][e] M[e][q]
  Planes Hd = f->Hd;
  Hd.R = R1;
  if (rc == LAS_OK) rc = slice_contig(RowsContig{H, n}, Hd, f->Hexp, st, true);
  if (rc == LAS_OK)
    rc = ozaki_gemm(Hd, 0, f->Hexp, R1, f->Mdig, 0, f->Mexp, nmo, n, 1, 0, T, nmo, 0, 0, 0,
                    s->status, st);
  if (rc != LAS_OK) return rc;
  const long kb = (nL + BK - 1) / BK;
  if (ppaa) {
    // Eq. ppaa: ppaa[(p,q)][(u,v)] (+)= sum_L T[L][(p,q)] T[L][a0+u][a0+v]
    Planes A = f->Tpl, B = f->Taa;
    A.K = nL;
    B.R = (long)ma * ma;
    B.K = nL;
    // rows (p,q) of T^T with per-row exponents
    rc = slice_transposed(T, A, f->Texp, f->mx, false, st);
    if (rc == LAS_OK)
      rc = slice_cols(RowsAA{T, n2, nmo, a0, ma}, B, f->Taaexp, st, true);
    const long out = n2 * ma * ma;
    const int ks = balanced_ksplit(ozaki_tiles(n2, (long)ma * ma, 0), kb,
                                   std::max(1L, std::min(kb, part_elems / out)));
    if (rc == LAS_OK)
      rc = ozaki_gemm(A, 0, f->Texp, n2, B, 0, f->Taaexp, (long)ma * ma, nL, ks, 0, part,
                      (long)ma * ma, out, 0, 0, s->status, st);
    if (rc != LAS_OK) return rc;
    launch_reduce_partials(part, ks, out, ppaa, accumulate, st);
  }
  if (papa) {
    // Eq. papa: papa[(p,u)][(q,v)] (+)= sum_L T[L][p][a0+u] T[L][q][a0+v] (lower triangle; the
    // caller mirrors it once all chunks are in)
    Planes A = f->Tpa;
    A.R = (long)nmo * ma;
    A.K = nL;
    rc = slice_cols(RowsPA{T, n2, nmo, a0, ma}, A, f->Tpaexp, st, true);
    const long m = (long)nmo * ma, out = m * m;
    const int ks = balanced_ksplit(ozaki_tiles(m, m, 1), kb,
                                   std::max(1L, std::min(kb, part_elems / out)));
    if (rc == LAS_OK)
      rc = ozaki_gemm(A, 0, f->Tpaexp, m, A, 0, f->Tpaexp, m, nL, ks, 0, part, m, out, 0, 0,
                      s->status, st, 1);
    if (rc != LAS_OK) return rc;
    launch_reduce_partials(part, ks, out, papa, accumulate, st);
  }
  return LAS_OK;
}

// ------------------------------------------------------------------------------------------
// Self-test of the bounded waits: one CTA waits on an mbarrier that nothing ever arrives on,
// with a short poll limit; the wait must give up, record LAS_ERR_TIMEOUT and let the kernel
// return, leaving the context usable.
// ------------------------------------------------------------------------------------------
namespace lasdf_split {
__global__ void k_selftest_wait(int* status, long limit) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    sm100::mbar_init(&bar, 1);
    abort_flag = 0;
    sm100::fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0)
    sm100::mbar_wait(&bar, 0, (volatile int*)&abort_flag, status, LAS_ERR_TIMEOUT, 0, limit);
  __syncthreads();
}
}  // namespace lasdf_split

extern "C" las_status las_selftest_bounded_wait(void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  int* status = nullptr;
  LAS_CUDA_TRY(cudaMalloc(&status, sizeof(int)));
  las_status rc = LAS_OK;
  cudaError_t e = cudaMemsetAsync(status, 0, sizeof(int), st);
  if (e == cudaSuccess) {
    k_selftest_wait<<<1, 32, 0, st>>>(status, 1L << 16);
    las_count_launch();
    e = cudaGetLastError();
  }
  int h = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, status, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    las_record_cuda_error(e, "bounded-wait self-test", __FILE__, __LINE__);
    rc = LAS_ERR_CUDA;
  } else {
    rc = (las_status)h;
  }
  cudaFree(status);
  return rc;
}

// ------------------------------------------------------------------------------------------
// Allocation-free variant of las_split_gemm
//
// Some callers cannot allocate device memory at the point where they need a product: plugins
// whose host application owns every device allocation through its own pool, and
// latency-critical loops where a cudaMalloc could synchronise the device. This entry point takes
// its scratch from a fixed array that is part of the library image instead of asking for a
// buffer: the digit planes and exponents of both operands live in `g_noalloc_scratch`, a
// LAS_NOALLOC_SCRATCH_BYTES (64 MiB) file-scope device array that every GPU which loads the
// library holds until the process exits.  Like las_split_gemm it waits for its stream and reads
// its status word back before returning.
// ------------------------------------------------------------------------------------------
#include <mutex>

static __device__ __align__(256) unsigned char g_noalloc_scratch[LAS_NOALLOC_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
void* g_noalloc_addr[kMaxDevices];  // device address of g_noalloc_scratch, per device ordinal
}  // namespace

extern "C" las_status las_split_gemm_noalloc(long M, long N, long K, const double* A, long lda,
                                             const double* B, long ldb, double* C, long ldc,
                                             void* stream) {
  if (M < 0 || N < 0 || K < 0) return LAS_ERR_ARG;
  if (M == 0 || N == 0) return LAS_OK;
  if (!A || !B || !C) return LAS_ERR_ARG;
  if (lda < K || ldb < N || ldc < N) return LAS_ERR_ARG;
  if (K > 0 && sgemm_ws(M, N, K) > (size_t)LAS_NOALLOC_SCRATCH_BYTES) return LAS_ERR_WORKSPACE;
  int dev = 0;
  LAS_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return LAS_ERR_UNSUPPORTED;
  void* scratch = nullptr;
  {
    // Set-up, once per device with that device current: in host code the array's name is only
    // a host-side stand-in, so its device address must be looked up.
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
      void* p = nullptr;
      LAS_CUDA_TRY(cudaGetSymbolAddress(&p, g_noalloc_scratch));
      g_noalloc_addr[dev] = p;
    }
    scratch = g_noalloc_addr[dev];
  }
  // The shared array keeps whatever the previous call left: las_split_gemm clears the status word it
  // keeps there, and writes every digit of the M rows and N columns.  The planes' padding rows stay
  // as they are; tiles read them, but only for rows and columns of the product that are not stored.
  return las_split_gemm(M, N, K, A, lda, B, ldb, C, ldc, scratch, LAS_NOALLOC_SCRATCH_BYTES,
                        stream);
}
