// Storage of the digit planes and the boxes in which a product reads them: index arithmetic only,
// without CUDA calls, so that it compiles for the host alone (the layout is checked there).
#pragma once
#include <stddef.h>
#include <string.h>

#ifdef __CUDACC__
#include <cuda_bf16.h>
#define LAS_HD __host__ __device__ __forceinline__
#else
struct __nv_bfloat16;
#define LAS_HD inline
#endif

namespace lasdf_split {

constexpr int NDIG = 6;
constexpr int BM = 128;          // rows per CTA tile (tcgen05 M)
constexpr int BK = 16;           // K per pipeline stage (one 32-byte swizzle row of BF16)

// Digit planes are stored K-blocked: the 16 values of K block k / BK of row r of plane s lie at
//   s*plane + (k / BK) * (Rpad * BK) + r * BK,   Rpad = R rounded up to ROWPAD,
// so that every pipeline stage of every tile is one contiguous block per plane, and the two
// 8-value halves of such a 32-byte row are swapped when bit 2 of r is set.  That is the image the
// MMA's 32-byte-swizzle operand has in shared memory (16-byte chunk index ^= address bit 7), so a
// stage is a plain copy: the tensor maps see rows of 256 elements (16 stored rows, 512 bytes) and
// do not swizzle.  The TMA unit works through a box row by row, about 1.4 clocks per row however
// short it is: loads of 32-byte rows with the swizzle done by the TMA took 1810 clocks per 42 KB
// stage on every SM, as long as the MMAs, and 512-byte rows take 760 (18 TB/s over the chip).  Row
// coordinates of a box are therefore multiples of ROWGRAN (box_skip).
// A tile box that reaches past Rpad reads the next K block's rows (finite digits) or, at the end
// of a plane, the TMA's zero fill: those rows only feed output rows or columns beyond M or N,
// which are never stored.
constexpr long ROWPAD = 384;
constexpr int ROWGRAN = 16;      // stored rows per 512-byte row of the tensor maps

struct Planes {
  __nv_bfloat16* p;
  long R, Rpad, K, nkb, plane;   // rows, padded rows, K, K blocks, elements per plane
  LAS_HD long idx(int s, long r, long k) const {
    return s * plane + (k / BK) * (Rpad * BK) + swz(r, (int)(k % BK));
  }
  // Position of value c (0..15) of row r inside a K block: the 8-value halves swap with bit 2 of r.
  static LAS_HD long swz(long r, int c) {
    return r * BK + (c ^ ((int)(r & 4) << 1));
  }
};

static inline long planes_rpad(long R) { return (R + ROWPAD - 1) / ROWPAD * ROWPAD; }
static inline long planes_nkb(long K) { return (K + BK - 1) / BK; }
static inline size_t planes_bytes(long R, long K) {
  return (size_t)NDIG * planes_rpad(R) * planes_nkb(K) * BK * 2;
}
static inline Planes make_planes(void* p, long R, long K) {
  Planes P;
  P.p = (__nv_bfloat16*)p;
  P.R = R;
  P.Rpad = planes_rpad(R);
  P.K = K;
  P.nkb = planes_nkb(K);
  P.plane = P.nkb * P.Rpad * BK;
  return P;
}

// The Cholesky vectors as digit planes in packed-triangle form.  The first n1 = 128 nb1 rows of
// every b^L lie in full 128-row blocks, of which only the lower tiles (I >= J) are stored (the
// diagonal tiles whole): T = nb1 (nb1 + 1) / 2 tiles per L, tile (I, J) of L at index
// L T + I (I + 1) / 2 + J, each as 8 K blocks of 128 rows x 16 (the Planes layout with 128 rows
// and 8 X T K blocks).  The half transform reads a tile as it is stored for the rows of block I
// and MN-major (transposed) for the rows of block J.  The r = n - n1 ragged rows mu >= n1 of each
// b^L are stored whole (rows (L, mu - n1), K = nu; when there are full blocks each L's rows are
// padded with zero rows to rp, a multiple of ROWGRAN, so that every L starts at a box coordinate);
// they are read as they are for their own rows and MN-major for the columns nu >= n1 of the full
// blocks.  One exponent per L (max |b^L| < 2^e(L)), so that a stored element has the same scale for
// both rows that use it.
struct BPacked {
  int n, X, nb1, T, r, rp, n1;
  Planes tiles;       // R = Rpad = 128, nkb = 8 X T
  Planes rag;         // rows (L, j), j < rp, of all X rp; K = n
  int* exp;           // [X]
  unsigned long long* mx;   // [X] max |b^L| as ordered bit patterns (set-up scratch)
};

static inline BPacked bpacked_geometry(int n, int X) {
  BPacked b;
  memset(&b, 0, sizeof(b));
  b.n = n;
  b.X = X;
  b.nb1 = n / 128;
  b.T = b.nb1 * (b.nb1 + 1) / 2;
  b.n1 = 128 * b.nb1;
  b.r = n - b.n1;
  b.rp = b.nb1 > 0 ? (b.r + ROWGRAN - 1) / ROWGRAN * ROWGRAN : b.r;
  return b;
}
static inline size_t bpacked_tile_bytes(const BPacked& b) {
  return (size_t)NDIG * 8 * (size_t)b.X * b.T * 128 * BK * 2;
}

// Boxes.  A K-major box of K block kb starts at row row0 + m0 of an operand (multiples of ROWGRAN):
// its row coordinate in the tensor map's 512-byte rows.
LAS_HD int box_row(int kb, int rpad, int row0, int m0) {
  return (int)(((long)kb * rpad + row0 + m0) / ROWGRAN);
}
// A product whose first row lies between two box rows starts that many rows early.
LAS_HD int box_skip(long row0) { return (int)(row0 % ROWGRAN); }

// Packed-triangle A, per row tile `mt` of a chunk from L0 on: its row block R of b^L, the K block of
// stored tile (R, 0), the index of stored tile (R, R) less R (R + 1) / 2, and the ragged row of K
// block 0, so that each stage adds its K block kb = 8 J + kk only.
struct PackedBoxes {
  int R;
  long row, col, rag;
  // row coordinate of K block kb of the stored lower tiles (R, J), J <= R (K-major)
  LAS_HD int lower(int kb) const { return (int)((row + kb) * (BM / ROWGRAN)); }
  // K-block coordinate of the stored tile (J, R), R < J < nb1 (MN-major, row coordinate kb % 8)
  LAS_HD int mirror(int J) const { return (int)((col + J * (J + 1) / 2) * 8); }
  // row coordinate of the ragged rows nu = 16 kb.. (MN-major, K-block coordinate 8 R)
  LAS_HD int ragged(int kb) const { return (int)((rag + (long)kb * BK) / ROWGRAN); }
};
LAS_HD PackedBoxes packed_boxes(int L0, int mt, int nb1, int T, int rp) {
  PackedBoxes b;
  const int Lr = mt / nb1;
  const long L = (long)L0 + Lr;
  b.R = mt - Lr * nb1;
  b.row = (L * T + b.R * (b.R + 1) / 2) * 8;
  b.col = L * T + b.R;
  b.rag = L * rp - 8L * nb1 * BK;
  return b;
}

}  // namespace lasdf_split
