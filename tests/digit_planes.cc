// Host check of csrc/digit_planes.h: planes are filled through its storage functions, boxes are read
// at its coordinates as the tensor maps describe them (rows of 256 values, 16 stored rows; nothing
// swizzled), and every value that the MMA's 32-byte-swizzle operand takes from there is compared with
// the one that the product needs.  Prints "ok" and the number of values compared.
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>

#include <vector>

#include "digit_planes.h"

using namespace lasdf_split;

static long checked = 0;
static void fail(const char* what, long a, long b, long c) {
  printf("%s: %ld %ld %ld\n", what, a, b, c);
  exit(1);
}

// value of row r and column k of operand L: nothing else has this id
static int64_t id(long L, long r, long k) { return 1 + (L * 4096 + r) * 4096 + k; }

struct Image {   // one plane of ids
  Planes P;
  std::vector<int64_t> v;
  explicit Image(const Planes& p) : P(p), v((size_t)p.plane, 0) {}
  // 3D map: dims {256, nkb * Rpad / 16}, box {256, rows / 16} at row y
  std::vector<int64_t> box(long y, int rows) const {
    std::vector<int64_t> o((size_t)rows * BK, 0);
    for (long i = 0; i < (long)o.size(); ++i) {
      const long at = y * ROWGRAN * BK + i;
      if (y < 0) fail("box starts below zero", y, 0, 0);
      if (at < (long)v.size()) o[i] = v[at];
    }
    return o;
  }
  // 4D map: dims {256, Rpad / 16, nkb}, box {256, 1, BM / BK} at (y, z); outside it reads zero
  std::vector<int64_t> box_mn(long y, long z) const {
    std::vector<int64_t> o((size_t)BM * BK, 0);
    if (y < 0 || z < 0) fail("box starts below zero", y, z, 0);
    for (int b = 0; b < BM / BK; ++b)
      for (int i = 0; i < ROWGRAN * BK; ++i)
        if (y < P.Rpad / ROWGRAN && z + b < P.nkb)
          o[(size_t)b * ROWGRAN * BK + i] = v[(z + b) * P.Rpad * BK + y * ROWGRAN * BK + i];
    return o;
  }
};

// Byte address in a tile that starts at a multiple of 256 -> where the swizzled operand finds it: bit
// 4 (the 16-byte chunk) ^= bit 7.
static long swizzled(long byte) { return byte ^ ((byte >> 3) & 16); }
static int64_t k_major(const std::vector<int64_t>& t, int m, int k) {
  return t[swizzled(2L * (m * BK + k)) / 2];
}
// MN-major: atoms of 16 values of M by 16 of K, 512 bytes each
static int64_t mn_major(const std::vector<int64_t>& t, int m, int k) {
  return t[swizzled(512L * (m / 16) + 2L * (k * BK + m % 16)) / 2];
}
static void expect(const char* what, int64_t got, int64_t want, long a, long b, long c) {
  ++checked;
  if (got != want) fail(what, a, b, c);
}

// Rows [row0, row0 + M) of an R x K operand, K-major, and the same planes read MN-major
static void full_rows(long R, long K, long row0, long M) {
  Image A(make_planes(nullptr, R, K));
  for (long r = 0; r < R; ++r)
    for (long k = 0; k < K; ++k) A.v[A.P.idx(0, r, k)] = id(0, r, k);
  const int skip = box_skip(row0);
  const long start = row0 - skip;
  if (start % ROWGRAN || skip < 0 || skip >= ROWGRAN) fail("start", row0, skip, 0);
  for (long m0 = 0; m0 < M + skip; m0 += BM)
    for (int kb = 0; kb < A.P.nkb; ++kb) {
      const auto t = A.box(box_row(kb, (int)A.P.Rpad, (int)start, (int)m0), BM);
      for (int m = 0; m < BM; ++m)
        for (int k = 0; k < BK; ++k) {
          const long row = m0 + m - skip;            // row of the product
          if (row < 0 || row >= M) continue;         // computed, not stored
          const long kk = (long)kb * BK + k;
          expect("K-major", k_major(t, m, k), kk < K ? id(0, row0 + row, kk) : 0, row, kk, m0);
        }
    }
  // MN-major: the product's M is K here, and its K the rows
  for (long m0 = 0; m0 < K; m0 += BM)
    for (int kb = 0; kb < (R + BK - 1) / BK; ++kb) {
      const auto t = A.box_mn(kb, m0 / BK);
      for (int m = 0; m < BM && m0 + m < K; ++m)
        for (int k = 0; k < BK; ++k) {
          const long r = (long)kb * BK + k;
          expect("MN-major", mn_major(t, m, k), r < R ? id(0, r, m0 + m) : 0, m0 + m, r, 0);
        }
    }
}

// Every stage of the packed-triangle form of X symmetric n x n matrices, and its ragged rows
static void packed(int n, int X) {
  BPacked b = bpacked_geometry(n, X);
  auto sym = [](long L, long r, long c) { return r > c ? id(L, r, c) : id(L, c, r); };
  Planes tp;
  memset(&tp, 0, sizeof(tp));
  tp.R = tp.Rpad = BM;
  tp.nkb = 8L * X * b.T;
  tp.K = tp.nkb * BK;
  tp.plane = tp.nkb * BM * BK;
  if (bpacked_tile_bytes(b) != (size_t)NDIG * tp.plane * 2) fail("bytes", n, X, 0);
  Image tiles(tp), rag(make_planes(nullptr, (long)X * b.rp, n));
  for (long L = 0; L < X; ++L) {
    for (int I = 0; I < b.nb1; ++I)
      for (int J = 0; J <= I; ++J)
        for (int r = 0; r < BM; ++r)
          for (int c = 0; c < BM; ++c) {
            const long kb = (L * b.T + I * (I + 1) / 2 + J) * 8 + c / BK;
            tiles.v[tiles.P.idx(0, r, kb * BK + c % BK)] = sym(L, BM * I + r, BM * J + c);
          }
    for (int j = 0; j < b.r; ++j)
      for (int k = 0; k < n; ++k) rag.v[rag.P.idx(0, L * b.rp + j, k)] = sym(L, b.n1 + j, k);
  }
  const int kbs = (int)planes_nkb(n);
  for (int L0 = 0; L0 < X; L0 += 2)
    for (int mt = 0; mt < (X - L0) * b.nb1; ++mt) {
      const PackedBoxes pk = packed_boxes(L0, mt, b.nb1, b.T, b.rp);
      const long L = L0 + mt / b.nb1;
      for (int kb = 0; kb < kbs; ++kb) {
        const int J = kb >> 3;
        const bool mn = J > pk.R;
        const auto t = !mn ? tiles.box(pk.lower(kb), BM)
                       : J < b.nb1 ? tiles.box_mn(kb & 7, pk.mirror(J))
                                   : rag.box_mn(pk.ragged(kb), pk.R * (BM / BK));
        for (int m = 0; m < BM; ++m)
          for (int k = 0; k < BK; ++k) {
            const long row = (long)BM * pk.R + m, nu = (long)kb * BK + k;
            expect("packed", mn ? mn_major(t, m, k) : k_major(t, m, k), nu < n ? sym(L, row, nu) : 0,
                   row, nu, L);
          }
      }
    }
  if (b.nb1 > 0 && b.r > 0 && (b.rp % ROWGRAN || b.rp < b.r)) fail("rp", n, b.rp, b.r);
  // the ragged rows as rows (L, j) of their own product
  for (int L0 = 0; L0 < X; L0 += 2) {
    const long row0 = (long)L0 * b.rp, M = (X - L0) * (long)b.rp;
    const int skip = box_skip(row0);
    for (long m0 = 0; m0 < M + skip; m0 += BM)
      for (int kb = 0; kb < kbs; ++kb) {
        const auto t = rag.box(box_row(kb, (int)rag.P.Rpad, (int)(row0 - skip), (int)m0), BM);
        for (int m = 0; m < BM; ++m)
          for (int k = 0; k < BK; ++k) {
            const long row = m0 + m - skip, nu = (long)kb * BK + k;
            if (row < 0 || row >= M || row % b.rp >= b.r) continue;
            expect("ragged", k_major(t, m, k), nu < n ? sym(L0 + row / b.rp, b.n1 + row % b.rp, nu) : 0,
                   row, nu, L0);
          }
      }
  }
}

int main() {
  for (long n : {16L, 37L, 100L, 400L})
    for (long l0 : {0L, 7L, 12L}) full_rows(n * 13, n, l0 * n, (13 - l0) * n);
  full_rows(384, 17, 5, 379);
  full_rows(385, 33, 384, 1);
  for (int n : {16, 100, 127, 128, 129, 143, 144, 145, 256, 300, 383}) packed(n, 5);
  printf("ok %ld\n", checked);
  return 0;
}
