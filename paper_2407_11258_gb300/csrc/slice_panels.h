// Panels of a digit-plane product (gemm_slices.cu) in a bounded workspace: host arithmetic only.
#pragma once
#include <algorithm>
#include <cstddef>

namespace lnocc {

constexpr int kSliceChunk = 512;  // columns that share one exponent
constexpr int kDigits = 9;        // BF16 digit planes of an operand (and one plane of its magnitudes)
constexpr int kFarDigits = 12;    // the same for products of rows that decay away from centres far apart

// Device bytes of the planes and chunk exponents of `rows` rows of Kp columns.
inline size_t slice_bytes(long long rows, int Kp, int digits = kDigits) {
  const size_t planes = static_cast<size_t>(rows) * Kp * 2 * (digits + 1);
  const size_t ex = static_cast<size_t>(rows) * ((Kp + kSliceChunk - 1) / kSliceChunk) * 4;
  return (planes + 255) / 256 * 256 + (ex + 255) / 256 * 256;
}

// C = A B^T with M rows of A and N rows of B, Kp columns (a multiple of 64): panels of nb rows of B and mb rows
// of A, kw columns each, both cut into one workspace, B's planes first.
struct SlicePanels {
  int kw = 0, nb = 0, mb = 0;  // kw == 0: the workspace is too small
};

// Invariant: slice_bytes(nb, kw, digits) + slice_bytes(mb, kw, digits) <= room. The K panel is the whole of K unless even a few
// row tiles of it would not fit. B stays whole while it leaves a quarter of the workspace, and at least one row
// tile of A, to the other operand; otherwise it is cut into panels of about half of the workspace. Whole tiles:
// 128 rows of A, 64 of B.
inline SlicePanels plan_slice_panels(int M, int N, int Kp, size_t room, int digits = kDigits) {
  SlicePanels p;
  if (M < 1 || N < 1 || Kp < 1) return p;
  auto bytes = [&](int rows, int k) { return slice_bytes(rows, k, digits); };
  auto fits = [&](int m, int n, int k) { return bytes(m, k) + bytes(n, k) <= room; };
  const int m1 = std::min(M, 512), n1 = std::min(N, 256);
  if (!fits(m1, n1, std::min(Kp, 2 * kSliceChunk))) return p;
  int kw = Kp;
  while (kw > 2 * kSliceChunk && !fits(m1, n1, kw)) kw = (kw / 2 + kSliceChunk - 1) / kSliceChunk * kSliceChunk;
  const int m0 = std::min(M, 128);
  int nb = N;
  if (!fits(M, N, kw) && (bytes(N, kw) > room / 4 * 3 || !fits(m0, N, kw))) {
    nb = std::min(N, std::max(64, static_cast<int>(room / 2 / bytes(64, kw)) * 64));
    while (nb > 64 && !fits(m0, nb, kw)) nb = (nb - 1) / 64 * 64;
  }
  if (!fits(m0, nb, kw)) return p;
  int mb = M;
  if (!fits(M, nb, kw)) mb = std::max(m0, static_cast<int>((room - bytes(nb, kw)) / bytes(128, kw)) * 128);
  p.kw = kw;
  p.nb = nb;
  p.mb = mb;
  return p;
}

// f(k0, kw, n0, nn, m0, mm, first): one panel product after the other; `first` marks the first one of a B panel.
// sym (A == B): panels wholly below the diagonal are left out.
template <typename F>
inline void for_each_slice_panel(const SlicePanels& p, int M, int N, int Kp, bool sym, F&& f) {
  for (int k0 = 0; k0 < Kp; k0 += p.kw)
    for (int n0 = 0; n0 < N; n0 += p.nb) {
      const int nn = std::min(p.nb, N - n0);
      for (int m0 = 0; m0 < M; m0 += p.mb) {
        if (sym && n0 + nn <= m0) continue;
        f(k0, std::min(p.kw, Kp - k0), n0, nn, m0, std::min(p.mb, M - m0), m0 == 0);
      }
    }
}

}  // namespace lnocc
