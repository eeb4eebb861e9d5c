"""Panels of the FP64 digit-plane products (csrc/slice_panels.h): host arithmetic, compiled here and swept."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_11258_gb300", "csrc")

SRC = r"""
#include <cstdint>
#include <vector>
#include "slice_panels.h"
using namespace lnocc;
// -1: refused; 0: sound; 1: past the workspace; 2: a panel exceeds the operands or the plan; 3: an element of C and
// a K panel not covered exactly once; 4: a B panel is read before it is cut
extern "C" int check(int M, int N, int Kp, unsigned long long room, int sym, int digits) {
  const SlicePanels p = plan_slice_panels(M, N, Kp, room, digits);
  if (p.kw == 0) return -1;
  int bad = 0;
  long long area = 0, want = 0;
  std::vector<uint8_t> seen(static_cast<size_t>(M) * N <= 40000 ? static_cast<size_t>(M) * N : 0);
  const int kpanels = (Kp + p.kw - 1) / p.kw;
  int cut_k = -1, cut_n = -1;
  for_each_slice_panel(p, M, N, Kp, sym != 0, [&](int k0, int kw, int n0, int nn, int m0, int mm, bool first) {
    if (slice_bytes(nn, kw, digits) + slice_bytes(mm, kw, digits) > room) bad = bad ? bad : 1;
    if (kw < 1 || nn < 1 || mm < 1 || k0 + kw > Kp || n0 + nn > N || m0 + mm > M || nn > p.nb || mm > p.mb ||
        (k0 + kw < Kp && kw % kSliceChunk != 0) || k0 % kSliceChunk != 0)
      bad = bad ? bad : 2;
    if (first) cut_k = k0, cut_n = n0;
    if (cut_k != k0 || cut_n != n0) bad = bad ? bad : 4;
    area += static_cast<long long>(mm) * nn;
    if (!seen.empty())
      for (int m = m0; m < m0 + mm; ++m)
        for (int n = n0; n < n0 + nn; ++n) ++seen[static_cast<size_t>(m) * N + n];
  });
  if (!sym && area != static_cast<long long>(M) * N * kpanels) bad = bad ? bad : 3;
  for (size_t x = 0; x < seen.size(); ++x) {
    const int m = static_cast<int>(x / N), n = static_cast<int>(x % N);
    if (seen[x] > kpanels || (seen[x] < kpanels && !(sym && n < m))) bad = bad ? bad : 3;
  }
  return bad;
}
extern "C" int sweep(const int* Ms, int nm, const int* Ns, int nn, const int* Ks, int nk, unsigned long long room, int sym,
                     int* at) {
  int plans = 0;
  for (int a = 0; a < nm; ++a)
    for (int b = 0; b < nn; ++b)
      for (int c = 0; c < nk; ++c) {
        if (sym && Ms[a] != Ns[b]) continue;
        for (int digits : {kDigits, kFarDigits}) {
          const int r = check(Ms[a], Ns[b], Ks[c], room, sym, digits);
          if (r > 0) { at[0] = Ms[a], at[1] = Ns[b], at[2] = Ks[c], at[3] = r; return -1; }
          plans += r == 0;
        }
      }
  return plans;
}
"""


@pytest.fixture(scope="module")
def planner(tmp_path_factory):
    d = tmp_path_factory.mktemp("panels")
    src, lib = d / "panels.cpp", d / "panels.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, str(src), "-o", str(lib)], check=True)
    return ctypes.CDLL(str(lib))


def sweep(planner, Ms, Ns, Ks, room, sym=0):
    arr = [(ctypes.c_int * len(x))(*x) for x in (Ms, Ns, Ks)]
    at = (ctypes.c_int * 4)()
    n = planner.sweep(arr[0], len(Ms), arr[1], len(Ns), arr[2], len(Ks), ctypes.c_ulonglong(room), sym, at)
    assert n >= 0, f"M, N, Kp = {list(at)[:3]}, room {room}: fault {at[3]}"
    return n


CAP = 256 << 20  # the largest workspace of a handle


def test_panels_stay_inside_the_largest_workspace(planner):
    """Few rows of A, a few hundred of B and a long K: B takes most of the workspace."""
    Ms = list(range(80, 260)) + [1, 16, 64, 511, 512, 513, 900]
    Ns = list(range(240, 400, 3)) + [1, 64, 255, 256, 257, 900, 4000]
    Ks = [k // 64 * 64 for k in (20000, 30000, 33700, 35000, 38000, 40000, 42048, 44000, 47040, 52000, 70016, 200000)]
    assert sweep(planner, Ms, Ns, Ks, CAP) > 0
    for M, N, K in [(100, 260, 47040), (130, 290, 42048), (144, 300, 40000), (92, 260, 95680), (120, 300, 162048)]:
        assert planner.check(M, N, K, ctypes.c_ulonglong(CAP), 0, 9) == 0


def test_panels_stay_inside_any_workspace(planner):
    sizes = [1, 3, 63, 64, 65, 127, 128, 129, 130, 191, 256, 257, 300, 384, 511, 512, 513, 640, 1500]
    Ks = [64, 128, 512, 576, 1024, 1088, 2048, 4160]
    plans = 0
    for room in [1 << s for s in range(14, 29)] + [3 << s for s in range(14, 26)] + [5000000, 12345678]:
        plans += sweep(planner, sizes, sizes, Ks, room)
        plans += sweep(planner, sizes, sizes, Ks, room, sym=1)
    assert plans > 5000


def test_panels_cover_small_products_once(planner):
    sizes = [1, 64, 65, 100, 128, 129, 180, 200]
    for room in (3 << 20, 5 << 20, 7 << 20, 9 << 20):
        sweep(planner, sizes, sizes, [64, 512, 1088, 1600, 3072], room)
        sweep(planner, sizes, sizes, [64, 512, 1088, 1600, 3072], room, sym=1)


def test_workspace_that_cannot_hold_two_panels_is_refused(planner):
    for M, N, K in [(512, 256, 1024), (4000, 4000, 8192)]:
        assert planner.check(M, N, K, ctypes.c_ulonglong(1 << 20), 0, 9) == -1

