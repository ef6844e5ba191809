"""The split of a launch's items among its processing elements (at_items.cuh,
plain arithmetic): every item has one owner, the elements' runs differ by one
item at most, and with fewer items than elements so do the CTAs' counts, the
first element of a CTA before its others."""
import subprocess

from test_abi import ROOT

_SRC = r"""
#include <cstdio>
#include <initializer_list>
#include <vector>
#include "at_items.cuh"
int main() {
  const long long counts[] = {1, 2, 3, 4, 5, 7, 16, 17, 27, 64, 100, 152, 200, 600, 607, 608, 609, 1823, 1824, 1825, 4096, 65536};
  for (int W : {1, 2, 4, 8}) for (long long G : {1, 2, 3, 16, 100, 152, 456}) for (long long total : counts) {
    std::vector<int> owners((size_t)total, 0);
    long long most = 0, least = total, cmost = 0, cleast = total;
    for (long long g = 0; g < G; ++g) {
      long long cta = 0;
      for (int w = 0; w < W; ++w) {
        const atk::ItemRange r = atk::cta_items(total, G, W, g, w);
        if (r.lo < 0 || r.hi < r.lo || r.hi > total) { std::printf("range: %lld %lld %d\n", total, G, W); return 1; }
        if (w > 0 && cta == 0 && r.hi > r.lo) { std::printf("first: %lld %lld %d\n", total, G, W); return 1; }
        for (long long i = r.lo; i < r.hi; ++i) ++owners[(size_t)i];
        cta += r.hi - r.lo;
        if (r.hi - r.lo > most) most = r.hi - r.lo;
        if (r.hi - r.lo < least) least = r.hi - r.lo;
      }
      if (cta > cmost) cmost = cta;
      if (cta < cleast) cleast = cta;
    }
    for (int o : owners) if (o != 1) { std::printf("owners: %lld %lld %d\n", total, G, W); return 1; }
    if (most - least > 1) { std::printf("elements: %lld %lld %d\n", total, G, W); return 1; }
    if (total < G * W && cmost - cleast > 1) { std::printf("CTAs: %lld %lld %d: %lld %lld\n", total, G, W, cleast, cmost); return 1; }
  }
  return 0;
}
"""


def test_items_of_ctas(tmp_path):
    src, exe = tmp_path / "split.cpp", tmp_path / "split"
    src.write_text(_SRC)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", f"{ROOT}/paper_1911_05769_gb300/csrc", str(src), "-o",
                           str(exe)])
    r = subprocess.run([str(exe)], text=True, capture_output=True)
    assert r.returncode == 0, r.stdout
