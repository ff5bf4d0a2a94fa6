"""What the EC kernel's staging area rests on (host code, compiled with nvcc,
no GPU), over the staging capacities (multiples of 8), lanes and slab counts
that occur: a tile's share is a multiple of 16 bytes; the area of the slab
masks holds an id per staged bead and a bit per bead and slab; the slabs
cover the tile's box and fit 10 bits; and every capacity that the settings
accept fits a block, with more lanes or, last, with what fits."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include "ec_kernel.cuh"
using namespace ecmc;
int main() {
  long n = 0, bad = 0;
  auto check = [&](bool ok, const char *what, int S, int G, int k) {
    ++n;
    if (!ok && ++bad < 10) std::printf("%s S=%d G=%d %d\n", what, S, G, k);
  };
  for (int G : {4, 8, 16, 32})
    for (int S = 8; S <= 65504; S += 8)
      for (int nsl : {10, 11, 30, 1000}) {
        const int MQ = mask_quads(S, G, nsl);
        check((size_t)MQ * 16 >= (size_t)S * 4, "ids", S, G, nsl);
        check((long long)MQ * 128 / (3 * (nsl + 1)) >= S, "bits", S, G, nsl);
        for (int M : {8, (S / 24) * 8 + 8, S})
          for (int M64 : {0, S}) check(group_bytes(S, M64, M, MQ) % 16 == 0, "share", S, G, nsl);
      }
  // slabs: counted from the box's lower end by rint, so e_max / side + 1 of
  // them, and one for rounding
  for (int G : {4, 8, 16, 32})
    for (double sigma : {1e-3, 1.0, 50.0})
      for (double e = 1.5; e < 2e4; e *= 1.13)
        for (int S : {32, 160, 512, 4096, 14016})
          for (size_t budget : {(size_t)0, (size_t)2048, (size_t)192 * G}) {
            const SlabPick k = pick_slabs(e * sigma, sigma, S, G, budget);
            check(k.nsl >= 10 && k.nsl <= 1000, "nsl", S, G, k.nsl);
            check(e * sigma * k.inv <= k.nsl - 1.0, "cover", S, G, k.nsl);
          }
  const size_t room = 232448;
  for (int S = 32; S <= 65504; S += 32)
    for (int M = 32; M <= S; M += 32) {
      const bool whole = staging_budget(S, M, M, 1, 1) <= room;
      bool packed = false;
      for (int G : {4, 8, 16})
        packed = packed || staging_budget(S, 0, M, 1, 32 / G) + request_budget(32 / G) <= room;
      if (!whole && !packed) break;
      const int s = fit_stage(S, M, 32, room);
      check(s >= M && s <= S && group_bytes(s, 0, M, mask_quads(s, 32, 10)) <= room, "fit", S, 32, M);
      check(s == S || group_bytes(s + 32, 0, M, mask_quads(s + 32, 32, 10)) > room, "most", S, 32, M);
    }
  std::printf("checked %ld bad %ld\n", n, bad);
  return bad != 0;
}
"""


def test_staging_area(tmp_path):
    nvcc = shutil.which(os.environ.get("NVCC", "nvcc"))
    if nvcc is None:
        pytest.skip("nvcc not found")
    src = tmp_path / "t.cu"
    src.write_text(SRC)
    exe = tmp_path / "t"
    r = subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a",
                        "-I", os.path.join(ROOT, "paper_1502_06447_gb300", "csrc"),
                        "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    if r.returncode != 0:
        pytest.fail(r.stderr[-3000:])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and "bad 0" in out.stdout, out.stdout[-2000:]
