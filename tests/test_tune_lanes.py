"""Lanes that a tile runs with when few tiles are there, and the autotuner under
that rule: settings that run the same kernel instance are one point, timed once
and returned under the lanes that ran."""
import os
import subprocess

import pytest

from paper_1502_06447_gb300 import ecmc
from paper_1502_06447_gb300.configs import Melt

from helpers import gpu_context

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")

SRC = r"""
#include <cstdio>
#include <vector>
#include "ecmc_internal.h"
using namespace ecmc;
int main() {
  long bad = 0;
  for (int lanes : {4, 8, 16, 32})
    for (long n : {1L, 27L, 1824L, 1825L, 3648L, 3649L, 7296L, 7297L, 1000000L, 2147483647L}) {
      const int want = n <= 1824 ? 32 : (n <= 3648 ? 16 : (n <= 7296 ? 8 : 4));
      bad += spread_lanes(n, lanes, 0, 152) != (want > lanes ? want : lanes);
      bad += spread_lanes(n, lanes, 2, 152) != lanes;
    }
  // 1,000 tiles at 4.2 sigma, 2,000 below 4: lanes asked for and lanes run
  auto ran = [](const TunePoint &p) { return spread_lanes(p.tile_side < 4.0 ? 2000 : 1000, p.lanes, 0, 152); };
  std::vector<TunePoint> seen;
  auto trial = [&](const TunePoint &p, TuneScore *s) -> ecmc_status {
    for (const TunePoint &q : seen)
      bad += q.lanes == p.lanes && q.tile_side == p.tile_side && q.cell_side == p.cell_side && q.ecs == p.ecs &&
             q.warps == p.warps && q.tight == p.tight;
    seen.push_back(p);
    bad += p.lanes != ran(p);
    s->ecs_per_s = (p.tile_side == 3.8 ? 2.0 : 1.0) + (p.lanes == 16 ? 0.5 : 0.0);
    return ECMC_OK;
  };
  TunePoint best{};
  TuneScore bs{};
  int n = 0;
  bad += tune_search(TunePoint{8, 4.2, 1.05, 1, 1, 1.08}, trial, &best, &bs, &n, ran) != ECMC_OK;
  bad += n != (int)seen.size() || best.tile_side != 3.8 || best.lanes != 16;
  // a start that is not admissible itself (another axis off its default)
  auto odd = [&](const TunePoint &p, TuneScore *s) -> ecmc_status {
    if (p.tight != 1.08) return ECMC_EINVAL;
    s->ecs_per_s = 1.0;
    return ECMC_OK;
  };
  bad += tune_search(TunePoint{8, 4.2, 1.05, 1, 1, 1.0}, odd, &best, &bs, &n, ran) != ECMC_OK || best.lanes != 32;
  std::printf("bad %ld\n", bad);
  return bad != 0;
}
"""


def test_spread_rule_and_search_host(tmp_path):
    if not os.path.isdir(CUDA_INC):
        pytest.skip("CUDA headers not found")
    src = tmp_path / "t.cpp"
    src.write_text(SRC)
    exe = tmp_path / "t"
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1502_06447_gb300", "csrc"),
                        "-I", os.path.join(ROOT, "include"), "-I", CUDA_INC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    if r.returncode != 0:
        pytest.fail(r.stderr[-3000:])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and "bad 0" in out.stdout, out.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("kw", [dict(precision=ecmc.PREC_FP64), dict(precision=ecmc.PREC_FP32F, k_spring=30.0)])
def test_autotune_returns_the_lanes_that_ran(kw):
    """A few hundred tiles: FP64 and springs run 32 lanes whatever is asked
    for, so lanes give no points of their own (at most 12 of the other axes
    in the first round and 10 in the second)."""
    m = Melt("tune_24", (24, 24, 24), 1.05, 12, ell=2.0, seed=0xEC0A71, mode="domain", dir_mode="iso",
             sweeps=1, D=(6, 6, 6))
    ctx = gpu_context(m, lanes=8, **kw)
    t = ctx.autotune(m.ell, seed=m.seed, trial_sweeps=1)
    assert t["lanes"] == 32 and t["block_tiles"] == 0
    assert t["n_trials"] <= 22


@pytest.mark.gpu
def test_batch_autotune_returns_the_lanes_that_ran():
    b = ecmc.Batch([dict(dims=(12, 12, 12), spacing=1.05, N=8)] * 3, jitter=0.01, seed=1)
    b.configure(dir_mode=ecmc.DIR_ISO, precision=ecmc.PREC_FP64, lanes=8)
    t = b.autotune(2.0, seed=1, trial_sweeps=1)
    assert t["lanes"] == 32 and t["block_tiles"] == 0
