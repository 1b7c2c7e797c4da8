"""What the projection kernels rely on in their plans, for every shape of a range: compiled for the host, no GPU."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_20357_b200", "csrc")
# clusters of 1 .. 8 CTAs that a B200 (148 SMs) keeps resident, one CTA per SM
FIT = (0, 148, 74, 45, 33, 26, 22, 15, 15)

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "proj_plan.h"
using namespace tabed;
static const int fit[9] = {%s};
static ProjPlan plan(int rows, int K, int n, int can_norm) { return plan_proj((rows + kTcM - 1) / kTcM, (K + kTcKC - 1) / kTcKC, n, can_norm != 0, fit); }
int main(int argc, char** argv) {
  if (argc == 5) {
    const ProjPlan p = plan(atoi(argv[1]), atoi(argv[2]), atoi(argv[3]), atoi(argv[4]));
    printf("%%d %%d %%d %%d %%u %%zu\n", p.n_pad, p.ks, p.n_stages, (int)p.norm, p.recv_off, p.smem);
    return 0;
  }
  long bad = 0, shapes = 0;
  for (int rows = 32; rows <= 12288; rows += rows < 1024 ? 96 : 1376)
    for (int K = 32; K <= 8192; K += K < 1024 ? 104 : 1400)
      for (int n = 1; n <= 4096; n += n < 80 ? 1 : (n < 1100 ? 37 : 499))
        for (int can_norm = 0; can_norm < 2; ++can_norm, ++shapes) {
          const ProjPlan p = plan(rows, K, n, can_norm);
          const int chunks = (K + kTcKC - 1) / kTcKC;
          const size_t a = tc_block_bytes(kTcM), b = tc_block_bytes(p.n_pad), slab = (size_t)p.n_pad * kTcM * 4;
          const size_t operands = p.norm ? (size_t)p.cps * proj_norm_block_bytes(p.n_pad) + p.n_stages * a : p.n_stages * (a + b);
          bool ok = p.us < 1e29f && p.n_pad %% 16 == 0 && p.n_pad >= 16 && p.n_pad <= kTcMaxN && p.n_tiles * p.n_pad >= n;
          ok = ok && (p.n_tiles - 1) * p.n_pad < n && p.n_tiles * p.n_pad <= n + kTcMaxN && (can_norm || !p.norm);     // operand buffers
          ok = ok && p.ks >= 1 && p.ks <= kProjMaxSplit && p.ks * p.cps >= chunks && (p.ks - 1) * p.cps < chunks;      // no split is empty
          ok = ok && p.n_stages >= 1 && p.n_stages <= kProjMaxStages && operands <= p.smem && p.smem <= kProjMaxSmem;
          if (p.recv_off) ok = ok && p.ks > 1 && p.recv_off >= operands && p.recv_off %% 128 == 0 && p.recv_off + (size_t)p.ks * proj_owned(p.n_pad, p.ks) * kTcM * 4 <= p.smem;
          else ok = ok && slab <= p.smem;
          // an SM has 228 KB of shared memory (1 KB of it a CTA's own overhead) and 512 columns of tensor memory
          const size_t side_by_side = 228u * 1024u / (p.smem + 1024u);
          ok = ok && side_by_side * tc_tmem_cols(p.n_pad) <= 512 && (size_t)tc_tmem_cols(p.n_pad) * 228u * 1024u <= 512u * (p.smem + 4096u);
          if (!ok && bad++ < 5) printf("rows %%d K %%d n %%d norm %%d: n_pad %%d ks %%d stages %%d smem %%zu\n", rows, K, n, can_norm, p.n_pad, p.ks, p.n_stages, p.smem);
        }
  printf("%%ld of %%ld\n", bad, shapes);
  return bad != 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(PROGRAM % ", ".join(map(str, FIT)))
    exe = str(d / "plan")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, "-o", exe, str(d / "plan.cpp")], check=True)
    return exe


def test_plans_keep_to_the_memory_that_a_cta_and_its_neighbours_have(program):
    res = subprocess.run([program], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout


def test_a_long_down_projection_pulls_its_partial_sums(program):
    """1024 columns from 4096 at 800 positions: no room for a receive buffer beside the operands (the GPU test of that form
    relies on it)."""
    n_pad, ks, stages, norm, recv_off, smem = map(int, subprocess.run([program, "1024", "4096", "800", "0"], capture_output=True, text=True, check=True).stdout.split())
    assert ks > 1 and recv_off == 0
