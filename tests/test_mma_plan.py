"""The shared-memory layout of linear_mma_kernel's launches, by arithmetic on the CPU: every chunk
size from empty to dense, every batch, matrices from one chunk to thousands, both value types.  The
areas that the kernel uses must lie one behind the other inside the bytes that the launch asks for.
(A request 64 bytes short of the control area was met once, at some chunk sizes only.)"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include "sp_mma_plan.h"
using namespace sp;
using namespace sp::mma;

static long checked = 0;
static const sp_matrix* H;
static int B;
static MmaChoice C;
#define CHECK(cond) do { if (!(cond)) { \
  std::printf("%s: RB %d T %d chunk %llu esize %d M %d, form nt %d rw %d cw %d occ %d cluster %d\n", #cond, H->RB, H->T, \
              (unsigned long long)H->max_chunk, H->esize, B, C.nt, C.rw, C.cw, C.occ, C.cluster); std::exit(1); } } while (0)

int main() {
  sp_matrix h = {};
  H = &h;
  const int rbs[] = {1, 2, 8, 32, 40, 96, 152, 153, 172, 313, 2000}, ts[] = {1, 2, 3, 7, 16, 18, 64, 100, 172, 400};
  const int sms[] = {152, 148, 132};
  for (int sm : sms)
    for (int rb : rbs)
      for (int t : ts)
        for (int es = 1; es <= 2; ++es)
          for (uint64_t chunk = kMaskBytes; chunk <= kMaskBytes + (uint64_t)kRows * kTileK * es; chunk += 16)
            for (int M = 1; M <= kMmaMaxRows; M += M < 10 || M > 30 ? 1 : 3) {
              h.RB = rb, h.T = t, h.num_sms = sm, h.esize = es, h.max_chunk = chunk, h.N = (int64_t)rb * kRows;
              h.K = (int64_t)t * kTileK;
              B = M;
              MmaPlan p;
              C = MmaChoice{};
              CHECK(choose(&h, M, &C, &p));
              ++checked;
              const int groups = C.cw * C.rw / kRows;
              CHECK(C.nt * 8 >= M && C.cluster >= 1 && C.cluster <= 16 && C.cluster <= t);
              CHECK(p.cluster == C.cluster && p.slots <= kMaxSlots && p.slots >= (groups < 4 ? groups + 1 : groups));
              // occ CTAs and the 1 KB that the system keeps for each fit an SM
              CHECK(p.smem % 128 == 0 && C.occ * (p.smem + 1024) <= 228 * 1024 && p.smem <= 227 * 1024);
              // x tiles, chunks, the sums that take their place, tables
              CHECK(p.chunk_region >= chunk && p.chunk_region % 128 == 0 && p.ring_off % 1024 == 0);
              CHECK(p.ring_off >= (uint32_t)p.slots * C.nt * 1024);
              CHECK(p.tab_off >= p.ring_off + (uint64_t)p.slots * p.chunk_region && p.tab_off % 16 == 0);
              CHECK(p.tab_off >= (uint64_t)groups * M * kRows * 4);
              // the word after a value is read too (four INT8 values are placed at a time)
              CHECK(p.tab_off + 8 <= p.smem);
              // full, empty, quarter index, tag of each slot; 16-entry table; receive area
              CHECK(p.bar_off >= p.tab_off + (uint32_t)(C.cw * C.rw * 16) && p.bar_off % 8 == 0);
              CHECK(p.lut_off >= p.bar_off + kMaxSlots * 28 && p.lut_off % 64 == 0);
              CHECK(p.rx_off >= p.lut_off + 64 && p.rx_off % 4 == 0);
              const bool push = C.nt == 1 && C.cw == 8 && C.cluster > 1;
              const uint64_t own = (M + C.cluster - 1) / C.cluster;  // tokens that a CTA owns, at most
              CHECK(p.rx_off + (push ? own * C.cluster * kRows * 4 : 0) <= p.smem);
            }
  std::printf("%ld layouts\n", checked);
  return 0;
}
"""


def _cuda_include():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")


def test_areas_lie_within_the_request(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text(HARNESS)
    subprocess.check_call([cxx, "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_2405_03594_gb300", "csrc"),
                           "-I", _cuda_include(), str(src), "-o", str(exe)])
    p = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stdout
    assert int(p.stdout.split()[0]) > 10**6
