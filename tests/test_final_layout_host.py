"""Regions of the final contraction (csrc/finlayout.cuh), compiled for the host: M^T and V of every cut that a
network can meet lie inside the regions sized for its widest one."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = r"""
#include "finlayout.cuh"
using namespace td;
// cuts (m x n) whose columns leave the regions of chi_mps, bond D; W: V shares its region with T1
extern "C" long run(int nt, int cm, int D) {
  const int cmx = cm > 2 ? cm : 2, n_max = cmx * D * 2, m_max = cm * D;
  const int64_t mt = final_mt_elems(nt, n_max, m_max), v = final_v_elems(nt, n_max, m_max);
  const int64_t t1 = (int64_t)cm * D * 2 * D * cmx, w = v > t1 ? v : t1;
  long bad = 0;
  for (int m = 1; m <= m_max; ++m)
    for (int n = 1; n <= n_max; n += n < 64 ? 1 : 31) {
      const int g = team_svd_group(nt, n, m), ldm = final_ld(n, g, m, mt), ldv = final_ld(m, g, m, w);
      bad += ldm < n || ldv < m || (int64_t)m * ldm > mt || (int64_t)m * ldv > w;
    }
  return bad;
}
"""


@pytest.mark.parametrize("threads", [256, 512, 1024])
def test_cuts_stay_inside_their_regions(tmp_path, threads):
    src, lib = str(tmp_path / "t.cpp"), str(tmp_path / "t.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(HERE, "..", "paper_2310_10722_gb300", "csrc"), src, "-o", lib], check=True)
    run = ctypes.CDLL(lib).run
    run.restype = ctypes.c_long
    caps = [(cm, D) for cm in (*range(1, 34), 64, 128, 1024) for D in range(1, 33) if cm * D <= 1024]
    assert [c for c in caps if run(threads, *c)] == []
