"""The pages a decode step's linears ask into L2: the numbering of their blocks and the addresses, run on the host and compared
with a list made here.  (The requests change no result, so no comparison of outputs can see a wrong one.)"""
import os
import shutil
import subprocess

import numpy as np
import pytest

from conftest import ROOT
from paper_2607_21042_b200 import build

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "common.cuh"
using namespace ttsgpt;
int main(int argc, char **argv) {
  KvPrefetch p;
  const int n_cta[3] = {atoi(argv[1]), atoi(argv[2]), atoi(argv[3])};
  p.rows = atoi(argv[4]); p.cap = atoi(argv[5]); p.blocks = atoi(argv[6]); p.pps = atoi(argv[7]);
  p.block_bytes = kPageElems * 2; p.n_parts = 3;
  std::vector<int> pages(p.rows * p.pps);
  std::vector<int4> slots(p.rows);
  for (int z = 0; z < p.rows; ++z) { if (scanf("%d", &slots[z].y) != 1) return 1; }
  for (int &x : pages) if (scanf("%d", &x) != 1) return 1;
  p.slots = slots.data(); p.slot_pages = pages.data();
  p.layer = reinterpret_cast<const unsigned char *>(uintptr_t(1) << 40);
  for (p.part = 0; p.part < 3; ++p.part)
    for (int cta = 0; cta < n_cta[p.part]; ++cta)
      for (int lane = 0; lane < 32; ++lane)
        for (int u = kv_prefetch_first(p, cta, lane); u < kv_prefetch_total(p); u += kv_prefetch_stride(p, n_cta[p.part]))
          if (const unsigned char *q = kv_prefetch_address(p, u)) printf("%lld\n", (long long)(q - p.layer));
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = build.nvcc_path()
    if not (shutil.which(nvcc) or os.path.exists(nvcc)):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("kv_prefetch")
    (d / "p.cu").write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", os.path.join(ROOT, "paper_2607_21042_b200", "csrc"),
                    "-o", str(d / "p"), str(d / "p.cu")], check=True)
    return str(d / "p")


@pytest.mark.parametrize("rows,cap,heads,pps,n_cta", [(8, 6, 20, 32, (160, 213, 216)), (11, 4, 20, 12, (160, 160, 216)), (48, 1, 20, 32, (40, 80, 40)),
                                                      (2, 32, 8, 32, (1, 2, 3)), (3, 5, 18, 7, (1000, 1, 7))])
def test_every_complete_page_is_asked_for_once(program, rows, cap, heads, pps, n_cta):
    rng = np.random.default_rng(rows)
    edges = [1, 64, 65, 128, 129, pps * 64]       # a page is complete when a token lies behind it
    n_tok = [edges[z] if z < len(edges) else int(rng.integers(1, pps * 64 + 1)) for z in range(rows)]
    pages = rng.permutation(rows * pps).reshape(rows, pps)
    text = " ".join(map(str, n_tok)) + " " + " ".join(map(str, pages.reshape(-1)))
    out = subprocess.run([program, *map(str, n_cta), str(rows), str(cap), str(2 * heads), str(pps)], input=text, capture_output=True, text=True, check=True)
    got = sorted(int(x) for x in out.stdout.split())
    want = sorted((int(pages[z, j]) * 2 * heads + b) * 8192 for z in range(rows) for j in range(min(cap, (n_tok[z] - 1) // 64)) for b in range(2 * heads))
    assert got == want
