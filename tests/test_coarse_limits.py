"""Coarse meshes beyond the small dense solver's limit: no entry of its index lists is read for
them, and creating a handle on one is refused."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <stdio.h>
#include <vector>
#define __host__
#define __device__
#include "dense_lists.h"
// prints, for meshes of n cells per side (right triangles), whether the lists were built and
// how many entries a handle uploads from its array of kDenseMaxLists
int main() {
  for (int n = 2; n <= 100; n += n < 12 ? 1 : 11) {
    const int m = n - 1;
    std::vector<int> tri;
    auto id = [&](int i, int j) { return i < 1 || j < 1 || i >= n || j >= n ? -1 : i - 1 + (j - 1) * m; };
    for (int j = 0; j < n; ++j)
      for (int i = 0; i < n; ++i)
        for (int v : {id(i, j), id(i + 1, j), id(i + 1, j + 1), id(i, j), id(i + 1, j + 1), id(i, j + 1)})
          tri.push_back(v);
    std::vector<uint16_t> out(fmg::kDenseMaxLists);
    fmg::DenseLists d;
    const bool ok = fmg::build_dense_lists(m * m, 2 * n * n, 3, tri.data(), out.data(), &d);
    printf("%d %d %d %d\n", n, ok, ok ? d.total(m * m) : 0, d.stored(m * m));
    if (d.stored(m * m) > fmg::kDenseMaxLists) return 1;
  }
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a C++ compiler")
def test_stored_entries_stay_within_the_list_array(tmp_path):
    src = tmp_path / "lists.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "lists"
    inc = os.path.join(ROOT, "paper_1502_04657_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-I", inc, "-o", str(exe), str(src)], check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    rows = [tuple(map(int, line.split())) for line in run.stdout.splitlines()]
    assert run.returncode == 0, rows[-1]
    for n, ok, total, stored in rows:
        assert ok == (n <= 9)
        assert stored == (-(-total // 8) * 8 if ok else 0)


@pytest.mark.gpu
@pytest.mark.parametrize("dim,cells", [(2, 10), (2, 80), (3, 5), (3, 20)])
def test_create_refuses_larger_coarse_meshes(dim, cells):
    from paper_1502_04657_gb300 import fmg

    with pytest.raises(fmg.FmgError) as e:
        fmg.Solver(fmg.Problem(dim=dim, coarse_cells=cells, levels=1))
    assert e.value.code == fmg.FMG_ENOTSUP
