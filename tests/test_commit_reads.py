"""Pass 1 of the tensor-core commit reads whole chunks of rows: up to 63 rows
past the last one, of the row exponents and of every column.  Builds a host
program against the kernels' header (no GPU needed) and checks that those
reads stay inside the regions make_layout hands out."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2108_05345_gb300", "csrc")

CASES = [(977, 16, 152), (977, 16, 1), (77, 5, 1), (96, 40, 152), (256, 512, 152), (511, 300, 1), (1000, 64, 152),
         (1025, 9, 152), (4096, 2048, 152)]

PROGRAM = r"""
#include <cstdio>
#include "lhdm_kernels.cuh"
int main() {
  const int cases[][3] = {%s};
  for (const auto& c : cases) {
    const lhdm::ScratchLayout L = lhdm::make_layout(c[0], c[1], c[2]);
    std::printf("%%d %%d %%zu %%zu %%d %%zu %%zu %%zu\n", c[0], c[1], L.Ver, L.csign, L.ldw, L.W, L.bt, L.w);
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def layouts(tmp_path_factory):
    nvcc = shutil.which(os.environ.get("NVCC", "nvcc"))
    if not nvcc:
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("reads")
    src = d / "reads.cu"
    src.write_text(PROGRAM % ", ".join("{%d, %d, %d}" % c for c in CASES))
    exe = d / "reads"
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")
    return [list(map(int, line.split())) for line in out if line.strip()]


def read_end(m, nP, kp):
    """First row of W (counted from the panel's first row) that pass 1 of a
    commit of kp reflectors at nP does not read; None: no tensor-core form."""
    L = m - nP
    if kp < 5 or L < kp + 72 or L > 16384:
        return None
    r0d = kp + (8 - ((nP + kp) & 7)) % 8
    groups = (((L - r0d + 7) >> 3) + 1) & ~1
    g1 = 8 if kp <= 16 else 4
    return r0d + -(-groups // g1) * g1 * 8


def test_chunk_reads_stay_inside_their_regions(layouts):
    worst = 0
    for m, n, ver, csign, ldw, W, bt, w in layouts:
        for nP in range(0, min(m, n), 1 if m < 2000 else 7):
            for kp in range(5, min(64, min(m, n) - nP) + 1):
                end = read_end(m, nP, kp)
                if end is None:
                    continue
                worst = max(worst, end - (m - nP))
                assert ver + (nP & 7) + end <= csign, (m, n, nP, kp)
                assert W + (n - 1) * ldw + nP + end <= w  # the last column
                assert bt + nP + end <= w                 # Q^T b
    assert worst == 63
