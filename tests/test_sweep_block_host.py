"""Index arithmetic of the sweep by blocks (csrc/ff_block.cuh), compiled for the host."""
from __future__ import annotations

import os
import subprocess

from paper_1703_02563_gb300 import _build

# Every warp of a strip forms its row's addresses and loads that row's first query,
# whether or not the row exists.  So over all strips of all clusters, those past the level
# among them, each has to be a row of the level; and the rows that exist come once each.
ROWS = r"""
#include <cstdio>
#include <vector>
#include "ff_block.cuh"
int main() {
    using namespace ffk;
    const int per = kBlkRows * kBlkCluster;
    int bad = 0;
    for (int V = 1; V <= 4096; V += V < 140 ? 1 : 97)
        for (int flip = 0; flip < 2; flip++) {
            std::vector<int> seen(V, 0);
            for (int v = 0; v < (V + per - 1) / per * per; v++) {
                const int gy = block_row(v, V, flip);
                if (gy < 0 || gy >= V) {
                    if (bad++ < 5) printf("V %d v %d flip %d: row %d\n", V, v, flip, gy);
                } else if (v < V) {
                    seen[gy]++;
                }
            }
            for (int r = 0; r < V; r++) bad += seen[r] != 1;
        }
    return bad != 0;
}
"""


# A vector load has no order among its words: a tag must not share one with what it stands for.
TAGS = r"""
#include <cstddef>
#include "ff_block.cuh"
int main() {
    using namespace ffk;
    const size_t stage = offsetof(BlockShared, stage), tag = offsetof(BlockShared, tag);
    const size_t end = stage + sizeof(BlockShared::stage);
    return sizeof(BlockStage) % 16 || stage % 16 || !(tag >= (end + 15) / 16 * 16 || tag < stage);
}
"""


def _run(text, tmp_path):
    src, exe = tmp_path / "check.cu", tmp_path / "check"
    src.write_text(text)
    inc = os.path.join(_build.ROOT, "include")
    subprocess.run([_build.nvcc(), *_build.ARCH, "-std=c++17", "-I", _build.CSRC, "-I", inc,
                    "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_every_row_of_a_strip_is_a_row_of_the_level(tmp_path):
    _run(ROWS, tmp_path)


def test_staged_tags_share_no_vector_with_the_staged_values(tmp_path):
    _run(TAGS, tmp_path)
