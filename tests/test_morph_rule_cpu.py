"""The morphing forward transform's choice of form (csrc/morph_rule.cuh) over every plane that is admitted, also
planes of one row and up to 2^31 - 2^20 nodes, against the same rule in whole numbers of any size."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1001_1588_gb300", "csrc")
TOP = 2 ** 31 - 2 ** 20
SHAPES = [(1, TOP, 1), (1, 500_000_000, 1), (3, 600_000_000, 2), (4, TOP // 4, 20), (1, 64, 1), (2048, 2048, 20), (2400, 65, 6),
          (62, 173, 9), (256, 256, 4), (46000, 46000, 3), (TOP, 1, 1), (5, 430_000_001, 65535)]


def _rule(ny, nx, K, sms):
    tiles = -(-nx // 64)
    if ny * nx * K <= 3 * sms * 256 or 5 * nx < 3 * 64 * tiles:
        return 0
    return 2 if tiles * -(-ny // 16) * K >= 8 * sms else 1


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_form_of_every_plane(tmp_path):
    (tmp_path / "t.cc").write_text(
        '#include <cstdio>\n#include <cstdlib>\n#include "morph_rule.cuh"\n'
        "int main(int n, char** a) { for (int i = 1; i + 2 < n; i += 3)"
        ' std::printf("%d ", fftenkf::morph_form(std::atoi(a[i]), std::atoi(a[i + 1]), std::atoi(a[i + 2]), 152)); }\n')
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover", "-I", CSRC, str(tmp_path / "t.cc"), "-o", exe],
                   check=True)
    out = subprocess.run([exe] + [str(v) for s in SHAPES for v in s], capture_output=True, text=True, check=True).stdout
    assert [int(x) for x in out.split()] == [_rule(ny, nx, K, 152) for ny, nx, K in SHAPES]
