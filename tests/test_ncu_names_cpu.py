"""The launch lists of ncu_summary.py keep every kernel of the library."""

import os
import re

import ncu_summary

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1001_1588_gb300", "csrc")


def test_every_kernel_is_listed():
    names = set()
    for f in os.listdir(CSRC):
        if f.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, f), encoding="utf-8") as src:
                names |= set(re.findall(r"__global__ void(?:\s+__launch_bounds__\((?:[^()]|\([^()]*(?:\([^()]*\))*[^()]*\))*\))?\s+(\w+)\(", src.read()))
    assert len(names) >= 25, names
    assert not [n for n in names if not ncu_summary.OURS.search("void fftenkf::%s<1>(P)" % n)]
