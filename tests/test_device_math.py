"""Quotients, reciprocals and roots on the device are CUDA's own, at their full
accuracy: no kernel refines a hardware seed by hand or divides approximately."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1611_03189_gb300", "csrc")


def test_no_approximate_quotients_or_roots():
    seeds = re.compile(r"\b(rcp|rsqrt|sqrt|div)\.(approx|full)|__fdividef|__frcp_r[duz]|use_fast_math|prec-div|ftz=true")
    found = []
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            found += [(name, i, line.strip()) for i, line in enumerate(f, 1) if seeds.search(line)]
    assert found == []
