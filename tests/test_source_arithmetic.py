"""The kernels' divisions, reciprocals and roots are the correctly rounded ones.

The interface pivots of the preconditioner feed a closure that, for a nearly singular lowest mode, magnifies any
difference in them, so an approximate reciprocal has no place there; nor has a compiler switch that would turn every
division into one.  Checked on the sources, since no result shows the last bit of a pivot.
"""
import os
import re

ROOT = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1512_02548_gb300")
APPROXIMATE = re.compile(r"__fdividef|__frcp_r[zud]|__frsqrt_|__(?:exp|log|sin|cos|tan|pow)f\b|"
                         r"\b(?:rcp|div|sqrt|rsqrt|ex2|lg2|sin|cos)\.approx|use_fast_math|prec-div=false|prec-sqrt=false")


def test_no_approximate_arithmetic():
    found = []
    for base, _, files in os.walk(ROOT):
        for name in files:
            if name.endswith((".cu", ".cuh", ".cpp", ".h", ".py")):
                with open(os.path.join(base, name), encoding="utf-8") as f:
                    found += [f"{name}:{n}" for n, line in enumerate(f, 1) if APPROXIMATE.search(line)]
    assert not found, found
