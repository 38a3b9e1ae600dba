"""Kernels of the adjoint's reverse chain are launched while the kernel before them
still runs and wait for it inside the grid. What that kernel writes must not be
declared const __restrict__, which allows loads from the read-only cache, or
ahead of the wait. Read from the source: a stale load depends on timing.
"""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2103_08301_gb300", "csrc",
                   "lbm_adjoint.cu")
KERNEL = re.compile(r"__global__ void __launch_bounds__\([^)]*\)\s+(\w+)\(([^)]*)\)\s*\{(.*?)\n\}", re.S)


def test_chained_kernels_promise_no_constant_inputs():
    text = open(SRC).read()
    chained = [(n, args) for n, args, body in KERNEL.findall(text) if "chain_start()" in body]
    assert {n for n, _ in chained} == {"adj_local", "adj_finish", "adj_finish_terms"}
    for name, args in chained:
        promised = {a.split()[-1].lstrip("*") for a in args.split(",") if "__restrict__" in a}
        assert promised <= {"fld"}, (name, promised)  # the fields of a run are complete before its first kernel
