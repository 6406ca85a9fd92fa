"""Loads by the read-only path in the kernels of the dependent chain.

A kernel launched as a dependent may be resident while the kernels before it
on the stream (the library's or a user's) still write, so __ldg, which takes
its data for constant while the kernel lives, is for tables that no kernel
writes: the plan's and the context's.  Every __ldg of a file whose kernels
start so is checked by the name of what it reads."""
import os
import re

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2410_04090_gb300", "csrc")
# taps, projections, sector and pattern tables, corner table
TABLES = {"L.tapx", "L.tapy", "R.projx", "R.projy", "b.bin_cosf", "b.bin_sinf", "b.disk_mask", "b.corner_lut", "pat"}


def _read_only_loads(text):
    return [re.match(r"[A-Za-z_][\w.]*", m.group(1)).group(0)
            for m in re.finditer(r"__ldg\(\s*((?:[^()]|\([^()]*\))*)\)?", text)]


def test_read_only_loads_are_of_tables():
    files = {f: open(os.path.join(CSRC, f)).read() for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh"))}
    chain = [f for f, text in files.items() if "after_previous()" in text]
    assert {"k_pyramid.cu", "k_detect.cu", "k_pyca.cu", "k_orb_match.cu", "k_refine.cu"} <= set(chain)
    found = 0
    for f in chain:
        loads = _read_only_loads(files[f])
        found += len(loads)
        assert set(loads) <= TABLES, (f, sorted(set(loads) - TABLES))
    assert found >= 8  # the pattern of the search still meets the sources
