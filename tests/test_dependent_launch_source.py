"""Loads through the read-only data path (ld.global.nc, __ldg) ask that nothing writes the data
while the kernel runs.  A kernel under programmatic dependent launch is running before the kernel
ahead of it has finished writing, so in the sources that use such launches only tables that no
kernel writes (damping profile, tile prefix sums, chunk tables) may be read that way."""
import glob
import os
import re

TABLES = {"t", "tab", "base", "tbase", "pbase", "table"}


def _sources(root):
    for p in sorted(glob.glob(os.path.join(root, "paper_2401_16322_gb300", "csrc", "*.cu*"))):
        txt = open(p).read()
        yield os.path.basename(p), re.sub(r"//[^\n]*", "", txt)


def test_read_only_loads_are_of_tables(repo_root):
    launched, bad = [], []
    for name, txt in _sources(repo_root):
        if "pdl_wait()" not in txt or name == "pdl.cuh":
            continue
        launched.append(name)
        assert "ld.global.nc" not in txt, name
        for arg in re.findall(r"__ldg\(\s*(?:reinterpret_cast<[^>]*>\()?\s*&?(\w+)", txt):
            if arg not in TABLES:
                bad.append((name, arg))
    assert len(launched) >= 4          # the 2D and 3D TMA passes, the plain passes, the scalars
    assert not bad, bad


def test_restricted_kernel_parameters_are_tables(repo_root):
    """`const T* __restrict__` lets the compiler choose the same path by itself."""
    for name, txt in _sources(repo_root):
        if "pdl_wait()" not in txt:
            continue
        for typ, arg in re.findall(r"const (\w+)\s*\*\s*__restrict__\s+(\w+)", txt):
            assert (typ, arg) == ("ProblemDev", "probs") or (typ == "int" and arg in TABLES | {"tile_prob"}), (name, arg)
