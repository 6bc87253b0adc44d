"""The rules that kernels launched as programmatic dependents keep (csrc/sgp_internal.cuh, at
launch_pdl), read off the CUDA sources: every kernel waits, and what other grids of the stream
write is not loaded through the read-only path."""

import glob
import os
import re

import pytest

from paper_2106_06695_gb300 import build_lib

SOURCES = {os.path.basename(p): open(p).read()
           for p in sorted(glob.glob(os.path.join(build_lib.CSRC, "*.cu*")))}

# arrays that do not change after the build (which ends with a synchronisation), the server's
# table (constant while a lane's graph runs), and lists derived from them
FIXED = {"nbr", "nbr_j", "plane", "idx", "w", "perm", "seg", "items", "act", "chain", "pw",
         "huge_rows", "med_rows", "rank", "T"}


def kernels(text):
    """(name, parameters, body) of every __global__ function."""
    for at in re.finditer(r"__global__", text):
        head = text.index("{", at.end())
        sig = text[at.end():head]
        name = re.search(r"(k[b]?_\w+)\s*\(", sig)
        depth, end = 1, head + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[end], 0)
            end += 1
        yield name.group(1), sig[name.end():], text[head:end]


def test_sources_are_read():
    assert sum(1 for t in SOURCES.values() for _ in kernels(t)) > 80


@pytest.mark.parametrize("name", sorted(SOURCES))
def test_every_kernel_waits(name):
    for kernel, _, body in kernels(SOURCES[name]):
        assert "pdl_enter()" in body or "SLOT_AHEAD_IN_LOOP" in body, kernel


def test_read_only_rows_are_for_ordinary_launches():
    """The read-only loads of lattice rows (ro8) stand under RO alone, in one kernel, and that
    instance is never launched as a dependent."""
    for name, text in SOURCES.items():
        if name != "values.cuh":
            for line in text.splitlines():
                assert "ro8(" not in line or "if constexpr (RO)" in line, line
    mvm = SOURCES["mvm.cu"]
    assert mvm.count("k_blur_pipe<true, S><<<") == 1
    assert not re.search(r"launch_pdl\w*\([^;]*<true, S>", mvm)


@pytest.mark.parametrize("name", sorted(SOURCES))
def test_read_only_path_is_for_fixed_arrays(name):
    fixed = set() if name == "build.cu" else FIXED  # the build itself writes all of them
    if name == "values.cuh":
        fixed = fixed | {"p"}  # ro8
    for pointer in re.findall(r"const [\w ]+\* ?__restrict__ (\w+)", SOURCES[name]):
        assert pointer in fixed, pointer
    for pointer in re.findall(r"__ldg\(\(?(?:reinterpret_cast<[^>]*>\()?(\w+)", SOURCES[name]):
        assert pointer in fixed, pointer
