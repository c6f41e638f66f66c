"""The rules of pdl.cuh for kernels launched with programmatic stream serialisation, checked on the source:
their life begins before the kernel ahead of them has ended, so what that kernel writes must not be read in
ways that declare it read-only for the kernel's life and let the load move above the wait."""
import glob
import os
import re

import pytest

from paper_1905_10182_gb300 import buildlib

# parameters behind const __restrict__ that only the host writes (copies, or kernels it waits for)
HOST_WRITTEN = {"k_batch_step": {"dom", "tiles", "ntiles_p", "links"}}


def code(path):
    text = open(path, encoding="utf-8").read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


FILES = sorted(glob.glob(os.path.join(buildlib.CSRC, "*.cu")) + glob.glob(os.path.join(buildlib.CSRC, "*.cuh")))


def past(text, i):
    """The place after the bracket that closes the one at i."""
    depth = 0
    for j in range(i, len(text)):
        depth += {"(": 1, "{": 1, ")": -1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return j + 1


def kernels(text):
    """name -> (parameters, body) of the kernels in the source."""
    found = {}
    for m in re.finditer(r"__global__\s+void\s+", text):
        i = m.end()
        if text.startswith("__launch_bounds__", i):
            i = past(text, text.index("(", i))
        name = re.match(r"\s*(\w+)\s*", text[i:])
        args = i + name.end()
        end = past(text, args)
        if text[end:].lstrip().startswith("{"):
            found[name.group(1)] = (text[args:end], text[end:past(text, text.index("{", end))])
    return found


KERNELS = {k: v for f in FILES for k, v in kernels(code(f)).items()}


def launched():
    """Kernels that are named in a launch_pdl call, or in a table that such a call picks from: all that are not
    launched with <<< >>>, their own or that of a dispatch macro."""
    text = "\n".join(code(f) for f in FILES)
    return {k for k in KERNELS if not re.search(r"\b%s\s*(?:<[^;()]*>)?\s*<<<|\w+_DISPATCH\(%s\b" % (k, k), text)}


def test_the_kernels_are_found():
    assert {"k_stream_collide", "k_stream_collide_x2", "k_psi", "k_cg_step", "k_mhd_step", "k_batch_step", "k_map_act", "k_gemm_bf16_tma",
            "k_project_v", "k_adam_v"} <= launched()
    assert len(launched()) >= 40


@pytest.mark.parametrize("name", sorted(launched()))
def test_waits_and_reads_through_plain_pointers(name):
    params, body = KERNELS[name]
    assert "pdl_wait();" in body
    readonly = set(re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", params))
    assert readonly <= HOST_WRITTEN.get(name, set())


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_no_read_only_loads(path):
    text = code(path)
    if "pdl_wait" in text or path.endswith(".cuh"):
        assert not re.search(r"__ldg\s*\(|ld\.global\.nc", text)
