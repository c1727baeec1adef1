"""CPU checks of the sources of kernels that start while the kernel before them still runs (they call
pdl_wait): what that kernel writes is never read through the read-only path.  CUDA wants data read
with __ldg, or through a const __restrict__ pointer, unwritten for the kernel's whole lifetime,
which here overlaps the writer's; such loads may also move above the wait."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_13379_gb300", "csrc")
# written once, when the operator is created or its live-pair lists are built
STATIC = {"xyz", "rs", "perm", "pairs", "sc", "W0", "Wlo", "K"}


def _functions(text, pattern):
    """(signature, body) of the definitions whose signature starts at a match of pattern."""
    for m in re.finditer(pattern, text):
        brace, semi = text.find("{", m.start()), text.find(";", m.start())
        if brace < 0 or 0 <= semi < brace:
            continue
        depth = 0
        for i in range(brace, len(text)):
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            if depth == 0:
                yield text[m.start():brace], text[brace:i + 1]
                break


def _sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        yield os.path.basename(path), text


def overlapped_kernels():
    return [(name, re.search(r"(\w+)\s*\([^()]*(\([^()]*\)[^()]*)*\)\s*$", sig).group(1), sig, body)
            for name, text in _sources() for sig, body in _functions(text, r"__global__\s") if "pdl_wait()" in body]


KERNELS = overlapped_kernels()


def test_the_overlapped_kernels_are_found():
    assert {k[1] for k in KERNELS} >= {"mf_sym_kernel", "mf_multi_kernel", "adj_sym_kernel", "gemv_kernel",
                                       "gemv_sym_kernel", "rk4_stage_kernel", "reduce_I_kernel",
                                       "adj_epilogue_kernel", "mf_pair_packed_kernel"}


@pytest.mark.parametrize("file,kernel,sig,body", KERNELS, ids=[k[1] for k in KERNELS])
def test_no_read_only_loads_of_overlapped_data(file, kernel, sig, body):
    for name in re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", sig):
        assert name in STATIC, f"{file}: {kernel} promises that nothing writes {name} while it runs"
    for arg in re.findall(r"__ldg\(\s*(?:reinterpret_cast<[^>]*>\(\s*)?([\w.]+)", body):
        assert arg.startswith("nd.") or arg in STATIC, f"{file}: {kernel} reads {arg} through the read-only path"


def test_slot_sums_take_ordinary_loads():
    (sig, body), = [f for _, text in _sources() for f in _functions(text, r"__device__[^;{}]*\bsum_slots\(")]
    assert "__restrict__" not in sig and "__ldg" not in body
