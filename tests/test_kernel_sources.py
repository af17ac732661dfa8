"""CPU checks of the CUDA sources for faults that no GPU run may be made to show."""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2606_09514_gb300" / "csrc"


def code(path):
    """The file without comments."""
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", path.read_text(), flags=re.S)


def kernels(text):
    """(name, body) of each kernel."""
    for m in re.finditer(r"__global__", text):
        end = text.index("{", text.index(")", re.compile(r"\b\w+_kernel\s*\(").search(text, m.start()).end()))
        depth, at = 1, end + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[at], 0)
            at += 1
        yield re.search(r"(\w+_kernel)\s*\(", text[m.start():end]).group(1), text[end:at]


def remote_kernels():
    for f in sorted(CSRC.glob("*.cu")):
        for name, body in kernels(code(f)):
            if "dsmem_addr" in body:
                yield pytest.param(body, id=name)


# A CTA's shared memory may be accessed by its cluster only once it has started:
# a cluster barrier comes before the first access.
@pytest.mark.parametrize("body", list(remote_kernels()))
def test_cluster_barrier_before_remote_shared_memory(body):
    before = body[:body.index("dsmem_addr")]
    started = "cluster_arrive_started" in before and "cluster_wait_started" in before
    assert started or "cluster_sync" in before


def test_remote_kernels_are_found():
    assert {p.id for p in remote_kernels()} == {"attn_cl_kernel", "gemm_pf_kernel", "pool_refresh_kernel"}


# What a function keeps between calls would be shared by contexts on other devices and
# by host threads: only constants may be static in a function.
def test_no_state_kept_in_functions():
    found = [f"{f.name}: {line.strip()}" for f in sorted(CSRC.glob("*.cu*")) + sorted(CSRC.glob("*.h"))
             for line in code(f).splitlines() if re.match(r"\s+static\s+(?!const\b|constexpr\b)", line)]
    assert not found
