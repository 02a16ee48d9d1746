"""Properties of the kernel sources that no run can show (no GPU, no build)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_11536_gb300", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu*")))


def text(path):
    """A source without its comments."""
    s = open(path).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", s, flags=re.S))


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_no_bulk_load_multicasts_to_a_cluster(path):
    """Replicas on several GPUs load this library."""
    s = re.sub(r'"\s*\n?\s*"', "", text(path))  # adjacent literals are one instruction
    for instruction in re.findall(r"cp\.async\.bulk[^;\[]*", s):
        assert ".multicast::cluster" not in instruction, instruction


def body(s, start):
    """From `start` to the end of the brace block that opens after it."""
    i = s.index("{", start)
    depth, k = 1, i + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(s[k], 0)
        k += 1
    return s[start:k]


# what kernels launched early may read through the non-coherent path: tables, keys, the resident DB
READ_ONLY = {"tw", "src", "db", "a.perm", "a.mon", "a.mon_sh", "key"}  # src: of Pairs, twiddles


def non_coherent(s):
    """The first names of the operands of __ldg and of ldg4, which is __ldg of four words."""
    operands = [m.group(1) for m in re.finditer(r"__ldg\((?:reinterpret_cast<[^>]*>\()?([A-Za-z_.]+)", s)]
    return operands + [m.group(1) for m in re.finditer(r"(?<!void )\bldg4\(\w+(?:\[\w+\])?, ([A-Za-z_.]+)", s)]


def test_kernels_launched_early_read_their_input_by_plain_loads():
    """A kernel that waits in chain_wait is resident while its input is still being written: no
    load of that may be a non-coherent one, nor go through a __restrict__ pointer."""
    found = []
    for path in SOURCES:
        s = text(path)
        for m in re.finditer(r"__global__", s):
            kernel = body(s, m.start())
            if "chain_wait();" not in kernel:
                continue
            name = re.search(r"\b(k_\w+)\(", kernel).group(1)
            found.append(name)
            assert "__restrict__" not in kernel, name
            assert set(non_coherent(kernel)) <= READ_ONLY, (name, non_coherent(kernel))
    assert len(set(found)) >= 9, found
    # what those kernels call
    row = text(os.path.join(CSRC, "ntt_row.cuh"))
    assert "ld.global.nc" not in row and set(non_coherent(row)) <= READ_ONLY
    for helper in ("load16", "store16", "ld_global32"):
        assert "__restrict__" not in body(row, row.index(helper + "(")), helper
    first = text(os.path.join(CSRC, "query_ntt.cu"))
    first = body(first, first.index("first_pass("))
    assert set(non_coherent(first)) <= {"tw"} and "const uint32_t *__restrict__" not in first
    raw = text(os.path.join(CSRC, "ntt.cu"))
    assert "__ldg" not in body(raw, raw.index("raw_coeff("))


def test_stage_releases_are_waited_for_before_a_cta_leaves():
    """An MMA commit arrives on its barrier some time after it was issued, with a pair in both CTAs.
    Every barrier that releases a stage is waited for after the last stage (the completed phase,
    where a refill waits for the one before: parity ^ 1), in both CTAs, before the kernel ends."""
    kernels = 0
    for path in SOURCES:
        s = text(path)
        for m in re.finditer(r"__global__", s):
            kernel = body(s, m.start())
            released = set(re.findall(r"commit(?:_pair)?(?:<CG>)?\((empty\w*) \+", kernel))
            kernels += bool(released)
            for bar in released:
                waits = [w.split(";")[0].split("{")[0] for w in re.findall(r"if \(([^\n]*)", kernel) + re.findall(
                    r"(\w+ = __all_sync[^\n]*)", kernel) if "wait_bounded(" + bar in w or "wait_bounded(empty " in w]
                drained = [w for w in waits if "^ 1" not in w]
                assert any("rank == 0" not in w for w in drained), (re.search(r"k_\w+", kernel).group(0), bar, waits)
    assert kernels == 4
