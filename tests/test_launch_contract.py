"""Kernels that are launched through csrc/launch.cuh may come up before the kernel in front of them has finished (programmatic dependent launch), so each of
them has to wait for it; those that do not wait go through launch_beside, which never lets a kernel come up early.  On the GPU a missing wait shows only
where the overlap happens; here it is looked up in the sources."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2110_02987_b200", "csrc")


def sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = open(path).read()
        text = re.sub(r"//[^\n]*", "", text)
        yield os.path.basename(path), re.sub(r"/\*.*?\*/", "", text, flags=re.S)


def closing(text, at, pair):
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == pair[0]) - (text[i] == pair[1])
        if depth == 0:
            return i
    raise ValueError("unbalanced")


def kernels(text):
    """Name -> body of every __global__ function."""
    out = {}
    for m in re.finditer(r"__global__", text):
        head = re.compile(r"\b(\w+_kernel)\s*\(").search(text, m.end())
        end = closing(text, head.end() - 1, "()")
        brace = text.index("{", end)
        out[head.group(1)] = text[brace:closing(text, brace, "{}") + 1]
    return out


def launched_with_overlap(text):
    """Kernels named in the arguments of launch, launch_share, launch_tail, launch_spread and launch_cluster, in those of a local lambda around one of
    them, or in what such a lambda's kernel variable is set to."""
    names = set()
    for m in re.finditer(r"\b(?:launch|launch_share|launch_tail|launch_spread|launch_cluster|go)\s*\(", text):
        names |= set(re.findall(r"\b\w+_kernel\b", text[m.end():closing(text, m.end() - 1, "()")]))
    return names


CASES = [(f, k, body) for f, t in sources() for k, body in kernels(t).items() if k in launched_with_overlap(t)]


def test_the_launches_are_found():
    names = {k for _, k, _ in CASES}
    assert {"gemm_rows_kernel", "gemm_tn_kernel", "spmm_items_kernel", "spmm_finish_kernel", "reduce_chunks_kernel", "step_sums_consensus_kernel",
            "narrow_bwd_kernel", "small_rows_kernel", "split_weights_kernel"} <= names, names


def test_kernels_beside_never_come_up_early():
    text = open(os.path.join(CSRC, "launch.cuh")).read()
    body = text[text.index("launch_beside("):]
    assert "Early::kNever" in body[:body.index("\n}")]
    assert re.search(r"== st\.stream && early != Early::kNever\) \{", text)


@pytest.mark.parametrize("file,kernel,body", CASES, ids=[k for _, k, _ in CASES])
def test_a_kernel_that_may_come_up_early_waits(file, kernel, body):
    assert re.search(r"\bpdl_wait\(\)", body), "%s: %s does not wait for the kernel in front" % (file, kernel)
