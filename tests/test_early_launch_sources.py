"""Kernels that may start before the kernel ahead of them has finished (those that call
launch_wait()) must not read what that kernel writes through loads that are taken for
read-only: such loads may move above the wait, or be served from lines cached before it.  A
wrong one need not show up in results, so the sources themselves are checked."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1905_00444_gb300", "csrc")


def early_kernels():
    """(name, parameter list, body) of every kernel whose body calls launch_wait()."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\b", text):
            name = re.compile(r"(\w+_kernel)\s*\(").search(text, m.end())
            depth, i = 1, name.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(text[i], 0)
                i += 1
            params = text[name.end():i - 1]
            start = text.index("{", i)
            depth, j = 1, start + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[j], 0)
                j += 1
            body = text[start:j]
            if "launch_wait()" in body:
                out.append((name.group(1), params, body))
    return out


def test_the_early_kernels_are_found():
    names = {k[0] for k in early_kernels()}
    assert {"cgemm_pair_kernel", "split_site_kernel", "cgemm_step_kernel", "small_parts_kernel", "fold_kernel",
            "fold_scale_kernel", "accumulate_kernel", "grads_kernel", "fold_backward_kernel"} <= names


@pytest.mark.parametrize("kernel", early_kernels(), ids=lambda k: k[0])
def test_no_read_only_loads(kernel):
    assert not re.search(r"__ldg|ld\.global\.(\w+\.)*nc", kernel[2])


# the plan's tables, which a copy ahead of the call's first kernel has written
TABLES = {"FoldSite": {"sites"}, "FoldEvent": {"events"}, "float": {"matsf"}, "CutDev": {"cuts"},
          "int32_t": {"open_perm", "gate_ev"}, "int64_t": {"part_off"}}


@pytest.mark.parametrize("kernel", early_kernels(), ids=lambda k: k[0])
def test_restrict_is_for_tables_only(kernel):
    for param in kernel[1].split(","):
        if "__restrict__" in param:
            kind, name = re.fullmatch(r"\s*const\s+(\w+)\s*\*\s*__restrict__\s+(\w+)\s*", param).groups()
            assert name in TABLES.get(kind, ()), param


@pytest.mark.parametrize("kernel", early_kernels(), ids=lambda k: k[0])
def test_successors_start_behind_the_wait(kernel):
    """A kernel that lets its successor start before its own wait lets the whole chain become
    resident at once, which crowds the blocks of small grids onto some of the SMs."""
    body = kernel[2]
    assert body.count("launch_wait()") == 1
    if "launch_next()" in body:
        assert body.index("launch_wait()") < body.index("launch_next()")
