"""Kernels that start before their predecessor on the stream has ended
(griddepcontrol): their sources, read on the CPU.  What such a kernel reads
may still be written while it is alive, so its value pointers must not be
declared read-only (const and __restrict__ together) nor loaded with __ldg,
and a load that is an asm of its own (__ldcs, through ld_stream) must go
through a pointer that depends on the wait."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2303_08953_gb300", "csrc")


def _kernels():
    """(name, parameters, body) of every kernel that calls wait_previous."""
    out = []
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith(".cu"):
            continue
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\(", src):
            i, depth = m.end(), 1
            while depth:
                depth += {"(": 1, ")": -1}.get(src[i], 0)
                i += 1
            params = src[m.end():i - 1]
            b, depth = src.index("{", i) + 1, 1
            e = b
            while depth:
                depth += {"{": 1, "}": -1}.get(src[e], 0)
                e += 1
            if "wait_previous()" in src[b:e]:
                out.append((m.group(1), params, src[b:e]))
    return out


KERNELS = _kernels()


def test_they_are_found():
    assert {k[0] for k in KERNELS} >= {"sell_kernel", "dot_tile_kernel", "dot_small_kernel",
                                       "reduce_parts_kernel", "update_kernel",
                                       "update_thin_kernel"}


@pytest.mark.parametrize("name,params,body", KERNELS, ids=[k[0] for k in KERNELS])
def test_the_wait_comes_first(name, params, body):
    # (compile-time declarations apart)
    body = re.sub(r"\s*(constexpr|static_assert)\b[^;]*;", "", body)
    assert re.match(r"\s*(sval \+= )?wait_previous\(\);\s*release_next\(\);", body)


@pytest.mark.parametrize("name,params,body", KERNELS, ids=[k[0] for k in KERNELS])
def test_no_value_pointer_is_declared_read_only(name, params, body):
    bad = re.findall(r"const\s+(?:double|float|T)\s*\*\s*__restrict__\s+\w+", params)
    assert not bad, bad
    # (row order and offsets are index arrays, complete before any launch)
    assert set(re.findall(r"__ldg\(\s*(\w+)", body)) <= {"sperm"}


def test_sell_rows_gather_x_with_plain_loads():
    src = open(os.path.join(CSRC, "k_spmv.cu")).read()
    helpers = src[src.index("sell_chunk("):src.index("sell_kernel(")]
    assert "__ldg(" not in helpers
    assert not re.search(r"const T\* __restrict__ x\b", helpers)
    assert "sval += wait_previous();" in src
