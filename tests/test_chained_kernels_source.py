"""The sources of the chained kernels (csrc/chain.cuh): a kernel of a step is
resident while the kernels before it still write, and waits in its first
statement.  What the compiler may move above that wait is not visible in any
result, so the rules are held on the text: every kernel that launch_chained
starts opens with after_previous(); none of its pointers carries __restrict__
(an access through one is not ordered by the wait, and a load through a const
one may be non-coherent), but for a batch's descriptors and tile lists, which no
kernel writes; and nothing is loaded by __ldg, whose target may not change while
the kernel is resident."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_20461_gb300", "csrc")
CONSTANT = {"gd", "tiles"}


def _sources():
    out = {}
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(f) as fh:
            out[os.path.basename(f)] = re.sub(r"/\*.*?\*/|//[^\n]*", " ", fh.read(), flags=re.S)
    return out


def _kernels():
    """name -> (file, parameters, body's beginning)"""
    out = {}
    for f, s in _sources().items():
        for m in re.finditer(r"__global__", s):
            depth, i, last = 0, m.end(), 0  # last: where the last outermost parenthesis (the parameters) opens
            while depth or s[i] not in "{;":
                if s[i] == "(":
                    last, depth = (i if depth == 0 else last), depth + 1
                elif s[i] == ")":
                    depth -= 1
                i += 1
            if s[i] == "{":
                out[re.search(r"(\w+)\s*$", s[:last]).group(1)] = (f, s[last:i], s[i + 1 : i + 600])
    return out


KERNELS = _kernels()
LAUNCHED = sorted({n for s in _sources().values() for call in re.findall(r"launch_chained\(([^;]*);", s)
                   for n in re.findall(r"\w+", call) if n in KERNELS})


def test_the_chained_kernels_are_found():
    assert {"cell_poly_kernel", "step_flux_kernel", "step_update_kernel", "dt_from_speed_kernel", "step1d_kernel",
            "step1d_short_kernel", "nc_stage_kernel", "nc_short_kernel", "bk_poly", "bk_flux", "bk_update"} <= set(LAUNCHED)


@pytest.mark.parametrize("name", LAUNCHED)
def test_waits_first_and_orders_every_pointer(name):
    f, sig, body = KERNELS[name]
    first = [st.strip() for st in body.split(";")]
    first = next(st for st in first if not re.match(r"(constexpr|__shared__)", st))
    assert first == "after_previous()", (f, first)
    assert set(re.findall(r"__restrict__\s+(\w+)", sig)) <= CONSTANT, f


def test_item_functions_do_not_bring_the_promise_back():
    """the functions inlined into these kernels (csrc/*.cuh, k1d_nc.cu): no __restrict__ pointer parameter"""
    for f in ("chain.cuh", "kernels.cuh", "step_flux.cuh", "step_1d.cuh", "k1d_nc.cu"):
        for sig in re.findall(r"__device__ __forceinline__ [^{;]*{", _sources()[f]):
            assert "__restrict__" not in sig, (f, sig[:80])


def test_no_load_that_assumes_constant_memory():
    for f, s in _sources().items():
        assert "__ldg" not in s and "ld.global.nc" not in s, f
