"""The kernels of the likelihood's chain read what the kernels before them wrote,
and may be resident before that is visible (programmatic dependent launch).  So no
such read may be one that the compiler can move to before the wait on the kernel
before: a load through a __restrict__ kernel parameter, or an __ldg, whose address
is known before the wait."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_13196_gb300", "csrc")


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


ALL = "\n".join(_code(f) for f in ("fg21_kernels.cu", "fg21_tc.cu", "fg21_noalloc.cu"))


def _function(name):
    """(parameters, body) of a function by name."""
    m = re.search(r"\b%s\(([^;{]*?)\)\s*\{(.*?)\n\}" % name, ALL, flags=re.S)
    assert m, name
    return m.group(1), m.group(2)


DEPENDENT = sorted(set(re.findall(r"launch_dependent\((\w+)<", ALL)) | {"prep_tc_kernel"})   # (launched by pointer)


def test_dependent_kernels_are_found():
    assert set(DEPENDENT) == {"prep_tiles_kernel", "prep_tc_kernel", "simt_kernel", "reduce_kernel", "tc_loglike_kernel"}


@pytest.mark.parametrize("kernel", DEPENDENT)
def test_descriptor_is_read_after_the_wait(kernel):
    params, body = _function(kernel)
    wait = body.index("pdl_wait()")
    assert not re.search(r"\breqs\b|\bone\b|\br\.", body[:wait])
    if kernel == "prep_tc_kernel":
        # reads reqs of several requests only (there before the call's first kernel), one request by value
        assert "ONE ? one : reqs[blockIdx.y]" in body and not re.search(r"\breqs\b", body.replace("reqs[blockIdx.y]", ""))
    else:
        assert not re.search(r"ReqDesc\s*\*\s*__restrict__", params)
        assert not re.search(r"ReqDesc\s*\*\s*__restrict__", body)


def test_by_value_descriptors_are_followed_by_plain_loads():
    """Where the descriptor is a kernel argument, addresses are known before the wait."""
    by_value = {n for n, params in re.findall(r"__global__[^;{]*?\b(\w+_kernel)\(([^{;]*)\)\s*\{", ALL)
                if re.search(r"__grid_constant__ (const )?ReqDesc|const ReqDesc r\b", params)}
    assert by_value == {"prep_stats_kernel", "prep_tc_kernel", "store_desc_kernel"}
    for f in by_value | {"gather_stats", "row_stats", "finish_stats", "prep_finalize", "prep_points", "begin_call"}:
        params, body = _function(f)
        assert "__ldg" not in body and "ld.global.nc" not in body, f
        assert not re.search(r"__restrict__ \w+ = r\.", body), f
