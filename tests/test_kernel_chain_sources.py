"""The kernels of the likelihood's chain read what the kernels before them wrote,
and may be resident before those have finished (programmatic dependent launch).
So none of those reads may be declared read-only for the kernel's duration: the
compiler could then move them to before the wait on the kernel before."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_13196_gb300", "csrc")


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


@pytest.mark.parametrize("name", ["fg21_kernels.cu", "fg21_tc.cu", "fg21_noalloc.cu"])
def test_chain_memory_is_not_declared_unchanging(name):
    code = _code(name)
    assert not re.findall(r"ReqDesc\s*\*\s*__restrict__\s*\w*", code)
    assert not re.findall(r"__ldg\s*\([^;]*;|ld\.global\.nc|__restrict__ \w+ = r\.\w+", code)


def test_dependent_kernels_wait_before_they_read():
    """Every kernel launched as a dependent one calls pdl_wait() before it names its descriptors."""
    kernels, tc = _code("fg21_kernels.cu"), _code("fg21_tc.cu")
    launched = set(re.findall(r"launch_dependent\((\w+)<", kernels)) | set(re.findall(r"launch_dependent\((\w+)<", tc))
    launched.add("prep_tc_kernel")           # launched through a pointer to the chosen instantiation
    assert launched >= {"prep_tiles_kernel", "prep_tc_kernel", "simt_kernel", "reduce_kernel", "tc_loglike_kernel"}
    for k in launched:
        body = re.search(r"__global__[^;{]*?\b%s\([^{]*\{(.*?)\n\}" % k, kernels + tc, flags=re.S).group(1)
        wait = body.index("pdl_wait()")
        assert not re.search(r"\breqs\b|\bone\b|\br\.", body[:wait]), k
