"""What a kernel launched before the work ahead of it has ended has to keep to
(launch_after), read from the sources: it waits for that work (grid_wait); it
takes no pointer as `const __restrict__`, whose loads need not stay behind the
wait and may be served by a cache that does not see the writes ahead; and one
that allocates TMEM releases the next launch only behind a barrier that follows
the allocation, so that no later kernel's block can hold the columns it waits
for.
"""
import glob
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = "\n".join(re.sub(r"//[^\n]*", "", open(f).read())
                 for f in sorted(glob.glob(os.path.join(ROOT, "paper_2007_14283_gb300", "csrc", "*.cu*"))))
LAUNCHED = sorted(set(re.findall(r"launch_after\(\s*(k_\w+)", CODE)))


def balanced(text, at, opening, closing):
    """text from the bracket at `at` to the one that closes it."""
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == opening) - (text[i] == closing)
        if depth == 0:
            return text[at:i + 1]
    raise AssertionError("unbalanced")


def kernel(name):
    """(parameters, body) of a __global__ function."""
    for m in re.finditer(r"\b%s\s*\(" % name, CODE):
        head = CODE[max(0, m.start() - 200):m.start()]
        if "__global__" not in head.rsplit(";", 1)[-1].rsplit("}", 1)[-1]:
            continue
        params = balanced(CODE, m.end() - 1, "(", ")")
        brace = CODE.index("{", m.end() - 1 + len(params))
        return params, balanced(CODE, brace, "{", "}")
    raise AssertionError(name)


def check(params, body):
    assert "grid_wait()" in body and "grid_release()" in body
    for p in params.split(","):
        assert not ("__restrict__" in p and re.search(r"\bconst\b", p)), p
    if "tmem_alloc(" in body:
        release = body.index("grid_release()")
        assert "__syncthreads()" in body[body.index("tmem_alloc("):release]


def test_the_kernels_are_found():
    assert {"k_finalize", "k_shift_tc", "k_shift_f32_tc", "k_vmf_tc", "k_vmf_adj_tc"} <= set(LAUNCHED)


@pytest.mark.parametrize("name", LAUNCHED)
def test_launch_contract(name):
    check(*kernel(name))


def test_the_checker_sees_planted_breaches():
    ok = "{ tmem_alloc(slot, 512); __syncthreads(); grid_release(); grid_wait(); }"
    check("(const float* X, float* __restrict__ y)", ok)
    for params, body in (("(const float* __restrict__ X)", ok),
                         ("(const float* X)", "{ grid_release(); tmem_alloc(slot, 512); __syncthreads(); grid_wait(); }"),
                         ("(const float* X)", "{ tmem_alloc(slot, 512); grid_release(); __syncthreads(); grid_wait(); }"),
                         ("(const float* X)", "{ grid_release(); }")):
        with pytest.raises((AssertionError, ValueError)):
            check(params, body)
