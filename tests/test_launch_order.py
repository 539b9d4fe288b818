"""The order of programmatically launched kernels, by their source.

Such a kernel lets the next one start at its own top (pdl_trigger), and the
next one's pdl_wait covers this grid alone: "every earlier kernel has
finished" holds only if CTAs of every grid pass pdl_wait before they end.  So
none leaves before it, but groups of rows past a launch's end: the first group
of a launch never is one."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2305_17341_gb300", "csrc")


def _kernels():
    """(file, kernel, body) of every __global__ function that calls pdl_trigger."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(", text):
            i = text.index("{", m.end())
            depth, j = 1, i + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[j], 0)
                j += 1
            body = text[i:j]
            if "pdl_trigger()" in body:
                out.append((os.path.basename(path), m.group(1), body))
    return out


KERNELS = _kernels()


def test_the_kernels_are_found():
    assert {"k_ntt_fwd_fast", "k_ntt_inv_fast", "k_msum", "k_multsum_giants", "k_relin_ms", "k_relin_up",
            "k_modup_bconv", "k_moddown_bconv", "k_pmul_acc"} <= {k for _, k, _ in KERNELS}


@pytest.mark.parametrize("file,kernel,body", KERNELS, ids=[k for _, k, _ in KERNELS])
def test_no_cta_leaves_before_the_wait(file, kernel, body):
    rest = re.sub(r"pdl_wait\(\);\s*return;", "", body)   # leaving after the wait
    rest = re.sub(r"if \((ROWS && )?pm\.row >= nr\) return;", "", rest)
    wait = re.search(r"(?<!\) )pdl_wait\(\);", rest)      # an unconditional one
    assert wait, (file, kernel)
    assert not re.search(r"\breturn\b", rest[:wait.start()]), (file, kernel)
