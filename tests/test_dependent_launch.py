"""Kernels launched with sg_launch_pdl overlap the kernel before them on the
stream: what that kernel writes is not constant during their lifetime, so they
must not read it on the read-only path, which is what __ldg asks for and const
__restrict__ pointer arguments permit.  And an update kernel changes parameters
from its first finished CTA on, so whether the step counts must be settled before
it: a wait that may run out has no place there.  Read from the sources (no GPU)."""

import os
import re

import pytest

from paper_2305_04180_gb300 import build


def _strip(text):
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def _kernels():
    """{name: (arguments, body)} of every kernel that sg_launch_pdl launches."""
    text = "".join(_strip(open(os.path.join(build.CSRC, f)).read())
                   for f in sorted(os.listdir(build.CSRC)) if f.endswith(".cu"))
    names = set()
    for m in re.finditer(r"sg_launch_pdl\(([^;]*?);", text, flags=re.S):
        names |= set(re.findall(r"\bk_\w+", m.group(1).split("grid")[0]))
    out = {}
    for n in names:
        m = re.search(r"__global__[^;{}]*?\b%s\s*\(" % n, text)
        at = m.end()
        args = text[at:text.index("{", at)]
        i = text.index("{", at)
        depth, j = 0, i
        while True:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
            if depth == 0:
                break
        out[n] = (args, text[i:j])
    return out


KERNELS = _kernels()


def test_every_dependent_launch_is_found():
    assert {"k_td_tile", "k_td_tc", "k_td_update", "k_td_update_split", "k_step_finish"} <= set(KERNELS)


@pytest.mark.parametrize("name", sorted(KERNELS))
def test_no_read_only_loads_of_what_the_kernel_before_writes(name):
    args, body = KERNELS[name]
    assert "pdl_wait();" in body
    assert not re.search(r"const\s+[\w:]+\s*\*\s*__restrict__", args), "read-only pointer argument"
    assert "__ldg(" not in body


@pytest.mark.parametrize("name", [n for n in sorted(KERNELS) if "update" in n])
def test_updates_hold_no_wait_that_may_run_out(name):
    body = KERNELS[name][1]
    assert "mbar_wait" not in body and "kTcTries" not in body
    # the one failure word is read once, before any parameter is written
    assert body.count("u.fail") == 1 and body.index("u.fail") < body.index("upd_adam(")


@pytest.mark.parametrize("name", ["k_td_tile", "k_td_tc"])
def test_a_repeated_tile_is_gathered_behind_an_acquire(name):
    """A CTA that repeats its first tile with a later step counter has read rows
    that lie beside the new ones: its L1 must not answer for those."""
    body = KERNELS[name][1]
    assert len(re.findall(r"st = steps_sh\[1\];", body)) == 1
    assert re.search(r"st = steps_sh\[1\];\s*if \(tid == 0\) ring_steps\(rp\);\s*(__syncthreads|lt_sync)\(\);", body)
