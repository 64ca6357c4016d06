"""Codes of the bounded waits: each kernel has its own, and pico_sync names it.

No wait is made to run out: the codes are read from the sources, and the message
from a status word that the host sets.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_09590_gb300", "csrc")


def test_no_two_kernels_share_a_code():
    head = open(os.path.join(CSRC, "kernels.cuh")).read()
    enum = dict(re.findall(r"\b(kWait\w+) = (\d+)", head))
    assert len(set(enum.values())) == len(enum)
    owner = {}
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        kernel = ""
        for line in open(os.path.join(CSRC, name)):
            m = re.search(r"\b(k_[a-z0-9_]+)\(", line)
            if m:
                kernel = m.group(1)
            for code in re.findall(r"atomicCAS\([a-z.]*err, 0, (\w+)\)", line) + \
                    re.findall(r"set_err\([a-z.]*err, (\w+)\)", line):
                if code == "code":       # the helper itself
                    continue
                if code.isdigit():       # gram.cu and colcg_persist.cu number theirs in a range of their own
                    lo, hi = {"gram.cu": ("kWaitGramFirst", "kWaitGramLast"),
                              "colcg_persist.cu": ("kWaitPersistFirst", "kWaitPersistLast")}[name]
                    assert int(enum[lo]) <= int(code) <= int(enum[hi])
                else:
                    assert owner.setdefault(code, (name, kernel)) == (name, kernel), code
    assert len(owner) == 5


@pytest.mark.gpu
@pytest.mark.parametrize("code,text", [(3, "Gram"), (10, "column pass"), (11, "exchange"), (12, "inverse row pass"),
                                       (13, "row adjoint"), (14, "forward row pass"), (22, "per-column CG")])
def test_sync_names_the_wait(code, text):
    import paper_2605_09590_gb300 as pico
    import synth
    op = pico.Operator(synth.coil_maps(64, 48, 2, 3), mask=synth.mask_pe(64, 2, 4), power_iters=0, max_batch=2)
    pico.pico_inject_error(op.ctx, pico.PICO_E_TIMEOUT, code)
    with pytest.raises(pico.PicoError) as ei:
        op.sync()
    assert ei.value.status == pico.PICO_E_TIMEOUT
    assert f"code {code}: " in str(ei.value) and text in str(ei.value)
    op.sync()
    op.close()
