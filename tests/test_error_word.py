"""Who may write the workspace's error word and when, read from the kernels'
sources on CPU. The advantage kernel, the call's first, resets the word; the
sweep is launched as its programmatic dependent and runs beside it. A wait of
the sweep that runs out before the reset must not be lost to it, so every
record of one waits for the advantage kernel. (The shortest stall that the test
hook can make is some 250 us, long past the reset: the outputs of a run do not
show the order.)"""

import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2609_08368_gb300", "csrc")


def _source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def test_a_timeout_is_recorded_after_the_advantage_kernel():
    helper = re.search(r"void record_timeout\(uint32_t\* err\) \{([^}]*)\}", _source("common.cuh")).group(1)
    assert re.fullmatch(r"\s*pdl_wait\(\);\s*atomicOr\(err, kErrTimeout\);\s*", helper)
    uses = []
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        name = os.path.basename(path)
        uses += [name for _ in re.finditer(r"\bkErrTimeout\b", _source(name))]
    assert uses == ["common.cuh"] * 2  # its definition and the helper


def test_the_sweeps_write_other_errors_after_their_wait():
    for name, kernel in (("k_short.cuh", "k_short"), ("k_sweep.cuh", "k_sweep"),
                         ("k_stream.cuh", "k_stream")):
        src = _source(name)
        body = src[re.search(r"__global__ .*\b" + kernel + r"\(", src).end():]
        for m in re.finditer(r"atomicOr\(", body):
            assert "pdl_wait()" in body[:m.start()], (kernel, body[m.start():m.start() + 60])
