"""A call whose launch fails half way still makes its stream wait for the kernels it
has forked onto the internal streams: the next call may overwrite the workspace they
read.  Run against a CUDA runtime that only logs (no GPU needed)."""
import os
import subprocess

import pytest

from paper_2301_09310_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
MAIN, AUX, JOIN = 1, range(100, 108), 200


@pytest.fixture(scope="module", params=["api", "bwa"])
def probe(request, tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("join") / "probe")
    # PTX only: the kernels are never run
    subprocess.run([build.nvcc(), "-gencode", "arch=compute_103a,code=compute_103a", "-O0", "-std=c++17",
                    "-cudart", "none", f"-I{build.INCLUDE}", f"-I{build.CSRC}",
                    os.path.join(HERE, f"join_{request.param}_probe.cu"),
                    os.path.join(HERE, "fake_cuda.cpp"), "-o", exe,
                    "-Xlinker", "--unresolved-symbols=ignore-all"], check=True, capture_output=True)

    def run(fail_at, branches):
        r = subprocess.run([exe, str(fail_at), str(branches)], capture_output=True, text=True, check=True)
        return [line.split() for line in r.stdout.splitlines()]

    return run


@pytest.mark.parametrize("branches", [1, 3, 8])
def test_forked_streams_are_joined(probe, branches):
    launches = sum(line[0] == "launch" for line in probe(-1, branches))
    assert launches >= 6
    for fail_at in [-1, *range(launches)]:
        log = probe(fail_at, branches)
        assert (log[-1] == ["status", "0"]) == (fail_at < 0)
        busy = {}  # stream -> place of its last launch in the log
        for at, line in enumerate(log):
            if line[0] == "launch" and int(line[1]) in AUX:
                busy[int(line[1])] = at
        for st, at in busy.items():
            ev = str(JOIN + st - AUX[0])
            rec = [k for k in range(at, len(log)) if log[k] == ["record", ev, str(st)]]
            assert rec and ["wait", str(MAIN), ev] in log[rec[0]:], (fail_at, st, log)
