"""The order in which a decode step enqueues its work, read off the library's own host code with the CUDA runtime and the kernel
launchers replaced by fakes (tests/fakes/step_runtime.cpp): no GPU, and any of the calls can be made to report an error."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if not (shutil.which(NVCC) and shutil.which("g++")):
        pytest.skip("no compiler")
    d = tmp_path_factory.mktemp("step_order")
    csrc, inc = os.path.join(ROOT, "paper_2607_24555_b200", "csrc"), os.path.join(ROOT, "include")
    api, fakes = str(d / "api.o"), os.path.join(ROOT, "tests", "fakes", "step_runtime.cpp")
    subprocess.run([NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-I", inc, "-I", csrc, "-c", os.path.join(csrc, "api.cu"), "-o", api],
                   check=True, capture_output=True)
    exe = str(d / "step_order")
    # what no decode step calls stays unresolved
    subprocess.run(["g++", "-std=c++17", "-I", inc, "-I", os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include"), "-o", exe, fakes, api,
                    "-Wl,--unresolved-symbols=ignore-all"], check=True, capture_output=True)
    return exe


def trace(program, early, append, call, nth):
    """[(step, operation)], the pairs (i, j) of which i is over before j starts, and what the steps returned."""
    out = subprocess.run([program, str(int(early)), str(int(append)), call, str(nth)], check=True, capture_output=True, text=True, timeout=60).stdout
    ops, before, returned = [], [], []
    stream, event, step = {}, {}, 0      # stream / event -> operations that are over when it is reached
    for line in out.splitlines():
        w = line.split()
        if w[0] == "step":
            step = int(w[1])
        elif w[0] == "op":
            done = stream.setdefault(w[2], set())
            before.append(set(done))
            done.add(len(ops))
            ops.append((step, w[1]))
        elif w[0] == "record":
            event[w[1]] = set(stream.setdefault(w[2], set()))
        elif w[0] == "wait":
            stream.setdefault(w[2], set()).update(event[w[1]])
        elif w[0] == "returns":
            returned.append(int(w[1]))
    return ops, before, returned


CALLS = [("none", 1)] + [(c, 1) for c in ("build", "scan", "select", "attend")] + [("record", 1), ("record", 2), ("wait", 1), ("wait", 2)]


@pytest.mark.parametrize("call,nth", CALLS)
@pytest.mark.parametrize("append", [False, True])
@pytest.mark.parametrize("early", [False, True])
def test_a_step_follows_all_of_the_step_before(program, early, append, call, nth):
    ops, before, returned = trace(program, early, append, call, nth)
    assert returned == [0 if call == "none" else -4, 0], returned
    first = [i for i, (s, _) in enumerate(ops) if s == 0]
    second = [i for i, (s, _) in enumerate(ops) if s == 1]
    assert [n for s, n in ops if s == 1 and n != "clear"] == (["build", "scan", "select", "attend"] if early else ["scan", "build", "select", "attend"])
    for j in second:
        assert set(first) <= before[j], (ops[j], [ops[i] for i in first if i not in before[j]])
    # arrivals that a broken-off step may have counted in part are cleared when nothing is left that counts
    if early and call != "none":
        clear = [i for i in first if ops[i][1] == "clear"]
        assert clear and all(i in before[clear[-1]] for i in first if ops[i][1] in ("build", "select"))
