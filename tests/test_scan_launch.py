"""What the scan's launcher decides on the host, from the library's own code with the CUDA runtime replaced by fakes
(tests/fakes/scan_launch.cpp)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FORMAT = {"f32": 0, "i4": 1, "i8": 2, "bf16": 3}
STRIDED, BALANCED = 1, 2


@pytest.fixture(scope="module")
def decide(tmp_path_factory):
    """decide([(B, Hq, Hkv, rank, format, query bits, batch, pages, partition), ..]) -> [(partials, slots, CTAs, early build), ..]"""
    if not (shutil.which(NVCC) and shutil.which("g++")):
        pytest.skip("no compiler")
    d = tmp_path_factory.mktemp("scan_launch")
    csrc, inc = os.path.join(ROOT, "paper_2607_24555_b200", "csrc"), os.path.join(ROOT, "include")
    scan, exe = str(d / "scan.o"), str(d / "scan_launch")
    subprocess.run([NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O0", "-Xcicc", "-O0", "-Xptxas", "-O0", "-I", inc, "-I", csrc,
                    "-c", os.path.join(csrc, "scan.cu"), "-o", scan], check=True, capture_output=True)
    subprocess.run(["g++", "-std=c++17", "-I", inc, "-I", csrc, "-I", os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include"), "-o", exe,
                    os.path.join(ROOT, "tests", "fakes", "scan_launch.cpp"), scan, "-Wl,--unresolved-symbols=ignore-all"], check=True, capture_output=True)

    def run(cases):
        text = "\n".join(" ".join(str(x) for x in (*c[:4], FORMAT[c[4]], 1 if c[5] == 16 else 0, *c[6:])) for c in cases)
        out = subprocess.run([exe], input=text, check=True, capture_output=True, text=True, timeout=60).stdout.split("\n")[:-1]
        assert len(out) == len(cases)
        return [tuple(int(x) for x in line.split()) for line in out]
    return run


def test_partials_fit_their_row(decide):
    """The selector reads a problem's partials before it knows how many of them this sequence has."""
    cases = [(16, 4 * Hkv, Hkv, rank, "i4", 16, batch, pages, part) for Hkv in (1, 2, 3, 8) for rank in (8, 4, 2) for batch in (1, 2, 3, 5, 40)
             for pages in (1, 8, 9, 24, 40, 100, 1000) for part in (STRIDED, BALANCED)]
    for case, (partials, slots, _, _) in zip(cases, decide(cases)):
        assert 1 <= partials <= slots, (case, partials, slots)


def test_builds_start_beside_scans_that_leave_room(decide):
    """16-token pages: the CTAs of the scan that is launched, whichever it is, and those of the build (four page-heads each) take at
    most two places on an SM.  Wider pages: always, since the build lasts several times as long as the rest of the step."""
    cases = [(B, 4 * Hkv, Hkv, rank, fmt, 16 if dtype == "bf16" else 32, batch, pages, STRIDED) for B in (16, 32, 64) for Hkv in (1, 2, 8)
             for rank in (8, 2) for fmt, dtype in (("i4", "bf16"), ("i4", "f32"), ("i8", "bf16"), ("bf16", "bf16"), ("f32", "f32")) for batch in (1, 2, 4, 9, 40)
             for pages in (8, 100, 300, 576, 1100)]
    rooms = set()
    for case, (_, _, ctas, room) in zip(cases, decide(cases)):
        fits = ctas + -(-case[6] * case[2] // 4) <= 2 * 148
        assert room == (case[0] != 16 or fits), (case, ctas, room)
        rooms.add((case[0], case[4], case[5], room))
    assert {(16, f, d, r) for f, d in (("i4", 16), ("i4", 32), ("i8", 16), ("bf16", 16), ("f32", 32)) for r in (0, 1)} <= rooms
