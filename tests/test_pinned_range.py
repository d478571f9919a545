"""Which host ranges the library lets a kernel address: those that are page-locked throughout. The
arithmetic alone, on made-up address spaces (no GPU, no such buffer is handed to a kernel)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def view(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("pinned") / "pinned_range")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-O1", os.path.join(ROOT, "tests", "pinned_range_program.cpp"),
                    "-o", exe], check=True)

    def call(spans, at, nbytes):
        text = ",".join(":".join(str(v) for v in s) for s in spans)
        return int(subprocess.run([exe, text, str(at), str(nbytes)], check=True, capture_output=True, text=True).stdout)
    return call


ONE = [(4096, 4096, 8192)]
HOLE = [(4096, 4096, 4096), (16384, 16384, 4096)]          # page-locked at both ends, pageable in between
JOINED = [(4096, 4096, 4096), (8192, 8192, 100), (8292, 8292, 4096)]
MOVED = [(4096, 50_000, 8192)]                             # device addresses of their own
APART = [(4096, 50_000, 4096), (8192, 90_000, 4096)]       # neighbours for the host, not for the device


@pytest.mark.parametrize("spans,at,nbytes,device", [
    (ONE, 4096, 8192, 4096), (ONE, 4097, 8191, 4097), (ONE, 12287, 1, 12287),          # up to the last byte
    (ONE, 4097, 8192, 0), (ONE, 4095, 2, 0), (ONE, 12288, 1, 0), ([], 4096, 1, 0),
    (HOLE, 4096, 16384, 0), (HOLE, 8191, 8194, 0), (HOLE, 4096, 4097, 0), (HOLE, 16384, 4096, 16384),
    (JOINED, 4096, 8292, 4096), (JOINED, 8191, 102, 8191), (JOINED, 4096, 8293, 0),
    (MOVED, 4100, 8188, 50_004), (MOVED, 4100, 8189, 0),
    (APART, 4096, 4096, 50_000), (APART, 8192, 4096, 90_000), (APART, 8191, 2, 0),
])
def test_range_is_page_locked_throughout(view, spans, at, nbytes, device):
    assert view(spans, at, nbytes) == device
