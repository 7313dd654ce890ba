"""Host arithmetic of the digit products' workspace (csrc/digit_ws.h): what setup allocates for a batch
holds every launch of that batch, the panel solves included, whose planes span a full panel of 64
columns however few are eliminated.  Through a host-only build of the same header."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2101_02959_gb300", "csrc")
PANEL, SLICE_K = 64, 1024
DIMS = {"d": (7, 128), "f": (3, 64)}  # digits, columns of a scaling group


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("ws") / "digit_ws")
    src = os.path.join(ROOT, "tests", "native", "digit_ws_harness.cu")
    r = subprocess.run([nvcc, "-std=c++17", "-I", CSRC, "-gencode", "arch=compute_103a,code=sm_103a", src,
                        "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


def _parts(t, rows, cols):
    """Bytes of one matrix's row planes, inverse planes, row exponents, inverse exponents."""
    digits, group = DIMS[t]
    padded = -(-rows // 128) * 128
    block = 64 * 32 * 2
    return ((-(-cols // 32)) * digits * (padded // 64) * block, (PANEL // 32) * digits * block,
            (-(-cols // group)) * padded * 4, 64 * 4)


@pytest.mark.parametrize("t", ["d", "f"])
def test_workspace_holds_every_launch(harness, t):
    queries = []
    for count in (1, 2, 5, 304):
        for e in (1, 2, 18, 31, 32, 33, 63, 64, 65, 127, 128, 129, 700, 1024, 1030):
            for rows in (e, 2 * e, 2 * e + 131):
                # the panel solve, the in-block and outer updates (at most e columns), the final one
                for cols in {PANEL, min(e, 128), min(e, 512), min(e, SLICE_K)}:
                    queries.append((t, count, rows, e, cols))
    text = "\n".join(" ".join(map(str, q)) for q in queries)
    r = subprocess.run([harness], input=text, capture_output=True, text=True, check=True)
    lines = r.stdout.strip().splitlines()
    assert len(lines) == len(queries)
    for q, line in zip(queries, lines):
        ws, run, inv, ex, ex_inv, end = map(int, line.split())
        assert 1 <= run <= q[1], q
        at = 0
        for got, part in zip((inv, ex, ex_inv, end), _parts(t, q[2], q[4])):
            at += run * part
            assert got == at, q
        assert end <= ws, q


def test_small_class_needs_a_whole_panel(harness):
    """One deluxe class of order 18 (two subdomains that share 3 x 3 nodes)."""
    for t in "df":
        r = subprocess.run([harness], input=f"{t} 1 36 18 64", capture_output=True, text=True, check=True)
        assert int(r.stdout.split()[0]) >= sum(_parts(t, 36, 64))
