"""A bounded wait that runs out in the row kernel and in the streaming kernel of calls with a bitmask, in the form that
tests/test_gpu_wait_expiry.py describes: a test-only build in a child process, one copy announced and never issued."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2607_20475_b200 import build as lib_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def child(path, env):
    if not os.path.exists(lib_build.WAITTEST_LIB):
        lib_build.build_waittest()
    run = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "wait_expiry", "child_paths.py"), path],
                         capture_output=True, text=True, timeout=600, cwd=ROOT, env={**os.environ, **env})
    assert run.returncode == 0, run.stdout[-2000:] + run.stderr[-2000:]
    line = [ln for ln in run.stdout.splitlines() if ln.startswith("RESULT ")][-1]
    r = json.loads(line[len("RESULT "):])
    sure = np.array(r["sure"])
    assert sure.sum() >= len(sure) - 1
    assert np.array_equal(np.array(r["sample"]["good"])[sure], np.array(r["oracle"])[sure])
    for name in ("sample", "verify", "topk"):
        if name in r:
            assert not any(r[name]["flagged"])
            for e in r[name]["withheld"]:
                # the call returned and its error is known; sticky until the workspace is initialised; then as before
                assert e["error"] & 1 and all(e["sticky"])
                assert e["recovered"] and not any(e["after"]) and not e["tickets"]
    return r


@pytest.mark.gpu
def test_row_kernel_reports_the_rows_whose_copy_never_came():
    r = child("row", {"SONIC_TEST_ROW": "1"})
    B = len(r["sample"]["good"])
    for i, e in enumerate(r["sample"]["withheld"]):
        row, part = i // 2, 3 * (i % 2)
        # (a greedy row's other parts report to the first)
        assert e["expired"] == [q == row for q in range(B)], (row, part)
        assert e["tokens"][row] == -1
        assert all(e["tokens"][q] == r["sample"]["good"][q] for q in range(B) if q != row)
    for i, e in enumerate(r["verify"]["withheld"]):
        assert e["expired"] == [q == i // 3 for q in range(3)], i
        assert all(t == -1 for t in e["tokens"][i // 3])
        assert all(e["tokens"][q] == r["verify"]["good"][q] for q in range(3) if q != i // 3)
    assert r["topk"]["withheld"][0]["expired"] == [False, True, False]


@pytest.mark.gpu
def test_masked_streaming_kernel_reports_every_row():
    r = child("masked", {})
    for e in r["sample"]["withheld"]:
        assert all(e["expired"]) and all(t == -1 for t in e["tokens"])
