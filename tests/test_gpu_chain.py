"""The chain of kernels of large calls on the small calls of the other tests: they are written for its edges (tiles cut into parts,
crowded crossing bins, list entries in one tile, thousands of rows, residual passes), but in the library itself calls of few rows
are one launch of the row kernel.  The trace variant of the library sends every call through the chain; here those tests run once
more against it, in a child process.  And one workspace shared by calls of both kinds."""
import os
import re
import subprocess
import sys

import numpy as np
import pytest

from paper_2607_20475_b200 import build as lib_build, workloads as wl

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = ("import sys, pytest; from paper_2607_20475_b200 import build; build.LIB = build.TRACE_LIB; "
         "sys.exit(pytest.main(sys.argv[1:]))")


# (left out: what an infinite processed logit gives is defined for the row kernel alone)
@pytest.mark.parametrize("files", [["test_gpu_dense.py"], ["test_gpu_more.py"], ["test_gpu_fuzz.py"], ["test_gpu_parity.py"],
                                   ["test_gpu_rows.py", "-k", "not overflow"]])
def test_the_chain_passes_the_tests_of_small_calls(files):
    lib_build.build_trace()
    run = subprocess.run([sys.executable, "-c", CHILD, "-q", "-x", "-m", "gpu", "-p", "no:cacheprovider",
                          os.path.join(ROOT, "tests", files[0]), *files[1:]],
                         capture_output=True, text=True, timeout=900, cwd=ROOT)
    assert run.returncode == 0, run.stdout[-4000:] + run.stderr[-1000:]
    assert int(re.search(r"(\d+) passed", run.stdout).group(1)) > 0 and "skipped" not in run.stdout, run.stdout[-500:]


def test_calls_of_both_kinds_share_one_workspace():
    # one row-kernel call and one call of the chain of every operation, replayed in turn from graphs: each leaves the workspace's
    # header as the others need it
    import torch
    from oracle import oracle
    from paper_2607_20475_b200 import harness
    from tests.parity import compare_sample, compare_topk, compare_verify
    few, many = wl.config2(B=5, V=30000), wl.config2(B=90, V=30000)
    vfew, vmany = wl.config4(B=3, K=2, V=20000), wl.config4(B=30, K=2, V=20000)
    for v in (vfew, vmany):
        v.sample.top_k[::2] = 0
        v.sample.mode[::2] &= ~np.uint32(wl.TOP_K)
    x = np.random.default_rng(2).standard_normal((90, 20000)).astype(np.float32)
    tops = [wl.TopKWorkload(name="t", B=n, V=20000, dtype=wl.DTYPE_F32, logits=x[:n]) for n in (4, 90)]
    nbytes = max(harness.sonic_workspace_bytes(90, 30000), harness.sonic_workspace_bytes(90, 20000, 3000))
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    harness.sonic_workspace_init(ws)
    devs = [harness.DeviceSample(few, ws=ws), harness.DeviceSample(many, ws=ws), harness.DeviceVerify(vfew, ws=ws), harness.DeviceVerify(vmany, ws=ws),
            harness.DeviceTopK(tops[0], 300, ws=ws), harness.DeviceTopK(tops[1], 3000, ws=ws)]

    def results(d):
        r = d.results()
        return r if isinstance(r, dict) else dict(vals=r[0], idx=r[1])

    first, graphs = [], []
    for d in devs:
        d.run()
        first.append(results(d))
    for w, f in zip((few, many), first[:2]):
        compare_sample(f, oracle.sample(w), w)
    for v, f in zip((vfew, vmany), first[2:4]):
        compare_verify(f, oracle.verify(v), v, max_near=v.B)
    for t, k, f in zip(tops, (300, 3000), first[4:]):
        compare_topk(f["vals"], f["idx"], *oracle.topk(t.logits_f32(), k))
    for d in devs:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            d.run()
        graphs.append(g)
    order = np.random.default_rng(3).integers(0, len(devs), 600)
    for i, c in enumerate(order):
        graphs[c].replay()
        if i % 29 == 0 or i >= 580:
            again = results(devs[c])
            for key in first[c]:
                assert np.array_equal(first[c][key], again[key]), (i, c, key)
    assert not ws[512:512 + 4 * 4096].view(torch.int32).any()
    hdr = ws[:32].view(torch.int32).cpu().numpy()
    assert not hdr[[0, 2, 3, 4, 5, 6, 7]].any(), hdr[:8]
