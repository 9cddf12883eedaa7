"""Child process of tests/test_gpu_wait_expiry_paths.py: the test-only build of the library (waits give up after 4096 rounds, one
chosen copy is announced but never issued) on the paths that tests/wait_expiry/child.py does not take.  argv: "row" (the row
kernel; SONIC_TEST_ROW is set by the parent) or "masked" (the streaming kernel of calls with a bitmask).  No wait is unbounded,
nothing faults; what was seen is printed as one JSON line."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
sys.path.insert(0, ROOT)

import numpy as np
import torch

from paper_2607_20475_b200 import build as _build

_build.LIB = _build.WAITTEST_LIB           # before the binding loads the library
from oracle import oracle  # noqa: E402
from paper_2607_20475_b200 import binding, harness, workloads as wl  # noqa: E402
from tests.helpers import make_sample, pack_bits  # noqa: E402

WS_TEST_WITHHOLD = 100                      # header word of the test-only build
ROW_PARTS = 16                              # the row kernel numbers the parts of row r from r * 16


def sample_calls(masked):
    V, B = 40000, 7
    rng = np.random.default_rng(78)
    x = rng.standard_normal((B, V)).astype(np.float32) * 2
    mode = np.array([wl.GREEDY, wl.TOP_K | wl.TEMPERATURE, wl.TOP_P, wl.MIN_P | wl.TEMPERATURE, wl.TOP_K | wl.TOP_P, wl.TEMPERATURE, wl.TOP_K], np.uint32)
    kw = {}
    if masked:
        mode |= wl.GRAMMAR
        kw["bitmask"] = pack_bits(rng.random((B, V)) < np.array([.02, .5, 1, .02, .9, .1, .02])[:, None])
    return make_sample(x, mode, temperature=[1, .8, 1, 1.2, 1, .9, 1], top_k=[0, 40, 0, 0, 900, 0, 4000], top_p=[1, 1, .9, 1, .8, 1, 1],
                       min_p=[0, 0, 0, .05, 0, 0, 0], seed=np.arange(B) + 5, **kw)


class Call:
    """A device workload with its results as {name: array of one entry per row}, and what says that a row's wait ran out."""

    def __init__(self, dev, kind):
        self.dev, self.kind = dev, kind
        self.ws = dev.ws
        self.hdr = self.ws[:512].view(torch.int32)

    def run(self):
        self.dev.run()
        r = self.dev.results()
        if self.kind == "topk":
            return r[1].tolist(), (r[1] == -1).all(1).tolist()
        token = r["tokens"] if self.kind == "verify" else r["token"]
        return token.tolist(), ((r["flags"] & 16) != 0).tolist()


def observe(call, words):
    """words: what is withheld, one call each; after each the error is sticky until the workspace is initialised again."""
    good, flagged = call.run()
    out = {"good": good, "flagged": flagged, "withheld": []}
    for word in words:
        call.hdr[WS_TEST_WITHHOLD] = word
        torch.cuda.synchronize()
        tokens, expired = call.run()
        error = int(call.hdr[0].item())
        call.hdr[WS_TEST_WITHHOLD] = 0
        sticky = call.run()[1]
        binding.sonic_workspace_init(call.ws)
        again, after = call.run()
        tickets = bool(call.ws[512:512 + 4 * 4096].view(torch.int32).any().item())
        out["withheld"].append({"tokens": tokens, "expired": expired, "error": error, "sticky": sticky, "recovered": again == good,
                                "after": after, "tickets": tickets})
    return out


def main(path):
    binding.lib()
    out = {}
    w = sample_calls(path == "masked")
    ref = oracle.sample(w)
    if path == "row":
        out["sample"] = observe(Call(harness.DeviceSample(w), "sample"), [r * ROW_PARTS + p + 1 for r in range(w.B) for p in (0, 3)])
        vw = wl.config4(B=3, K=2, V=32003)
        vw.sample.top_k[0] = 0
        vw.sample.mode[0] &= ~np.uint32(wl.TOP_K)
        out["verify"] = observe(Call(harness.DeviceVerify(vw), "verify"), [r * ROW_PARTS + 1 + 1 for r in range(9)])
        tw = wl.TopKWorkload(name="t", B=3, V=32003, dtype=wl.DTYPE_F32, logits=np.random.default_rng(1).standard_normal((3, 32003)).astype(np.float32))
        out["topk"] = observe(Call(harness.DeviceTopK(tw, 700), "topk"), [1 * ROW_PARTS + 2 + 1])
    else:
        tiles = (w.V + 8191) // 8192
        # (not the last row: nothing is copied for the tiles of the cluster kernel's rows)
        out["sample"] = observe(Call(harness.DeviceSample(w), "sample"), [2 * tiles + 1 + 1, 0 * tiles + 1, 4 * tiles + 4 + 1])
    out["sure"] = (ref["margin"] >= 1e-6).tolist()
    out["oracle"] = ref["token"].tolist()
    print("RESULT " + json.dumps(out))


if __name__ == "__main__":
    main(sys.argv[1])
