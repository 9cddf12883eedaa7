"""GPU parity test of the streaming kernel of calls without sparse lists (no list code, a four-stage ring for bf16): one tile per row to
more tiles than stages, partial last tiles; zeros of both signs, subnormals, the lowest and the highest finite values, ties, rows
with fewer finite entries than asked for."""
import numpy as np
import pytest

from paper_2607_20475_b200 import workloads as wl
from tests.helpers import make_sample
from tests.parity import compare_sample, compare_topk

pytestmark = pytest.mark.gpu


def rounded(x):
    return wl.bf16_bits_to_f32(wl.f32_to_bf16_bits(x))


def rows_of_extremes(rng, B, V):
    x = rounded((rng.standard_normal((B, V)) * 2).astype(np.float32))
    x[1::8] = np.round(x[1::8])                                                    # ties
    x[2::8] = rng.choice(np.array([0.0, -0.0, 9.2e-41, -9.2e-41], np.float32), (len(x[2::8]), V))      # 9.2e-41: the smallest subnormal
    x[3::8] = -np.inf
    x[3::8, ::997] = rng.standard_normal(x[3::8, ::997].shape)
    x[4::8] = -3.3895314e38                                                        # the lowest finite value
    x[4::8, V // 2] = 3.3895314e38
    x[5::8, :min(V, 8192)] = -np.inf
    x[6::8] = -np.abs(x[6::8]) * 1e30
    return rounded(x)


@pytest.mark.parametrize("V", [8191, 8192, 16384, 16385, 24576, 40000])
@pytest.mark.parametrize("dtype", [wl.DTYPE_F32, wl.DTYPE_BF16])
def test_calls_without_lists(V, dtype):
    from oracle import oracle
    from paper_2607_20475_b200 import harness
    B = 80                                                       # more clusters of the row kernel than are resident: the chain
    rng = np.random.default_rng(V)
    x = rows_of_extremes(rng, B, V)
    tw = wl.TopKWorkload(name="t", B=B, V=V, dtype=dtype, logits=x if dtype == wl.DTYPE_F32 else wl.f32_to_bf16_bits(x))
    for k in (1, 7, 64, 300, 2500):
        dev = harness.DeviceTopK(tw, k)
        dev.run()
        compare_topk(*dev.results(), *oracle.topk(x, k))
    mode = np.array([wl.TOP_K | wl.TEMPERATURE | wl.TOP_P, wl.TOP_K, wl.TOP_K | wl.TEMPERATURE, wl.GREEDY])[np.arange(B) // 8 % 4]
    # (temperature at or above 1: max / 0.8 would leave the range of finite values, 4.2e38 > 3.4e38, which is not what this test is about)
    w = make_sample(x, mode, dtype=dtype, temperature=np.full(B, 1.25), top_k=np.full(B, 50), top_p=np.full(B, 0.9),
                    seed=np.arange(B) + V, offset=np.arange(B))
    dev = harness.DeviceSample(w)
    dev.run()
    compare_sample(dev.results(), oracle.sample(w), w, max_near=B)
