"""GPU parity test of the streaming kernel of calls with a grammar bitmask, at the sizes where it can go wrong: vocabularies at
the edges of a tile and of a mask word; masks of a few ids, of one id, of whole empty tiles, dense ones and rows without the mode
bit; histories below, at and beyond what a CTA keeps in shared memory."""
import numpy as np
import pytest

from paper_2607_20475_b200 import workloads as wl
from tests.helpers import make_sample, pack_bits
from tests.parity import compare_sample

pytestmark = pytest.mark.gpu

T = wl.TEMPERATURE
KINDS = [(wl.GREEDY, 0), (wl.GREEDY | T, 0), (wl.TOP_K | T, 1), (wl.TOP_K | T, 50), (wl.TOP_K | T | wl.TOP_P, 100), (wl.TOP_K, 1000),
         (wl.TOP_P | T, 0), (wl.MIN_P, 0), (wl.TOP_K | wl.MIN_P, 20)]
HISTORY = [0, 1, 511, 512, 513, 700]


@pytest.mark.parametrize("V", [8191, 8192, 8193, 9000, 20001, 32800])
@pytest.mark.parametrize("dtype", [wl.DTYPE_F32, wl.DTYPE_BF16])
def test_masked_batches(V, dtype):
    from oracle import oracle
    from paper_2607_20475_b200 import harness
    B = 80                                                       # more clusters of the row kernel than are resident: the chain
    rng = np.random.default_rng(V * 2 + dtype)
    x = (rng.standard_normal((B, V)) * 2).astype(np.float32)
    mode = np.array([KINDS[r % len(KINDS)][0] for r in range(B)], np.uint32)
    k = np.array([KINDS[r % len(KINDS)][1] for r in range(B)])
    share = np.array([0.02, 0.002, 0.5, 0.98])[rng.integers(0, 4, B)]
    allowed = rng.random((B, V)) < share[:, None]
    allowed[5::16, :min(V - 1, 8192)] = False                    # nothing in the first tile
    allowed[6::16, 4096:] = False                                # nothing beyond the first half tile
    allowed[7::16] = False                                       # the last id alone
    allowed[np.arange(B), np.where(np.arange(B) % 16 == 6, 0, V - 1)] = True
    mode[rng.random(B) < 0.8] |= wl.GRAMMAR
    lists = rng.random(B) < 0.7
    mode[lists] |= wl.REPETITION | wl.FREQUENCY | wl.PRESENCE | wl.BIAS
    hist = [{int(i): int(c) for i, c in zip(rng.choice(V, HISTORY[r % 6], replace=False), rng.integers(1, 5, HISTORY[r % 6]))}
            for r in range(B)]
    bias = [{int(i): float(b) for i, b in zip(rng.choice(V, 8, replace=False), rng.uniform(-4, 4, 8))} for _ in range(B)]
    w = make_sample(x, mode, dtype=dtype, temperature=rng.uniform(0.6, 1.4, B), top_k=k, top_p=np.full(B, 0.9), min_p=np.full(B, 0.05),
                    rep=np.full(B, 1.2), freq=np.full(B, 0.2), pres=np.full(B, 0.3), bitmask=pack_bits(allowed), hist=hist, bias=bias,
                    seed=np.arange(B) + V, offset=np.arange(B) * 5)
    dev = harness.DeviceSample(w)
    dev.run()
    got = dev.results()
    compare_sample(got, oracle.sample(w), w, max_near=B)          # (each near-margin row is held to an admissible outcome)
    dev.run()
    again = dev.results()
    for key in got:
        assert np.array_equal(got[key], again[key]), key


@pytest.mark.parametrize("temperature", [1.0, 0.7, 1e38, 1e-39, 1e-40])
@pytest.mark.parametrize("dtype", [wl.DTYPE_F32, wl.DTYPE_BF16])
def test_masked_greedy_rows(dtype, temperature):
    # dense, sparse and missing masks; logits a few units in the last place apart, which an extreme temperature makes equal (the
    # lowest index wins) or sends to -inf (no token)
    from oracle import oracle
    from paper_2607_20475_b200 import harness
    B, V = 80, 20001
    rng = np.random.default_rng(9)
    x = rng.standard_normal((B, V)).astype(np.float32)
    step = 2.0 ** -22 if dtype == wl.DTYPE_F32 else 2.0 ** -8
    x[::4] = np.float32(0.1) * (1 + np.arange(V) * np.float32(step) / 64)
    x[1::4] = -np.float32(0.3) * (1 + np.arange(V)[::-1] * np.float32(step) / 64)
    if temperature < 1e-30:
        x = -np.abs(x)
        x[::8, 777] = -2 * temperature
    allowed = rng.random((B, V)) < np.array([0.02, 0.3, 0.9, 1.0])[rng.integers(0, 4, B)][:, None]
    mode = np.full(B, wl.GREEDY | wl.TEMPERATURE, np.uint32)
    mode[rng.random(B) < 0.7] |= wl.GRAMMAR
    w = make_sample(x, mode, dtype=dtype, temperature=np.full(B, temperature), bitmask=pack_bits(allowed))
    dev = harness.DeviceSample(w)
    dev.run()
    compare_sample(dev.results(), oracle.sample(w), w)


@pytest.mark.parametrize("share", [0.3, 1.0])
@pytest.mark.parametrize("dtype", [wl.DTYPE_F32, wl.DTYPE_BF16])
def test_masked_rows_whose_values_depend_on_the_position(dtype, share):
    # the cutoff that a CTA keeps from its first tile of a row lies far below a later tile's values: the rows have to be right, and
    # but for the few that miss their proof (half the row is as good as not there) the merge has to finish them
    from oracle import oracle
    from paper_2607_20475_b200 import harness
    B, V = 128, 131072                                             # (several tiles of a row in a CTA)
    rng = np.random.default_rng(17)
    x = rng.standard_normal((B, V)).astype(np.float32)
    x[0::2, V // 2:] += 6                                          # the second half
    x[1::2] += 6 * (np.arange(V) // 8192 % 2)                      # every other tile
    allowed = rng.random((B, V)) < share
    w = make_sample(x, np.full(B, wl.TOP_K | wl.TEMPERATURE | wl.TOP_P | wl.GRAMMAR), dtype=dtype, temperature=np.full(B, 0.8),
                    top_k=np.array([8, 20, 64, 100])[np.arange(B) // 4 % 4], top_p=np.full(B, 0.95), bitmask=pack_bits(allowed),
                    seed=np.arange(B), offset=np.arange(B))
    dev = harness.DeviceSample(w)
    dev.run()
    got = dev.results()
    compare_sample(got, oracle.sample(w), w, max_near=B)
    assert ((got["flags"] & 4) != 0).sum() <= B // 8, np.nonzero(got["flags"] & 4)[0]
