"""GPU parity tests of the row kernel (calls whose rows are resident at once: one cluster per row) and of the bucket sort of
large candidate sets, at the sizes where they can go wrong: vocabularies at the edges of a CTA's part, every cluster size,
supports at the limits of the short finish, ties, outliers that squash the bins, crowded buckets."""
import numpy as np
import pytest

from paper_2607_20475_b200 import workloads as wl
from tests.helpers import make_sample, pack_bits
from tests.parity import compare_sample, compare_topk, compare_verify

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sonic():
    from paper_2607_20475_b200 import harness
    harness.lib()
    return harness


@pytest.fixture(scope="module")
def oracle():
    from oracle import oracle as o
    return o


def rows_of_every_class(rng, B, V, dtype):
    """Greedy, small and large top-k, top-k beyond the gather, top-p, min-p, both, neither; lists and a mask on some."""
    x = rng.standard_normal((B, V)).astype(np.float32) * 1.5
    x[1::4] = (-1.1 * np.log(rng.permuted(np.tile(np.arange(1, V + 1), (len(x[1::4]), 1)), axis=1))).astype(np.float32)
    x[2::4, :1] += 9.0
    T = wl.TEMPERATURE
    kinds = [(wl.GREEDY, 0), (wl.TOP_K | T, 20), (wl.TOP_K | T | wl.TOP_P, 100), (wl.TOP_K | T, 1000), (wl.TOP_P | T, 0),
             (wl.MIN_P | T, 0), (wl.TOP_P | wl.MIN_P | T, 0), (T, 0), (wl.TOP_K | T | wl.TOP_P, 3000), (wl.TOP_K | wl.MIN_P, 128)]
    mode = np.array([kinds[r % len(kinds)][0] for r in range(B)], np.uint32)
    k = np.array([min(kinds[r % len(kinds)][1], V) for r in range(B)])
    allowed = rng.random((B, V)) < 0.3
    allowed[:, -1] = True
    mode[3::7] |= wl.GRAMMAR
    mode[::2] |= wl.REPETITION | wl.FREQUENCY | wl.PRESENCE | wl.BIAS
    n = min(V, 40)
    hist = [{int(i): int(c) for i, c in zip(rng.choice(V, n, replace=False), rng.integers(1, 5, n))} for _ in range(B)]
    bias = [{int(i): float(v) for i, v in zip(rng.choice(V, min(V, 6), replace=False), rng.uniform(-5, 5, 6))} for _ in range(B)]
    return make_sample(x, mode, dtype=dtype, temperature=rng.uniform(0.6, 1.4, B), top_k=k, top_p=np.full(B, 0.93),
                       min_p=np.full(B, 0.03), rep=np.full(B, 1.2), freq=np.full(B, 0.2), pres=np.full(B, 0.3),
                       bitmask=pack_bits(allowed), hist=hist, bias=bias, seed=np.arange(B) + V, offset=np.arange(B) * 3)


@pytest.mark.parametrize("B,V", [(10, 1), (10, 5), (10, 2047), (10, 2048), (10, 2049), (10, 8192), (10, 8193), (12, 32767), (11, 32769),
                                 (30, 65537), (40, 40960), (3, 262144), (11, 262143), (18, 200003), (74, 9000)])
@pytest.mark.parametrize("dtype", [wl.DTYPE_F32, wl.DTYPE_BF16])
def test_rows_of_every_class(sonic, oracle, B, V, dtype):
    w = rows_of_every_class(np.random.default_rng(B * 1000003 + V), B, V, dtype)
    dev = sonic.DeviceSample(w)
    dev.run()
    got = dev.results()
    compare_sample(got, oracle.sample(w), w, max_near=B)         # (each near-margin row is held to an admissible outcome)
    dev.run()
    again = dev.results()
    for key in got:
        assert np.array_equal(got[key], again[key]), key


@pytest.mark.parametrize("dtype", [wl.DTYPE_F32, wl.DTYPE_BF16])
def test_ties_outliers_and_empty_parts(sonic, oracle, dtype):
    # one value, two values, a single finite entry in the last CTA's part, a huge outlier, -1e9 in place of a mask
    V = 50021
    rng = np.random.default_rng(31)
    base = rng.standard_normal(V).astype(np.float32)
    rows = [np.zeros(V, np.float32), np.where(rng.random(V) < 0.4, 1.0, 0.0).astype(np.float32), np.full(V, -np.inf, np.float32),
            base.copy(), np.where(rng.random(V) < 0.01, base, np.float32(-1e9)).astype(np.float32), base * 40, np.round(base * 4) / 4]
    rows[2][V - 1] = 3.0
    rows[3][77] = 1000.0
    for mode, kw in ((wl.TOP_K, dict(top_k=50)), (wl.TOP_K | wl.TEMPERATURE, dict(top_k=700, temperature=1.7)),
                     (wl.TOP_P | wl.TEMPERATURE, dict(top_p=0.9, temperature=1.3)), (wl.TOP_P | wl.MIN_P, dict(top_p=0.97, min_p=0.2)),
                     (wl.TOP_K | wl.TOP_P, dict(top_k=5000, top_p=0.6)), (wl.GREEDY, {})):
        B = len(rows)
        w = make_sample(np.stack(rows), np.full(B, mode), dtype=dtype, seed=np.arange(B) + mode, offset=np.arange(B),
                        **{n: np.full(B, v) for n, v in kw.items()})
        dev = sonic.DeviceSample(w)
        dev.run()
        compare_sample(dev.results(), oracle.sample(w), w, max_near=B)


@pytest.mark.parametrize("B,K,V", [(1, 0, 3000), (3, 2, 32003), (9, 3, 17000), (2, 7, 131072)])
def test_verification_of_few_requests(sonic, oracle, B, K, V):
    vw = wl.config4(B=B, K=K, V=V) if K else None
    if vw is None:
        full = wl.config4(B=B, K=1, V=V)
        full.sample.logits = np.ascontiguousarray(full.sample.logits[::2])
        vw = wl.VerifyWorkload(name="k0", B=B, K=0, V=V, sample=full.sample, draft_tokens=np.zeros((B, 0), np.int32),
                               draft_probs=np.zeros((B, 0, V), np.float32))
    else:
        vw.draft_tokens[0, 0] = int(np.argmin(vw.sample.logits_f32()[0]))        # rejected
    dev = sonic.DeviceVerify(vw)
    dev.run()
    got = dev.results()
    compare_verify(got, oracle.verify(vw), vw, max_near=B)
    dev.run()
    again = dev.results()
    for key in got:
        assert np.array_equal(got[key], again[key]), key


@pytest.mark.parametrize("B", [3, 80])                             # row kernel (k up to 2048), streaming chain
@pytest.mark.parametrize("k", [100, 101, 129, 513, 1024, 2048, 2049, 4096])
def test_large_top_k_sorts(sonic, oracle, B, k):
    # smooth values, low-precision ties (crowded buckets), an outlier that squashes the buckets, few distinct values
    V = 20001
    rng = np.random.default_rng(k)
    x = rng.standard_normal((B, V)).astype(np.float32)
    x[1] = np.round(x[1] * 8) / 8
    x[2] = np.where(rng.random(V) < 0.5, x[2], np.round(x[2]))
    x[0, 5] = 1e30
    tw = wl.TopKWorkload(name="t", B=B, V=V, dtype=wl.DTYPE_F32, logits=x)
    dev = sonic.DeviceTopK(tw, k)
    dev.run()
    gv, gi = dev.results()
    compare_topk(gv, gi, *oracle.topk(x, k))


@pytest.mark.parametrize("V", [8193, 9000, 12000, 16384, 17999])
@pytest.mark.parametrize("dtype", [wl.DTYPE_F32, wl.DTYPE_BF16])
def test_top_k_that_the_streaming_chain_would_not_take(sonic, oracle, V, dtype):
    # short vocabularies with a large k, at both sides of what the chain's candidates prove (1003 | 1005 at V = 8193): every
    # output has to be written, through both entry points
    rng = np.random.default_rng(V + dtype)
    for B, k in ((1, 1003), (8, 1005), (3, 1500), (8, 2048)):
        x = rng.standard_normal((B, V)).astype(np.float32)
        x[0, ::3] = -np.inf
        tw = wl.TopKWorkload(name="t", B=B, V=V, dtype=dtype, logits=x if dtype == wl.DTYPE_F32 else wl.f32_to_bf16_bits(x))
        ref = oracle.topk(tw.logits_f32(), k)
        dev = sonic.DeviceTopK(tw, k)
        for static in (False, True):
            dev.out_vals.fill_(-7.0)
            dev.out_idx.fill_(-7)
            if static:
                sonic.sonic_topk_static(dev.logits, dtype, B, V, dev.logits.shape[1], k, dev.out_vals, dev.out_idx)
            else:
                dev.run()
            compare_topk(*dev.results(), *ref)


@pytest.mark.parametrize("dtype", [wl.DTYPE_F32, wl.DTYPE_BF16])
def test_processed_logits_that_overflow(sonic, oracle, dtype):
    # finite logits over a temperature of 0.5: ten ids become +inf and share the whole mass (the limit of the softmax); no
    # truncation, top-p, min-p, a top-k beyond the gather; then the same as verification rows, whose requests must be finished
    import torch
    V, n = 20001, 10
    rng = np.random.default_rng(5 + dtype)
    ids = np.sort(rng.choice(V, n, replace=False))
    x = rng.standard_normal((4, V)).astype(np.float32)
    x[:, ids] = 3e38
    T = wl.TEMPERATURE
    w = make_sample(x, [T, T | wl.TOP_P, T | wl.MIN_P, T | wl.TOP_K], dtype=dtype, temperature=np.full(4, 0.5), top_p=np.full(4, 0.85),
                    min_p=np.full(4, 0.1), top_k=np.full(4, 3000), seed=np.arange(4) + 11, offset=np.arange(4))
    dev = sonic.DeviceSample(w)
    dev.run()
    got = dev.results()
    assert np.isin(got["token"], ids).all() and not (got["flags"] & 0x13).any()
    assert got["support"].tolist() == [V, 9, n, 3000]                # (elements without weight count where nothing cuts them off)
    assert np.allclose(got["prob"], [1 / n, 1 / 9, 1 / n, 1 / n], rtol=1e-5)
    B, K = 2, 1
    vw = wl.VerifyWorkload(name="v", B=B, K=K, V=V, sample=make_sample(x[:B], [T | wl.TOP_P, T | wl.MIN_P], dtype=dtype,
                           temperature=np.full(B, 0.5), top_p=np.full(B, 0.85), min_p=np.full(B, 0.1), seed=np.arange(B), offset=np.arange(B)),
                           draft_tokens=np.array([[ids[-1]], [ids[0]]], np.int32), draft_probs=np.zeros((B, K, V), np.float32))
    vw.draft_probs[0, 0, ids[:5]] = 0.2                           # (the first draft lies outside the top-p support: rejected)
    vw.draft_probs[1, 0, ids[0]] = 0.05
    vw.sample.logits = w.logits
    dv = sonic.DeviceVerify(vw)
    for _ in range(3):
        dv.run()
        got = dv.results()
        assert got["accept_len"].tolist() == [0, 1] and got["tokens"][1, 0] == ids[0]
        assert got["tokens"][0, 0] in ids[5:9] and got["tokens"][0, 1] == -1 and got["tokens"][1, 1] in ids
        assert not dv.ws[512:512 + 4 * 4096].view(torch.int32).any()                # the requests' tickets


@pytest.mark.parametrize("octaves", [1, 4, 8, 16, 32, 41])
def test_smallest_weight_at_the_edge_of_an_octave(sonic, oracle, octaves):
    # the row's smallest value a whole number of halvings below its largest, give or take a unit in the last place: every
    # weight must stay within the bins that this number is given
    V = 30011
    rng = np.random.default_rng(octaves)
    x = (rng.random((12, V)) * -(octaves * np.log(2.0))).astype(np.float32)
    low = np.float32(-octaves * np.log(2.0))
    for r in range(12):
        edge = low
        for _ in range(abs(r - 6)):
            edge = np.nextafter(edge, np.float32(-np.inf if r < 6 else np.inf))
        x[r] = np.maximum(x[r], edge)
        x[r, rng.choice(V, V // 3, replace=False)] = edge
        x[r, r * 100] = 0.0
    w = make_sample(x, np.full(12, wl.TOP_P), top_p=np.where(np.arange(12) % 2, 0.9999, 0.6), seed=np.arange(12) + 3, offset=np.arange(12))
    dev = sonic.DeviceSample(w)
    dev.run()
    compare_sample(dev.results(), oracle.sample(w), w, max_near=12)


@pytest.mark.parametrize("B,k", [(8, 1500), (80, 1500), (148, 3000)])
def test_repeated_sorts_of_large_candidate_sets(sonic, oracle, B, k):
    # many sorts of thousands of candidates under load, in the row kernel and in the merge: the same rows every time
    import torch
    V = 20001
    x = np.random.default_rng(k).standard_normal((B, V)).astype(np.float32)
    dev = sonic.DeviceTopK(wl.TopKWorkload(name="t", B=B, V=V, dtype=wl.DTYPE_F32, logits=x), k)
    dev.run()
    vals, idx = dev.results()
    compare_topk(vals, idx, *oracle.topk(x, k))
    vals, idx = torch.from_numpy(vals).cuda(), torch.from_numpy(idx).cuda()
    for _ in range(300):
        dev.out_vals.fill_(-7.0)
        dev.out_idx.fill_(-7)
        dev.run()
        assert torch.equal(dev.out_vals, vals) and torch.equal(dev.out_idx, idx)


@pytest.mark.parametrize("temperature", [3e38, 1e38, 1e-39, 1e-40, 0.3])
@pytest.mark.parametrize("dtype", [wl.DTYPE_F32, wl.DTYPE_BF16])
def test_values_that_become_equal_under_the_temperature(sonic, oracle, temperature, dtype):
    # quotients that are subnormal (steps of 1e-6 of the value) or overflow: ascending logits a few units in the last place
    # apart, so that the largest index holds the largest logit but the lowest index among its equals wins
    V = 9000
    rng = np.random.default_rng(8)
    x = np.full((6, V), -1.0, np.float32)
    for r in range(6):
        ids = np.sort(rng.choice(V, 400, replace=False))
        x[r, ids] = np.float32(0.1) * (1 + np.arange(400) * np.float32(2.0 ** -22 if dtype == wl.DTYPE_F32 else 2.0 ** -8) * (r + 1))
    if temperature < 1e-30:
        x = np.where(x < 0, x, -x * 3)                            # (below 1e-38 most quotients are -inf)
        x[:, 5] = -temperature
    mode = np.full(6, wl.TOP_K | wl.TEMPERATURE, np.uint32)
    mode[5] = wl.GREEDY | wl.TEMPERATURE
    w = make_sample(x, mode, dtype=dtype, temperature=np.full(6, temperature), top_k=[1, 2, 20, 50, 90, 0], seed=np.arange(6) + 7, offset=np.arange(6))
    dev = sonic.DeviceSample(w)
    dev.run()
    compare_sample(dev.results(), oracle.sample(w), w, max_near=6)


@pytest.mark.parametrize("B", [8, 80])                             # row kernel (k up to 2048), streaming chain
@pytest.mark.parametrize("k", [513, 1024, 2048, 3000])
def test_sorts_with_hundreds_of_equal_values(sonic, oracle, B, k):
    # a dozen distinct values among the wanted ones, hundreds of each: buckets beyond what a warp sorts, most candidates unwanted
    V = 65536
    rng = np.random.default_rng(k + B)
    x = (np.round(rng.standard_normal((B, V)) * 8) / 8).astype(np.float32)
    x[1::3] = np.round(x[1::3] * 2) / 2
    x[2::3, rng.choice(V, k // 2, replace=False)] += np.float32(40.0)
    tw = wl.TopKWorkload(name="t", B=B, V=V, dtype=wl.DTYPE_F32, logits=x)
    dev = sonic.DeviceTopK(tw, k)
    dev.run()
    compare_topk(*dev.results(), *oracle.topk(x, k))


@pytest.mark.parametrize("B,V", [(14, 40000), (15, 40000), (18, 245761), (17, 200003), (33, 20001), (34, 20001), (37, 131072), (71, 9000), (74, 9000), (75, 9000)])
@pytest.mark.parametrize("dtype", [wl.DTYPE_F32, wl.DTYPE_BF16])
def test_row_counts_at_the_edges_of_the_cluster_sizes(sonic, oracle, B, V, dtype):
    # as many rows as there are clusters of 16, 8 or 4 CTAs at once, one more, as many as there are CTA slots for; top-k at both
    # sides of what the group maxima serve
    w = rows_of_every_class(np.random.default_rng(B * 7 + V), B, V, dtype)
    dev = sonic.DeviceSample(w)
    dev.run()
    compare_sample(dev.results(), oracle.sample(w), w, max_near=B)
    tw = wl.TopKWorkload(name="t", B=B, V=V, dtype=dtype, logits=w.logits)
    vals, idx = oracle.topk(tw.logits_f32(), 101)
    for k in (2, 63, 65, 88, 89, 101):
        dev = sonic.DeviceTopK(tw, k)
        dev.run()
        compare_topk(*dev.results(), vals[:, :k].copy(), idx[:, :k].copy())
