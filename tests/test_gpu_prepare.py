"""Preparation at the edges of its splits (needs a GPU): the length sort's order
around 1,024 PCFs against a stable host sort, the key sort's tiles of 8,192 keys
(one key, one tile, a partial one, shared and distinct times, digits that all
keys share) through exact float32 walks, and validation split over warps."""
import numpy as np
import pytest

import oracle
from paper_2404_07183_gb300 import synth

from conftest import gpu_available, max_rel_error

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pcf():
    if not gpu_available():
        pytest.skip("no CUDA device")
    import paper_2404_07183_gb300 as P
    P.build.build()
    return P


def _set(lens, seed, gaps=lambda r, m: r.exponential(1.0, m)):
    rng = np.random.default_rng(seed)
    return synth.from_lengths(lens, gaps,
                              lambda r, o: np.where(np.isin(np.arange(o[-1]), o[1:] - 1), 0.0,
                                                    r.standard_normal(o[-1])), rng, np.float64)


@pytest.mark.parametrize("n", [1, 2, 31, 33, 97, 1000, 1023, 1024, 1025, 2049])
@pytest.mark.parametrize("top", [9, 600])
def test_sort_order_is_the_stable_host_sort(pcf, n, top):
    rng = np.random.default_rng(n + top)
    s = _set(rng.integers(1, top, n), n)
    x = pcf.PcfTensors.from_numpy(s, "cuda")
    ws = pcf.pcf_prepare(x, "f64")
    perm = pcf.pcf_sort_order(x, ws, "f64").cpu().numpy()
    lens = s.lengths()
    last = s.times[s.offsets[1:] - 1].astype(np.float32)
    bucket = np.where(lens <= 256, lens, 256 + (lens - 256) // 32)
    scale = np.where((lens > 256) & (lens.max() > 256), last, 0.0)
    np.testing.assert_array_equal(perm, np.lexsort((scale, bucket)))


@pytest.mark.parametrize("keys", [1, 8191, 8192, 8193, 20000, 70000])
@pytest.mark.parametrize("kind", ["random", "integers", "close"])
def test_key_sort_tiles(pcf, keys, kind):
    """Exact comparisons at every number of tiles: integer times share keys and
    digits; times a few float64 ulps apart differ in the lowest digit only."""
    import torch
    n = 1 if keys == 1 else 7
    lens = np.full(n, keys // n + 1, np.int64)
    lens[0] += keys - int((lens - 1).sum())
    if kind == "random":
        s = _set(lens, keys)
    elif kind == "integers":
        s = _set(lens, keys, lambda r, m: r.integers(1, 4, m).astype(np.float64))
    else:
        rng = np.random.default_rng(keys)
        s = _set(lens, keys)
        t = s.times.copy()
        for i in range(s.n):
            a, b = int(s.offsets[i]), int(s.offsets[i + 1])
            t[a + 1:b] = 1.0 + 2.0 ** -44 * np.cumsum(rng.integers(1, 4, b - a - 1))
        s = synth.PcfSet(s.offsets, t, s.values)
    x = pcf.PcfTensors.from_numpy(s, "cuda")
    got = pcf.pcf_pairwise(x, ["l1"], precision="f32c", out_dtype=torch.float64)[0].cpu().numpy()
    assert max_rel_error("l1", got, oracle.matrix(s, metric="l1")) <= 1e-5


@pytest.mark.parametrize("n,length", [(3, 40000), (400, 300), (5000, 9)])
def test_errors_of_split_validation(pcf, n, length):
    """The smallest offending element is reported whichever warp finds it."""
    s = _set(np.full(n, length, np.int64), 3)
    t = s.times.copy()
    k = int(s.offsets[n // 2]) + length // 2
    t[k] = t[k - 1]
    t[k + 1:int(s.offsets[n // 2 + 1])] = np.nan
    x = pcf.PcfTensors.from_numpy(synth.PcfSet(s.offsets, t, s.values), "cuda")
    with pytest.raises(pcf.PcfError) as e:
        pcf.pcf_pairwise(x, ["l1"])
    assert (e.value.detail, e.value.index) == (3, k)


@pytest.mark.parametrize("prec,dtype", [("f64", np.float64), ("f32c", np.float64), ("f64", np.float32)])
@pytest.mark.parametrize("bad,detail", [
    ([-0.0, -0.0], 3), ([-0.0, 0.0], 3), ([0.0, -0.0], 3), ([0.0, -1.0], 3), ([-1.0, -0.5], 2),
    ([0.0, 1.0, 1.0], 3), ([0.0, np.nan, 1.0], 4), ([0.0, np.inf], 4), ([0.0, -np.inf, 2.0], 4),
    ([5e-324, 1.0], 2), ([0.0, 2.0, 1.0, 3.0], 3)], ids=str)
def test_time_checks(pcf, bad, detail, prec, dtype):
    """Zeros of either sign, negative and non-finite times: reason and index."""
    t = np.concatenate([[0.0, 1.0], bad, [0.0, 3.0]])
    o = np.array([0, 2, 2 + len(bad), 4 + len(bad)])
    x = pcf.PcfTensors.from_numpy(synth.PcfSet(o, t.astype(dtype), np.zeros(t.size, dtype)), "cuda")
    if dtype == np.float32 and bad[0] == 5e-324:
        return                                       # 0 in float32
    k = 2 if detail == 2 else 2 + next(
        i for i in range(1, len(bad)) if not (np.isfinite(bad[i]) and bad[i] > bad[i - 1]))
    with pytest.raises(pcf.PcfError) as e:
        pcf.pcf_pairwise(x, ["l1"], precision=prec)
    assert (e.value.detail, e.value.index) == (detail, k)


@pytest.mark.parametrize("t", [[-0.0, 1.0, 2.0], [-0.0], [0.0, 5e-324, 1e-310]], ids=str)
def test_times_that_pass(pcf, t):
    import torch
    s = synth.PcfSet([0, 1, 1 + len(t)], np.concatenate([[0.0], t]),
                     np.concatenate([[0.0], np.arange(len(t), dtype=float)[::-1]]))
    got = pcf.pcf_pairwise(pcf.PcfTensors.from_numpy(s, "cuda"), ["l1"], precision="f64",
                           out_dtype=torch.float64)[0].cpu().numpy()
    np.testing.assert_array_equal(got, oracle.matrix(s, metric="l1"))
