"""The cooperative merge path at the edges of its slabs, groups and parts
(needs a GPU).  A warp copies float64 pairs of up to 256 advances, a CTA takes
2,048 per slab; above 1,024 breakpoints per pair on average a long longest pair
sends the call to CTAs, and few long pairs to clusters of 2, 4 or 8 of them above
8,192, 16,384 and 32,768."""
import numpy as np
import pytest

import oracle
from paper_2404_07183_gb300 import synth

from conftest import gpu_available, max_rel_error

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "f32c": 1e-5, "f32b": 1e-5}
LENGTHS = [[1, 1, 2], [128, 129, 130, 1], [300, 213, 43, 600], [1025, 1024, 1023, 3],
           [2049, 2048, 4100, 1], [4097, 4096, 5000], [9001, 8192, 7000], [16385, 20000, 12001]]


@pytest.fixture(scope="module")
def pcf():
    if not gpu_available():
        pytest.skip("no CUDA device")
    import paper_2404_07183_gb300 as P
    P.build.build()
    return P


@pytest.mark.parametrize("lens", LENGTHS, ids=lambda v: str(max(v)))
@pytest.mark.parametrize("prec,dtype", [("f64", np.float64), ("f32c", np.float64),
                                        ("f32c", np.float32), ("f32b", np.float32)])
def test_slab_edges(pcf, lens, prec, dtype):
    import torch
    rng = np.random.default_rng(sum(lens))
    s = synth.from_lengths(lens, lambda r, m: r.exponential(1.0, m),
                           lambda r, o: np.where(np.isin(np.arange(o[-1]), o[1:] - 1), 0.0,
                                                 r.standard_normal(o[-1])), rng, dtype)
    x = pcf.PcfTensors.from_numpy(s, "cuda")
    s64 = synth.PcfSet(s.offsets, s.times.astype(np.float64), s.values.astype(np.float64))
    diag = np.array([oracle.segment_sq(*s64.pcf(i)) for i in range(s64.n)])
    got = pcf.pcf_pairwise(x, ["l1", "l2", "gram"], precision=prec, out_dtype=torch.float64,
                           schedule="mergepath")
    again = pcf.pcf_pairwise(x, ["l1", "l2", "gram"], precision=prec, out_dtype=torch.float64,
                             schedule="mergepath")
    for m, g, h in zip(("l1", "l2", "gram"), got, again):
        assert max_rel_error(m, g.cpu().numpy(), oracle.matrix(s64, metric=m), diag) <= TOL[prec], m
        assert torch.equal(g, h), m                     # fixed order: the same bits


@pytest.mark.parametrize("lens", [[300, 213, 43, 600], [9001, 8192, 7000]], ids=str)
def test_dyadic_bitwise(pcf, lens):
    """Integer times with many shared breakpoints: every partial sum is exact."""
    import torch
    rng = np.random.default_rng(5)
    s = synth.from_lengths(lens, lambda r, m: r.integers(1, 3, m).astype(np.float64),
                           lambda r, o: np.where(np.isin(np.arange(o[-1]), o[1:] - 1), 0.0,
                                                 r.integers(-6, 7, o[-1])), rng, np.float64)
    x = pcf.PcfTensors.from_numpy(s, "cuda")
    for prec in ("f64", "f32c"):
        got = pcf.pcf_pairwise(x, ["l1", "gram"], precision=prec, out_dtype=torch.float64,
                               schedule="mergepath")
        for m, g in zip(("l1", "gram"), got):
            if prec == "f32c" and max(lens) > 1000:
                continue                                # sums beyond 2^24
            np.testing.assert_array_equal(g.cpu().numpy(), oracle.matrix(s, metric=m))


@pytest.mark.parametrize("lens", [[300, 213, 43], [20000, 16385, 12001]], ids=str)
def test_captured_call(pcf, lens):
    """A captured call (plain and cluster launches) replays with new contents."""
    import torch
    sets = [synth.from_lengths(lens, lambda r, m: r.exponential(1.0, m),
                               lambda r, o: np.where(np.isin(np.arange(o[-1]), o[1:] - 1), 0.0,
                                                     r.standard_normal(o[-1])),
                               np.random.default_rng(seed), np.float64) for seed in (1, 2)]
    x = pcf.PcfTensors.from_numpy(sets[0], "cuda")
    for prec in ("f64", "f32c"):
        graph = pcf.PairwiseGraph(x, ["l1"], precision=prec, out_dtype=torch.float64)
        y = pcf.PcfTensors.from_numpy(sets[1], "cuda")
        x.times.copy_(y.times)
        x.values.copy_(y.values)
        got = graph.replay()[0].clone()
        graph.check()
        want = pcf.pcf_pairwise(y, ["l1"], precision=prec, out_dtype=torch.float64)[0]
        assert torch.equal(got, want)


def test_auto_keeps_what_windows_and_rounding_accept(pcf):
    """200 PCFs (fewer tiles than half the SMs): an explicit window larger than any
    tile kernel's, and rounded times with more coincident ones than a window holds,
    go to the merge path."""
    import torch
    s = synth.random_set(200, seed=3, min_len=5, max_len=30)
    x = pcf.PcfTensors.from_numpy(s, "cuda")
    got = pcf.pcf_pairwise(x, ["l1"], precision="f32c", schedule=("auto", 4000), out_dtype=torch.float64)[0]
    assert max_rel_error("l1", got.cpu().numpy(), oracle.matrix(s, metric="l1")) <= 1e-5
    t = np.concatenate([[0.0], 4096.0 + 2.0 ** -20 * np.arange(1, 600)])
    o = np.arange(0, 200 * t.size + 1, t.size)
    v = np.tile(np.concatenate([np.arange(t.size - 1) % 7, [0.0]]), 200)
    pcf.pcf_pairwise(pcf.PcfTensors.from_numpy(synth.PcfSet(o, np.tile(t, 200), v), "cuda"), ["l1"],
                     precision="f32c_round")


@pytest.mark.parametrize("lens", [[40000, 33000, 20001], [2, 60000, 50000, 1]], ids=str)
@pytest.mark.parametrize("prec,dtype", [("f64", np.float64), ("f32c", np.float64), ("f32c", np.float32)])
def test_clusters_of_eight(pcf, lens, prec, dtype):
    """Eight CTAs per pair, also where some of them get no advance, whole and in
    shards."""
    import torch
    rng = np.random.default_rng(len(lens))
    s = synth.from_lengths(lens, lambda r, m: r.exponential(1.0, m),
                           lambda r, o: np.where(np.isin(np.arange(o[-1]), o[1:] - 1), 0.0,
                                                 r.standard_normal(o[-1])), rng, dtype)
    x = pcf.PcfTensors.from_numpy(s, "cuda")
    s64 = synth.PcfSet(s.offsets, s.times.astype(np.float64), s.values.astype(np.float64))
    diag = np.array([oracle.segment_sq(*s64.pcf(i)) for i in range(s64.n)])
    metrics = ["l1", "l2", "gram"]
    got = pcf.pcf_pairwise(x, metrics, precision=prec, out_dtype=torch.float64, schedule="mergepath")
    parts = [torch.full_like(g, -7.0) for g in got]
    for k in range(4):
        pcf.pcf_pairwise(x, metrics, precision=prec, out=parts, schedule="mergepath", shard=(k, 4))
    for m, g, p in zip(metrics, got, parts):
        assert max_rel_error(m, g.cpu().numpy(), oracle.matrix(s64, metric=m), diag) <= TOL[prec], m
        assert torch.equal(g, p), m


@pytest.mark.parametrize("prec,dtype", [("f64", np.float64), ("f32c", np.float64), ("f32c", np.float32),
                                        ("f32b", np.float32), ("f32", np.float32)])
@pytest.mark.parametrize("kind", ["short", "edge of the copy", "one long", "many", "skewed"])
def test_warps_and_ctas(pcf, kind, prec, dtype):
    """A warp per pair around its copied length (256 advances) and for many pairs
    of more than 1,024; one very long curve decides for CTAs on the device."""
    import torch
    rng = np.random.default_rng(21)
    lens = {"short": rng.integers(1, 40, 60),
            "edge of the copy": np.array([128, 129, 130, 131, 1, 2, 256, 257, 258, 127]),
            "one long": np.concatenate([rng.integers(5, 30, 40), [5000]]),
            "many": rng.integers(500, 800, 50),
            "skewed": np.concatenate([rng.integers(100, 300, 78), [30000, 9000]])}[kind]
    s = synth.from_lengths(lens, lambda r, m: r.exponential(1.0, m),
                           lambda r, o: np.where(np.isin(np.arange(o[-1]), o[1:] - 1), 0.0,
                                                 r.standard_normal(o[-1])), rng, dtype)
    x = pcf.PcfTensors.from_numpy(s, "cuda")
    s64 = synth.PcfSet(s.offsets, s.times.astype(np.float64), s.values.astype(np.float64))
    diag = np.array([oracle.segment_sq(*s64.pcf(i)) for i in range(s64.n)])
    tol = {**TOL, "f32": 5e-4}[prec]
    for metrics in (["l1"], ["l1", "l2", "gram"], [("lp", 3.0)]):
        got = pcf.pcf_pairwise(x, metrics, precision=prec, out_dtype=torch.float64,
                               schedule="mergepath")
        for m, g in zip(metrics, got):
            code, p = (m, 1.0) if isinstance(m, str) else m
            assert max_rel_error(code, g.cpu().numpy(), oracle.matrix(s64, metric=code, p=p),
                                 diag) <= tol, m
