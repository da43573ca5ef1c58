"""PCF_SCHED_AUTO between the tiles and the merge path (needs a GPU): where a call
has few tiles but many pairs, collections with a few very long curves take the
merge path and even ones the tiles, whichever form, call or precision; captured
calls choose again at every replay."""
import numpy as np
import pytest

import oracle
from paper_2404_07183_gb300 import synth

from conftest import gpu_available, max_rel_error

pytestmark = pytest.mark.gpu

FORMS = [("f32c", np.float32, 200), ("f32c", np.float64, 200), ("f32b", np.float32, 351),
         ("f64", np.float64, 320), ("f64", np.float32, 320)]


@pytest.fixture(scope="module")
def pcf():
    if not gpu_available():
        pytest.skip("no CUDA device")
    import paper_2404_07183_gb300 as P
    P.build.build()
    return P


def _set(n, long, dtype, seed=3):
    rng = np.random.default_rng(seed)
    lens = rng.integers(20, 26, n)
    if long:
        lens[[3, 50]] = long
    return synth.from_lengths(lens, lambda r, m: r.exponential(1.0, m),
                              lambda r, o: np.where(np.isin(np.arange(o[-1]), o[1:] - 1), 0.0,
                                                    r.standard_normal(o[-1])), rng, dtype)


@pytest.mark.parametrize("prec,dtype,n", FORMS)
@pytest.mark.parametrize("metrics", [["l1"], ["l1", "l2", "gram"]], ids=str)
@pytest.mark.parametrize("long", [0, 9000])
def test_lengths_decide(pcf, prec, dtype, n, metrics, long):
    """AUTO gives the bits of the schedule it should have taken (an even call of
    25,000 pairs or fewer may take either)."""
    import torch
    s = _set(n, long, dtype)
    x = pcf.PcfTensors.from_numpy(s, "cuda")
    run = lambda sched, **kw: pcf.pcf_pairwise(x, metrics, precision=prec, out_dtype=torch.float64,
                                               schedule=sched, **kw)
    auto, merge = run("auto"), run("mergepath")
    if long:
        for a, m in zip(auto, merge):
            assert torch.equal(a, m)
        ws = pcf.pcf_prepare(x, prec)
        for a, m in zip(auto, run("auto", workspace=ws, prepared=True)):
            assert torch.equal(a, m)
        parts = [torch.full_like(a, -7.0) for a in auto]
        for k in range(3):
            pcf.pcf_pairwise(x, metrics, precision=prec, out=parts, shard=(k, 3))
        for a, p in zip(auto, parts):
            assert torch.equal(a, p)
    elif n > 300:
        tiles = run("tile512x2") if prec == "f64" or len(metrics) > 1 else run("tile512x3")
        for a, t in zip(auto, tiles):
            assert torch.equal(a, t)
    s64 = synth.PcfSet(s.offsets, s.times.astype(np.float64), s.values.astype(np.float64))
    diag = np.array([oracle.segment_sq(*s64.pcf(i)) for i in range(s64.n)])
    for m, a in zip(metrics, auto):
        assert max_rel_error(m, a.cpu().numpy(), oracle.matrix(s64, metric=m),
                             diag) <= (1e-12 if prec == "f64" else 1e-5), m


@pytest.mark.parametrize("long", [0, 9000])
def test_other_calls(pcf, long):
    """Cross, to the host, AUTO64 and captured calls."""
    import torch
    s = _set(330, long, np.float64)
    x = pcf.PcfTensors.from_numpy(s, "cuda")
    want = pcf.pcf_pairwise(x, ["l1", "gram"], precision="f32c", out_dtype=torch.float64)
    host = pcf.pcf_pairwise_to_host(x, ["l1", "gram"], precision="f32c", out_dtype=torch.float64)
    torch.cuda.synchronize()
    both = pcf.pcf_pairwise(x, ["l1", "gram"], precision="f32c_auto64", out_dtype=torch.float64)
    graph = pcf.PairwiseGraph(x, ["l1", "gram"], precision="f32c", out_dtype=torch.float64)
    replayed = [r.clone() for r in graph.replay()]
    graph.check()
    for w, h, b, g in zip(want, host, both, replayed):
        assert torch.equal(w.cpu(), h.cpu()) and torch.equal(w, b) and torch.equal(w, g)
    cross = pcf.pcf_cross(x, x, 5, 320, ["l1", "gram"], precision="f32c", out_dtype=torch.float64)
    for w, c in zip(want, cross):
        torch.testing.assert_close(c, w[5:320], rtol=1e-5, atol=1e-5 * float(w.abs().max()))


def test_a_replay_chooses_again(pcf):
    """Even lengths, two long curves among as many breakpoints, even lengths."""
    import torch
    n = 330
    uneven = _set(n, 1200, np.float64, 4)
    nnz = uneven.times.size
    lens = np.full(n, nnz // n)
    lens[:nnz - int(lens.sum())] += 1
    rng = np.random.default_rng(9)
    even = synth.from_lengths(lens, lambda r, m: r.exponential(1.0, m),
                              lambda r, o: np.where(np.isin(np.arange(o[-1]), o[1:] - 1), 0.0,
                                                    r.standard_normal(o[-1])), rng, np.float64)
    x = pcf.PcfTensors.from_numpy(even, "cuda")
    graph = pcf.PairwiseGraph(x, ["l1"], precision="f32c", out_dtype=torch.float64)
    for s in (even, uneven, even):
        y = pcf.PcfTensors.from_numpy(s, "cuda")
        x.offsets.copy_(y.offsets)
        x.times.copy_(y.times)
        x.values.copy_(y.values)
        got = graph.replay()[0].clone()
        graph.check()
        want = pcf.pcf_pairwise(y, ["l1"], precision="f32c", out_dtype=torch.float64)[0]
        assert torch.equal(got, want)
        assert max_rel_error("l1", got.cpu().numpy(), oracle.matrix(s, metric="l1")) <= 1e-5


@pytest.mark.parametrize("long", [0, 9000])
def test_promoted_and_weighted_calls(pcf, long):
    """AUTO64 where the float64 walk runs, and a weight PCF."""
    import torch
    s = _set(330, long, np.float64)
    big = synth.PcfSet(s.offsets, s.times, s.values * 1e60)
    x, y = pcf.PcfTensors.from_numpy(s, "cuda"), pcf.PcfTensors.from_numpy(big, "cuda")
    want = pcf.pcf_pairwise(y, ["l1"], precision="f64", out_dtype=torch.float64)[0]
    got = pcf.pcf_pairwise(y, ["l1"], precision="f32c_auto64", out_dtype=torch.float64)[0]
    assert torch.equal(got, want)
    one = (np.array([0.0]), np.array([1.0]))
    plain = pcf.pcf_pairwise(x, ["l1"], precision="f64", out_dtype=torch.float64)[0]
    weighted = pcf.pcf_pairwise_weighted(x, one, ["l1"], precision="f64", out_dtype=torch.float64)[0]
    torch.testing.assert_close(weighted, plain, rtol=1e-12, atol=0.0)
