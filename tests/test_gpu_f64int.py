"""float64 walks and their adjoint where the integer widths and products begin
and end (needs a GPU): magnitudes inside and outside their ranges, ends that
span more than ten octaves, values that differ in the last bit, zeros."""
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


def _set(kind, tscale, vscale, n=40):
    rng = np.random.default_rng(7)
    lens = rng.integers(1, 90, n)
    s = synth.from_lengths(lens, lambda r, m: r.exponential(1.0, m),
                           lambda r, o: r.standard_normal(o[-1]), rng, np.float64)
    t, v = s.times.copy(), s.values.copy()
    for i in range(n):
        a, b = int(s.offsets[i]), int(s.offsets[i + 1])
        if kind == "octaves":                        # ends over 60 octaves
            t[a + 1:b] = np.sort(2.0 ** rng.uniform(-30, 30, b - a - 1))
        if kind == "last bit":
            v[a:b] = 1.0 + 2.0 ** -52 * rng.integers(0, 3, b - a)
        v[b - 1] = 0.0
    if kind == "one wild value":
        v[int(s.offsets[n // 2])] = 1e-160
    return synth.PcfSet(s.offsets, t * tscale, v * vscale)


CASES = [("plain", 1.0, 1.0), ("octaves", 1.0, 1.0), ("last bit", 1.0, 1.0),
         ("one wild value", 1.0, 1.0), ("plain", 2.0 ** -700, 1.0), ("plain", 2.0 ** 600, 1.0),
         ("plain", 2.0 ** -760, 2.0 ** 20), ("plain", 1.0, 2.0 ** -398), ("plain", 1.0, 2.0 ** 480),
         ("plain", 1.0, 2.0 ** -420)]


@pytest.mark.parametrize("kind,tscale,vscale", CASES)
@pytest.mark.parametrize("sched", ["tile1024", "tile512x2", ("tile512x2", 8)], ids=str)
def test_walk(pcf, kind, tscale, vscale, sched):
    import torch
    s = _set(kind, tscale, vscale)
    x = pcf.PcfTensors.from_numpy(s, "cuda")
    metrics = [("l1", "l1"), (("l2", False), "l2"), ("gram", "gram")]
    got = pcf.pcf_pairwise(x, [m for m, _ in metrics], precision="f64", out_dtype=torch.float64,
                           schedule=sched)
    for (m, name), g in zip(metrics, got):
        want = oracle.matrix(s, metric=name, apply_root=isinstance(m, str))
        diag = np.array([oracle.segment_sq(*s.pcf(i)) for i in range(s.n)])
        if name == "gram" and (vscale < 2.0 ** -300 or tscale < 2.0 ** -300):
            continue                                 # products of norms leave float64
        if not np.all(want[np.isfinite(want)] < 1e300):
            continue
        assert max_rel_error(name, g.cpu().numpy(), want, diag) <= 1e-12, name


@pytest.mark.parametrize("kind,tscale,vscale", CASES[:4] + [("plain", 2.0 ** -100, 2.0 ** 30)])
@pytest.mark.parametrize("metric", ["l1", "l2", "gram"])
def test_adjoint(pcf, kind, tscale, vscale, metric):
    import torch
    s = _set(kind, tscale, vscale)
    G = np.random.default_rng(1).standard_normal((s.n, s.n))
    x = pcf.PcfTensors.from_numpy(s, "cuda")
    gv, gt = pcf.pcf_pairwise_backward(x, (metric, False), torch.from_numpy(G).cuda())
    ov, ot = oracle.backward(s, G, metric=metric, p=2.0 if metric == "l2" else 1.0)
    for a, b in ((gv.cpu().numpy(), ov), (gt.cpu().numpy(), ot)):
        assert np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(b))
