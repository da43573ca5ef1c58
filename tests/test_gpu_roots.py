"""float32 results are the float64 results rounded once (needs a GPU): the roots
of all forms are taken in float64, over integrals from below the smallest normal
float32 to near the largest."""
import numpy as np
import pytest

from paper_2404_07183_gb300 import synth

from conftest import gpu_available

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pcf():
    if not gpu_available():
        pytest.skip("no CUDA device")
    import paper_2404_07183_gb300 as P
    P.build.build()
    return P


@pytest.mark.parametrize("metrics", [["l2"], [("lp", 3.0)], ["l1", "l2", "gram"],
                                     ["l1", "l2", ("lp", 3.0)], [("lp", 2.5)]], ids=str)
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("sched", ["tile1024", "tile512x2"])
def test_float32_results_are_rounded_once(pcf, metrics, dtype, sched):
    import torch
    n = 3001 if metrics != [("lp", 2.5)] else 301
    rng = np.random.default_rng(11)
    s = synth.from_lengths(rng.integers(2, 8, n), lambda r, m: r.exponential(1.0, m),
                           lambda r, o: r.standard_normal(o[-1]), rng, np.float64)
    v = s.values * np.repeat(2.0 ** rng.uniform(-46.0, 41.0, n), s.lengths())
    v[s.offsets[1:] - 1] = 0.0
    x = pcf.PcfTensors.from_numpy(synth.PcfSet(s.offsets, s.times.astype(dtype), v.astype(dtype)),
                                  "cuda")
    for prec in ("f32c", "f32b", "f32"):
        one = pcf.pcf_pairwise(x, metrics, precision=prec, out_dtype=torch.float32, schedule=sched)
        two = pcf.pcf_pairwise(x, metrics, precision=prec, out_dtype=torch.float64, schedule=sched)
        for m, a, b in zip(metrics, one, two):
            # (a sum beyond float32's range is NaN in both)
            np.testing.assert_array_equal(a.cpu().numpy(), b.float().cpu().numpy(), err_msg=f"{prec} {m}")
