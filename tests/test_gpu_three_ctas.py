"""Tile walks with three CTAs per SM (needs a GPU): every combination of metrics
and form, with a small window and split into shards, gives the bits of one CTA
per SM."""
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


@pytest.mark.parametrize("metrics", [["l1"], ["l2"], ["gram"], [("lp", 3.0)], [("lp", 2.5)],
                                     ["l1", "l2", "gram"], ["l1", "l2", ("lp", 3.0)]], ids=str)
@pytest.mark.parametrize("prec,dtype", [("f32c", np.float32), ("f32c", np.float64),
                                        ("f32c_round", np.float64), ("f32", np.float32),
                                        ("f32b", np.float32)])
def test_shards_and_windows(pcf, metrics, prec, dtype):
    import torch
    s = synth.random_set(150, seed=17, max_len=120)
    x = pcf.PcfTensors.from_numpy(
        synth.PcfSet(s.offsets, s.times.astype(dtype), s.values.astype(dtype)), "cuda")
    for window in (0, 40):
        want = pcf.pcf_pairwise(x, metrics, precision=prec, out_dtype=torch.float64,
                                schedule=("tile1024", window))
        for out in (torch.float64, torch.float32):
            whole = pcf.pcf_pairwise(x, metrics, precision=prec, out_dtype=out,
                                     schedule=("tile512x3", window))
            parts = [torch.full_like(w, -3.0) for w in whole]
            for k in range(3):
                pcf.pcf_pairwise(x, metrics, precision=prec, out=parts,
                                 schedule=("tile512x3", window), shard=(k, 3))
            for m, w, a, p in zip(metrics, want, whole, parts):
                assert torch.equal(a, p), m
                # (float32 blocks of the block-compensated sums follow the windows)
                if out == torch.float64 and not (prec == "f32b" and window):
                    assert torch.equal(w, a), m
