"""The key sort when one of its waits gives up (needs a GPU): the call ends with
the wait's status, no rank is written and nothing behind the workspace changes."""
import ctypes

import numpy as np
import pytest

from conftest import gpu_available

pytestmark = pytest.mark.gpu

GUARD = 1 << 20


@pytest.fixture(scope="module")
def pcf():
    if not gpu_available():
        pytest.skip("no CUDA device")
    import paper_2404_07183_gb300 as P
    P.build.build()
    return P


def _run(pcf, keys, missing, polls):
    """(status or 0, reason, ranks, whether the guard bytes are untouched)"""
    import torch
    from paper_2404_07183_gb300 import abi, api
    lib = abi.load()
    used = ctypes.c_size_t()
    assert lib.pcf_selftest_sort_wait(keys, missing, polls, None, 0, ctypes.byref(used),
                                      api._stream_handle(None)) == abi.PCF_ENOWS
    n = used.value
    buf = torch.full((n + GUARD,), 0xA5, dtype=torch.uint8, device="cuda")
    assert lib.pcf_selftest_sort_wait(keys, missing, polls, ctypes.c_void_p(buf.data_ptr()), n,
                                      ctypes.byref(used), api._stream_handle(None)) == abi.PCF_OK
    status, reason = 0, 0
    try:
        api.pcf_check(buf)
    except pcf.PcfError as e:
        status, reason = e.code, e.detail
    tail = (16 * keys + 255) // 256 * 256
    ranks = buf[n - tail:n - tail + 16 * keys].cpu().numpy().view(np.uint32).reshape(-1, 4)
    return status, reason, ranks, bool((buf[n:] == 0xA5).all().item())


@pytest.mark.parametrize("keys", [1, 8192, 8193, 70001])
def test_whole_sort(pcf, keys):
    status, _, ranks, intact = _run(pcf, keys, -1, 1 << 20)
    assert status == 0 and intact
    key = (np.arange(1, keys + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)) >> np.uint64(1)
    place = np.empty(keys, np.int64)
    place[np.argsort(key, kind="stable")] = np.arange(keys)
    np.testing.assert_array_equal(ranks[:, 0], 2 * (place + 1))
    assert not ranks[:, 1:].any()


@pytest.mark.parametrize("missing", [-1, 3])
def test_wide_states(pcf, missing):
    """2^27 keys and more: states without a pass number, cleared before each pass."""
    import torch
    from paper_2404_07183_gb300 import abi
    keys = (1 << 27) + 5
    status, _, ranks, intact = _run(pcf, keys, missing, 1 << 20 if missing < 0 else 500)
    assert intact
    if missing >= 0:
        assert status == abi.PCF_ETIMEOUT and not ranks.any()
        return
    i = torch.arange(1, keys + 1, dtype=torch.int64, device="cuda")
    key = (i * -7046029254386353131 >> 1) & 0x7FFFFFFFFFFFFFFF     # 0x9e3779b97f4a7c15
    place = torch.empty_like(i)
    place[torch.argsort(key)] = torch.arange(keys, dtype=torch.int64, device="cuda")
    got = torch.from_numpy(np.ascontiguousarray(ranks[:, 0]).astype(np.int64))
    assert status == 0 and torch.equal(got, 2 * (place.cpu() + 1))


@pytest.mark.parametrize("missing", range(9))
@pytest.mark.parametrize("keys", [8193, 70001, 3000000])
def test_a_wait_that_gives_up_stops_the_sort(pcf, keys, missing):
    from paper_2404_07183_gb300 import abi
    status, reason, ranks, intact = _run(pcf, keys, missing, 500)
    assert (status, reason) == (abi.PCF_ETIMEOUT, 9)
    assert intact and not ranks.any()


def test_the_next_call_is_right(pcf):
    """Nothing of a sort that gave up stays behind."""
    import oracle
    import torch
    from paper_2404_07183_gb300 import synth
    _run(pcf, 20000, 0, 500)
    s = synth.random_set(12, seed=5, max_len=40)
    got = pcf.pcf_pairwise(pcf.PcfTensors.from_numpy(s, "cuda"), ["l1"], precision="f32c",
                           out_dtype=torch.float64)[0].cpu().numpy()
    want = oracle.matrix(s, metric="l1")
    assert np.max(np.abs(got - want)) <= 1e-5 * np.max(want)
