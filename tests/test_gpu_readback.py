"""Read-back into device arrays (one kernel) against read-back into host arrays
(copies): counts around a vector pair, arrays that are 8- but not 16-byte
aligned, high words wanted or not, an array too small, a state with an error, a
reset not yet carried out; circuits of a batch; readouts and measurements whose
words lie in device, pinned and pageable memory."""

import ctypes

import numpy as np
import pytest

from paper_2105_01533_gb300 import sps
from paper_2105_01533_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2105_01533_gb300 import build as B
    B.build()
    sps.load_library()
    yield


def device_arrays(n, offset):
    import torch
    i = [torch.full((n + 3,), -7, dtype=torch.int64, device="cuda")[offset:] for _ in range(2)]
    f = [torch.full((n + 3,), -7.0, dtype=torch.float64, device="cuda")[offset:] for _ in range(2)]
    return i + f


def host(t, n):
    a = t[:n].cpu().numpy()
    return a.view(np.uint64) if a.dtype == np.int64 else a


@pytest.mark.parametrize("nq", [20, 64, 90])
@pytest.mark.parametrize("n", [1, 2, 3, 511, 4097, 300001])
@pytest.mark.parametrize("offset", [0, 1])
def test_device_arrays_equal_host_arrays(nq, n, offset):
    rng = np.random.default_rng(n)
    lo = np.arange(n, dtype=np.uint64) * np.uint64(3)
    hi = lo % np.uint64(7) if nq > 70 else np.zeros_like(lo)
    re, im = rng.normal(size=n), rng.normal(size=n)
    st = sps.SparseState(nq, n)
    st.set_amplitudes(hi, lo, re, im)
    want = st.get_amplitudes(sort=False)
    for with_hi in (True, False):
        h, l, r, i = device_arrays(n, offset)
        got = sps.sps_get_amplitudes(st.handle, h if with_hi else None, l, r, i, n)
        assert got == n
        for t, w, used in zip((h, l, r, i), want, (with_hi, True, True, True)):
            if used:
                np.testing.assert_array_equal(host(t, n), w)
            assert float(t[n]) == -7.0   # nothing past the entries
    h, l, r, i = device_arrays(n, 0)
    with pytest.raises(sps.SpsError) as e:
        sps.sps_get_amplitudes(st.handle, h, l, r, i, n - 1)
    assert e.value.status == sps.SPS_ERR_CAPACITY and float(r[0]) == -7.0
    st.reset()
    assert sps.sps_get_amplitudes(st.handle, h, l, r, i, n) == 1
    assert (host(l, 1)[0], host(r, 1)[0], host(i, 1)[0]) == (0, 1.0, 0.0)
    st.close()


def test_nothing_is_copied_from_a_state_with_an_error():
    st = sps.SparseState(20, 4)
    st.set_option(sps.SPS_OPT_SMALL_RUN_CAP, 0)
    h, l, r, i = device_arrays(8, 0)
    st.apply(W.to_array([W.H(q) for q in range(3)]), 0.0)
    with pytest.raises(sps.SpsError) as e:
        sps.sps_get_amplitudes(st.handle, h, l, r, i, 8)
    assert e.value.status == sps.SPS_ERR_CAPACITY and float(r[0]) == -7.0
    n = sps.sps_get_amplitudes(st.handle, h, l, r, i, 8)   # the error is cleared
    want = st.get_amplitudes(sort=False)
    assert n == len(want[1])
    np.testing.assert_array_equal(host(r, n), want[2])
    st.close()


def test_batch_and_words_of_the_caller():
    import torch
    b = sps.Batch()
    for nq, cap in ((20, 301), (70, 1 << 9), (30, 255)):
        b.add(nq, cap, W.to_array([W.H(q) for q in range(7)] + [W.CX(3, nq - 1), W.T(2)]), 0.0)
    b.run()
    b.sync()
    for k in range(3):
        want = b.get_amplitudes(k, sort=False)
        h, l, r, i = device_arrays(512, 1)
        got = ctypes.c_uint64(0)
        assert sps.load_library().sps_batch_get_amplitudes(
            b.handle, k, h.data_ptr(), l.data_ptr(), r.data_ptr(), i.data_ptr(), 512,
            ctypes.byref(got)) == sps.SPS_OK
        assert got.value == len(want[1])
        for t, w in zip((h, l, r, i), want):
            np.testing.assert_array_equal(host(t, got.value), w)
    b.close()
    st = sps.SparseState(66, 1 << 12)
    st.apply(W.to_array([W.Ry(q, 0.3 + q) for q in range(12)]), 0.0)
    places = [torch.zeros(2, dtype=torch.float64, device="cuda"),
              torch.zeros(2, dtype=torch.float64, pin_memory=True), np.zeros(2)]
    for m in places:
        ptr = m.ctypes.data if isinstance(m, np.ndarray) else m.data_ptr()
        p = st.probability((6, 0), (2, 0))   # (the sum's order is the state's layout)
        st.probability_async((6, 0), (2, 0), ptr)
        st.sync()
        assert float(m[0]) == p
        st.apply(W.to_array([W.Ry(q, 0.3 + q) for q in range(12)]), 0.0)
        st.measure_async(1, 0.5, ptr)
        st.sync()
        assert float(m[0]) in (0.0, 1.0) and 0.0 < float(m[1]) <= 1.0
        st.reset()
        st.apply(W.to_array([W.Ry(q, 0.3 + q) for q in range(12)]), 0.0)
    st.close()
