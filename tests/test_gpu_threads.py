"""Distinct states used from several host threads at once."""

import threading

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


@pytest.mark.parametrize("form", ["fused", "expand"])
def test_long_and_short_op_streams_side_by_side(form):
    """Runs of 512 and of 400 dependent Y gates on 100 qubits (op streams of
    different lengths past the default shared memory) applied 400 times each from
    two threads, on states and streams of their own: every launch is accepted and
    an even number of Y on one qubit leaves the state as it was."""
    import torch
    n, d = 100, 6
    errors = []

    def work(ngates):
        try:
            stream = torch.cuda.Stream()
            st = sps.SparseState(n, 1 << d, stream=stream.cuda_stream)
            st.set_option(sps.SPS_OPT_SMALL_RUN_CAP, 0)
            st.set_option(sps.SPS_OPT_BITSLICE_MIN_OPS, 0)
            head = W.to_array([W.H(64 + q) for q in range(d)])
            run = W.to_array([W.Y(67)] * ngates)
            both = np.concatenate([head, run])
            st.apply(head, 1e-14)
            for _ in range(400):
                if form == "expand":
                    st.reset()
                    st.apply(both, 1e-14)
                else:
                    st.apply(run, 1e-14)
            got = st.get_amplitudes()
            np.testing.assert_array_equal(got[0], np.arange(1 << d, dtype=np.uint64))
            np.testing.assert_allclose(got[2], 2.0 ** (-d / 2), rtol=1e-12)
            st.close()
        except BaseException as e:   # noqa: BLE001 (handed to the main thread)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in (512, 400)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
