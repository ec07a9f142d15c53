"""Pauli exponentials of Z factors only (one kernel) against the run of CNOTs, Rz
and CNOTs that they stand for and count as: strings of one qubit to all, on low
and high qubits, with controls, from one entry to two rounds of the grid."""

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


@pytest.mark.parametrize("nq,n", [(12, 1), (20, 33), (63, 257), (64, 4099), (100, 1000), (127, 700001)])
@pytest.mark.parametrize("zq,cq", [([0], []), ([1, 5], [2]), ([0, 3, 7, 11], [1, 4]), ("high", "low")])
def test_equals_its_ladder(nq, n, zq, cq):
    if zq == "high":
        zq, cq = [nq - 1, nq - 2, 3], [0]
    rng = np.random.default_rng(nq)
    lo = (np.arange(n, dtype=np.uint64) * np.uint64(2654435761)) % np.uint64(1 << min(nq, 60))
    lo = np.unique(lo)
    hi = (lo * np.uint64(40503)) % np.uint64(1 << min(nq - 64, 60)) if nq > 64 else np.zeros_like(lo)
    init = (hi, lo, rng.normal(size=len(lo)), rng.normal(size=len(lo)))
    mask = lambda qs: (sum(1 << q for q in qs if q < 64), sum(1 << (q - 64) for q in qs if q >= 64))
    ladder = [W.CX(q, zq[-1]) for q in zq[:-1]]
    got = []
    for form in (0, 1):
        st = sps.SparseState(nq, len(lo))
        st.set_amplitudes(*init)
        for theta in (0.7, -2.9):
            if form:
                st.apply(W.to_array(ladder + [W.Rz(zq[-1], theta, *cq)] + ladder[::-1]), 0.0)
            else:
                st.pauli_exp((0, 0), mask(zq), mask(cq), theta, 0.0)
        got.append(st.get_amplitudes() + (st.updates(), st.counters().gates))
        st.close()
    for a, b in zip(got[0][:2], got[1][:2]):
        np.testing.assert_array_equal(a, b)
    for a, b in zip(got[0][2:4], got[1][2:4]):   # two products of |a| < 6, each within 2^-52
        np.testing.assert_allclose(a, b, rtol=0, atol=6e-15)
    assert got[0][4:] == got[1][4:]
