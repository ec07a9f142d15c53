"""The op stream of direct fused passes (ops sorted into levels, walked in
pairs, narrow and wide steps) where its layout can go wrong: chains that leave
every pair half empty, streams longer than 48 KB of shared memory, stretches
of ops on the low qubits between ops on the high ones, every fire slot of a
pass; at label counts around a warp and a block, every count of labels a
thread, against the oracle. Amplitudes take at most one product per table byte
and the pi/4 step, so the bound of the suite (1e-12) holds with room."""

import pytest

from oracle import OracleState
from paper_2105_01533_gb300 import sps
from paper_2105_01533_gb300 import workloads as W

from helpers import compare_states

pytestmark = pytest.mark.gpu

EPS = 1e-14


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2105_01533_gb300 import build as B
    B.build()
    sps.load_library()
    yield


def chain(nq):
    """512 gates that each read what the last one flipped; with Y on a top
    qubit every op is two phase ops and a flip."""
    a, b = nq - 1, nq - 2
    return [W.Y(a, b) if i % 2 else W.Y(b, a) for i in range(512)]


def stretches(nq):
    """Long and short stretches on the low qubits between ops on the high ones."""
    out, rng = [], W.SplitMix64(3)
    for length in (1, 3, 7, 20, 40, 2, 9, 30):
        for _ in range(length):
            c, d, t = rng.distinct(12, 3)
            out += [W.CCX(c, d, t), W.CRz(c, t, rng.angle()) if length == 7 else W.T(d)]
        out += [W.CX(nq - 1, 2), W.CCX(1, 3, nq - 1), W.S(nq - 1), W.CX(5, nq - 2)]
    return out


def slots(nq):
    """Every fire slot of one pass (61: 30 Rz and a P), then more."""
    rng = W.SplitMix64(4)
    out = []
    for k in range(40):
        c, t = rng.distinct(nq, 2)
        out += [W.CRz(c, t, rng.angle()), W.CX(t, c), W.Sdg(t, c)]
    return out


@pytest.mark.parametrize("lanes", [0, 1, 2, 4, 8])
@pytest.mark.parametrize("nq,log2n", [(20, 0), (20, 5), (63, 9), (64, 8), (100, 11), (127, 13)])
@pytest.mark.parametrize("make", [chain, stretches, slots])
def test_direct_walk(make, nq, log2n, lanes):
    spread = [W.H(q) for q in range(log2n)] + [W.CX(q, nq - 1 - q % 6) for q in range(log2n)]
    spread += [W.X(nq - 1), W.X(nq - 2)]
    st = sps.SparseState(nq, 1 << log2n)
    st.set_option(sps.SPS_OPT_SMALL_RUN_CAP, 0)
    st.set_option(sps.SPS_OPT_BITSLICE_MIN_OPS, 0)
    st.set_option(sps.SPS_OPT_EXPAND_WALK, 0)
    st.set_option(sps.SPS_OPT_FOLD, 0)
    st.set_option(sps.SPS_OPT_FUSED_LABELS, lanes)
    orc = OracleState(nq)
    for g in (spread, make(nq)):
        st.apply(W.to_array(g), EPS)
        orc.apply(W.to_array(g), eps=EPS)
    compare_states(st.get_amplitudes(), orc.get(), EPS)
    st.close()


@pytest.mark.parametrize("make", [chain, stretches, slots])
def test_walk_in_one_block_and_after_expansion(make):
    for opts in ([], [(sps.SPS_OPT_SMALL_RUN_CAP, 0)]):
        n = 70
        g = W.to_array([W.H(q) for q in range(10)] + make(n))
        st = sps.SparseState(n, 1 << 10)
        for o, v in opts:
            st.set_option(o, v)
        st.apply(g, EPS)
        orc = OracleState(n)
        orc.apply(g, eps=EPS)
        compare_states(st.get_amplitudes(), orc.get(), EPS)
        st.close()


def ladder(nq):
    """Every gate reads what the last one flipped: single flips."""
    return [W.CX(i % nq, (i + 1) % nq) for i in range(300)]


def adder(nq):
    """One and two flips a level in turn."""
    n = (nq - 1) // 2
    up = [(2 * n if i == 0 else i - 1, i, n + i) for i in range(n)]
    return [g for c, x, y in up for g in (W.CX(x, y), W.CX(x, c), W.CCX(c, y, x))] + \
           [g for c, x, y in up[::-1] for g in (W.CCX(c, y, x), W.CX(x, c), W.CX(c, y))]


def ladder_with_phases(nq):
    """A phase op between the flips it waits for: steps of either kind, a long
    stretch of flips alone, then a level with many phase ops."""
    out = []
    for i in range(20):
        a, b = i % nq, (i + 1) % nq
        out += [W.CX(a, b), W.Rz(b, 0.1 + i), W.CX(a, b), W.Y(b, a)]
    return out + ladder(nq) + [W.CZ(i % nq, (i + 3) % nq) for i in range(40)] + [W.CX(0, 1), W.S(1)]


@pytest.mark.parametrize("small", [0, 2048])
@pytest.mark.parametrize("nq,log2n", [(9, 5), (24, 0), (63, 10), (64, 7), (100, 11), (127, 12)])
@pytest.mark.parametrize("make", [ladder, adder, ladder_with_phases])
def test_single_steps(make, nq, log2n, small):
    g = W.to_array([W.H(q) for q in range(log2n)] + make(nq))
    for walk in (0, 1):
        st = sps.SparseState(nq, 1 << log2n)
        st.set_option(sps.SPS_OPT_SMALL_RUN_CAP, small)
        st.set_option(sps.SPS_OPT_BITSLICE_MIN_OPS, 0)
        st.set_option(sps.SPS_OPT_EXPAND_WALK, walk)
        st.set_option(sps.SPS_OPT_FOLD, 0)
        st.apply(g, EPS)
        orc = OracleState(nq)
        orc.apply(g, eps=EPS)
        compare_states(st.get_amplitudes(), orc.get(), EPS)
        st.close()
