"""The group stage of the fallback launch (runs of three or more branching
gates on disjoint qubits on states that they change): against the passes as
separate launches, bit for bit with their update count, and the oracle; where
it hands the run back (groups over 64 members, members over the capacity)
and where absent members, pruned values, stored zeros, appended leaders and
partial rounds meet."""

import itertools

import numpy as np
import pytest

from oracle import OracleState
from paper_2105_01533_gb300 import sps
from paper_2105_01533_gb300 import workloads as W

from helpers import compare_states

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


def random_state(nq, count, seed, zeros=0):
    rng = np.random.default_rng(seed)
    lo = set()
    while len(lo) < count:
        lo.add(int(rng.integers(0, 1 << min(nq, 14))))
    lo = np.array(sorted(lo), np.uint64)
    rng.shuffle(lo)
    hi = np.zeros_like(lo)
    if nq > 64:   # the same values on the top qubits
        hi = (lo & np.uint64(127)) << np.uint64(nq - 64 - 7)
        lo = lo >> np.uint64(7)
    re, im = rng.normal(size=count), rng.normal(size=count)
    re[:zeros] = 0.0
    im[:zeros] = 0.0
    return hi, lo, re, im


def layer(nq, kind, gates, rng):
    """`gates` disjoint gates over the qubits random_state populates."""
    low = 7 if nq > 64 else min(nq, 14)
    qs = list(range(low)) + (list(range(nq - 7, nq)) if nq > 64 else [])
    qs = [qs[i] for i in rng.distinct(len(qs), len(qs))]
    out = []
    while len(out) < gates:
        t = rng.angle()
        if kind == "givens":
            out.append(W.Givens(qs.pop(), qs.pop(), t))
        elif kind == "controlled":
            out.append(W.Givens(qs.pop(), qs.pop(), t) if len(out) % 2 else
                       W.Rx(qs.pop(), t, qs.pop()))
        else:
            out.append([W.H(qs.pop()), W.Rx(qs.pop(), t)][len(out) % 2] if len(qs) > 1 else
                       W.Ry(qs.pop(), t))
    return out


def both(nq, init, parts, eps, cap, lay=4):
    got = []
    for chain in (1, 0):
        st = sps.SparseState(nq, cap)
        st.set_option(sps.SPS_OPT_SMALL_RUN_CAP, 0)
        st.set_option(sps.SPS_OPT_EXPAND, 0)
        st.set_option(sps.SPS_OPT_LAYER_GATES, lay)
        st.set_option(sps.SPS_OPT_FALLBACK_CHAIN, chain)
        st.set_amplitudes(*init)
        for g in parts:
            st.apply(W.to_array(g), eps)
        try:
            st.sync()
            err = None
        except sps.SpsError as e:
            err = (e.status, e.failed_gate)
        got.append((err, st.get_amplitudes(), st.updates()))
        st.close()
    (e1, a1, u1), (e0, a0, u0) = got
    assert e1 == e0
    for x, y in zip(a1, a0):
        np.testing.assert_array_equal(x, y)
    assert u1 == u0
    return e1, a1


@pytest.mark.parametrize("kind,gates", [("givens", 3), ("givens", 6), ("controlled", 4), ("all", 3),
                                        ("all", 5), ("all", 6), ("all", 7)])
@pytest.mark.parametrize("nq,count", [(14, 1), (14, 31), (14, 700), (63, 2500), (64, 33),
                                      (100, 900), (127, 65)])
def test_runs_equal_their_passes(kind, gates, nq, count):
    rng = W.SplitMix64(31 * nq + count + gates)
    init = random_state(nq, count, count + gates, zeros=count // 16)
    parts = [layer(nq, kind, gates, rng) + [W.CZ(0, 2), W.T(1)] for _ in range(3)]
    for eps in (0.0, 1e-14, 0.2):
        err, got = both(nq, init, parts, eps, 1 << 17)
        assert err is None
        orc = OracleState(nq)
        orc.set(*init)
        for g in parts:
            orc.apply(W.to_array(g), eps=eps)
        if eps == 1e-14:   # (at 0 and 0.2 rounding decides which values are kept)
            compare_states(got, orc.get(), eps, atol=1e-12)


@pytest.mark.parametrize("cap", [640, 641, 900, 1279, 1280, 5119, 5120, 6000])
def test_capacity_edges(cap):
    """640 labels; three H make up to 5,120: passes that overflow, overflow on
    the way only, or just fit are reported as by the passes one by one."""
    init = random_state(20, 640, 5)
    parts = [[W.H(15), W.H(16), W.H(17)], [W.H(15), W.H(16), W.H(17)]]
    both(20, init, parts, 1e-14, cap, lay=1)


def test_sector_fills_as_its_passes_fill_it():
    g = W.givens_workload(seed=8, nqubits=70, modes=3, layers=7)
    parts = [g[3 + 70 * k:3 + 70 * (k + 1)] for k in range(7)]
    one = [np.array([0], np.uint64), np.array([7], np.uint64), np.array([1.0]), np.array([0.0])]
    err, got = both(70, one, parts, 1e-14, 60000)
    assert err is None
    orc = OracleState(70)
    orc.set(*one)
    for p in parts:
        orc.apply(p, eps=1e-14)
    compare_states(got, orc.get(), 1e-14)


def test_epochs_of_one_launch_do_not_wrap():
    """The fallback launch draws an epoch for its group stage and one a pass. Drawn
    across the wrap of the 16-bit counter, one turn later the slots it left would
    pass for labels of a state that lies over the older one's entries (2,048
    labels, of which the later states hold 1,025 and lack the others)."""
    n, nq = 2048, 20
    lo = np.arange(n, dtype=np.uint64)
    rng = np.random.default_rng(3)
    re, im = rng.normal(size=n), rng.normal(size=n)
    st = sps.SparseState(nq, 8 * n)
    for o, v in ((sps.SPS_OPT_SMALL_RUN_CAP, 0), (sps.SPS_OPT_EXPAND, 0),
                 (sps.SPS_OPT_LAYER_GATES, 1), (sps.SPS_OPT_AMP_ONLY, 0)):
        st.set_option(o, v)
    one = [np.zeros(1, np.uint64), np.zeros(1, np.uint64), np.ones(1), np.zeros(1)]

    def passes(count):   # one epoch each
        st.set_amplitudes(*one)
        st.apply(np.tile(W.to_array([W.H(19)]), count), 1e-14)

    passes(65532)
    st.set_option(sps.SPS_OPT_AMP_ONLY, 1)
    st.set_amplitudes(np.zeros_like(lo), lo, re, im)
    st.apply(W.to_array([W.H(12), W.H(13), W.H(14)]), 1e-14)   # epochs 65533 ..
    assert st.nnz() == 8 * n
    st.set_option(sps.SPS_OPT_AMP_ONLY, 0)
    passes(65521)
    m = n // 2 + 1
    a = np.zeros(n, np.complex128)
    a[:m] = re[:m] + 1j * im[:m]
    r = np.sqrt(0.5)
    want = np.concatenate([r * a[:n // 2] + r * a[n // 2:], r * a[:n // 2] - r * a[n // 2:]])
    for _ in range(14):   # up to and past the next wrap
        st.set_amplitudes(np.zeros_like(lo[:m]), lo[:m], re[:m], im[:m])
        st.apply(W.to_array([W.H(10)]), 1e-14)
        _, klo, kre, kim = st.get_amplitudes()
        np.testing.assert_array_equal(klo, lo)
        # two products and a sum
        np.testing.assert_allclose(kre + 1j * kim, want, rtol=0, atol=2e-15)
    st.close()


def chain_flags(nq, init, runs, cap, eps=1e-14, lay=4):
    """The profile flags of the fallback launches that had something to do."""
    st = sps.SparseState(nq, cap)
    for o, v in ((sps.SPS_OPT_SMALL_RUN_CAP, 0), (sps.SPS_OPT_EXPAND, 0),
                 (sps.SPS_OPT_LAYER_GATES, lay), (sps.SPS_OPT_PROFILE, 1)):
        st.set_option(o, v)
    st.set_amplitudes(*init)
    for g in runs:
        st.apply(W.to_array(g), eps)
    out = [(r["flags"], r["n_in"], r["n_out"]) for r in st.profile_read() if r["kind"] == 11 and r["n_in"]]
    try:
        st.sync()
    except sps.SpsError as e:
        assert e.status == sps.SPS_ERR_CAPACITY
    st.close()
    return out


@pytest.mark.parametrize("kind,gates,took", [("givens", 3, True), ("givens", 6, True), ("controlled", 4, True),
                                             ("all", 3, True), ("all", 6, True), ("all", 7, False),
                                             ("all", 2, False)])
@pytest.mark.parametrize("nq,count", [(14, 700), (63, 2500), (100, 900)])
def test_which_runs_are_taken_as_groups(kind, gates, took, nq, count):
    rng = W.SplitMix64(nq + gates)
    init = random_state(nq, count, count)
    recs = chain_flags(nq, init, [layer(nq, kind, gates, rng)], 1 << 17)
    assert len(recs) == 1 and recs[0][1] == count
    assert bool(recs[0][0] & 64) == took and count < recs[0][2] <= 1 << 17


def test_members_over_the_capacity_are_handed_back():
    """640 labels with 8 members each: taken at a capacity of 5,120, not of 5,119
    (where the passes find the error)."""
    init = random_state(20, 640, 5)
    run = [W.H(15), W.H(16), W.H(17)]
    (flags, _, n), = chain_flags(20, init, [run], 5120, lay=1)
    assert flags & 64 and n == 5120
    (flags, _, n), = chain_flags(20, init, [run], 5119, lay=1)
    assert not flags & 64 and flags & 128 and n == 2560


def sector(nq, k):
    lo = np.array([sum(1 << q for q in c) for c in itertools.combinations(range(nq), k)], np.uint64)
    rng = np.random.default_rng(k)
    lo = rng.permutation(lo)
    return [np.zeros_like(lo), lo, rng.normal(size=len(lo)), rng.normal(size=len(lo))]


def test_runs_that_cannot_be_taken_are_seldom_tried():
    """Givens layers where some labels activate more than 6 gates and some do not
    (16 qubits, 8 particles): handed back, then 1, 2, 4 .. runs are not tried.
    Seven gates that every label activates: never tried. The state is the passes'."""
    init = sector(16, 8)
    run = [W.Givens(q, q + 8, 0.2 + 0.1 * q) for q in range(8)]
    recs = chain_flags(16, init, [run] * 21, 1 << 14)
    assert len(recs) == 21 and not any(f & 64 for f, _, _ in recs)
    assert [i for i, (f, _, _) in enumerate(recs) if f & 128] == [0, 2, 5, 10, 19]
    both(16, init, [run] * 3, 1e-14, 1 << 14)
    rng = W.SplitMix64(5)
    recs = chain_flags(14, random_state(14, 700, 2), [layer(14, "all", 7, rng)] * 3, 1 << 14)
    assert recs and not any(f & 192 for f, _, _ in recs)


def test_a_run_that_holds_is_taken_after_one_that_does_not():
    init = sector(16, 8)
    bad = [W.Givens(q, q + 8, 0.2 + 0.1 * q) for q in range(8)]
    good = [[W.Givens(q, q + 8, 0.2 + 0.1 * q) for q in range(4)] + [W.H(16 + j)] for j in range(2)]
    recs = chain_flags(20, init, [bad] + good, 1 << 16)
    assert [f & 192 for f, _, _ in recs] == [128, 0, 192]


@pytest.mark.parametrize("kind", ["givens", "all"])
@pytest.mark.parametrize("nq", [20, 100])
def test_large_bounds_take_the_instances_of_three_blocks(kind, nq):
    """Seven gates on 9,000 labels with a bound past 2^20, with the group stage
    (tried, then skipped) and without."""
    rng = W.SplitMix64(nq)
    init = random_state(nq, 9000, 4)
    parts = [layer(nq, kind, 7, rng) + [W.T(1)] for _ in range(2)]
    err, got = both(nq, init, parts, 1e-14, 1 << 21)
    assert err is None
    orc = OracleState(nq)
    orc.set(*init)
    for g in parts:
        orc.apply(W.to_array(g), eps=1e-14)
    # amplitudes of modulus up to 4, seven butterflies twice: some 60 roundings
    compare_states(got, orc.get(), 1e-14, atol=1e-12)
