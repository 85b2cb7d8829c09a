"""Long queued runs on states large enough for the pass on bit planes (2^19 slots; with
factors 2^20, or 2^22 for a key word of more than 32 bits), dense and after a merge
(segments part full), against the same gates flushed three at a time, which takes the
pass branch by branch: keys bit for bit, amplitudes to the roundings of the folded
factors.  The kernels that ran are read from the profiler."""
import numpy as np
import pytest

import oracle
from paper_2503_15118_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KINDS = ("x", "cx", "ccx", "add", "sub", "swap")
FACTORS = KINDS + ("phase", "cphase")


@pytest.fixture(scope="module")
def sqs():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_15118_gb300 import sqs as S
    S.load()
    return S


def _gates(rng, widths, n, factors):
    qs = [(r, b) for r, w in enumerate(widths) for b in range(w)]
    out = []
    for _ in range(n):
        g = W._draw_gate(rng, FACTORS if factors else KINDS, qs, widths, 0)
        if rng.random() < 0.3 and g[0] in ("add", "sub", "swap"):
            used = {g[1], g[2]}
            free = [q for q in qs if q[0] not in used]
            if free:  # a controlled operation, values 0 and 1
                c = tuple(free[i] + (int(rng.integers(2)),)
                          for i in rng.choice(len(free), size=min(3, len(free)), replace=False))
                g = g[:-1] + (c,)
        if factors and rng.random() < 0.1:  # a predicate over most of the key
            some = [q + (int(rng.integers(2)),) for q in qs[:: int(rng.integers(2, 5))]]
            g = ("phase", tuple(some), 0.31)
        out.append(g)
    return out


def _kernels(f):
    """Names of the kernels that f() launches (None where the profiler gives none)."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        f()
        torch.cuda.synchronize()
    names = {e.key for e in p.key_averages() if "sqs::" in e.key}
    return names or None


def _pass(sqs, widths, amp32, state, gates, every, segmented, on_planes=True):
    st = sqs.State(widths, amp32=amp32, merge=sqs.MERGE_HASH | sqs.FUSE_OFF)
    st.import_(*state)
    if segmented:
        st.ry(len(widths) - 1, 1, 0.83)
    st.sync()

    def go():
        for i, g in enumerate(gates):
            st.apply(g)
            if every and i % every == every - 1:
                st.flush()
        st.flush()

    names = _kernels(go)
    if names is not None:
        planes = any("k_apply_planes" in n for n in names)
        singly = any("k_apply_inplace" in n for n in names)
        assert planes if on_planes and not every else singly and not planes, names
    return st


def _compare(one, three, amp32, n_factors):
    (l1, h1, a1), (l2, h2, a2) = one.export(), three.export()
    assert np.array_equal(l1, l2) and np.array_equal(h1, h2)
    # Phases of one launch are folded into one factor: on either side at most one
    # rounding of a factor (1 unit) and of a complex product (sqrt(5)) per phase.
    tol = 2 * 3.25 * n_factors * (2.0 ** -24 if amp32 else 2.0 ** -53)
    assert np.max(np.abs(a1 - a2) / np.abs(a2)) <= tol
    assert one.nnz() == three.nnz() and one.peak_nnz() == three.peak_nnz()
    return l1, h1, a1


def _fp32(state, amp32):
    return state[:2] + (state[2].astype(np.complex64).astype(np.complex128),) if amp32 else state


@pytest.mark.parametrize("amp32", [False, True])
@pytest.mark.parametrize("widths", [[9, 14, 9], [16, 16, 16, 16], [31, 33, 31, 33],
                                    [64, 13, 13, 20]])
@pytest.mark.parametrize("extra,length", [(0, 12), (1, 90), (4095, 40), (4097 + 31, 150)])
def test_dense_states(sqs, widths, amp32, extra, length):
    """Whole tiles of 4096, one branch over, one short of a tile; a run of the
    fewest operations that goes to planes, and runs of more than a launch."""
    rng = np.random.default_rng(sum(widths) + extra)
    if length == 12:  # exactly so many operations after packing: controlled X
        qs = [(r, b) for r, w in enumerate(widths) for b in range(w)]
        gates = [("x",) + qs[int(rng.integers(1, len(qs)))] + ((qs[0] + (i & 1,),),)
                 for i in range(12)]
    else:
        gates = _gates(rng, widths, length, False)
    state = _fp32(W.random_state(widths, (1 << 19) + extra, seed=extra), amp32)
    one = _pass(sqs, widths, amp32, state, gates, 0, False)
    three = _pass(sqs, widths, amp32, state, gates, 3, False)
    _compare(one, three, amp32, 0)


@pytest.mark.parametrize("amp32", [False, True])
@pytest.mark.parametrize("widths,size", [([9, 14, 9], 20), ([31, 33, 31, 33], 20),
                                         ([64, 13, 13, 20], 20), ([16, 16, 16, 16], 22)])
@pytest.mark.parametrize("length", [40, 90])
def test_factors(sqs, widths, size, amp32, length):
    """Phases among the operations: more predicate bits or factors than the smaller
    list takes, indices of a few bits and of all ten."""
    gates = _gates(np.random.default_rng(sum(widths)), widths, length, True)
    n = (1 << size) + 33
    i = np.arange(n, dtype=np.uint64)
    lo = i * np.uint64(0x9E3779B97F4A7C15)  # odd: distinct below 2^22 in the low 32 bits too
    hi = i >> np.uint64(2) if sum(widths) > 64 else np.zeros(n, np.uint64)
    if sum(widths) < 64:
        lo &= np.uint64((1 << sum(widths)) - 1)
    elif sum(widths) < 128:
        hi &= np.uint64((1 << (sum(widths) - 64)) - 1)
    rng = np.random.default_rng(length)
    a = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    state = _fp32((lo, hi, a), amp32)
    one = _pass(sqs, widths, amp32, state, gates, 0, False)
    three = _pass(sqs, widths, amp32, state, gates, 3, False)
    _compare(one, three, amp32, len(gates))


@pytest.mark.parametrize("n,length,phases", [(1 << 19, 30, 2), (1 << 20, 14, 2), ((1 << 19) - 1, 30, 0),
                                             (1 << 20, 11, 0)])
def test_lists_that_stay_branch_by_branch(sqs, n, length, phases):
    """Too few slots or operations for planes: with a factor table the line is higher."""
    widths = [20, 16]
    gates = [("x", 1, i % 16, ((0, i % 20, i & 1),)) for i in range(length - phases)]
    gates += [("phase", ((1, i, 1),), 0.3) for i in range(phases)]
    state = W.random_state(widths, n, seed=1)
    one = _pass(sqs, widths, False, state, gates, 0, False, on_planes=False)
    three = _pass(sqs, widths, False, state, gates, 3, False)
    _compare(one, three, False, phases)


@pytest.mark.parametrize("amp32", [False, True])
@pytest.mark.parametrize("widths", [[16, 16, 16, 16], [31, 33, 31, 33]])
def test_segmented_states(sqs, widths, amp32):
    """After a merge every segment holds a number of branches of its own.  (The
    storage order after a merge is not fixed; the sorted exports are compared.)"""
    factors = sum(widths) > 64
    gates = _gates(np.random.default_rng(4), widths, 70, factors)
    state = _fp32(W.random_state(widths, (1 << 18) + 77, seed=6, pair_fraction=0.4,
                                 target=(len(widths) - 1, 1)), amp32)
    one = _pass(sqs, widths, amp32, state, gates, 0, True)
    three = _pass(sqs, widths, amp32, state, gates, 3, True)
    _compare(one, three, amp32, len(gates))


def test_against_the_oracle(sqs):
    widths = [20, 32, 32]
    gates = _gates(np.random.default_rng(2), widths, 30, True)
    state = W.random_state(widths, (1 << 20) + 1003, seed=8)
    got = _pass(sqs, widths, False, state, gates, 0, False).export()
    o = oracle.OracleState(widths, 1e-14)
    o.import_(*state)
    for g in gates:
        o.apply(g)
    lo, hi, ref = o.export()
    assert np.array_equal(got[0], lo) and np.array_equal(got[1], hi)
    assert np.max(np.abs(got[2] - ref)) <= 1e-12 * np.max(np.abs(ref))
