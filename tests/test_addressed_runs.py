"""Rotations that read their QRAM table themselves, and fused runs by direct
addressing.

A register-valued rotation between a QRAM load into its angle register and
the unload runs as one step when no table entry depends on the rotated qubit;
held steps (and a phase between two of them) whose state has few varying key
bits run by direct addressing, also where a step reads or repeats another
step's target.  Both must give the state of the operations one by one
(SQS_MERGE_PLAIN) bit for bit, peak count included, and the oracle's within
its tolerance."""
import math

import numpy as np
import pytest

import oracle
from paper_2503_15118_gb300 import qlss
from paper_2503_15118_gb300 import workloads as W
from tests.helpers import compare_states

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sqs():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_15118_gb300 import sqs as S
    S.load()
    return S


def _compare(sqs, circ, amp32=False, merge=None, fused=None, with_oracle=True):
    a = sqs.State(circ["widths"], amp32=amp32, eps=circ["eps"],
                  merge=sqs.FUSE_ALWAYS if merge is None else merge).run(circ)
    b = sqs.State(circ["widths"], amp32=amp32, eps=circ["eps"], merge=sqs.MERGE_PLAIN).run(circ)
    da, db = a.to_dict(), b.to_dict()
    assert set(da) == set(db)
    assert all(da[k] == db[k] for k in da)
    assert a.peak_nnz() == b.peak_nnz()
    if fused is not None:
        assert a.stats()["runs_fused"] >= fused, a.stats()
    if not amp32 and with_oracle:
        ref = oracle.run_circuit(circ).to_dict()
        assert set(da) == set(ref)
        assert compare_states(da, ref, eps=circ["eps"], atol=1e-12) >= 1 - 1e-12
    return a


def _tables(rng, n_bits, free_bit, entries):
    """A table whose entries do not depend on address bit `free_bit` (None: on
    every bit), cut to `entries` entries."""
    t = rng.integers(0, 2 ** 32, size=1 << n_bits, dtype=np.uint64).astype(np.uint32)
    if free_bit is not None:
        i = np.arange(1 << n_bits)
        t = t[i & ~(1 << free_bit)]
    return t[:entries]


@pytest.mark.parametrize("amp32", [False, True])
@pytest.mark.parametrize("pad", [1, 60])
@pytest.mark.parametrize("free,entries", [(1, 64), (None, 64), (1, 37), (1, 33), (5, 32)])
def test_rotation_reads_its_table(sqs, amp32, pad, free, entries):
    """Load, rotations, unload over an address of two registers (6 bits): the
    target inside the address on a bit the table ignores, on one it does not
    (a table of 37 or 33 entries reads 0 past its end, so that flipping a bit
    can leave it), and outside the address.  pad = 60 puts the angle register
    across the two key words."""
    rng = np.random.default_rng(10 + entries + pad)
    widths = [4, 2, pad, 32, 2]
    t = _tables(rng, 6, free, entries)
    u = _tables(rng, 6, 5, 64)
    gates = [("h", 0, b, ()) for b in range(3)] + [("h", 1, 1, ()), ("h", 4, 0, ())]
    sc = qlss.ANGLE_SCALE
    for tab, targets in ((0, [(0, 1), (4, 1)]), (1, [(1, 1), (0, 0)]), (0, [(0, 1)])):
        gates.append(("qload", (0, 2), 3, tab))
        for r, b in targets:
            gates.append(("ry_reg", r, b, 3, sc, 0.1, ((4, 0, 1),)))
        gates.append(("qunload", (0, 2), 3, tab))
    gates += [("qload", (0, 2), 3, 0), ("x", 3, 5, ()), ("ry_reg", 0, 1, 3, sc, 0.0, ()),
              ("x", 3, 5, ()), ("qunload", (0, 2), 3, 0), ("qload", (0, 2), 3, 1)]
    circ = {"widths": widths, "eps": 1e-14, "tables": [t, u], "gates": gates}
    for merge in (sqs.FUSE_ALWAYS, sqs.FUSE_OFF, sqs.MERGE_HASH, sqs.MERGE_SORT):
        _compare(sqs, circ, amp32, merge)


@pytest.mark.parametrize("amp32", [False, True])
@pytest.mark.parametrize("widths", [[5, 4, 3], [9, 6, 3], [5, 57, 4, 3], [3, 62, 12, 2]])
def test_runs_with_repeated_and_read_targets(sqs, amp32, widths):
    """Random steps on few targets with controls and angle registers on other
    targets, single phases between steps, and Hadamards undone on the spot
    (copy-pair folds inside a run); small states (part of one area) up to
    several areas, slots spread over both key words."""
    rng = np.random.default_rng(sum(widths))
    few = [(0, b) for b in range(min(5, widths[0]))] + [(len(widths) - 2, b) for b in range(3)]
    last = len(widths) - 1
    gates = [("h", 0, b, ()) for b in range(widths[0])] + [("x", last, 0, ())]
    gates += [("h", len(widths) - 2, b, ()) for b in range(min(widths[-2], 8))]
    for _ in range(45):
        (r, b), (cr, cb) = (few[i] for i in rng.choice(len(few), size=2, replace=False))
        ctrl = ((cr, cb, int(rng.integers(2))),) if rng.random() < 0.6 else ()
        k = int(rng.integers(7))
        if k == 0:
            gates.append(("h", r, b, ctrl))
        elif k == 1:
            gates.append(("u1q", r, b, W.random_unitary(rng), ctrl))
        elif k == 2:
            gates.append(("ry", r, b, float(rng.uniform(0, 6)), ctrl))
        elif k == 3:
            gates.append(("ry_reg", r, b, last if rng.random() < 0.5 else
                          (0 if r != 0 else len(widths) - 2), 0.41, 0.2, ctrl))
        elif k == 4:
            gates.append(("phase", ((r, b, 1),) + ctrl, float(rng.uniform(0, 6))))
        elif k == 5:
            gates += [("h", last, 1, ()), ("h", last, 1, ())]
        else:
            gates.append(("x", r, b, ctrl))
    circ = {"widths": widths, "eps": 1e-14, "tables": [], "gates": gates}
    _compare(sqs, circ, amp32, fused=3)


@pytest.mark.parametrize("n,inst", [(3, 0), (6, 0), (4, 9)])
def test_walks_run_addressed(sqs, n, inst):
    """Whole walk steps, one system and a batch (a step counter stays known
    constant through its additions), with the default choice of paths."""
    if inst:
        cfg = qlss.config5(seed=3, n_inst=inst, n_max=n, T=20)
        circ = qlss.batched_circuit(cfg, 2)
    else:
        cfg = qlss.config4(seed=3, N=1 << n, half_band=2, kappa=10.0, T=20)
        circ = qlss.walk_circuit(cfg, n_steps=12)
        circ["gates"] = circ["gates"][:n] + circ["gates"][-2 * len(qlss.walk_step(cfg, 0.5)):]
    a = _compare(sqs, circ, merge=0)
    s = a.stats()
    assert s["runs_fused"] > 0 and s["steps_hash"] == 0


def test_arithmetic_on_known_fields(sqs):
    """Additions, multiplications and loads on registers known constant, under
    controls known to hold, known to fail and unknown, then steps whose
    shortcuts rely on what is known."""
    widths = [4, 4, 5, 4]
    t = np.arange(16, dtype=np.uint8)
    gates = [("x", 0, 1, ()), ("add", 1, 0, 0, ()), ("add", 1, -1, 5, ((0, 1, 1),)),
             ("sub", 1, 0, 0, ((0, 0, 1),)), ("mulc", 1, 7, ()), ("h", 3, 0, ()),
             ("add", 2, 1, 0, ((3, 0, 1),)), ("h", 1, 0, ()), ("h", 2, 1, ()),
             ("sub", 0, -1, 3, ()), ("h", 0, 0, ()), ("qload", 1, 2, 0), ("qload", 1, 2, 0),
             ("h", 2, 4, ()), ("add", 3, 1, 0, ()), ("h", 3, 1, ()), ("h", 1, 3, ((0, 3, 1),))]
    circ = {"widths": widths, "eps": 1e-14, "tables": [t], "gates": gates}
    for merge in (0, sqs.FUSE_ALWAYS, sqs.MERGE_SORT):
        _compare(sqs, circ, merge=merge)


def test_eager_runs_leave_a_captured_graph_its_buffers(sqs):
    """An addressed run may hold up to a branch per slot; after a capture it
    runs only where that fits the buffers the graph holds."""
    import torch
    widths = [10, 4]
    gates = [("h", 0, b, ()) for b in range(6)] + [("x", 1, 0, ((0, 1, 1),))]
    gates += [("ry", 0, b, 0.3 + b, ()) for b in range(6, 10)]
    gates += [("ry", 0, b, -0.3 - b, ()) for b in range(6, 10)]
    circ = {"widths": widths, "eps": 1e-14, "tables": [], "gates": gates}
    stream = torch.cuda.Stream()
    st = sqs.State(widths, stream=stream.cuda_stream, merge=sqs.FUSE_ALWAYS)
    graph = st.capture(circ, static_bound=1 << 10)
    graph.launch()
    want = st.to_dict()
    st.reset()
    st.run(circ)
    assert st.to_dict() == want
    graph.launch()
    assert st.to_dict() == want
    graph.close()
    st.close()


@pytest.mark.parametrize("bits", [10, 11, 19])
def test_slot_areas_at_their_edges(sqs, bits):
    """One area exactly, two, and many; 12 targets and every group size of the
    last run; each basis amplitude against the product of its rotations."""
    widths = [bits]
    th = [0.2 + 0.05 * b for b in range(bits)]
    gates = [("ry", 0, b, th[b], ()) for b in range(bits)]
    circ = {"widths": widths, "eps": 0.0, "tables": [], "gates": gates}
    st = sqs.State(widths, eps=0.0, merge=sqs.FUSE_ALWAYS).run(circ)
    lo, _, a = st.export()
    assert lo.shape[0] == 1 << bits and np.array_equal(lo, np.arange(1 << bits, dtype=np.uint64))
    want = np.ones(1)
    for t in reversed(th):  # register bit 0 varies fastest
        want = np.kron(want, [math.cos(t / 2), math.sin(t / 2)])
    # Each rotation rounds once: at most `bits` units of 2^-53 relative, and
    # the host's product as many.
    assert np.max(np.abs(a - want) / want) <= 4 * bits * 2.0 ** -53
    assert st.stats()["runs_fused"] == (bits + 11) // 12


@pytest.mark.parametrize("amp32", [False, True])
@pytest.mark.parametrize("widths", [[20, 12], [30, 34, 20]])
@pytest.mark.parametrize("spread", [0, 3, 9, 13])
def test_bucketed_runs_on_wide_states(sqs, amp32, widths, spread):
    """More varying bits than can be addressed: runs of up to five targets over
    hash buckets, with repeated targets, controls and angle registers inside
    and outside the run, phases between steps, runs longer than five targets
    (split), rotations undone inside a run, growth and an almost empty state;
    2^spread branches when the runs begin (one bucket up to many)."""
    rng = np.random.default_rng(spread + sum(widths))
    lastr = len(widths) - 1
    gates = [("h", 0, b, ()) for b in range(spread)]
    # Every bit varies (or is not known constant) from here on.
    gates += [("mulc", r, int(rng.integers(1 << 20)) * 2 + 1, ((0, 0, 0),)) for r in range(1, lastr + 1)]
    gates += [("add", r, 0 if r else lastr, 0, ()) for r in range(lastr + 1)]
    for n_t, ctrls in ((4, False), (5, True), (7, True), (2, True)):
        picks = [(int(r), int(rng.integers(widths[r]))) for r in rng.integers(lastr + 1, size=n_t)]
        th = rng.uniform(0.2, 6, size=n_t)
        steps = []
        for (r, b), t in zip(picks, th):
            c = ()
            if ctrls and rng.random() < 0.6:
                cr, cb = picks[int(rng.integers(n_t))] if rng.random() < 0.5 else (lastr, 3)
                if (cr, cb) != (r, b):
                    c = ((cr, cb, int(rng.integers(2))),)
            k = int(rng.integers(3))
            if k == 0:
                steps.append(("ry", r, b, float(t), c))
            elif k == 1:
                steps.append(("u1q", r, b, W.random_unitary(rng), c))
            else:
                steps.append(("ry_reg", r, b, 0 if r else lastr, 0.37, 0.1, c))
        gates += steps[: n_t // 2] + [("phase", ((0, 1, 1), picks[0] + (0,)), 0.7)] + steps[n_t // 2:]
        gates += [W.inverse_gate(g) for g in reversed(steps[n_t // 2:])]
        gates += [("x", 0, 2, ((lastr, 1, 1),)), ("add", lastr, 0, 0, ())]
    circ = {"widths": widths, "eps": 1e-14, "tables": [], "gates": gates}
    if amp32:
        circ["eps"] = 1e-7
    # Angles of up to 0.37 * 2^30 radians carry an FP64 rounding of their own of
    # 10^-8 and more, so only the steps one by one are an exact reference.
    _compare(sqs, circ, amp32, merge=0, fused=2, with_oracle=False)


def test_bucketed_runs_of_whole_groups(sqs):
    """Every group of the run holds one of its 2^5 members, or all of them: the
    buckets hold whole groups without an overflow (2^17 branches)."""
    widths = [17, 60]
    spread = [("h", 0, b, ()) for b in range(17)]
    run = [("ry", 0, b, 0.3 + b, ()) for b in (0, 3, 7, 11, 16)]
    run += [("u1q", 0, b, W.random_unitary(np.random.default_rng(b)), ()) for b in (16, 0)]
    mixed = [("add", 1, 0, 0, ()), ("mulc", 1, 977, ()), ("mulc", 0, 31, ())]
    for gates in (spread + mixed + run,                # groups of one branch
                  spread + mixed[2:] + [("mulc", 1, 3, ((0, 5, 1),))] + run):  # whole groups
        c = {"widths": widths, "eps": 1e-14, "tables": [], "gates": gates}
        a = sqs.State(c["widths"]).run(c)
        b = sqs.State(c["widths"], merge=sqs.MERGE_PLAIN).run(c)
        x, y = a.export(), b.export()
        assert all(np.array_equal(p, q) for p, q in zip(x, y))
        assert a.peak_nnz() == b.peak_nnz()
