"""What a graph capture reserves, and for how long: the buffers a live graph holds stay
where they are, and once every graph is destroyed the state is as free as before."""
import numpy as np
import pytest

from paper_2503_15118_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sqs():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_15118_gb300 import sqs as S
    S.load()
    return S


def _state(sqs, widths, **kw):
    import torch
    return sqs.State(widths, stream=torch.cuda.Stream().cuda_stream, **kw)


SMALL = {"widths": [], "eps": 1e-14, "tables": [], "gates": [("h", 0, 0, ()), ("h", 0, 1, ())]}


def test_runs_grow_buffers_again_after_the_last_graph(sqs):
    """Three steps on 2^14 branches of a 40-bit register: one bucketed run, whose
    buffers are larger than those of the captures before it."""
    widths = [40]
    lo, hi, amps = W.random_state(widths, 1 << 14, seed=4)
    gates = [("ry", 0, b, 0.3 + b, ()) for b in (3, 20, 33)]

    def run(st):
        before = st.stats()["runs_fused"]
        st.import_(lo, hi, amps)
        for g in gates:
            st.apply(g)
        out = st.to_dict()
        return out, st.stats()["runs_fused"] - before

    want, fused = run(_state(sqs, widths))
    assert fused == 1
    st = _state(sqs, widths)
    first, second = st.capture(SMALL, 64), st.capture(SMALL, 64)
    first.close()
    second.launch()
    st.sync()
    second.close()
    got, fused = run(st)
    assert got == want and fused == 1


def test_a_later_capture_reserves_its_own_slots(sqs):
    """Four steps on a state with 21 varying bits, one run of two launches: 2^21
    slots, which a bound of 2^18 branches reserves and one of 2^10 does not."""
    widths = [21, 2]
    gates = [("h", 0, b, ()) for b in range(8)] + [("mulc", 0, 3 ** 12, ())]
    gates += [("ry", 0, b, 0.3, ()) for b in (9, 12, 15, 18)] + [("x", 0, 2, ())]
    circ = {"widths": widths, "eps": 1e-14, "tables": [], "gates": gates}

    def replay(st):
        graph = st.capture(circ, 1 << 18)
        n = st.launch_count()
        graph.launch()
        n = st.launch_count() - n
        out = st.to_dict()
        graph.close()
        return n, out

    fresh = _state(sqs, widths, merge=sqs.FUSE_ALWAYS)
    used = _state(sqs, widths, merge=sqs.FUSE_ALWAYS)
    used.capture(SMALL, 1 << 10).close()
    (n0, want), (n1, got) = replay(fresh), replay(used)
    assert got == want and n1 == n0


def test_graphs_and_states_closed_in_either_order(sqs):
    a, b = _state(sqs, [4]), _state(sqs, [4])
    ga, gb, gc = a.capture(SMALL, 16), b.capture(SMALL, 16), b.capture(SMALL, 16)
    ga.close()
    a.close()
    gb.close()
    b.close()
    gc.close()


@pytest.mark.parametrize("amp32", [False, True])
def test_capture_without_room_for_slots(sqs, monkeypatch, amp32):
    """The slots of addressed runs are larger than all other buffers of a small
    bound; where the allocator has none, the captured steps run one by one."""
    widths = [8, 8, 8]
    circ = W.random_circuit(widths, 60, seed=5, kinds=("x", "cx", "ry", "phase", "add"))
    # Rotations back to back, undone again: what an addressed run takes.
    run = [("ry", 1, b, 0.2 + b, ()) for b in range(4)]
    circ["gates"] = [("h", 0, b, ()) for b in range(4)] + circ["gates"][:20] + run + \
        [W.inverse_gate(g) for g in reversed(run)]
    bound = 1 << 13
    eager = _state(sqs, widths, amp32=amp32).run(circ)
    want = eager.to_dict()
    assert eager.peak_nnz() <= bound
    given = sqs._TorchAllocator.alloc
    monkeypatch.setattr(sqs._TorchAllocator, "alloc",
                        lambda self, ctx, n, s: None if n > 4 << 20 else given(self, ctx, n, s))
    st = _state(sqs, widths, amp32=amp32)
    graph = st.capture(circ, bound)
    for _ in range(2):
        graph.launch()
        assert st.to_dict() == want
    graph.close()


@pytest.mark.parametrize("before", [0, 1, 2])
@pytest.mark.parametrize("after", ["prune", "diag"])
def test_a_small_merge_leaves_room_for_what_follows(sqs, before, after):
    """A state whose two buffers differ in size (an import grows the one it fills): what
    follows the merge of a captured circuit writes as many segments as the merge into
    the other buffer."""
    widths = [13, 3]
    gates = [("h", 0, b, ()) for b in range(13)] + [("phase", ((0, 5, 1),), 0.4)]
    gates += [("prune", 1e-14)] * before + [("ry", 0, 5, 0.3, ()), ("x", 1, 0, ((0, 2, 1),))]
    gates += [("prune", 1e-14)] if after == "prune" else \
        [("u1q", 0, 1, [[0.6 + 0.8j, 0], [0, 1j]], ())]
    circ = {"widths": widths, "eps": 1e-14, "tables": [], "gates": gates}
    want = _state(sqs, widths).run(circ).to_dict()
    st = _state(sqs, widths)
    st.import_(np.arange(50000, dtype=np.uint64), None, np.full(50000, 50000.0 ** -0.5, complex))
    graph = st.capture(circ, 1 << 13)
    for _ in range(2):
        graph.launch()
        assert st.to_dict() == want
    st.reset()
    st.run(circ)             # eager again: the graph's buffers stay where they are
    assert st.to_dict() == want
    graph.launch()
    assert st.to_dict() == want
    graph.close()
