"""The Python binding's own work, on the CPU: what State.run() looks up and refuses."""
import pytest

from paper_2503_15118_gb300 import sqs as S


@pytest.fixture
def state():
    """A binding object without a device state behind it."""
    st = S.State.__new__(S.State)
    st.lib = S.load()
    st.h = None
    st.widths, st.kw, st._tables = [4, 4], 1, {}
    yield st
    st.h = None  # nothing to destroy


def test_a_closed_state_refuses_a_circuit_as_it_refuses_a_gate(state):
    circ = {"widths": [4, 4], "gates": [("h", 0, 0, ())]}
    with pytest.raises(S.SqsError) as one:
        state.apply(circ["gates"][0])
    with pytest.raises(S.SqsError) as run:
        state.run(circ)
    assert (run.value.status, str(run.value)) == (one.value.status, str(one.value))
    assert state.run({"widths": [4, 4], "gates": []}) is state
