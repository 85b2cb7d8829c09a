"""Fused runs on an allocator that refuses their buffers.

A held run needs more memory than its steps one by one (a slot per setting of
the varying bits, or room for every group to fill).  Where the allocator has
none, the steps run one by one, after the operations queued before them, and
give the same state."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LIMIT = 12 << 20  # bytes the allocator gives at once


@pytest.fixture(scope="module")
def sqs():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_15118_gb300 import sqs as S
    S.load()
    return S


def _whole_groups(bits, targets, groups, seed):
    """`groups` random keys of `bits` bits, each with every setting of `targets`."""
    rng = np.random.default_rng(seed)
    clear = np.uint64(sum(1 << t for t in targets))
    base = np.unique(rng.integers(0, 1 << bits, size=groups, dtype=np.uint64) & ~clear)
    keys = base
    for t in targets:
        keys = np.concatenate([keys, keys | np.uint64(1 << t)])
    amps = rng.normal(size=keys.size) + 1j * rng.normal(size=keys.size)
    return keys, amps / np.linalg.norm(amps)


@pytest.mark.parametrize("kind", ["addressed", "bucketed"])
@pytest.mark.parametrize("before", [(), (("x", 0, 7, ()), ("phase", ((0, 9, 1),), 0.4), ("prune", 1e-14))])
def test_refused_buffers(sqs, monkeypatch, kind, before):
    # 2^20 slots of 16 bytes; room for 40000 x 2^5 branches of 16 bytes.
    bits, targets, groups = (20, (1, 4, 11, 17), 64) if kind == "addressed" else \
        (40, (1, 4, 11, 17, 38), 1250)
    keys, amps = _whole_groups(bits, targets, groups, len(before))
    run = [("h", 0, targets[0], ())]
    run += [("ry", 0, t, 0.3 + t, ((0, p, 1),)) for p, t in zip(targets, targets[1:])]

    def state(merge=0):
        st = sqs.State([bits], merge=merge)
        st.import_(keys, None, amps)
        for g in list(before) + run:
            st.apply(g)
        st.flush()
        return st

    assert state().stats()["runs_fused"] == 1
    given = sqs._TorchAllocator.alloc
    monkeypatch.setattr(sqs._TorchAllocator, "alloc",
                        lambda self, ctx, n, stream: None if n > LIMIT else given(self, ctx, n, stream))
    got, ref = state(), state(sqs.MERGE_PLAIN)
    assert got.stats()["runs_fused"] == 0
    a, b = got.to_dict(), ref.to_dict()
    assert set(a) == set(b) and all(a[k] == b[k] for k in a)
    assert got.peak_nnz() == ref.peak_nnz()
