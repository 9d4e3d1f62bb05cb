"""The kept C structs of the binding's buffers follow the tensors: replaced, set
or resized ones are seen by the next call (on the CPU, no launch)."""
import copy
import pickle

import pytest
import torch

rps = pytest.importorskip("paper_2608_11742_gb300.rps")


def addresses(buf):
    st = buf._c()
    return [getattr(st, n) or 0 for n, _ in st._fields_]


def expected(buf, names):
    return [0 if getattr(buf, n) is None else getattr(buf, n).data_ptr() for n in names]


@pytest.mark.parametrize("make", [
    lambda: rps.RowStatsBuf.alloc(5, 3, "cpu"),
    lambda: rps.RowStatsBuf.alloc(5, 0, "cpu"),
    lambda: rps.PivotsBuf.alloc(2, 4, 3, 2, "cpu"),
    lambda: rps.ScoresBuf.alloc(2, 3, 2, "cpu"),
    lambda: rps.CommitBuf.alloc(2, 4, 3, "cpu"),
])
def test_kept_struct_follows_the_tensors(make):
    buf = make()
    names = [n for n, _ in type(buf)._struct._fields_]
    assert addresses(buf) == expected(buf, names)
    assert buf._c() is buf._c(), "kept while nothing moved"
    first = names[0]
    setattr(buf, first, torch.zeros_like(getattr(buf, first)))       # replaced
    assert addresses(buf) == expected(buf, names)
    getattr(buf, first).set_(torch.zeros(64, dtype=getattr(buf, first).dtype))  # another storage
    assert addresses(buf) == expected(buf, names)
    getattr(buf, names[1]).resize_(1 << 16)                           # moved by a resize
    assert addresses(buf) == expected(buf, names)
    for other in (copy.copy(buf), copy.deepcopy(buf), pickle.loads(pickle.dumps(buf))):
        assert addresses(other) == expected(other, names)


def test_a_subclass_may_form_its_own_struct():
    """``c()`` of a subclass is what the calls pass on."""
    class Own(rps.ScoresBuf):
        def c(self):
            return rps.RpsBranchScores(64, 2, 3, 4)

    class Other:
        def c(self):
            return rps.RpsBranchScores(1, 2, 3, 4)

    name = rps.RpsBranchScores._fields_[0][0]
    plain = rps.ScoresBuf.alloc(2, 3, 2, "cpu")
    own = Own(*(getattr(plain, n) for n, _ in rps.RpsBranchScores._fields_))
    assert getattr(rps._cs(own), name) == 64
    assert getattr(rps._cs(Other()), name) == 1
    assert getattr(rps._cs(plain), name) == getattr(plain, name).data_ptr()
