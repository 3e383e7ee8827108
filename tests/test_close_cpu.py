"""A destroy call that reports an error has freed the handle all the same, so closing an object a second
time (its finaliser does) must not pass the handle to the library again.  No GPU: the library is a fake."""
import ctypes as C

import pytest

from paper_1202_6351_gb300 import lbm


class FakeLibrary:
    def __init__(self):
        self.destroyed = []

    def _destroy(self, h):
        self.destroyed.append(h)
        return lbm.LBM_ECUDA  # an error left behind by earlier work

    lbm_destroy = lbm_batch_destroy = lbm3_destroy = _destroy

    def lbm_last_error(self):
        return b"fake"


@pytest.mark.parametrize("cls,attr", [(lbm.Lattice, "h"), (lbm.Batch, "b"), (lbm.Lattice3, "h")])
def test_a_handle_is_destroyed_once(monkeypatch, cls, attr):
    fake = FakeLibrary()
    monkeypatch.setattr(lbm, "load_library", lambda *a: fake)
    obj = cls.__new__(cls)
    obj.lib = fake
    setattr(obj, attr, C.c_void_p(1))
    try:
        with pytest.raises(lbm.LBMError):
            obj.close()
        obj.close()
    finally:
        setattr(obj, attr, None)
    assert len(fake.destroyed) == 1
