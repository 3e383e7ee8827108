"""A call that finds no device memory is tried once more after PyTorch's allocator has given back what
it holds unused.  No GPU: the call and the allocator are fakes."""
import sys
import types

import pytest

from paper_1202_6351_gb300 import lbm


@pytest.mark.parametrize("answers,initialized,calls,emptied,code", [
    ([lbm.LBM_OK], True, 1, 0, None),
    ([lbm.LBM_ENOMEM, lbm.LBM_OK], True, 2, 1, None),
    ([lbm.LBM_ENOMEM, lbm.LBM_ENOMEM], True, 2, 1, lbm.LBM_ENOMEM),
    ([lbm.LBM_ENOMEM, lbm.LBM_OK], False, 1, 0, lbm.LBM_ENOMEM),  # PyTorch holds nothing
    ([lbm.LBM_EINVAL, lbm.LBM_OK], True, 1, 0, lbm.LBM_EINVAL),
])
def test_one_more_try_after_the_cache_is_emptied(monkeypatch, answers, initialized, calls, emptied, code):
    log = []
    cuda = types.SimpleNamespace(is_initialized=lambda: initialized, empty_cache=lambda: log.append("empty"))
    monkeypatch.setitem(sys.modules, "torch", types.SimpleNamespace(cuda=cuda))

    def call(a, b):
        log.append((a, b))
        return answers[log.count((a, b)) - 1]

    if code is None:
        lbm._check_alloc(call, 1, 2)
    else:
        with pytest.raises(lbm.LBMError) as e:
            lbm._check_alloc(call, 1, 2)
        assert e.value.code == code
    assert log.count((1, 2)) == calls and log.count("empty") == emptied
