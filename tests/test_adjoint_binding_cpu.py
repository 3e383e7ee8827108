"""The adjoint's workspace has to lie on the device of the run's fields: another device's memory would
fault.  No GPU: tensors and library are fakes, and the check comes before either is used."""
import types

import pytest

from paper_1202_6351_gb300 import lbm


@pytest.mark.parametrize("device,error", [("cuda:1", ValueError), ("cuda:0", None)])
def test_workspace_of_another_device_is_refused(monkeypatch, device, error):
    class Reached(Exception):
        pass

    def field(device):
        return types.SimpleNamespace(is_cuda=True, device=device, data_ptr=lambda: 256, numel=lambda: 1 << 20,
                                     element_size=lambda: 1, is_contiguous=lambda: True)

    def run(*a):
        raise Reached

    torch = pytest.importorskip("torch")
    monkeypatch.setattr(lbm, "_dev", lambda t, shape: t.data_ptr())
    monkeypatch.setattr(torch, "empty", lambda *a, **k: field("cuda:0"))
    L = lbm.Lattice.__new__(lbm.Lattice)
    L.h, L.nx, L.ny, L.lib = None, 8, 8, types.SimpleNamespace(lbm_adjoint_run_in=run)
    with pytest.raises(error or Reached):
        L.adjoint_run(4, 2, field("cuda:0"), field("cuda:0"), workspace=field(device))
