"""The binding's lazily built tables under concurrent first calls: a second thread that arrives while the first one is
still building them gets complete tables."""
import threading

import pytest


@pytest.mark.parametrize("at", ["int16", "uint16", "complex64", "complex128"])
def test_dtype_tables_first_use(monkeypatch, at):
    import torch
    from paper_2309_04841_gb300 import qaoa as Q
    seen = []

    def second():
        try:
            seen.append((Q.state_type_of(torch.empty(1, dtype=torch.complex64)), Q.cost_type_of(torch.empty(1, dtype=torch.int32)),
                         Q.cost_type_of(torch.empty(1, dtype=torch.uint16))))
        except Exception as e:  # noqa: BLE001 (what a caller would see)
            seen.append(repr(e))

    class Torch:
        """torch, with another thread's first call let in where the tables read the dtype `at`."""
        started = False

        def __getattr__(self, name):
            if name == at and not Torch.started:
                Torch.started = True
                t = threading.Thread(target=second)
                t.start()
                t.join(20)
            return getattr(torch, name)

    monkeypatch.setattr(Q, "_dtype_codes", None)
    monkeypatch.setattr(Q, "_torch", lambda proxy=Torch(): proxy)
    assert Q.state_type_of(torch.empty(1, dtype=torch.complex128)) == Q.C128
    assert seen == [(Q.C64, Q.COST_I32, Q.COST_U16)]
