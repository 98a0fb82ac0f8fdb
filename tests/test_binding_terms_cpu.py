"""Host logic of the Python binding without a GPU: the split-term setting belongs
to the library's handle, which other callers (the C interface, other threads) may
change, so a call that depends on it sets it again every time."""
import pytest

torch = pytest.importorskip("torch")


class _FakeLib:
    def __init__(self):
        self.terms = []

    def cola_create(self, device, out):
        return 0

    def cola_set_split_terms(self, handle, factor, vector):
        self.terms.append((factor, vector))
        return 0


def test_split_terms_are_set_on_every_call(monkeypatch):
    import paper_2309_03060_gb300 as cola
    lib = _FakeLib()
    monkeypatch.setattr(cola, "_lib", lambda: lib)
    ctx = cola.Context(0)
    for terms in (3, 3, (2, 1), (2, 1)):
        ctx._set_split_terms(terms)
    assert lib.terms == [(3, 3), (3, 3), (2, 1), (2, 1)]
