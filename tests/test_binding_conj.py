"""A lazily conjugated symbol tensor is refused: its memory holds the values before conjugation."""
import pytest


def test_conjugated_symbols_are_refused():
    import torch

    import paper_2405_01808_gb300 as g

    x = torch.ones((2, 32), dtype=torch.complex64)
    assert g._interleaved(x) == x.data_ptr()
    with pytest.raises(RuntimeError):
        g._interleaved(x.conj())
    y = x.conj().resolve_conj()
    assert g._interleaved(y) == y.data_ptr()
