"""A batch takes one signal, filter bank and output per problem: lists of another
length are refused before a pointer table is made (the kernels read as many
pointers as the batch has problems).  No GPU: the batch is a stand-in whose
launch records that it was reached."""
import pytest
import torch

import paper_1910_01972_gb300 as ols


class Batch(ols.BatchPlan):
    def __init__(self, B):
        self._h, self.device, self.B = None, torch.device("cpu"), B
        self.Ns, self.M, self.F, self.Nout = [8] * B, [3] * B, [2] * B, [6] * B
        self.launched = None

    def launch(self, s_table, y_table):
        self.launched = s_table.tolist(), y_table.tolist()


def signals(n):
    return [torch.zeros(8, dtype=torch.complex64) for _ in range(n)]


def outputs(n):
    return [torch.zeros((2, 6), dtype=torch.complex64) for _ in range(n)]


@pytest.mark.parametrize("ns,ny", [(2, 3), (0, 3), (3, 2), (4, 3), (3, 4), (2, 2)])
def test_lists_of_another_length_are_refused(ns, ny):
    b = Batch(3)
    with pytest.raises((ValueError, IndexError)):
        b.convolve(signals(ns), outputs(ny))
    assert b.launched is None
    if ny == 3:
        with pytest.raises((ValueError, IndexError)):
            b.convolve(signals(ns))
        assert b.launched is None


def test_full_lists_keep_their_order():
    b, s, y = Batch(3), signals(3), outputs(3)
    assert b.convolve(s, y) is y
    assert b.launched == ([t.data_ptr() for t in s], [t.data_ptr() for t in y])


@pytest.mark.parametrize("n", [0, 2, 4])
def test_filter_lists_of_another_length_are_refused(n, monkeypatch):
    reached = []
    monkeypatch.setattr(ols._native, "ols_batch_set_filters", lambda *a: reached.append(a) or 0)
    monkeypatch.setattr(ols, "_stream_ptr", lambda device: 0)
    with pytest.raises((ValueError, IndexError)):
        Batch(3).set_filters([torch.zeros((2, 3), dtype=torch.complex64) for _ in range(n)])
    assert not reached
