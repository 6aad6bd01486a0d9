"""The binding's batch calls hand the library the handles of the streams they are given (no compute, no library)."""
import torch

from paper_2609_35115_b200 import binding


class _Lib:
    """Opens streams as ever new handles."""

    def __init__(self):
        self.opened = 0

    def dc_stream_open(self, model, out):
        self.opened += 1
        out._obj.value = 0x1000 + 64 * self.opened
        return 0

    def dc_stream_close(self, handle):
        return 0


def _model():
    m = binding.Model.__new__(binding.Model)
    m.lib, m.handle = _Lib(), None
    return m


# a Stream object that is dropped leaves its address to the next one, closed or not
def test_a_new_stream_is_not_taken_for_the_one_before():
    m, x = _model(), torch.zeros(2, 1, 4)
    for i in range(16):
        a, b = m.open_stream(), m.open_stream()
        assert list(binding._batch_args(m, [a, b], x, x)[1]) == [a.handle.value, b.handle.value]
        assert list(binding._batch_args(m, [b, a], x, x)[1]) == [b.handle.value, a.handle.value]
        if i % 2:
            a.close()
            b.close()
        del a, b


def test_a_closed_stream_has_no_handle():
    m, x = _model(), torch.zeros(1, 1, 4)
    s = m.open_stream()
    binding._batch_args(m, [s], x, x)
    s.close()
    assert list(binding._batch_args(m, [s], x, x)[1]) == [None]
