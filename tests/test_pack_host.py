"""Native packing of the binding's host arrays."""
import struct

import pytest
import torch


class Fake:
    def data_ptr(self):
        return (1 << 63) + 5


@pytest.mark.parametrize("n", [0, 1, 3, 200])
def test_pointers(n):
    from paper_2608_15943_b200 import kvp
    ts = [(torch.zeros(4)[i % 3:], None, torch.nn.Parameter(torch.zeros(2)), Fake())[i % 4] for i in range(n)]
    want = struct.pack(f"{n}Q", *[0 if t is None else t.data_ptr() for t in ts])
    assert kvp._ptr_array(ts) == want and kvp._ptr_array(tuple(ts)) == want


@pytest.mark.parametrize("xs", [[], [0], [0, 1, 1, -3], (2**31 - 1, -2**31), [True, 2.0, torch.tensor(7)]])
def test_donors(xs):
    from paper_2608_15943_b200 import kvp
    assert kvp._donors(xs) == struct.pack(f"{len(xs)}i", *map(int, xs))


def test_refused():
    from paper_2608_15943_b200 import kvp
    for bad, err in (([2**31], OverflowError), (["x"], ValueError), (3, TypeError)):
        with pytest.raises(err):
            kvp._donors(bad)
    for bad, err in (([1.5], AttributeError), (None, TypeError)):
        with pytest.raises(err):
            kvp._ptr_array(bad)
