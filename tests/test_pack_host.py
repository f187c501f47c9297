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


def test_packing_is_built_anew_for_another_torch(monkeypatch, tmp_path):
    """_pack.so is laid out for one Python and one torch: a build for another is not kept, whatever its time."""
    import os
    from paper_2608_15943_b200 import build
    os.makedirs(tmp_path / "obj")
    monkeypatch.setattr(build, "OBJ", str(tmp_path / "obj"))
    monkeypatch.setattr(build, "PACK", str(tmp_path / "_pack.so"))
    runs = []

    class Done:
        returncode, stdout, stderr = 0, "", ""

    def run(cmd, **kw):
        runs.append(cmd)
        open(build.PACK, "w").close()
        return Done()
    monkeypatch.setattr(build.subprocess, "run", run)
    build._build_pack(False)
    build._build_pack(False)
    assert len(runs) == 1
    key = build._pack_key
    monkeypatch.setattr(build, "_pack_key", lambda d: key(d) + "another")
    build._build_pack(False)
    build._build_pack(False)
    assert len(runs) == 2
