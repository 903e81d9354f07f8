"""The autotuner creates no more lattices than there are shapes to time."""
import pytest

from paper_2208_09267_gb300 import lbm, tune

pytestmark = pytest.mark.gpu


def test_fp16_has_one_row_shape_to_time(tmp_path, monkeypatch):
    made = []

    class Counted(lbm.Lattice):
        def __init__(self, *args, **kw):
            made.append(kw.get("kernel"))
            super().__init__(*args, **kw)

    monkeypatch.setattr(lbm, "Lattice", Counted)
    cache = tune.Cache(str(tmp_path / "tune.json"), seed=None)
    best, ms = tune.tune_step("D3Q19", "fp16", (64, 16, 16), steps=4, warmup=2, cache=cache, blocks=[(64, 2)],
                              row_shapes=[(0, 0), (5, 2), (6, 3)])
    assert made == [2, 1] and sum(name.startswith("row") for name in ms) == 1
    assert best in ({"kernel": 2, "block": [0, 0], "row_shape": [16, 8]},
                    {"kernel": 1, "block": [64, 2], "row_shape": None})
