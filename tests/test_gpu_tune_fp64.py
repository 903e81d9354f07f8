"""Tuning an FP64 lattice does not lose the kernel that small ones step in."""
import pytest

from paper_2208_09267_gb300 import lbm, tune

pytestmark = pytest.mark.gpu


def test_small_fp64_lattices_keep_the_default(tmp_path, monkeypatch):
    """64 x 64 cells: the split step takes two thirds of the time of the best
    block shape, so the tuned choice is the default and the handle launches it."""
    monkeypatch.setenv("LBM_TUNE_CACHE", str(tmp_path / "tune.json"))
    monkeypatch.setattr(tune, "SEED_CACHE", None)
    best, ms = tune.tune_step("D2Q9", "fp64", (64, 64, 1), steps=60, warmup=20, cache=tune.Cache(seed=None))
    assert "default" in ms and "cell32x1" in ms
    assert best == {"kernel": 1, "block": [0, 0], "row_shape": None}
    tuned = lbm.Lattice("D2Q9", (64, 64, 1), tau=0.6, storage="fp64")
    plain = lbm.Lattice("D2Q9", (64, 64, 1), tau=0.6, storage="fp64", tuned=False)
    assert tuned.tuned_from and tuned.launch_shape == plain.launch_shape
    tuned.close()
    plain.close()
