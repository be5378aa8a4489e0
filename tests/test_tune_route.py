"""The POD tuner gives no leaf height to calls whose automatic choice is the
Gram route (CPU)."""
import pytest

import paper_2405_15529_gb300 as pg
from paper_2405_15529_gb300 import tune


@pytest.mark.parametrize("energy,r_max,height", [(0.99, None, 0), (0.0, 40, 0), (0.0, None, 13797), (0.0, 256, 13797),
                                                 (1.0, None, 13797), (1.0 - 1e-4, None, 0)])
def test_heights_only_for_calls_that_use_leaves(energy, r_max, height, tmp_path, monkeypatch):
    monkeypatch.setattr(tune, "CACHE", str(tmp_path / "c.json"))
    monkeypatch.setattr(tune, "gpu_name", lambda: "cpu")
    monkeypatch.delenv("PYLOM_TREE", raising=False)
    tune._save({"cpu|pod|prec0|N4194304|M256": 13797})
    assert tune.pod_leaf_rows_for(1 << 22, 256, pg.PREC_FP64, tune=True, energy=energy, r_max=r_max) == height
    monkeypatch.setenv("PYLOM_TREE", "pipe")
    assert tune.pod_leaf_rows_for(1 << 22, 256, pg.PREC_FP64, energy=energy, r_max=r_max) == 13797
