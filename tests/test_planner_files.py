"""Saved cost models of the twelve-feature network are still read, and predict what they predicted."""
import json

import numpy as np
import pytest

from oracle import mlp
from paper_2310_03983_gb300 import planner


def _save(path, in_dim, params):
    path.write_text(json.dumps({"in_dim": in_dim, "hidden": planner.HIDDEN, "y_shift": 0.5, "params": params}))
    return str(path)


def test_a_file_without_the_last_feature_is_read(tmp_path):
    old = mlp.init(planner.IN_DIM - 1, seed=4).astype(np.float32)
    m = planner.CostModel.load(_save(tmp_path / "old.json", planner.IN_DIM - 1, old.tolist()), device="cpu")
    assert m.y_shift == 0.5
    x = np.array([planner.features(n, p, dt, a, c) for n, p, dt in ((100, 0.2, "int32"), (1024, 0.4, "float32"))
                  for a, c in planner.applicable(n)])
    got = mlp.forward(m.params.numpy().astype(np.float64), x)[0]
    want = mlp.forward(old.astype(np.float64), x[:, :-1])[0]
    assert np.allclose(got, want, rtol=0, atol=1e-12)


def test_other_networks_stay_refused(tmp_path):
    for in_dim in (planner.IN_DIM - 2, planner.IN_DIM + 1):
        with pytest.raises(ValueError):
            planner.CostModel.load(_save(tmp_path / "x.json", in_dim, mlp.init(in_dim, seed=1).tolist()), device="cpu")
