"""The batched-query tuner's cache: what other kernels were tuned to is not
applied, what these were is found again."""
import json

import numpy as np
import pytest

pytest.importorskip("torch")


def test_entries_of_other_kernels_are_not_found(tmp_path, monkeypatch):
    import torch

    from paper_1506_03872_gb300 import autotune
    path = tmp_path / "tuned.json"
    monkeypatch.setenv("MAD_TUNE_CACHE", str(path))
    s_q = np.array([1000, 50_000])
    dev = torch.cuda.get_device_name() if torch.cuda.is_available() else "cpu"
    # The key of the entries that were stored for the per-query hash regions.
    old = f"{dev}|d=300|n=1000000|nq=2|s=[1000,50000]|sum={float('5.1e+04')}|tp=100|t=5"
    path.write_text(json.dumps({old: {"best": {"region_lg": 2, "chunk_mult": 1}}}))
    key = autotune.shape_key(300, 1_000_000, s_q, 100, 5)
    assert autotune.load(key) is None
    autotune.store(key, {"best": dict(autotune.DEFAULT)})
    assert autotune.load(key)["best"] == autotune.DEFAULT
    assert autotune.load(old) is not None   # (left to whoever stored it)
