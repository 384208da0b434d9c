"""The batched build does not take launch shapes that were timed for earlier forms of its kernels: their
entries of the tuning file have other names, stay as they are, and the present names are added."""
import json

import numpy as np
import pytest

from gpu_common import to_dev

pytestmark = pytest.mark.gpu


def test_entries_of_earlier_kernels_are_not_taken(tmp_path, monkeypatch):
    from paper_2202_03655_gb300 import hdf
    path = tmp_path / "tune.json"
    monkeypatch.setenv("HDF_AUTOTUNE_CACHE", str(path))
    g = np.random.default_rng(0)
    x, off = to_dev(g.uniform(-1, 1, (900, 3))), [0, 300, 900]

    def build():
        hdf.build_batched(x, off, "gaussian", [0.5, 0.7], 1e-5).free()
        return json.loads(path.read_text())

    now = build()
    radial = [k for k in now if k.startswith("batch_radial_")]
    assert len(radial) == 1 and build() == now                  # found again
    for old in ("v1", "v2", "v3"):
        name = "batch_radial_" + old + radial[0][radial[0].index(":"):]
        path.write_text(json.dumps({name: 101}))
        after = build()
        assert after[name] == 101 and radial[0] in after and radial[0] != name
