"""Small trees, whose default sort is one launch, use the tuner's cached sort
like every other build, and the tuner times that launch against its variants."""
from __future__ import annotations

import json

import numpy as np
import pytest

from paper_2402_00665_gb300 import _build, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    _build.build()
    from paper_2402_00665_gb300 import lbvh
    return lbvh.load()


def launches(tree, p, bits):
    from paper_2402_00665_gb300 import lbvh
    before = lbvh.kernel_launches()
    tree.build(p, lbvh.POINTS, bits).check()
    return lbvh.kernel_launches() - before


@pytest.mark.parametrize("n,bits", [(900, 30), (8192, 30), (900, 63), (16384, 63)])
def test_a_cached_choice_decides(tmp_path, n, bits):
    from paper_2402_00665_gb300 import lbvh
    p = torch.from_numpy(inputs.uniform_points(n, seed=n)).cuda()
    one, fixed = lbvh.Tree(), lbvh.Tree()
    fixed.set_tuning(3, -1)
    lbvh.tune_clear()
    fewer, more = launches(one, p, bits), launches(fixed, p, bits)
    assert fewer < more
    path = tmp_path / "tune.json"
    path.write_text(json.dumps({"lbvh_tune_cache": 1, "entries": [
        {"gpu": torch.cuda.get_device_name(), "n_log2": int(n - 1).bit_length(), "bits": bits, "kind": 0, "qkind": -1,
         "instances": 1, "sort_variant": 3, "sort_ms": 0.1, "walk_variant": -1, "walk_ms": 0}]}))
    try:
        lbvh.tune_load(str(path))
        assert launches(one, p, bits) == more
        a, b = one.export(), fixed.export()
        for key in ("perm", "sorted", "left", "skip_internal", "skip_leaf"):
            assert np.array_equal(a[key], b[key]), key
    finally:
        lbvh.tune_clear()
    assert launches(one, p, bits) == fewer
    one.close()
    fixed.close()


@pytest.mark.parametrize("n,bits", [(1000, 30), (1000, 63)])
def test_the_tuner_times_the_one_launch(tmp_path, n, bits):
    from paper_2402_00665_gb300 import lbvh
    p = torch.from_numpy(inputs.uniform_points(n, seed=5)).cuda()
    lbvh.tune_clear()
    try:
        t = lbvh.Tree()
        default = launches(t, p, bits)
        sv, _ = t.autotune(p, lbvh.POINTS, bits)
        assert sv == -1  # 41 and 45 us against 87 and 180
        assert lbvh.tune_entries() == 1
        assert launches(t, p, bits) == default
        lbvh.tune_save(str(tmp_path / "tune.json"))
        lbvh.tune_load(str(tmp_path / "tune.json"))
        assert launches(t, p, bits) == default
        t.close()
    finally:
        lbvh.tune_clear()
