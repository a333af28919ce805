"""Sorted runs (tests/checked_sorted_cases.py): the checked build runs them without an index out
of range and gives the default build's bits; they really sort, and give the unsorted bits, also
where a sorted set was saved and loaded on the way."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def default():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0912_3223_gb300 import build
    build.build()
    build.build(checked=True)
    import checked_sorted_cases
    return checked_sorted_cases.run_cases()


def test_checked_build_is_clean_and_identical(default, tmp_path):
    out = str(tmp_path / "checked.npz")
    code = ("import sys; sys.path[:0] = [%r, %r]; import numpy as np; "
            "import checked_sorted_cases as c; np.savez(%r, **c.run_cases())" % (HERE, ROOT, out))
    env = dict(os.environ, LPM_CHECKED_BUILD="1")
    run = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True,
                         timeout=900)
    assert run.returncode == 0, run.stderr[-3000:]
    got = np.load(out)
    assert sorted(got.files) == sorted(default)
    for k, v in default.items():
        assert np.array_equal(got[k], v), k


def test_sorted_equals_unsorted(default):
    import checked_sorted_cases as c
    for name, (cfg, kw, dosage) in c.cases().items():
        ref = c.run_case(cfg, {"sort_every": 0}, dosage)
        sorts = (c.STEPS // 2 + 2) // kw["sort_every"]
        # two or three launches a sort, and one more for every segment that a sort cuts off
        assert default[f"{name}_launches"] >= ref["launches"] + 2 * sorts, name
        for k, v in ref.items():
            if k != "launches":
                assert np.array_equal(default[f"{name}_{k}"], v), (name, k)
