"""The bounds-checked build on maps of long tile lists (tests/_checked_lists.py: cut, gathered and
full lists, each build in its own process): no index out of bounds, images the normal build's bit
for bit, none of them empty."""
import subprocess
import sys

import numpy as np
import pytest

from tests._util import ROOT, ensure_built

pytestmark = pytest.mark.gpu


def test_checked_build_on_long_lists(tmp_path):
    ensure_built()
    runs = []
    for which in ("normal", "checked"):
        path = tmp_path / f"{which}.npz"
        r = subprocess.run([sys.executable, "-m", "tests._checked_lists", which, str(path)], cwd=ROOT, capture_output=True,
                           text=True, timeout=600)
        assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
        runs.append(dict(np.load(path)))
    normal, checked = runs
    assert not bool(normal["checked"]) and bool(checked["checked"])
    for name, route in (("cut", (1, 0)), ("gathered", (3, 0)), ("in_full", (1, 1)), ("odd", (1, 0))):
        assert tuple(normal[f"{name}_route"]) == tuple(checked[f"{name}_route"]) == route, name
        assert normal[f"{name}_alpha"].max() > 0.1
        for k in ("color", "depth", "alpha"):
            np.testing.assert_array_equal(checked[f"{name}_{k}"], normal[f"{name}_{k}"], err_msg=f"{name}_{k}")
