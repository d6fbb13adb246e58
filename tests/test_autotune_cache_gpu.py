"""The autotuner's cache holds the kernels' version in its keys: a shape timed
on earlier kernels is measured again, one of the current kernels is taken."""
import json

import pytest

from paper_2310_13143_gb300 import binding, gridgen as gg

pytestmark = pytest.mark.gpu


def test_entries_of_earlier_kernels_are_not_used(tmp_path):
    path = str(tmp_path / "shapes.json")

    def tune():
        s = binding.Solver(gg.two_bus(), precision="fp64")
        out = s.autotune(path, iters=4)
        s.close()
        return out

    shape, us = tune()
    assert us > 0
    assert tune() == (shape, -1.0)
    (entry,) = json.load(open(path))
    version, rest = entry["key"].split("-", 1)
    for old in range(1, 5):
        with open(path, "w") as f:
            f.write("[\n  " + json.dumps(dict(entry, key=f"v{old}-{rest}")) + "\n]\n")
        assert tune()[1] > 0
        # both are in the file then; the earlier kernels' entry is not touched
        assert sorted(e["key"] for e in json.load(open(path))) == [f"v{old}-{rest}", f"{version}-{rest}"]
