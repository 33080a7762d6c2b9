"""A persisted autotune file written by a build whose shape numbers meant other kernels (lines
without the shape table's version, or with another one) is not used: its keys are timed again."""
import json

import pytest

from test_gpu_autotune_cache import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("version", [None, 1])
def test_lines_of_other_shape_tables_are_ignored(tmp_path, version):
    path = str(tmp_path / "tune.jsonl")
    _run(path)
    line = json.loads(open(path).read())
    table = line.pop("shapes", None)
    old = {"device": line.pop("device")}
    if version is not None:
        assert table != version
        old["shapes"] = version
    old.update(line)
    open(path, "w").write(json.dumps(old, separators=(",", ":")) + "\n")
    second = _run(path)
    assert second["launches"] > 1
    assert len(open(path).readlines()) == 2      # the new choice was appended
    assert _run(path)["launches"] == 1           # and is read
