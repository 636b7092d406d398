"""A cached tuning choice is re-applied only to the shape that it was timed on."""
import json

import pytest

from paper_2106_06161_gb300 import _lib, autotune, build


@pytest.fixture
def cache(tmp_path, monkeypatch):
    build.build()
    monkeypatch.setattr(autotune, "device_key", lambda device=None: "gpu")
    autotune.reset()
    path = tmp_path / "tuning.json"
    yield lambda entry: (path.write_text(json.dumps({"gpu": entry})), autotune.apply_cached(str(path)))[1]
    autotune.reset()


@pytest.mark.parametrize("kernel", sorted(autotune.KERNELS))
def test_stale_choices_are_passed_over(cache, kernel):
    kid = autotune.KERNELS[kernel]
    shapes = [{k: v for k, v in c.items() if k != "config"} for c in _lib.bshuffle_kernel_configs(kid)]
    selected = lambda: _lib.bshuffle_kernel_selected(kid, 8)  # noqa: E731
    assert cache({kernel: {"8": {"config": 1, "shape": shapes[1]}}}) and selected() == 1
    autotune.reset()
    for rec in ({"config": 1},                                                  # a file without shapes
                {"config": 1, "shape": dict(shapes[1], items=shapes[1]["items"] + 1)},
                {"config": len(shapes), "shape": shapes[1]}):
        assert not cache({kernel: {"8": rec}}) and selected() == 0, rec
    # the others of the file are applied
    assert cache({kernel: {"4": {"config": 1}, "8": {"config": 1, "shape": shapes[1]}}}) and selected() == 1
    assert _lib.bshuffle_kernel_selected(kid, 4) == 0
