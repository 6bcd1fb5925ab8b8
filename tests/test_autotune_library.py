"""The autotuner's stored choices belong to the library that timed them (host
logic, no GPU; the library calls are test_autotune_cache's fake)."""
import json
import os

from paper_2102_01366_gb300 import _build, gks
from test_autotune_cache import _state, calls  # noqa: F401


def test_another_library_is_tuned_anew(calls, tmp_path, monkeypatch):
    """A choice stored by a library with other sources is not taken: its
    variant was the fastest of other kernels."""
    cache = str(tmp_path / "autotune.json")
    _state().autotune(cache=cache)
    assert _state().autotune(cache=cache)["cached"] is True
    copy = tmp_path / "csrc"
    copy.mkdir()
    for p in sum(_build._sources(), []):
        (copy / os.path.basename(p)).write_bytes(open(p, "rb").read())
    (copy / "gks_flux.cu").write_text(open(copy / "gks_flux.cu").read() + "// another kernel\n")
    monkeypatch.setattr(_build, "CSRC", str(copy))
    assert _state().autotune(cache=cache)["cached"] is False
    # without the sources, the library file stands for them
    monkeypatch.setattr(_build, "CSRC", str(tmp_path / "none"))
    monkeypatch.setattr(gks, "LIB_PATH", str(copy / "gks_api.cpp"))
    assert _state().autotune(cache=cache)["cached"] is False
    assert _state().autotune(cache=cache)["cached"] is True
    # an entry keyed without the library, as older versions wrote them
    (old,) = {k.split("|lib=")[0] for k in json.load(open(cache))}
    open(cache, "w").write(json.dumps({old: {"variant": [0, 3, 0], "fused": 0}}))
    assert _state().autotune(cache=cache)["cached"] is False
