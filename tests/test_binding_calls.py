"""The per-step calls as native functions and through ctypes: the same arguments, the same refusals (no GPU needed)."""
import importlib.machinery
import os

import pytest

from paper_2605_29986_b200 import _build
from paper_2605_29986_b200 import binding as cz

NAMES = sorted(cz._STEP_CALLS)


def test_the_native_module_is_of_this_interpreter():
    assert cz._calls is not None and cz._calls.__file__ == _build.CALLS_PATH
    assert any(os.path.basename(_build.CALLS_PATH) == "_calls" + s for s in importlib.machinery.EXTENSION_SUFFIXES[:1])


@pytest.mark.parametrize("name", NAMES)
def test_both_ways_take_and_refuse_the_same(name):
    kinds, required, names = cz._STEP_CALLS[name][0], cz._STEP_CALLS[name][1], cz._STEP_CALLS[name][2].split()
    assert len(kinds) == len(names) == len(cz._SIGNATURES[name][1])
    null = {"p": None, "s": None, "i": 0, "f": 0.5}
    values = [null[k] for k in kinds]
    for call in (getattr(cz, name), cz._through_ctypes(name)):
        for args, given in ((values, {}), (values[:required], {}), (values[:2], dict(zip(names[2:], values[2:]))),
                            ([], dict(zip(names[:required], values)))):
            with pytest.raises(cz.CfgzipError) as e:  # (no context)
                call(*args, **given)
            assert e.value.status in (cz.E_ARG, cz.E_RANGE)
        for args, given in ((values + [0], {}), (values[:required - 1], {}), (values, {names[0]: None}), (values[:required], {"nothing": 1}),
                            ([object()] + values[1:], {})):
            with pytest.raises(TypeError):
                call(*args, **given)


def test_import_without_a_compiler(tmp_path, monkeypatch):
    monkeypatch.setattr(_build, "CALLS_PATH", str(tmp_path / "_calls.so"))
    monkeypatch.setattr(_build.shutil, "which", lambda name: str(tmp_path / name))
    assert _build.build_calls() is False and not os.path.exists(_build.CALLS_PATH)
    (tmp_path / "_calls.so").write_text("of an older source")
    os.utime(tmp_path / "_calls.so", (1, 1))
    assert _build.build_calls() is False and not os.path.exists(_build.CALLS_PATH)
