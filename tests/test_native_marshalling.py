"""The native marshalling of the binding (csrc/lla_binding.cpp) takes only ordinary calls: to anything
else it answers None, and the Python marshalling accepts or refuses the call as without it (no GPU; what it
takes is tested with real CUDA tensors in test_native_marshalling_gpu.py)."""
import inspect

import pytest
import torch

from helpers import ensure_library

FAKE = 0x10000


@pytest.fixture(scope="module")
def lla():
    ensure_library()
    from paper_2607_15456_gb300 import lla as m
    return m


def _args(lla, name, x):
    """The native function's arguments for a call of lla.<name> with x in every tensor's place."""
    geom, cache = lla.Geometry(4, 2, 128, 96, 160), lla.Cache(x, 4, x, 2)
    cd = lla.Codec(x, x, x, x)
    scalar = {"geom": geom, "codec": cd, "cache": cache, "codecs": [cd], "caches": [cache], "max_ctx": 64, "max_len": 64,
              "loop": 0, "rope_base": 10000.0, "rope_pairing": 0, "d_rope": 64, "stream": 0}
    names = list(inspect.signature(getattr(lla, "lla_" + name)).parameters)
    return [scalar[n] if n in scalar else ([x] if name == "encode_layers" and n in ("x_k", "x_v") else x) for n in names]


NAMES = ["encode", "encode_2d", "encode_layers", "decode_attn", "decode_attn_2d", "decode_attn_loops", "decode_attn_rope",
         "decode_attn_decoupled", "prefill_attn", "prefill_attn_rope"]


@pytest.mark.parametrize("name", NAMES)
@pytest.mark.parametrize("what", ["host tensor", "address", "other object", "host parameter"])
def test_unusual_arguments_are_left_to_python(lla, name, what):
    x = {"host tensor": torch.zeros(4, 4, 2, 128), "address": FAKE, "other object": "x",
         "host parameter": torch.nn.Parameter(torch.zeros(4, 4, 2, 128))}[what]
    assert getattr(lla._native(), name)(*_args(lla, name, x)) is None
    if what in ("host tensor", "host parameter"):
        with pytest.raises(ValueError, match="CUDA tensors"):
            getattr(lla, "lla_" + name)(*_args(lla, name, x))


@pytest.mark.parametrize("name", NAMES)
def test_wrong_number_of_arguments(lla, name):
    with pytest.raises(TypeError):
        getattr(lla._native(), name)(None)


def test_a_missing_module_leaves_every_call_to_python(lla, monkeypatch):
    def missing(name, package=None):
        raise ImportError("no such module")

    monkeypatch.setattr(lla, "_native_module", None)
    monkeypatch.setattr(lla.importlib, "import_module", missing)
    with pytest.warns(UserWarning, match="marshalled in Python"):
        assert lla._native().encode(1, 2, 3) is None
    for name in NAMES:
        args = _args(lla, name, torch.zeros(4, 4, 2, 128))
        assert getattr(lla._native(), name)(*args) is None
        with pytest.raises(ValueError, match="CUDA tensors"):
            getattr(lla, "lla_" + name)(*args)


def test_a_binding_that_does_not_compile_does_not_fail_the_build(lla, monkeypatch, tmp_path, capsys):
    from paper_2607_15456_gb300 import build
    stale = tmp_path / "_lla_native.so"
    stale.write_bytes(b"")
    monkeypatch.setattr(build, "NATIVE", str(stale))
    monkeypatch.setattr(build, "library_up_to_date", lambda: True)
    monkeypatch.setattr(build, "binding_up_to_date", lambda: False)

    def fails():
        raise RuntimeError("g++ on lla_binding.cpp failed")

    monkeypatch.setattr(build, "compile_binding", fails)
    assert build.build() == build.LIB
    assert not stale.exists() and "marshalled in Python" in capsys.readouterr().err


def test_a_binding_of_another_torch_is_neither_loaded_nor_up_to_date(lla, monkeypatch):
    from paper_2607_15456_gb300 import build
    assert build.binding_up_to_date()
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    assert not build.binding_up_to_date()
    monkeypatch.setattr(lla, "_native_module", None)
    with pytest.warns(UserWarning, match="built for"):
        assert lla._native().encode(1, 2, 3) is None
