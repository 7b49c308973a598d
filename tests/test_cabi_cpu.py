"""The C-ABI library builds for sm_100a, loads without a GPU and exports every declared symbol."""
import ctypes
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def libpath():
    from paper_2608_15383_b200 import build
    return build.build()


def declared_symbols():
    text = open(os.path.join(ROOT, "include", "exmoe.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(exmoe_[a-z_0-9]+)\s*\(", text)))


def test_header_declares_the_boundary():
    names = declared_symbols()
    for must in ("exmoe_pack", "exmoe_packed_bytes", "exmoe_cache_create", "exmoe_moe_forward",
                 "exmoe_cache_workspace_bytes", "exmoe_cache_destroy", "exmoe_status", "exmoe_strerror"):
        assert must in names


def test_library_exports_every_declared_symbol(libpath):
    lib = ctypes.CDLL(libpath)
    for name in declared_symbols():
        assert hasattr(lib, name), name


def test_binding_covers_every_declared_symbol(libpath):
    from paper_2608_15383_b200 import binding
    assert sorted(binding._SIGNATURES) == declared_symbols()
    binding.lib()


def test_host_only_calls(libpath):
    """Entry points that touch no device: size model (Eq. 4), argument checks, error strings."""
    from paper_2608_15383_b200 import binding, synth
    assert binding.exmoe_packed_bytes(synth.OLMOE) == 3244032
    assert binding.exmoe_packed_bytes(synth.TINY) == 50688
    slot_total, ws = binding.exmoe_cache_workspace_bytes(synth.OLMOE, 16, 16, 64)
    assert slot_total == 16 * 16 * 3244032
    assert ws >= 64 * 8 * (1024 * 2 + 2048 * 4)
    for bad in (synth.Shape(200, 128, 4, 2), synth.Shape(256, 128, 4, 8), synth.Shape(256, 128, 4, 2, group_size=64)):
        with pytest.raises(binding.ExmoeError) as ei:
            binding.exmoe_packed_bytes(bad)
        assert ei.value.code == binding.EXMOE_ERR_SHAPE
    with pytest.raises(binding.ExmoeError):
        binding.exmoe_cache_workspace_bytes(synth.OLMOE, 1, 4, 16)      # C < k
    assert "pinned" in binding.strerror(binding.EXMOE_ERR_NOT_PINNED)
    assert binding.exmoe_launch_count() == 0


def test_missing_library_fails_loudly(monkeypatch, tmp_path):
    from paper_2608_15383_b200 import binding
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "LIB_PATH", str(tmp_path / "nope.so"))
    with pytest.raises(FileNotFoundError):
        binding.lib()


def test_serving_calls_take_what_int_takes(libpath):
    """Layer numbers and shape dimensions go through int(): floats, strings of digits, numpy scalars.  With host tensors where
    device tensors belong, a call that got past its numbers ends at the tensors."""
    import types

    import numpy as np
    import torch

    from paper_2608_15383_b200 import binding
    binding.lib()
    h = torch.zeros((1, 256), dtype=torch.bfloat16)
    for layer in (0, 1.0, np.int64(1), np.float32(2.0), "1", torch.tensor(1), True):
        with pytest.raises(ValueError, match="hidden"):
            binding.Cache.forward(types.SimpleNamespace(_address=0), layer, h, None, None)
    for bad in (None, "x", [1]):
        with pytest.raises((TypeError, ValueError), match="int"):
            binding.Cache.forward(types.SimpleNamespace(_address=0), bad, h, None, None)
    for d in (256, 256.0, np.float64(256), "256"):
        with pytest.raises(ValueError, match="hidden"):
            binding.exmoe_route(types.SimpleNamespace(d_model=d, d_ff=128, num_experts=8, top_k=2), h, h)


def test_only_the_serving_calls_need_the_native_module(libpath, monkeypatch, tmp_path):
    import torch

    from paper_2608_15383_b200 import binding, synth
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "_native", None)
    monkeypatch.setattr(binding, "NATIVE_PATH", str(tmp_path / "nope.so"))
    assert binding.exmoe_packed_bytes(synth.TINY) == 50688
    with pytest.raises(FileNotFoundError):
        binding.exmoe_route(synth.TINY, torch.zeros((1, 256)), torch.zeros((8, 256)))


def test_a_native_module_of_another_torch_is_rebuilt_and_not_loaded(libpath, monkeypatch, tmp_path):
    import torch

    from paper_2608_15383_b200 import binding, build, synth
    assert build.native_is_current()
    other = tmp_path / "other.so"
    with open(build.NATIVE, "rb") as f:
        other.write_bytes(f.read().replace(torch.__version__.encode(), b"9" * len(torch.__version__)))
    assert not build.native_is_current(str(other))
    monkeypatch.setattr(binding, "_native", None)
    monkeypatch.setattr(binding, "NATIVE_PATH", str(other))
    with pytest.raises(ImportError, match="another torch"):
        binding.exmoe_route(synth.TINY, torch.zeros((1, 256)), torch.zeros((8, 256)))
