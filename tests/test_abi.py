"""The C-ABI library builds, loads without a GPU and exports every symbol the header declares."""
import ctypes
import os
import re
import subprocess
import sys

import pytest
import torch

from paper_2510_18239_b200 import binding, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_symbols():
    with open(os.path.join(ROOT, "include", "lime.h")) as f:
        text = f.read()
    return re.findall(r"LIME_API\s+[\w\s\*]+?\b(lime_\w+)\s*\(", text)


def test_library_exports_every_declared_symbol():
    lib_path = build.build()
    assert os.path.exists(lib_path)
    names = declared_symbols()
    assert len(names) >= 12 and "lime_score_candidates" in names and "lime_encode_user" in names
    lib = ctypes.CDLL(lib_path)
    for n in names:
        assert hasattr(lib, n), n
    assert set(names) == set(binding.EXPORTS)


def test_version_string_and_host_side_validation():
    lib = binding.load_library()
    assert b"sm_100a" in lib.lime_version()
    # NULL config / out pointer are rejected before any CUDA call
    assert lib.lime_create(None, None) == 1
    h = ctypes.c_void_p()
    bad = binding.lime_config(d=30, H=2, ell=8, n_layers=1, d_ff=0, dtype=0, phi=0, ln=1, gated_mlp=1)
    assert lib.lime_create(ctypes.byref(bad), ctypes.byref(h)) == 2          # d % 8 != 0
    bad = binding.lime_config(d=32, H=3, ell=8, n_layers=1, d_ff=0, dtype=0, phi=0, ln=1, gated_mlp=1)
    assert lib.lime_create(ctypes.byref(bad), ctypes.byref(h)) == 2          # d % H != 0
    bad = binding.lime_config(d=32, H=2, ell=0, n_layers=1, d_ff=0, dtype=0, phi=0, ln=1, gated_mlp=1)
    assert lib.lime_create(ctypes.byref(bad), ctypes.byref(h)) == 1
    bad = binding.lime_config(d=32, H=2, ell=8, n_layers=17, d_ff=0, dtype=0, phi=0, ln=1, gated_mlp=1)
    assert lib.lime_create(ctypes.byref(bad), ctypes.byref(h)) == 2
    bad = binding.lime_config(d=32, H=2, ell=8, n_layers=1, d_ff=0, dtype=7, phi=0, ln=1, gated_mlp=1)
    assert lib.lime_create(ctypes.byref(bad), ctypes.byref(h)) == 1
    assert lib.lime_destroy(None) == 0
    assert lib.lime_workspace_bytes(None, 1, 1) == 0


def test_struct_layouts_match_header():
    assert ctypes.sizeof(binding.lime_config) == 13 * 4          # 12 fields of the paper's model + cand_heads
    assert ctypes.sizeof(binding.lime_weights) == 8 * (1 + 6 * binding.LIME_MAX_LAYERS + 3)
    assert ctypes.sizeof(binding.lime_ffn) == 4 * 4 + 8 * 8      # n_hidden + 3 widths, 4 weight and 4 bias pointers


def test_ffn_entry_points_validate_on_the_host():
    lib = binding.load_library()
    assert lib.lime_set_head(None, None, None) == 1
    assert lib.lime_set_context_mlp(None, 4, None, None) == 1
    assert lib.lime_contextualize_links(None, None, 1, None, None) == 1
    assert lib.lime_head_workspace_bytes(None, 4) == 0
    assert lib.lime_score_candidates_head(None, None, 1, None, None, None, 1, 1, None, 0, None, None, None, 0, None) == 1


def test_native_binding_refuses_what_is_no_cuda_tensor():
    """The native half of the binding loads without a GPU and checks what it is given before anything is launched."""
    import pytest
    import torch
    native = binding._native()
    with pytest.raises(TypeError):
        native.lengths_to_offsets(None, [1, 2])
    with pytest.raises(TypeError):
        native.encode_user(None, 8, 32)
    cpu = torch.zeros((3, 32))
    for call in (lambda: native.lengths_to_offsets(None, cpu), lambda: native.gather_history(None, 32, cpu, cpu, None),
                 lambda: native.precompute_candidate_links(None, 8, cpu),
                 lambda: native.score_candidates(None, cpu, cpu, cpu, 1, None, None, None, None, None)):
        with pytest.raises(ValueError):
            call()
    with pytest.raises(OverflowError):
        native.score_candidates(None, cpu, cpu, cpu, 1, None, None, 1 << 70, None, None)


def test_python_marshalling_refuses_what_is_no_cuda_tensor():
    """The same without the native half."""
    plain = binding._PlainCalls
    with pytest.raises(TypeError):
        plain.lengths_to_offsets(None, [1, 2])
    with pytest.raises(TypeError):
        plain.encode_user(None, 8, 32)
    cpu = torch.zeros((3, 32))
    for call in (lambda: plain.lengths_to_offsets(None, cpu), lambda: plain.gather_history(None, 32, cpu, cpu, None),
                 lambda: plain.precompute_candidate_links(None, 8, cpu),
                 lambda: plain.score_candidates(None, cpu, cpu, cpu, 1, None, None, None, None, None)):
        with pytest.raises(ValueError):
            call()


def test_the_library_builds_without_what_the_binding_needs(monkeypatch, tmp_path, capsys):
    """No g++ (or no torch, no Python.h): the C-ABI library all the same, and a word about what is left out."""
    monkeypatch.setattr(build, "BINDING", str(tmp_path / "_torch_binding.so"))
    monkeypatch.setattr(build, "MADE_FOR", str(tmp_path / "made_for"))
    which = build.shutil.which
    monkeypatch.setattr(build.shutil, "which", lambda name: None if name == "g++" else which(name))
    assert build.build() == build.LIB and not (tmp_path / "_torch_binding.so").exists()
    assert "g++ not found" in capsys.readouterr().err


def test_the_binding_is_rebuilt_for_another_torch(monkeypatch, tmp_path):
    made = []

    def compiler(cmd, **kw):
        made.append(cmd)
        open(build.BINDING, "w").close()
        return subprocess.CompletedProcess(cmd, 0, "", "")
    monkeypatch.setattr(build, "BINDING", str(tmp_path / "_torch_binding.so"))
    monkeypatch.setattr(build, "MADE_FOR", str(tmp_path / "made_for"))
    monkeypatch.setattr(build.subprocess, "run", compiler)
    assert build.build_binding() == build.BINDING == build.build_binding() and len(made) == 1
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    assert build.build_binding() == build.BINDING == build.build_binding() and len(made) == 2
    assert any("torch 0.0.0" in a for a in made[1])


@pytest.mark.parametrize("made_for", [None, "another torch"])
def test_calls_go_through_python_without_a_fitting_extension(monkeypatch, made_for):
    """The extension missing, or built against another torch or Python: a warning, and the calls through ctypes."""
    monkeypatch.setattr(binding, "_native_module", None)
    binding._native()
    native = sys.modules["paper_2510_18239_b200._torch_binding"]
    monkeypatch.setattr(binding, "_native_module", None)
    if made_for is None:
        monkeypatch.setitem(sys.modules, "paper_2510_18239_b200._torch_binding", None)
        monkeypatch.delattr(sys.modules["paper_2510_18239_b200"], "_torch_binding", raising=False)
    else:
        monkeypatch.setattr(native, "made_for", made_for)
    with pytest.warns(UserWarning, match="marshalled in Python"):
        assert binding._native() is binding._PlainCalls
