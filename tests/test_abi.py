"""CPU-side checks: the shared library builds, loads and exports every symbol the header declares;
host-side validation answers without a GPU; the N>1 'replicas only' layout of bench.py."""
import ctypes as C
import os
import re
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_2502_18394_b200 import build, binding
    build.build()
    return binding.lib()


def test_every_declared_symbol_is_exported(lib):
    from paper_2502_18394_b200 import binding
    header = open(os.path.join(ROOT, "include", "spectre.h")).read()
    header = re.sub(r"/\*.*?\*/", "", header, flags=re.S)
    declared = set(re.findall(r"\b(spectre_[a-z_0-9]+)\s*\(", header))
    assert declared, "no declarations found"
    for name in declared:
        assert hasattr(lib, name), name
    assert declared == set(binding.EXPORTS)


def test_status_strings(lib):
    assert lib.spectre_status_string(0) == b"ok"
    for s in range(1, 6):
        assert lib.spectre_status_string(s) not in (b"ok", b"unknown status")
    assert lib.spectre_status_string(99) == b"unknown status"


@pytest.mark.parametrize("B,H,D,N,nrows,r", [(1, 1, 64, 2, 1, 0), (3, 5, 40, 700, 2, 0), (2, 12, 64, 4096, 3, 2)])
def test_decode_workspace_holds_what_the_step_uses(lib, B, H, D, N, nrows, r):
    # partial rows of every 256 bins, a counter per head, the gate's scratch (raw gate of a banded update, 1024 hidden units, one copy of the sums)
    def up(x):
        return (x + 255) // 256 * 256
    K = N // 2 + 1
    gate = (up(B * H * K * 8) if r else 0) + up(B * H * 1024 * 4) + up(B * H * D * 4)
    rows = up(B * H * ((K + 255) // 256) * {1: 1, 2: 2, 3: 4}[nrows] * D * 4)
    assert lib.spectre_decode_workspace_bytes(None, B, H, D, N, nrows, r) == rows + up(B * H * 4) + gate


def test_struct_layouts_match_the_header():
    from paper_2502_18394_b200 import binding as b
    assert C.sizeof(b.Act) == 8 + 4 * 5 + 4 + 8 * 3        # ptr, dtype+BLHD, pad, strides
    assert C.sizeof(b.Cache) == 4 * 6 + 8 * 4
    assert b.GateParams.ln_eps.offset == 32 and b.GateParams.W1.offset == 40
    assert C.sizeof(b.Wavelet) == 16 + 8 * 7 and b.Wavelet.skip.offset == 16 + 8 * 6


def test_null_arguments_fail_without_a_device(lib):
    import torch
    if torch.cuda.is_available():
        pytest.skip("covers the no-device behaviour")
    h = C.c_void_p()
    assert lib.spectre_create(C.byref(h), 0) == 4            # no CUDA device -> SPECTRE_ERR_CUDA, no fallback
    assert b"no CPU fallback" in lib.spectre_last_error()
    assert lib.spectre_mixer_forward(None, None, None, None, None, 8, None, None, 0) == 1
    assert lib.spectre_prefix_cache_append(None, None, None, None, None, 0) == 1


def test_native_calls_with_another_number_of_arguments_are_refused():
    # in a process of its own: a call that reads beyond its argument array ends the process
    code = ("from paper_2502_18394_b200 import build, binding\nbuild.build()\next = binding._native()\n"
            "for name in ('gate', 'mixer_forward', 'wavelet_refine', 'prefill', 'append', 'decode_step', 'readout', 'project_qv', "
            "'mixer_backward'):\n"
            "    for n in (0, 1, 4, 30):\n"
            "        try:\n            getattr(ext, name)(*[None] * n)\n"
            "        except TypeError as e:\n            assert 'arguments, got %d' % n in str(e), (name, n, e)\n"
            "        else:\n            raise SystemExit(name)\n")
    res = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr


def test_a_flag_without_a_truth_value_raises_its_own_error(lib):
    import torch
    from paper_2502_18394_b200 import binding
    x, w = torch.zeros(1, 8, 1, 64, dtype=torch.bfloat16), torch.zeros(1, 64, 64)
    both = torch.zeros(2)                                    # bool() of it raises
    ext = binding._native()
    with pytest.raises(RuntimeError, match="[Bb]oolean value"):
        ext.mixer_backward(None, x, x, torch.zeros(1, 1, 5, 2), None, both, True, None, None)
    with pytest.raises(RuntimeError, match="[Bb]oolean value"):
        ext.project_qv(None, x, w, w, None, None, None, both, None, None)


def test_the_extension_is_rebuilt_for_another_torch(lib, monkeypatch):
    import torch
    from paper_2502_18394_b200 import build
    assert not build.native_is_stale()
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    assert build.native_is_stale()
