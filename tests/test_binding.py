"""The extension module of the binding against ctypes: the same calls accepted, refused and answered alike."""
import os
import subprocess
import sys
import types

import numpy as np
import pytest
import torch

from paper_2602_02864_b200 import fdc

THROUGH_CTYPES = types.SimpleNamespace(**{n: (lambda *a: None) for n in ("frontier", "build_masks", "kv_append", "decode_attn")})
T = torch.zeros(8, dtype=torch.int64)


def outcome(f):
    try:
        return f()
    except Exception as e:  # noqa: BLE001
        return type(e), str(e)


def calls(plan, x, layer, scale, nbytes, stream, batch):
    kv = fdc.fdc_kv_desc()
    return [lambda: fdc.fdc_frontier(plan, batch, x, None, T, T, T, T, T, x, stream),
            lambda: fdc.fdc_build_masks(plan, batch, T, x, T, T, T, stream),
            lambda: fdc.fdc_kv_append(plan, kv, layer, T, T, x, T, stream),
            lambda: fdc.fdc_decode_attn(plan, kv, layer, T, T, T, T, x, T, scale, T, nbytes, stream)]


# (without a plan every accepted call answers FDC_ERR_NULL: nothing is launched)
@pytest.mark.parametrize("odd", [{}, {"x": None}, {"x": 4096}, {"x": np.zeros(4)}, {"x": 1.5}, {"x": "a"}, {"layer": 2 ** 40}, {"layer": -1},
                                 {"layer": np.int64(3)}, {"layer": 1.0}, {"layer": True}, {"scale": 1}, {"scale": np.float32(0.5)}, {"scale": "b"},
                                 {"nbytes": -1}, {"nbytes": 2.5}, {"nbytes": 2 ** 63}, {"batch": 2 ** 33}, {"batch": None}, {"plan": None}, {"stream": -1}])
def test_odd_arguments_end_as_they_do_through_ctypes(odd, monkeypatch):
    args = dict(plan=0, x=T, layer=0, scale=0.125, nbytes=1 << 20, stream=0, batch=1)
    args.update(odd)
    got = [outcome(f) for f in calls(**args)]
    monkeypatch.setattr(fdc, "_fdc_bind", THROUGH_CTYPES)
    assert got == [outcome(f) for f in calls(**args)]


def test_usual_arguments_do_not_go_through_ctypes():
    kv = fdc.fdc_kv_desc()
    assert fdc._fdc_bind.kv_append(0, kv, 0, T, T, T, T, 0) == fdc.FDC_ERR_NULL
    assert fdc._fdc_bind.decode_attn(0, kv, 0, T, T, T, T, T, T, 0.5, None, 0, 0) == fdc.FDC_ERR_NULL
    assert fdc._fdc_bind.frontier(0, 1, T, None, T, T, T, T, T, T, 0) == fdc.FDC_ERR_NULL
    assert fdc._fdc_bind.build_masks(0, 1, T, T, T, T, T, 0) == fdc.FDC_ERR_NULL


def test_without_the_module_every_call_goes_through_ctypes():
    code = ("import sys; sys.modules['paper_2602_02864_b200._fdc_bind'] = None\n"       # (an import of it raises ImportError)
            "from paper_2602_02864_b200 import fdc\n"
            "kv = fdc.fdc_kv_desc()\n"
            "for f in (lambda: fdc.fdc_frontier(0, 1, 0, None, 0, 0, 0, 0, 0, 0, 0), lambda: fdc.fdc_build_masks(0, 1, 0, 0, 0, 0, 0, 0),\n"
            "          lambda: fdc.fdc_kv_append(0, kv, 0, 0, 0, 0, 0, 0), lambda: fdc.fdc_decode_attn(0, kv, 0, 0, 0, 0, 0, 0, 0, 0.5, 0, 0, 0)):\n"
            "    try: f()\n"
            "    except fdc.FdcError as e: print(e.code)\n")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert r.stdout.split() == [str(fdc.FDC_ERR_NULL)] * 4


def test_the_library_is_built_without_a_c_compiler(monkeypatch, tmp_path):
    from paper_2602_02864_b200 import build
    build.build()
    monkeypatch.setenv("CC", str(tmp_path / "no_such_compiler"))
    monkeypatch.setattr(build, "BIND", str(tmp_path / "_fdc_bind.so"))
    assert build.build() == build.LIB and os.path.exists(build.LIB)
