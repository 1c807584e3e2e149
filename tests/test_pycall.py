"""CPU-only: the extension module behind the binding's per-token calls, and ctypes in its place, hand their arguments to the library
as they came.
Every call here ends at the library's own argument checks, before anything touches a GPU."""
import ctypes
import sysconfig

import pytest

import paper_2503_24358_b200 as sq
from paper_2503_24358_b200 import build as sq_build

A, MISALIGNED = 4096, 4100                 # addresses that are checked, never read


@pytest.fixture(scope="module", autouse=True)
def built():
    sq_build.build()


def _values(meta16=False, v=A, dtype=1, T=32, bits=2, G=32, stride_t=128, out=A):
    return sq.binding._direct().quantize_values(meta16, v, dtype, 1, 1, T, 128, 0, 0, stride_t, bits, G, out, out, out, 0, 0, None)


@pytest.fixture(params=["extension", "ctypes"], autouse=True)
def route(request, monkeypatch):
    """Either way into the library: the extension module, and ctypes for an installation that has no compiler or headers."""
    assert sq.binding.PYCALL == sq_build.PYCALL
    if request.param == "ctypes":
        monkeypatch.setattr(sq.binding, "PYCALL", sq.binding.PYCALL + ".missing")
    monkeypatch.setattr(sq.binding, "_lib", None)
    monkeypatch.setattr(sq.binding, "_call", None)
    is_module = type(sq.binding._direct()).__name__ == "module"
    assert is_module == (request.param == "extension")
    return request.param


def test_build_without_compiler_or_headers(monkeypatch, tmp_path):
    assert sq_build.build_pycall() == sq_build.PYCALL and sysconfig.get_config_var("SOABI") in sq_build.PYCALL
    monkeypatch.setenv("CC", "no-such-compiler")
    assert sq_build.build_pycall(force=True) is None
    monkeypatch.delenv("CC")
    monkeypatch.setattr(sysconfig, "get_paths", lambda: {"include": str(tmp_path)})
    assert sq_build.build_pycall(force=True) is None


@pytest.mark.parametrize("kw, status", [
    (dict(v=None), 1), (dict(v=MISALIGNED), 1), (dict(v=2 ** 64 - 12), 1), (dict(dtype=7), 1), (dict(stride_t=64), 1),
    (dict(bits=3), 3), (dict(G=48), 3), (dict(T=0, v=None, out=None), 0)])
@pytest.mark.parametrize("meta16", [False, True])
def test_each_argument_arrives_in_its_place(kw, status, meta16):
    assert _values(meta16, **kw) == status


def test_other_entry_points_report_status():
    call = sq.binding._direct()
    assert call.quantize_keys(False, None, A, 1, 1, 1, 32, 128, 0, 0, 128, 2, 32, A, A, A, 0, 0, None) == 1
    assert call.dequantize(True, 5, A, A, A, 1, 1, 32, 128, 2, 32, 0, 0, A, 0, None) == 1
    assert call.dequantize(False, 0, A, A, A, 1, 1, 33, 128, 2, 32, 0, 0, A, 0, None) == 2
    assert call.decode_attention(0.0, None, 1, 1, 32, 32, 128, A, A, A, A, A, A, False, 32, 0, 0, 2, 32,
                                 None, None, 0, 0, None, 0, 0, A, A, 0, None) == 1


def test_wrong_calls_raise(route):
    call = sq.binding._direct()
    with pytest.raises(TypeError):
        call.dequantize(False, 0, A)
    with pytest.raises((TypeError, ctypes.ArgumentError)):
        _values(bits=2.0)
    if route == "extension":
        with pytest.raises(OverflowError):
            _values(v=2 ** 64)
