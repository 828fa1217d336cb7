"""The binding's own callables of the C ABI (csrc/calls.c): which interpreter they are for, what they convert and what they refuse."""
import ctypes
import os
import re
import shutil
import subprocess
import sys
import sysconfig

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PACKAGE = os.path.join(ROOT, "paper_2609_33135_b200")


@pytest.fixture(scope="module")
def binding():
    from paper_2609_33135_b200 import binding, build
    build.build()
    binding.lib()
    return binding


def entries():
    """name -> (kinds, members) of the ENTRY lines."""
    text = open(os.path.join(PACKAGE, "csrc", "calls.c")).read()
    return {m.group(1): (m.group(2), re.findall(r"v\[(\d+)\]\.(\w)", m.group(3)))
            for m in re.finditer(r'^ENTRY\((\w+), "(\w+)",([^;]*?)\)\n(?=ENTRY|\n)', text, flags=re.M)}


def test_the_module_is_named_for_its_interpreter_and_no_other_is_taken(binding, tmp_path):
    """Another interpreter's module, or one whose name does not say whose it is, is left alone; the typed and the host-only functions
    work without any, and the wrappers say what is missing."""
    from paper_2609_33135_b200 import build
    assert build.CALLS.endswith("_mpfa_calls" + sysconfig.get_config_var("EXT_SUFFIX")) and os.path.exists(build.CALLS)
    copy = tmp_path / "paper_2609_33135_b200"
    copy.mkdir()
    for f in ("__init__.py", "binding.py", "build.py", "libmpfa.so"):
        shutil.copy(os.path.join(PACKAGE, f), copy / f)
    for other in ("_mpfa_calls.so", "_mpfa_calls.cpython-399-x86_64-linux-gnu.so"):
        shutil.copy(build.CALLS, copy / other)
    child = """
import ctypes, torch
from paper_2609_33135_b200 import binding as B
L = B.lib()
assert L.mpfa_version() >= 100 and L.mpfa_v_fp8_bytes(1, 1, 1) == 128 * 128
assert L.mpfa_prefill(None, None, None, None, None, 1.0, 0, 1.0, None, None, None, None) == -1
try:
    L.packed_mpfa_prefill(None)
except B.MpfaError as e:
    assert "build it with" in str(e), e
else:
    raise AssertionError("the call went through")
"""
    r = subprocess.run([sys.executable, "-c", child], cwd=tmp_path, env=dict(os.environ, PYTHONPATH=str(tmp_path)), capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


def test_kinds_are_the_declared_argument_types(binding):
    """A kind that differs from the member that is passed, or from the C ABI's type, would go unnoticed by the compiler."""
    found = entries()
    assert len(found) == 7
    letter = {ctypes.c_int: "i", ctypes.c_float: "f", ctypes.c_size_t: "z"}
    for name, (kinds, members) in found.items():
        assert kinds == "".join(letter.get(t, "p") for t in getattr(binding.lib(), name).argtypes), name
        assert members == [(str(k), c) for k, c in enumerate(kinds)], name


@pytest.mark.parametrize("name", sorted(entries()))
def test_conversions_and_what_is_refused(binding, name):
    kinds = entries()[name][0]
    call = getattr(binding.lib(), "packed_" + name)
    null = [{"p": None, "i": 1, "f": 1.0, "z": 0}[c] for c in kinds]
    assert call(*null) == -1 and call(*[0 if c == "p" else x for c, x in zip(kinds, null)]) == -1   # None and 0 are null pointers
    for args in (null[:-1], null + [None]):
        with pytest.raises(TypeError, match="arguments"):
            call(*args)
    bad = {"p": ("text", 1.5, bytearray(8)), "i": (None, 1.5, b"1"), "f": (None, "1"), "z": (None, 1.5)}
    for k, c in enumerate(kinds):
        for x in bad[c]:
            with pytest.raises(TypeError):
                call(*null[:k], x, *null[k + 1:])
        for x in {"i": (1 << 31, -(1 << 31) - 1, 1 << 70), "z": (-1, 1 << 64)}.get(c, ()):
            with pytest.raises(OverflowError):
                call(*null[:k], x, *null[k + 1:])
    with pytest.raises(KeyError):
        binding._calls().bind(name + "_", 0)


def test_quantize_qkv_status_codes(binding):
    """What the call refuses before any CUDA call (well-aligned addresses that nothing dereferences), by both kinds of function."""
    a = 1 << 20
    st, q, k = binding._Stats(a, a, a, a), binding._Fp4(a, a, 1, 8, 100), binding._Fp4(a, a, 1, 2, 100)
    good = dict(q=a, k=a, v=a, B=1, N_q=100, N_kv=100, H_q=8, H_kv=2, flags=1, v_scale=1.0, st=st, q_out=q, k_out=k, v_fp8=a, delta=a, ws=a,
                nbytes=0, stream=None)
    cases = [({}, -4),                                                       # everything but the workspace's size
             ({"v": None}, -1), ({"v_fp8": None}, -1), ({"N_kv": 0}, -1), ({"B": 0}, -1),
             ({"v_scale": 0.0}, -1), ({"v_scale": -1.0}, -1), ({"v_scale": float("nan")}, -1),
             ({"v": a + 8}, -3), ({"v_fp8": a + 512}, -3),
             ({"B": 65536}, -2), ({"H_kv": 65536}, -2),
             ({"k": None}, -4), ({"q": None}, -1), ({"ws": None}, -1), ({"delta": None}, -1)]
    typed, packed = binding.lib().mpfa_quantize_qkv, binding.lib().packed_mpfa_quantize_qkv
    for change, want in cases:
        args = list(dict(good, **change).values())
        assert packed(*[bytes(x) if isinstance(x, ctypes.Structure) else x for x in args]) == want, change
        assert typed(*[ctypes.byref(x) if isinstance(x, ctypes.Structure) else x for x in args]) == want, change
