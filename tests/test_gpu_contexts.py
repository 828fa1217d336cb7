"""A device can have more than one context in a process (a library that makes its own, or a reset of the primary one).  What the
library has told the driver about a kernel in one of them does not hold in another."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.gpu

CHILD = r"""
import ctypes, sys
sys.path.insert(0, sys.argv[1])
from paper_2609_33135_b200 import binding
cu = ctypes.CDLL("libcuda.so.1")
def ok(rc):
    assert rc == 0, rc
ok(cu.cuInit(0))
dev = ctypes.c_int()
ok(cu.cuDeviceGet(ctypes.byref(dev), 0))
primary, other = ctypes.c_void_p(), ctypes.c_void_p()
ok(cu.cuDevicePrimaryCtxRetain(ctypes.byref(primary), dev))
ok(cu.cuCtxCreate_v2(ctypes.byref(other), 0, dev))
L = binding.lib()

def calls():
    def mem(n):
        p = ctypes.c_uint64()
        ok(cu.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(n)))
        ok(cu.cuMemsetD8_v2(p, ctypes.c_ubyte(0), ctypes.c_size_t(n)))
        return p.value
    m = [mem(1 << 20) for _ in range(12)]     # zeros: scores and outputs 0, contexts without keys
    st = binding._Stats(m[0], m[1], m[2], m[3])
    q, k = binding._Fp4(m[4], m[5], 1, 4, 100), binding._Fp4(m[6], m[7], 1, 2, 100)
    kv = binding._PagedKV(m[6], m[7], m[8], None, 4, 64, 4, 2)
    b = ctypes.byref
    rc = [L.mpfa_prefill_variant(b(q), b(k), m[8], None, b(st), 1.0, 0, 0.1, v, m[9], None, m[10], None) for v in (0, 2)]
    rc.append(L.mpfa_prefill_paged(b(q), b(kv), m[11], 4, m[11], None, b(st), 1.0, 0.1, m[9], None, m[10], None))
    q1 = binding._Fp4(m[4], m[5], 1, 4, 1)
    rc.append(L.mpfa_decode(b(q1), b(kv), m[11], 4, m[11], b(st), 1.0, 0.1, m[9], None, m[1], 1 << 20, m[10], None))
    ok(cu.cuCtxSynchronize())
    status = ctypes.c_int(-1)
    ok(cu.cuMemcpyDtoH_v2(ctypes.byref(status), ctypes.c_uint64(m[10]), ctypes.c_size_t(4)))
    return rc, status.value

for ctx in (primary, other, primary):
    ok(cu.cuCtxSetCurrent(ctx))
    print(*calls(), flush=True)
"""


def test_calls_in_a_second_context_of_the_device():
    out = subprocess.run([sys.executable, "-c", CHILD, ROOT], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    assert out.stdout.split("\n")[:3] == ["[0, 0, 0, 0] 0"] * 3, out.stdout


def test_a_failed_launch_does_not_fail_the_next_call():
    """A launch that the driver refuses (more batch elements than a grid's third dimension holds) is reported by its own call only."""
    import torch
    from paper_2609_33135_b200 import binding
    small = torch.ones(1, 1, 1, 128, dtype=torch.bfloat16, device="cuda")
    many = torch.zeros(65536, 1, 1, 128, dtype=torch.bfloat16, device="cuda")
    out = torch.empty(binding.lib().mpfa_v_fp8_bytes(65536, 1, 1), dtype=torch.uint8, device="cuda")
    for _ in range(2):
        with pytest.raises(binding.MpfaError, match="CUDA"):
            binding.mpfa_quantize_v(many, 1.0, out)
        tiles = binding.mpfa_pack_v_bf16(small)
        torch.cuda.synchronize()
        assert float(tiles[0, 0, 0].float().min()) == 1.0
