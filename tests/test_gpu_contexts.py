"""A program with two CUDA contexts on a device: the kernels' attributes (dynamic shared memory) belong to a context, so a
call in the second one sets them again.  In a process of its own, which makes the second context."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import ctypes
import torch
from paper_2608_17336_b200 import binding as tm

cu = ctypes.CDLL("libcuda.so.1")


def check(rc):
    assert rc == 0, rc


class Buf:                                  # memory of the context that is current now
    def __init__(self, data):
        self.n, self.data = len(data), data
        self.p = ctypes.c_uint64()
        check(cu.cuMemAlloc_v2(ctypes.byref(self.p), ctypes.c_size_t(self.n)))
        check(cu.cuMemcpyHtoD_v2(self.p, data, ctypes.c_size_t(self.n)))

    def read(self):
        out = ctypes.create_string_buffer(self.n)
        check(cu.cuMemcpyDtoH_v2(out, self.p, ctypes.c_size_t(self.n)))
        return out.raw


def run(L, Hq, Hk, d):
    """Raw bytes of every result: quantise, pack, attend, then a decode step over the codes; in the current context."""
    gen = torch.Generator().manual_seed(d)
    fp16 = lambda *shape: torch.randn(shape, generator=gen).half().numpy().tobytes()  # noqa: E731
    p = tm.problem(1, Hq, Hk, L, d, d, d, 1)
    q, k, v = Buf(fp16(1, Hq, L, d)), Buf(fp16(1, Hk, L, d)), Buf(fp16(1, Hk, L, d))
    nq, nk, blocks = Hq * L * d, Hk * L * d, p.T_m
    zeros = lambda n: Buf(bytes(n))  # noqa: E731
    q8, k8, qs, ks = zeros(nq), zeros(nk), zeros(4 * Hq * blocks), zeros(4 * Hk * blocks)
    v8, vs = zeros(nk), zeros(4 * Hk * blocks)
    route = Buf(bytes(i % 2 for i in range(Hk * p.T_m * p.T_mask)))
    words, counts, out, ws = zeros(4 * Hk * p.T_m * p.W), zeros(16 * Hk), zeros(2 * nq), zeros(4096)
    lib, ref = tm.lib(), ctypes.byref(p)
    check(lib.tilemix_quantize_qk(ref, q.p.value, k.p.value, q8.p.value, k8.p.value, qs.p.value, ks.p.value, None))
    check(lib.tilemix_quantize_qk(ref, None, v.p.value, None, v8.p.value, None, vs.p.value, None))
    check(lib.tilemix_pack_routing_mask(ref, route.p.value, 0, words.p.value, counts.p.value, None))
    check(lib.tilemix_attention_fwd(ref, q.p.value, k.p.value, v.p.value, q8.p.value, k8.p.value, qs.p.value, ks.p.value,
                                    words.p.value, out.p.value, None, ws.p.value, 4096, None, None))
    dp = tm.decode_problem(1, Hq, Hk, d, L, d, 1)
    size = tm.tilemix_decode_workspace_size(dp)
    dws, dout, lens = zeros(size), zeros(2 * Hq * d), Buf((L - 1).to_bytes(4, "little"))
    row = Buf(bytes([0xff] * (4 * Hk)))
    check(lib.tilemix_decode_int8kv(ctypes.byref(dp), q.p.value, k.p.value, k8.p.value, ks.p.value, v8.p.value, vs.p.value,
                                    row.p.value, lens.p.value, dout.p.value, None, None, None, dws.p.value, size, None))
    check(cu.cuCtxSynchronize())
    return [b.read() for b in (q8, k8, qs, ks, v8, vs, words, counts, out, dout)]


torch.zeros(1, device="cuda")               # the primary context, current
shapes = [(300, 2, 1, 64), (300, 2, 1, 128)]
first = [run(*s) for s in shapes]
ctx, primary = ctypes.c_void_p(), ctypes.c_void_p()
check(cu.cuCtxGetCurrent(ctypes.byref(primary)))
check(cu.cuCtxCreate_v2(ctypes.byref(ctx), 0, 0))
second = [run(*s) for s in shapes]
check(cu.cuCtxSetCurrent(primary))
again = [run(*s) for s in shapes]
assert first == second and first == again
assert any(any(b) for b in first[0][8:])
print("same")
'''


def test_a_second_context_of_the_device():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "same", r.stdout[-500:] + r.stderr[-1500:]
