"""The library from a second CUDA context of the same device: a kernel's shared-memory limit belongs to
the context it was set in, so calls that need more than the default have to work in every context."""
import subprocess
import sys
import textwrap

import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu

CHILD = """
import ctypes
import numpy as np
import torch
from paper_2608_04771_gb300 import build, reco
from paper_2608_04771_gb300 import workloads as W
build.build()
L = reco.lib()
wl = W.WORKLOADS["tiny"].reduced(L=300, decode_steps=1)
K, V = W.make_cache(wl, "cuda", canary=False)
qw, (q, kn, vn) = W.make_qwin(wl, "cuda"), W.make_decode_step(wl, 0, "cuda")
lens = torch.full(K.shape[:3], 280, dtype=torch.int32, device="cuda")
kv = reco.make_kv(K, V, wl.h_q)
ws = reco.workspace(reco.RECO_OP_SCORE, kv, wl.w), reco.workspace(reco.RECO_OP_DECODE, kv)
scores = torch.zeros(K.shape[:4], dtype=torch.float32, device="cuda")
out = torch.zeros(q.shape, dtype=torch.float32, device="cuda")
lse = torch.zeros(q.shape[:3], dtype=torch.float32, device="cuda")
host = [t.cpu().numpy().copy() for t in (K, V, qw, q, lens, *ws, scores, out, lse)]
reco.reco_score_cache(kv, qw, lens, wl.w, wl.pool, wl.scale(), scores, ws[0])
reco.reco_decode_attn(kv, q, None, None, lens, wl.scale(), out, lse, ws[1])
reco.reco_check()
want = [t.cpu().numpy() for t in (scores, out, lse)]

cu = ctypes.CDLL("libcuda.so.1")
def ok(status):
    assert status == 0, status
ctx = ctypes.c_void_p()
dev = ctypes.c_int()
ok(cu.cuDeviceGet(ctypes.byref(dev), 0))
ok(cu.cuCtxCreate_v2(ctypes.byref(ctx), 0, dev))  # current on this thread from here on
ptr = []
for x in host:
    p = ctypes.c_uint64()
    ok(cu.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(x.nbytes)))
    ok(cu.cuMemcpyHtoD_v2(p, ctypes.c_void_p(x.ctypes.data), ctypes.c_size_t(x.nbytes)))
    ptr.append(p.value)
pK, pV, pqw, pq, plens, pws0, pws1, pscores, pout, plse = ptr
kv2 = reco.reco_kv(pK, pV, kv.n_layers, kv.B, kv.H_q, kv.H_kv, kv.L_cap, kv.d, kv.dtype)
reco._ok(L.reco_score_cache(ctypes.byref(kv2), pqw, plens, None, wl.w, wl.pool, wl.scale(), pscores, pws0,
                            ws[0].numel(), None))
reco._ok(L.reco_decode_attn(ctypes.byref(kv2), pq, None, None, plens, wl.scale(), pout, reco.RECO_F32, plse, pws1,
                            ws[1].numel(), None))
ok(cu.cuCtxSynchronize())
for p, x, y in zip((pscores, pout, plse), host[-3:], want):
    ok(cu.cuMemcpyDtoH_v2(ctypes.c_void_p(x.ctypes.data), ctypes.c_uint64(p), ctypes.c_size_t(x.nbytes)))
    np.testing.assert_array_equal(x, y)
for p in ptr:
    ok(cu.cuMemFree_v2(ctypes.c_uint64(p)))
ok(cu.cuCtxDestroy_v2(ctx))
print("same results in both contexts")
"""


def test_second_context_of_the_device():
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(CHILD)], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and "same results in both contexts" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]
