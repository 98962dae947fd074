"""Indexed queues on a part of the GPU: their compaction is a cooperative
launch, which is refused where its CTAs do not fit on the SMs at once.  The
part is a green context of a few SMs, in a process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes as C
import sys
import numpy as np
import torch
import oracle as O
from paper_2608_01657_gb300 import binding as B
from paper_2608_01657_gb300 import workloads as W
from _util import compare_outputs, ctl_word

torch.zeros(1, device="cuda")
cu = C.CDLL("libcuda.so.1")
SM = 1  # CU_DEV_RESOURCE_TYPE_SM; a CUdevResource is 144 bytes, its SM count at byte 96


def call(name, *args):
    rc = getattr(cu, name)(*args)
    if rc:
        print("unavailable: %s returned %d" % (name, rc))
        sys.exit(77)


dev, nparts = C.c_int(), C.c_uint(1)
whole, part, rest = ((C.c_ubyte * 144)() for _ in range(3))
desc, green, ctx, primary = (C.c_void_p() for _ in range(4))
call("cuDeviceGet", C.byref(dev), 0)
call("cuCtxGetCurrent", C.byref(primary))
call("cuDeviceGetDevResource", dev, whole, SM)
call("cuDevSmResourceSplitByCount", part, C.byref(nparts), whole, rest, 0, 16)
call("cuDevResourceGenerateDesc", C.byref(desc), part, 1)
call("cuGreenCtxCreate", C.byref(green), desc, dev, 1)
call("cuCtxFromGreenCtx", C.byref(ctx), green)
sms = int.from_bytes(bytes(part[96:100]), "little")
assert 0 < sms < 100, sms


class on_part:  # the library's calls run in the part, torch's in the whole
    def __enter__(self):
        torch.cuda.synchronize()
        call("cuCtxSetCurrent", ctx)

    def __exit__(self, *a):
        call("cuCtxSynchronize")
        call("cuCtxSetCurrent", primary)


N, G, R = 40, 3, 8
kw = dict(rho=(2.0,), beta=(6.0,), flags=B.PS_FLAG_INDEXED_QUEUES)
steps = W.fuzz_steps(3, G, R, 120, docs_per_group=3, doc_blocks=6, fresh_max_blocks=1, now_stride=2)
L = B.load()
p = B.Params(**kw).to_c(G)
nbytes = L.ps_workspace_bytes(N, 16, G, C.byref(p), R, 4096)
gpu = B.Cache.__new__(B.Cache)  # torch's allocations here, the handle in the part
gpu.workspace = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
i32, i64 = dict(dtype=torch.int32, device="cuda"), dict(dtype=torch.int64, device="cuda")
B4 = 4096 // 16
gpu.out = {"hit_blocks": torch.empty(R, **i32), "admitted_blocks": torch.empty(R, **i32),
           "admitted_offsets": torch.empty(R + 1, **i32), "admitted_ids": torch.empty(B4, **i32),
           "evicted_ids": torch.empty(B4, **i32), "invalidated_ids": torch.empty(B4, **i32),
           "counts": torch.zeros(4, **i32), "debt_raw": torch.empty(G, **i64), "debt_norm": torch.empty(G, **i64)}
out = B.step_out(gpu.out)
h = C.c_void_p()
with on_part():
    assert L.ps_create(C.byref(h), N, 16, G, B.POLICIES["prefixshield"], C.byref(p), gpu.workspace.data_ptr(), nbytes,
                       R, 4096, None) == 0
orc = O.OracleCache(N, 16, G, "prefixshield", O.Params(**kw))
buffers = set()
for k, st in enumerate(steps):
    g, o, t = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (st.groups, st.offsets, st.tokens))
    with on_part():
        rc = L.ps_step(h, None, st.now, st.num_requests, g.data_ptr(), o.data_ptr(), t.data_ptr(), None, None, C.byref(out))
    assert rc == 0, "step %d returned %d" % (k, rc)
    compare_outputs(gpu.fetch(st.num_requests), orc.step(st.now, st.groups, st.offsets, st.tokens), "step %d" % k)
    buffers.add(int(ctl_word(gpu, "lg_buf", torch.int32).item()))
assert buffers == {0, 1}, "no compaction ran"
with on_part():
    assert L.ps_uses_graph(h) == 1
    L.ps_destroy(h)
print("ok on %d SMs" % sms)
"""


def test_indexed_queues_on_a_few_sms():
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([ROOT, os.path.join(ROOT, "tests")]))
    r = subprocess.run([sys.executable, "-c", CHILD], env=env, cwd=ROOT, capture_output=True, text=True, timeout=120)
    if r.returncode == 77:
        pytest.skip(r.stdout.strip())
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    assert "ok on" in r.stdout
