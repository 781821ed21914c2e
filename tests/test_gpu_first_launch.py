"""The first launch of any of the library's kernels beside another thread's capture.

In a process of its own, where nothing has run: a kernel that its first launch
had to load would synchronise the context and end the capture."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

RUN = """
import sys, threading, time
sys.path.insert(0, sys.argv[1])
import torch
from paper_0908_0673_gb300 import bem, inputs as I
a = torch.arange(1000.0, device="cuda")
b = (a + 1) * 2
t0 = time.time()
ctx = bem.bem_ctx_create(0)
print("context", time.time() - t0)
err = []

def work():
    try:
        m = I.cube(6, I.TRI6)
        mesh = bem.bem_mesh_create(ctx, m.nodes, m.elems, m.elem_type)
        n, nc = bem.bem_mesh_sizes(mesh)
        for precision in (bem.BEM_F64, bem.BEM_MIXED):
            for green, dt in ((bem.BEM_LAPLACE, torch.float64), (bem.BEM_HELMHOLTZ, torch.complex128)):
                plan = bem.bem_plan_create(mesh, green, 2.0, bem.bem_fmm_params_default(precision=precision, leaf_size=32))
                chi, phi, pts = vec[dt][:nc], out[dt][:n], points
                code, _ = bem.bem_solve(plan, chi, phi)
                assert code == bem.BEM_OK
                bem.bem_field(plan, phi, chi, pts, out[dt][-16:])
                bem.bem_plan_destroy(plan)
    except Exception as e:
        err.append(repr(e))

vec = {dt: torch.ones(20000, device="cuda", dtype=dt) for dt in (torch.float64, torch.complex128)}
out = {dt: torch.zeros(20000, device="cuda", dtype=dt) for dt in (torch.float64, torch.complex128)}
points = 3.0 + torch.arange(48.0, device="cuda", dtype=torch.float64).reshape(16, 3)
g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
torch.cuda.synchronize()
with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
    c = a + 1
    th = threading.Thread(target=work)
    th.start()
    th.join()
    d = c * 2
g.replay()
torch.cuda.synchronize()
assert not err, err
assert torch.equal(d, b)
assert all(torch.isfinite(torch.view_as_real(o) if o.is_complex() else o).all() for o in out.values())
"""


def test_beside_a_capture():
    r = subprocess.run([sys.executable, "-X", "faulthandler", "-c", RUN, os.path.dirname(os.path.dirname(os.path.abspath(__file__)))],
                       capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    print(r.stdout)
