"""Plans built, run, read and destroyed while other host threads capture graphs.

Nothing here may wait for the whole device: such a wait fails beside a capture
and ends it.  The stress runs in a process of its own."""
import os
import subprocess
import sys
import threading

import pytest

from gpu_util import Plan
from paper_0908_0673_gb300 import bem, inputs as I

pytestmark = pytest.mark.gpu

PRM = dict(p=8, leaf_size=32, eta=2.0, precision=bem.BEM_MIXED)


def test_another_threads_capture_survives():
    import torch
    m = I.icosphere(3)
    ctx = bem.bem_ctx_create(0)
    mesh = bem.bem_mesh_create(ctx, m.nodes, m.elems, m.elem_type)
    n = bem.bem_mesh_sizes(mesh)[0]
    x = torch.tensor(I.random_vector(n, 80), device="cuda")
    prm = bem.bem_fmm_params_default(**PRM)

    def request(out, plans):
        s = torch.cuda.Stream()
        for plan in plans:                           # destroyed with its product still running
            bem.bem_matvec(plan, bem.BEM_OP_A, x, torch.empty_like(x), s)
            bem.bem_plan_destroy(plan)
        plan = bem.bem_plan_create(mesh, bem.BEM_LAPLACE, 0.0, prm, s)   # on the blocks given back
        y = torch.empty_like(x)
        bem.bem_matvec(plan, bem.BEM_OP_A, x, y, s)
        d = bem.bem_plan_diagonal(plan, n)
        bem.bem_plan_export_tree(plan)
        assert bem.bem_plan_device_status(plan) == 0
        s.synchronize()
        bem.bem_plan_destroy(plan)
        out += [y, d]

    ref = []
    request(ref, [bem.bem_plan_create(mesh, bem.BEM_LAPLACE, 0.0, prm)])   # also loads every kernel
    plans = [bem.bem_plan_create(mesh, bem.BEM_LAPLACE, 0.0, prm) for _ in range(3)]
    got, err = [], []

    def body():
        try:
            request(got, plans)
        except Exception as e:
            err.append(e)

    a = torch.arange(1000.0, device="cuda")
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
        b = a + 1
        th = threading.Thread(target=body)
        th.start()
        th.join()
        c = b * 2
    g.replay()
    torch.cuda.synchronize()
    assert not err, err
    assert torch.equal(c, (a + 1) * 2)
    assert torch.equal(got[0], ref[0]) and (got[1] == ref[1]).all()
    bem.bem_mesh_destroy(mesh)
    bem.bem_ctx_destroy(ctx)


def test_plan_used_under_the_callers_capture():
    """Replays are not the plan's to see: its memory is freed after a wait by cudaFree, its state read after one."""
    import torch
    P = Plan(I.icosphere(3), **PRM)
    x = torch.tensor(I.random_vector(P.n_phi, 81), device="cuda")
    y, ref = torch.empty_like(x), torch.empty_like(x)
    bem.bem_matvec_noalloc(P.plan, bem.BEM_OP_A, x, ref)
    torch.cuda.synchronize()
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
        bem.bem_matvec_noalloc(P.plan, bem.BEM_OP_A, x, y, s)
    for _ in range(20):
        g.replay()
    assert bem.bem_plan_device_status(P.plan) == 0
    torch.cuda.synchronize()
    assert torch.equal(y, ref)
    del g
    P.close()


STRESS = """
import sys, threading, time
sys.path.insert(0, sys.argv[1])
import torch
from paper_0908_0673_gb300 import bem, inputs as I
torch.cuda.init()
prm = bem.bem_fmm_params_default(p=8, leaf_size=32, precision=bem.BEM_MIXED)
bad, done = [], [0]
ctx = bem.bem_ctx_create(0)

def work(level, end):
    try:
        s, ref, m = torch.cuda.Stream(), None, I.icosphere(level)
        mesh = bem.bem_mesh_create(ctx, m.nodes, m.elems, m.elem_type)
        x = torch.arange(bem.bem_mesh_sizes(mesh)[0], device="cuda", dtype=torch.float64)
        torch.cuda.current_stream().synchronize()
        while time.time() < end or ref is None:
            y = torch.empty_like(x)
            plan = bem.bem_plan_create(mesh, bem.BEM_LAPLACE, 0.0, prm, s)
            bem.bem_matvec(plan, bem.BEM_OP_A, x, y, s)
            bem.bem_plan_destroy(plan)
            s.synchronize()
            ref = y if ref is None else ref
            assert torch.equal(y, ref)
            done[0] += 1
    except Exception as e:
        bad.append(repr(e))

for level in (2, 3):                             # loads every kernel (a load ends captures too)
    work(level, 0.0)
end = time.time() + 4.0
work_threads = [threading.Thread(target=work, args=(2 + i % 2, end)) for i in range(3)]
[t.start() for t in work_threads]
[t.join() for t in work_threads]
assert not bad, bad
assert done[0] > 30, done
"""


def test_threads_building_and_destroying():
    here = os.path.dirname(os.path.abspath(__file__))
    r = subprocess.run([sys.executable, "-X", "faulthandler", "-c", STRESS, os.path.dirname(here)],
                       capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
