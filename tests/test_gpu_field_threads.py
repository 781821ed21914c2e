"""Fields of plans of different orders on two host threads at once: the launches
need different amounts of shared memory, and neither may limit the other's."""
import threading

import pytest

from gpu_util import Plan
from paper_0908_0673_gb300 import bem, inputs as I

pytestmark = pytest.mark.gpu


def test_orders_on_two_threads():
    import torch
    plans = [Plan(I.icosphere(1), bem.BEM_HELMHOLTZ, 1.0, p=p, leaf_size=16) for p in (2, 20)]
    n, nc = plans[0].n_phi, plans[0].n_chi
    phi = torch.ones(n, device="cuda", dtype=torch.complex128)
    chi = torch.ones(nc, device="cuda", dtype=torch.complex128)
    pts = torch.full((1, 3), 2.0, device="cuda", dtype=torch.float64)
    bad = []

    def work(P):
        s = torch.cuda.Stream()
        u = torch.zeros(1, device="cuda", dtype=torch.complex128)
        try:
            for _ in range(1500):
                bem.bem_field(P.plan, phi, chi, pts, u, s)
            s.synchronize()
        except Exception as e:
            bad.append(str(e))

    torch.cuda.synchronize()
    th = [threading.Thread(target=work, args=(P,)) for P in plans]
    [t.start() for t in th]
    [t.join() for t in th]
    assert not bad, bad
    [P.close() for P in plans]
