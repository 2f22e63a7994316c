"""The heat step whose products run beside its evaluation takes no longer than the one in order.  Outputs in
one buffer (Jv over c) keep the order."""
import pytest
import torch

from paper_2510_03932_gb300 import ocp, synth
from test_euler_subsets_gpu import best_us

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("free", [1, 13, 26, 60])        # SMs without an evaluation CTA
@pytest.mark.parametrize("cells", [8, 16, 32, 48, 64])
def test_products_beside_the_evaluation_pay(cells, free):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    w = dict(synth.workload("heat_n2e4"), nx=cells, params=[float(cells)], q=[1.0] * cells, xref=[0.5] * cells, x0=[0.0] * cells,
             N=31 * (sms - free) - 1)
    H = ocp.OCP.from_workload(w)
    g = torch.Generator(device="cuda").manual_seed(2)
    U = lambda k: torch.rand(k, generator=g, device="cuda", dtype=torch.float64) * 0.8 + 0.1
    x, y, vn, vm = U(H.n), U(H.m), U(H.n), U(H.m)
    outs = list(H.eval_step(x, y, 0.5, vn, vm))
    want = [H.jprod(x, vn), H.jtprod(x, vm), H.hprod(x, y, 0.5, vn)]
    assert all(torch.equal(a, b) for a, b in zip(outs[5:], want))
    beside = best_us(lambda: H.eval_step(x, y, 0.5, vn, vm, outs))
    shared = outs[:5] + [outs[1]] + outs[6:]
    in_order = best_us(lambda: H.eval_step(x, y, 0.5, vn, vm, shared))
    assert beside < 1.05 * in_order
    H.close()
