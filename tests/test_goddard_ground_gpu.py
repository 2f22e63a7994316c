"""The rocket at altitude r = 1, where the drag's exponent is exactly zero: one pass over the nodes, and the
values of neighbouring calls."""
import pytest
import torch

from paper_2510_03932_gb300 import ocp, synth
from test_euler_subsets_gpu import best_us

pytestmark = pytest.mark.gpu


def test_nodes_on_the_ground_take_one_pass():
    N = 1000 * torch.cuda.get_device_properties(0).multi_processor_count
    H = ocp.OCP.from_workload(dict(synth.workload("goddard_n1e3"), N=N))
    g = torch.Generator(device="cuda").manual_seed(5)
    U = lambda k: torch.rand(k, generator=g, device="cuda", dtype=torch.float64) * 0.8 + 0.1
    x, y, vn, vm = U(H.n), U(H.m), U(H.n), U(H.m)
    X = x[:3 * (N + 1)].view(N + 1, 3)
    X[:, 0], x[-1] = 1.0, 0.2
    outs = list(H.eval_step(x, y, 0.5, vn, vm))
    want = (H.eval_cons(x), H.eval_grad(x), H.jac_coo_values(x), H.hess_coo_values(x, y, 0.5), H.jprod(x, vn), H.jtprod(x, vm),
            H.hprod(x, y, 0.5, vn))
    assert all(torch.equal(a, b) for a, b in zip(outs[1:], want))
    ground = best_us(lambda: H.eval_step(x, y, 0.5, vn, vm, outs))
    X[:, 0], X[:, 1] = 1.01, 0.0     # exact zeros: the FP64 pipe's products
    fp64 = best_us(lambda: H.eval_step(x, y, 0.5, vn, vm, outs))
    assert ground < 1.25 * fp64      # (integer products first, then these: 1.8)
    H.close()
