"""Forward Euler's single calls and its fused step have the same bits in every range of launch sizes."""
import pytest
import torch

from paper_2510_03932_gb300 import ocp, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [288, 19_500, 30_000, 39_000])   # small, middle (plain products) and large (integer products)
@pytest.mark.parametrize("name", ["quadrotor_n1e3", "cartpole_n1e5"])
def test_euler_single_calls_equal_the_step(name, N):
    H = ocp.OCP.from_workload(dict(synth.workload(name), N=N, scheme="euler"))
    g = torch.Generator(device="cuda").manual_seed(6)
    U = lambda k: torch.rand(k, generator=g, device="cuda", dtype=torch.float64) * 0.8 + 0.1
    x, y, vn, vm = U(H.n), U(H.m), U(H.n), U(H.m)
    f, c, gr, jv, hv, o1, o2, o3 = H.eval_step(x, y, 0.5, vn, vm)
    for got, want in ((H.eval_cons(x), c), (H.eval_grad(x), gr), (H.jac_coo_values(x), jv), (H.hess_coo_values(x, y, 0.5), hv),
                      (H.jprod(x, vn), o1), (H.jtprod(x, vm), o2), (H.hprod(x, y, 0.5, vn), o3), (H.eval_obj(x), f)):
        assert torch.equal(got, want)
