"""Outputs other than H do not need the multipliers."""
import pytest
import torch

from paper_2510_03932_gb300 import ocp, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,N", [("vdp_mu_n1e6", 900), ("cartpole_n1e5", 900), ("cartpole_n1e5", 50_000), ("quadrotor_n1e3", 900),
                                    ("goddard_n1e3", 900), ("goddard_n1e3", 50_000), ("heat_n2e4", 900), ("heat_n2e4", 9000),
                                    ("cartpole_n1e5:euler", 900), ("cartpole_n1e5:euler", 50_000)])
def test_outputs_without_multipliers(name, N):
    # y is needed for H alone
    w = dict(synth.workload(name.split(":")[0]), N=N)
    if name.endswith(":euler"):
        w["scheme"] = "euler"
    H = ocp.OCP.from_workload(w)
    x = torch.rand(H.n, generator=torch.Generator(device="cuda").manual_seed(4), device="cuda", dtype=torch.float64) * 0.8 + 0.1
    want = dict(f=H.eval_obj(x), c=H.eval_cons(x), g=H.eval_grad(x), jvals=H.jac_coo_values(x))
    for some in (("f", "c"), ("g", "jvals"), ("f", "c", "g", "jvals")):
        outs = {k: torch.zeros_like(want[k]) for k in some}
        H.eval_all(x, None, 0.5, alloc=False, **outs)
        assert all(torch.equal(outs[k], want[k]) for k in some)


def test_batch_outputs_without_multipliers():
    w = synth.workload("cartpole_n1e5")
    H = [ocp.OCP.from_workload(dict(w, N=N)) for N in (1, 2, 300)]
    B = ocp.OCPBatch(H)
    x = torch.rand(B.n, generator=torch.Generator(device="cuda").manual_seed(4), device="cuda", dtype=torch.float64) * 0.8 + 0.1
    new = lambda k: torch.zeros(k, device="cuda", dtype=torch.float64)
    f, c, g, jv = new(3), new(B.m), new(B.n), new(B.nnzj)
    B.eval_all(x, None, 0.5, f, c, g, jv, None)
    for i, h in enumerate(H):
        xi = x[int(B.xoff[i]):int(B.xoff[i + 1])].clone()
        assert torch.equal(c[int(B.coff[i]):int(B.coff[i + 1])], h.eval_cons(xi))
        assert torch.equal(jv[int(B.joff[i]):int(B.joff[i + 1])], h.jac_coo_values(xi))
        assert torch.equal(g[int(B.xoff[i]):int(B.xoff[i + 1])], h.eval_grad(xi))
