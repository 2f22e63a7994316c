"""The objective's gradient written over x, in launches of every size."""
import pytest
import torch

from paper_2510_03932_gb300 import ocp, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_sm", [1, 200, 300])
@pytest.mark.parametrize("name", ["vdp_n1e3", "cartpole_n1e5", "quadrotor_n1e3", "quadrotor_n1e3:euler"])
def test_gradient_over_x(name, per_sm):
    w = dict(synth.workload(name.split(":")[0]), N=per_sm * torch.cuda.get_device_properties(0).multi_processor_count)
    if name.endswith(":euler"):
        w["scheme"] = "euler"
    w.update(xref=[0.5] * w["nx"], xslope=None, xamp=None, xfreq=None)
    H = ocp.OCP.from_workload(w)
    x = torch.rand(H.n, generator=torch.Generator(device="cuda").manual_seed(9), device="cuda", dtype=torch.float64) * 0.8 + 0.1
    x[:w["nx"] * (w["N"] + 1)].view(-1, w["nx"])[::7] = 0.5    # nodes on the reference: products of zeros, done again
    want = H.eval_grad(x)
    H.eval_grad(x, x)
    assert torch.equal(x, want)
