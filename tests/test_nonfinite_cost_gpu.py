"""A reference that is not a number on a component with a zero weight gives NaN in launches of every size
(0 times NaN), as it does from one call per output."""
import math

import pytest
import torch

from paper_2510_03932_gb300 import ocp, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [math.nan, math.inf])
@pytest.mark.parametrize("name", ["vdp_n1e3", "cartpole_n1e5", "quadrotor_n1e3", "heat_n2e4", "cartpole_n1e5:euler"])
def test_zero_weight_on_a_reference_that_is_not_finite(name, value):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    base = dict(synth.workload(name.split(":")[0]))
    if name.endswith(":euler"):
        base["scheme"] = "euler"
    nx = base["nx"]
    q, xref = list(base["q"]), list(base.get("xref") or [0.0] * nx)
    q[0], xref[0] = 0.0, value
    base.update(q=q, xref=xref, xslope=None, xamp=None, xfreq=None)
    for N in (30, (40 if "heat" in name else 300) * sms):    # a small and a large launch (integer products)
        H = ocp.OCP.from_workload(dict(base, N=N))
        g = torch.Generator(device="cuda").manual_seed(4)
        x = torch.rand(H.n, generator=g, device="cuda", dtype=torch.float64) * 0.8 + 0.1
        f, c, gr, jv, hv = H.eval_all(x, torch.ones(H.m, device="cuda", dtype=torch.float64), 0.5)
        nodes = N if base.get("scheme") == "euler" else N + 1
        for grad in (gr, H.eval_grad(x)):
            X = grad[:nx * nodes].view(nodes, nx)
            assert bool(torch.isnan(X[:, 0]).all()) and not bool(torch.isnan(X[:, 1:]).any())
        assert math.isnan(f.item()) and math.isnan(H.eval_obj(x).item())
        H.close()
