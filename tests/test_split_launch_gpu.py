"""The split evaluation of the smallest launches gives the bits of one call per output."""
import pytest
import torch

from paper_2510_03932_gb300 import ocp, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [False, True])
@pytest.mark.parametrize("name", ["quadrotor_n1e3", "cartpole_n1e5"])
@pytest.mark.parametrize("N", [2, 62, 63, 64, 1000, "last", "next"])
def test_split_equals_separate_calls(name, N, rows):
    edge = 64 * torch.cuda.get_device_properties(0).multi_processor_count   # nodes of the largest split launch
    w = dict(synth.workload(name), N={"last": edge - 1, "next": edge}.get(N, N))
    H = ocp.OCP.from_workload(synth.with_bineq(synth.with_path(w)) if rows else w)
    g = torch.Generator(device="cuda").manual_seed(3)
    U = lambda k: torch.rand(k, generator=g, device="cuda", dtype=torch.float64) * 0.8 + 0.1
    x, y, vn, vm = U(H.n), U(H.m) - 0.5, U(H.n), U(H.m)
    f, c, gr, jv, hv, o1, o2, o3 = H.eval_step(x, y, 0.5, vn, vm)
    want = dict(f=H.eval_obj(x), c=H.eval_cons(x), g=H.eval_grad(x), jvals=H.jac_coo_values(x),
                hvals=H.hess_coo_values(x, y, 0.5))
    assert torch.equal(o1, H.jprod(x, vn)) and torch.equal(o2, H.jtprod(x, vm)) and torch.equal(o3, H.hprod(x, y, 0.5, vn))
    every = dict(f=f, c=c, g=gr, jvals=jv, hvals=hv)
    assert all(torch.equal(every[k], want[k]) for k in want)
    for some in (tuple(want), ("c",), ("f", "g"), ("hvals",), ("f", "c", "hvals"), ("g", "jvals")):
        outs = {k: torch.zeros_like(want[k]) for k in some}
        H.eval_all(x, y, 0.5, alloc=False, **outs)
        assert all(torch.equal(outs[k], want[k]) for k in some)
