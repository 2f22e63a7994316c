"""Forward Euler: a call for some outputs does not work longer than the call for all of them."""
import pytest
import torch

from paper_2510_03932_gb300 import ocp, synth

pytestmark = pytest.mark.gpu


def best_us(fn):
    """Least time of a call among rounds of twenty."""
    times = []
    for _ in range(6):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(20):
            fn()
        e1.record()
        torch.cuda.synchronize()
        times.append(e0.elapsed_time(e1) * 50.0)
    return min(times)


@pytest.mark.parametrize("name", ["vdp_mu_n1e6", "cartpole_n1e5"])
def test_outputs_without_the_hessian_take_no_second_pass(name):
    # large launches (integer products); a second pass over the nodes took 1.26 to 1.98 times the full call
    N = 4000 * torch.cuda.get_device_properties(0).multi_processor_count
    H = ocp.OCP.from_workload(dict(synth.workload(name), N=N, scheme="euler"))
    g = torch.Generator(device="cuda").manual_seed(8)
    U = lambda k: torch.rand(k, generator=g, device="cuda", dtype=torch.float64) * 0.8 + 0.1
    x, y = U(H.n), U(H.m)
    f, c, gr, jv, hv = H.eval_all(x, y, 0.5)
    every = best_us(lambda: H.eval_all(x, y, 0.5, f, c, gr, jv, hv))
    for some in (dict(f=f, c=c), dict(f=f, c=c, g=gr, jvals=jv)):
        assert best_us(lambda: H.eval_all(x, y, 0.5, alloc=False, **some)) < 1.1 * every
