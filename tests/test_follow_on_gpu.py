"""Launches that overlap the end of the one before them give the results of separate calls."""
import pytest
import torch

from paper_2510_03932_gb300 import ocp, synth

pytestmark = pytest.mark.gpu


def _heat(cells, N):
    w = synth.workload("heat_n2e4")
    return ocp.OCP.from_workload(dict(w, nx=cells, N=N, params=[float(cells)], q=[1.0] * cells, xref=[0.5] * cells, x0=[0.25] * cells, xf=None))


def _draw(H, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    U = lambda k, lo, hi: torch.rand(k, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo
    return U(H.n, 0.1, 0.9), U(H.m, -1, 1), U(H.n, -1, 1), U(H.m, -1, 1)


def _empty(H):
    e = lambda k: torch.empty(k, device="cuda", dtype=torch.float64)
    return [e(1), e(H.m), e(H.n), e(H.nnzj), e(H.nnzh), e(H.m), e(H.n), e(H.n)]


def _separate(H, x, y, vn, vm):
    f, c, g, jv, hv, o1, o2, o3 = _empty(H)
    H.eval_all(x, y, 0.5, f, c, g, jv, hv)
    torch.cuda.synchronize()
    H.jprod(x, vn, o1)
    torch.cuda.synchronize()
    H.jtprod(x, vm if vm is not None else c, o2)
    torch.cuda.synchronize()
    H.hprod(x, y, 0.5, vn, o3)
    return [f, c, g, jv, hv, o1, o2, o3]


@pytest.mark.parametrize("cells,N", [(2, 3), (17, 30), (64, 31 * 152), (37, 7003), (64, 20000)])
def test_heat_step_products_beside_the_evaluation(cells, N):
    H = _heat(cells, N)
    outs = _empty(H)
    for seed in range(3):   # the inputs are written by the launches just before the step
        x, y, vn, vm = _draw(H, seed)
        got = [t.clone() for t in H.eval_step(x, y, 0.5, vn, vm, outs=outs)]
        for a, b in zip(got, _separate(H, x, y, vn, vm)):
            assert torch.equal(a, b)


def test_heat_step_with_arrays_that_share_memory():
    # w is the array that c is written to: the products come after the evaluation
    H = _heat(64, 20000)
    x, y, vn, _ = _draw(H, 5)
    outs = _empty(H)
    got = H.eval_step(x, y, 0.5, vn, outs[1], outs=outs)
    for a, b in zip(got, _separate(H, x, y, vn, None)):
        assert torch.equal(a, b)
