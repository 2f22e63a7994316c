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


@pytest.mark.parametrize("cells,N", [(2, 3), (17, 30), (64, 3000), (64, 31 * 152), (37, 7003), (64, 20000)])
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


def _chain(H, b, x, y, v, after=lambda: None):
    """Calls that each read what the launch before wrote, or write what it read."""
    b["x"].copy_(x), b["y"].copy_(y), b["v"].copy_(v)
    f, c, g, jv, hv, o1, o2, o3 = b["outs"]
    for call in (lambda: H.eval_all(b["x"], b["y"], 0.5, f, c, g, jv, hv),
                 lambda: H.kkt_values(hv, jv, None, 1e-3, 1e-8, out=b["kkt"]),
                 lambda: H.jprod(b["x"], b["v"], o1),
                 lambda: H.jtprod(b["x"], o1, o2),
                 lambda: H.hprod(b["x"], o1, 0.5, o2, o3),
                 lambda: H.eval_step(b["x"], o1, 0.5, o2, b["y"], outs=b["step"]),
                 lambda: H.eval_grad(b["x"], o2),
                 lambda: H.eval_cons(b["x"], o1),
                 lambda: H.eval_all(b["x"], o1, 0.5, f, c, g, jv, hv),
                 lambda: H.eval_obj(b["x"], f),
                 lambda: H.jac_coo_values(b["x"], b["step"][3]),
                 lambda: H.hess_coo_values(b["x"], c, 0.5, b["step"][4])):
        call()
        after()
    return [t.clone() for t in (*b["outs"], *b["step"], b["kkt"])]


@pytest.mark.parametrize("path", [False, True])
@pytest.mark.parametrize("name,N", [("vdp_mu_n1e6", 50), ("vdp_mu_n1e6", 70_001), ("cartpole_n1e5", 1234),
                                    ("quadrotor_n1e3", 3001), ("goddard_n1e3", 999), ("heat_n2e4", 500)])
def test_chained_launches(name, N, path):
    w = dict(synth.workload(name), N=N)
    H = ocp.OCP.from_workload(synth.with_bineq(synth.with_path(w)) if path else w)
    new = lambda: dict(x=_empty(H)[2], y=_empty(H)[1], v=_empty(H)[2], outs=_empty(H), step=_empty(H),
                       kkt=torch.empty(H.kkt_nnz(), device="cuda", dtype=torch.float64))
    draws = [_draw(H, s)[:3] for s in range(3)]
    b = new()
    want = [_chain(H, b, *d, after=torch.cuda.synchronize) for d in draws]
    same = lambda got: all(torch.equal(p.view(torch.int64), q.view(torch.int64)) for p, q in zip(got, want[-1]))
    b = new()
    got = [_chain(H, b, *d) for d in draws]
    for a, r in zip(got, want):
        assert all(torch.equal(p.view(torch.int64), q.view(torch.int64)) for p, q in zip(a, r))
    b, st = new(), torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        for d in draws:
            got = _chain(H, b, *d)
    torch.cuda.synchronize()
    assert same(got)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = _chain(H, b, *draws[-1])
    for t in (*b["outs"], *b["step"], b["kkt"]):
        t.fill_(0.0)
    graph.replay()
    graph.replay()
    assert same(got)
