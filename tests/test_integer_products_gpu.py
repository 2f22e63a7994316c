"""Products on the integer pipes (csrc/soft_mul.cuh) against the FP64 pipe's, bit for bit.

Launches of at least 256 nodes per SM use them.  A warp that holds a zero input does its work with
the FP64 pipe's products, so the same problem is evaluated twice: as drawn, and with a zero put into one node of every sixteen (every warp then
holds one; the heat model decides per warp and cell: into all its cells).  Whatever depends on untouched nodes alone must have the same bits, over ordinary
inputs, inputs over thirty decades (products near both ends of the integer products' range, which
are done again) and multipliers whose sums vanish."""
import numpy as np
import pytest
import torch

from paper_2510_03932_gb300 import synth
from test_parity_gpu import dev, host, named, ocp  # noqa: F401  (ocp: the module fixture)

pytestmark = pytest.mark.gpu

NAMES = ["vdp_n1e3", "cartpole_n1e5", "quadrotor_n1e3", "goddard_n1e3", "vdp_n1e3:euler", "cartpole_n1e5:euler",
         "quadrotor_n1e3:euler", "heat_n2e4"]


def every_output(H, d, sigma):
    x, y, vn, vm = (dev(d[k]) for k in ("x", "y", "vn", "vm"))
    f, c, g, jv, hv, Jv, Jtv, Hv = H.eval_step(x, y, sigma, vn, vm)
    out = dict(step=(c, g, jv, hv, Jv, Jtv, Hv), parts=(H.eval_cons(x), H.eval_grad(x), H.jac_coo_values(x),
                                                        H.hess_coo_values(x, y, sigma), H.jprod(x, vn), H.jtprod(x, vm),
                                                        H.hprod(x, y, sigma, vn)),
               all=H.eval_all(x, y, sigma)[1:])
    if H.nparams and H.model != "goddard" and not d["euler"]:
        out["vjp"] = (H.vjp_params(x, vm)[0],)
    return {k: [host(t) for t in v] for k, v in out.items()}


@pytest.mark.parametrize("kind", ["ordinary", "wide", "cancelling"])
@pytest.mark.parametrize("name", NAMES)
def test_integer_products_have_the_bits_of_the_fp64_pipe(ocp, name, kind):  # noqa: F811
    N = 5000 if name == "heat_n2e4" else 40_007   # (the heat model counts a node n / 8 times)
    w = named(name, N)
    d = synth.draw(w)
    nx, nu, nun = w["nx"], w["nu"], synth.control_nodes(w)
    nX = nx * (N + 1)
    rng = np.random.default_rng(11)
    H = ocp.OCP.from_workload(w)
    if kind == "wide":   # magnitudes over thirty decades (angles and Goddard's states stay in their range)
        fixed = {"cartpole": [2], "quadrotor": [6, 7, 8], "goddard": [0, 1, 2]}.get(w["model"], [])
        X = d["x"][:nX].reshape(N + 1, nx)
        for k in range(nx):
            if k not in fixed:
                X[:, k] *= 10.0 ** rng.uniform(-15, 15, N + 1)
        d["x"][nX:nX + nu * nun] *= 10.0 ** rng.uniform(-15, 15, nu * nun)
        for k in ("y", "vn", "vm"):
            d[k] *= 10.0 ** rng.uniform(-15, 15, d[k].size)
    if kind == "cancelling":   # y_{k,j-1} + y_{k,j} = 0 and w likewise at every third node
        nb = nx + synth.final_rows(w)
        for v in (d["y"], d["vm"]):
            rows = v[nb:nb + nx * N].reshape(nx, N)
            rows[:, 2::3] = -rows[:, 1:-1:3][:, :rows[:, 2::3].shape[1]]
    d["euler"] = w.get("scheme") == "euler"
    base = every_output(H, d, 0.75)
    # a zero into one state of every sixteenth node
    e = dict(d, x=d["x"].copy())
    hit = np.zeros(N + 1, bool)
    hit[3::16] = True
    cols = {"goddard": slice(1, 2), "heat": slice(0, nx)}.get(w["model"], slice(0, 1))
    e["x"][:nX].reshape(N + 1, nx)[hit, cols] = 0.0
    other = every_output(H, e, 0.75)
    # nodes of the variables and rows (tf, the last variable, depends on every node)
    var = np.concatenate([np.repeat(np.arange(N + 1), nx), np.repeat(np.arange(nun), nu)] + ([[3]] if w.get("free_tf") else []))
    rows = np.zeros(H.m, bool)
    nb = nx + synth.final_rows(w)
    rows[nb:] = np.tile(hit[:-1] | hit[1:], nx)
    rows[:nx] = hit[0]
    (jr, jc), (hr, hc) = ([host(t) for t in s] for s in (H.jac_coo_structure(), H.hess_coo_structure()))
    jbad = hit[var[jc]] | (rows[jr] if w.get("free_tf") else False)
    hbad = hit[var[hc]] | hit[var[hr]] * (hr < nX + nu * nun)
    vbad = hit[var]
    if d["euler"]:
        rows[nb:] = np.tile(hit[:-1] | hit[1:], nx)
    if w.get("free_tf"):
        vbad[-1] = True
    bad = dict(step=(rows, vbad, jbad, hbad, rows, vbad, vbad), parts=(rows, vbad, jbad, hbad, rows, vbad, vbad),
               all=(rows, vbad, jbad, hbad), vjp=(vbad,))
    for key, outs in base.items():
        for i, (p, q, b) in enumerate(zip(outs, other[key], bad[key])):
            keep = ~np.asarray(b)
            assert keep.sum() > 0.5 * keep.size
            same = (p == q) | (np.isnan(p) & np.isnan(q))
            assert np.all(same[keep]), (key, i, np.flatnonzero(keep & ~same)[:5])
    # and the calls agree with each other
    for i in range(7):
        assert np.array_equal(base["step"][i], base["parts"][i], equal_nan=True), i
    H.close()


@pytest.mark.parametrize("name", ["vdp_n1e3", "cartpole_n1e5"])
def test_large_batch_slices_have_the_bits_of_small_plain_problems(ocp, name):  # noqa: F811
    """A batch is one launch, large by its total (integer products), while each of its problems
    alone is small (the FP64 pipe's)."""
    Ns = [20_000, 1, 130, 19_999]
    ws = [dict(named(name, N), seed=50 + i) for i, N in enumerate(Ns)]
    ds = [synth.draw(w) for w in ws]
    Hs = [ocp.OCP.from_workload(w) for w in ws]
    B = ocp.OCPBatch(Hs)
    x, y = (dev(np.concatenate([d[k] for d in ds])) for k in ("x", "y"))
    for threads, npt in ((128, 1), (64, 1), (256, 1), (128, 2)):
        B.set_config(npt, threads, 0)
        f, c, g, jv, hv = B.outputs()
        B.eval_all(x, y, 0.75, f, c, g, jv, hv)
        for i, H in enumerate(Hs):
            _, c1, g1, j1, h1 = H.eval_all(dev(ds[i]["x"]), dev(ds[i]["y"]), 0.75)
            for got, off, want in ((c, B.coff, c1), (g, B.xoff, g1), (jv, B.joff, j1), (hv, B.hoff, h1)):
                assert torch.equal(got[off[i]:off[i + 1]], want), (i, threads, npt)
    B.close()
