"""Inputs with exact zeros in large launches (where warps that hold one leave the integer products, see
csrc/soft_mul.cuh): the bits of a small problem, whose kernels have the FP64 pipe's products alone.

The small problem is the first eighth of the large one: its horizon (and final time) is an eighth too, so
the step is the same number and every interior node and defect row has the same values."""
import numpy as np
import pytest
import torch

from paper_2510_03932_gb300 import ocp, synth

pytestmark = pytest.mark.gpu

NAMES = ["vdp_n1e3", "cartpole_n1e5", "quadrotor_n1e3", "goddard_n1e3", "heat_n2e4", "vdp_n1e3:euler", "cartpole_n1e5:euler",
         "quadrotor_n1e3:euler"]


def with_zeros(w, d, kind):
    """Exact zeros of one sign in one state, the multipliers, most of the directions, or all of x and y."""
    zero = -0.0 if kind == "negative" else 0.0
    X = d["x"][:w["nx"] * (w["N"] + 1)].reshape(w["N"] + 1, w["nx"])
    if kind in ("state", "negative"):
        X[:, 1 if w["model"] == "goddard" else 0] = zero
    if kind in ("multipliers", "all"):
        d["y"][:] = zero
    if kind in ("directions", "negative"):
        for k in ("vn", "vm"):
            d[k][np.arange(d[k].size) % 97 != 5] = zero
    if kind == "all" and w["model"] != "goddard":
        d["x"][:] = zero


def first_part(w, d, N):
    """The inputs of the problem on the first N intervals."""
    nx, nu, nun, big = w["nx"], w["nu"], synth.control_nodes(dict(w, N=N)), w["N"]
    nb = nx + synth.final_rows(w)
    out = {}
    for k in ("x", "vn"):
        v = d[k]
        U = v[nx * (big + 1):]
        out[k] = np.concatenate([v[:nx * (N + 1)], U[:nu * nun], [v[-1] * N / big] if w.get("free_tf") else []])
    for k in ("y", "vm"):
        v = d[k]
        out[k] = np.concatenate([v[:nb], v[nb:nb + nx * big].reshape(nx, big)[:, :N].reshape(-1)])
    return out


def outputs(w, d, N, T):
    """The nodes and rows below N of every output, from the fused step and from the separate calls."""
    H = ocp.OCP.from_workload(dict(w, N=d["N"], T=T))
    n = {k: torch.from_numpy(np.ascontiguousarray(d[k])).cuda() for k in ("x", "y", "vn", "vm")}
    x, y, vn, vm = (n[k] for k in ("x", "y", "vn", "vm"))
    step = H.eval_step(x, y, 0.75, vn, vm)[1:]
    parts = (H.eval_cons(x), H.eval_grad(x), H.jac_coo_values(x), H.hess_coo_values(x, y, 0.75), H.jprod(x, vn), H.jtprod(x, vm),
             H.hprod(x, y, 0.75, vn))
    L = H.value_layout()
    nx, nu, big = w["nx"], w["nu"], d["N"]
    nun = synth.control_nodes(dict(w, N=big))
    nb, tf = L["nb"], 1 if w.get("free_tf") else 0

    def rows(v):
        return [v[nb:nb + nx * big].reshape(nx, big)[:, :N]]

    def nodes(v, a=nx, b=nu, over=big + 1):
        return [v[:a * over].reshape(over, a)[:N], v[a * over:a * over + b * nun].reshape(nun, b)[:N]]

    def jac(v):
        out, at = [], nb
        for c in L["jcount"]:
            out.append(v[at:at + c * big].reshape(big, c)[:N, :c - tf])
            at += c * big
        return out

    res = []
    for call in (step, parts):
        c, g, jv, hv, Jv, Jtv, Hv = (t.cpu().numpy() for t in call)
        # (the objective has no terms of its own on Euler's last node; H has a block per node with a control)
        res += rows(c) + nodes(g) + jac(jv) + nodes(hv, L["hx"], L["hu"], nun) + rows(Jv) + nodes(Jtv) + nodes(Hv)
    H.close()
    return res


@pytest.mark.parametrize("kind", ["none", "state", "multipliers", "directions", "negative", "all"])
@pytest.mark.parametrize("name", NAMES)
def test_large_launches_have_the_bits_of_small_ones(name, kind):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    per = 40 if name == "heat_n2e4" else 60      # nodes per SM of the small problem (the heat model counts a node 8 times)
    w = dict(synth.workload(name.split(":")[0]), N=8 * per * sms)
    if name.endswith(":euler"):
        w["scheme"] = "euler"
    d = synth.draw(w)
    with_zeros(w, d, kind)
    N = w["N"] // 8
    large = outputs(w, dict(d, N=w["N"]), N, w["T"])
    small = outputs(w, dict(first_part(w, d, N), N=N), N, w["T"] / 8)
    for i, (p, q) in enumerate(zip(large, small)):
        assert p.size and np.array_equal(np.ascontiguousarray(p).view(np.int64), np.ascontiguousarray(q).view(np.int64)), i
