"""The calls a solver makes around the evaluation: the KKT values' blocks of output slots, and the
path and boundary terms' one launch, at the sizes and values where they can go wrong."""
import numpy as np
import pytest
import torch

from paper_2510_03932_gb300 import synth
from test_parity_gpu import dev, host, named, ocp  # noqa: F401  (ocp: the module fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,N", [("goddard_n1e3", 510), ("goddard_n1e3", 511), ("goddard_n1e3", 512), ("goddard_n1e3", 2500),
                                    ("vdp_n1e3", 682), ("vdp_n1e3", 683), ("quadrotor_n1e3+path+bineq+bolza", 227),
                                    ("cartpole_n1e5:euler+path", 1023), ("heat_n2e4", 33), ("dint", 1)])
def test_kkt_values_across_blocks(ocp, name, N):  # noqa: F811
    """Every slot of K = [H + diag(sigma_x + delta_w), .; J, -delta_c I], bit for bit, where the
    regions of uniform layout end inside, at and after a block of 2048 slots (the tf row's
    4 (N + 1) + 1 slots, rows of 3, 5 and 6 entries)."""
    w = named(name, N)
    d = synth.draw(w)
    H = ocp.OCP.from_workload(w)
    x, y = dev(d["x"]), dev(d["y"])
    _, _, _, jv, hv = H.eval_all(x, y, 0.5)
    sx = np.random.default_rng(3).uniform(0.0, 5.0, H.n)
    dw, dc = 0.25, 1e-3
    got = host(H.kkt_values(hv, jv, dev(sx), dw, dc))
    (jr, jc), (hr, hc), (kr, kc) = ([host(t) for t in s] for s in
                                    (H.jac_coo_structure(), H.hess_coo_structure(), H.kkt_structure()))
    diag = np.arange(H.n + H.m)
    rows = np.concatenate([hr, jr + H.n, diag])
    cols = np.concatenate([hc, jc, diag])
    vals = np.concatenate([host(hv), host(jv), sx + dw, np.full(H.m, -dc)])
    o = np.lexsort((np.arange(rows.size), cols, rows))   # (an H diagonal before its addition)
    rows, cols, vals = rows[o], cols[o], vals[o]
    first = np.concatenate([[True], (rows[1:] != rows[:-1]) | (cols[1:] != cols[:-1])])
    want = vals[first]
    dup = np.flatnonzero(~first)
    want[np.cumsum(first)[dup] - 1] = vals[dup - 1] + vals[dup]
    assert np.array_equal(rows[first], kr) and np.array_equal(cols[first], kc)
    assert np.array_equal(got, want)
    H.close()


@pytest.mark.parametrize("bad", [float("inf"), -float("inf"), float("nan"), 1e300, 0.0, -0.0])
def test_path_rows_of_unusual_values(ocp, bad):  # noqa: F811
    """Squared-only and linear-only path terms skip what their zero coefficient multiplies; the
    rows of a node with an infinite, NaN, huge or zero value still are what the whole form
    a (z - b)^2 + l z gives (0 times infinity is NaN)."""
    w = named("cartpole_n1e5+path", 300)
    d = synth.draw(w)
    H = ocp.OCP.from_workload(w)
    xh = d["x"].copy()
    for j, k in ((7, 0), (8, 2), (0, 2), (300, 0)):   # states of the ellipse's row
        xh[4 * j + k] = bad
    U0 = 4 * 301
    xh[U0 + 7] = bad                                # the control's row
    c = host(H.eval_cons(dev(xh)))
    jv = host(H.jac_coo_values(dev(xh)))
    X, U = xh[:U0].reshape(301, 4), xh[U0:U0 + 301]
    r0 = H.m - 2 * 301
    with np.errstate(all="ignore"):
        def val(a, b, l, z):
            return a * (z - b) * (z - b) + l * z
        ell = (0.0 + val(0.25, 0.0, 0.0, X[:, 0])) + val(1.0, 0.0, 0.0, X[:, 2]) - 1.0
        u2 = (0.0 + val(1.0, 0.0, 0.0, U)) - 100.0
        je = np.stack([0.5 * (X[:, 0] - 0.0) + 0.0, 2.0 * (X[:, 2] - 0.0) + 0.0], 1).ravel()
        ju = 2.0 * (U - 0.0) + 0.0
    np.testing.assert_array_equal(c[r0:r0 + 301], ell)
    np.testing.assert_array_equal(c[r0 + 301:], u2)
    np.testing.assert_array_equal(jv[-903:-301], je)
    np.testing.assert_array_equal(jv[-301:], ju)
    H.close()


@pytest.mark.parametrize("name,N", [("heat_n2e4+path+bineq+bolza", 1), ("heat_n2e4+path+bineq+bolza", 70),
                                    ("quadrotor_n1e3+path+bineq+bolza", 513), ("vdp_n1e3:euler+path+bolza", 257),
                                    ("goddard_n1e3+path+bineq+bolza", 2)])
def test_step_with_path_and_boundary_terms_equals_the_separate_calls(ocp, name, N):  # noqa: F811
    """The fused step's outputs with every kind of extra term, against the separate calls, bit for
    bit (nodes 0 and N take path and boundary additions in one order)."""
    w = named(name, N)
    d = synth.draw(w)
    H = ocp.OCP.from_workload(w)
    x, y, vn, vm = (dev(d[k]) for k in ("x", "y", "vn", "vm"))
    f, c, g, jv, hv, Jv, Jtv, Hv = H.eval_step(x, y, 0.75, vn, vm)
    for got, want in ((f, H.eval_obj(x)), (c, H.eval_cons(x)), (g, H.eval_grad(x)), (jv, H.jac_coo_values(x)),
                      (hv, H.hess_coo_values(x, y, 0.75)), (Jv, H.jprod(x, vn)), (Jtv, H.jtprod(x, vm)),
                      (Hv, H.hprod(x, y, 0.75, vn))):
        assert torch.equal(got, want)
    H.close()
