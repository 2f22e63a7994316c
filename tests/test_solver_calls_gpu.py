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
