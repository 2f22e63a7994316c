"""The heat objective's sum over tiles in CTAs of one, two, four and eight warps, at tile counts around the
places that it is summed in (256 and their multiples)."""
import pytest
import torch

from paper_2510_03932_gb300 import ocp, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tiles", [1, 255, 256, 257, 761, 1024, 1025, 2047, 2050, 3100])
@pytest.mark.parametrize("cells", [2, 8, 12, 30, 40])
def test_objective_against_a_plain_sum(cells, tiles):
    q, xref, r = [0.5 + 0.01 * k for k in range(cells)], [0.3] * cells, 0.02
    w = dict(synth.workload("heat_n2e4"), nx=cells, params=[float(cells)], q=q, xref=xref, r=[r], x0=[0.0] * cells, N=31 * tiles - 1)
    H = ocp.OCP.from_workload(w)
    N, g = w["N"], torch.Generator(device="cuda").manual_seed(tiles + cells)
    x = torch.rand(H.n, generator=g, device="cuda", dtype=torch.float64)
    X, U = x[:cells * (N + 1)].view(N + 1, cells), x[cells * (N + 1):]
    per = ((X - 0.3) ** 2 * torch.tensor(q, device="cuda", dtype=torch.float64)).sum(1) + r * U * U
    per[0] *= 0.5
    per[-1] *= 0.5
    want = (per.sum() * (w["T"] / N)).item()
    # terms of one sign: every rounding is within 2^-53 of the sum; at most 40 + 30 of them lie on a term's way
    # (its cells and tile, 13 tiles a place, the places), and fewer than a thousand on the plain sum's
    f = H.eval_obj(x)
    assert abs(f.item() - want) <= 1100 * 2.0 ** -53 * want
    assert torch.equal(f, H.eval_obj(x))
    assert torch.equal(f, H.eval_all(x, None, 0.5, torch.empty_like(f), torch.empty(H.m, device="cuda", dtype=torch.float64),
                                     alloc=False)[0])
    H.close()
