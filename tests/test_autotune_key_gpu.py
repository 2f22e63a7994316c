"""The autotuning cache: a configuration that was stored by a library with other kernels is not taken."""
import re

import pytest
import torch

from paper_2510_03932_gb300 import build, ocp, synth

pytestmark = pytest.mark.gpu


def test_lines_of_other_kernels_are_ignored(tmp_path, monkeypatch):
    path = tmp_path / "tune.txt"
    monkeypatch.setenv("OCP_AUTOTUNE_CACHE", str(path))
    B = ocp.OCPBatch([ocp.OCP.from_workload(synth.with_horizon(synth.workload("cartpole_n1e5"), n)) for n in (700, 1500)])
    x, y = (torch.ones(k, device="cuda", dtype=torch.float64) for k in (B.n, B.m))
    outs = B.outputs()
    B.autotune(x, y, 1.0, *outs)
    (line,) = path.read_text().splitlines()
    assert "kernels=" + build.kernels_tag() in line
    key = line.split("\t")[0]
    # the same shape under another tag, and as a line without one: with a time that no batch has
    for other in (re.sub(r"kernels=\S+", "kernels=0123456789ab", key), re.sub(r" kernels=\S+", "", key)):
        path.write_text(other + "\t64 2 1 12345.0\n")
        assert B.autotune(x, y, 1.0, *outs) < 1000.0
        assert len(path.read_text().splitlines()) == 2
    path.write_text(key + "\t64 2 1 12345.0\n")   # and its own line is
    assert B.autotune(x, y, 1.0, *outs) == 12345.0
    assert B.get_config() == dict(nodes_per_thread=2, threads=64, ctas_per_sm=1)
