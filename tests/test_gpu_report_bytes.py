"""Bytes that kernel_report gives for a sweep: a Schwarz sweep applies the whole operator once, so with
and without the finest level's zero pattern it differs by what the operator application differs by."""
import dataclasses

import pytest

torch = pytest.importorskip("torch")

import paper_2512_08728_gb300 as pkg
from workloads import make_problem

pytestmark = pytest.mark.gpu


def test_schwarz_sweep_counts_the_stored_entries():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()
    pr = make_problem(3, 2, (16, 16, 8), 3, nu_kind="jump", seed=1)
    dense = pr.blocks.copy()
    dense[0, 0, 1, 2] = 1e-9                     # modes x and y: zero in a tensor basis
    rep = []
    for blocks in (pr.blocks, dense):
        s = pkg.KCycleSolver(dataclasses.replace(pr, blocks=blocks), smoother="as", omega=0.5, sweeps=2)
        rep.append(s.kernel_report(reps=1))
        s.close()
    pattern, full = rep
    saved = full["spmv_bytes"] - pattern["spmv_bytes"]
    assert saved > 0.6 * full["spmv_bytes"]
    assert full["sweep_bytes"] - pattern["sweep_bytes"] == pytest.approx(saved, rel=1e-12)
