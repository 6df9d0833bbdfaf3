"""Host-side arithmetic of bench.py (no GPU)."""
import os
import sys
from unittest import mock

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

N, P, K = 512, 84, 924
NNZ = 5 * (N - 1) ** 2 - 4 * (N - 1)


@pytest.mark.parametrize("flux,kbytes,form", [
    (1, K * 2 * N * (N - 1) * 4, "edge-flux"),
    (0, K * NNZ * 4 + NNZ * 4 + ((N - 1) ** 2 + 1) * 4, "five-slot"),
])
def test_large_workload_counts_the_bytes_of_the_form_that_runs(monkeypatch, flux, kbytes, form):
    """The 512^2 apply's roofline follows the operator's form: the edge form
    reads 2.5 times fewer values than five slots."""
    import bench
    sg, torch = mock.MagicMock(), mock.MagicMock()
    prob = sg.sg_setup.return_value
    prob.n, prob.P, prob.K, prob.nnzA = (N - 1) ** 2, P, K, NNZ
    sg.sg_apply_flux.return_value = flux
    sg.sg_profile_read.return_value = (100, 100.0)                 # 1 ms a launch
    info = {"outer_it": 30, "relres": 1e-9, "fallback_used": 0}
    sg.sg_train_precond.return_value = {"t_train": 1.0, "loss_last": 0.3}
    monkeypatch.setattr(bench, "ev_time", lambda *a: (100.0, info))
    monkeypatch.setattr(bench, "peaks", lambda: (6772.2, "measured"))
    roof = bench.large_workload(sg, torch, None)["roofline"]
    assert roof["bytes_per_launch"] == kbytes + 2 * (N - 1) ** 2 * P * 4
    assert form in roof["kernel"]
    assert roof["achieved"] == round(roof["bytes_per_launch"] / 1e6, 1)
