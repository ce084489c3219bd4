"""Solver blocks on forms that the bundled robots do not have: the wide controller's per-step reverse
launches without a compiled topology. Against the one-warp kernels, bounds as in test_gpu_blocks."""
import numpy as np
import pytest

pytest.importorskip("torch")

from paper_1611_01652_gb300 import workloads as WL  # noqa: E402

from test_gpu_blocks import run  # noqa: E402

pytestmark = pytest.mark.gpu


def same_gradients(got, ref):
    for a, b in zip(got[1], ref[1]):
        assert np.isfinite(a).all()
        assert np.linalg.norm(a - b) <= 1e-4 * max(np.linalg.norm(b), 1e-12), (a.shape, np.linalg.norm(a - b), np.linalg.norm(b))


def test_wide_controller_on_a_run_time_topology(monkeypatch):
    m = WL.quadruped(B=33, horizon=6, widths=[64, 320, 320, 8])
    monkeypatch.setenv("DP_FORCE_RUNTIME_TOPOLOGY", "1")
    got = run(m, 6, 5, None, True)
    monkeypatch.setenv("DP_SINGLE_WARP_BACKWARD", "1")
    same_gradients(got, run(m, 6, 5, None, True))
