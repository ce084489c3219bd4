"""The reverse pass of the compiled topologies forms every sum row by row in slot order, whatever the
schedule: the initial state's adjoint of quadrupeds whose gradients amplify a rounding (bfloat16
controller, damped warm start, 100 steps) against stored values of a sequential walk over the rows,
and recomputed segments against the whole tape.

Tolerance: the same sums in the same order, so the same bits; 1e-6 of the norm leaves a few last bits
(2^-24 = 6e-8 each) to the conversion of the seeded inputs. Another order of sums is 2.1e-4 (recurrent)
and 1.7e-4 (feed-forward) away on these robots."""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1611_01652_gb300 import workloads as WL  # noqa: E402
from paper_1611_01652_gb300.binding import WS_PARAMS, World  # noqa: E402

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "quadruped_reverse.npz")
CASES = {"recurrent": (50, 8), "feed_forward": (71, 0)}  # seed, recurrent state


def reverse(name, ckpt=None):
    seed, rec = CASES[name]
    m = WL.quadruped(B=32, seed=seed, horizon=100, iters=14, n_recurrent=rec)
    w = World(m, horizon=100, iters=14, ckpt_every=ckpt, warmstart=True)
    w.set_warmstart(torch.zeros(WS_PARAMS, device="cuda"), 0.7)
    w.rollout(torch.tensor(m.W, device="cuda"), torch.zeros(m.B, device="cuda"))
    dW = torch.zeros(w.n_params, device="cuda")
    ds = torch.zeros(m.B, m.nb, 18, device="cuda")
    w.backward(torch.full((m.B,), 1.0 / m.B, device="cuda"), dW, ds)
    w.sync()
    return ds, dW


@pytest.mark.parametrize("name", sorted(CASES))
def test_state_adjoint_is_the_sequential_walks(name):
    ds, _ = reverse(name)
    ref = np.load(GOLDEN)[name].astype(np.float64)
    assert np.linalg.norm(ds.cpu().double().numpy() - ref) <= 1e-6 * np.linalg.norm(ref)


@pytest.mark.parametrize("name", sorted(CASES))
def test_segments_give_the_tapes_bits(name):
    a, b = reverse(name), reverse(name, ckpt=16)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
