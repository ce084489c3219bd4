"""The rollout and reverse kernels on solver blocks against the one-warp kernels, which walk the
constraint rows one after the other: robots of one block (a ball, a lone hinge), of two bodies in
contact, of chains and trees, at sweep counts around the reverse pass's ring of three sweeps and at
batches around a group of 32 instances, with the whole tape and with recomputed segments.

States and losses: the blocks keep every body's rows in order; what may differ is the rounding of a
row of a robot without a compiled topology (2^-24 a sum, some 1e3 sums a step on one velocity over
at most 12 steps): 1e-5. Gradients: the sums over rows and sweeps are formed in another order, about
1e4 terms of either sign: 1e-4 of the gradient's norm."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1611_01652_gb300 import workloads as WL  # noqa: E402
from paper_1611_01652_gb300.binding import WS_PARAMS, World  # noqa: E402

pytestmark = pytest.mark.gpu

ROBOTS = {
    "ball": lambda B: WL.ball(B=B, horizon=60),
    "hinge": lambda B: WL.pendulum1(B=B, horizon=12),
    "spheres": lambda B: WL.two_spheres(B=B, e=0.3, mu=0.4),
    "chain": lambda B: WL.pendulum3(B=B, horizon=12),
    "arm": lambda B: WL.arm4dof(B=B, horizon=12),
    "quadruped": lambda B: WL.quadruped(B=B, horizon=12),
    "quadruped, recurrent": lambda B: WL.quadruped(B=B, horizon=12, n_recurrent=8),
}


def run(m, horizon, iters, ckpt, warm):
    w = World(m, horizon=horizon, iters=iters, ckpt_every=ckpt, warmstart=warm)
    if warm:
        w.set_warmstart(torch.zeros(WS_PARAMS, device="cuda"), 0.7)
    W = torch.tensor(m.W, device="cuda") if m.W is not None and len(m.W) else None
    loss = torch.zeros(m.B, device="cuda")
    w.rollout(W, loss)
    dW = torch.zeros(w.n_params, device="cuda") if w.n_params else None
    ds = torch.zeros(m.B, m.nb, 18, device="cuda")
    dp = {"mass": torch.zeros(m.B, m.nb, device="cuda"), "inertia": torch.zeros(m.B, m.nb, 3, device="cuda")}
    w.backward(torch.ones(m.B, device="cuda"), dW, ds, dp)
    x = w.get_state(torch.zeros(m.B, m.nb, 18, device="cuda"))
    w.sync()
    state = [t.cpu().double().numpy() for t in (loss, x)]
    return state, [t.cpu().double().numpy() for t in ([dW] if dW is not None else []) + [ds, dp["mass"], dp["inertia"]]]


@pytest.mark.parametrize("robot", sorted(ROBOTS))
@pytest.mark.parametrize("B,iters,ckpt,warm", [(1, 1, None, False), (33, 2, None, True), (40, 3, 5, True), (32, 7, 1, False)])
def test_blocks_match_rows(monkeypatch, robot, B, iters, ckpt, warm):
    m = ROBOTS[robot](B)
    m.ctrl_fp32 = 1  # (a bfloat16 rounding that falls the other way is another robot)
    T = 60 if robot == "ball" else 12  # the ball lands within its sixty steps
    got = run(m, T, iters, ckpt, warm)
    monkeypatch.setenv("DP_SINGLE_WARP_FORWARD", "1")
    monkeypatch.setenv("DP_SINGLE_WARP_BACKWARD", "1")
    ref = run(m, T, iters, ckpt, warm)
    for a, b in zip(got[0], ref[0]):
        assert (np.abs(a - b) <= 1e-5 * np.maximum(1.0, np.abs(b))).all(), np.abs(a - b).max()
    for a, b in zip(got[1], ref[1]):
        assert np.isfinite(a).all()
        assert np.linalg.norm(a - b) <= 1e-4 * max(np.linalg.norm(b), 1e-12), (a.shape, np.linalg.norm(a - b), np.linalg.norm(b))
