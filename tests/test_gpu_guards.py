"""Sums whose ends are easy to miss: what lies around a texture gradient is not even added a zero to, and
the warm-start network's gradient of a few rows against the oracle's; recomputed segments of robots
without a compiled topology give the whole tape's bits with a tensor-core controller too."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1611_01652_gb300 import binding as Bd  # noqa: E402
from paper_1611_01652_gb300 import workloads as WL  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tex_size,W,H", [(1, 32, 16), (3, 144, 48), (5, 288, 96), (64, 64, 38)])
def test_texture_gradient_leaves_its_surroundings(tex_size, W, H):
    """The 16-byte reductions add zeros around the texels they are for: negative zeros next to the buffer
    would turn positive."""
    cs = WL.camera_scene(B=6, W=W, H=H, tex_size=tex_size, mixed=True)
    rig = Bd.CameraRig(cs)
    st = torch.tensor(np.asarray(cs.states, np.float32), device="cuda")
    tex = torch.tensor(np.asarray(cs.textures, np.float32), device="cuda")
    dimg = torch.randn(6, H, W, 3, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    for shift in (4, 5):
        buf = torch.full((tex.numel() + 32,), -0.0, device="cuda")
        rig.render_backward(st, tex, dimg, torch.zeros_like(st), buf[shift:shift + tex.numel()].view(tex.shape))
        torch.cuda.synchronize()
        around = torch.cat([buf[:shift], buf[shift + tex.numel():]])
        assert torch.signbit(around).all() and (around == 0).all()


@pytest.mark.parametrize("n", [1, 2, 33, 257])
def test_weight_gradient_of_few_rows_matches_oracle(n):
    """Bounds as for larger row counts in test_gpu_warmstart: bfloat16 storage points that fall the other
    way on few of the units."""
    rng = np.random.default_rng(n)
    rows = rng.normal(size=(n, Bd.WS_ROW)).astype(np.float32)
    W = WL.xavier_weights([16, 64, 64, 3], 0, rng)
    L_o, g_o = O.ws_loss_grad(W, rows)
    loss, dW = torch.zeros(1, device="cuda"), torch.zeros(Bd.WS_PARAMS, device="cuda")
    Bd.ws_loss_grad(torch.tensor(W, device="cuda"), torch.tensor(rows, device="cuda"), loss, dW, Bd.ws_workspace(n))
    torch.cuda.synchronize()
    assert abs(loss.item() - L_o) <= 1e-3 * abs(L_o)
    d = dW.cpu().double().numpy() - g_o
    assert np.linalg.norm(d) <= 1e-2 * np.linalg.norm(g_o)


@pytest.mark.parametrize("robot", ["arm", "quadruped"])
def test_segments_give_the_tapes_bits(monkeypatch, robot):
    monkeypatch.setenv("DP_FORCE_RUNTIME_TOPOLOGY", "1")
    m = WL.arm4dof(B=33, horizon=40) if robot == "arm" else WL.quadruped(B=33, horizon=40, iters=5)
    if robot == "arm":  # (its output layer starts at zero)
        m.W = WL.xavier_weights(m.widths, 0, np.random.default_rng(1))
    out = []
    for ckpt in (None, 16):
        w = Bd.World(m, horizon=40, iters=5, ckpt_every=ckpt, warmstart=True)
        w.set_warmstart(torch.zeros(Bd.WS_PARAMS, device="cuda"), 0.7)
        assert w.controller_kind == 2  # tensor cores in the step
        w.rollout(torch.tensor(m.W, device="cuda"), torch.zeros(m.B, device="cuda"))
        dW, ds = torch.zeros(w.n_params, device="cuda"), torch.zeros(m.B, m.nb, 18, device="cuda")
        w.backward(torch.ones(m.B, device="cuda"), dW, ds)
        w.sync()
        assert torch.isfinite(dW).all() and dW.norm() > 0
        out.append((dW, ds))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
