"""Solver blocks on forms that the bundled robots do not have: blocks of a part of an item's rows, ball
joints, more than 32 blocks, robots past the schedule's limits or whose reverse pass does not fit, bodies
that do touch, and the wide controller without a compiled topology. Against the one-warp kernels, which
walk the constraint rows one after the other; bounds as in test_gpu_blocks (states 2^-24 a sum, some 1e3
sums a step over a few dozen steps: 1e-5; gradients some 1e4 terms of either sign: 1e-4 of the norm)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1611_01652_gb300 import workloads as WL  # noqa: E402
from paper_1611_01652_gb300.binding import PARAM_GRADS, WS_PARAMS, World  # noqa: E402

pytestmark = pytest.mark.gpu

BALL, HINGE, BOTH = WL.BALL, WL.HINGE, WL.FLAG_LIMIT | WL.FLAG_MOTOR
JLIN, JANG, LIMIT, MOTOR, GN, GT, PN, PT = range(8)  # slot kinds of World.schedule()


def robot(B, pos, joints, spheres, pairs=(), ground_z=0.0, speed=0.2, seed=3):
    """Bodies at ``pos`` (no rotation, random speeds), joints (type, parent, child, pivot, axis, flags),
    spheres (body, offset, radius), pairs of spheres. Limits are active at the start (the lower bound lies
    above the angle), servos hold zero."""
    rng = np.random.default_rng(seed)
    pos = np.asarray(pos, float)
    nb, nj, ns = len(pos), len(joints), len(spheres)
    d = WL._empty(B, nb, nj, ns)
    d["mass"][:] = rng.uniform(0.8, 1.2, size=(B, nb))
    d["inertia"][:] = rng.uniform(0.01, 0.02, size=(B, nb, 3))
    for i in range(B):
        for b in range(nb):
            v, w = rng.uniform(-speed, speed, size=(2, 3))
            d["state0"][i, b] = WL._state(pos[b], np.eye(3), v, w)
    for j, (_, a, b, pivot, axis, _) in enumerate(joints):
        pivot = np.asarray(pivot, float)
        d["anchor"][:, j, 0] = pivot - (pos[a] if a >= 0 else 0.0)
        d["anchor"][:, j, 1] = pivot - pos[b]
        d["axis"][:, j, :] = axis
        d["ref"][:, j, :] = np.roll(axis, 1)
    d["limit"][:] = [0.01, 1.0]
    d["motor"][:] = [10.0, 1.0, 2.0]
    for q, (_, off, rad) in enumerate(spheres):
        d["sph_off"][:, q] = off
        d["sph_rad"][:, q] = rad
    d["sph_mu"][:] = rng.uniform(0.3, 0.5, size=(B, ns))
    d["sph_e"][:] = 0.2
    d["loss_target"][:] = rng.uniform(-1, 1, size=(B, 3))
    WL._finish(d)
    return WL.Model(name="test", B=B, joint_type=np.array([j[0] for j in joints], np.int32),
                    joint_body=np.array([j[1:3] for j in joints], np.int32).reshape(nj, 2),
                    joint_flags=np.array([j[5] for j in joints], np.int32),
                    sphere_body=np.array([s[0] for s in spheres], np.int32),
                    pair_sphere=np.array(pairs, np.int32).reshape(len(pairs), 2), nb=nb, dt=0.002, iters=5, horizon=12,
                    ground_z=ground_z, loss_kind=WL.L_SQDIST, loss_mode=WL.M_MEAN, loss_body=nb - 1, **d)


def pile(B):
    """Three balls in a row on the ground, each touching the next: two pairs that share a sphere."""
    r, x = [0.1, 0.12, 0.09], [0.0]
    for a, b in zip(r, r[1:]):
        x.append(x[-1] + np.sqrt((a + b) ** 2 - (a - b) ** 2) - 0.004)
    return robot(B, [[x[k], 0.0, r[k] - 0.002] for k in range(3)], [], [(k, [0, 0, 0], r[k]) for k in range(3)], [(0, 1), (1, 2)])


def hub(B, n=7):
    """A ball on the ground and n smaller ones around it that touch it: n pairs share its sphere."""
    R, r = 0.3, 0.1
    u = np.sqrt((R + r) ** 2 - (R - r) ** 2) - 0.003
    ang = 0.1 + 2 * np.pi * np.arange(n) / n
    pos = [[0.0, 0.0, R - 0.002]] + [[u * np.cos(a), u * np.sin(a), r - 0.002] for a in ang]
    return robot(B, pos, [], [(0, [0, 0, 0], R)] + [(k + 1, [0, 0, 0], r) for k in range(n)], [(0, k + 1) for k in range(n)])


def mixed_chain(B):
    """A ball joint, then two hinges with limits and servos, two contacts on the last link: the second
    hinge's linear and angular rows fall apart, and so does the second contact."""
    return robot(B, [[0, 0, -0.2], [0, 0, -0.6], [0, 0, -1.0]],
                 [(BALL, -1, 0, [0, 0, 0], [0, 1, 0], 0), (HINGE, 0, 1, [0, 0, -0.4], [0, 1, 0], BOTH),
                  (HINGE, 1, 2, [0, 0, -0.8], [1, 0, 0], BOTH)],
                 [(2, [0.05, 0, -0.2], 0.05), (2, [-0.05, 0, -0.2], 0.05)], ground_z=-1.248)


def split_pair(B):
    """A hinge to the world and a ball joint leave a hole in one body's colours that takes a pair's normal
    and first friction row; the other falls behind a contact."""
    u = np.sqrt(0.22 ** 2 - 0.02 ** 2) - 0.003
    return robot(B, [[0, 0, 0.3], [0.4, 0, 0.3], [0.4 + u, 0, 0.12]],
                 [(HINGE, -1, 0, [0, 0, 0.5], [0, 1, 0], 0), (BALL, 1, 0, [0.2, 0, 0.3], [0, 1, 0], 0)],
                 [(2, [0, 0, 0], 0.12), (1, [0, 0, -0.2], 0.1), (0, [0, 0, -0.2], 0.1)], [(1, 0)], ground_z=0.002)


def plates(B):
    """Two plates of sixteen contact spheres each, a ball joint and a hinge with limit and servo: 36 blocks."""
    grid = [[0.05 * (k % 4), 0.05 * (k // 4), -0.45] for k in range(16)]
    return robot(B, [[0, 0, 0.5], [0.6, 0, 0.5]],
                 [(BALL, -1, 0, [0, 0, 0.9], [0, 1, 0], 0), (HINGE, 0, 1, [0.3, 0, 0.5], [0, 1, 0], BOTH)],
                 [(b, o, 0.05) for b in range(2) for o in grid], ground_z=0.002)


def one_plate(B):
    """A body on a hinge with 32 contacts: 35 levels, more than the schedule holds (one warp)."""
    grid = [[0.05 * (k % 8), 0.05 * (k // 8), -0.45] for k in range(32)]
    return robot(B, [[0, 0, 0.5]], [(HINGE, -1, 0, [0, 0, 0.9], [0, 1, 0], BOTH)], [(0, o, 0.05) for o in grid], ground_z=0.002)


def ball_chain(B):
    """Thirteen links on ball joints and a contact: the rollout fits on blocks, the reverse pass does not."""
    return robot(B, [[0, 0, -0.1 - 0.2 * k] for k in range(13)],
                 [(BALL, k - 1, k, [0, 0, -0.2 * k], [0, 1, 0], 0) for k in range(13)], [(12, [0, 0, -0.1], 0.05)], ground_z=-2.648)


# robot, blocks of its schedule, items that are split (type, index)
JOINT, CONTACT, PAIR = "joint", "contact", "pair"
ROBOTS = {
    "mixed chain": (mixed_chain, 11, {(JOINT, 2), (CONTACT, 1)}),
    "split pair": (split_pair, 7, {(PAIR, 0)}),
    "plates": (plates, 36, set()),
    "one plate": (one_plate, 35, set()),
    "ball chain": (ball_chain, 14, set()),
    "pile": (pile, 5, set()),
    "hub": (hub, 15, set()),
}


def blocks(w):
    """The schedule's blocks: a row joins its item's block when that is the last one on each of its
    bodies. Returns their number and the items in more than one block."""
    s = w.schedule()
    item = {JLIN: JOINT, JANG: JOINT, LIMIT: LIMIT, MOTOR: MOTOR, GN: CONTACT, GT: CONTACT, PN: PAIR, PT: PAIR}
    last, made = {}, []
    for o in s["order"]:
        it = (item[s["kind"][o]], int(s["idx"][o]))
        bodies = [x for x in (s["body_a"][o], s["body_b"][o]) if x >= 0]
        on = {last.get(x) for x in bodies}
        if len(on) == 1 and None not in on and made[list(on)[0]] == it and it[0] not in (LIMIT, MOTOR):
            continue
        made.append(it)
        for x in bodies:
            last[x] = len(made) - 1
    return len(made), {it for it in made if made.count(it) > 1}


def solve(m, horizon, iters, ckpt, warm, net=None, **kw):
    """(loss, final state), every gradient, the activity log and the schedule."""
    w = World(m, horizon=horizon, iters=iters, ckpt_every=ckpt, warmstart=warm, **kw)
    if warm:
        w.set_warmstart(torch.zeros(WS_PARAMS, device="cuda") if net is None else net, 0.7)
    W = torch.tensor(m.W, device="cuda") if m.W is not None and len(m.W) else None
    loss = torch.zeros(m.B, device="cuda")
    act = torch.zeros(horizon, m.B, w.n_slots, dtype=torch.uint8, device="cuda")
    w.rollout(W, loss, None, act)
    dW = torch.zeros(w.n_params, device="cuda") if w.n_params else None
    ds = torch.zeros(m.B, m.nb, 18, device="cuda")
    dp = {k: torch.zeros(getattr(m, k).shape, device="cuda") for k in PARAM_GRADS if getattr(m, k).size}
    w.backward(torch.ones(m.B, device="cuda"), dW, ds, dp)
    x = w.get_state(torch.zeros(m.B, m.nb, 18, device="cuda"))
    w.sync()
    grads = dict(dp, state0=ds, **({"W": dW} if dW is not None else {}))
    return [t.cpu().double().numpy() for t in (loss, x)], {k: t.cpu().numpy() for k, t in grads.items()}, act.cpu().numpy(), w


def same(got, ref):
    for a, b in zip(got[0], ref[0]):
        assert (np.abs(a - b) <= 1e-5 * np.maximum(1.0, np.abs(b))).all(), np.abs(a - b).max()
    for k in ref[1]:
        a, b = got[1][k].astype(np.float64), ref[1][k].astype(np.float64)
        assert np.isfinite(a).all(), k
        assert np.linalg.norm(a - b) <= 1e-4 * max(np.linalg.norm(b), 1e-12), (k, np.linalg.norm(a - b), np.linalg.norm(b))


def one_warp(monkeypatch):
    monkeypatch.setenv("DP_SINGLE_WARP_FORWARD", "1")
    monkeypatch.setenv("DP_SINGLE_WARP_BACKWARD", "1")


def test_wide_controller_on_a_run_time_topology(monkeypatch):
    m = WL.quadruped(B=33, horizon=6, widths=[64, 320, 320, 8])
    monkeypatch.setenv("DP_FORCE_RUNTIME_TOPOLOGY", "1")
    got = solve(m, 6, 5, None, True)
    monkeypatch.setenv("DP_SINGLE_WARP_BACKWARD", "1")
    same(got, solve(m, 6, 5, None, True))


def test_gradients_of_touching_spheres_repeat_bit_for_bit():
    """Ground contacts and pairs add to the parameters of the same spheres: always in the same order."""
    m = hub(64)
    _, first, act, w = solve(m, 12, 5, None, True)
    kind = w.schedule()["kind"]
    assert act[:, :, kind == GN].any() and act[:, :, kind == PN].any()
    for _ in range(8):
        again = solve(m, 12, 5, None, True)[1]
        for k in first:
            assert np.array_equal(first[k], again[k]), k


@pytest.mark.parametrize("name", sorted(ROBOTS))
@pytest.mark.parametrize("B,iters,ckpt,warm", [(1, 1, 1, False), (33, 3, None, True), (40, 5, 5, True), (32, 7, None, False)])
def test_general_robots_match_rows(monkeypatch, name, B, iters, ckpt, warm):
    make, n, split = ROBOTS[name]
    m = make(B)
    got = solve(m, 12, iters, ckpt, warm)
    assert blocks(got[3]) == (n, split)
    kind = got[3].schedule()["kind"]
    for k in (LIMIT, GN, PN):  # every kind of row that comes and goes was there
        assert not (kind == k).any() or got[2][:, :, kind == k].any(), k
    one_warp(monkeypatch)
    same(got, solve(m, 12, iters, ckpt, warm))


def test_colliding_spheres_match_rows(monkeypatch):
    """Two spheres in free flight that meet within sixty steps."""
    m = WL.two_spheres(B=40, e=0.3, mu=0.4)
    got = solve(m, 60, 5, 16, True)
    assert got[2][:, :, got[3].schedule()["kind"] == PN].any()
    one_warp(monkeypatch)
    same(got, solve(m, 60, 5, 16, True))


def test_many_balls_record_on_one_warp():
    """At seven groups an SM and above, recorded rollouts of robots without joints take one warp a group,
    their reverse pass blocks: against the one-warp kernels."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    few = WL.ball(B=64, horizon=20)
    m = few.subset(np.arange(32 * (7 * sms + 1) - 5) % few.B)
    m.state0[:, :, 14] = np.where(np.arange(m.B) % 3 == 0, -1.0, m.state0[:, 0, 14])[:, None]  # a third hits the ground at once
    got = solve(m, 20, 3, None, True)
    assert got[2].any()
    same(got, solve(m, 20, 3, None, True, one_warp=True))


@pytest.mark.parametrize("name", sorted(ROBOTS))
def test_learned_start_matches_rows(monkeypatch, name):
    """A warm-start network that is not zero, two steps (a bfloat16 rounding of its features or hidden units
    that falls the other way shows later)."""
    net = torch.tensor(0.05 * WL.xavier_weights([16, 64, 64, 3], 0, np.random.default_rng(2)), device="cuda")
    m = ROBOTS[name][0](33)
    got = solve(m, 2, 3, None, True, net)
    one_warp(monkeypatch)
    same(got, solve(m, 2, 3, None, True, net))
