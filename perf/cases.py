"""Performance cases: what programs do with this package, through its public entry points.

One case is a dict of plain values. `kind` names the call and the other values give its size:

  round      one IRLS round of the epipolar adjustment (`refine`), streaming iterations
  quadratic  the same round on the pre-aggregated quadratic form
  learned    rounds with the network's reweighting (`refine_learned`), streaming or quadratic
  autograd   `epipolar_loss` forward and backward, for poses that a torch program optimises
  create     a new scene: `Problem` from device arrays, the L1 loss with its gradient, residuals
  train      minibatch steps of the inlier-weight network
  rotation   the global rotation stage: initialisation and refinement steps
  translation  the global translation stage: several runs advanced together, then their losses
  vote       the focal-length vote over candidate focal lengths

Inputs are synthetic scenes made on the GPU from the seed: cameras on a closed path that winds
around a point cloud and looks inward, image pairs of neighbouring views, matches of random points
of the cloud with pixel noise and a share of uniform random wrong matches, heavy-tailed match
counts, and initial poses that are a few degrees off.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import learned

F = 500.0                      # focal length in pixels of a 640 x 480 image
HALF_W, HALF_H = 0.64, 0.48    # half the image in normalised coordinates
CHUNK = 1 << 24                # point pairs handled at once while inputs are made or checked
ON_CHIP = 100e6                # bytes that the GPU's L2 keeps from one iteration to the next


def listed():
    return [
        # the smallest adjustment: 16 views on a ring, every pair matched; launches and latency count
        dict(name="ring16_round", kind="round", cams=16, near=15, points=119064, tail="flat", storage="fp32",
             iters=25, outliers=0.10, sigma_px=0.5),
        # an object-centred capture of 128 views with their 16 nearest views, plain FP32
        dict(name="sphere128_round", kind="round", cams=128, near=16, points=3131047, tail="lognormal",
             storage="fp32", iters=25, outliers=0.15, sigma_px=1.0),
        # the largest adjustment: 4,000 views, heavy-tailed match counts, FP16 keypoints
        dict(name="traj4000_round", kind="round", cams=4000, near=20, points=140559465, tail="pareto",
             storage="fp16", iters=25, outliers=0.25, sigma_px=1.5),
        # 1,000 views iterating on the quadratic form, the cheapest kind of round
        dict(name="loop1000_quadratic", kind="quadratic", cams=1000, near=20, points=48865055, tail="lognormal",
             storage="fp16", iters=25, outliers=0.20, sigma_px=1.0),
        # the network's reweighting on a long capture: first round without a history, second with one
        dict(name="loop1000_learned", kind="learned", cams=1000, near=20, points=48865055, tail="lognormal",
             storage="fp16", iters=25, outliers=0.30, sigma_px=1.0, quadratic=False),
        # the network's reweighting at the size it was trained on, with quadratic-form iterations
        dict(name="sphere128_learned", kind="learned", cams=128, near=16, points=3131047, tail="lognormal",
             storage="fp32", iters=25, outliers=0.30, sigma_px=1.0, quadratic=True),
        # the objective inside a torch program: one forward and backward over 1,000 views
        dict(name="traj1000_autograd", kind="autograd", cams=1000, near=20, points=48865055, tail="lognormal",
             storage="fp16", outliers=0.20, sigma_px=1.0, recompute=False),
        # a new scene whose matches come in any order, and what a program first asks of it
        dict(name="sphere128_create", kind="create", cams=128, near=16, points=3131047, tail="lognormal",
             storage="fp16", outliers=0.15, sigma_px=1.0, shuffled=True),
        # training of the inlier-weight network: minibatches of the shipped training run
        dict(name="mlp_train", kind="train", batch=16384, steps=8),
        # global rotations of 1,000 views from noisy relative rotations
        dict(name="loop1000_rotation", kind="rotation", cams=1000, near=20, steps=100, noise_deg=1.0),
        # global positions of 1,000 views: eight random starts advanced together
        dict(name="loop1000_translation", kind="translation", cams=1000, near=20, runs=8, steps=100, noise_deg=1.0),
        # one focal length for a capture of 1,000 views
        dict(name="loop1000_vote", kind="vote", pairs=11669, candidates=256, known=0.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["round", "round", "quadratic", "learned", "autograd", "create", "train", "rotation",
                       "translation", "vote"])
    if kind == "train":
        return dict(kind=kind, batch=_log_int(rng, 200, 65536), steps=rng.randint(1, 8))
    if kind == "vote":
        return dict(kind=kind, pairs=_log_int(rng, 1, 47903), candidates=_log_int(rng, 1, 256),
                    known=rng.choice([0.0, 0.3]))
    cams = _log_int(rng, 8, 2000)
    near = min(rng.randint(4, 24), cams - 1)
    if kind in ("rotation", "translation"):
        c = dict(kind=kind, cams=cams, near=near, steps=rng.randint(5, 100), noise_deg=rng.uniform(0.2, 2.0))
        if kind == "translation":
            c["runs"] = rng.randint(1, 8)
        return c
    points = cams * near * _log_int(rng, 20, 4000) // 2 + rng.randint(0, 999)
    c = dict(kind=kind, cams=cams, near=near, points=points, tail=rng.choice(["flat", "lognormal", "pareto"]),
             storage=rng.choice(["fp32", "fp16"]), outliers=rng.choice([0.1, 0.2, 0.3]), sigma_px=rng.choice([0.5, 1.0, 1.5]))
    if kind in ("round", "quadratic", "learned"):
        c["iters"] = rng.choice([10, 25, 50])
    if kind == "learned":
        c["quadratic"] = rng.random() < 0.5
    if kind == "autograd":
        c["recompute"] = rng.random() < 0.3
    if kind == "create":
        c["shuffled"] = rng.random() < 0.5
    return c


# ---- inputs ------------------------------------------------------------------------------------
def _hat(v):
    z = torch.zeros_like(v[..., 0])
    return torch.stack([torch.stack([z, -v[..., 2], v[..., 1]], -1), torch.stack([v[..., 2], z, -v[..., 0]], -1),
                        torch.stack([-v[..., 1], v[..., 0], z], -1)], -2)


def _unit(n, g):
    v = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
    return v / v.norm(dim=-1, keepdim=True)


def _turn(n, degrees, g):
    return torch.linalg.matrix_exp(_hat(_unit(n, g) * (math.radians(degrees))))


def _cameras(case, g):
    """True rotations and centres, and the image pairs of neighbouring views (i < j)."""
    n, near = case["cams"], case["near"]
    s = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) / n
    laps = max(1, n // 50)
    elev = math.radians(70.0) * torch.cos(2 * math.pi * s) * (1.0 if n > 32 else 0.0)
    theta = 2 * math.pi * laps * s
    C = torch.stack([torch.cos(elev) * torch.cos(theta), torch.cos(elev) * torch.sin(theta), torch.sin(elev)], -1)
    C = 3.0 * C * (1 + 0.05 * torch.randn(n, 1, generator=g, device="cuda", dtype=torch.float64))
    z = -C / C.norm(dim=-1, keepdim=True)
    y = torch.tensor([0.0, 0.0, -1.0], device="cuda", dtype=torch.float64) + z * z[:, 2:3]
    y = y / y.norm(dim=-1, keepdim=True)
    R = _turn(n, 5.0, g) @ torch.stack([torch.linalg.cross(y, z), y, z], 1)
    d = torch.cdist(C, C)
    d.fill_diagonal_(float("inf"))
    k = torch.arange(n, device="cuda")
    nn = torch.topk(d, near, dim=1, largest=False).indices
    a = torch.cat([k[:, None].expand_as(nn).reshape(-1), k[:-1]])    # and every view with the next one
    b = torch.cat([nn.reshape(-1), k[1:]])
    key = torch.unique(torch.minimum(a, b) * n + torch.maximum(a, b))
    return R, C, key // n, key % n


def _scene(case, g):
    """Cameras, pairs, and matches in normalised coordinates, in pair order."""
    R, C, i, j = _cameras(case, g)
    B, P = i.numel(), max(case["points"], i.numel())
    if case["tail"] == "flat":
        x = torch.ones(B, device="cuda", dtype=torch.float64)
    elif case["tail"] == "lognormal":
        x = torch.exp(0.9 * torch.randn(B, generator=g, device="cuda", dtype=torch.float64))
    else:
        x = torch.rand(B, generator=g, device="cuda", dtype=torch.float64).clamp_min(0.003) ** (-1 / 1.5)
    counts = 1 + torch.floor((P - B) * (x / x.sum())).to(torch.int64)
    counts[torch.argmax(counts)] += P - int(counts.sum())
    pid = torch.repeat_interleave(torch.arange(B, device="cuda", dtype=torch.int32), counts)
    x1 = torch.empty(P, 2, device="cuda")
    x2 = torch.empty(P, 2, device="cuda")
    score = torch.empty(P, device="cuda")
    Rf, Cf = R.float(), C.float()
    sigma = case["sigma_px"] / F
    for p in range(0, P, CHUNK):
        q = slice(p, min(P, p + CHUNK))
        m = pid[q].numel()
        X = torch.randn(m, 3, generator=g, device="cuda")
        X *= torch.rand(m, 1, generator=g, device="cuda") ** (1 / 3) / X.norm(dim=1, keepdim=True)
        for cam, out in ((i, x1), (j, x2)):
            c = cam[pid[q].long()]
            Y = (Rf[c] @ (X - Cf[c])[:, :, None])[:, :, 0]
            out[q] = Y[:, :2] / Y[:, 2:] + sigma * torch.randn(m, 2, generator=g, device="cuda")
        wrong = torch.rand(m, generator=g, device="cuda") < case["outliers"]
        rnd = (2 * torch.rand(m, 2, generator=g, device="cuda") - 1) * torch.tensor([HALF_W, HALF_H], device="cuda")
        x2[q] = torch.where(wrong[:, None], rnd, x2[q])
        u = torch.rand(m, generator=g, device="cuda")
        score[q] = torch.where(wrong, 0.8 * u, 0.3 + 0.7 * u)
    base = (C[i] - C[j]).norm(dim=1).median()
    R0 = _turn(R.shape[0], 3.0, g) @ R
    C0 = C + 0.1 * base * _unit(R.shape[0], g)
    return dict(R=R0, C=C0, i=i, j=j, pid=pid, x1=x1, x2=x2, score=score, base=float(base), sigma=sigma)


def _schedule(case, sc, rounds=1):
    return fm.Schedule(rounds=rounds, iters_per_round=case["iters"], tau0=0.1, tau_min=4 * sc["sigma"], tau_factor=0.8,
                       decay=0.985, lr_rot=3e-3, lr_c=1e-2 * sc["base"], delta=sc["sigma"], beta2=0.99)


def _translations(R, C):
    return -(R @ C[:, :, None])[:, :, 0]


def _problem(case, sc, options):
    return fm.Problem(sc["R"], _translations(sc["R"], sc["C"]), sc["i"], sc["j"], sc["pid"], sc["x1"], sc["x2"],
                      options=options)


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _moved(sc, g):
    """Poses a little off the initial ones, as an optimiser's next evaluation has them."""
    n = sc["R"].shape[0]
    return _turn(n, 0.2, g) @ sc["R"], sc["C"] + 0.01 * sc["base"] * _unit(n, g)


def _batches(case, g):
    """Features as the network sees them (log residuals, score, pair statistics) and inlier labels."""
    out = []
    for _ in range(case["steps"]):
        y = (torch.rand(case["batch"], generator=g, device="cuda") < 0.6).float()
        r = torch.randn(case["batch"], 8, generator=g, device="cuda")
        scale = torch.tensor([1.5, 1.5, 0.5, 0.2, 0.15, 0.05, 0.0, 1.5], device="cuda")
        shift = torch.tensor([-1.0, 0.0, 0.0, 0.5, 0.6, 0.8, 0.3, -1.0], device="cuda")
        sep = torch.tensor([-1.5, -1.5, 0.0, 0.2, 0.0, 0.0, 0.0, -1.5], device="cuda")
        out.append(((shift + scale * r + y[:, None] * sep).to(torch.bfloat16), y))
    return out


def _trained():
    return np.load(os.path.join(os.path.dirname(os.path.abspath(learned.__file__)), "data", "mlp_inlier.npy"))


def _rotation_inputs(case, g):
    R, C, i, j = _cameras(case, g)
    ang = math.radians(case["noise_deg"]) * torch.randn(i.numel(), 1, generator=g, device="cuda", dtype=torch.float64)
    noise = torch.linalg.matrix_exp(_hat(_unit(i.numel(), g) * ang))
    return i.cpu().numpy(), j.cpu().numpy(), (noise @ R[j] @ R[i].transpose(1, 2)).cpu().numpy()


def _translation_inputs(case, g):
    R, C, i, j = _cameras(case, g)
    d = (R[j] @ (C[i] - C[j])[:, :, None])[:, :, 0]
    ang = math.radians(case["noise_deg"]) * torch.randn(i.numel(), 1, generator=g, device="cuda", dtype=torch.float64)
    d = (torch.linalg.matrix_exp(_hat(_unit(i.numel(), g) * ang)) @ d[:, :, None])[:, :, 0]
    d = d / d.norm(dim=1, keepdim=True)
    o = torch.randn(case["runs"], case["cams"], 3, generator=g, device="cuda", dtype=torch.float64)
    return tuple(v.cpu().numpy() for v in (R, i, j, d, o))


def _vote_inputs(case, g):
    """Fundamental matrices of noisy relative poses, a tenth of them wrong; known focal lengths of some sides."""
    B = case["pairs"]
    ang = math.radians(25.0) * torch.randn(B, 1, generator=g, device="cuda", dtype=torch.float64)
    E = _hat(_unit(B, g)) @ torch.linalg.matrix_exp(_hat(_unit(B, g) * ang))
    E = E + 1e-3 * torch.randn(B, 3, 3, generator=g, device="cuda", dtype=torch.float64)
    wrong = torch.rand(B, generator=g, device="cuda") < 0.1
    E = torch.where(wrong[:, None, None], torch.randn(B, 3, 3, generator=g, device="cuda", dtype=torch.float64), E)
    k = torch.tensor([F, F, 1.0], device="cuda", dtype=torch.float64)
    out = [(E / (k[:, None] * k[None, :])).cpu().numpy(), np.geomspace(0.3 * F, 3.0 * F, case["candidates"])]
    for _ in range(2):
        known = torch.rand(B, generator=g, device="cuda") < case["known"]
        out.append((F * known.double()).cpu().numpy() if case["known"] else None)
    return out


def prepare(case, seed):
    g = _generator(seed)
    kind = case["kind"]
    s = dict(case=case)
    if kind == "train":
        s["net"] = fm.Mlp(learned.init_params(seed % 1000))
        s["batches"] = _batches(case, g)
        return s
    if kind == "rotation":
        i, j, rel = _rotation_inputs(case, g)
        s["stage"] = fm.Rotation(i, j, rel, case["cams"])
        return s
    if kind == "translation":
        s["stage"] = fm.Translation(*_translation_inputs(case, g))
        return s
    if kind == "vote":
        s["inputs"] = _vote_inputs(case, g)
        return s
    sc = _scene(case, g)
    if kind == "create":
        if case["shuffled"]:
            at = torch.randperm(sc["pid"].numel(), generator=g, device="cuda")
            sc["pid"], sc["x1"], sc["x2"] = sc["pid"][at].contiguous(), sc["x1"][at].contiguous(), sc["x2"][at].contiguous()
        s["poses"] = tuple(v.cpu().numpy() for v in (sc["R"], _translations(sc["R"], sc["C"]), sc["i"], sc["j"]))
        s["scene"] = sc
        return s
    if kind == "autograd":
        s["problem"] = _problem(case, sc, fm.default_options(storage=case["storage"], delta=sc["sigma"]))
        s["problem"].irls_weights(0.1)
        R, C = _moved(sc, g)
        s["R"], s["C"] = R.requires_grad_(True), C.requires_grad_(True)
        return s
    s["schedule"] = _schedule(case, sc, 2 if kind == "learned" else 1)
    s["problem"] = _problem(case, sc, s["schedule"].options(storage=case["storage"]))
    if kind == "learned":
        s["problem"].set_scores(sc["score"])
        s["net"] = fm.Mlp(_trained())
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("round", "quadratic"):
        fm.refine(state["problem"], state["schedule"], quadratic=kind == "quadratic")
        return state["problem"].get_poses()
    if kind == "learned":
        learned.refine_learned(state["problem"], state["net"], state["schedule"], quadratic=case["quadratic"])
        return state["problem"].get_poses()
    if kind == "autograd":
        R, C = state["R"], state["C"]
        R.grad = C.grad = None
        loss = fm.epipolar_loss(state["problem"], R, C, case["recompute"])
        loss.backward()
        return loss.detach(), R.grad, C.grad
    if kind == "create":
        sc = state["scene"]
        with fm.Problem(*state["poses"], sc["pid"], sc["x1"], sc["x2"],
                        options=fm.default_options(storage=case["storage"], loss="l1")) as p:
            loss, grad = p.loss_grad()
            return loss, grad, p.residuals()
    if kind == "train":
        for x, y in state["batches"]:
            state["net"].train_step(x, y, 3e-3, want_loss=False)
        return state["net"].params()
    if kind == "rotation":
        stage = state["stage"]
        stage.initialize()
        start = stage.rotations()
        stage.step(case["steps"])
        return start, stage.rotations()
    if kind == "translation":
        stage = state["stage"]
        loss, grad, cam_loss = stage.loss_grad()
        stage.step(case["steps"])
        return loss, grad, cam_loss, stage.centres()
    f, cand, k1, k2 = state["inputs"]
    return fm.focal_vote(f, cand, 0.01, k1, k2)


# ---- the same results in 64 bits ----------------------------------------------------------------
def _essential(R, C, i, j):
    Rn = R[j] @ R[i].transpose(1, 2)
    t = (R[j] @ (C[i] - C[j])[:, :, None])[:, :, 0]
    return _hat(t / t.norm(dim=1, keepdim=True)) @ Rn


def _homogeneous(x):
    return torch.cat([x.double(), torch.ones_like(x[:, :1], dtype=torch.float64)], 1)


def _residuals(E, sc, q):
    return ((E[sc["pid"][q].long()] @ _homogeneous(sc["x1"][q])[:, :, None])[:, :, 0] * _homogeneous(sc["x2"][q])).sum(1)


def _exact_loss(sc, R, C, weights, l1):
    """(loss, gradient for left rotation increments, gradient for the centres), FP64; weights: of a chunk, or None."""
    n, P = R.shape[0], sc["pid"].numel()
    phi = torch.zeros(n, 3, device="cuda", dtype=torch.float64, requires_grad=True)
    Cv = C.detach().clone().requires_grad_(True)
    E = _essential(R.detach() + _hat(phi) @ R.detach(), Cv, sc["i"], sc["j"])
    G = torch.zeros(E.numel() // 9, 9, device="cuda", dtype=torch.float64)
    loss = 0.0
    for p in range(0, P, CHUNK // 4):
        q = slice(p, min(P, p + CHUNK // 4))
        e = _residuals(E.detach(), sc, q)
        w = None if l1 else weights(q)
        loss += float((e.abs() if l1 else w * e * e).sum()) / P
        s = (e.sign() if l1 else 2 * w * e) / P
        a = (s[:, None] * _homogeneous(sc["x2"][q]))[:, :, None] * _homogeneous(sc["x1"][q])[:, None, :]
        G.index_add_(0, sc["pid"][q].long(), a.reshape(-1, 9))
    g_phi, g_c = torch.autograd.grad(E, (phi, Cv), G.reshape(-1, 3, 3))
    return loss, g_phi, g_c


def _exact_train(case, seed, g):
    """Adam on the mean cross-entropy: weights and activations rounded to BF16, all else in 64 bits."""
    def rounded(v):
        return v.float().to(torch.bfloat16).double()

    p = torch.from_numpy(learned.init_params(seed % 1000)).double().cuda()
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    for t, (x, y) in enumerate(_batches(case, g), 1):
        W1, b1, W2, b2, W3, b3 = (u for u in torch.split(p, [256, 32, 1024, 32, 32, 1]))
        W1, W2, W3 = rounded(W1).reshape(8, 32), rounded(W2).reshape(32, 32), rounded(W3)
        x, y = x.double(), y.double()
        z1 = x @ W1 + b1
        h1 = rounded(z1.clamp_min(0))
        z2 = h1 @ W2 + b2
        h2 = rounded(z2.clamp_min(0))
        d3 = (torch.sigmoid(h2 @ W3 + b3) - y) / y.numel()
        d2 = (z2 > 0) * d3[:, None] * W3
        d1 = (z1 > 0) * (d2 @ W2.T)
        grad = torch.cat([(x.T @ d1).reshape(-1), d1.sum(0), (h1.T @ d2).reshape(-1), d2.sum(0), h2.T @ d3, d3.sum()[None]])
        m = 0.9 * m + 0.1 * grad
        v = 0.999 * v + 0.001 * grad * grad
        p = p - 3e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return p.cpu().numpy()


def _exact_rotation(case, g):
    """The column-wise initialisation by dense solves (camera 0 held at the identity)."""
    i, j, rel = _rotation_inputs(case, g)
    n, B = case["cams"], len(i)
    i, j, rel = torch.from_numpy(i).cuda(), torch.from_numpy(j).cuda(), torch.from_numpy(rel).cuda()
    eye = torch.eye(3, device="cuda", dtype=torch.float64)
    A = torch.zeros(n, n, 3, 3, device="cuda", dtype=torch.float64)
    deg = torch.bincount(torch.cat([i, j]), minlength=n).double()
    k = torch.arange(n, device="cuda")
    A[k, k] = deg[:, None, None] * eye
    A.index_put_((j, i), -rel, accumulate=True)
    A.index_put_((i, j), -rel.transpose(1, 2), accumulate=True)

    def solve(M, axis):
        full = M.permute(0, 2, 1, 3).reshape(3 * n, 3 * n)
        x = torch.linalg.solve(full[3:, 3:], -full[3:, axis])
        x = torch.cat([eye[axis], x]).reshape(n, 3)
        return x / x.norm(dim=1, keepdim=True)

    c1 = solve(A, 0)
    M = A / B
    M[k, k] += c1[:, :, None] * c1[:, None, :] / n
    c2 = solve(M, 1)
    c2 = c2 - (c1 * c2).sum(1, keepdim=True) * c1
    c2 = c2 / c2.norm(dim=1, keepdim=True)
    return torch.stack([c1, c2, torch.linalg.cross(c1, c2)], 2).cpu().numpy()


def _exact_translation(case, g):
    R, i, j, d, o = (torch.from_numpy(v).cuda() for v in _translation_inputs(case, g))
    target = -(R[j].transpose(1, 2) @ d[:, :, None])[:, :, 0]
    u = o[:, j] - o[:, i]
    nrm = u.norm(dim=2, keepdim=True)
    r = u / nrm - target
    term = r.abs().sum(2)
    s = r.sign()
    gu = (s - (u / nrm) * ((u / nrm) * s).sum(2, keepdim=True)) / nrm
    grad = torch.zeros_like(o).index_add_(1, j, gu).index_add_(1, i, -gu) / i.numel()
    tot = torch.zeros(o.shape[:2], device="cuda", dtype=torch.float64).index_add_(1, i, term).index_add_(1, j, term)
    deg = torch.bincount(torch.cat([i, j]), minlength=o.shape[1]).clamp_min(1)
    return term.mean(1).cpu().numpy(), grad.cpu().numpy(), (tot / deg).cpu().numpy(), None


def _exact_vote(case, g):
    """Singular values from the closed form of the eigenvalues of E^T E."""
    f, cand, k1, k2 = _vote_inputs(case, g)
    f = torch.from_numpy(f).cuda()
    f = f / f.flatten(1).norm(dim=1)[:, None, None]
    out = []
    for c in cand:
        side = [torch.full((f.shape[0],), float(c), device="cuda", dtype=torch.float64) for _ in range(2)]
        for a, k in enumerate((k1, k2)):
            if k is not None:
                side[a] = torch.where(torch.from_numpy(k).cuda() > 0, torch.from_numpy(k).cuda(), side[a])
        one = torch.ones_like(side[0])
        E = torch.stack([side[1], side[1], one], 1)[:, :, None] * f * torch.stack([side[0], side[0], one], 1)[:, None, :]
        M = E.transpose(1, 2) @ E
        q = torch.einsum("naa->n", M) / 3
        D = M - q[:, None, None] * torch.eye(3, device="cuda", dtype=torch.float64)
        p = ((D * D).sum((1, 2)) / 6).sqrt()
        half = (torch.linalg.det(D / p[:, None, None]) / 2).clamp(-1, 1)
        a = torch.acos(half) / 3
        hi = q + 2 * p * torch.cos(a)
        mid = q + 2 * p * torch.cos(a - 2 * math.pi / 3)
        out.append(float(torch.exp((1 - (hi / mid).sqrt()) / 0.01).sum()))
    return np.array(out)


def exact(case, seed):
    g = _generator(seed)
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed, g)
    if kind == "rotation":
        return _exact_rotation(case, g), None
    if kind == "translation":
        return _exact_translation(case, g)
    if kind == "vote":
        return _exact_vote(case, g)
    if kind == "autograd":
        sc = _scene(case, g)
        R, C = _moved(sc, g)
        E0 = _essential(sc["R"], sc["C"], sc["i"], sc["j"])

        def weights(q):
            e = _residuals(E0, sc, q).abs()
            return torch.where(e <= 0.1, 1 / e.clamp_min(sc["sigma"]), torch.zeros_like(e))

        loss, g_phi, g_c = _exact_loss(sc, R, C, weights, False)
        return torch.tensor(loss, dtype=torch.float64), 0.5 * _hat(g_phi) @ R, g_c
    if kind == "create":
        s = prepare(case, seed)
        sc = s["scene"]
        loss, g_phi, g_c = _exact_loss(sc, sc["R"], sc["C"], None, True)
        E, P = _essential(sc["R"], sc["C"], sc["i"], sc["j"]), sc["pid"].numel()
        e = torch.cat([_residuals(E, sc, slice(p, min(P, p + CHUNK // 4))) for p in range(0, P, CHUNK // 4)])
        return loss, torch.cat([g_phi, g_c], 1).cpu().numpy(), e.cpu().numpy()
    return None    # a round of Adam steps: its poses follow the rounding of every step before them


def work(case):
    """Bytes read and written once (per iteration where they do not fit the L2 cache) and arithmetic operations."""
    kind = case["kind"]
    if kind == "train":
        macs = 8 * 32 + 32 * 32 + 32
        return dict(bytes=case["steps"] * case["batch"] * 20 + 1377 * 4 * 6, flops=case["steps"] * case["batch"] * 6 * macs)
    if kind == "vote":
        return dict(bytes=case["pairs"] * 72 + case["candidates"] * 16, flops=case["pairs"] * case["candidates"] * 300)
    pairs = case["cams"] * min(0.6 * case["near"], (case["cams"] - 1) / 2)
    if kind == "rotation":
        return dict(bytes=pairs * 80 + case["cams"] * 300, flops=pairs * (200 * 2 * 18 + case["steps"] * 200))
    if kind == "translation":
        return dict(bytes=pairs * 24 + case["runs"] * case["cams"] * 80,
                    flops=case["runs"] * pairs * (case["steps"] + 1) * 40)
    P = max(case["points"], pairs)
    size = P * (20 if case["storage"] == "fp32" else 10)
    if kind == "create":
        return dict(bytes=P * 20 + 3 * size + P * 4, flops=P * 60)
    if kind == "autograd":
        return dict(bytes=size * (2 if case["recompute"] else 1), flops=P * 40 * (2 if case["recompute"] else 1))
    it = case["iters"]
    passes = it if size > ON_CHIP else 1
    if kind == "round":
        return dict(bytes=passes * size, flops=P * it * 40)
    if kind == "quadratic":
        return dict(bytes=size + pairs * 224 * it, flops=P * 130 + pairs * it * 800)
    net = P * (16 if case["storage"] == "fp16" else 28)
    if case["quadratic"]:
        return dict(bytes=2 * (net + size + pairs * 224 * it), flops=2 * (P * (2700 + 130) + pairs * it * 800))
    return dict(bytes=2 * (net + (passes - 1) * size), flops=2 * (P * 2700 + P * it * 40))
