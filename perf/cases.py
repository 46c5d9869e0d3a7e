"""Performance cases: the work that users of the library have it do, through its public entry points.

``listed()`` names the cases and ``draw(rng)`` draws one more from the same ranges.  Kinds of work:

* ``softmin``     -- one sweep of ``otgb.softmin`` (a custom loop's step): 3-D points and fiber vectors, from a
                     thousand points (latency) to a whole density map.
* ``dense``       -- ``otgb.sinkhorn_divergence`` on one scale: the small registration problem (a rotated cloud of
                     a few thousand points), balanced and unbalanced, in 3-D and on short fiber sets.
* ``density``     -- the coarse-to-fine solve on two track-density maps (3-D voxels, grid clusters, unbalanced).
* ``fibers``      -- the coarse-to-fine solve on two tractograms (k-means clusters, unbalanced), in float32 and in
                     the tensor-core form.
* ``transfer``    -- ``otgb.transport_apply``: label transfer from an atlas of fiber bundles to a subject.
* ``grad``        -- ``otgb.sinkhorn_grad_x``: the gradient of the divergence in the points.
* ``barycenter``  -- ``otgb.sinkhorn_barycenter``: a gradient step of the track-density atlas.
* ``mlp_infer``, ``mlp_grad`` -- the warm-start network: inference over a subject, loss and gradient of a batch.

Solves run the paper's schedule and then a fixed number of steps at the final scale (``fixed_iters``), so that
every solve of a case does the same work.  Inputs have the shapes and distributions of
``paper_2107_02010_gb300.synth``, drawn on the GPU.
"""
import math

import numpy as np
import torch

from paper_2107_02010_gb300 import otgb, synth

GRID = 64           # voxels per axis of a density volume
TUBE_SIGMA = 1.5
N_BUNDLES = 20
FIBER_EPS = 4.0     # blur 2 mm
STEPS = 10          # steps at the final scale, dense and density solves
FIBER_STEPS = 5


# ------------------------------------------------------------------ cases ---
def listed():
    return [
        # the smallest calls: one step of a custom loop on a thousand points, where launches and latency count
        {"name": "softmin_3d_1k", "kind": "softmin", "D": 3, "n": 1000, "m": 800},
        # one dense sweep over a whole pair of density maps
        {"name": "softmin_3d_100k", "kind": "softmin", "D": 3, "n": 100_000, "m": 100_000},
        # one dense sweep over two small tractograms, ragged sizes
        {"name": "softmin_60d_20k", "kind": "softmin", "D": 60, "n": 19_997, "m": 20_011},
        # the balanced single-scale problem: a rigidly moved noisy cloud of 2,000 points
        {"name": "dense_cloud_2k", "kind": "dense", "D": 3, "n": 2000, "m": 2000, "reach": 0.0},
        # the track-density workload: 100,000 voxels per side, unbalanced
        {"name": "density_100k", "kind": "density", "n": 100_000, "m": 100_000, "reach": 10.0},
        # subject against the 300,000-fiber atlas, float32
        {"name": "fibers_300k_fp32", "kind": "fibers", "P": 20, "n": 300_000, "m": 300_000, "tc": False},
        # the scale test: a million fibers per side, tensor-core form
        {"name": "fibers_1m_tc", "kind": "fibers", "P": 20, "n": 1_000_000, "m": 1_000_000, "tc": True},
        # bundle labels of an atlas carried to a subject
        {"name": "transfer_60k", "kind": "transfer", "P": 20, "n": 60_013, "m": 50_000, "L": 20},
        # gradient in the points of a density map against another one
        {"name": "grad_3d_50k", "kind": "grad", "D": 3, "n": 50_000, "m": 50_000},
        # one gradient step of a track-density atlas, with the objective before and after
        {"name": "barycenter_2x5k", "kind": "barycenter", "K": 2, "n": 5000},
        # the warm-start network over one subject
        {"name": "mlp_infer_400k", "kind": "mlp_infer", "P": 20, "H": 256, "n": 400_000},
        # loss and gradient of one training batch
        {"name": "mlp_grad_16k", "kind": "mlp_grad", "P": 20, "H": 256, "n": 16_384},
    ]


def _size(rng, lo, hi):
    """A size between lo and hi, uniform in its logarithm; mostly no multiple of anything."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["softmin", "softmin", "dense", "density", "fibers", "fibers", "transfer", "grad",
                       "barycenter", "mlp_infer", "mlp_grad"])
    P = rng.choice([8, 12, 16, 20])
    if kind == "softmin":
        D = rng.choice([2, 3, 3, 3 * P, 60])
        hi = 100_000 if D <= 3 else 30_000
        return {"kind": kind, "D": D, "n": _size(rng, 300, hi), "m": _size(rng, 300, hi)}
    if kind == "dense":
        D = rng.choice([2, 3, 3, 3 * P])
        return {"kind": kind, "D": D, "n": _size(rng, 200, 6000), "m": _size(rng, 200, 6000),
                "reach": rng.choice([0.0, 0.5, 1.0])}
    if kind == "density":
        return {"kind": kind, "n": _size(rng, 10_000, 100_000), "m": _size(rng, 10_000, 100_000),
                "reach": rng.choice([5.0, 10.0, 20.0])}
    if kind == "fibers":
        tc = rng.random() < 0.5
        hi = 1_000_000 if tc else 300_000
        n = _size(rng, 20_000, hi)
        return {"kind": kind, "P": P, "n": n, "m": min(hi, max(20_000, int(n * rng.uniform(0.5, 2.0)))), "tc": tc}
    if kind == "transfer":
        return {"kind": kind, "P": P, "n": _size(rng, 2000, 60_000), "m": _size(rng, 2000, 50_000),
                "L": rng.randint(2, 40)}
    if kind == "grad":
        D = rng.choice([3, 3, 60, 3 * P])
        hi = 50_000 if D <= 3 else 15_000
        return {"kind": kind, "D": D, "n": _size(rng, 500, hi), "m": _size(rng, 500, hi)}
    if kind == "barycenter":
        return {"kind": kind, "K": rng.randint(1, 3), "n": _size(rng, 1000, 5000)}
    if kind == "mlp_infer":
        return {"kind": kind, "P": P, "H": rng.choice([128, 256]), "n": _size(rng, 1000, 400_000)}
    return {"kind": kind, "P": P, "H": rng.choice([128, 256]), "n": _size(rng, 128, 65_536)}


# ----------------------------------------------------------------- inputs ---
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _density(n, seed, mass):
    """The n strongest voxels of a GRID^3 volume of 30 Gaussian tubes (the recipe of synth.density_map)."""
    r = np.random.default_rng(seed)
    ax = torch.arange(GRID, device="cuda", dtype=torch.float32) + 0.5
    vox = torch.stack(torch.meshgrid(ax, ax, ax, indexing="ij"), dim=-1).reshape(-1, 3)
    dens = torch.zeros(vox.shape[0], device="cuda")
    t = np.linspace(0.0, 1.0, 256)[:, None]
    for _ in range(30):
        c = r.uniform(GRID / 8.0, GRID * 7.0 / 8.0, size=(4, 3))
        curve = (1 - t) ** 3 * c[0] + 3 * (1 - t) ** 2 * t * c[1] + 3 * (1 - t) * t ** 2 * c[2] + t ** 3 * c[3]
        curve = torch.from_numpy(curve.astype(np.float32)).cuda()
        d2 = sum((vox[:, None, k] - curve[None, :, k]) ** 2 for k in range(3)).amin(dim=1)
        dens += torch.where(d2 < (6 * TUBE_SIGMA) ** 2, torch.exp(-d2 / (2 * TUBE_SIGMA ** 2)), torch.zeros_like(d2))
    n = min(n, int((dens > 0).sum()))
    idx = torch.topk(dens, n).indices.sort().values
    w = dens[idx].double()
    return vox[idx].contiguous(), (w / w.sum() * mass).float().contiguous()


def _centrelines(P, seed):
    """Bundle centrelines, P points equally spaced in arc length, and their control points (perturbed by the seed)."""
    ctrl = synth.bundle_centrelines(N_BUNDLES, P=P)
    ctrl = ctrl + np.random.default_rng(seed).normal(0.0, 3.0, size=ctrl.shape)
    t = np.linspace(0.0, 1.0, 512)[:, None]
    lines = []
    for c in ctrl:
        curve = (1 - t) ** 3 * c[0] + 3 * (1 - t) ** 2 * t * c[1] + 3 * (1 - t) * t ** 2 * c[2] + t ** 3 * c[3]
        s = np.concatenate([[0.0], np.cumsum(np.linalg.norm(np.diff(curve, axis=0), axis=1))])
        u = np.linspace(0.0, s[-1], P)
        lines.append(np.stack([np.interp(u, s, curve[:, d]) for d in range(3)], axis=1))
    return np.stack(lines)


def _fibers(n, P, seed):
    """n fibers of P points around the bundles, canonically oriented, times 1/sqrt(P) (synth.fiber_bundles)."""
    g = _gen(seed)
    lines = _centrelines(P, seed)
    # a fiber keeps the orientation in which its first point is the lexicographically smaller end
    lines = np.stack([ln if tuple(ln[0]) < tuple(ln[-1]) else ln[::-1] for ln in lines])
    lines = torch.from_numpy(lines.astype(np.float32)).cuda()
    lab = torch.randint(0, N_BUNDLES, (n,), generator=g, device="cuda")
    x = lines[lab] + 2.0 * _normal(g, n, 1, 3) + 0.5 * _normal(g, n, P, 3)
    return (x.reshape(n, 3 * P) / math.sqrt(P)).contiguous(), lab.int()


def _cloud(n, m, D, seed):
    """A cloud in the unit cube and a moved, noisy copy (synth.rotated_cloud in any dimension)."""
    g = _gen(seed)
    x = torch.rand(n, D, generator=g, device="cuda")
    y = torch.rand(m, D, generator=g, device="cuda")
    if D >= 2:
        a = math.radians(5.0 + 10.0 * (seed % 7) / 7.0)
        c, s = math.cos(a), math.sin(a)
        u, v = y[:, 0] - 0.5, y[:, 1] - 0.5
        y = torch.cat([(c * u - s * v + 0.5)[:, None], (s * u + c * v + 0.5)[:, None], y[:, 2:]], dim=1)
    y[:, 0] += 0.1
    y = y + 0.01 * _normal(g, m, D)
    return x.contiguous(), y.contiguous()


def _points(n, m, D, seed):
    """Two weighted point sets of dimension D and their eps: a cloud in voxels, or fibers."""
    if D > 3:
        P = D // 3
        x, y = _fibers(n, P, seed)[0], _fibers(m, P, seed + 1000)[0]
        a = torch.full((n,), 1.0 / n, device="cuda")
        b = torch.full((m,), 1.0 / m, device="cuda")
        return x, a, y, b, FIBER_EPS
    if D == 3 and n >= 5000 and m >= 5000:
        x, a = _density(n, seed, 1.0)
        y, b = _density(m, seed + 1000, 1.2)
        return x, a, y, b, 1.0
    x, y = _cloud(n, m, D, seed)
    g = _gen(seed + 1)
    a, b = (torch.rand(k, generator=g, device="cuda") + 0.5 for k in (n, m))
    return x, (a / a.sum()).contiguous(), y, (b / b.sum()).contiguous(), 0.05 ** 2


def _softmin_t(q, p, w, pot, eps, lam=1.0, dtype=torch.float32):
    """-lam eps log sum_j w_j exp((pot_j - |q_i - p_j|^2 / 2) / eps) in plain torch."""
    q, p, lw = q.to(dtype), p.to(dtype), torch.log(w.to(dtype))
    pot = pot.to(dtype)
    c = p.mean(dim=0)
    q, p = q - c, p - c
    h = lw + (pot - 0.5 * (p * p).sum(1)) / eps
    hq = 0.5 * (q * q).sum(1)
    out = torch.empty(q.shape[0], device=q.device, dtype=dtype)
    step = max(1, 200_000_000 // p.shape[0])
    for i in range(0, q.shape[0], step):
        e = torch.addmm(h[None, :], q[i:i + step], p.T, alpha=1.0 / eps)
        out[i:i + step] = -lam * (eps * torch.logsumexp(e, dim=1) - hq[i:i + step])
    return out


def _duals(x, a, y, b, eps, rho, want_self, dtype):
    """Annealed duals near a solution, in plain torch: what a solve hands to transfer and gradient."""
    f = torch.zeros(x.shape[0], device="cuda", dtype=dtype)
    g = torch.zeros(y.shape[0], device="cuda", dtype=dtype)
    s = torch.zeros_like(f)
    for k in (64.0, 16.0, 4.0, 1.0, 1.0):
        lam = 1.0 / (1.0 + k * eps / rho)
        f = _softmin_t(x, y, b, g, k * eps, lam, dtype)
        g = _softmin_t(y, x, a, f, k * eps, lam, dtype)
        if want_self:
            s = 0.5 * (s + _softmin_t(x, x, a, s, k * eps, lam, dtype))
    return f.float(), g.float(), s.float()


def _theta(D, H, seed):
    """Network parameters in the library's flat order, drawn as a fresh network's."""
    r = np.random.default_rng(seed)
    parts = []
    for fan_in, out, lim in ((D, H, 6.0), (H, H, 6.0), (H, H, 6.0), (H, 1, 3.0)):
        k = math.sqrt(lim / fan_in)
        parts.append(r.uniform(-k, k, size=fan_in * out))
        parts.append(r.uniform(-0.1, 0.1, size=out))
    return np.concatenate(parts).astype(np.float32)


def _mlp_inputs(case, seed):
    x, _ = _fibers(case["n"], case["P"], seed)
    D = x.shape[1]
    mean, scale = x.double().mean(0).float(), x.double().std(0).float() + 1e-3
    r = np.random.default_rng(seed + 7)
    v = torch.from_numpy(r.normal(0.0, 1.0, size=(D, 4)).astype(np.float32)).cuda() / math.sqrt(D)
    f = 40.0 * torch.sin(((x - mean) / scale) @ v).sum(1)  # a smooth dual-like target
    return x, f.contiguous(), mean.cpu().numpy(), scale.cpu().numpy(), 0.0, 60.0, _theta(D, case["H"], seed)


# ---------------------------------------------------------------- prepare ---
def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind, "ctx": otgb.Context()}
    if kind == "softmin":
        x, a, y, b, eps = _points(case["n"], case["m"], case["D"], seed)
        g = _gen(seed + 2)
        # a potential a few eps deep and old values of the same size; the unbalanced damping of the workloads
        st.update(x=x, y=y, b=b, eps=eps, pot=eps * 3.0 * _normal(g, y.shape[0]), old=eps * 3.0 * _normal(g, x.shape[0]),
                  lam=1.0 / 1.01)
    elif kind == "dense":
        if case["D"] > 3:
            x, a, y, b, _ = _points(case["n"], case["m"], case["D"], seed)
            blur, reach = 2.0, 20.0 * case["reach"]
        else:
            x, y = _cloud(case["n"], case["m"], case["D"], seed)
            a = torch.full((x.shape[0],), 1.0 / x.shape[0], device="cuda")
            b = torch.full((y.shape[0],), 1.0 / y.shape[0], device="cuda")
            blur, reach = 0.05, case["reach"]
        st.update(x=x, a=a, y=y, b=b, p=otgb.default_params(blur=blur, reach=reach, scaling=0.5, fixed_iters=STEPS))
    elif kind == "density":
        x, a = _density(case["n"], seed, 1.0)
        y, b = _density(case["m"], seed + 1000, 1.2)
        st.update(x=x, a=a, y=y, b=b, p=otgb.default_params(blur=1.0, reach=case["reach"], scaling=0.5, multiscale=1,
                                                            cluster=0, cell=4.0, fixed_iters=STEPS))
    elif kind == "fibers":
        x, a, y, b, _ = _points(case["n"], case["m"], 3 * case["P"], seed)
        st.update(x=x, a=a, y=y, b=b, p=_fiber_params(case["n"], FIBER_STEPS, case["tc"]))
    elif kind == "transfer":
        P, n, m = case["P"], case["n"], case["m"]
        x, _ = _fibers(n, P, seed)
        y, lab = _fibers(m, P, seed + 1000)
        a = torch.full((n,), 1.0 / n, device="cuda")
        b = torch.full((m,), 1.0 / m, device="cuda")
        f, g, _ = _duals(x, a, y, b, FIBER_EPS, 400.0, False, torch.float32)
        plan = otgb.sinkhorn_divergence(st["ctx"], x, a, y, b, _fiber_params(n, 1, True), want_plan=True)["plan"]
        lab = (lab * 7 + torch.arange(m, device="cuda", dtype=torch.int32) // 4096) % case["L"]
        st.update(plan=plan, f=f, g=g, labels=lab.int().contiguous(), L=case["L"], b=b, x=x, y=y)
    elif kind == "grad":
        x, a, y, b, eps = _points(case["n"], case["m"], case["D"], seed)
        f, g, s = _duals(x, a, y, b, eps, 100.0 * eps, True, torch.float64 if case["D"] <= 3 else torch.float32)
        st.update(x=x, a=a, y=y, b=b, eps=eps, f=f, g=g, s=s)
    elif kind == "barycenter":
        maps = [_density(case["n"], seed + 1000 * k, 1.0) for k in range(case["K"])]
        ys = [y for y, _ in maps]
        bs = [torch.from_numpy(synth.unit_mass(w.cpu().numpy())).cuda() for _, w in maps]
        vox, inv = torch.unique(torch.cat(ys), dim=0, return_inverse=True)
        dens = torch.zeros(vox.shape[0], device="cuda", dtype=torch.float64)
        dens.index_put_((inv,), torch.cat(bs).double(), accumulate=True)
        # the strongest voxels of the average map, as many as a map has, each up-sampled into 6 points
        idx = torch.topk(dens, case["n"]).indices.sort().values
        x0 = vox[idx].repeat_interleave(6, dim=0) - 0.5
        x0 += torch.rand(x0.shape[0], 3, generator=_gen(seed), device="cuda")
        w0 = synth.unit_mass(np.repeat(dens[idx].cpu().numpy(), 6))
        st.update(x0=x0.contiguous(), a0=torch.from_numpy(w0).cuda(), ys=ys, bs=bs,
                  p=otgb.default_params(blur=1.0, reach=0.0, scaling=0.5, multiscale=1, cluster=0, cell=4.0,
                                        fixed_iters=STEPS))
    else:
        x, f, mean, scale, om, os_, theta = _mlp_inputs(case, seed)
        net = otgb.Mlp(st["ctx"], x.shape[1], case["H"], seed=1)
        net.set_normalization(mean, scale, om, os_)
        net.set_params(theta)
        st.update(net=net, x=x, f=f)
    return st


def _fiber_params(n, steps, tc):
    return otgb.default_params(blur=2.0, reach=20.0, scaling=0.5, multiscale=1, cluster=1,
                               k_clusters=max(2, n // 1000), seed=0, fixed_iters=steps, precision=1 if tc else 0)


# -------------------------------------------------------------------- run ---
def run(st):
    kind, ctx = st["kind"], st["ctx"]
    if kind == "softmin":
        return otgb.softmin(ctx, st["x"], st["y"], st["b"], st["pot"], st["eps"], lam=st["lam"], old=st["old"])
    if kind in ("dense", "density", "fibers"):
        r = otgb.sinkhorn_divergence(ctx, st["x"], st["a"], st["y"], st["b"], st["p"], want_self=True)
        return {k: r[k] for k in ("S", "f", "g", "a_self", "b_self")}
    if kind == "transfer":
        sc, am, rm = otgb.transport_apply(ctx, st["plan"], st["f"], st["g"], st["labels"], st["L"])
        return {"scores": sc, "argmax": am, "row_mass": rm}
    if kind == "grad":
        return otgb.sinkhorn_grad_x(ctx, st["x"], st["a"], st["y"], st["b"], st["eps"], st["f"], st["g"], st["s"])
    if kind == "barycenter":
        x = st["x0"].clone()
        hist = otgb.sinkhorn_barycenter(ctx, x, st["a0"], st["ys"], st["bs"], st["p"], iters=1)
        return {"x": x, "S": hist}
    if kind == "mlp_infer":
        return st["net"].infer(st["x"])
    loss, grad = st["net"].grad(st["x"], st["f"])
    return {"loss": loss, "grad": grad}


# ------------------------------------------------------------------- work ---
def work(case):
    """Bytes (inputs once, outputs once) and operations.  The coarse-to-fine solves count the pairs that the
    truncation has to keep: about 5 % of all pairs for 20 bundles, 15 % for density maps at blur 1 voxel."""
    kind, n, m = case["kind"], case["n"], case.get("m", 0)
    D = case.get("D", 3 * case.get("P", 1))
    pair = 2.0 * D + 4.0
    if kind == "softmin":
        return {"bytes": 4.0 * (n * (D + 2) + m * (D + 2)), "flops": pair * n * m}
    if kind in ("dense", "density", "fibers"):
        D = 3 if kind == "density" else D
        kept, steps = {"dense": (1.0, 16), "density": (0.15, 12), "fibers": (0.05, 8)}[kind]
        return {"bytes": 4.0 * (n + m) * (D + 3),
                "flops": (2.0 * D + 4.0) * kept * steps * (float(n) * n + float(m) * m + 2.0 * n * m)}
    if kind == "transfer":
        return {"bytes": 4.0 * (n * (D + 3 + case["L"]) + m * (D + 3)), "flops": pair * n * m}
    if kind == "grad":
        return {"bytes": 4.0 * (n * (2 * D + 3) + m * (D + 2)), "flops": (5.0 * D + 4.0) * n * (n + m)}
    if kind == "barycenter":
        s = 6.0 * n  # support points
        return {"bytes": 4.0 * (8.0 * s + 4.0 * n * case["K"]),
                "flops": 10.0 * 0.15 * 26 * case["K"] * (s * s + 2.0 * s * n + float(n) * n)}
    H = case["H"]
    layer = 2.0 * (D * H + 2.0 * H * H + H)
    params = D * H + 2 * H * H + 5 * H
    if kind == "mlp_infer":
        return {"bytes": 4.0 * (n * (D + 1) + params), "flops": layer * n}
    return {"bytes": 4.0 * (n * (D + 1) + 2 * params), "flops": 3.0 * layer * n}


# ------------------------------------------------------------------ exact ---
def _divergence_t(x, a, y, b, blur, reach, q, steps):
    """The Algorithm on one scale in double precision: schedule, then `steps` steps at blur, with the translation of
    (f, g) after each step when the problem is unbalanced."""
    x, a, y, b = (t.double() for t in (x, a, y, b))
    box = torch.cat([x, y])
    d = float((box.amax(0) - box.amin(0)).square().sum().sqrt())
    sched = [d * q ** k for k in range(math.ceil(math.log(d / blur) / math.log(1.0 / q)))] if d > blur else []
    rho = reach * reach if reach > 0 else math.inf
    f, g, s, t = (torch.zeros(k, device="cuda", dtype=torch.float64)
                  for k in (x.shape[0], y.shape[0], x.shape[0], y.shape[0]))
    for sigma in sched + [blur] * (steps + 1):
        eps = sigma * sigma
        lam = 1.0 / (1.0 + eps / rho)
        sm = lambda u, v, w, pot: _softmin_t(u, v, w, pot, eps, lam, torch.float64)  # noqa: E731
        s2, t2, g2, f2 = sm(x, x, a, s), sm(y, y, b, t), sm(y, x, a, f), sm(x, y, b, g)
        s, t, g, f = 0.5 * (s + s2), 0.5 * (t + t2), 0.5 * (g + g2), 0.5 * (f + f2)
        if reach > 0:
            c = 0.5 * rho * torch.log((a * torch.exp(-f / rho)).sum() / (b * torch.exp(-g / rho)).sum())
            f, g = f + c, g - c
    if reach > 0:
        S = -(rho + 0.5 * blur * blur) * ((a * torch.exp(-s / rho) * torch.expm1(-(f - s) / rho)).sum()
                                          + (b * torch.exp(-t / rho) * torch.expm1(-(g - t) / rho)).sum())
    else:
        S = (a * (f - s)).sum() + (b * (g - t)).sum()
    return {"S": S, "f": f, "g": g, "a_self": s, "b_self": t}


def _net_t(u, theta, D, H):
    """The network on normalised inputs u in double precision; theta: the flat parameter vector."""
    o = 0
    for fan_in, out in ((D, H), (H, H), (H, H), (H, 1)):
        W = theta[o:o + fan_in * out].reshape(out, fan_in)
        bias = theta[o + fan_in * out:o + fan_in * out + out]
        o += fan_in * out + out
        u = u @ W.T + bias
        if out > 1:
            u = torch.nn.functional.silu(u)
    return u[:, 0]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("density", "fibers", "barycenter"):
        return None  # clusters and truncation decide which steps run on which pairs
    if kind in ("mlp_infer", "mlp_grad"):
        x, f, mean, scale, om, os_, theta = _mlp_inputs(case, seed)
        D, H = x.shape[1], case["H"]
        mean, scale, th = (torch.from_numpy(v).double().cuda() for v in (mean, scale, theta))
        if kind == "mlp_infer":
            return torch.cat([om + os_ * _net_t((c.double() - mean) / scale, th, D, H) for c in x.split(65_536)])
        th.requires_grad_(True)
        res = _net_t((x.double() - mean) / scale, th, D, H) - (f.double() - om) / os_
        loss = 0.5 * res.square().mean()
        loss.backward()
        return {"loss": loss.detach(), "grad": th.grad}
    st = prepare(case, seed)
    if kind == "softmin":
        tilde = _softmin_t(st["x"], st["y"], st["b"], st["pot"], st["eps"], st["lam"], torch.float64)
        return 0.5 * (st["old"].double() + tilde)
    if kind == "dense":
        p = st["p"]
        return _divergence_t(st["x"], st["a"], st["y"], st["b"], p.blur, p.reach, p.scaling, STEPS)
    x, y, b, f, g = (st[k].double() for k in ("x", "y", "b", "f", "g"))
    if kind == "transfer":
        eps = FIBER_EPS
        onehot = torch.nn.functional.one_hot(st["labels"].long(), case["L"]).double() * b[:, None]
        sc = [torch.exp((u[:, None] + g[None, :] - 0.5 * _sq(v, y)) / eps) @ onehot
              for u, v in zip(f.split(2048), x.split(2048))]
        sc = torch.cat(sc)
        return {"scores": sc, "argmax": None, "row_mass": sc.sum(1)}
    a, s, eps = st["a"].double(), st["s"].double(), st["eps"]
    out = []
    for v, u, t in zip(x.split(2048), f.split(2048), s.split(2048)):
        pi = torch.exp((u[:, None] + g[None, :] - 0.5 * _sq(v, y)) / eps) * b[None, :]
        pa = torch.exp((t[:, None] + s[None, :] - 0.5 * _sq(v, x)) / eps) * a[None, :]
        out.append(pi.sum(1, keepdim=True) * v - pi @ y - pa.sum(1, keepdim=True) * v + pa @ x)
    return a[:, None] * torch.cat(out)


def _sq(u, v):
    """|u_i - v_j|^2 in double precision."""
    return (u * u).sum(1)[:, None] + (v * v).sum(1)[None, :] - 2.0 * (u @ v.T)
