"""The work a user of the registration framework has it do, as measurable cases.

Each case names a public entry point and its sizes:
  eval        loss and gradient of one series at its finest level (`Muster.eval`): one forward
              pass and adjoint over every ordered pair, the body of every gradient step and of
              a caller's own optimiser;
  run         a whole registration on a context that is kept (`Muster.set_images`,
              `Muster.run`, the velocities read back), as a service runs one subject after another;
  similarity  the windowed similarity of two volumes and its gradient (`op_similarity`);
  exp         the exponential of one velocity field (`op_exp`);
  jacobian    a Jacobian determinant map (`op_jacobian_det`);
  metrics     the deformation metrics of an estimate against a reference (`op_deformation_metrics`).

Inputs are seeded synthetic heads made on the GPU (tissue classes, texture, smooth deformations
from session to session, bias field, Rician noise) and smooth random velocities. `exact` states
the same quantities in 64 bits with plain torch.
"""
import math

import numpy as np
import torch
import torch.nn.functional as nnf

import paper_2412_14671_gb300 as m

# the weights of the benchmark's registrations
ALPHA = dict(alpha_ss=0.05, alpha_l2=0.005, lr=0.05)

# the most pair-voxels (ordered pairs x voxels) whose 64-bit evaluation stays within seconds
EXACT_PAIR_VOXELS = 5.0e8
# the most pair-voxels of a drawn series (the largest listed one has 4.0e9)
DRAW_PAIR_VOXELS = 4.8e8


def listed():
    return [
        # the smallest call: one pair of small volumes, where launches and latency count
        dict(name="similarity small", op="similarity", D=48, H=48, W=48, window=5, kind=0),
        # one pair of brain volumes at 1 mm, the benchmark's window
        dict(name="similarity brain", op="similarity", D=160, H=192, W=160, window=7, kind=0),
        # one velocity field of a brain series (flow grid of 160 x 192 x 160 images)
        dict(name="exp brain", op="exp", D=80, H=96, W=80, K=7, sign=1, rms=1.0),
        # the map a user makes of a registered session
        dict(name="jacobian brain", op="jacobian", D=160, H=192, W=160),
        # accuracy of an estimate within the head
        dict(name="metrics brain", op="metrics", D=160, H=192, W=160, roi=True),
        # a small series evaluated for a caller's optimiser
        dict(name="eval small", op="eval", N=3, D=48, H=48, W=48, K=6, window=5, kind=0, det=0),
        # odd extents, normalised cross-correlation, bit-reproducible sums, uneven time gaps
        dict(name="eval odd", op="eval", N=5, D=91, H=109, W=91, K=7, window=5, kind=1, det=1, ts=0.05),
        # smoothed velocities and rigid motion estimated together, the method's own 3^3 window
        dict(name="eval smooth rigid", op="eval", N=6, D=128, H=128, W=128, K=7, window=3, kind=0, det=0, omega=0.08,
             rigid=1),
        # the benchmark's series at its finest level
        dict(name="eval brain", op="eval", N=10, D=160, H=192, W=160, K=7, window=7, kind=0, det=0),
        # the large series: 240 pairs of 256^3, squaring intermediates recomputed
        dict(name="eval large", op="eval", N=16, D=256, H=256, W=256, K=8, window=9, kind=0, det=0, recompute=1),
        # a small registration from images to velocities, where launches and latency count
        dict(name="run small", op="run", N=3, D=48, H=48, W=48, K=6, window=5, kind=0, levels=1, steps=20),
        # the benchmark's registration over its four levels with a short schedule
        dict(name="run brain", op="run", N=10, D=160, H=192, W=160, K=7, window=7, kind=0, levels=4, steps=10),
    ]


def _axes(rng, lo, hi):
    """Three extents around one size that is spread over the logarithm of lo..hi."""
    s = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return [int(min(hi, max(lo, round(s * rng.uniform(0.8, 1.25))))) for _ in range(3)]


def draw(rng):
    op = rng.choice(["eval"] * 7 + ["similarity"] * 4 + ["run"] * 2 + ["exp"] * 3 + ["jacobian"] * 2 + ["metrics"] * 2)
    if op == "exp":
        D, H, W = _axes(rng, 24, 128)
        return dict(op=op, D=D, H=H, W=W, K=rng.randint(5, 8), sign=rng.choice([1, -1]), rms=round(rng.uniform(0.3, 1.5), 2))
    if op == "jacobian":
        D, H, W = _axes(rng, 40, 256)
        return dict(op=op, D=D, H=H, W=W)
    if op == "metrics":
        D, H, W = _axes(rng, 40, 256)
        return dict(op=op, D=D, H=H, W=W, roi=rng.random() < 0.5)
    if op == "similarity":
        D, H, W = _axes(rng, 40, 256)
        return dict(op=op, D=D, H=H, W=W, window=rng.choice([3, 5, 7, 7, 9, 11]), kind=rng.choice([0, 0, 1]))
    N = rng.randint(2, 12)
    D, H, W = _axes(rng, 40, 224)
    if rng.random() < 0.5:  # half of the series have extents that divide by 8
        D, H, W = [max(40, 8 * round(a / 8)) for a in (D, H, W)]
    while N * (N - 1) * D * H * W > DRAW_PAIR_VOXELS:
        N -= 1
    c = dict(op=op, N=N, D=D, H=H, W=W, K=rng.randint(6, 8), window=rng.choice([3, 5, 7, 7, 9]), kind=rng.choice([0, 0, 0, 1]))
    if op == "run":
        c.update(window=rng.choice([5, 7]), kind=0, levels=rng.choice([2, 3]) if min(D, H, W) >= 64 else 1, steps=rng.randint(5, 10))
        return c
    c.update(det=rng.choice([0, 1]))
    extra = rng.random()
    if extra < 0.15:
        c.update(ts=0.05)
    elif extra < 0.3:
        c.update(omega=round(rng.uniform(0.05, 0.2), 3))
    elif extra < 0.45:
        c.update(rigid=1)
    elif extra < 0.6:
        c.update(recompute=1)
    return c


# ---------------------------------------------------------------------- inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _smooth(gen, channels, shape, spacing, rms):
    """Smooth random fields (channels, *shape) with `rms` over each voxel's channels: white noise
    on a grid `spacing` times coarser, interpolated."""
    small = [max(2, -(-a // spacing)) for a in shape]
    x = torch.randn([1, channels] + small, generator=gen, device="cuda")
    x = nnf.interpolate(x, size=tuple(shape), mode="trilinear", align_corners=True)[0]
    return x * (rms / x.square().sum(0).mean().sqrt())


def _grid(shape, dtype=torch.float32):
    return torch.stack(torch.meshgrid(*[torch.arange(a, device="cuda", dtype=dtype) for a in shape], indexing="ij"))


def _head(P, shape, tex):
    """Tissue intensities at the points P (3, D, H, W) of a head that fills the volume."""
    c = [(a - 1) / 2 for a in shape]
    ax = [0.42 * shape[0], 0.44 * shape[1], 0.40 * shape[2]]
    R = sum(((P[k] - c[k]) / ax[k]) ** 2 for k in range(3)).sqrt()
    edge = 0.6 * min(ax) / max(min(shape) / 160.0, 0.3)
    brain = torch.sigmoid((0.90 - R) * edge)
    I = 0.02 + 0.55 * torch.sigmoid((1.0 - R) * edge) * (1 - brain)
    I = I + brain * (0.25 + 0.30 * torch.sigmoid((0.86 - R) * edge) + 0.30 * torch.sigmoid((0.74 - R) * edge))
    vent = 0.0
    for side in (-1.0, 1.0):
        vc = [c[0], c[1] - 0.05 * shape[1], c[2] + side * 0.08 * shape[2]]
        va = [0.07 * shape[0], 0.16 * shape[1], 0.045 * shape[2]]
        rv = sum(((P[k] - vc[k]) / va[k]) ** 2 for k in range(3)).sqrt()
        vent = torch.maximum(torch.sigmoid((1.0 - rv) * min(va)), torch.as_tensor(vent, device="cuda"))
    I = I * (1 - vent) + 0.25 * vent
    q = torch.stack([P[2] / max(shape[2] - 1, 1), P[1] / max(shape[1] - 1, 1), P[0] / max(shape[0] - 1, 1)], -1) * 2 - 1
    return I + brain * nnf.grid_sample(tex[None], q[None], align_corners=True, padding_mode="border")[0, 0]


def _series(shape, N, seed):
    """N sessions of one head: (N, D, H, W) float32."""
    gen = _generator(seed)
    tex = _smooth(gen, 1, shape, 3, 0.04)
    x, d = _grid(shape), torch.zeros([3] + list(shape), device="cuda")
    out = torch.empty([N] + list(shape), device="cuda")
    for i in range(N):
        if i:
            d += _smooth(gen, 3, shape, 10, 0.5)
        I = _head(x + d, shape, tex)
        I *= 1.0 + 0.2 * torch.tanh(_smooth(gen, 1, shape, max(8, min(shape) // 3), 0.7))[0]
        a, b = (torch.randn(shape, generator=gen, device="cuda") for _ in range(2))
        out[i] = ((I.clamp_min(0) + 0.03 * a).square() + (0.03 * b).square()).sqrt()
    return out


def _shape(c):
    return [c["D"], c["H"], c["W"]]


def _velocities(c, seed):
    """(N-1, 3, d, h, w) velocities on the flow grid as a registration under way has them."""
    gen = _generator(seed + 77)
    nf = [(a + 1) // 2 for a in _shape(c)]
    return torch.stack([_smooth(gen, 3, nf, 6, 0.5) for _ in range(c["N"] - 1)])


def _rigid(c, seed):
    """(N-1, 6) angles of about a degree and translations of about half a voxel."""
    r = np.random.default_rng(int(seed) + 5).normal(size=(c["N"] - 1, 6)) * np.array([0.02] * 3 + [0.5] * 3)
    return r.astype(np.float32)


def _times(c):
    """Acquisition times: uneven gaps where the temporal regulariser is on, else the default."""
    return [i + 0.25 * (i % 3) for i in range(c["N"])] if c.get("ts") else None


def _disp_pair(c, seed):
    gen = _generator(seed)
    true = _smooth(gen, 3, _shape(c), 12, 1.5)
    est = 0.9 * true + _smooth(gen, 3, _shape(c), 6, 0.3) + 0.05
    roi = None
    if c.get("roi"):
        roi = (_head(_grid(_shape(c)) + true, _shape(c), torch.zeros([1] + _shape(c), device="cuda")) > 0.1).to(torch.uint8)
    return true, est, roi


def _volumes(c, seed):
    s = _series(_shape(c), 2, seed)
    return s[0].contiguous(), s[1].contiguous()


def _context(c):
    kw = dict(ALPHA, n_squarings=c["K"], window=c["window"], similarity=c["kind"], deterministic=c.get("det", 0),
              recompute_squaring=c.get("recompute", 0), alpha_ts=c.get("ts", 0.0), smooth_omega=c.get("omega", 0.0),
              rigid=c.get("rigid", 0))
    L = c.get("levels", 1)
    return m.Muster(_shape(c), c["N"], n_levels=L, steps_per_level=[c.get("steps", 1)] * L, **kw)


def prepare(case, seed):
    c, op = case, case["op"]
    if op == "similarity":
        F, W = _volumes(c, seed)
        return dict(case=c, F=F, W=W)
    if op == "exp":
        return dict(case=c, phi=_smooth(_generator(seed), 3, _shape(c), 6, c["rms"]))
    if op == "jacobian":
        return dict(case=c, u=_smooth(_generator(seed), 3, _shape(c), 12, 1.5))
    if op == "metrics":
        true, est, roi = _disp_pair(c, seed)
        return dict(case=c, true=true, est=est, roi=roi)
    reg = _context(c)
    imgs = _series(_shape(c), c["N"], seed)
    if op == "run":
        return dict(case=c, reg=reg, imgs=imgs)
    reg.set_images(imgs, times=_times(c))
    if c.get("rigid"):
        reg.set_level(0)
        reg.set_rigid(_rigid(c, seed))
    return dict(case=c, reg=reg, v=_velocities(c, seed))


def run(state):
    c = state["case"]
    op = c["op"]
    if op == "similarity":
        loss, grad = m.op_similarity(state["F"], state["W"], c["window"], c["kind"])
        return dict(loss=loss, grad=grad)
    if op == "exp":
        return m.op_exp(state["phi"], c["K"], float(c["sign"]))
    if op == "jacobian":
        return m.op_jacobian_det(state["u"])
    if op == "metrics":
        return m.op_deformation_metrics(state["true"], state["est"], state["roi"])
    reg = state["reg"]
    if op == "run":
        reg.set_images(state["imgs"])
        loss = reg.run()
        return dict(loss=loss, velocities=reg.velocities(c["levels"] - 1))
    grad = torch.empty_like(state["v"])
    out = dict(loss=reg.eval(state["v"], 0, grad), grad=grad)
    if c.get("rigid"):
        out["rigid_grad"] = reg.rigid(grad=True)[1].astype(np.float32)
    return out


# ---------------------------------------------------------------------- bytes and operations
def work(case):
    """Inputs read once and outputs written once; operations of the method with running box sums
    (the transforms of one field or pair: about 60 per trilinear vector sample, twice that with its
    adjoint; per pair-voxel about 140 for the warp, the window sums and their adjoints)."""
    c, op = case, case["op"]
    V = float(c["D"] * c["H"] * c["W"])
    if op == "similarity":
        return {"bytes": 12 * V, "flops": 60 * V}
    if op == "exp":
        return {"bytes": 24 * V, "flops": 60 * V * c["K"]}
    if op == "jacobian":
        return {"bytes": 16 * V, "flops": 30 * V}
    if op == "metrics":
        return {"bytes": (25 if c.get("roi") else 24) * V, "flops": 60 * V}
    N, P = c["N"], c["N"] * (c["N"] - 1)

    def step(V):
        Vf = V / 8
        return 140 * P * V + Vf * (180 * 2 * (N - 1) * c["K"] + 180 * (N - 1) * (N - 2) + 40 * (N - 1))

    vel = 12 * (N - 1) * V / 8
    if op == "eval":
        return {"bytes": 4 * N * V + 2 * vel, "flops": step(V)}
    return {"bytes": 4 * N * V + vel, "flops": sum(c["steps"] * step(V / 8**l) for l in range(c["levels"]))}


# ---------------------------------------------------------------------- the same in 64 bits
class _Sample(torch.autograd.Function):
    """Trilinear samples of f (C, D, H, W) at index coordinates q (3, ...), clamped to the grid;
    the derivative is 0 along an axis whose coordinate was clamped."""

    @staticmethod
    def _cells(f, q):
        n = f.shape[1:]
        i0, i1, t, inside = [], [], [], []
        for a in range(3):
            c = q[a].clamp(0, n[a] - 1)
            lo = c.floor()
            i0.append(lo.long())
            i1.append((lo.long() + 1).clamp_max(n[a] - 1))
            t.append(c - lo)
            inside.append(c == q[a])
        return n, i0, i1, t, inside

    @staticmethod
    def _corners(n, i0, i1, t):
        for b in range(8):
            bits = (b >> 2 & 1, b >> 1 & 1, b & 1)
            z, y, x = (i1[a] if bits[a] else i0[a] for a in range(3))
            yield bits, (z * n[1] + y) * n[2] + x, [t[a] if bits[a] else 1 - t[a] for a in range(3)]

    @staticmethod
    def forward(ctx, f, q):
        ctx.save_for_backward(f, q)
        n, i0, i1, t, _ = _Sample._cells(f, q)
        flat = f.reshape(f.shape[0], -1)
        out = 0
        for _, o, w in _Sample._corners(n, i0, i1, t):
            out = out + flat[:, o] * (w[0] * w[1] * w[2])
        return out

    @staticmethod
    def backward(ctx, g):
        f, q = ctx.saved_tensors
        n, i0, i1, t, inside = _Sample._cells(f, q)
        flat = f.reshape(f.shape[0], -1)
        gf = torch.zeros_like(flat) if ctx.needs_input_grad[0] else None
        gq = [0, 0, 0] if ctx.needs_input_grad[1] else None
        for bits, o, w in _Sample._corners(n, i0, i1, t):
            if gf is not None:
                gf.index_add_(1, o.reshape(-1), (g * (w[0] * w[1] * w[2])).reshape(f.shape[0], -1))
            if gq is not None:
                s = (flat[:, o] * g).sum(0)
                for a in range(3):
                    b, c = (k for k in range(3) if k != a)
                    gq[a] = gq[a] + (s if bits[a] else -s) * w[b] * w[c]
        if gq is not None:
            gq = torch.stack([x * i for x, i in zip(gq, inside)])
        return (gf.reshape(f.shape) if gf is not None else None), gq


class _Box(torch.autograd.Function):
    """Sums over the w^3 windows that lie inside the volume."""

    @staticmethod
    def _sum(x, w):
        for a in range(3):
            n = x.shape[a] - w + 1
            y = x.narrow(a, 0, n).clone()
            for k in range(1, w):
                y += x.narrow(a, k, n)
            x = y
        return x

    @staticmethod
    def forward(ctx, x, w):
        ctx.w = w
        return _Box._sum(x, w)

    @staticmethod
    def backward(ctx, g):
        return _Box._sum(nnf.pad(g, [ctx.w - 1] * 6), ctx.w), None


def _similarity64(F, W, w, kind, eps=1e-6):
    n = float(w**3)
    f, v = F - F.mean(), W - W.mean().detach()
    sf, sv = _Box._sum(f, w), _Box.apply(v, w)
    sff, svv = _Box._sum(f * f, w) - sf * sf / n, _Box.apply(v * v, w) - sv * sv / n
    sfv = _Box.apply(f * v, w) - sf * sv / n
    if kind == 0:
        return ((svv - sfv * sfv / (sff + eps)) / n).mean()
    return (1 - sfv / (sff * svv + eps).sqrt()).mean()


def _exp64(phi, K, x, sign=1.0):
    u = phi * (sign / 2**K)
    for _ in range(K):
        u = u + _Sample.apply(u, x + u)
    return u


def _smooth64(theta, omega, spacing):
    f2 = 0
    for a in range(3):
        f = torch.fft.fftfreq(theta.shape[2 + a], d=spacing, device="cuda", dtype=torch.float64)
        f2 = f2 + f.reshape([-1 if b == a else 1 for b in range(3)]) ** 2
    return torch.fft.ifftn(torch.fft.fftn(theta, dim=(2, 3, 4)) * torch.exp(-0.5 * f2 / omega**2), dim=(2, 3, 4)).real


def _rotation64(a):
    R = torch.eye(3, dtype=torch.float64, device="cuda")
    for k in range(3):
        u, w = (k + 1) % 3, (k + 2) % 3
        c, s, M = torch.cos(a[k]), torch.sin(a[k]), {}
        M[k, k] = torch.ones_like(c)
        M[u, u] = M[w, w] = c
        M[u, w], M[w, u] = -s, s
        z = torch.zeros_like(c)
        R = R @ torch.stack([torch.stack([M.get((i, j), z) for j in range(3)]) for i in range(3)])
    return R


def _eval64(c, imgs, v, rho, times):
    """Loss, dL/dv and (with rigid motion) dL/drho of a series."""
    N, F, K = c["N"], c["N"] - 1, c["K"]
    ni, nf = list(imgs.shape[1:]), list(v.shape[2:])
    th = v.double().requires_grad_()
    phi = _smooth64(th, float(np.float32(c["omega"])), 2.0) if c.get("omega") else th
    x = _grid(nf, torch.float64)
    U = {}
    for i in range(F):
        U[i + 1, i] = _exp64(phi[i], K, x)
        U[i, i + 1] = _exp64(phi[i], K, x, -1.0)
    for d in range(2, N):
        for i in range(N - d):
            U[i + d, i] = U[i + d - 1, i] + _Sample.apply(U[i + d, i + d - 1], x + U[i + d - 1, i])
        for i in range(d, N):
            U[i - d, i] = U[i - d + 1, i] + _Sample.apply(U[i - d, i - d + 1], x + U[i - d + 1, i])
    r = torch.tensor(rho, dtype=torch.float64, device="cuda").requires_grad_() if rho is not None else None
    p = _grid(ni, torch.float64)
    centre = torch.tensor([(a - 1) / 2 for a in ni], dtype=torch.float64, device="cuda")
    total, keys, grads, rgrad = 0.0, list(U), [], 0
    for k, i in keys:
        u = U[k, i].detach().requires_grad_()
        q = p + 2 * _Sample.apply(u, (p - 0.5) / 2)
        if r is not None and i > 0:
            R = _rotation64(r[i - 1, :3])
            q = q + torch.einsum("ab,bdhw->adhw", R - torch.eye(3, dtype=torch.float64, device="cuda"), p)
            q = q + (centre - R @ centre + r[i - 1, 3:]).reshape(3, 1, 1, 1)
        W = _Sample.apply(imgs[k].double()[None], q)[0]
        s = _similarity64(imgs[i].double(), W, c["window"], c["kind"])
        got = torch.autograd.grad(s, [u] + ([r] if r is not None and i > 0 else []))
        grads.append(got[0])
        if len(got) > 1:
            rgrad = rgrad + got[1]
        total += float(s)
    a_ss, a_l2, a_ts = ALPHA["alpha_ss"], ALPHA["alpha_l2"], c.get("ts", 0.0)
    reg = a_l2 * phi.square().sum() / math.prod(nf) / F
    for a in range(3):
        if nf[a] > 1:
            d = phi.diff(dim=2 + a).square().sum() / (math.prod(nf) * (nf[a] - 1) / nf[a])
            reg = reg + a_ss * d / F
    if a_ts and N >= 3:
        t = times or list(range(N))
        rate = torch.stack([phi[i] / (t[i + 1] - t[i]) for i in range(F)])
        reg = reg + a_ts * rate.diff(dim=0).square().sum() / math.prod(nf) / (N - 2)
    torch.autograd.backward([U[k] for k in keys] + [reg], grads + [torch.ones_like(reg)])
    out = dict(loss=np.float64(total + float(reg)), grad=th.grad)
    if r is not None:
        out["rigid_grad"] = rgrad
    return out


def exact(case, seed):
    c, op = case, case["op"]
    if op == "run":
        return None
    if op == "similarity":
        F, W = _volumes(c, seed)
        w = W.double().requires_grad_()
        s = _similarity64(F.double(), w, c["window"], c["kind"])
        s.backward()
        return dict(loss=s.detach(), grad=w.grad)
    if op == "exp":
        phi = _smooth(_generator(seed), 3, _shape(c), 6, c["rms"]).double()
        return _exp64(phi, c["K"], _grid(_shape(c), torch.float64), float(c["sign"]))
    if op == "jacobian":
        u = _smooth(_generator(seed), 3, _shape(c), 12, 1.5).double()
        M = torch.stack([torch.stack(torch.gradient(u[k])) for k in range(3)])
        M = M + torch.eye(3, dtype=torch.float64, device="cuda").reshape(3, 3, 1, 1, 1)
        return ((M[0, 0] * (M[1, 1] * M[2, 2] - M[1, 2] * M[2, 1])) - M[0, 1] * (M[1, 0] * M[2, 2] - M[1, 2] * M[2, 0])
                + M[0, 2] * (M[1, 0] * M[2, 1] - M[1, 1] * M[2, 0]))
    if op == "metrics":
        true, est, roi = _disp_pair(c, seed)
        keep = roi.bool().reshape(-1) if roi is not None else torch.ones(true[0].numel(), dtype=torch.bool, device="cuda")
        t, e = true.double().reshape(3, -1)[:, keep], est.double().reshape(3, -1)[:, keep]
        mt, me = t.mean(1, keepdim=True), e.mean(1, keepdim=True)
        tc, ec = t - mt, e - me
        A = (ec @ tc.T) @ torch.linalg.inv(tc @ tc.T)
        return dict(A=A, B=A.trace() / 3, Eu=(t - e).square().sum(0).sqrt().mean(),
                    PCC=(tc * ec).sum() / (tc.square().sum().sqrt() * ec.square().sum().sqrt()), b=(me - A @ mt)[:, 0],
                    count=None)
    if c["N"] * (c["N"] - 1) * float(c["D"] * c["H"] * c["W"]) > EXACT_PAIR_VOXELS:
        return None
    return _eval64(c, _series(_shape(c), c["N"], seed), _velocities(c, seed), _rigid(c, seed) if c.get("rigid") else None,
                   _times(c))
