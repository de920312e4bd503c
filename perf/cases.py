"""Performance cases: the calls that a user of the package makes, over the sizes they make them at.

A case names one operation and its sizes:

    reconstruct  particles -> CIC density -> smoothing, floor, mean 1 -> solve -> displacement and delta_r
    solve        density -> potential, FP64 or mixed precision
    batch        several densities of uneven sizes solved together
    gradient     loss on the output of the FP64 solve, differentiated with respect to the density
    density      particles -> NGP / CIC / TSC density -> smoothing, floor, mean 1
    displace     potential and density -> displacement and delta_r
    gaussianise  rank mapping of delta_r onto Gaussian quantiles

Inputs are seeded Zel'dovich particles (P(k) ~ k^-1.5 exp(-k^2), as in ``synth``) and what plain torch makes of them.
``exact`` evaluates the same quantities in 64 bits with torch alone.
"""
from __future__ import annotations

import math

import torch

from paper_1709_06350_gb300 import autograd, autotune, recon

# sides whose multigrid hierarchy ends at 16^3 or below: 2^k times 4, 6, 10 or 14
SIDES = (64, 80, 96, 112, 128, 160, 192, 224, 256, 320, 384, 448, 512)
FLOOR = 0.05


def _case(name, op, N, L, sigma, R, **more):
    return {"name": name, "op": op, "N": N, "L": float(L), "sigma": sigma, "R": float(R), **more}


def listed():
    return [
        # the headline workload: one snapshot of 512^3 particles in 512 Mpc/h, the whole method, tuned schedule
        _case("reconstruct_512", "reconstruct", 512, 512, 1.0, 2.0, tuned=True),
        # a whole reconstruction of a small mock, where launches and host reads count
        _case("reconstruct_96", "reconstruct", 96, 192, 0.8, 4.0, tuned=False),
        # the smallest solve of the batched workload: latency
        _case("solve_mixed_64", "solve", 64, 128, 0.8, 4.0, precision="mixed"),
        # a side that is no multiple of 64 in a box whose cell is no power of two
        _case("solve_mixed_160", "solve", 160, 500, 0.8, 6.25, precision="mixed"),
        # an ordinary solve at the default options
        _case("solve_mixed_256", "solve", 256, 512, 0.8, 4.0, precision="mixed"),
        # a large solve at the default options, beyond the tuned sizes
        _case("solve_mixed_768", "solve", 768, 768, 1.0, 2.0, precision="mixed"),
        # the paper's 128^3 grid in plain FP64, as for a reference answer
        _case("solve_f64_128", "solve", 128, 256, 0.8, 4.0, precision="f64"),
        # many mocks of uneven sizes together, two of each size of the batched workload, tuned schedules
        _case("batch_10", "batch", 256, 512, 0.8, 4.0, count=10),
        # forward and backward: gradient of a loss on psi and delta_r with respect to the density
        _case("gradient_128", "gradient", 128, 256, 0.8, 4.0),
        # one-point Gaussianisation of a reconstructed field (delta_r of the output step has FP32 digits)
        _case("gaussianise_256", "gaussianise", 256, 512, 0.8, 4.0, digits=32),
        # density by TSC from 256^3 tracers in the paper's 500 Mpc/h box
        _case("density_tsc_256", "density", 256, 500, 0.8, 4.0, scheme="tsc", particles=256),
        # the output step alone, 384^3 in 500 Mpc/h
        _case("displace_384", "displace", 384, 500, 0.8, 2.7),
    ]


def draw(rng):
    op = rng.choice(("reconstruct", "solve", "solve", "solve", "batch", "gradient", "density", "displace", "gaussianise"))
    more, most = {}, 512
    if op == "reconstruct":
        more["tuned"] = rng.random() < 0.5
    elif op == "solve":
        more["precision"] = rng.choice(("mixed", "mixed", "f64"))
        most = 192 if more["precision"] == "f64" else 512
    elif op == "batch":
        more["count"], most = rng.randint(3, 12), 192
    elif op == "gradient":
        most = 160
    elif op == "density":
        more["scheme"] = rng.choice(("ngp", "cic", "tsc"))
    N = rng.choice([s for s in SIDES if s <= most])
    if op == "gaussianise":
        more["digits"] = rng.choice((32, 64))   # delta_r of the output step, or of its FP64 form
    if op == "density":
        # tracer : mesh ratios of 1 : 8, 1 : 1 and 8 : 1 per volume
        more["particles"] = rng.choice((N // 2, N, N, min(2 * N, 512)))
    # cells of 1 to 4 Mpc/h, half of them powers of two
    h = float(rng.choice((1, 2, 4))) if rng.random() < 0.5 else round(math.exp(rng.uniform(0.0, math.log(4.0))), 3)
    sigma = round(rng.uniform(0.4, 0.9), 3)
    R = round(rng.uniform(1.8, 2.6) * h, 3)
    c = _case("", op, N, N * h, sigma, R, **more)
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs in plain torch, 64 bits
def _dev():
    return torch.device("cuda", torch.cuda.current_device()) if torch.cuda.is_available() else torch.device("cpu")


def _k(N, L):
    kf = 2.0 * math.pi / L
    k = torch.fft.fftfreq(N, d=1.0 / N, dtype=torch.float64, device=_dev()) * kf
    kz = torch.arange(N // 2 + 1, dtype=torch.float64, device=_dev()) * kf
    return k[:, None, None], k[None, :, None], kz[None, None, :]


def _linear(n, L, sigma, seed):
    """Transform of a seeded Gaussian field of rms sigma, divided by k^2."""
    g = torch.Generator(device=_dev()).manual_seed(int(seed) * 7919 + 17)
    dh = torch.fft.rfftn(torch.randn((n, n, n), generator=g, dtype=torch.float64, device=_dev()))
    kx, ky, kz = _k(n, L)
    k2 = kx * kx + ky * ky + kz * kz
    k2[0, 0, 0] = 1.0
    dh *= k2 ** -0.375 * torch.exp(-0.5 * k2)
    dh[0, 0, 0] = 0.0
    rms = torch.fft.irfftn(dh, s=(n, n, n)).square().mean().sqrt()
    return dh * (sigma / (rms * k2))


def _particles(n, L, sigma, seed):
    """n^3 Zel'dovich particles of a seeded Gaussian field, [n^3, 3]."""
    dh = _linear(n, L, sigma, seed)
    kx, ky, kz = _k(n, L)
    q = (torch.arange(n, dtype=torch.float64, device=_dev()) + 0.5) * (L / n)
    pos = torch.empty((n, n, n, 3), dtype=torch.float64, device=_dev())
    for d, k in enumerate((kx, ky, kz)):
        shape = [1, 1, 1]
        shape[d] = n
        pos[..., d] = torch.remainder(torch.fft.irfftn(1j * k * dh, s=(n, n, n)) + q.view(shape), L)
    return pos.view(-1, 3)


def _assign(pos, N, L, scheme):
    """Density of mean 1 on N^3 by NGP, CIC or TSC."""
    rho = torch.zeros(N ** 3, dtype=torch.float64, device=pos.device)
    for p in pos.split(1 << 25):
        u = p * (N / L)
        if scheme == "cic":
            u = u - 0.5
        i = torch.floor(u)
        t = (u - i).unbind(1)
        if scheme == "ngp":
            w, first = [[torch.ones_like(x)] for x in t], 0
        elif scheme == "cic":
            w, first = [[1.0 - x, x] for x in t], 0
        else:
            w, first = [[0.5 * (1.0 - x) ** 2, 0.75 - (x - 0.5) ** 2, 0.5 * x * x] for x in t], -1
        i = i.long().unbind(1)
        at = [[torch.remainder(i[d] + first + s, N) for s in range(len(w[d]))] for d in range(3)]
        for a in range(len(w[0])):
            for b in range(len(w[0])):
                row, wr = (at[0][a] * N + at[1][b]) * N, w[0][a] * w[1][b]
                for c in range(len(w[0])):
                    rho.index_add_(0, row + at[2][c], wr * w[2][c])
    return rho.view(N, N, N) * (N ** 3 / pos.shape[0])


def _smooth(rho, L, R):
    """Gaussian window of width R, floor, mean 1."""
    kx, ky, kz = _k(rho.shape[0], L)
    h = torch.fft.rfftn(rho)
    for k in (kx, ky, kz):
        h *= torch.exp(-0.5 * R * R * k * k)
    b = torch.fft.irfftn(h, s=rho.shape).clamp_(min=FLOOR)
    return b / b.mean()


def _density(c, N, L, seed):
    return _smooth(_assign(_particles(N, L, c["sigma"], seed), N, L, "cic"), L, c["R"]).contiguous()


def _skewed(c, N, L, seed):
    """A field with the range of delta_r (below 3, skewed), in as many digits as the output step gives it."""
    kx, ky, kz = _k(N, L)
    k2 = kx * kx + ky * ky + kz * kz
    d = torch.fft.irfftn(_linear(N, L, c["sigma"], seed) * k2 * torch.exp(-0.5 * c["R"] ** 2 * k2), s=(N, N, N))
    x = 3.0 - 3.0 * torch.exp(-d / 3.0)
    return (x.float().double() if c["digits"] == 32 else x).contiguous()


def _potential(b, L):
    """The linear potential of a density: lap phi = (b - mean b) limited to |delta| < 0.8."""
    d = b.clamp(max=1.8) - 1.0
    return _inverse_laplacian(d, L / b.shape[0]).contiguous()


def _batch_sizes(c):
    sizes = [s for s in (64, 96, 128, 192, 256) if s <= c["N"]]
    return [sizes[i % len(sizes)] for i in range(c["count"])]


# ---------------------------------------------------------------- the calls
def prepare(case, seed):
    c, N, L, op = case, case["N"], case["L"], case["op"]
    s = {"case": c}
    mixed = recon.RECON_MIXED
    if op == "reconstruct":
        s["pos"] = _particles(N, L, c["sigma"], seed)
    elif op == "density":
        s["pos"] = _particles(c["particles"], L, c["sigma"], seed)
    elif op == "batch":
        sizes = _batch_sizes(c)
        boxes = [L / N * n for n in sizes]
        s["b"] = [_density(c, n, box, 100 * seed + i) for i, (n, box) in enumerate(zip(sizes, boxes))]
        s["phi"] = [torch.zeros_like(b) for b in s["b"]]
    elif op == "gaussianise":
        s["field"] = _skewed(c, N, L, seed)
    else:
        s["b"] = _density(c, N, L, seed)
    if op == "displace":
        s["phi"] = _potential(s["b"], L)
    if op == "gradient":
        g = torch.Generator(device=_dev()).manual_seed(int(seed))
        s["w"] = [torch.randn(n, generator=g, dtype=torch.float64, device=_dev()) for n in ((3, N, N, N), (N, N, N))]
        s["b"].requires_grad_(True)
    torch.cuda.empty_cache()   # the handle's workspace does not come from torch's pool
    if op == "batch":
        s["solver"] = recon.Batch(sizes, boxes)
        autotune.apply(s["solver"])
    else:
        f64 = op == "gradient" or c.get("precision") == "f64"
        s["solver"] = recon.Solver(N, L, recon.RECON_F64 if f64 else mixed)
        if c.get("tuned"):
            autotune.apply(s["solver"])
    return s


def run(s):
    c, solver = s["case"], s["solver"]
    op = c["op"]
    if op == "reconstruct":
        b = solver.smooth_density(solver.deposit_cic(s["pos"]), c["R"])
        phi, stats = solver.solve(b, tol=1e-8, max_cycles=40)
        psi, dl = solver.displace(phi, b)
        return {"b": b, "phi": phi, "c": stats["compat_c"], "psi": psi, "delta_r": dl}
    if op == "solve":
        phi, stats = solver.solve(s["b"], tol=1e-10 if c["precision"] == "f64" else 1e-8, max_cycles=40)
        return {"phi": phi, "c": stats["compat_c"]}
    if op == "batch":
        phis, stats = solver.solve(s["b"], phis=s["phi"], tol=1e-8, max_cycles=40)
        return {"phi": phis, "c": [t["compat_c"] for t in stats]}
    if op == "gradient":
        b = s["b"]
        phi = autograd.solve(b, solver, tol=1e-11)
        psi, dl = autograd.displace(phi, b, solver)
        loss = (psi * s["w"][0]).sum() + (dl * dl * s["w"][1]).sum()
        (grad,) = torch.autograd.grad(loss, b)
        return {"psi": psi.detach(), "delta_r": dl.detach(), "grad": grad}
    if op == "density":
        rho = solver.deposit(s["pos"], c["scheme"])
        return {"rho": rho, "b": solver.smooth_density(rho, c["R"])}
    if op == "displace":
        psi, dl = solver.displace(s["phi"], s["b"])
        return {"psi": psi, "delta_r": dl}
    if op == "gaussianise":
        return solver.gaussianise(s["field"])
    raise ValueError(op)


def work(case):
    """Bytes of the inputs and outputs, each moved once, and the operations that no evaluation of the result goes without
    (for a solve, one residual: about 60 per cell)."""
    c, n, op = case, case["N"] ** 3, case["op"]
    if op == "reconstruct":
        return {"bytes": 24 * n + 48 * n, "flops": 250 * n}
    if op == "batch":
        n = sum(m ** 3 for m in _batch_sizes(c))
    if op in ("solve", "batch"):
        return {"bytes": 16 * n, "flops": 60 * n}
    if op == "gradient":
        return {"bytes": (8 + 32 + 32 + 8) * n, "flops": 400 * n}
    if op == "density":
        p = c["particles"] ** 3
        corners = {"ngp": 1, "cic": 8, "tsc": 27}[c["scheme"]]
        return {"bytes": 24 * p + 16 * n, "flops": 2 * corners * p + 60 * n}
    if op == "displace":
        return {"bytes": 16 * n + 32 * n, "flops": 100 * n}
    return {"bytes": 16 * n, "flops": 20 * n}


# ---------------------------------------------------------------- the same results in plain torch, 64 bits
def _laplacian_symbol(N, h, dtype):
    c = 2.0 * torch.cos(2.0 * math.pi * torch.arange(N, dtype=torch.float64, device=_dev()) / N) - 2.0
    s = (c[:, None, None] + c[None, :, None] + c[None, None, :N // 2 + 1]) / (h * h)
    s[0, 0, 0] = 1.0
    return s.to(dtype)


def _inverse_laplacian(f, h, symbol=None):
    s = _laplacian_symbol(f.shape[0], h, f.dtype) if symbol is None else symbol
    g = torch.fft.rfftn(f) / s
    g[0, 0, 0] = 0.0
    return torch.fft.irfftn(g, s=f.shape)


def _at(a, *shift):
    """a at (i, j, k) + shift."""
    return torch.roll(a, [-x for x in shift], (0, 1, 2))


PAIRS = ((0, 1), (1, 2), (0, 2))


def _unit(d, s=1):
    return tuple(s if x == d else 0 for x in range(3))


def _second(a, d, h):
    return (_at(a, *_unit(d)) + _at(a, *_unit(d, -1)) - 2.0 * a) / (h * h)


def _cross(a, p, h):
    def e(x, y):
        v = [0, 0, 0]
        v[p[0]], v[p[1]] = x, y
        return _at(a, *v)
    return ((e(1, 1) + e(-1, -1)) - (e(1, -1) + e(-1, 1))) / (4.0 * h * h)


def _hessian(phi, h):
    """A = I + H phi: (xx, yy, zz, xy, yz, xz)."""
    return [1.0 + _second(phi, d, h) for d in range(3)] + [_cross(phi, p, h) for p in PAIRS]


def _det(A):
    xx, yy, zz, xy, yz, xz = A
    return xx * (yy * zz - yz * yz) - xy * (xy * zz - yz * xz) + xz * (xy * yz - yy * xz)


def _adj(A):
    xx, yy, zz, xy, yz, xz = A
    return [yy * zz - yz * yz, xx * zz - xz * xz, xx * yy - xy * xy,
            xz * yz - xy * zz, xy * xz - xx * yz, xy * yz - xz * yy]


def _jacobian(adj, e, h):
    out = sum(adj[d] * _second(e, d, h) for d in range(3))
    return out + 2.0 * sum(adj[3 + n] * _cross(e, p, h) for n, p in enumerate(PAIRS))


def _jacobian_t(adj, e, h):
    out = sum(_second(adj[d] * e, d, h) for d in range(3))
    return out + 2.0 * sum(_cross(adj[3 + n] * e, p, h) for n, p in enumerate(PAIRS))


def _krylov(apply, rhs, rtol, most=150):
    """BiCGSTAB."""
    x = torch.zeros_like(rhs)
    r, r0 = rhs.clone(), rhs.clone()
    rho = alpha = omega = 1.0
    v = p = torch.zeros_like(rhs)
    goal = rtol * float(rhs.norm())
    for _ in range(most):
        rho, old = float((r0 * r).sum()), rho
        if rho == 0.0:
            break
        p = r + (rho / old) * (alpha / omega) * (p - omega * v)
        v = apply(p)
        alpha = rho / float((r0 * v).sum())
        s = r - alpha * v
        t = apply(s)
        tt = float((t * t).sum())
        omega = float((t * s).sum()) / tt if tt > 0.0 else 0.0
        x = x + alpha * p + omega * s
        r = s - omega * t
        if omega == 0.0 or float(r.norm()) < goal:
            break
    return x


def _solved(b, L):
    """(phi, c) with det(I + H phi) = b + c and mean(phi) = 0: Newton steps, each linear system by preconditioned
    BiCGSTAB in 32 bits, residuals in 64."""
    N = b.shape[0]
    h = L / N
    symbol = _laplacian_symbol(N, h, torch.float32)
    phi = torch.zeros_like(b)

    def residual(p, target):
        A = _hessian(p, h)
        r = target - _det(A)
        return A, r - r.mean()

    for t in (0.3, 0.6, 0.85, 1.0):
        target = 1.0 + t * (b - 1.0)
        A, r = residual(phi, target)
        size = float(target.sub(1.0).norm())
        for _ in range(30):
            rel = float(r.norm()) / size
            if rel < (1e-2 if t < 1.0 else 1e-14):
                break
            adj = [a.float() for a in _adj(A)]
            inv = 3.0 / (adj[0] + adj[1] + adj[2])
            inv = torch.where(inv > 0, inv.clamp(max=50.0), torch.ones_like(inv))
            mean = inv.mean()

            def project(w):
                return w - (w.mean() / mean) * inv

            def apply(y):
                return project(inv * _jacobian(adj, _inverse_laplacian(y, h, symbol), h))
            scale = float(r.abs().max())
            y = _krylov(apply, project(inv * (r / scale).float()), 1e-3)
            e = _inverse_laplacian(y, h, symbol).double() * scale
            step = 1.0
            while True:
                A2, r2 = residual(phi + step * e, target)
                if float(r2.norm()) < float(r.norm()) or step < 0.02:
                    break
                step *= 0.5
            if float(r2.norm()) >= float(r.norm()):
                break   # the floor of 64 bits
            phi, A, r = phi + step * e, A2, r2
            phi = phi - phi.mean()
    return phi, float((_det(_hessian(phi, h)) - b).mean())


def _solved_adjoint(phi, g, L):
    """lam with J^T lam + mu 1 = g, sum(lam) = 0."""
    h = L / phi.shape[0]
    symbol = _laplacian_symbol(phi.shape[0], h, torch.float32)
    adj = _adj(_hessian(phi, h))
    low = [a.float() for a in adj]
    inv = 3.0 / (low[0] + low[1] + low[2])
    inv = torch.where(inv > 0, inv.clamp(max=50.0), torch.ones_like(inv))
    mean = inv.mean()

    def lift(y):
        z = _inverse_laplacian(y, h, symbol)
        return inv * (z - (z * inv).mean() / mean)

    def apply(y):
        w = _jacobian_t(low, lift(y), h)
        return w - w.mean()
    lam = torch.zeros_like(g)
    goal = 1e-14 * float(g.norm())
    best = math.inf
    for _ in range(30):
        r = g - _jacobian_t(adj, lam, h)
        r = r - r.mean()
        if float(r.norm()) < goal or float(r.norm()) > 0.9 * best:
            break
        best = float(r.norm())
        scale = float(r.abs().max())
        lam = lam + lift(_krylov(apply, (r / scale).float(), 1e-3)).double() * scale
        lam = lam - lam.mean()
    return lam


def _displaced(phi, b, L):
    """psi and delta_r."""
    N = phi.shape[0]
    h = L / N
    grad = [(_at(phi, *_unit(d)) - _at(phi, *_unit(d, -1))) / (2.0 * h) for d in range(3)]
    A = _hessian(phi, h)
    adj = _adj(A)
    v = 3.0 - (adj[0] + adj[1] + adj[2]) / _det(A)
    num = torch.zeros(N ** 3, dtype=torch.float64, device=phi.device)
    den = torch.zeros_like(num)
    cells = torch.arange(N, dtype=torch.float64, device=phi.device)
    at, w = [], []
    for d in range(3):
        shape = [1, 1, 1]
        shape[d] = N
        u = grad[d] / h + cells.view(shape)
        i = torch.floor(u.detach())
        f = u - i
        i = i.long()
        at.append([torch.remainder(i, N).reshape(-1), torch.remainder(i + 1, N).reshape(-1)])
        w.append([(1.0 - f).reshape(-1), f.reshape(-1)])
        del u, i, f
    bv, bb = (b * v).reshape(-1), b.reshape(-1)
    del A, adj, v
    for x in range(2):
        for y in range(2):
            for z in range(2):
                id_ = (at[0][x] * N + at[1][y]) * N + at[2][z]
                wt = w[0][x] * w[1][y] * w[2][z]
                num = num.index_add(0, id_, bv * wt)
                den = den.index_add(0, id_, bb * wt)
    return -torch.stack(grad), (num / den.clamp(min=1e-12)).view(N, N, N)


def exact(case, seed):
    c, N, L, op = case, case["N"], case["L"], case["op"]
    if op == "density":
        rho = _assign(_particles(c["particles"], L, c["sigma"], seed), N, L, c["scheme"])
        return {"rho": rho, "b": _smooth(rho, L, c["R"])}
    if op == "reconstruct":
        b = _density(c, N, L, seed)
        if N > 160:   # the solve takes too long here
            return {"b": b, "phi": None, "c": None, "psi": None, "delta_r": None}
        phi, comp = _solved(b, L)
        psi, dl = _displaced(phi, b, L)
        return {"b": b, "phi": phi, "c": comp, "psi": psi, "delta_r": dl}
    if op == "solve":
        if N > 256:
            return None
        phi, comp = _solved(_density(c, N, L, seed), L)
        return {"phi": phi, "c": comp}
    if op == "batch":
        got = []
        for i, n in enumerate(_batch_sizes(c)):
            box = L / N * n
            got.append(_solved(_density(c, n, box, 100 * seed + i), box) if n <= 128 else (None, None))
        return {"phi": [g[0] for g in got], "c": [g[1] for g in got]}
    if op == "displace":
        b = _density(c, N, L, seed)
        psi, dl = _displaced(_potential(b, L), b, L)
        return {"psi": psi, "delta_r": dl}
    if op == "gaussianise":
        x = _skewed(c, N, L, seed).reshape(-1)
        n = x.numel()
        order = torch.sort(x, stable=True).indices
        z = torch.special.ndtri((torch.arange(n, dtype=torch.float64, device=x.device) + 0.5) / n)
        out = torch.empty_like(x)
        out[order] = x.mean() + x.std(unbiased=False) * z
        return out.view(N, N, N)
    if op == "gradient":
        b = _density(c, N, L, seed)
        g = torch.Generator(device=_dev()).manual_seed(int(seed))
        w = [torch.randn(n, generator=g, dtype=torch.float64, device=_dev()) for n in ((3, N, N, N), (N, N, N))]
        phi, _ = _solved(b, L)
        phi.requires_grad_(True)
        b.requires_grad_(True)
        psi, dl = _displaced(phi, b, L)
        gphi, gb = torch.autograd.grad((psi * w[0]).sum() + (dl * dl * w[1]).sum(), (phi, b))
        lam = _solved_adjoint(phi.detach(), gphi, L)
        return {"psi": psi.detach(), "delta_r": dl.detach(), "grad": gb + lam}
    raise ValueError(op)
