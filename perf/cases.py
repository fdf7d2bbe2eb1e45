"""Performance cases: what a user of this framework has it compute, through its public entry points.

A case is a plain dict; its ``kind`` names one of the stages of the method:
  volume     field of one solved sample on a 3-D grid (``Plan.synthesize``)
  fresh      the same for a solution that has just come in (``Plan.set_layers`` + ``synthesize``)
  sweep      many wavelengths as one batch (``BatchedPlan.synthesize``)
  points     field at lateral points on every plane (``Plan.synthesize_points``)
  solve      refractive-index sample -> modes and amplitudes (``Solver.solve``)
  grad       loss and gradient of the learned surrogate (``Surrogate.forward_backward``)
  infer      field and error estimate of the surrogate (``Surrogate.infer``)
The copy-bound host-memory call (``synthesize_host``) is left to the benchmark, which times it
beside the machine's copy rates.

``listed`` gives the fixed cases, ``draw`` more of the same ranges, ``prepare`` the inputs and the plan or handle
that a program keeps, ``run`` one pass, ``work`` the bytes and operations a pass cannot do
without and ``exact`` the outputs in 64 bits.
"""
import math

import numpy as np
import torch

import paper_2404_07293_gb300 as scw

GRID, MODES, SLICES, IN_GRID, WIDTH = 64, 16, 8, 32, 32  # the surrogate's configuration
INTERIOR = 0.25  # layer thickness in wavelengths of the solved samples


def listed():
    return [
        # the tiny sphere: 16x16x4 voxels, 7x7 orders. A small unit cell viewed interactively; launches count
        dict(name="sphere_small", kind="volume", U=7, V=7, L=4, per_layer=8, Fx=64, Fy=64, precision="split_bf16",
             illuminations=1, tiles=1, outside=0),
        # the headline workload: one wavelength, 21x21 orders, 32 layers, 256^3 voxels, the plan replayed per sample
        dict(name="volume_256", kind="volume", U=21, V=21, L=32, per_layer=8, Fx=256, Fy=256, precision="split_bf16",
             illuminations=1, tiles=1, outside=0),
        # the plain FP32 path at the surrogate study's 15x15 orders: users who want no split precision
        dict(name="volume_fp32", kind="volume", U=15, V=15, L=16, per_layer=8, Fx=128, Fy=128, precision="fp32",
             illuminations=1, tiles=1, outside=0),
        # microscopy: 16 incident fields of one solved sample at camera resolution
        dict(name="illuminations_16", kind="volume", U=21, V=21, L=32, per_layer=8, Fx=128, Fy=128,
             precision="split_bf16", illuminations=16, tiles=1, outside=0),
        # a design or reconstruction loop: every pass brings another solution, odd sizes, planes above and below
        # the sample, an offset grid and an objective's pupil
        dict(name="fresh_solution", kind="fresh", U=15, V=13, L=12, per_layer=7, Fx=200, Fy=136,
             precision="split_bf16", illuminations=1, tiles=1, outside=6),
        # mid-infrared spectroscopy: every fourth wavenumber of the 128-point sweep, 9x9 to 25x25 orders
        dict(name="sweep_32", kind="sweep", items=32, of=128, Fx=128, Fy=128, planes=64, precision="split_bf16"),
        # one x-z cross-section through the headline sample
        dict(name="xz_plane", kind="points", U=21, V=21, L=32, per_layer=8, points=256, line=True,
             precision="split_bf16"),
        # a zoomed window off the pixel grid, on every plane
        dict(name="zoom_window", kind="points", U=21, V=21, L=32, per_layer=8, points=65536, line=False,
             precision="split_bf16"),
        # the solve of the tiny sample, the step every field starts from
        dict(name="solve_small", kind="solve", U=7, V=7, L=4, N=16),
        # the surrogate's training batch: loss and gradient
        dict(name="surrogate_grad", kind="grad", batch=256, layers=4),
        # surrogate inference over a batch of candidates
        dict(name="surrogate_infer", kind="infer", batch=256, layers=4),
        # surrogate inference inside a reconstruction loop: few samples, latency counts
        dict(name="surrogate_infer_few", kind="infer", batch=5, layers=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["volume", "volume", "volume", "fresh", "sweep", "points", "solve", "grad", "infer"])
    if kind in ("volume", "fresh"):
        c = dict(kind=kind, U=rng.randint(3, 23), V=rng.randint(3, 23), L=_log_int(rng, 2, 32),
                 per_layer=rng.randint(1, 24), Fx=8 * _log_int(rng, 4, 32), Fy=8 * _log_int(rng, 4, 32),
                 precision=rng.choice(["split_bf16", "split_bf16", "fp16", "fp32"]),
                 illuminations=rng.choice([1, 1, 2, _log_int(rng, 3, 16)]), tiles=rng.choice([1, 1, 1, 2]),
                 outside=rng.choice([0, 0, 2, 5]))
        while c["L"] * c["per_layer"] * c["Fx"] * c["Fy"] * c["illuminations"] * c["tiles"] ** 2 > 16 * 2 ** 22:
            c["per_layer"], c["illuminations"] = (c["per_layer"] + 1) // 2, (c["illuminations"] + 1) // 2
            c["Fx"] = max(32, c["Fx"] // 16 * 8)
        return c
    if kind == "sweep":
        return dict(kind=kind, items=rng.randint(3, 32), of=128, Fx=8 * rng.randint(6, 16), Fy=8 * rng.randint(6, 16),
                    planes=rng.randint(16, 64), precision=rng.choice(["split_bf16", "split_bf16", "fp16"]))
    if kind == "points":
        return dict(kind=kind, U=rng.randint(5, 21), V=rng.randint(5, 21), L=_log_int(rng, 4, 32),
                    per_layer=rng.randint(2, 8), points=_log_int(rng, 40, 65536), line=rng.random() < 0.5,
                    precision=rng.choice(["split_bf16", "split_bf16", "fp16", "fp32"]) if rng.random() < 0.7
                    else "split_bf16")
    if kind == "solve":
        return dict(kind=kind, U=rng.randint(3, 7), V=rng.randint(3, 7), L=rng.randint(1, 4), N=rng.choice([14, 16, 18]))
    batch = _log_int(rng, 1, 255)
    return dict(kind=kind, batch=batch + (batch == 5), layers=rng.randint(2, 5) if batch < 200 else rng.randint(2, 4))


# ------------------------------------------------------------------ inputs ---
def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + salt)
    return g


def _normal(g, *shape, dtype=torch.complex128):
    return torch.randn(shape, dtype=dtype, device="cuda", generator=g)


def _layers(seed, salt, U, V, L, illuminations=1):
    """Modes and amplitudes with a solved sample's structure: W rows scaled to unit fields, forward modes with
    Re gamma in [0.3, 1.6] and 5 % evanescent ones, backward = -forward with amplitudes ten times smaller."""
    M, g = U * V, _gen(seed, salt)
    f64 = dict(dtype=torch.float64, device="cuda", generator=g)
    re, im = 0.3 + 1.3 * torch.rand((L, 2 * M), **f64), 0.01 * -torch.log1p(-torch.rand((L, 2 * M), **f64))
    evanescent = torch.rand((L, 2 * M), **f64) < 0.05
    re = torch.where(evanescent, 0.05 * torch.rand((L, 2 * M), **f64), re)
    im = torch.where(evanescent, 0.1 + 0.9 * torch.rand((L, 2 * M), **f64), im)
    forward = torch.complex(re, im)
    W = _normal(g, L, 3 * M, 4 * M, dtype=torch.complex64).mul_(1.0 / math.sqrt(3 * M))
    a = [_normal(g, L, 2 * M) * (s / math.sqrt(2 * M)) for _ in range(illuminations) for s in (1.0, 0.1)]
    alpha = torch.stack([torch.cat(a[2 * i:2 * i + 2], dim=1) for i in range(illuminations)])
    p = [_normal(g, illuminations, 3, M) / math.sqrt(M) for _ in range(3)]
    if illuminations == 1:
        alpha, p = alpha[0], [x[0] for x in p]
    return W, torch.cat([forward, -forward], dim=1), alpha, p


def _geometry(c):
    """The arguments of Plan for a volume, fresh or points case."""
    L, n, out = c["L"], c["per_layer"] * c["L"], c.get("outside", 0)
    zb = INTERIOR * np.arange(L + 1)
    step = zb[-1] / n
    lead = out // 2
    zp = (np.arange(n + out) - lead + 0.5) * step
    kw = dict(U=c["U"], V=c["V"], L=L, lam=1.0, X=16.0, Y=16.0, z_bounds=zb, Fx=c.get("Fx", 256), Fy=c.get("Fy", 256),
              z_planes=zp, precision=c["precision"])
    if c.get("illuminations", 1) > 1:
        kw["illuminations"] = c["illuminations"]
    if c.get("tiles", 1) > 1:
        kw["tiles"] = (c["tiles"], c["tiles"])
    if out:
        kw.update(exterior=True, pupil_na=0.5, n_bot=1.5, z_inc=-0.5, x0=0.3, y0=-0.2)
    return kw


def _sweep_items(c):
    """Wavenumbers 1000..1800 / cm over 16 layers of 1 um, orders growing with the wavenumber."""
    out = []
    for k in range(c["items"]):
        i = k * c["of"] // c["items"]
        U = 9 + 2 * ((9 * i) // c["of"])
        zb = np.arange(17.0)
        zp = (np.arange(c["planes"]) + 0.5) * (16.0 / c["planes"])
        out.append(dict(U=U, V=U, L=16, lam=1e4 / (1000.0 + 800.0 * i / (c["of"] - 1)), X=64.0, Y=64.0, z_bounds=zb,
                        Fx=c["Fx"], Fy=c["Fy"], z_planes=zp))
    return out


def _xy(c, seed):
    n = c["points"]
    r = np.random.default_rng(seed)
    if c["line"]:
        return np.stack([16.0 * np.arange(n) / n, np.full(n, 16.0 * r.random())], axis=1)
    x0, y0 = 12.0 * r.random(2)
    side = int(math.isqrt(n))
    i = np.arange(n)
    return np.stack([x0 + 4.0 * (i % side) / side, y0 + 4.0 * (i // side) / side], axis=1)


def _ellipsoids(seed, salt, B, nz, ny, nx, axes, n_top=1.0):
    """B refractive-index volumes [B][nz][ny][nx]: up to 8 ellipsoids of n in 1.33..1.6 + i 0..0.05 each."""
    g = _gen(seed, salt)

    def uniform(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(shape, dtype=torch.float64, device="cuda", generator=g)

    z, y, x = torch.meshgrid(*(torch.arange(s, dtype=torch.float64, device="cuda") + 0.5 for s in (nz, ny, nx)),
                             indexing="ij")
    vol = torch.full((B, nz, ny, nx), n_top, dtype=torch.complex128, device="cuda")
    count = torch.randint(1, 9, (B, 1, 1, 1), device="cuda", generator=g)
    for k in range(8):
        ax, ctr = uniform(axes[0], axes[1], 3, B, 1, 1, 1), uniform(0.0, 1.0, 3, B, 1, 1, 1)
        inside = (((x - nx * ctr[0]) / ax[0]) ** 2 + ((y - ny * ctr[1]) / ax[1]) ** 2 + ((z - nz * ctr[2]) / ax[2]) ** 2) <= 1
        n = torch.complex(uniform(1.33, 1.6, B, 1, 1, 1), uniform(0.0, 0.05, B, 1, 1, 1))
        vol = torch.where(inside & (k < count), n, vol)
    return vol


def _solve_inputs(c, seed):
    """A sample of N x N x L voxels of a quarter wavelength and a focused beam."""
    N, period = c["N"], INTERIOR * c["N"]
    n = _ellipsoids(seed, 11, 1, c["L"], N, N, (1.5, 6.0))[0]
    r = (torch.arange(N, dtype=torch.float64, device="cuda") - 0.5 * N) * INTERIOR
    image = torch.exp(-(r[:, None] ** 2 + r[None, :] ** 2) / (0.3 * period) ** 2).to(torch.complex128)
    geometry = dict(U=c["U"], V=c["V"], L=c["L"], lam=1.0, X=period, Y=period, z_bounds=INTERIOR * np.arange(c["L"] + 1),
                    Nx=N, Ny=N)
    return geometry, n.contiguous(), image


def _parameter_groups(layers):
    """(size, scale) of the surrogate's flat parameters: lift, Fourier layers, projection, error head."""
    C, S2 = WIDTH, 2 * SLICES
    groups = [(C * S2, S2 ** -0.5), (C, S2 ** -0.5)]
    groups += [(MODES * MODES * C * C * 2, 1.0 / C), (C * C, C ** -0.5), (C, C ** -0.5)] * layers
    return groups + [(6 * C, C ** -0.5), (6, C ** -0.5), (C, C ** -0.5), (1, C ** -0.5)]


def _surrogate_inputs(c, seed):
    r = np.random.default_rng([seed, 7])
    flat = np.concatenate([r.uniform(-s, s, n) for n, s in _parameter_groups(c["layers"])]).astype(np.float32)
    n = _ellipsoids(seed, 21, c["batch"], SLICES, IN_GRID, IN_GRID, (2.0, 8.0)).to(torch.complex64).contiguous()
    g = _gen(seed, 22)
    # exit fields: a transmitted plane wave with scattered light in the 15x15 lowest orders
    k, x = torch.arange(-7, 8, device="cuda"), torch.arange(GRID, device="cuda")
    E = torch.exp(2j * math.pi * k[:, None] * x[None, :] / GRID).to(torch.complex64)
    spectrum = 0.3 * _normal(g, c["batch"], 3, 15, 15, dtype=torch.complex64) / (1.0 + (k[:, None] ** 2 + k[None, :] ** 2))
    spectrum[:, 0, 7, 7] += 0.8
    target = torch.einsum("bcvu,vy,ux->bcyx", spectrum, E, E).contiguous()
    return flat, n, target


# ---------------------------------------------------------------- a pass -----
def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind in ("volume", "fresh", "points"):
        W, gamma, alpha, p = _layers(seed, 1, c["U"], c["V"], c["L"], c.get("illuminations", 1))
        args = (W, gamma, alpha) + (tuple(p) if c.get("outside", 0) else ())
        plan = scw.Plan(**_geometry(c))
        if kind == "fresh":
            return dict(case=c, plan=plan, args=args)
        plan.set_layers(*args)
        state = dict(case=c, plan=plan)
        if kind == "points":
            plan.set_points(_xy(c, seed))
            state["out"] = torch.empty(plan.points_shape(), dtype=torch.complex64, device="cuda")
        else:
            state["out"] = torch.empty(plan.out_shape(), dtype=torch.complex64, device="cuda")
        return state
    if kind == "sweep":
        items = _sweep_items(c)
        plan = scw.BatchedPlan(items, precision=c["precision"])
        for i, it in enumerate(items):
            plan.set_layers(i, *_layers(seed, 100 + i, it["U"], it["V"], it["L"])[:3])
        outs = [torch.empty(s, dtype=torch.complex64, device="cuda") for s in plan.shapes]
        return dict(case=c, plan=plan, outs=outs, table=plan.item_table(outs))
    if kind == "solve":
        geometry, n, image = _solve_inputs(c, seed)
        solver = scw.Solver(**geometry)
        return dict(case=c, solver=solver, n=n, p_inc=solver.incident(image))
    flat, n, target = _surrogate_inputs(c, seed)
    net = scw.Surrogate(grid=GRID, modes=MODES, layers=c["layers"], slices=SLICES, in_grid=IN_GRID, batch_max=c["batch"])
    net.set_params(flat)
    return dict(case=c, net=net, n=n, target=target)


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "volume":
        return state["plan"].synthesize(state["out"])
    if kind == "fresh":
        state["plan"].set_layers(*state["args"])
        return state["plan"].synthesize()
    if kind == "points":
        return state["plan"].synthesize_points(state["out"])
    if kind == "sweep":
        state["plan"].synthesize_table(state["table"])
        return state["outs"]
    if kind == "solve":
        return state["solver"].solve(state["n"], state["p_inc"])
    if kind == "grad":
        loss = state["net"].forward_backward(state["n"], state["target"])
        return loss, state["net"].grads()
    field, est, fallback = state["net"].infer(state["n"], threshold=0.5)
    return field, est, fallback


# ------------------------------------------------------------------- work ----
def _synthesis_work(U, V, L, planes, fields, pixels, convert=False):
    """Layers' W read once (and written once where a pass converts it), spectra -> field written once. planes:
    plane slots inside the sample; fields: component planes written, of `pixels` each."""
    M = U * V
    w = L * 3 * M * 4 * M * 8
    flops = 8.0 * 3 * M * 4 * M * planes + fields * 8.0 * (U * V * 16 + 16 * pixels)
    return dict(bytes=w * (2 if convert else 1) + 8.0 * fields * pixels, flops=flops)


def work(case):
    c, kind = case, case["kind"]
    if kind in ("volume", "fresh"):
        I, t = c["illuminations"], c["tiles"]
        inside, total = c["L"] * c["per_layer"] * I, (c["L"] * c["per_layer"] + c["outside"]) * I
        return _synthesis_work(c["U"], c["V"], c["L"], inside, 3 * total, c["Fx"] * c["Fy"] * t * t)
    if kind == "points":
        planes, M, P = c["L"] * c["per_layer"], c["U"] * c["V"], c["points"]
        return dict(bytes=8.0 * (c["L"] * 12 * M * M + M * 3 * planes + 3 * planes * P + 2 * P),
                    flops=8.0 * M * (12 * M * planes + 3 * planes * P))
    if kind == "sweep":
        parts = [_synthesis_work(it["U"], it["V"], 16, c["planes"], 3 * c["planes"], c["Fx"] * c["Fy"])
                 for it in _sweep_items(c)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if kind == "solve":
        M, L = c["U"] * c["V"], c["L"]
        # per layer: the product of the two off-diagonal blocks, ~25 n^3 of a 2M eigenproblem, the LU solve of 4M
        flops = L * 8.0 * ((25 + 2) * (2 * M) ** 3 + (4 * M) ** 3 * 4 / 3) + 8.0 / 3 * (6 * M) ** 3
        return dict(bytes=16.0 * (L * c["N"] ** 2 + 8 * M * L + 9 * M) + 8.0 * L * 12 * M * M, flops=flops)
    B, px, C, m2 = c["batch"], GRID * GRID, WIDTH, MODES * MODES
    n_par = sum(n for n, _ in _parameter_groups(c["layers"]))
    # row-column transforms of the kept modes, per-mode C x C products, 1x1 convolutions, lift and projection
    fourier = B * C * (GRID * GRID * MODES * 4.0 + GRID * m2 * 8.0)
    layer = 2 * fourier + 8.0 * B * m2 * C * C + 2.0 * B * px * C * C
    one = c["layers"] * layer + 2.0 * B * px * C * (2 * SLICES + 6)
    io = 8.0 * B * (SLICES * IN_GRID * IN_GRID + 3 * px)
    if kind == "infer":
        return dict(bytes=io + 2.0 * n_par + 5.0 * B, flops=one)
    # a backward pass is twice the forward; the activations of every layer (BF16) are kept for it
    return dict(bytes=io + 2.0 * n_par + 4.0 * n_par + 2 * 2.0 * c["layers"] * B * C * px, flops=3 * one)


# ------------------------------------------------------------------ exact ----
def _orders(U, V):
    u, v = torch.arange(U, device="cuda") - U // 2, torch.arange(V, device="cuda") - V // 2
    return u.double(), v.double()


def _cis(t):
    return torch.exp(2j * math.pi * t)


def _sz(n, sx, sy):
    """sqrt(n^2 - sx^2 - sy^2) on the decaying branch."""
    w = torch.sqrt(torch.as_tensor(complex(n) ** 2, dtype=torch.complex128, device="cuda") - (sx ** 2 + sy ** 2))
    return torch.where((w.imag < 0) | ((w.imag == 0) & (w.real < 0)), -w, w)


def _spectra(kw, W, gamma, alpha, p=None):
    """S [Fz][3][M] of every plane in 64 bits."""
    U, V, L, lam, zb = kw["U"], kw["V"], kw["L"], kw["lam"], kw["z_bounds"]
    M, zp = U * V, np.asarray(kw["z_planes"])
    S = torch.zeros((len(zp), 3 * M), dtype=torch.complex128, device="cuda")
    region = np.minimum(np.searchsorted(zb, zp, side="right") - 1, L - 1)
    for l in range(L):
        f = np.nonzero((region == l) & (zp >= zb[0]) & (zp <= zb[-1]))[0]
        if not len(f):
            continue
        z = torch.as_tensor(zp[f], device="cuda")
        ref = torch.cat([torch.full((2 * M,), zb[l]), torch.full((2 * M,), zb[l + 1])]).to(z)
        g = torch.exp(2j * math.pi / lam * gamma[l][:, None] * (z[None, :] - ref[:, None]))
        S[torch.as_tensor(f, device="cuda")] = (W[l].to(torch.complex128) @ (alpha[l][:, None] * g)).T
    S = S.reshape(-1, 3, M)
    if p is not None:
        u, v = _orders(U, V)
        sx, sy = (lam * u / kw["X"]).repeat(V), (lam * v / kw["Y"]).repeat_interleave(U)
        top, bot = _sz(kw.get("n_top", 1.0), sx, sy), _sz(kw.get("n_bot", 1.0), sx, sy)
        na = kw.get("pupil_na", 0.0)
        pupil = ((sx ** 2 + sy ** 2) <= na * na * (1 + 1e-12)) if na > 0 else torch.ones_like(sx)
        for f, z in enumerate(zp):
            if z < zb[0]:
                S[f] = p[0] * _cis(top * (z - kw["z_inc"]) / lam) + p[1] * _cis(-top * (z - zb[0]) / lam)
            elif z > zb[-1]:
                S[f] = p[2] * pupil * _cis(bot * (z - zb[-1]) / lam)
    return S


def _to_grid(kw, S):
    """E [3][Fz][Fy][Fx] of the spectra on the pixel grid."""
    U, V, Fx, Fy = kw["U"], kw["V"], kw["Fx"], kw["Fy"]
    u, v = _orders(U, V)
    x = torch.arange(Fx, device="cuda").double() / Fx + kw.get("x0", 0.0) / kw["X"]
    y = torch.arange(Fy, device="cuda").double() / Fy + kw.get("y0", 0.0) / kw["Y"]
    S = S.reshape(-1, 3, V, U).permute(1, 0, 2, 3)
    E = torch.matmul(_cis(v[None, :] * y[:, None]), torch.matmul(S, _cis(u[:, None] * x[None, :])))
    t = kw.get("tiles", (1, 1))
    return E.repeat(1, 1, t[1], t[0])


def _exact_solve(c, seed):
    """Reflected and transmitted amplitudes from the layers' transfer matrices expm(i k D d)."""
    geo, n, image = _solve_inputs(c, seed)
    U, V, L, N, X = c["U"], c["V"], c["L"], c["N"], geo["X"]
    M, k, zb = U * V, 2 * math.pi, geo["z_bounds"]
    u, v = _orders(U, V)
    uu, vv = u.repeat(V), v.repeat_interleave(U)
    sx, sy = uu / X, vv / X
    du, dv = (uu[:, None] - uu[None, :]).long() % N, (vv[:, None] - vv[None, :]).long() % N
    D_, I = torch.diag, torch.eye(M, dtype=torch.complex128, device="cuda")
    Sx, Sy, Z = D_(sx).to(I), D_(sy).to(I), torch.zeros_like(I)
    K = torch.eye(4 * M, dtype=torch.complex128, device="cuda")
    for l in range(L):
        phi = (torch.fft.fft2(n[l] ** 2) / N ** 2)[dv, du]
        psi = (torch.fft.fft2(n[l] ** -2) / N ** 2)[dv, du]
        A = torch.cat([torch.cat([Sx @ psi @ Sy, I - Sx @ psi @ Sx], 1), torch.cat([Sy @ psi @ Sy - I, -Sy @ psi @ Sx], 1)])
        B = torch.cat([torch.cat([-Sx @ Sy, Sx @ Sx - phi], 1), torch.cat([phi - Sy @ Sy, Sy @ Sx], 1)])
        D = torch.cat([torch.cat([torch.zeros_like(A), A], 1), torch.cat([B, torch.zeros_like(B)], 1)])
        K = torch.linalg.matrix_exp(1j * k * D * float(zb[l + 1] - zb[l])) @ K
    sz = _sz(1.0, sx, sy)

    def to_r(z):
        rows = [[I, Z, Z], [Z, I, Z], [Z, -D_(z), Sy], [D_(z), Z, -Sx]]
        return torch.cat([torch.cat(r, 1) for r in rows])

    p = torch.zeros((3, M), dtype=torch.complex128, device="cuda")
    p[0] = (torch.fft.fft2(image) / N ** 2)[vv.long() % N, uu.long() % N]
    p[2] = -(sx * p[0] + sy * p[1]) / sz
    A = torch.zeros((6 * M, 6 * M), dtype=torch.complex128, device="cuda")
    A[:4 * M, :3 * M], A[:4 * M, 3 * M:] = -K @ to_r(-sz), to_r(sz)
    A[4 * M:5 * M, :3 * M] = torch.cat([Sx, Sy, -D_(sz)], 1)
    A[5 * M:, 3 * M:] = torch.cat([Sx, Sy, D_(sz)], 1)
    b = torch.cat([K @ (to_r(sz) @ p.reshape(-1)), torch.zeros(2 * M, dtype=torch.complex128, device="cuda")])
    x = torch.linalg.solve(A, b)
    # an eigenvector has a free phase and the modes a free order: W, gamma and alpha have no one value
    return None, None, None, x[:3 * M].reshape(3, M), x[3 * M:].reshape(3, M)


def _exact_surrogate(c, seed, training):
    flat, n, target = _surrogate_inputs(c, seed)
    flat = torch.from_numpy(flat).to("cuda", torch.float64).requires_grad_(training)
    C, S2, m, N = WIDTH, 2 * SLICES, MODES, GRID
    parts = list(torch.split(flat, [size for size, _ in _parameter_groups(c["layers"])]))
    k, x = torch.arange(m, device="cuda") - m // 2, torch.arange(N, device="cuda")
    E = _cis((k[:, None] * x[None, :]).double() / N)
    B = c["batch"]
    loss = [torch.zeros((), dtype=torch.float64, device="cuda") for _ in range(2)]
    fields, ests, grads = [], [], torch.zeros_like(flat)
    for s in range(0, B, 32):  # the loss is a mean over samples: gradients of the parts add up
        nb, T = n[s:s + 32].to(torch.complex128), target[s:s + 32].to(torch.complex128)
        a = torch.stack([nb.real - 1.0, nb.imag], dim=2).reshape(len(nb), S2, IN_GRID, IN_GRID)
        a = a.repeat_interleave(N // IN_GRID, 2).repeat_interleave(N // IN_GRID, 3)
        h = torch.einsum("oc,bcyx->boyx", parts[0].reshape(C, S2), a) + parts[1][:, None, None]
        for l in range(c["layers"]):
            R, Wl, cl = parts[2 + 3 * l:5 + 3 * l]
            R = torch.view_as_complex(R.reshape(m, m, C, C, 2))
            vh = torch.einsum("biyx,vy,ux->bivu", h.to(torch.complex128), E.conj(), E.conj())
            wh = torch.einsum("vuoi,bivu->bovu", R, vh)
            z = torch.einsum("bovu,vy,ux->boyx", wh, E, E).real / N ** 2
            z = z + torch.einsum("oi,biyx->boyx", Wl.reshape(C, C), h) + cl[:, None, None]
            h = torch.nn.functional.gelu(z) if l < c["layers"] - 1 else z
        Q, q, e, e0 = parts[-4:]
        F = torch.einsum("jo,boyx->bjyx", Q.reshape(6, C), h) + q[:, None, None]
        field = torch.complex(F[:, 0::2], F[:, 1::2])
        head = h.detach().mean(dim=(2, 3)) @ e + e0  # the head is trained on a constant trunk
        if not training:
            fields.append(field)
            ests.append(torch.exp(head))
            continue
        rel2 = (field - T).abs().square().sum((1, 2, 3)) / T.abs().square().sum((1, 2, 3))
        part = (rel2.sum() / B, (head - 0.5 * torch.log(rel2.detach() + 1e-12)).square().sum() / B)
        grads = grads + torch.autograd.grad(part[0] + part[1], flat, retain_graph=s + 32 < B)[0]
        loss = [x + y.detach() for x, y in zip(loss, part)]
    if training:
        return torch.stack([loss[0] + loss[1], loss[0], loss[1]]), grads
    est = torch.cat(ests)
    return torch.cat(fields), est, None


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "solve":
        return _exact_solve(c, seed)
    if kind == "grad":
        return _exact_surrogate(c, seed, True)
    if kind == "infer":
        with torch.no_grad():
            return _exact_surrogate(c, seed, False)
    if kind == "sweep":
        return [_to_grid(it, _spectra(it, *_layers(seed, 100 + i, it["U"], it["V"], it["L"])[:3]))
                for i, it in enumerate(_sweep_items(c))]
    kw, I = _geometry(c), c.get("illuminations", 1)
    W, gamma, alpha, p = _layers(seed, 1, c["U"], c["V"], c["L"], I)
    p = p if c.get("outside", 0) else None
    if kind == "points":
        S, (u, v) = _spectra(kw, W, gamma, alpha), _orders(c["U"], c["V"])
        xy = torch.as_tensor(_xy(c, seed), device="cuda")
        phi = _cis(u.repeat(c["V"])[:, None] * xy[:, 0] / kw["X"] + v.repeat_interleave(c["U"])[:, None] * xy[:, 1] / kw["Y"])
        return torch.matmul(S.permute(1, 0, 2), phi)
    if I == 1:
        return _to_grid(kw, _spectra(kw, W, gamma, alpha, p))
    return torch.stack([_to_grid(kw, _spectra(kw, W, gamma, alpha[i], None if p is None else [x[i] for x in p]))
                        for i in range(I)])
