"""What the speed of this framework is measured on: single operators and whole reconstructions through the
public binding (``paper_1901_01893_gb300.smsm``), at the sizes its workloads, tests and benchmark use.

Geometry of a case: L simultaneously excited slices, Ns shots, Nc coils, N x N images, filter r, CAIPI shift
FOV/div, D diffusion directions (the plan's batch).  Inputs are made on the GPU with plain torch in 64 bits from the
seed alone (elliptic phantoms, polynomial shot phases, Gaussian coil maps, complex Gaussian noise at an amplitude
ratio of 30) and rounded to the types the calls take.
"""
import math

import torch

from paper_1901_01893_gb300 import smsm

DEV = "cuda"
LAM = 1e-2


def _case(name, op, L, Ns, Nc, N, r, div, D, **more):
    c = {"op": op, "L": L, "Ns": Ns, "Nc": Nc, "N": N, "r": r, "div": div, "D": D}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the forward model of one small slice group: the smallest call a user makes (a data-consistency check)
        _case("forward_64_single", "forward", 2, 4, 8, 64, 5, 2, 1),
        # simulating data at the largest matrix of the workloads, three slices, FOV/3 (not a whole number of pixels)
        _case("forward_256_thirds", "forward", 3, 4, 32, 256, 6, 3, 2),
        # A^H y of a whole diffusion series of one slice group: the start of every reconstruction
        _case("adjoint_128_series", "adjoint", 2, 4, 32, 128, 6, 2, 26),
        # the Hankel Gram of a series (FP32 form): rank studies of the shots, the solver's own first half
        _case("gram_128_series", "gram", 2, 4, 32, 128, 6, 2, 26),
        # the annihilating-filter penalty for given weights, as another solver around this operator calls it
        _case("penalty_256", "penalty", 3, 4, 8, 256, 6, 3, 4),
        # SMS-SENSE with known shot phases (the comparison reconstruction), 2 shots, 30 CG steps
        _case("sense_192_phase", "sense", 3, 2, 16, 192, 4, 3, 4, J=30, phase=True),
        # one small slice group with the library's default schedule (10 x 10): single-call latency
        _case("solve_64_single", "solve", 2, 4, 8, 64, 5, 2, 1, K=10, J=10, precision=0),
        # one direction of the paper's acquisition (128 x 128, 32 coils, 4 shots): a scanner console's call
        _case("solve_128_single", "solve", 2, 4, 32, 128, 6, 2, 1, K=20, J=15, precision=0),
        # a whole series of that acquisition in the BF16 split form: throughput, the benchmark's workload
        _case("solve_128_series", "solve", 2, 4, 32, 128, 6, 2, 26, K=20, J=15, precision=1),
        # the high-resolution acquisition with a FOV/3 shift, a short first schedule (a longer one grows the
        # rounding of any two FP32 solves of this geometry apart)
        _case("solve_256_thirds", "solve", 3, 4, 32, 256, 6, 3, 4, K=2, J=4, precision=0),
        # 8 shots with a 6x6 filter: the largest Gram (C = 288) of the batched workload, a short schedule too
        _case("solve_192_8shots", "solve", 2, 8, 16, 192, 6, 2, 2, K=3, J=5, precision=0),
        # the learned warm start's network applied to the k-space of two slice groups before their solve
        _case("learned_start_256", "start", 3, 4, 2, 256, 6, 3, 2, width=64, layers=6),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any of the operations, geometry over the workloads' whole range (matrices 48 to 256 with
    factors of 3 among them, 1 to 3 slices, 1 to 8 shots, 2 to 32 coils), batches up to the cost of the largest."""
    while True:
        op = rng.choice(["forward", "adjoint", "gram", "penalty", "sense", "solve", "solve", "start"])
        N = rng.choice([48, 64, 72, 96, 108, 128, 144, 192, 256])
        Ns = rng.choice([1, 2, 3, 4, 6, 8])
        if N % Ns or (N // Ns) % 2 or N // Ns < 8:
            continue
        L = rng.randint(1, 3)
        Nc = _log(rng, 2, 32)
        r = rng.randint(2, {1: 9, 2: 8, 3: 6, 4: 6, 6: 6, 8: 6}[Ns])
        div = rng.choice([L, L, 2, 3, 4])
        pixels = L * Ns * N * N
        D = _log(rng, 1, max(1, min(26, int(26 * 2 * 4 * 128 * 128 / pixels))))
        more = {}
        if op == "start":
            D, Nc = min(D, max(1, 2 * 256 * 256 // (N * N))), 2
            more = {"width": rng.choice([16, 24, 40, 48, 64]), "layers": rng.randint(2, 6)}
        elif op == "sense":
            more = {"J": rng.randint(3, 30), "phase": rng.random() < 0.5}
        elif op == "solve":
            C = Ns * r * r
            big = N >= 192
            Nc = max(4, Nc)
            more = {"K": 2 if big else rng.randint(2, 3), "J": rng.randint(3, 4 if big else 5),
                    "precision": 1 if C <= 144 and rng.random() < 0.4 else 0}
        elif op in ("gram", "penalty"):
            Nc = 2
        return _case(None, op, L, Ns, Nc, N, r, div, D, **more)


# --- inputs, 64 bits on the GPU ------------------------------------------------------------------


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _uniform(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _crandn(g, *shape):
    return torch.complex(torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64),
                         torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64))


def _grid(N):
    u = (torch.arange(N, device=DEV, dtype=torch.float64) - N / 2) / (N / 2)
    return u[:, None], u[None, :]


def _phantom(g, L, N):
    Y, X = _grid(N)
    img = torch.zeros(L, N, N, device=DEV, dtype=torch.float64)
    for _ in range(10):
        cx, cy, a, b, th, amp = (_uniform(g, lo, hi, L, 1, 1) for lo, hi in
                                 ((-0.3, 0.3), (-0.3, 0.3), (0.1, 0.4), (0.1, 0.4), (0.0, math.pi), (0.1, 1.0)))
        xr = (X - cx) * torch.cos(th) + (Y - cy) * torch.sin(th)
        yr = (Y - cy) * torch.cos(th) - (X - cx) * torch.sin(th)
        img = img + amp * ((xr / a) ** 2 + (yr / b) ** 2 <= 1.0)
    return img


def _shot_phase(g, L, Ns, N):
    Y, X = _grid(N)
    ph = torch.zeros(L, Ns, N, N, device=DEV, dtype=torch.float64)
    for a in range(4):
        for b in range(4 - a):
            ph = ph + _uniform(g, -math.pi, math.pi, L, Ns, 1, 1) * (X / 2) ** a * (Y / 2) ** b
    return torch.polar(torch.ones_like(ph), ph)


def _coils(L, Nc, N):
    Y, X = _grid(N)
    c = torch.arange(Nc, device=DEV, dtype=torch.float64)[:, None, None]
    ang = 2 * math.pi * c / Nc
    zc = torch.where(c % 2 == 0, 0.4, -0.4).to(torch.float64)
    S = []
    for l in range(L):
        z = (l - (L - 1) / 2) * 0.6
        m = torch.exp(-((X - 1.2 * torch.cos(ang)) ** 2 + (Y - 1.2 * torch.sin(ang)) ** 2 + (z - zc) ** 2) / 0.72)
        S.append(torch.polar(m / torch.sqrt((m ** 2).sum(0, keepdim=True)), ang.expand_as(m)))
    return torch.stack(S)


def _c64(t):
    return t.to(torch.complex64).contiguous()


def _images(c, seed):
    """[D][L][Ns][N][N] images of the shots and their phases, 64 bits."""
    g = _gen(seed)
    rho = _phantom(g, c["L"], c["N"])
    ph = torch.stack([_shot_phase(g, c["L"], c["Ns"], c["N"]) for _ in range(c["D"])])
    return rho[None, :, None] * ph, ph


def _lead(c, t):
    return t if c["D"] > 1 else t[0]


def _inputs(c, seed):
    """The tensors a call takes, by name, rounded to its types: a pure function of the case and the seed."""
    op, D, L, Ns, Nc, N = c["op"], c["D"], c["L"], c["Ns"], c["Nc"], c["N"]
    g = _gen(seed + 1000003)
    img, ph = _images(c, seed)
    out = {"sens": _c64(_coils(L, Nc, N))}
    if op in ("gram", "penalty", "forward", "start"):
        x = _fft2c(img)
        out["x"] = _c64(_lead(c, x / torch.sqrt((x.abs() ** 2).mean())))
        if op == "penalty":
            C = Ns * c["r"] ** 2
            A = _crandn(g, D, L, C, max(1, C // 2)) / math.sqrt(C)
            W = 0.1 * torch.eye(C, device=DEV, dtype=torch.complex128) + A @ A.mH  # a weight: Hermitian, positive
            out["W"] = _lead(c, 0.5 * (W + W.mH)).contiguous()
        if op == "start":
            params, w, n = [], c["width"], c["layers"]
            for k in range(n):
                ci, co = (L * Ns if k == 0 else w), (L * Ns if k + 1 == n else w)
                params += [(_crandn(g, co * ci * 9) / math.sqrt(9 * ci)), 0.01 * _crandn(g, co)]
            out["params"] = _c64(torch.cat(params))
        return out
    S = out["sens"].to(torch.complex128)
    y = torch.stack([_forward(_fft2c(v), S, c["div"]) for v in img])
    nz = _crandn(g, *y.shape)
    y = y + nz * (torch.linalg.vector_norm(y) / (30.0 * torch.linalg.vector_norm(nz)))
    out["y"] = _c64(_lead(c, y / torch.sqrt((y.abs() ** 2).mean())))
    if c.get("phase"):
        out["phase"] = _c64(_lead(c, ph))
    return out


# --- the calls -----------------------------------------------------------------------------------


def prepare(case, seed):
    c, v = case, _inputs(case, seed)
    s = dict(v, case=c)
    s["plan"] = smsm.Plan(c["L"], c["Ns"], c["Nc"], c["N"], c["r"], caipi_div=c["div"], batch=c["D"],
                          precision=c.get("precision", 0))
    s["plan"].set_sens(v["sens"])
    if c["op"] == "solve":
        s["params"] = smsm.default_params(lam=LAM, outer_iters=c["K"], cg_iters=c["J"])
    if c["op"] == "start":
        s["net"] = smsm.CNN(c["L"] * c["Ns"], c["N"], c["N"], width=c["width"], layers=c["layers"], max_batch=c["D"])
        s["net"].set_params(v["params"])
    return s


def run(s):
    op = s["case"]["op"]
    if op == "forward":
        return s["plan"].forward(s["x"])
    if op == "adjoint":
        return s["plan"].adjoint(s["y"])
    if op == "gram":
        return s["plan"].hankel_gram(s["x"])
    if op == "penalty":
        return s["plan"].apply_filters(s["W"], s["x"])
    if op == "sense":
        return s["plan"].sense(s["y"], phase=s.get("phase"), cg_iters=s["case"]["J"], report=False)[0]
    if op == "solve":
        x = s["plan"].reconstruct(s["y"], params=s["params"], report=False)[0]
        return list(x) if s["case"]["D"] > 1 else x  # one output per direction
    return smsm.learned_start(s["plan"], s["net"], s["x"])


# --- what a pass cannot do without ---------------------------------------------------------------


def work(case):
    c = case
    D, L, Ns, Nc, N, r = c["D"], c["L"], c["Ns"], c["Nc"], c["N"], c["r"]
    B, NN = L * Ns, N * N
    fft = 10 * NN * math.log2(N)  # one N x N transform
    if c["op"] == "start":
        mac = 9 * (2 * B * c["width"] + c["width"] ** 2 * (c["layers"] - 2))
        return {"bytes": 8 * (2 * D * B * NN + mac), "flops": D * (8 * NN * mac + 2 * B * fft)}
    x, y, sens, C, R2 = 8 * D * B * NN, 8 * D * Nc * NN, 8 * L * Nc * NN, Ns * r * r, 2 * r - 1
    P = (N - r + 1) ** 2
    # per coil, slice and shot: the coil products and, along y, the N/Ns-point transform of the kept lines; per coil
    # line kept the x transform; per slice-shot image one transform
    A = D * (B * fft + Nc * B * (14 * NN + 5 * NN / Ns * math.log2(N / Ns)) + 5 * Nc * NN * math.log2(N))
    if c["op"] in ("forward", "adjoint"):
        return {"bytes": x + y + sens, "flops": A}
    gram = 4 * D * L * P * C * C
    # the filters from W, the periodic part in the image domain, the band within r - 1 of an edge tap by tap
    pen = D * (2 * B * fft + 8 * L * Ns * Ns * NN + 8 * L * Ns * Ns * (NN - max(0, N - 2 * r + 2) ** 2) * R2 * R2)
    filt = D * L * (8 * (Ns * (Ns + 1) // 2) * (R2 * R2 * N + R2 * NN) + 2 * C * C)
    if c["op"] == "gram":
        return {"bytes": x + 16 * D * L * C * C, "flops": gram}
    if c["op"] == "penalty":
        return {"bytes": 2 * x + 16 * D * L * C * C, "flops": pen + filt}
    if c["op"] == "sense":
        return {"bytes": y + sens + x / Ns + (x if c["phase"] else 0), "flops": (2 * c["J"] + 1) * A}
    # a CG step: A^H A through the coils' correlations (or, shift between pixels, coil by coil) and the penalty
    normal = 8 * D * B * B * NN if N % c["div"] == 0 else 2 * D * Nc * B * (14 * NN + 5 * NN / Ns * math.log2(N / Ns))
    step = normal + pen + 20 * D * B * NN
    return {"bytes": x + y + sens, "flops": A + c["K"] * (gram + D * L * 24 * C ** 3 + filt + (c["J"] + 1) * step)}


# --- the same in plain torch, 64 bits ------------------------------------------------------------


def _fft2c(v):
    ax = (-2, -1)
    return torch.fft.fftshift(torch.fft.fft2(torch.fft.ifftshift(v, dim=ax), norm="ortho"), dim=ax)


def _ifft2c(v):
    ax = (-2, -1)
    return torch.fft.fftshift(torch.fft.ifft2(torch.fft.ifftshift(v, dim=ax), norm="ortho"), dim=ax)


def _ramp(L, N, div):
    a = torch.arange(L, device=DEV, dtype=torch.float64)[:, None] * (torch.arange(N, device=DEV) - N / 2)[None]
    return torch.polar(torch.ones_like(a), -2 * math.pi * a / div)


def _forward(x, S, div, phase=None):
    """[L][Ns or 1][N][N] -> [Ns][Nc][N/Ns][N]"""
    L, N = x.shape[0], x.shape[-1]
    Ns = x.shape[1] if phase is None else phase.shape[1]
    ramp = _ramp(L, N, div)
    img = _ifft2c(x)
    if phase is not None:
        img = img * phase
    y = []
    for i in range(Ns):
        k = _fft2c(S * img[:, i, None])
        y.append((ramp[:, None, :, None] * k).sum(0)[:, i::Ns])
    return torch.stack(y)


def _adjoint(y, S, div, phase=None):
    Ns, Nc, _, N = y.shape
    ramp = _ramp(S.shape[0], N, div)
    out = []
    for i in range(Ns):
        full = torch.zeros(Nc, N, N, device=DEV, dtype=torch.complex128)
        full[:, i::Ns] = y[i]
        out.append((S.conj() * _ifft2c(ramp.conj()[:, None, :, None] * full)).sum(1))
    img = torch.stack(out, 1)
    if phase is not None:
        img = (phase.conj() * img).sum(1, keepdim=True)
    return _fft2c(img)


def _hankel(x, r):
    """[Ns][N][N] -> [(N-r+1)^2][Ns r r]"""
    Ns, N, _ = x.shape
    V = N - r + 1
    w = x.unfold(1, r, 1).unfold(2, r, 1)  # [Ns][V][V][r][r]
    return w.permute(1, 2, 0, 3, 4).reshape(V * V, Ns * r * r)


def _hankel_t(Y, Ns, N, r):
    V = N - r + 1
    Y = Y.reshape(V, V, Ns, r, r)
    out = torch.zeros(Ns, N, N, device=DEV, dtype=torch.complex128)
    for a in range(r):
        for b in range(r):
            out[:, a:a + V, b:b + V] += Y[:, :, :, a, b].permute(2, 0, 1)
    return out


def _penalty(x, W, r):
    return torch.stack([_hankel_t(_hankel(v, r) @ w, v.shape[0], v.shape[-1], r) for v, w in zip(x, W)])


def _cg(apply, b, x, J):
    r = b - apply(x)
    p, rr = r.clone(), (r.abs() ** 2).sum()
    for _ in range(J):
        q = apply(p)
        a = rr / (p.conj() * q).sum().real
        x, r = x + a * p, r - a * q
        new = (r.abs() ** 2).sum()
        p, rr = r + (new / rr) * p, new
    return x


def _solve(y, S, c):
    b = _adjoint(y, S, c["div"])
    x, eps, r = b, None, c["r"]
    for k in range(c["K"]):
        G = torch.stack([h.mH @ h for h in (_hankel(v, r) for v in x)])
        s, V = torch.linalg.eigh(G)
        eps = 1e-2 * s.max() if eps is None else torch.maximum(eps / 1.5, low)
        low = 1e-2 * eps if k == 0 else low
        W = (V / torch.sqrt(s.clamp_min(0) + eps)[:, None, :]) @ V.mH
        x = _cg(lambda v: _adjoint(_forward(v, S, c["div"]), S, c["div"]) + LAM * _penalty(v, W, r), b, x, c["J"])
    return x


def _start(x, params, c):
    """[L][Ns][N][N] k-space -> F(a + f(a)), a = F^-1 x; products take the weights rounded to BF16"""
    B, w, n = c["L"] * c["Ns"], c["width"], c["layers"]
    p = torch.view_as_real(params).to(torch.bfloat16).double()
    img = _ifft2c(x).reshape(1, B, c["N"], c["N"])
    h, at = torch.cat([img.real, img.imag], 1), 0
    for k in range(n):
        ci, co = (B if k == 0 else w), (B if k + 1 == n else w)
        re, im = (p[at:at + co * ci * 9, j].reshape(co, ci, 3, 3) for j in (0, 1))
        at += co * ci * 9
        W = torch.cat([torch.cat([re, -im], 1), torch.cat([im, re], 1)], 0)
        bias = torch.cat([p[at:at + co, 0], p[at:at + co, 1]])
        at += co
        with torch.backends.cudnn.flags(enabled=False):  # native double convolution
            h = torch.nn.functional.conv2d(torch.relu(h) if k else h, W, bias, padding=1)
    return _fft2c((img + torch.complex(h[:, :B], h[:, B:])).reshape(x.shape))


def exact(case, seed):
    c = case
    v = _inputs(c, seed)
    up = {k: t.to(torch.complex128) for k, t in v.items()}
    S, D = up["sens"], c["D"]
    if D == 1:
        up = {k: (t if k in ("sens", "params") else t[None]) for k, t in up.items()}
    ph = up.get("phase")
    got = []
    for d in range(D):
        if c["op"] == "forward":
            got.append(_forward(up["x"][d], S, c["div"]))
        elif c["op"] == "adjoint":
            got.append(_adjoint(up["y"][d], S, c["div"]))
        elif c["op"] == "gram":
            got.append(torch.stack([h.mH @ h for h in (_hankel(x, c["r"]) for x in up["x"][d])]))
        elif c["op"] == "penalty":
            got.append(_penalty(up["x"][d], up["W"][d], c["r"]))
        elif c["op"] == "start":
            got.append(_start(up["x"][d], v["params"], c))
        elif c["op"] == "solve" and d >= 3:
            got.append(None)  # three directions of a series say it
        elif c["op"] == "sense":
            one = ph[d] if ph is not None else torch.ones(c["L"], c["Ns"], c["N"], c["N"], device=DEV, dtype=torch.complex128)
            b = _adjoint(up["y"][d], S, c["div"], one)
            got.append(_cg(lambda x: _adjoint(_forward(x, S, c["div"], one), S, c["div"], one), b, torch.zeros_like(b), c["J"]))
        else:
            got.append(_solve(up["y"][d], S, c))
    if D == 1:
        return got[0]
    return got if c["op"] == "solve" else torch.stack(got)
