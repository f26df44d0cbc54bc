"""The work that this library is used for, as cases to be measured: coding of
patches (from device and from host memory, both precisions), coding of images,
projection, the dictionary update, and the way back from codes to pixels.

Sizes are the ones of the package's own workloads: the 11 x 11 patches (J = 6
rings, harmonics to 8) with the small, the 10^6-patch and the serving
dictionary, the 21 x 21 patches (J = 10, harmonics to 12) of the image
workload, and the ragged shapes of the tests.  Inputs follow the package's
synthetic recipe (three steered atoms at continuous angles plus noise; line
textures for images), drawn on the GPU from the seed alone."""
import math

import numpy as np
import torch

import paper_1806_04374_gb300 as rsc

F64 = torch.float64


# ------------------------------------------------------------------- cases

def _code(name, P, M, R, K, J=6, kmax=8, sigma=0.1, precision="f16"):
    return {"name": name, "kind": "code", "P": P, "M": M, "R": R, "K": K, "J": J, "kmax": kmax,
            "sigma": sigma, "precision": precision}


def _images(name, sides, N, J, kmax, M, R, K):
    return {"name": name, "kind": "images", "sides": sides, "N": N, "J": J, "kmax": kmax, "M": M,
            "R": R, "K": K, "precision": "f16"}


def listed():
    return [
        # a handful of patches coded on demand: launches and latency decide
        _code("code_small", 1000, 16, 32, 3, sigma=0.05),
        # odd angle count (no half-turn pairs), a small dictionary, ragged patch count
        _code("code_odd_angles", 60001, 7, 33, 3),
        # the benchmark workload: bulk coding of patches resident in HBM
        _code("code_1m", 1_000_000, 64, 64, 5),
        # the plain FP32 path, for users who code without the tensor cores
        _code("code_fp32", 100_003, 64, 64, 5, precision="fp32"),
        # patches in pinned host memory, codes back to host memory (the
        # end-to-end call), at the size of the learning runs
        dict(_code("code_host", 200_000, 128, 64, 5), kind="host"),
        # one batch of the image server: uneven images, 11 x 11 windows
        _images("images_11x11", "512x389,131x640,300x300", 11, 6, 8, 128, 64, 5),
        # the texture image workload: 21 x 21 windows, large dictionary
        _images("images_21x21", "96x96,160x160,224x224,288x288", 21, 10, 12, 256, 128, 8),
        # pixel -> coefficient step alone, one large image and one medium, odd-sized one
        {"name": "project_11x11", "kind": "project", "h": 2048, "w": 2048, "N": 11, "J": 6, "kmax": 8},
        {"name": "project_21x21", "kind": "project", "h": 487, "w": 641, "N": 21, "J": 10, "kmax": 12},
        # one dictionary update of the rotational K-SVD on 200,000 patches
        {"name": "learn_update", "kind": "update", "P": 200_000, "M": 128, "R": 64, "K": 5, "J": 6,
         "kmax": 8},
        # the way back: codes -> coefficients, coefficients -> pixels
        {"name": "reconstruct_1m", "kind": "reconstruct", "P": 1_000_000, "M": 64, "R": 64, "K": 5,
         "J": 6, "kmax": 8},
        {"name": "synthesize_1m", "kind": "synthesize", "P": 1_000_000, "N": 11, "J": 6, "kmax": 8},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["code", "code", "code", "host", "images", "project", "update", "reconstruct",
                       "synthesize"])
    wide = rng.random() < 0.3          # the 21 x 21 patches' coefficient sizes
    J, kmax, N = (10, 12, 21) if wide else (6, 8, 11)
    M, R, K = _logint(rng, 7, 256 if wide else 128), rng.choice([16, 32, 33, 60, 64, 64, 128]), \
        rng.randint(2, 8 if wide else 5)
    K = min(K, M)
    # steered atoms x coefficients x steps of one patch: what bounds the patch count
    per = M * R * (256 if wide else 112) * K
    if kind in ("code", "host"):
        c = _code("", _logint(rng, 500, min(1_000_000, int(2.0e12 / per))), M, R, K, J, kmax)
        c["kind"] = kind
        if kind == "code" and rng.random() < 0.25:
            c["precision"] = "fp32"
            c["P"] = min(c["P"], int(1.0e11 / per) + 1)
    elif kind == "images":
        top = min(600, int(math.sqrt(0.6e12 / per)))
        sides = ["%dx%d" % (_logint(rng, N + 12, max(top, N + 40)), _logint(rng, N + 12, max(top, N + 40)))
                 for _ in range(rng.randint(1, 4))]
        c = _images("", ",".join(sides), N, J, kmax, M, R, K)
    elif kind == "project":
        top = 900 if wide else 2048
        c = {"kind": kind, "h": _logint(rng, 64, top), "w": _logint(rng, 64, top), "N": N, "J": J,
             "kmax": kmax}
    elif kind == "update":
        c = {"kind": kind, "P": _logint(rng, 2000, 60_000 if wide else 200_000),
             "M": rng.choice([16, 24, 64, 100, 128]), "R": R, "K": rng.randint(2, 5), "J": 6, "kmax": 8}
    elif kind == "reconstruct":
        c = {"kind": kind, "P": _logint(rng, 1000, 400_000 if wide else 1_000_000), "M": M, "R": R, "K": K,
             "J": J, "kmax": kmax}
    else:
        c = {"kind": kind, "P": _logint(rng, 100, 300_000 if wide else 1_000_000), "N": N, "J": J,
             "kmax": kmax}
    c.pop("name", None)
    return c


# ------------------------------------------------------------------ inputs

def _generator(seed, part):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * int(seed) + part)
    return g


def _norm(c):
    """Coefficient-space norms of half spectra [..., H, J, 2]."""
    c = c.double()
    return (c[..., 0, :, 0].square().sum(-1) + 2.0 * c[..., 1:, :, :].square().sum((-1, -2, -3))).sqrt()


def _dictionary(M, J, kmax, seed):
    """Unit-norm atoms with Hermitian N(0, 1) spectra [M, H, J, 2] float32."""
    d = torch.randn((M, kmax + 1, J, 2), generator=_generator(seed, 1), device="cuda", dtype=F64)
    d[:, 0, :, 1] = 0.0
    return (d / _norm(d)[:, None, None, None]).float().contiguous()


def _steer(c, theta):
    """Half spectra [..., H, J] (complex) turned by theta [...]."""
    k = torch.arange(c.shape[-2], device=c.device, dtype=theta.dtype)
    ph = -theta[..., None] * k
    return c * torch.complex(ph.cos(), ph.sin())[..., None]


def _noise(P, H, J, sigma, g):
    n = torch.randn((P, H, J, 2), generator=g, device="cuda") * sigma
    n[:, 1:] *= math.sqrt(0.5)
    n[:, 0, :, 1] = 0.0
    return n


def _patches(d, P, sigma, seed):
    """Three steered atoms at continuous angles, N(0, 1) weights, noise."""
    M, H, J, _ = d.shape
    g = _generator(seed, 2)
    x = _noise(P, H, J, sigma, g)
    dc = torch.view_as_complex(d)
    for lo in range(0, P, 250_000):
        n = min(250_000, P - lo)
        for _ in range(3):
            m = torch.randint(0, M, (n,), generator=g, device="cuda")
            th = torch.rand((n,), generator=g, device="cuda") * (2.0 * math.pi)
            w = torch.randn((n,), generator=g, device="cuda")
            x[lo:lo + n] += torch.view_as_real(_steer(dc[m], th) * w[:, None, None])
    x[:, 0, :, 1] = 0.0
    return x.contiguous()


def _line_images(case, seed):
    """Textures of short line segments over noise (float32 [h, w] each)."""
    imgs = []
    for i, hw in enumerate(case["sides"].split(",") if "sides" in case else ["%dx%d" % (case["h"], case["w"])]):
        h, w = (int(v) for v in hw.split("x"))
        g = _generator(seed, 10 + i)
        img = 0.1 * torch.randn((h, w), generator=g, device="cuda")
        n = max(1, int(0.01 * h * w))
        cy = torch.rand((n,), generator=g, device="cuda") * h
        cx = torch.rand((n,), generator=g, device="cuda") * w
        th = torch.rand((n,), generator=g, device="cuda") * math.pi
        wt = torch.randn((n,), generator=g, device="cuda")
        u = torch.arange(-8, 9, device="cuda")
        yy = cy.floor().long()[:, None, None] + u[None, :, None]
        xx = cx.floor().long()[:, None, None] + u[None, None, :]
        dy, dx = yy - cy[:, None, None], xx - cx[:, None, None]
        co, si = th.cos()[:, None, None], th.sin()[:, None, None]
        along, across = dx * co + dy * si, dy * co - dx * si
        v = wt[:, None, None] * (5.5 - along.abs()).clamp(0.0, 1.0) * torch.exp(-0.5 * across.square())
        ok = (yy >= 0) & (yy < h) & (xx >= 0) & (xx < w)
        # whole numbers (2^-20) added up: the same image whatever the order of the additions
        q = torch.zeros(h * w, dtype=torch.int64, device="cuda")
        q.index_add_(0, (yy * w + xx)[ok], (v * 1048576.0).round().long()[ok])
        imgs.append((img + q.view(h, w).float() / 1048576.0).contiguous())
    return imgs


def _codes(P, M, R, K, g):
    """Codes as the coder writes them: K different atoms per patch, some atoms
    far more used than others, N(0, 1) weights in descending order."""
    pop = -1.0 * torch.log(1.0 + 0.05 * torch.arange(M, device="cuda", dtype=torch.float32))
    atom = torch.empty((P, K), dtype=torch.int32, device="cuda")
    for lo in range(0, P, 250_000):
        n = min(250_000, P - lo)
        u = torch.rand((n, M), generator=g, device="cuda").clamp_(1e-12, 1.0 - 1e-7)
        atom[lo:lo + n] = torch.topk(pop - torch.log(-torch.log(u)), K, dim=1).indices.int()
    ang = torch.randint(0, R, (P, K), generator=g, device="cuda", dtype=torch.int32)
    w = torch.randn((P, K), generator=g, device="cuda", dtype=F64)
    w = torch.gather(w, 1, torch.argsort(w.abs(), dim=1, descending=True)).contiguous()
    return {"atom": atom, "angle_idx": ang, "coef": w}


def _update_inputs(case, seed):
    """Patches made of planted atoms, their planted codes, and a dictionary
    that is some way off the planted one (an iteration in mid-learning)."""
    P, M, R, K, J, H = case["P"], case["M"], case["R"], case["K"], case["J"], case["kmax"] + 1
    true = _dictionary(M, J, case["kmax"], seed)
    off = true + 0.5 * _dictionary(M, J, case["kmax"], seed + 77_777)
    d = (off / _norm(off)[:, None, None, None].float()).contiguous()
    g = _generator(seed, 3)
    codes = _codes(P, M, R, K, g)
    x = _noise(P, H, J, 0.05, g)
    tc = torch.view_as_complex(true)
    for i in range(K):
        th = codes["angle_idx"][:, i].float() * (2.0 * math.pi / R)
        x += torch.view_as_real(_steer(tc[codes["atom"][:, i].long()], th)
                                * codes["coef"][:, i].float()[:, None, None])
    x[:, 0, :, 1] = 0.0
    return d, x.contiguous(), codes


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    if kind in ("code", "host"):
        d = _dictionary(case["M"], case["J"], case["kmax"], seed)
        s["dic"] = rsc.Dictionary(d, case["R"])
        s["x"] = _patches(d, case["P"], case["sigma"], seed)
        if kind == "host":
            P, K = case["P"], case["K"]
            s["x"] = s["x"].cpu().pin_memory()
            s["out"] = {"atom": torch.empty((P, K), dtype=torch.int32, pin_memory=True),
                        "angle_idx": torch.empty((P, K), dtype=torch.int32, pin_memory=True),
                        "angle": torch.empty((P, K), dtype=torch.float32, pin_memory=True),
                        "coef": torch.empty((P, K), dtype=F64, pin_memory=True),
                        "resid_norm2": torch.empty((P,), dtype=torch.float32, pin_memory=True)}
    elif kind in ("images", "project"):
        s["basis"] = rsc.Basis(case["N"], case["J"], case["kmax"])
        s["images"] = _line_images(case, seed)
        if kind == "images":
            s["dic"] = rsc.Dictionary(_dictionary(case["M"], case["J"], case["kmax"], seed), case["R"])
    elif kind == "update":
        d, s["x"], s["codes"] = _update_inputs(case, seed)
        s["dic"] = rsc.Dictionary(d, case["R"])
    elif kind == "reconstruct":
        s["dic"] = rsc.Dictionary(_dictionary(case["M"], case["J"], case["kmax"], seed), case["R"])
        s["codes"] = _codes(case["P"], case["M"], case["R"], case["K"], _generator(seed, 3))
    else:
        s["basis"] = rsc.Basis(case["N"], case["J"], case["kmax"])
        s["coef"] = _noise(case["P"], case["kmax"] + 1, case["J"], 1.0, _generator(seed, 3)).contiguous()
    return s


def run(s):
    c, kind = s["case"], s["kind"]
    if kind == "code":
        return rsc.encode(s["dic"], s["x"], c["K"], c["precision"])
    if kind == "host":
        return rsc.encode_host(s["dic"], s["x"], c["K"], c["precision"], out=s["out"])
    if kind == "images":
        return rsc.encode_images(s["dic"], s["basis"], s["images"], c["K"], c["precision"])
    if kind == "project":
        return rsc.project(s["basis"], s["images"][0])
    if kind == "update":
        new, used = rsc.ksvd_update(s["dic"], s["x"], s["codes"])
        return {"atoms": new, "used": used}
    if kind == "reconstruct":
        return rsc.reconstruct(s["dic"], s["codes"])
    return rsc.synthesize(s["basis"], s["coef"])


# -------------------------------------------------------------------- work

def _npix(N):
    c = (N - 1) / 2.0
    return sum((x - c) ** 2 + (y - c) ** 2 <= (N / 2.0) ** 2 for x in range(N) for y in range(N))


def _windows(case):
    sides = case.get("sides") or "%dx%d" % (case["h"], case["w"])
    hw = [tuple(int(v) for v in s.split("x")) for s in sides.split(",")]
    N = case["N"]
    return sum(max(h - N + 1, 0) * max(w - N + 1, 0) for h, w in hw), sum(h * w for h, w in hw)


def work(case):
    kind, J, kmax = case["kind"], case["J"], case["kmax"]
    vec, n = 2 * J * (kmax + 1), J * (2 * kmax + 1)
    coded = 0.0
    if "M" in case:
        M, R, K = case["M"], case["R"], case["K"]
        # per patch and step: the contraction per harmonic and a fast angle transform per atom
        coded = K * (2.0 * J * (1 + 4 * kmax) * M + 2.5 * R * math.log2(max(R, 2)) * M)
        codes = K * (4 + 4 + 8)
    if kind in ("code", "host"):
        return {"bytes": case["P"] * (4 * vec + codes + 4 * K + 4) + 4 * M * vec, "flops": case["P"] * coded}
    if kind in ("images", "project"):
        P, pixels = _windows(case)
        proj = 2.0 * _npix(case["N"]) * n
        if kind == "project":
            return {"bytes": 4 * pixels + P * 4 * vec, "flops": P * proj}
        return {"bytes": 4 * pixels + P * (codes + 4 * K + 4) + 4 * M * vec, "flops": P * (proj + coded)}
    P = case["P"]
    if kind == "update":
        # residuals, then one symmetric rank-1 term per patch and coded atom
        return {"bytes": P * (4 * vec + codes) + 2 * 4 * M * vec,
                "flops": P * K * (8.0 * vec + n * (n + 1))}
    if kind == "reconstruct":
        return {"bytes": P * (codes + 4 * vec) + 4 * M * vec, "flops": 8.0 * P * K * J * (kmax + 1)}
    npix = _npix(case["N"])
    return {"bytes": P * 4 * (vec + npix), "flops": 2.0 * P * n * npix}


# ---------------------------------------------------- the values in 64 bits

def _packed(c):
    """Half spectra [..., H, J] (complex128) as real vectors whose Euclidean
    product is the coefficient inner product."""
    a = c[..., 0, :].real
    b = torch.view_as_real(c[..., 1:, :].contiguous()).flatten(-3) * math.sqrt(2.0)
    return torch.cat([a, b], -1)


def _unpacked(v, H, J):
    out = torch.zeros(v.shape[:-1] + (H, J, 2), dtype=F64, device=v.device)
    out[..., 0, :, 0] = v[..., :J]
    out[..., 1:, :, :] = v[..., J:].reshape(v.shape[:-1] + (H - 1, J, 2)) / math.sqrt(2.0)
    return out


def _complex(c):
    z = torch.view_as_complex(c.double().contiguous()).clone()
    z[..., 0, :] = z[..., 0, :].real + 0j
    return z


def _omp64(x, d, R, K):
    """Orthogonal matching pursuit over the steered atoms in 64 bits."""
    P, (M, H, J, _) = x.shape[0], d.shape
    dc = _complex(d)
    th = torch.arange(R, device="cuda", dtype=F64) * (2.0 * math.pi / R)
    k = torch.arange(H, device="cuda", dtype=F64)
    wk = torch.where(k == 0, 1.0, 2.0)
    # Re(sum_k w_k e^{i k theta} G_k) as one real product over (k, re / im)
    tr = torch.stack([(k[:, None] * th).cos() * wk[:, None], -(k[:, None] * th).sin() * wk[:, None]], 1)
    tr = tr.reshape(2 * H, R)
    aug = _packed(_steer(dc[:, None].expand(M, R, H, J), th.expand(M, R))).reshape(M * R, -1)
    out = {"atom": torch.full((P, K), -1, dtype=torch.int32, device="cuda"),
           "angle_idx": torch.full((P, K), -1, dtype=torch.int32, device="cuda"),
           "angle": torch.zeros((P, K), dtype=F64, device="cuda"),
           "coef": torch.zeros((P, K), dtype=F64, device="cuda"),
           "resid_norm2": torch.zeros((P,), dtype=F64, device="cuda")}
    step = max(1024, int(6e8 / (M * R * 8)))
    for lo in range(0, P, step):
        xv = _packed(_complex(x[lo:lo + step]))
        r, n = xv, xv.shape[0]
        sel = torch.empty((n, 0), dtype=torch.long, device="cuda")
        for _ in range(K):
            rc = _complex(_unpacked(r, H, J))
            G = torch.matmul(rc.permute(1, 0, 2), dc.conj().permute(1, 2, 0))   # [H, n, M]
            G = torch.view_as_real(G).permute(1, 2, 0, 3).reshape(n, M, 2 * H)
            s = torch.matmul(G, tr).abs_().reshape(n, M * R)
            sel = torch.cat([sel, s.argmax(1)[:, None]], 1)
            A = aug[sel]                                                         # [n, t, N]
            a = torch.linalg.solve(A @ A.transpose(1, 2), (A @ xv[:, :, None]))[:, :, 0]
            r = xv - (a[:, None, :] @ A)[:, 0]
        hi = lo + n
        out["atom"][lo:hi], out["angle_idx"][lo:hi] = (sel // R).int(), (sel % R).int()
        out["angle"][lo:hi] = th[sel % R]
        out["coef"][lo:hi] = a
        out["resid_norm2"][lo:hi] = r.square().sum(1)
    return out


def _basis64(N, J, kmax):
    """Pixel offsets and the real synthesis matrix [npix, n] (packed order) of
    the steerable basis: Gaussian rings times circular harmonics, orthonormal
    within each harmonic, on the pixels within N / 2 of the centre."""
    c = (N - 1) / 2.0
    col, row = np.meshgrid(np.arange(N), np.arange(N))
    x, y = col - c, c - row
    rho, phi = np.hypot(x, y), np.arctan2(y, x)
    ok = rho <= N / 2.0
    rho, phi = rho[ok], phi[ok]
    prof = np.exp(-0.5 * (rho[:, None] - (N - 1) / (2.0 * J) * (np.arange(J) + 1)) ** 2)
    qs = []
    for drop in (False, True):
        B = prof * ~((rho == 0.0) & drop)[:, None]
        w, V = np.linalg.eigh(B.T @ B)
        qs.append(B @ (V / np.sqrt(w)) @ V.T)
    X = [qs[0]]
    for k in range(1, kmax + 1):
        cs = np.stack([np.cos(k * phi), -np.sin(k * phi)], -1)
        X.append((math.sqrt(2.0) * qs[1][:, :, None] * cs[:, None, :]).reshape(len(rho), 2 * J))
    return row[ok], col[ok], np.concatenate(X, 1)


def _project64(case, img):
    rows, cols, X = _basis64(case["N"], case["J"], case["kmax"])
    op = torch.from_numpy(np.linalg.pinv(X, rcond=1e-3)).cuda()
    N, J, H = case["N"], case["J"], case["kmax"] + 1
    h, w = img.shape
    img = img.double()
    out = torch.empty(((h - N + 1) * (w - N + 1), H, J, 2), dtype=F64, device="cuda")
    nw, step = w - N + 1, max(1, 200_000 // (w - N + 1))
    for r in range(0, h - N + 1, step):
        e = min(h - N + 1, r + step)
        px = torch.stack([img[r + dy:e + dy, dx:dx + nw].reshape(-1)
                          for dy, dx in zip(rows.tolist(), cols.tolist())], 1)
        out[r * nw:e * nw] = _unpacked(px @ op.T, H, J)
    return out


def _update64(case, seed):
    d, x, codes = _update_inputs(case, seed)
    M, R, K, J, H = case["M"], case["R"], case["K"], case["J"], case["kmax"] + 1
    dc, xc = _complex(d), _complex(x)
    atom, w = codes["atom"].long(), codes["coef"]
    th = codes["angle_idx"].double() * (2.0 * math.pi / R)
    e = xc.clone()
    for i in range(K):
        e -= _steer(dc[atom[:, i]], th[:, i]) * w[:, i, None, None]
    new = d.double().clone()
    used = torch.zeros(M, dtype=torch.int32)
    ys = [_packed(_steer(e, -th[:, i]) + dc[atom[:, i]] * w[:, i, None, None]) for i in range(K)]
    for m in range(M):
        Y = torch.cat([ys[i][atom[:, i] == m] for i in range(K)])
        used[m] = Y.shape[0]
        if Y.shape[0] == 0:
            return None  # an unused atom is reset: not a computed value
        v = np.linalg.eigh((Y.T @ Y).cpu().numpy())[1][:, -1]
        v = v * (1.0 if v[np.argmax(np.abs(v))] > 0 else -1.0)
        new[m] = _unpacked(torch.from_numpy(v.copy()).cuda(), H, J)
    return {"atoms": new, "used": used}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("code", "host"):
        d = _dictionary(case["M"], case["J"], case["kmax"], seed)
        return _omp64(_patches(d, case["P"], case["sigma"], seed), d, case["R"], case["K"])
    if kind == "project":
        return _project64(case, _line_images(case, seed)[0])
    if kind == "images":
        # which atom is picked turns on the last bits of the projected window
        # wherever two scores nearly tie: the weights have no value of their own
        return None
    if kind == "update":
        return _update64(case, seed)
    if kind == "reconstruct":
        d = _complex(_dictionary(case["M"], case["J"], case["kmax"], seed))
        c = _codes(case["P"], case["M"], case["R"], case["K"], _generator(seed, 3))
        out = torch.empty((case["P"],) + d.shape[1:] + (2,), dtype=F64, device="cuda")
        for lo in range(0, case["P"], 100_000):
            s = slice(lo, lo + 100_000)
            th = c["angle_idx"][s].double() * (2.0 * math.pi / case["R"])
            out[s] = torch.view_as_real((_steer(d[c["atom"][s].long()], th)
                                         * c["coef"][s][:, :, None, None]).sum(1))
        return out
    X = torch.from_numpy(_basis64(case["N"], case["J"], case["kmax"])[2]).cuda()
    coef = _noise(case["P"], case["kmax"] + 1, case["J"], 1.0, _generator(seed, 3))
    return torch.cat([_packed(_complex(coef[lo:lo + 100_000])) @ X.T for lo in range(0, case["P"], 100_000)])
