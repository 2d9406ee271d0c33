"""The work that programs have this library do, as cases that can be timed and compared.

A case is a dict of plain values.  ``listed()`` names the fixed ones, ``draw(rng)`` makes one more of the
same ranges, ``prepare(case, seed)`` builds what a program holds before the call (inputs from the seed alone,
geometry, batch or engine), ``run(state)`` is one pass through the public entry points, ``work(case)`` the
bytes and operations that a pass cannot do without, and ``exact(case, seed)`` the same outputs from plain
torch in 64 bits (written here from the definitions; nothing of the library is used).

Kinds of case:

- "project", "backproject": A x and B b alone, as programs that use the projector pair call them;
- "cgs2": one Arnoldi step of a caller's own Krylov loop;
- "solve": ab_gmres / ba_gmres as the README calls them;
- "batch": a handle made once, many different solves per call;
- "serve": a standing engine that takes a burst of requests and drains it.

Right-hand sides are A x_bar + white noise with x_bar an image of random ellipses, from the 64-bit projector
below.  Noise is 2-5 %, where the discrepancy principle stops early and the iterate is a well-conditioned
function of the rounding.  Coefficients and residual histories are FP32 sums in FP64 containers; they are
returned as FP32.
"""
import math
import random

import numpy as np
import torch

import paper_2110_01481_gb300 as P

SQRT2 = math.sqrt(2.0)


def _det(N, spacing=1.0):
    return math.ceil(SQRT2 * N / spacing)


def _geo(N, n_angles, n_det=None, start=0, range_=180, spacing=1.0, model="pixel"):
    return {"N": N, "angles": n_angles, "det": _det(N, spacing) if n_det is None else n_det, "start": start,
            "range": range_, "spacing": spacing, "model": model}


def listed():
    return [
        # the smallest problem of the test suite and of the paper-sized demos: launch latency
        {"name": "project_64", "kind": "project", **_geo(64, 90)},
        # A at the benchmark's size, the ordinary forward projection
        {"name": "project_512", "kind": "project", **_geo(512, 720)},
        # A at the largest configuration (2048 x 2048, 1800 angles): the most work of one call
        {"name": "project_2048", "kind": "project", **_geo(2048, 1800)},
        # B at the benchmark's size, the ordinary unmatched back projection
        {"name": "backproject_512", "kind": "backproject", **_geo(512, 720)},
        # A^T on an odd image with a ragged detector and a limited-angle scan: comparisons with the matched pair
        {"name": "backproject_matched_361", "kind": "backproject",
         **_geo(361, 187, n_det=517, range_=120, model="matched")},
        # an Arnoldi step deep in an unstopped solve on a 2048 x 2048 image: streaming the basis from HBM
        {"name": "cgs2_2048_k60", "kind": "cgs2", "L": 2048 * 2048, "k": 60},
        # a small solve with a fixed number of steps (64 x 64, 90 angles): the latency of a step
        {"name": "solve_ba_64", "kind": "solve", "variant": "ba", **_geo(64, 90), "noise": 0.02, "dp": False,
         "maxit": 8, "steps": 8, "basis": "fp32"},
        # AB-GMRES with the discrepancy stop at the benchmark's size, as in the README
        {"name": "solve_ab_512", "kind": "solve", "variant": "ab", **_geo(512, 720), "noise": 0.02, "dp": True,
         "maxit": 150, "steps": 11, "basis": "fp32"},
        # BA-GMRES with the discrepancy stop at the benchmark's size: a two-image projection in every step
        {"name": "solve_ba_512", "kind": "solve", "variant": "ba", **_geo(512, 720), "noise": 0.04, "dp": True,
         "maxit": 150, "steps": 9, "basis": "fp32"},
        # AB-GMRES with a 16-bit basis on a larger, odd-sized problem
        {"name": "solve_ab_fp16_1001", "kind": "solve", "variant": "ab", **_geo(1001, 900), "noise": 0.03, "dp": False,
         "maxit": 6, "steps": 6, "basis": "fp16"},
        # a batch of uneven solves (sizes, angle counts, scans, both variants) held by one handle
        {"name": "batch_16", "kind": "batch", "count": 16, "mix": 3, "sizes": "128,256,512"},
        # a burst of requests to a standing engine
        {"name": "serve_12", "kind": "serve", "count": 12, "mix": 5, "sizes": "128,256,512"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["project", "project", "backproject", "backproject", "cgs2", "solve", "solve", "batch"])
    if kind == "cgs2":
        L = _log_int(rng, 4096, 2048 * 2048)
        return {"kind": kind, "L": L, "k": min(_log_int(rng, 1, 150), max(1, 2048 * 2048 * 60 // L))}
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(2, 16), "mix": rng.randrange(1 << 20),
                "sizes": rng.choice(["128,256", "128,256,512", "64,200,333"])}
    top = 2048 if kind != "solve" else 1024
    N = _log_int(rng, 64, top)
    range_, start = rng.choice([(180, 0), (180, 0), (180, 15), (120, 0), (360, 0)])
    spacing = rng.choice([1.0, 1.0, 1.0, 0.75, 1.3])
    a = _log_int(rng, 60, 1800 if kind != "solve" else 900)
    g = _geo(N, a, n_det=_det(N, spacing) + rng.randint(0, 5), start=start, range_=range_, spacing=spacing)
    if kind == "project":
        return {"kind": kind, **g}
    if kind == "backproject":
        g["model"] = rng.choice(["pixel", "pixel", "matched"])
        return {"kind": kind, **g}
    variant = rng.choice(["ab", "ba"])
    dp = rng.random() < 0.5
    steps = rng.randint(3, 6)
    return {"kind": kind, "variant": variant, **g, "noise": round(rng.uniform(0.03, 0.05), 3), "dp": dp,
            "maxit": 8 if dp else steps, "steps": steps, "basis": "fp16" if variant == "ab" and rng.random() < 0.3 else "fp32"}


def _mix(case):
    """The solves of a batch or a burst: sizes, angle counts, a quarter limited-angle scans, AB and BA."""
    r = random.Random(case["mix"])
    sizes = [int(s) for s in case["sizes"].split(",")]
    out = []
    for i in range(case["count"]):
        N, a = r.choice(sizes), r.choice([60, 180, 360, 720])
        out.append({**_geo(N, a, range_=120 if r.random() < 0.25 else 180), "variant": "ab" if i % 2 == 0 else "ba",
                    "noise": round(r.uniform(0.02, 0.05), 4), "dp": True, "maxit": 60, "steps": 8, "basis": "fp32"})
    return out


# ---- inputs ------------------------------------------------------------------------------------------------


def _geometry(c):
    return P.Geometry(c["N"], c["angles"], c["det"], c["start"], c["range"], c["spacing"], back_model=c["model"])


def _ellipses(N, seed):
    """Random ellipses (painter's order) on [-1, 1]^2, as N x N floats on the GPU."""
    r = np.random.Generator(np.random.PCG64(seed))
    t = (torch.arange(N, device="cuda", dtype=torch.float32) - (N - 1) / 2) * (2.0 / N)
    y, x = t[:, None], t[None, :]
    img = torch.zeros(N, N, device="cuda")
    for _ in range(20):
        rad, phi = 0.7 * math.sqrt(r.uniform()), r.uniform(0, 2 * math.pi)
        ax, ay = r.uniform(0.05, 0.4, 2)
        th, val = r.uniform(0, math.pi), r.uniform()
        dx, dy = x - rad * math.cos(phi), y - rad * math.sin(phi)
        u = (dx * math.cos(th) + dy * math.sin(th)) / ax
        v = (dy * math.cos(th) - dx * math.sin(th)) / ay
        img = torch.where(u * u + v * v <= 1.0, torch.full_like(img, val), img)
    return img


def _noisy_data(c, seed):
    """b = A x_bar + e as FP32, and ||e||."""
    b = _forward64(c, _ellipses(c["N"], seed).double())
    gen = torch.Generator(device="cuda").manual_seed(seed)
    e = torch.randn(b.shape, generator=gen, device="cuda", dtype=torch.float64)
    e *= c["noise"] * torch.linalg.vector_norm(b) / torch.linalg.vector_norm(e)
    return (b + e).float().reshape(-1), float(torch.linalg.vector_norm(e))


def _basis(L, k, seed):
    """k orthonormal FP32 rows of length L (Cholesky QR, twice) and a vector with a part outside their span."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    ld = (L + 63) // 64 * 64
    W = torch.zeros(max(k, 1), ld, device="cuda")
    V = W[:, :L]
    V.normal_(generator=gen)
    for _ in range(2):
        G = torch.zeros(W.shape[0], W.shape[0], device="cuda", dtype=torch.float64)
        for s in range(0, L, 1 << 20):
            D = V[:, s:s + (1 << 20)].double()
            G += D @ D.T
        R = torch.linalg.inv(torch.linalg.cholesky(G))
        for s in range(0, L, 1 << 20):
            V[:, s:s + (1 << 20)] = (R @ V[:, s:s + (1 << 20)].double()).float()
    q = torch.randn(L, generator=gen, device="cuda")
    q += (torch.randn(V.shape[0], generator=gen, device="cuda") * math.sqrt(L)) @ V
    return W, q


def prepare(case, seed):
    kind = case["kind"]
    if kind == "project":
        g = _geometry(case)
        gen = torch.Generator(device="cuda").manual_seed(seed)
        # an iterate of a noisy solve: piecewise constant with noise on it
        x = _ellipses(case["N"], seed) + 0.05 * torch.randn(case["N"], case["N"], generator=gen, device="cuda")
        P.Context.get("cuda").tuning(g)      # the geometry's tables and tile shapes, made once by any program
        return {"kind": kind, "g": g, "x": x.contiguous()}
    if kind == "backproject":
        g = _geometry(case)
        gen = torch.Generator(device="cuda").manual_seed(seed)
        b = torch.randn(case["angles"], case["det"], generator=gen, device="cuda")
        t = torch.linspace(-1, 1, case["det"], device="cuda")
        P.Context.get("cuda").tuning(g)
        return {"kind": kind, "g": g, "b": (b + 4.0 * torch.sqrt(torch.clamp(1 - t * t, min=0.0))).contiguous()}
    if kind == "cgs2":
        W, q = _basis(case["L"], case["k"], seed)
        return {"kind": kind, "W": W, "k": case["k"], "q": q}
    if kind == "solve":
        b, e = _noisy_data(case, seed)
        g = _geometry(case)
        P.Context.get("cuda").tuning(g)
        return {"kind": kind, "g": g, "b": b, "variant": case["variant"], "maxit": case["maxit"],
                "noise_norm": e if case["dp"] else None, "basis": case["basis"]}
    probs = _mix(case)
    data = [_noisy_data(p, seed + i) for i, p in enumerate(probs)]
    asked = [{"geometry": _geometry(p), "variant": p["variant"], "maxit": p["maxit"], "tau": 1.02, "noise_norm": e}
             for p, (_, e) in zip(probs, data)]
    bs = [b for b, _ in data]
    if kind == "batch":
        # a handle's options hold the noise levels of its data
        return {"kind": kind, "batch": P.Batch(asked), "asked": asked, "bs": bs}
    return {"kind": kind, "engine": P.Engine(max_slots=64, hbm_budget_bytes=16 << 30), "asked": asked, "bs": bs}


# ---- one pass ----------------------------------------------------------------------------------------------


def _padded(history, maxit):
    """A history as the C call fills it: maxit + 1 entries, zero past the last step."""
    out = np.zeros(maxit + 1)
    out[:len(history)] = history
    return out


def _solved(r, maxit):
    return {"x": r.x, "history": _padded(r.history, maxit).astype(np.float32), "iters": r.iters}


def run(s):
    kind = s["kind"]
    if kind == "project":
        return P.project(s["g"], s["x"])
    if kind == "backproject":
        return P.backproject(s["g"], s["b"])
    if kind == "cgs2":
        q = s["q"].clone()                       # the step overwrites its vector
        h, w = P.cgs2(s["W"], s["k"], q)
        return {"h": h.float(), "w": w, "q": q}
    if kind == "solve":
        solve = P.ab_gmres if s["variant"] == "ab" else P.ba_gmres
        r = solve(s["g"], s["b"], s["maxit"], tau=1.02, noise_norm=s["noise_norm"], basis=s["basis"])
        return _solved(r, s["maxit"])
    if kind == "batch":
        return [_solved(r, a["maxit"]) for a, r in zip(s["asked"], s["batch"].solve(s["bs"]))]
    eng = s["engine"]
    for i, (a, b) in enumerate(zip(s["asked"], s["bs"])):
        eng.submit(a["geometry"], b, a["variant"], a["maxit"], a["tau"], a["noise_norm"], tag=i)
    return [_solved(r, s["asked"][i]["maxit"]) for i, r in sorted(eng.drain(), key=lambda d: d[0])]


# ---- the work of a pass ------------------------------------------------------------------------------------


def _turns(c):
    """(cos, sin, row-driven) of the angles, in 64 bits."""
    a = np.arange(c["angles"], dtype=np.int64)
    num = c["start"] * c["angles"] + a * c["range"]                    # theta_a * n_angles, in degrees
    T, half = num % (180 * c["angles"]), 180 * c["angles"]
    th = num / half * math.pi
    return np.cos(th), np.sin(th), (4 * T <= half) | (4 * T >= 3 * half)


def _taps(c):
    """Interpolations of one A: on a row of N pixels, (N + 1) |c| / spacing rays of an angle have a tap."""
    cs, sn, rd = _turns(c)
    return c["N"] * (c["N"] + 1) * float(np.where(rd, np.abs(cs), np.abs(sn)).sum()) / c["spacing"]


def _solve_work(c):
    n, m = c["N"] ** 2, c["angles"] * c["det"]
    L, es, k = (m if c["variant"] == "ab" else n), (2 if c["basis"] != "fp32" else 4), c["steps"]
    # BA's discrepancy test projects x_k as well
    fwd = (2 if c["variant"] == "ba" and c["dp"] else 1) * k + 1
    back = k + 1
    basis = sum(3 * j * L * es + 3 * L * 4 for j in range(1, k + 1)) + k * L * es
    return {"bytes": basis + 4 * (n + m) * (fwd + back), "flops": 4 * (fwd * _taps(c) + back * n * c["angles"]) + 2 * basis}


def work(case):
    kind = case["kind"]
    if kind in ("project", "backproject"):
        n, m = case["N"] ** 2, case["angles"] * case["det"]
        taps = _taps(case) if kind == "project" or case["model"] != "pixel" else n * case["angles"]
        return {"bytes": 4 * (n + m), "flops": 4 * taps}
    if kind == "cgs2":
        return {"bytes": 4 * case["L"] * (case["k"] + 3), "flops": 8 * case["L"] * case["k"]}
    if kind == "solve":
        return _solve_work(case)
    each = [_solve_work(p) for p in _mix(case)]
    return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}


# ---- 64-bit results from the definitions -------------------------------------------------------------------


def _chunks(sel, per):
    return [sel[i:i + per] for i in range(0, len(sel), per)]


def _forward64(c, x):
    """Joseph's A x (angles x det): lerp along rows (or columns) at the ray's crossing, over |cos| (|sin|)."""
    N, nd, ds = c["N"], c["det"], c["spacing"]
    cs, sn, rd = _turns(c)
    h = (N - 1) / 2
    t = torch.arange(N, device="cuda", dtype=torch.float64) - h
    sd = (torch.arange(nd, device="cuda", dtype=torch.float64) - (nd - 1) / 2) * ds
    out = torch.zeros(c["angles"], nd, device="cuda", dtype=torch.float64)
    for rows, img in ((True, x), (False, x.T)):
        pimg = torch.nn.functional.pad(img, (2, 2)).contiguous().reshape(-1)
        base = torch.arange(N, device="cuda") * (N + 4) + 2
        for sel in _chunks(np.flatnonzero(rd == rows), max(1, (1 << 27) // (N * nd))):
            ca = torch.tensor((cs if rows else sn)[sel], device="cuda")[:, None, None]
            sa = torch.tensor((sn if rows else cs)[sel], device="cuda")[:, None, None]
            u = (sd[None, :, None] - t[None, None, :] * sa) / ca + h
            j = torch.clamp(torch.floor(u), -2, N)
            f = torch.clamp(u - j, 0.0, 1.0)
            at = base + j.long()
            v0 = pimg[at]
            out[torch.as_tensor(sel, device="cuda")] = ((v0 + f * (pimg[at + 1] - v0)).sum(2) / ca[:, :, 0].abs())
    return out


def _back64(c, b, add=None):
    """B b (N x N): pixel-driven lerp on the detector, or the exact transpose of A ("matched")."""
    N, nd, ds = c["N"], c["det"], c["spacing"]
    cs, sn, rd = _turns(c)
    b = b.reshape(c["angles"], nd)
    wide = 2 + (0 if c["model"] == "pixel" else math.ceil(1 / ds))
    pb = torch.nn.functional.pad(b, (wide + 1, wide + 1))
    t = torch.arange(N, device="cuda", dtype=torch.float64) - (N - 1) / 2
    x = torch.zeros(N, N, device="cuda", dtype=torch.float64)
    for sel in _chunks(np.arange(c["angles"]), max(1, (1 << 26) // (N * N))):
        ca = torch.tensor(cs[sel], device="cuda")[:, None, None]
        sa = torch.tensor(sn[sel], device="cuda")[:, None, None]
        u = (t[None, None, :] * ca + t[None, :, None] * sa) / ds + (nd - 1) / 2
        d = torch.floor(u)
        f = u - d
        row = torch.as_tensor(sel, device="cuda")[:, None, None] * pb.shape[1] + wide + 1
        flat = pb.reshape(-1)

        def bins(e):
            return flat[row + torch.clamp(d + e, -wide - 1, nd + wide).long()]
        if c["model"] == "pixel":
            v0 = bins(0)
            x += (v0 + f * (bins(1) - v0)).sum(0)
            continue
        w = torch.tensor(np.where(rd, np.abs(cs), np.abs(sn))[sel], device="cuda")[:, None, None]
        reach = math.ceil(1 / ds)
        for e in range(1 - reach, reach + 1):
            x += (torch.clamp(1 - (e - f).abs() * ds / w, min=0.0) / w * bins(e)).sum(0)
    return x


def _gmres64(c, b, noise_norm):
    """AB- or BA-GMRES in 64 bits: (x_k, residual history, k)."""
    ab, target = c["variant"] == "ab", 1.02 * noise_norm if c["dp"] else 0.0
    b = b.double()

    def A(v):
        return _forward64(c, v.reshape(c["N"], c["N"])).reshape(-1)

    def B(v):
        return _back64(c, v).reshape(-1)
    norm = torch.linalg.vector_norm
    r0 = b if ab else B(b)
    beta, res = norm(r0), float(norm(b))
    W, H = [r0 / beta], np.zeros((c["maxit"] + 1, c["maxit"]))
    hist = [float(beta) if ab or not c["dp"] else res]
    x = torch.zeros(c["N"] ** 2, device="cuda", dtype=torch.float64)
    k = 0
    while k < c["maxit"] and not (c["dp"] and hist[-1] <= target):
        q = A(B(W[k])) if ab else B(A(W[k]))
        V = torch.stack(W)
        for _ in range(2):
            h = V @ q
            q = q - h @ V
            H[:k + 1, k] += h.cpu().numpy()
        H[k + 1, k] = float(norm(q))
        W.append(q / norm(q))
        k += 1
        rhs = np.zeros(k + 1)
        rhs[0] = float(beta)
        y = np.linalg.lstsq(H[:k + 1, :k], rhs, rcond=None)[0]
        u = torch.tensor(y, device="cuda") @ torch.stack(W[:k])
        if ab or not c["dp"]:
            hist.append(float(np.linalg.norm(rhs - H[:k + 1, :k] @ y)))
            x = u
        else:
            x = u
            hist.append(float(norm(b - A(x))))
    return {"x": B(x) if ab and k else x, "history": _padded(hist, c["maxit"]), "iters": None}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("project", "backproject"):
        if case["N"] ** 2 * case["angles"] > 2048 ** 2 * 1800:
            return None
        s = prepare(case, seed)
        if kind == "project":
            return _forward64(case, s["x"].double()).reshape(-1)
        return _back64(case, s["b"].double()).reshape(-1)
    if kind == "cgs2":
        s = prepare(case, seed)
        q, W = s["q"].double(), s["W"][:, :case["L"]]
        h = torch.zeros(W.shape[0], device="cuda", dtype=torch.float64)
        for _ in range(2):
            g = torch.stack([torch.dot(w.double(), q) for w in W])
            for gj, w in zip(g, W):
                q = q - gj * w.double()
            h += g
        nrm = torch.linalg.vector_norm(q)
        return {"h": torch.cat([h, nrm[None]]), "w": q / nrm, "q": q}
    if kind == "solve":
        b, e = _noisy_data(case, seed)
        return _gmres64(case, b, e)
    return [_gmres64(p, *_noisy_data(p, seed + i)) for i, p in enumerate(_mix(case))]
