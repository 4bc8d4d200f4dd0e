"""The calls a user of the slicing framework makes, as cases that can be timed and compared.

Sizes are those of the repository's own configurations: the real n = 2000, b = 32 matrix with
one slice of 100 eigenvalues, the complex n = 8192, b = 64 sequence with 8 slices of 205 and
subspaces of 267 columns, the b = 128 matrices, and the n = 16384 bands of the slice proposal.
"""
import math

import torch

import paper_2012_00506_gb300 as pk
from paper_2012_00506_gb300 import slicer

DEV = "cuda"


# --------------------------------------------------------------------------- cases
def listed():
    return [
        # single eigenvalues of a small band: a handful of shifts at a time, latency bound
        {"name": "bisect_small", "kind": "bisect", "n": 2000, "b": 32, "cplx": False, "count": 8},
        # exact counts at the boundaries of the 8 slices of one step of a sequence
        {"name": "counts_step", "kind": "counts", "n": 8192, "b": 64, "cplx": True, "count": 9},
        # a first partition of an unknown spectrum: hundreds of shifts at a time
        {"name": "propose", "kind": "propose", "n": 16384, "b": 64, "cplx": True, "count": 64},
        # one Adam step of the proposal network (forward, backward, update)
        {"name": "train_step", "kind": "train", "batch": 64},
        # the shifted systems of one slice in FP64
        {"name": "solve_fp64", "kind": "solve", "n": 2000, "b": 32, "cplx": False, "shifts": 8, "cols": 150,
         "mixed": False, "adjoint": False},
        # the shifted systems of one slice in complex64, the normal ones ...
        {"name": "solve_mixed", "kind": "solve", "n": 8192, "b": 64, "cplx": True, "shifts": 8, "cols": 267,
         "mixed": True, "adjoint": False},
        # ... and the adjoint ones of the conjugate nodes, on a wide band
        {"name": "solve_wide_adjoint", "kind": "solve", "n": 16384, "b": 128, "cplx": True, "shifts": 16,
         "cols": 201, "mixed": True, "adjoint": True},
        # the tall products of one Rayleigh-Ritz step of 8 slices
        {"name": "rr_products", "kind": "products", "n": 8192, "b": 64, "cplx": True, "blocks": 8, "cols": 267},
        # orthonormal bases of uneven blocks in FP64
        {"name": "cholqr_uneven", "kind": "cholqr", "n": 5003, "cplx": False, "blocks": 3, "cols": 131, "passes": 2},
        # the projected eigenproblems of 8 slices
        {"name": "eigh_slices", "kind": "eigh", "cplx": True, "blocks": 8, "cols": 267},
        # a whole call with nothing but defaults beside FP64: one slice, the norm by the library
        {"name": "slice_fp64", "kind": "slice", "n": 2000, "b": 32, "cplx": False, "slices": 1, "per": 100,
         "start": 0.25, "mixed": False, "norm": False},
        # a whole mixed-precision call: one step of the complex sequence from a random start
        {"name": "slice_step", "kind": "slice", "n": 8192, "b": 64, "cplx": True, "slices": 8, "per": 205,
         "start": 0.0, "mixed": True, "norm": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["bisect", "counts", "counts", "propose", "train", "solve", "solve", "solve", "products",
                       "cholqr", "eigh", "slice", "slice"])
    cplx = rng.random() < 0.5
    if kind == "bisect":
        return {"kind": kind, "n": _log(rng, 300, 5000), "b": _log(rng, 4, 64), "cplx": cplx,
                "count": rng.randint(1, 24)}
    if kind == "counts":
        return {"kind": kind, "n": _log(rng, 500, 16384), "b": _log(rng, 8, 140), "cplx": cplx,
                "count": _log(rng, 1, 150)}
    if kind == "propose":
        return {"kind": kind, "n": _log(rng, 1000, 12000), "b": _log(rng, 8, 64), "cplx": cplx,
                "count": rng.choice([8, 16, 32, 64])}
    if kind == "train":
        return {"kind": kind, "batch": rng.randint(1, 256)}
    if kind == "solve":
        mixed = rng.random() < 0.6
        return {"kind": kind, "n": _log(rng, 500, 16000 if mixed else 3000), "b": _log(rng, 8, 128 if mixed else 64),
                "cplx": cplx, "shifts": rng.randint(1, 16 if mixed else 8), "cols": _log(rng, 4, 267 if mixed else 160),
                "mixed": mixed, "adjoint": rng.random() < 0.5}
    if kind == "products":
        return {"kind": kind, "n": _log(rng, 1000, 9000), "b": _log(rng, 8, 128), "cplx": cplx,
                "blocks": rng.randint(1, 8), "cols": _log(rng, 20, 290)}
    if kind == "cholqr":
        return {"kind": kind, "n": _log(rng, 500, 8192), "cplx": cplx, "blocks": rng.randint(1, 4),
                "cols": _log(rng, 16, 200), "passes": rng.randint(1, 2)}
    if kind == "eigh":
        return {"kind": kind, "cplx": cplx, "blocks": rng.randint(1, 8), "cols": _log(rng, 12, 290)}
    mixed = rng.random() < 0.6
    return {"kind": "slice", "n": _log(rng, 1500, 7000 if mixed else 2400), "b": _log(rng, 8, 64 if mixed else 32),
            "cplx": cplx, "slices": rng.randint(1, 6 if mixed else 2), "per": rng.randint(30, 100),
            "start": rng.uniform(0.0, 0.5), "mixed": mixed, "norm": rng.random() < 0.5}


# --------------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _normal(g, shape, cplx, sigma=1.0):
    if cplx:
        x = torch.randn(tuple(shape) + (2,), generator=g, device=DEV, dtype=torch.float64) * (sigma * math.sqrt(0.5))
        return torch.view_as_complex(x)
    return torch.randn(shape, generator=g, device=DEV, dtype=torch.float64) * sigma


def _band(g, n, b, cplx, off):
    """Diagonal U[-1, 1], off-diagonals N(0, off^2), compact lower storage, zeros outside the matrix."""
    band = _normal(g, (n, b + 1), cplx, off)
    band[:, 0] = torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * 2.0 - 1.0
    j = torch.arange(n, device=DEV)[:, None]
    d = torch.arange(b + 1, device=DEV)[None, :]
    return torch.where(j + d < n, band, torch.zeros((), dtype=band.dtype, device=DEV)).contiguous()


def _sizes(blocks, cols):
    """Uneven column blocks of about `cols` columns (the first as given)."""
    return [max(1, cols - (37 * t) % max(2, cols // 2) if t % 3 else cols) for t in range(blocks)]


def prepare(case, seed):
    g = _gen(seed)
    k = case["kind"]
    s = {"case": case}
    if k in ("bisect", "counts", "propose", "solve", "slice", "products"):
        s["band"] = _band(g, case["n"], case["b"], case["cplx"], 0.1 if case["b"] <= 64 else 0.05)
    if k == "bisect":
        s["idx"] = torch.randperm(case["n"], generator=g, device=DEV)[:case["count"]].sort().values.cpu().numpy()
    elif k == "counts":
        s["sigma"] = (torch.rand(case["count"], generator=g, device=DEV, dtype=torch.float64) * 2.4
                      - 1.2).sort().values.cpu().numpy()
    elif k == "propose":
        s["params"] = slicer.init_params(seed % 1000, DEV)
    elif k == "train":
        s["trainer"] = slicer.Trainer(slicer.init_params(seed % 1000, DEV), lr=1e-3, max_batch=256)
        s["trainer"].t = 200  # a step in the middle of a training run: moments of the size of the gradient
        s["trainer"].m += 1e-3 * torch.randn(s["trainer"].m.shape, generator=g, device=DEV)
        s["trainer"].v += 1e-6 + 1e-5 * torch.rand(s["trainer"].v.shape, generator=g, device=DEV)
        s["x"] = torch.rand((case["batch"], slicer.N_FEAT), generator=g, device=DEV)
        s["t"] = torch.rand((case["batch"], slicer.N_BOUNDS), generator=g, device=DEV).sort(dim=1).values
    elif k == "solve":
        s["shifts"] = pk.contour_rule(case["shifts"], -0.31, -0.22)[0]
        s["rhs"] = _normal(g, (case["cols"], case["n"]), True)
    elif k in ("products", "cholqr"):
        s["m"] = _sizes(case["blocks"], case["cols"])
        s["q"] = _normal(g, (sum(s["m"]), case["n"]), case["cplx"])
        if k == "products":
            s["w"] = [_normal(g, (m, m), case["cplx"]) for m in s["m"]]
    elif k == "eigh":
        s["a"] = []
        for m in _sizes(case["blocks"], case["cols"]):
            # a projected matrix of a slice: eigenvalues spread over the slice, eigenvectors general
            x = _normal(g, (m, m), case["cplx"])
            s["a"].append((x + x.conj().T) / (2.0 * math.sqrt(m)))
    elif k == "slice":
        n, K, per = case["n"], case["slices"], case["per"]
        f0 = case["start"]
        p = slicer.propose_slices(s["band"], nslices=K, frac=(f0, f0 + K * per / n), count_tol=0)
        s["bounds"] = p.bounds
        s["m0"] = [min(n, max(math.ceil(1.3 * int(c)), int(c) + 10)) for c in p.counts]
        s["x0"] = _normal(g, (sum(s["m0"]), n), case["cplx"])
        s["opts"] = {"precision": pk.MIXED if case["mixed"] else pk.FP64}
        if case["norm"]:
            lo, hi = pk.bisect(s["band"], [0, n - 1], rtol=1e-6, fanout=16)
            s["opts"]["bnorm"] = float(max(abs(lo[0]), abs(hi[0]), abs(lo[1]), abs(hi[1])))
        o = pk.default_opts(**s["opts"])
        size = pk.workspace_size(n, case["b"], case["cplx"], s["m0"], 8, o)
        s["work"] = torch.empty(size, dtype=torch.uint8, device=DEV)
    return s


# --------------------------------------------------------------------------- one pass
def run(s):
    case = s["case"]
    k = case["kind"]
    if k == "bisect":
        return pk.bisect(s["band"], s["idx"], rtol=1e-12, fanout=8)
    if k == "counts":
        return pk.inertia(s["band"], s["sigma"])
    if k == "propose":
        p = slicer.propose_slices(s["band"], s["params"], nslices=case["count"], count_tol=16)
        return {"bounds": p.bounds, "counts": p.counts, "used": p.used_fallback, "evals": p.inertia_evals,
                "proposed": p.proposed_counts}
    if k == "train":
        tr = s["trainer"]
        loss = tr.step(s["x"], s["t"])
        return {"loss": loss, "params": tr.params, "m": tr.m, "v": tr.v}
    if k == "solve":
        return pk.shifted_solve(s["band"], s["shifts"], s["rhs"], trans=int(case["adjoint"]),
                                precision=pk.MIXED if case["mixed"] else pk.FP64)
    if k == "products":
        gram = pk.block_gemm(pk.GEMM_GRAM, s["q"], s["m"])
        bq = pk.band_matmul_tc(s["band"], s["q"])
        proj = pk.block_gemm(pk.GEMM_AHB, s["q"], s["m"], bq)
        x = pk.block_gemm(pk.GEMM_UPDATE, s["q"], s["m"], s["w"])
        return {"gram": gram, "bq": bq, "proj": proj, "x": x}
    if k == "cholqr":
        q, r = pk.cholqr(s["q"], s["m"], passes=case["passes"])
        return {"q": q, "r": r}
    if k == "eigh":
        pairs = pk.eigh(s["a"])
        return {"lam": [p[0] for p in pairs], "v": [p[1] for p in pairs]}
    r = pk.band_slice(s["band"], s["bounds"], s["m0"], s["x0"], workspace=s["work"], **s["opts"])
    out = {"counts": r.counts, "nfound": r.nfound, "lam": [], "v": []}
    for i in range(case["slices"]):
        lam, v = r.slice_pairs(i)
        out["lam"].append(lam)
        # at tol = 1e-10 a mixed-precision eigenvector is known to about tol ||B|| / gap: single precision
        out["v"].append(v.to(torch.complex64 if v.is_complex() else torch.float32) if case["mixed"] else v)
    return out


# --------------------------------------------------------------------------- what a pass cannot do without
def work(case):
    k = case["kind"]
    es, cm = (16, 4) if case.get("cplx") else (8, 1)
    n, b = case.get("n", 0), case.get("b", 0)
    band = n * (b + 1) * es
    if k == "bisect":  # 40 bits of every eigenvalue, one more per count
        return {"bytes": band + 24 * case["count"], "flops": 40.0 * case["count"] * cm * n * b * b}
    if k == "counts":
        return {"bytes": band + 16 * case["count"], "flops": 1.0 * case["count"] * cm * n * b * b}
    if k == "propose":
        return {"bytes": band, "flops": 1.0 * (case["count"] - 1) * cm * n * b * b + 31 * 8 * cm * 2 * n * (2 * b + 1)}
    if k == "train":
        np_ = 98 * 256 + 2 * 256 * 256 + 256 * 64 + 3 * 256 + 64
        return {"bytes": 4 * (6 * np_ + case["batch"] * (98 + 63)), "flops": 6.0 * np_ * case["batch"]}
    if k == "solve":
        c = case["cols"]
        return {"bytes": band + 16 * n * c * (1 + case["shifts"]),
                "flops": case["shifts"] * (16.0 * n * b * b + 24.0 * n * b * c)}
    if k == "products":
        m = _sizes(case["blocks"], case["cols"])
        tall, sq = sum(m) * n * es, sum(x * x for x in m)
        return {"bytes": band + 4 * tall + 3 * sq * es,
                "flops": cm * 2.0 * n * (2.5 * sq + (2 * b + 1) * sum(m))}
    if k == "cholqr":
        m = _sizes(case["blocks"], case["cols"])
        sq = sum(x * x for x in m)
        return {"bytes": (2 * sum(m) * n + sq) * es,
                "flops": case["passes"] * cm * (2.0 * n * sq + sum(x ** 3 for x in m) * 2.0 / 3)}
    if k == "eigh":
        m = _sizes(case["blocks"], case["cols"])
        return {"bytes": (2 * sum(x * x for x in m) + sum(m)) * es, "flops": cm * 9.0 * sum(x ** 3 for x in m)}
    M = case["slices"] * max(1.3 * case["per"], case["per"] + 10)
    m1 = M / case["slices"]
    both = 2 if case["cplx"] else 1
    # two passes over 8 nodes per slice, each with its Rayleigh-Ritz products; one factorization per node
    return {"bytes": band + 2 * M * n * es,
            "flops": 8 * case["slices"] * 16.0 * n * b * b
            + 2 * (8 * both * 24.0 * n * b * M + cm * 2.0 * n * M * (2.5 * m1 + 2 * (2 * b + 1)))}


# --------------------------------------------------------------------------- the same in 64 bits
def _dense(band):
    n, w = band.shape
    a = torch.zeros((n, n), dtype=band.dtype, device=band.device)
    for d in range(w):
        v = band[:n - d, d]
        if d == 0:
            a.diagonal().copy_(v.real if v.is_complex() else v)
        else:
            a.diagonal(-d).copy_(v)
            a.diagonal(d).copy_(v.conj())
    return a


def _band_times(band, x):
    """B x for the rows of x (ncols, n)."""
    n, w = band.shape
    d0 = band[:, 0].real if band.is_complex() else band[:, 0]
    y = x * d0
    for d in range(1, w):
        v = band[:n - d, d]
        y[:, d:] += x[:, :n - d] * v
        y[:, :n - d] += x[:, d:] * v.conj()
    return y


def _solve(band, shifts, rhs, adjoint):
    """(z I - B)^{-1} y by block elimination on blocks of the semi-bandwidth."""
    n, w = band.shape
    b = max(w - 1, 1)
    nb = -(-n // b)
    pad = nb * b - n
    z = torch.as_tensor(shifts, device=band.device)
    z = z.conj() if adjoint else z  # (z I - B)^H = conj(z) I - B
    S = z.numel()
    i = torch.arange(b, device=band.device)

    def block(r, c):  # B[rows of block r, columns of block c], r - c in (0, 1)
        rows, cols = r * b + i[:, None], c * b + i[None, :]
        d = rows - cols
        ok = (d >= 0) & (d < w) & (rows < n) & (cols < n)
        v = band[cols.clamp(max=n - 1), d.clamp(0, w - 1)].to(torch.complex128)
        return torch.where(ok, v, torch.zeros((), dtype=v.dtype, device=v.device))

    y = torch.nn.functional.pad(rhs, (0, pad)).T.reshape(nb, b, -1)
    eye = torch.eye(b, dtype=torch.complex128, device=band.device)
    ups, xs = [], []
    for k in range(nb):
        lo = block(k, k)
        diag = torch.tril(lo, -1)
        diag = diag + diag.conj().T + torch.diag(lo.diagonal().real.to(torch.complex128))
        m = z[:, None, None] * eye - diag
        r = y[k].expand(S, -1, -1)
        if k:
            sub = -block(k, k - 1)
            m = m - sub @ ups[-1]
            r = r - sub @ xs[-1]
        up = -block(k + 1, k).conj().T.expand(S, -1, -1) if k + 1 < nb else None
        sol = torch.linalg.solve(m, torch.cat([up, r], 2) if up is not None else r)
        ups.append(sol[:, :, :b] if up is not None else None)
        xs.append(sol[:, :, b:] if up is not None else sol)
    for k in range(nb - 2, -1, -1):
        xs[k] = xs[k] - ups[k] @ xs[k + 1]
    return torch.cat(xs, 1)[:, :n].transpose(1, 2).contiguous()


def _phase(v):
    """Columns scaled so that their first largest component is real and positive."""
    k = v.abs().argmax(0)
    p = v.gather(0, k[None, :])
    return v * (p.abs() / p).conj() if not v.is_complex() else v * (p.conj() / p.abs())


def _network(params, x):
    h = x
    for l, (wo, bo, fo, fi) in enumerate(slicer_layers()):
        h = h @ params[wo: wo + fo * fi].reshape(fo, fi).T + params[bo: bo + fo]
        if l < 3:
            h = torch.relu(h)
    return torch.cumsum(torch.softmax(h, 1), 1)[:, :-1]


def slicer_layers():
    """(weight offset, bias offset, out, in) of the network 98 -> 256 -> 256 -> 256 -> 64."""
    off, out = 0, []
    for fi, fo in ((98, 256), (256, 256), (256, 256), (256, 64)):
        out.append((off, off + fo * fi, fo, fi))
        off += fo * fi + fo
    return out


def exact(case, seed):
    k = case["kind"]
    if k in ("counts", "propose"):  # whole numbers, and bounds that only have to hold them
        return None
    if k == "slice" and case["n"] > 4096:
        return None
    s = prepare(case, seed)
    if k == "bisect":
        lam = torch.linalg.eigvalsh(_dense(s["band"]))[torch.as_tensor(s["idx"], device=DEV)]
        return lam, lam
    if k == "train":
        tr = s["trainer"]
        p = tr.params.double().requires_grad_(True)
        loss = ((_network(p, s["x"].double()) - s["t"].double()) ** 2).mean()
        g, = torch.autograd.grad(loss, p)
        t = tr.t + 1
        m = 0.9 * tr.m.double() + 0.1 * g
        v = 0.999 * tr.v.double() + 0.001 * g * g
        p = p.detach() - 1e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
        return {"loss": loss.detach().reshape(1), "params": p, "m": m, "v": v}
    if k == "solve":
        return _solve(s["band"], s["shifts"], s["rhs"], case["adjoint"])
    if k in ("products", "cholqr"):
        off = [0]
        for m in s["m"]:
            off.append(off[-1] + m)
        cols = [s["q"][off[t]: off[t + 1]].T for t in range(len(s["m"]))]
        if k == "products":
            bq = _band_times(s["band"], s["q"])
            gram = [c.conj().T @ c for c in cols]
            proj = [c.conj().T @ bq[off[t]: off[t + 1]].T for t, c in enumerate(cols)]
            x = torch.cat([(c @ w).T for c, w in zip(cols, s["w"])])
            return {"gram": gram, "bq": bq, "proj": proj, "x": x}
        qs, rs = [], []
        for c in cols:
            q, r = torch.linalg.qr(c)
            d = r.diagonal()
            ph = d / d.abs()
            qs.append((q * ph).T)
            rs.append(ph.conj()[:, None] * r)
        # with two passes the last factor is that of an orthonormal basis
        if case["passes"] > 1:
            rs = [torch.eye(r.shape[0], dtype=r.dtype, device=r.device) for r in rs]
        return {"q": torch.cat(qs), "r": rs}
    if k == "eigh":
        pairs = [torch.linalg.eigh(a) for a in s["a"]]
        return {"lam": [p[0] for p in pairs], "v": [_phase(p[1]) for p in pairs]}
    lam = torch.linalg.eigvalsh(_dense(s["band"]))
    bounds = torch.as_tensor(s["bounds"], device=DEV)
    inside = [lam[(lam >= bounds[i]) & (lam < bounds[i + 1])] for i in range(case["slices"])]
    n = [v.numel() for v in inside]
    return {"counts": torch.tensor(n, dtype=torch.int32), "nfound": torch.tensor(n, dtype=torch.int32), "lam": inside,
            "v": [None] * case["slices"]}
