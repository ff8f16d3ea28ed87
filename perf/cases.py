"""Performance cases: the calls a user of the PCA library makes, over the sizes they are made at.

Every case is one call of a public entry point on inputs of the kind it meets:
noisy linear mixtures, smooth scene-like mixtures, cubes with a planted
spectrum.  `listed` holds the fixed cases, `draw` gives more of the same ranges.

A case is a dict of
  op      fit | cov | eigh | project | backward | batch | host
  N, B, k pixels, bands, components (batch: tiles, n_lo, n_hi instead of N and B)
  dtype   f32 | bf16 | f16 (the cube's element type)
  prec    mix | p32 | p64
  data    mixture | scene | planted
  layout  bip | bsq (fit only)
  plain   fit only: the call as a newcomer writes it (outputs and workspace made by
          the call, which waits for the result); otherwise outputs and workspace are
          kept by the caller and the call only enqueues work
"""
import math

import numpy as np
import torch

import paper_2403_18321_gb300 as gbpca

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
TILE_BANDS = (64, 96, 128, 160, 200, 224, 256)


def _fit(name, N, B, k, prec="mix", dtype="f32", data="mixture", layout="bip", plain=False):
    return {"name": name, "op": "fit", "N": N, "B": B, "k": k, "prec": prec, "dtype": dtype,
            "data": data, "layout": layout, "plain": plain}


def listed():
    return [
        # the smallest image of the paper's tables, first component only: launches and latency
        _fit("fit_100x100x50", 100 * 100, 50, 1, plain=True),
        # the plain PCA configuration: a small mixed image, five components, default call
        _fit("fit_100x100x128", 100 * 100, 128, 5, plain=True),
        # a band-sequential image (the paper's GPU layout) in plain FP32
        _fit("fit_bsq_300x300x100_p32", 300 * 300, 100, 1, prec="p32", layout="bsq"),
        # an ordinary scene of one sensor pass, ten components
        _fit("fit_scene_512x217x224", 512 * 217, 224, 10, data="scene"),
        # the large 16-bit cube, twenty components
        _fit("fit_planted_2048x2048x224_bf16", 2048 * 2048, 224, 20, dtype="bf16", data="planted"),
        # a full-precision fit, as reference results are made
        _fit("fit_350x350x188_p64", 350 * 350, 188, 1, prec="p64", data="scene"),
        # covariance stage alone (a sharded fit's local step), odd band count, plain FP32
        {"name": "cov_610x340x103_p32", "op": "cov", "N": 610 * 340, "B": 103, "k": 1,
         "prec": "p32", "dtype": "f32", "data": "scene"},
        # eigen-decomposition of a pooled covariance, the most bands the library takes
        {"name": "eigh_256", "op": "eigh", "N": 1, "B": 256, "k": 1, "prec": "mix", "dtype": "f32",
         "data": "planted"},
        # projecting new pixels onto components fitted before
        {"name": "project_1024x1024x200_f16", "op": "project", "N": 1024 * 1024, "B": 200, "k": 16,
         "prec": "p32", "dtype": "f16", "data": "planted"},
        # the layer's backward pass in a training step
        {"name": "backward_512x512x200", "op": "backward", "N": 512 * 512, "B": 200, "k": 10,
         "prec": "p64", "dtype": "f32", "data": "planted"},
        # the tiles of a large mosaic in one planned run
        {"name": "batch_256_tiles", "op": "batch", "tiles": 256, "n_lo": 4096, "n_hi": 262144,
         "k": 8, "prec": "mix", "dtype": "f32", "data": "mixture"},
        # an image that starts and ends in host memory, copies included
        {"name": "host_512x614x224", "op": "host", "N": 512 * 614, "B": 224, "k": 1, "prec": "mix",
         "dtype": "f32", "data": "scene"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a call, a size (even and odd), an element type and an option of the ranges above."""
    op = rng.choice(("fit", "fit", "fit", "cov", "eigh", "project", "backward", "batch", "host"))
    if op == "batch":
        return {"op": "batch", "tiles": rng.randint(8, 96), "n_lo": 4096, "n_hi": _log_int(rng, 8192, 131072),
                "k": rng.randint(1, 8), "prec": rng.choice(("mix", "mix", "p32")), "dtype": "f32",
                "data": "mixture"}
    B = rng.randint(32, 256)
    if op == "eigh":
        return {"op": "eigh", "N": 1, "B": B, "k": 1, "prec": rng.choice(("mix", "p32", "p64")),
                "dtype": "f32", "data": "planted"}
    data = rng.choice(("mixture", "scene", "planted"))
    prec = rng.choice(("mix", "mix", "p32", "p64"))
    # 16-bit cubes are planted spectra in [0, 1]; scenes and mixtures are FP32
    dtype = rng.choice(("f32", "bf16", "f16")) if data == "planted" else "f32"
    top = {"mix": 1000000, "p32": 400000, "p64": 100000}[prec]
    c = {"op": op, "N": _log_int(rng, 2000, top), "B": B, "k": rng.randint(1, 10), "prec": prec,
         "dtype": dtype, "data": data}
    if op == "fit":
        c["layout"] = rng.choice(("bip", "bip", "bip", "bsq"))
        c["plain"] = rng.random() < 0.3
    if op == "project":
        c["k"], c["prec"] = rng.randint(1, 40) if B > 40 else rng.randint(1, B), "p32"
    if op == "backward":
        c["data"], c["dtype"], c["prec"] = "planted", "f32", "p64"
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _smooth_spectra(rng, count, bands):
    """Smoothed random walks scaled to [0, 8000]: reflectance-like spectra."""
    walk = np.cumsum(rng.standard_normal((count, bands)), axis=1)
    half = max(1, int(3 * bands / 20))
    g = np.exp(-0.5 * (np.arange(-half, half + 1) / max(bands / 20.0, 1e-6)) ** 2)
    pad = np.pad(walk, ((0, 0), (half, half)), mode="reflect")
    out = np.stack([np.convolve(p, g / g.sum(), mode="valid") for p in pad])
    lo, hi = out.min(axis=1, keepdims=True), out.max(axis=1, keepdims=True)
    return 8000.0 * (out - lo) / np.maximum(hi - lo, 1e-12)


def _planted_basis(rng, B, comps, ratio, floor):
    W, R = np.linalg.qr(rng.standard_normal((B, B)))
    s = np.full(B, floor)
    s[:comps] = ratio ** np.arange(min(comps, B))
    return W * np.sign(np.diag(R))[None, :], s


def _cube(N, B, k, dtype, data, seed):
    rng, g = np.random.default_rng(seed), _gen(seed)
    out = torch.empty(N, B, dtype=DTYPES[dtype], device="cuda")
    step = 1 << 20
    if data == "planted":
        W, s = _planted_basis(rng, B, max(20, k) if B > 20 else B, 0.7, 1e-3)
        M = torch.from_numpy((s[:, None] * W.T).astype(np.float32)).cuda()
        for i in range(0, N, step):
            n = min(step, N - i)
            u = torch.randn(n, B, generator=g, device="cuda")
            out[i:i + n] = (u @ M).mul_(0.08).add_(0.5).clamp_(0.0, 1.0).to(out.dtype)
        return out
    e = k + 2  # two more endmembers than components kept: the kept ones stand clear of the noise
    if data == "mixture":
        M = torch.from_numpy(rng.uniform(0.0, 1.0, (e, B)).astype(np.float32)).cuda()
    else:
        M = torch.from_numpy(_smooth_spectra(rng, e, B).astype(np.float32)).cuda()
    for i in range(0, N, step):
        n = min(step, N - i)
        a = torch.empty(n, e, device="cuda").exponential_(generator=g)
        if data == "scene":  # abundances that stay alike over 64-pixel patches
            patch = torch.empty((n + 63) // 64, e, device="cuda").exponential_(generator=g)
            a = 0.1 * a + 0.9 * patch.repeat_interleave(64, 0)[:n]
        a /= a.sum(1, keepdim=True)
        clean = a @ M
        noise = torch.randn(n, B, generator=g, device="cuda")
        out[i:i + n] = clean + (noise * 0.01 if data == "mixture" else noise * clean.clamp_min(0).sqrt())
    return out


def _cov_matrix(B, seed):
    """A covariance with a decaying spectrum, every eigenvalue apart from the next."""
    rng = np.random.default_rng(seed)
    W, _ = _planted_basis(rng, B, 1, 0.7, 1.0)
    lam = np.exp(-np.linspace(0.0, 9.0, B)) * (1.0 + 0.002 * rng.random(B))
    A = (W * lam[None, :]) @ W.T
    return torch.from_numpy((A + A.T) / 2).cuda()


def _moments64(Y):
    """Band means and covariance in FP64, in pieces."""
    N, B = Y.shape
    step = 1 << 18
    mu = torch.zeros(B, dtype=torch.float64, device=Y.device)
    for i in range(0, N, step):
        mu += Y[i:i + step].double().sum(0)
    mu /= N
    C = torch.zeros(B, B, dtype=torch.float64, device=Y.device)
    for i in range(0, N, step):
        x = Y[i:i + step].double() - mu
        C += x.T @ x
    return mu, C / (N - 1)


def _eig64(C):
    """Eigenvalues descending; each vector's largest entry positive."""
    lam, V = torch.linalg.eigh(C)
    lam, V = lam.flip(0), V.flip(1).contiguous()
    top = V.abs().argmax(0)
    V = V * torch.sign(V[top, torch.arange(V.shape[1], device=V.device)])[None, :]
    return lam.contiguous(), V.contiguous()


def _project64(Y, mu, Vk):
    step = 1 << 18
    return torch.cat([(Y[i:i + step].double() - mu) @ Vk for i in range(0, Y.shape[0], step)])


def _tiles(case, seed):
    rng = np.random.default_rng(seed)
    # the sizes are the case's, the same for every seed; the values are the seed's
    fixed = np.random.default_rng(case["tiles"])
    n = np.rint(np.exp(fixed.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), case["tiles"]))).astype(int)
    b = fixed.choice(np.array(TILE_BANDS), case["tiles"])
    return [(int(n[i]), int(b[i]), int(rng.integers(1 << 30))) for i in range(case["tiles"])]


def _tile_cubes(case, seed):
    return [_cube(n, b, case["k"], case["dtype"], case["data"], s) for n, b, s in _tiles(case, seed)]


# ------------------------------------------------------------------ the interface
def prepare(case, seed):
    op, st = case["op"], {"case": case}
    if op == "batch":
        st["batch"] = gbpca.Batch(_tile_cubes(case, seed), case["k"], tol=1e-8, precision=case["prec"])
        return st
    N, B, k = case["N"], case["B"], case["k"]
    if op == "eigh":
        st["A"] = _cov_matrix(B, seed)
        return st
    Y = _cube(N, B, k, case["dtype"], case["data"], seed)
    code = {"f32": 0, "bf16": 1, "f16": 2}[case["dtype"]]
    st["Y"] = Y
    if op == "fit":
        if case["layout"] == "bsq":
            st["Y"] = Y.t().contiguous()
        if not case["plain"]:
            st["ws"] = gbpca.make_workspace(N, B, k, code, case["prec"])
            st["out"] = (torch.empty(B, dtype=torch.float64, device="cuda"),
                         torch.empty(B, dtype=torch.float64, device="cuda"),
                         torch.empty(B, B, dtype=torch.float64, device="cuda"),
                         torch.empty(N, k, dtype=torch.float32, device="cuda"))
    elif op == "cov":
        st["ws"] = gbpca.make_workspace(N, B, 1, code, case["prec"])
    elif op == "project":
        rng = np.random.default_rng(seed + 1)
        W, _ = _planted_basis(rng, B, 1, 0.7, 1.0)
        st["V"] = torch.from_numpy(np.ascontiguousarray(W)).cuda()
        st["mu"] = Y[: 1 << 16].double().mean(0)
        st["ws"] = gbpca.make_workspace(N, B, k, code, "p32")
    elif op == "backward":
        mu, C = _moments64(Y)
        lam, V = _eig64(C)
        st.update(mu=mu, lam=lam, V=V,
                  dQ=torch.randn(N, k, generator=_gen(seed + 1), device="cuda"))
    elif op == "host":
        pin = lambda *shape, dtype: torch.empty(*shape, dtype=dtype, pin_memory=True)  # noqa: E731
        st["Y"] = pin(N, B, dtype=Y.dtype)
        st["Y"].copy_(Y)
        st["buf"] = gbpca.HostFit(N, B, k, Y.dtype, case["prec"])
        st["out"] = (pin(B, dtype=torch.float64), pin(B, dtype=torch.float64),
                     pin(B, B, dtype=torch.float64), pin(N, k, dtype=torch.float32))
    return st


def run(state):
    c = state["case"]
    op = c["op"]
    if op == "fit":
        if c["plain"]:
            mu, lam, V, Q, _ = gbpca.fit(state["Y"], c["k"], precision=c["prec"], layout=c["layout"])
        else:
            mu, lam, V, Q, _ = gbpca.fit(state["Y"], c["k"], precision=c["prec"], layout=c["layout"],
                                         out=state["out"], workspace=state["ws"], sync=False)
        return {"mu": mu, "eigvals": lam, "eigvecs": V, "proj": Q}
    if op == "cov":
        mu, C, _ = gbpca.covariance(state["Y"], c["prec"], workspace=state["ws"])
        return {"mu": mu, "cov": C}
    if op == "eigh":
        lam, V, _ = gbpca.eigh(state["A"], precision=c["prec"])
        return {"eigvals": lam, "eigvecs": V}
    if op == "project":
        return {"proj": gbpca.project(state["Y"], state["mu"], state["V"], c["k"], workspace=state["ws"])}
    if op == "backward":
        return {"dcube": gbpca.backward(state["Y"], state["mu"], state["lam"], state["V"], state["dQ"],
                                        sync=False)}
    if op == "batch":
        state["batch"].run()
        r = state["batch"].results
        return {name: torch.cat([t[i].reshape(-1) for t in r])
                for i, name in enumerate(("mu", "eigvals", "eigvecs", "proj"))}
    mu, lam, V, Q, _ = gbpca.fit_host(state["Y"], c["k"], precision=c["prec"], buffers=state["buf"],
                                      out=state["out"])
    return {"mu": mu, "eigvals": lam, "eigvecs": V, "proj": Q}


def work(case):
    """Bytes: inputs read once, outputs written once.  Flops: the covariance's upper triangle, a
    Jacobi of six sweeps (6 B^3 each), the projection; the adjoint's two products."""
    def one(N, B, k, el, op):
        small = 8 * (2 * B + B * B)
        cov, eig, proj = N * B * (B + 1), 36 * B ** 3, 2 * N * B * k
        if op == "cov":
            return N * B * el + small, cov
        if op == "eigh":
            return 2 * small, eig
        if op == "project":
            return N * B * el + 8 * B * (k + 1) + 4 * N * k, proj
        if op == "backward":
            return N * B * (el + 4) + 4 * N * k + small, 2 * N * B * (B + 2 * k)
        return N * B * el + small + 4 * N * k, cov + eig + proj
    el = 4 if case["dtype"] == "f32" else 2
    if case["op"] == "batch":
        w = [one(n, b, case["k"], el, "fit") for n, b, _ in _tiles(case, 0)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    b, f = one(case["N"], case["B"], case["k"], el, case["op"])
    return {"bytes": b, "flops": f}


def exact(case, seed):
    """In FP64.  Eigenvectors of the noise floor have no value of their own (a cluster's basis is
    arbitrary), so a fit's full eigenvector matrix is left out; its projection is not."""
    op, k = case["op"], case.get("k")

    def fit64(Y):
        mu, C = _moments64(Y)
        lam, V = _eig64(C)
        return mu, lam, _project64(Y, mu, V[:, :k])

    if op == "batch":
        got = [fit64(Y) for Y in _tile_cubes(case, seed)]
        mu, lam, Q = (torch.cat([t[i].reshape(-1) for t in got]) for i in range(3))
        return {"mu": mu, "eigvals": lam, "eigvecs": None, "proj": Q}
    if op == "eigh":
        lam, V = _eig64(_cov_matrix(case["B"], seed))
        return {"eigvals": lam, "eigvecs": V}
    Y = _cube(case["N"], case["B"], k, case["dtype"], case["data"], seed)
    if op == "cov":
        mu, C = _moments64(Y)
        return {"mu": mu, "cov": C}
    if op == "project":
        st = prepare(case, seed)
        return {"proj": _project64(Y, st["mu"], st["V"][:, :k])}
    if op == "backward":
        st = prepare(case, seed)
        N = case["N"]
        mu, lam, V, dQ = st["mu"], st["lam"], st["V"], st["dQ"].double()
        X = Y.double() - mu
        gap = lam[None, :] - lam[:, None]
        F = torch.where(gap.abs() > 1e-6 * lam[0].abs(), 1.0 / gap, torch.zeros_like(gap))
        F.fill_diagonal_(0.0)
        G = torch.zeros_like(V)
        G[:, :k] = V.T @ (X.T @ dQ)
        S = V @ (F * G) @ V.T
        return {"dcube": (dQ - dQ.mean(0)) @ V[:, :k].T + (X @ (S + S.T)) / (N - 1)}
    mu, lam, Q = fit64(Y)
    return {"mu": mu, "eigvals": lam, "eigvecs": None, "proj": Q}
