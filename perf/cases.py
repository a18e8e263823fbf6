"""The work this library is measured on: its calls at the sizes they are used at.

A case names one public call and its sizes; `prepare` renders the clip and
whatever a program holds before that call (measurement matrix, decomposition,
model, context), `run` makes the call once.  The clips are the kind the method
is for: a fixed camera, a textured static scene, a few moving objects, an
illumination ramp and sensor noise, as 8-bit frames.
"""
import math

import numpy as np
import torch

from paper_1512_04205_gb300 import cdmd as C
from paper_1512_04205_gb300 import selector as S

DEV = "cuda"


def listed():
    return [
        # One camera in HD, five 200-frame windows under one sensing matrix, learned selection: the
        # throughput setting of a server that segments a long video window by window.
        dict(name="run_shared_1080p", op="run_shared", W=1920, H=1080, n=200, clips=5, k=1000, r=20, K=10,
             prec="bf16x2", selector="mlp"),
        # The smallest clip in use (a thumbnail stream), whole call, the library's default precision:
        # launches and the small solves are all there is.
        dict(name="run_160x120", op="run", W=160, H=120, n=100, k=200, r=10, K=10, prec="fp32", selector="omp"),
        # The sketch of a single HD clip with a dense Gaussian matrix on the tensor cores.
        dict(name="sketch_gauss_1080p", op="sketch", W=1920, H=1080, n=200, k=1000, ctype="gaussian", prec="bf16x2"),
        # The same with the +1 / -1 matrix at 720p (the frame size the method was published for).
        dict(name="sketch_rad_720p", op="sketch", W=1280, H=720, n=200, k=1000, ctype="rademacher", prec="bf16x2"),
        # The default-precision sketch at 720x480, a mid-sized number of measurements.
        dict(name="sketch_fp32_480p", op="sketch", W=720, H=480, n=200, k=400, ctype="gaussian", prec="fp32"),
        # A long 4K clip with the sparse matrix (one entry in a thousand): the gather form.
        dict(name="gather_sparse_4k", op="gather", W=3840, H=2160, n=300, k=1000, density=1e-3),
        # The small solves of the HD window, and of the long 4K clip with its compressed modes.
        dict(name="decompose_n200", op="decompose", n=200, k=1000, r=20, K=10, selector="omp", phiy=False),
        dict(name="decompose_n300", op="decompose", n=300, k=1000, r=30, K=10, selector="omp", phiy=True),
        # The modes of the HD clip lifted back to pixels, ten of them.
        dict(name="lift_1080p", op="lift", W=1920, H=1080, n=200, r=20, K=10, prec="bf16x2"),
        # Background and threshold of the HD clip, the mask alone.
        dict(name="subtract_1080p", op="subtract", W=1920, H=1080, n=200, r=20, K=10, mode="modulus", bg=False),
        # Background and threshold at 720p where the program also keeps the background video.
        dict(name="subtract_bg_720p", op="subtract", W=1280, H=720, n=200, r=20, K=10, mode="modulus", bg=True),
        # The median post-pass on the masks of the HD clip.
        dict(name="median_1080p", op="median", W=1920, H=1080, n=200),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _size(rng, lo, hi):
    """A frame of lo..hi pixels (log-uniform), sides of any parity, between 1:1 and 2:1."""
    px = _log(rng, lo, hi)
    W = int(math.sqrt(px * rng.uniform(1.0, 2.0)))
    return dict(W=W, H=max(1, int(px / W)))


def draw(rng):
    op = rng.choice(["run", "run_shared", "sketch", "sketch", "gather", "decompose", "decompose", "lift", "subtract",
                     "subtract", "median"])
    n = int(_log(rng, 40, 300))
    r = rng.randint(6, max(6, min(20, n // 5)))
    K = rng.randint(3, min(r, 12))
    k = int(_log(rng, 100, 1000))
    if op == "run":
        prec = rng.choice(["fp32", "bf16x2"])
        return dict(op=op, **_size(rng, 160 * 120, 640 * 480), n=n, k=k, r=r, K=K, prec=prec,
                    selector=rng.choice(["omp", "mlp"]))
    if op == "run_shared":
        n = min(n, 200)
        return dict(op=op, **_size(rng, 320 * 240, 1280 * 720), n=n, clips=rng.randint(2, 5), k=k, r=r, K=K,
                    prec="bf16x2", selector=rng.choice(["omp", "mlp"]))
    if op == "sketch":
        prec = rng.choice(["fp32", "bf16x2", "bf16x2"])
        return dict(op=op, **_size(rng, 160 * 120, 640 * 480 if prec == "fp32" else 1920 * 1080), n=n, k=k,
                    ctype=rng.choice(["gaussian", "rademacher"]), prec=prec)
    if op == "gather":
        return dict(op=op, **_size(rng, 320 * 240, 1920 * 1080), n=n, k=k, density=_log(rng, 1e-4, 1e-3))
    if op == "decompose":
        n = int(_log(rng, 40, 512))
        r = rng.randint(6, max(6, min(32, n // 6)))
        return dict(op=op, n=n, k=k, r=r, K=rng.randint(3, min(r, 12)),
                    selector=rng.choice(["omp", "omp", "lstsq"]), phiy=rng.random() < 0.3)
    if op == "lift":
        return dict(op=op, **_size(rng, 320 * 240, 1920 * 1080), n=n, r=r, K=K, prec=rng.choice(["bf16x2", "bf16x2", "fp32"]))
    if op == "subtract":
        return dict(op=op, **_size(rng, 320 * 240, 1920 * 1080), n=n, r=r, K=K, mode=rng.choice(["modulus", "modulus", "real"]),
                    bg=rng.random() < 0.3)
    return dict(op="median", **_size(rng, 160 * 120, 1920 * 1080), n=n)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------


def _scene(W, H, n, seed):
    """A clip (n, W*H) uint8 on the GPU, row stride a multiple of 16 bytes as a decoder's frames have."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    m = W * H
    ldd = -(-m // 16) * 16
    D = torch.zeros((n, ldd), dtype=torch.uint8, device=DEV)
    y = torch.arange(H, dtype=torch.float32, device=DEV)[:, None]
    x = torch.arange(W, dtype=torch.float32, device=DEV)[None, :]
    scene = torch.full((H, W), 128.0, device=DEV)
    for _ in range(6):
        amp, per = rng.uniform(5.0, 25.0), rng.uniform(8.0, max(9.0, W / 2.0))
        th, ph = rng.uniform(0.0, math.pi), rng.uniform(0.0, 2.0 * math.pi)
        scene += amp * torch.sin((x * math.cos(th) + y * math.sin(th)) * (2.0 * math.pi / per) + ph)
    objs = []
    for _ in range(3):
        w, h = rng.uniform(W / 20.0, W / 6.0), min(rng.uniform(W / 20.0, W / 6.0), H - 2.0)
        grey = rng.choice([rng.uniform(0.0, 88.0), rng.uniform(168.0, 255.0)])
        v, a = rng.uniform(0.5, 3.0), rng.uniform(0.0, 2.0 * math.pi)
        objs.append([rng.uniform(0, W - w), rng.uniform(0, H - h), w, h, grey, v * math.cos(a), v * math.sin(a)])
    for t in range(n):
        f = scene.clone()
        for o in objs:
            x0, y0, w, h, grey, vx, vy = o
            f[max(0, int(y0)):max(0, int(y0 + h)), max(0, int(x0)):max(0, int(x0 + w))] = grey
            if not 0 <= x0 + vx <= W - w:
                o[5] = vx = -vx
            if not 0 <= y0 + vy <= H - h:
                o[6] = vy = -vy
            o[0], o[1] = x0 + vx, y0 + vy
        f *= 1.0 + 0.1 * (2.0 * t / (n - 1) - 1.0)
        f += 3.0 * torch.randn((H, W), generator=gen, device=DEV)
        D[t, :m] = (f + 0.5).floor_().clamp_(0, 255).to(torch.uint8).view(-1)
    return D[:, :m]


def _sketch_of(case, seed):
    """A k-measurement sketch (n, k) of a thumbnail clip, in 64 bits."""
    D = _scene(160, 120, case["n"], seed).double()
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) + 77)
    A = torch.randn((D.shape[1], case["k"]), generator=gen, device=DEV, dtype=torch.float64)
    return (D @ A).contiguous()


def _modes_of(D, r, K):
    """What a decomposition hands to the lift and the subtraction (G, lambda, beta, the K selected modes), from every
    s-th pixel of the clip."""
    Y = D[:, ::max(1, D.shape[1] // 20000)].double().cpu().numpy().T
    return _decompose(Y, r, K, "omp")


def _blob():
    return torch.from_numpy(np.array(S.load_model()[0], dtype=np.float32)).to(DEV)


def prepare(case, seed):
    op = case["op"]
    ctx = C.Context(0)
    st = dict(case=case, ctx=ctx, cseed=1000003 * (int(seed) + 1))
    if op in ("run", "run_shared"):
        st["D"] = [_scene(case["W"], case["H"], case["n"], 16 * int(seed) + i) for i in range(case.get("clips", 1))]
        st["params"] = C.make_params(case["k"], case["r"], case["K"], 25.0, seed=st["cseed"], prec=case["prec"],
                                     selector=case["selector"])
        if case["selector"] == "mlp":
            C.cdmd_selector_load(ctx, _blob())
    elif op == "sketch":
        st["D"] = _scene(case["W"], case["H"], case["n"], seed)
    elif op == "gather":
        st["D"] = _scene(case["W"], case["H"], case["n"], seed)
        st["meas"] = C.Measure(ctx, "sparse", case["W"] * case["H"], case["k"], st["cseed"], density=case["density"])
    elif op == "decompose":
        st["DY"] = _sketch_of(case, seed)
    elif op in ("lift", "subtract"):
        D = st["D"] = _scene(case["W"], case["H"], case["n"], seed)
        d = _modes_of(D, case["r"], case["K"])
        st.update({q: torch.from_numpy(np.ascontiguousarray(d[q])).to(DEV) for q in ("G", "lam", "beta", "sel")})
        if op == "subtract":
            st["Phi"] = _lift(D, st["G"], st["sel"]).float()
    elif op == "median":
        # a subtraction's mask: objects with ragged edges, and single false pixels
        W, H, n = case["W"], case["H"], case["n"]
        D = _scene(W, H, n, seed)
        fg = (D.int() - D.float().mean(0).int()).abs() > 25
        gen = torch.Generator(device=DEV)
        gen.manual_seed(int(seed))
        st["mask"] = torch.empty((n, -(-W * H // 32)), dtype=torch.int32, device=DEV)
        bits = torch.zeros((32 * st["mask"].shape[1],), dtype=torch.int64, device=DEV)
        two = 2 ** torch.arange(32, device=DEV)
        for t in range(n):
            bits[:W * H] = fg[t] ^ (torch.rand(W * H, generator=gen, device=DEV) < 0.02)
            st["mask"][t] = (bits.view(-1, 32) * two).sum(1).to(torch.int32)
    return st


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------


def run(st):
    case, ctx, op = st["case"], st["ctx"], st["case"]["op"]
    if op == "run":
        mask = C.cdmd_run(ctx, st["D"][0], st["params"])
        return dict(mask=[mask], modes=_modes(st))
    if op == "run_shared":
        masks = C.cdmd_run_shared(ctx, st["D"], st["params"])
        return dict(mask=masks, modes=_modes(st))
    if op == "sketch":
        return C.cdmd_sketch(ctx, st["D"], case["k"], st["cseed"], ctype=case["ctype"], prec=case["prec"])
    if op == "gather":
        return C.cdmd_sketch_gather(ctx, st["D"], st["meas"])
    if op == "decompose":
        out = C.cdmd_decompose(ctx, st["DY"], case["r"], case["K"], selector=case["selector"], with_phiy=case["phiy"])
        return {q: v for q, v in out.items() if v is not None}
    if op == "lift":
        return C.cdmd_lift(ctx, st["D"], st["G"], cols=st["sel"], ncols=case["K"], prec=case["prec"])
    if op == "subtract":
        out = C.cdmd_subtract(ctx, st["D"], st["Phi"], st["beta"], st["lam"], 25.0, cols=st["sel"], mode=case["mode"],
                              want_bg=case["bg"])
        return dict(mask=out[0], bg=out[1]) if case["bg"] else dict(mask=out)
    return C.cdmd_median3x3(ctx, st["mask"], case["W"], case["H"])


def _modes(st):
    """The modes behind the masks, which a program keeps beside them (of the last clip)."""
    c = st["case"]
    return C.workspace_tensors(st["ctx"], c["W"] * c["H"], c["n"], c["k"], c["r"], c["K"])


def work(case):
    op, n, m = case["op"], case["n"], case.get("W", 0) * case.get("H", 0)
    k, r, K, p = case.get("k", 0), case.get("r", 0), case.get("K", 0), case["n"] - 1
    words = -(-m // 32) * 4 * n
    small = k * n * n + 4 / 3 * p ** 3 + 4 * p * p * r + 25 * r ** 3 + 16 * p * r * r + 4 * p * p * r
    if op in ("run", "run_shared"):
        c = case.get("clips", 1)
        return dict(bytes=c * (m * n + words) + 8 * K * m + 8 * k * n,
                    flops=c * (2 * k * m * n + small + 4 * m * p * K + 8 * m * n * K))
    if op == "sketch":
        return dict(bytes=m * n + 8 * k * n, flops=2 * k * m * n)
    if op == "gather":
        nnz = case["density"] * m * k
        return dict(bytes=m * n + 4 * nnz + 8 * m + 8 * k * n, flops=nnz * n)
    if op == "decompose":
        return dict(bytes=8 * k * n + 16 * p * r + (16 * k * r if case["phiy"] else 0), flops=small)
    if op == "lift":
        return dict(bytes=m * p + 16 * p * r + 8 * K * m, flops=4 * m * p * K)
    if op == "subtract":
        return dict(bytes=m * n + 8 * K * m + words + (4 * m * n if case["bg"] else 0), flops=8 * m * n * K)
    return dict(bytes=2 * words, flops=0)


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------


def _philox(c0, c1, c2, seed):
    """Philox4x32-10 words (int64 tensors holding 32 bits) of counters (c0, c1, c2, 0)."""
    M = 0xFFFFFFFF
    k0, k1 = seed & M, (seed >> 32) & M
    c = [c0, c1, torch.full_like(c0 + c1, c2), torch.zeros_like(c0 + c1)]
    for _ in range(10):
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((b >> 32) & M) ^ c[1] ^ k0, b & M, ((a >> 32) & M) ^ c[3] ^ k1, a & M]
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return c


def _matrix(ctype, j0, j1, k, seed, density=0.0):
    """Columns j0..j1-1 of the measurement matrix, as (j1-j0, k) in 64 bits."""
    j = torch.arange(j0, j1, dtype=torch.int64, device=DEV)[:, None]
    if ctype == "rademacher":
        q = torch.arange(-(-k // 128), dtype=torch.int64, device=DEV)[None, :]
        w = torch.stack(_philox(j, q, 1, seed), 2)[..., None] >> torch.arange(32, device=DEV)
        return (1.0 - 2.0 * (w & 1).double()).reshape(j1 - j0, -1)[:, :k]
    q = torch.arange(-(-k // 4), dtype=torch.int64, device=DEV)[None, :]
    w = _philox(j, q, 2 if ctype == "sparse" else 0, seed)
    if ctype == "sparse":
        w = torch.stack(w, 2)
        v = torch.where(w < int(math.floor(2.0 ** 32 * density)), 1.0 - 2.0 * (w & 1).double(), 0.0)
    else:
        u = [(x.double() + 0.5) * 2.0 ** -32 for x in w]
        rad = [torch.sqrt(-2.0 * torch.log(u[i])) for i in (0, 2)]
        v = torch.stack([rad[0] * torch.cos(2 * math.pi * u[1]), rad[0] * torch.sin(2 * math.pi * u[1]),
                         rad[1] * torch.cos(2 * math.pi * u[3]), rad[1] * torch.sin(2 * math.pi * u[3])], 2)
    return v.reshape(j1 - j0, -1)[:, :k]


def _exact_sketch(D, ctype, k, seed, density=0.0):
    n, m = D.shape
    out = torch.zeros((n, k), dtype=torch.float64, device=DEV)
    step = max(1, (1 << 25) // k)
    for j in range(0, m, step):
        e = min(m, j + step)
        out += D[:, j:e].double() @ _matrix(ctype, j, e, k, seed, density)
    return out


def _lift(D, G, cols):
    """X' G[:, cols] as (m, K, 2) in 64 bits."""
    m = D.shape[1]
    g = G[cols.long()].permute(1, 0, 2).reshape(D.shape[0] - 1, -1)
    out = torch.empty((m, g.shape[1]), dtype=torch.float64, device=DEV)
    for j in range(0, m, 1 << 18):
        out[j:j + (1 << 18)] = D[1:, j:j + (1 << 18)].double().T @ g
    return out.view(m, -1, 2)


def _tridiagonal_basis(A):
    """Q of A = Q T Q^T by Householder reflections that send each column to -sign(x_1) ||x|| e_1."""
    p = A.shape[0]
    A, Q = A.copy(), np.eye(p)
    for j in range(p - 2):
        x = A[j + 1:, j].copy()
        if np.dot(x[1:], x[1:]) <= 1e-280:
            continue
        x[0] += math.copysign(np.linalg.norm(x), x[0])
        x /= np.linalg.norm(x)
        A[j + 1:] -= 2 * np.outer(x, x @ A[j + 1:])
        A[:, j + 1:] -= 2 * np.outer(A[:, j + 1:] @ x, x)
        Q[:, j + 1:] -= 2 * np.outer(Q[:, j + 1:] @ x, x)
    return Q


def _signs(V, Q):
    """The free sign of each singular vector, taken as the library takes it: its coordinates in the basis that makes
    Y^T Y tridiagonal have a positive product with a fixed positive vector."""
    p, r = V.shape
    M = 0xFFFFFFFF
    i = np.arange(1, p + 1, dtype=np.uint64)[:, None]
    w = np.arange(1, r + 1, dtype=np.uint64)[None, :]
    h = ((i * 0x9E3779B9) & M) ^ ((w * 0x85EBCA6B) & M)
    h ^= h >> np.uint64(15)
    h = (h * 0x2C1B3C6D) & M
    h ^= h >> np.uint64(12)
    b = 1.0 + (h & np.uint64(0xFFFF)).astype(np.float64) / 65536.0
    return np.where(np.sum((Q.T @ V) * b, 0) < 0, -1.0, 1.0)


def _decompose(DY, r, K, selector):
    """Compressed DMD of the sketch DY (k x n): rank-r SVD, eigenvalues, G = V S^-1 W, amplitudes of the selected modes."""
    Y, Y1 = DY[:, :-1], DY[:, 1:]
    if Y.shape[0] > 2 * Y.shape[1]:   # the same singular values and V from the triangular factor
        q, t = np.linalg.qr(Y)
        U, s, Vh = np.linalg.svd(t, full_matrices=False)
        U = q @ U[:, :r]
    else:
        U, s, Vh = np.linalg.svd(Y, full_matrices=False)
    U, s, V = U[:, :r], s[:r], Vh[:r].T
    sg = _signs(V, _tridiagonal_basis(Y.T @ Y))
    U, V = U * sg, V * sg
    lam, W = np.linalg.eig((U.T @ Y1 @ V) / s)
    lam, W = lam.astype(complex), W.astype(complex)
    heads = [i for i in range(r) if lam[i].imag >= 0]      # a pair goes where its first member goes
    order = []
    for i in sorted(heads, key=lambda i: (-abs(lam[i]), -lam[i].imag)):
        order.append(i)
        if lam[i].imag > 0:
            order.append(int(np.argmin(np.abs(lam - np.conj(lam[i])))))
    lam, W = lam[order], W[:, order] / np.linalg.norm(W[:, order], axis=0)
    top = W[np.argmax(np.abs(W), 0), np.arange(r)]
    W = W * (np.abs(top) / top)
    G = (V / s) @ W
    P = Y1 @ G
    y = DY[:, 0].astype(complex)
    norm = np.linalg.norm(P, axis=0)
    sel, amp, res = (list(range(r)), None, y) if selector == "lstsq" else ([], None, y)
    while len(sel) < (r if selector == "lstsq" else K):
        score = np.abs(P.conj().T @ res) / norm
        score[sel] = -1.0
        best = [i for i in range(r) if score[i] >= score.max() * (1.0 - 1e-9)]
        sel.append(max(best, key=lambda i: (lam[i].imag, -i)))
        amp = np.linalg.lstsq(P[:, sel], y, rcond=None)[0]
        res = y - P[:, sel] @ amp
    if amp is None:
        amp = np.linalg.lstsq(P, y, rcond=None)[0]
    beta = np.zeros(r, complex)
    beta[sel] = amp
    two = lambda z: np.stack([z.real, z.imag], -1)  # noqa: E731
    return dict(sigma=s, lam=two(lam), G=two(G.T), PhiY=two(P.T), beta=two(beta), sel=np.array(sel[:K], np.int32))


def exact(case, seed):
    op = case["op"]
    if op in ("run_shared", "median"):
        return None   # the mask decides nothing in 64 bits; the passes behind it are cases of their own
    st = prepare(case, seed)
    if op == "run":
        if case["selector"] == "mlp":
            return None
        D = st["D"][0]
        DY = _exact_sketch(D, "gaussian", case["k"], st["cseed"])
        d = _decompose(DY.cpu().numpy().T, case["r"], case["K"], "omp")
        G, sel = torch.from_numpy(d["G"]).to(DEV), torch.from_numpy(d["sel"]).to(DEV)
        return dict(mask=[None], modes=dict(DY=DY, sigma=d["sigma"], lam=d["lam"], G=d["G"], beta=d["beta"], sel=None,
                                            nsel=None, Phi=_lift(D, G, sel)))
    if op == "sketch":
        return _exact_sketch(st["D"], case["ctype"], case["k"], st["cseed"])
    if op == "gather":
        return _exact_sketch(st["D"], "sparse", case["k"], st["cseed"], case["density"])
    if op == "decompose":
        d = _decompose(st["DY"].cpu().numpy().T, case["r"], case["K"], case["selector"])
        out = dict(sigma=d["sigma"], lam=d["lam"], G=d["G"], beta=d["beta"], sel=None, nsel=None)
        return dict(out, PhiY=d["PhiY"]) if case["phiy"] else out
    if op == "lift":
        return _lift(st["D"], st["G"], st["sel"])
    if not case["bg"]:
        return None
    n, m = st["D"].shape
    cols = st["sel"].long()
    lam, beta = (torch.view_as_complex(st[q])[cols] for q in ("lam", "beta"))
    t = torch.arange(n, device=DEV, dtype=torch.float64)[:, None]
    T = lam[None, :] ** t * beta[None, :]
    bg = torch.empty((n, m), dtype=torch.float64, device=DEV)
    for j in range(0, m, 1 << 17):
        z = T @ torch.view_as_complex(st["Phi"][j:j + (1 << 17)].double()).T
        bg[:, j:j + (1 << 17)] = z.abs() if case["mode"] == "modulus" else z.real
    return dict(mask=None, bg=bg)
