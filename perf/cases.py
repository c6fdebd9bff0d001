"""Workloads of the matchgate-shadow overlap library, with their inputs, the call a user's
program makes, and the values that plain 64-bit torch gives for them.

A QC-AFQMC program holds a shadow snapshot set (an orthogonal Q_p and a measured bit string
b_p per snapshot) and, at every imaginary-time step, a fresh batch of walkers; it asks for
overlaps, gradients and force biases, now and then for local energies, and once per data set
for the shadow RDMs.  Every case here is one such call.  Inputs are synthetic, with the
distributions of the package's own workloads: Q Haar-random in O(2n) or a random signed
permutation, bits uniform or consistent with the parity of Q, walkers orthonormalised complex
Gaussians times a complex scale, Cholesky vectors symmetric real Gaussians.
"""
import math

import torch

from paper_2506_22408_gb300 import qcs

DEV = "cuda:0"

# One step of five molecules with different active spaces (n, ne, walkers, snapshots).
FIVE_SPACES = "8,4,1024,2000;12,6,512,5000;16,8,256,10000;20,10,128,20000;24,12,64,40000"


def listed():
    return [
        # The smallest useful call: a (4e, 4o)-sized active space, one small walker batch
        # against a few hundred snapshots.  Launches and latency count.
        dict(name="overlap_n8_small", kind="overlap", n=8, ne=4, W=16, P=256, ensemble="haar", bits="uniform",
             per_pair=False, precision="fp64"),
        # The paper-shaped step: an (8e, 8o) space, every walker of a node against the
        # snapshots of one shard.
        dict(name="overlap_n16_paper", kind="overlap", n=16, ne=8, W=1024, P=20000, ensemble="haar",
             bits="uniform", per_pair=False, precision="fp64"),
        # The paper's measurement ensemble: signed-permutation matchgates, only outcomes of
        # the right parity; ragged counts.
        dict(name="overlap_n16_signed_perm", kind="overlap", n=16, ne=8, W=321, P=6007, ensemble="signed_perm",
             bits="parity", per_pair=False, precision="fp64"),
        # Statistics over the shadows (variances, medians of means) read every pair's
        # estimate; a space below 16 modes and odd counts.
        dict(name="overlap_n12_per_pair", kind="overlap", n=12, ne=6, W=201, P=3001, ensemble="haar",
             bits="parity", per_pair=True, precision="fp64"),
        # Large sweep in the caller-selected split precision.
        dict(name="overlap_n16_split", kind="overlap", n=16, ne=8, W=1024, P=25000, ensemble="haar",
             bits="uniform", per_pair=False, precision="tf32x3"),
        # Several molecules in one call, mixed active spaces up to the largest supported one.
        dict(name="batch_five_spaces", kind="batch", systems=FIVE_SPACES),
        # One propagation step: overlaps, walker gradients and the force bias of every
        # Cholesky field.
        dict(name="grad_force_bias_n16", kind="grad", n=16, ne=8, W=512, P=10000, nchol=64, bits="uniform"),
        # Trial optimisation through torch.autograd: forward and backward on a small batch of
        # an odd size.
        dict(name="autograd_n10_small", kind="autograd", n=10, ne=4, W=23, P=701, bits="parity"),
        # Energy measurement every few steps on a sample of walkers.
        dict(name="local_energy_n16", kind="energy", n=16, ne=8, W=64, P=1000, nchol=64, bits="uniform"),
        # Once per data set: all two- and four-Majorana correlators, the 1-RDM and the
        # particle number from the snapshots alone.
        dict(name="rdm_n16", kind="rdm", n=16, P=60000, bits="parity", rotated=False),
        # Virtual-correlation-energy step: two spin sectors of a 200-orbital space carried to
        # the active space, then the active-space overlap.
        dict(name="vce_overlap_n16", kind="vce", NB=200, nc=20, na=8, nea=4, W=1024, P=1500),
        # New shadow data arrives: the snapshot set is built, its parities read and a first
        # walker batch evaluated.
        dict(name="new_snapshots_n16", kind="build", n=16, ne=8, W=16, P=20000, ensemble="haar", bits="uniform"),
    ]


# ------------------------------------------------------------------ drawn cases

def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _electrons(rng, n):
    return rng.choice([ne for ne in range(2, n + 1, 2) if n / 4 <= ne <= 3 * n / 4])


def _counts(rng, n, ne, cap, wlo, whi, plo, phi):
    """Walkers and snapshots, log-uniform, with the pair work at most cap flops."""
    W, P = _log_int(rng, wlo, whi), _log_int(rng, plo, phi)
    f = _pair_flops(n, ne)
    while W * P * f > cap and (W > wlo or P > plo):
        if P > plo and (W <= wlo or rng.random() < 0.5):
            P = max(plo, int(P * 0.7))
        else:
            W = max(wlo, int(W * 0.7))
    return W, P


def draw(rng):
    kind = rng.choice(["overlap"] * 5 + ["batch", "grad", "grad", "autograd", "energy", "rdm", "vce", "build"])
    if kind in ("overlap", "build"):
        n = rng.choice([6, 8, 10, 12, 13, 14, 15, 16, 16, 16, 16, 18, 20, 21, 24])
        ne = _electrons(rng, n)
        W, P = _counts(rng, n, ne, 4e11, 4, 1024, 200, 25000)
        ens, bits = rng.choice([("haar", "uniform"), ("haar", "parity"), ("signed_perm", "parity")])
        if kind == "build":
            return dict(kind=kind, n=n, ne=ne, W=min(W, 64), P=P, ensemble=ens, bits=bits)
        precision = rng.choice(["fp64", "fp64", "fp64", "tf32x3"])
        per_pair = precision == "fp64" and W * P < 2000000 and rng.random() < 0.4
        return dict(kind=kind, n=n, ne=ne, W=W, P=P, ensemble=ens, bits=bits, per_pair=per_pair,
                    precision=precision)
    if kind == "batch":
        out = []
        for _ in range(rng.randint(2, 5)):
            n = rng.choice([8, 10, 12, 14, 16, 18, 20, 22, 24])
            ne = _electrons(rng, n)
            W, P = _counts(rng, n, ne, 8e10, 16, 1024, 500, 40000)
            out.append(f"{n},{ne},{W},{P}")
        return dict(kind=kind, systems=";".join(out))
    if kind in ("grad", "autograd"):
        n = rng.choice([8, 10, 12, 13, 14, 16, 16, 16, 17, 18, 20])
        ne = _electrons(rng, n)
        big = kind == "grad"
        W, P = _counts(rng, n, ne, 1e11 if big else 1e10, 4, 512 if big else 64, 200, 10000 if big else 3000)
        bits = rng.choice(["uniform", "parity"])
        if big:
            return dict(kind=kind, n=n, ne=ne, W=W, P=P, nchol=rng.choice([1, 16, 37, 64]), bits=bits)
        return dict(kind=kind, n=n, ne=ne, W=W, P=P, bits=bits)
    if kind == "energy":
        n = rng.choice([8, 10, 12, 14, 16])
        ne = _electrons(rng, n)
        nchol = _log_int(rng, 4, 64)
        W, P = _counts(rng, n, ne, 1.5e11 / nchol, 2, 64, 100, 1000)
        return dict(kind=kind, n=n, ne=ne, W=W, P=P, nchol=nchol, bits=rng.choice(["uniform", "parity"]))
    if kind == "rdm":
        n = rng.choice([4, 6, 8, 11, 12, 14, 16])
        return dict(kind=kind, n=n, P=_log_int(rng, 500, 60000), bits="parity", rotated=rng.random() < 0.5)
    na = rng.choice([4, 6, 8])
    nea = rng.choice([e for e in range(2, na) if e <= na // 2 + 1])
    return dict(kind="vce", NB=_log_int(rng, 40, 200), nc=rng.randint(2, 20), na=na, nea=nea,
                W=_log_int(rng, 8, 1024), P=_log_int(rng, 200, 1500))


# ----------------------------------------------------------------------- inputs

def _rand(gen, *shape):
    return torch.randn(*shape, dtype=torch.float64, device=DEV, generator=gen)


def _haar(gen, N, P):
    """Haar-random O(N) matrices as products of Householder reflections, and their determinants."""
    sg = torch.randint(0, 2, (P, N), device=DEV, generator=gen).double().mul_(2).sub_(1)
    Q = torch.diag_embed(sg)
    for k in range(2, N + 1):
        v = _rand(gen, P, k)
        v[:, 0] += torch.copysign(v.norm(dim=1), v[:, 0])
        v /= v.norm(dim=1, keepdim=True)
        sub = Q[:, N - k:, N - k:]
        sub -= 2.0 * v[:, :, None] * torch.bmm(v[:, None, :], sub)
    return Q, sg.prod(dim=1) * (-1.0) ** (N - 1)


def _signed_perm(gen, N, P):
    perm = torch.rand(P, N, device=DEV, generator=gen).argsort(dim=1)
    sg = torch.randint(0, 2, (P, N), device=DEV, generator=gen).double().mul_(2).sub_(1)
    Q = torch.zeros(P, N, N, dtype=torch.float64, device=DEV).scatter_(2, perm[:, :, None], sg[:, :, None])
    upper = torch.ones(N, N, dtype=torch.bool, device=DEV).triu(1)
    inv = ((perm[:, :, None] > perm[:, None, :]) & upper).sum(dim=(1, 2))
    return Q, sg.prod(dim=1) * (1 - 2 * (inv % 2)).double()


def _shadows(gen, n, P, ensemble, bits):
    """Q (P, 2n, 2n), b (P, n) and the parities det(Q) (-1)^|b|."""
    Q, det = (_signed_perm if ensemble == "signed_perm" else _haar)(gen, 2 * n, P)
    b = torch.randint(0, 2, (P, n), device=DEV, generator=gen, dtype=torch.uint8)
    par = det * (1 - 2 * (b.sum(dim=1) % 2)).double()
    if bits == "parity":
        b[:, 0] ^= (par < 0).to(torch.uint8)
        par = par.abs()
    return Q.contiguous(), b.contiguous(), par


def _walkers(gen, W, n, ne):
    Z = torch.complex(_rand(gen, W, n, ne), _rand(gen, W, n, ne))
    L = torch.linalg.cholesky(Z.mH @ Z)
    Z = torch.linalg.solve_triangular(L.mH, Z, upper=True, left=False)
    u = torch.rand(W, 2, dtype=torch.float64, device=DEV, generator=gen)
    s = torch.polar(0.5 + 1.5 * u[:, 0], 2.0 * math.pi * u[:, 1])
    return (Z * s[:, None, None]).contiguous()


def _symmetric(gen, count, n):
    X = _rand(gen, count, n, n)
    return (0.5 * (X + X.transpose(1, 2))).to(torch.complex128).contiguous()


def _systems(case):
    return [tuple(int(x) for x in s.split(",")) for s in case["systems"].split(";")]


def _inputs(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(7919 * int(seed) + 13)
    k = case["kind"]
    if k == "batch":
        return [dict(zip(("Q", "b", "par"), _shadows(gen, n, P, "haar", "uniform")), Phi=_walkers(gen, W, n, ne))
                for n, ne, W, P in _systems(case)]
    n = 2 * case["na"] if k == "vce" else case["n"]
    x = dict(zip(("Q", "b", "par"), _shadows(gen, n, case["P"], case.get("ensemble", "haar"),
                                             case.get("bits", "uniform"))))
    if k == "rdm":
        x["R"] = _haar(gen, 2 * n, 1)[0][0].contiguous() if case["rotated"] else None
    elif k == "vce":
        for spin in ("up", "down"):
            x[spin] = _walkers(gen, case["W"], case["NB"], case["nc"] + case["nea"])
    else:
        x["Phi"] = _walkers(gen, case["W"], n, case["ne"])
    if "nchol" in case:
        x["L"] = _symmetric(gen, case["nchol"], n)
        x["h"] = _symmetric(gen, 1, n)[0].contiguous()
    return x


_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        torch.cuda.set_device(0)
        _ctx = qcs.Context(0)
    return _ctx


def prepare(case, seed):
    """The snapshot set (a handle that lives for a whole AFQMC run) and the step's walkers."""
    ctx = _context()
    x = _inputs(case, seed)
    st = dict(case=case, ctx=ctx)
    if case["kind"] == "batch":
        st["systems"] = [(qcs.Snapshots(ctx, y["Q"], y["b"]), y["Phi"]) for y in x]
    elif case["kind"] == "build":
        st.update(Q=x["Q"], b=x["b"], Phi=x["Phi"])
    else:
        st["snaps"] = qcs.Snapshots(ctx, x["Q"], x["b"])
        st.update({k: v for k, v in x.items() if k not in ("Q", "b", "par")})
    if case["kind"] == "autograd":
        st["Phi"].requires_grad_(True)
    torch.cuda.synchronize()
    return st


# ----------------------------------------------------------------- the user's call

def run(st):
    case, ctx = st["case"], st["ctx"]
    k = case["kind"]
    if k == "overlap":
        prec = qcs.QCS_TF32X3 if case["precision"] == "tf32x3" else qcs.QCS_FP64
        ov, pp = qcs.overlap(ctx, st["snaps"], st["Phi"], per_pair=case["per_pair"], precision=prec)
        return (ov, pp) if case["per_pair"] else (ov,)
    if k == "batch":
        return tuple(qcs.overlap_batched(ctx, st["systems"]))
    if k == "grad":
        ov, g = qcs.overlap_grad(ctx, st["snaps"], st["Phi"])
        return ov, g, qcs.force_bias(ctx, st["L"], st["Phi"].detach(), ov, g, sqrt_dt=0.1)
    if k == "autograd":
        Phi = st["Phi"]
        Phi.grad = None
        ov = qcs.OverlapFn.apply(Phi, ctx, st["snaps"])
        ov.abs().square().sum().backward()
        return ov.detach(), Phi.grad
    if k == "energy":
        return qcs.local_energy(ctx, st["snaps"], st["Phi"], st["L"], st["h"])
    if k == "rdm":
        return qcs.shadow_rdm(ctx, st["snaps"], st["R"])
    if k == "vce":
        nc, na, nea, W = case["nc"], case["na"], case["nea"], case["W"]
        act = torch.zeros(W, 2 * na, 2 * nea, dtype=torch.complex128, device=DEV)
        _, fu = qcs.vce_transform(ctx, st["up"], nc, na, nea, act=act, row0=0, col0=0)
        _, fd = qcs.vce_transform(ctx, st["down"], nc, na, nea, act=act, row0=na, col0=nea)
        ov, _ = qcs.overlap(ctx, st["snaps"], act)
        return (ov * fu * fd,)
    snaps = qcs.Snapshots(ctx, st["Q"], st["b"])  # build
    ov, _ = qcs.overlap(ctx, snaps, st["Phi"])
    return snaps.parity(), ov


# ------------------------------------------------------------------ necessary work

def _tri(m):
    return m * (m - 1) // 2


def _pair_flops(n, ne):
    """Congruence of the selected rows with the snapshot's covariance and the Pfaffians of
    the Gauss rule's nodes, the occupied block eliminated once."""
    m, d = 2 * n - ne, n - ne
    nodes = (d // 2 + 2) // 2
    f = 8.0 * n * n * n + 8.0 * n * n * m
    f += sum(16.0 * _tri(r - 2) for r in range(m, 2 * d, -2))
    return f + nodes * sum(16.0 * _tri(r - 2) for r in range(2 * d, 2, -2))


def _set_bytes(n, P):
    return P * (32.0 * n * n + n)


def work(case):
    k = case["kind"]
    if k == "batch":
        by = fl = 0.0
        for n, ne, W, P in _systems(case):
            by += _set_bytes(n, P) + 16.0 * W * (n * ne + 1)
            fl += 0.5 * W * P * _pair_flops(n, ne)
        return dict(bytes=by, flops=fl)
    P = case["P"]
    live = 0.5 if case.get("bits", "uniform") == "uniform" else 1.0  # parity -1 pairs are exactly zero
    if k == "rdm":
        n = case["n"]
        np_ = _tri(2 * n)
        return dict(bytes=_set_bytes(n, P) + 8.0 * (4 * n * n + math.comb(2 * n, 4)) + 16.0 * n * n,
                    flops=float(P) * np_ * (np_ + 1) + 4.0 * P * n * np_)
    if k == "vce":
        n, ne, W, e = 2 * case["na"], 2 * case["nea"], case["W"], case["nc"] + case["nea"]
        return dict(bytes=_set_bytes(n, P) + 16.0 * W * (2 * (case["nc"] + case["na"]) * e + 1),
                    flops=live * W * P * _pair_flops(n, ne) + 2.0 * W * 16.0 * e * e * case["nc"])
    n, ne, W = case["n"], case["ne"], case["W"]
    by = _set_bytes(n, P) + 16.0 * W * (n * ne + 1)
    pf = _pair_flops(n, ne)
    if k == "overlap" and case["per_pair"]:
        by += 16.0 * W * P
    if k == "build":
        by += P
    if k in ("grad", "autograd"):
        by += 16.0 * W * n * ne
        m, d = 2 * n - ne, n - ne
        nodes = (d // 2 + 2) // 2
        pf += nodes * sum(16.0 * r * r for r in range(2 * d - 2, 0, -2)) + 8.0 * n * n * m
        pf += sum(16.0 * r * r for r in range(2 * d, m, 2))
    if k == "grad":
        by += 16.0 * case["nchol"] * (n * n + W)
    if k == "energy":
        by += 16.0 * (case["nchol"] + 1) * n * n + 32.0 * W
        m, d = 2 * n - ne, n - ne
        pf += case["nchol"] * (4.0 * n * m * m + 16.0 * d * m * d)
    return dict(bytes=by, flops=live * W * P * pf)


# --------------------------------------------------- the same values in 64 bits

def _covariances(Q, b):
    """G_p = Q_p^T C_b Q_p (P, 2n, 2n)."""
    s = (1 - 2 * b.double())[:, :, None]
    even, odd = Q[:, 0::2, :], Q[:, 1::2, :] * s
    G = even.transpose(1, 2) @ odd
    return G - G.transpose(1, 2)


def _frames(Phi):
    """Unitary completion U and triangular factor R of each walker, with its selected rows X."""
    W, n, ne = Phi.shape
    U = torch.empty(W, n, n, dtype=Phi.dtype, device=Phi.device)
    R = torch.empty(W, ne, ne, dtype=Phi.dtype, device=Phi.device)
    A = Phi.clone()
    U[:] = torch.eye(n, dtype=Phi.dtype, device=Phi.device)
    for k in range(ne):  # complex Householder reflections, batched over the walkers
        x = A[:, k:, k]
        ph = x[:, 0] / x[:, 0].abs().clamp_min(1e-300)
        ph = torch.where(x[:, 0].abs() > 0, ph, torch.ones_like(ph))
        v = x.clone()
        v[:, 0] += ph * x.norm(dim=1)
        t = 2.0 / v.abs().square().sum(dim=1)
        A[:, k:, :] -= (t[:, None] * v)[:, :, None] * (v.conj()[:, None, :] @ A[:, k:, :])
        U[:, :, k:] -= (U[:, :, k:] @ v[:, :, None]) * (t[:, None] * v.conj())[:, None, :]
    R[:] = A[:, :ne, :].triu()
    T = torch.stack((U.transpose(1, 2), -1j * U.transpose(1, 2)), dim=-1).reshape(W, n, 2 * n)
    emp = torch.stack((T[:, ne:].real, -T[:, ne:].imag), dim=2).reshape(W, 2 * (n - ne), 2 * n)
    X = torch.cat((T[:, :ne] / math.sqrt(2.0), emp.to(T.dtype)), dim=1)
    return U, R, T, X


def _nodes(n, ne):
    """Points w_k on the unit circle and weights g_k with sum_x c_x C(2n,2x)/C(n,x) =
    sum_k g_k pf(B + w_k D) for a snapshot of parity +1 (roots of unity, one of each pair)."""
    d, l = n - ne, n - ne // 2
    N = d + 1
    wt = [math.comb(2 * n, 2 * (l - k)) / math.comb(n, l - k) for k in range(N)]
    out = []
    for j in range(N // 2 + 1):
        w = complex(math.cos(2 * math.pi * j / N), math.sin(2 * math.pi * j / N))
        g = sum(wt[k] * complex(math.cos(2 * math.pi * j * k / N), -math.sin(2 * math.pi * j * k / N))
                for k in range(N)) / N
        out.append((w, g if j == 0 or 2 * j == N else 2 * g))
    return out


def _pfaffian(A):
    """Pfaffians of a batch of complex skew-symmetric matrices (partial pivoting)."""
    m = A.shape[1]
    if m == 0:
        return torch.ones(A.shape[0], dtype=A.dtype, device=A.device)
    pf = None
    while m > 2:
        row = A[:, 0, 1:]
        p = row.abs().argmax(dim=1, keepdim=True)
        a = row.gather(1, p)[:, 0]
        rp = A.gather(1, (p + 1)[:, :, None].expand(-1, 1, m))[:, 0]
        r1 = A[:, 1, 1:].scatter(1, p, 0.0)
        f = torch.where(p[:, 0] == 0, a, -a)
        pf = f if pf is None else pf * f
        u = row.scatter(1, p, row[:, :1])[:, 1:]
        v = rp[:, 1:].scatter(1, p, rp[:, 1:2])[:, 1:]
        S = A[:, 1:, 1:]
        ix = p[:, :, None]
        S.scatter_(1, ix.expand(-1, 1, m - 1), r1[:, None, :])
        S.scatter_(2, ix.expand(-1, m - 1, 1), -r1[:, :, None])
        u = u / torch.where(a == 0, torch.ones_like(a), a)[:, None]
        m -= 2
        A = S[:, 1:, 1:]
        A = torch.addcmul(A, u[:, :, None], v[:, None, :], value=-1).addcmul_(v[:, :, None], u[:, None, :])
    return A[:, 0, 1] if pf is None else pf * A[:, 0, 1]


def _pair_blocks(X, G, entries):
    """(walker slice, snapshot slice, B (w, p, m, m)) over all pairs, `entries` complex values at a time."""
    W, m, N2 = X.shape
    P = G.shape[0]
    pc = max(1, min(P, 512))
    wc = max(1, min(W, entries // (pc * m * m)))
    Xr = torch.cat((X.real, X.imag), dim=1)
    for p0 in range(0, P, pc):
        g = G[p0:p0 + pc].transpose(0, 1).reshape(N2, -1)
        np_ = min(pc, P - p0)
        for w0 in range(0, W, wc):
            x = Xr[w0:w0 + wc]
            y = (x.reshape(-1, N2) @ g).reshape(-1, 2, m, np_, N2)
            y = torch.complex(y[:, 0], y[:, 1]).permute(0, 2, 1, 3).reshape(x.shape[0], -1, N2)
            B = (y @ X[w0:w0 + wc].transpose(1, 2)).reshape(x.shape[0], np_, m, m)
            yield slice(w0, w0 + wc), slice(p0, p0 + np_), B


def _with_node(B, w, ne):
    A = B.reshape(-1, B.shape[-2], B.shape[-1]).clone()
    i = torch.arange(ne, A.shape[1], 2, device=A.device)
    A[:, i, i + 1] += w
    A[:, i + 1, i] -= w
    return A


def _prefactor(R, n, ne):
    return torch.diagonal(R, dim1=1, dim2=2).prod(dim=1) * (2.0 * 1j ** (ne // 2) / 2.0 ** (n - ne // 2))


def _overlap64(Phi, Q, b, par, per_pair=False):
    W, n, ne = Phi.shape
    _, R, _, X = _frames(Phi)
    pos = (par > 0).nonzero()[:, 0]
    G = _covariances(Q[pos], b[pos])
    pref = _prefactor(R, n, ne)
    ov = torch.zeros(W, dtype=torch.complex128, device=DEV)
    pp = torch.zeros(W, Q.shape[0], dtype=torch.complex128, device=DEV) if per_pair else None
    for ws, ps, B in _pair_blocks(X, G, 40_000_000):
        S = 0
        for w, g in _nodes(n, ne):
            S = S + g * _pfaffian(_with_node(B, w, ne)).reshape(B.shape[:2])
        S = S * pref[ws, None]
        ov[ws] += S.sum(dim=1)
        if per_pair:
            pp[ws, pos[ps]] = S
    return ov / Q.shape[0], pp


def _gradient64(Phi, Q, b, par):
    """Overlaps and holomorphic gradients through d pf(A) = pf(A) tr(A^-1 dA) / 2."""
    W, n, ne = Phi.shape
    d, m = n - ne, 2 * n - ne
    U, R, T, X = _frames(Phi)
    pos = (par > 0).nonzero()[:, 0]
    G = _covariances(Q[pos], b[pos])
    S = torch.zeros(W, dtype=torch.complex128, device=DEV)
    Z = torch.zeros(W, 2 * n, m, dtype=torch.complex128, device=DEV)
    for ws, ps, B in _pair_blocks(X, G, 40_000_000):
        Y = 0
        for w, g in _nodes(n, ne):
            A = _with_node(B, w, ne)
            inv = torch.linalg.inv(A)
            pf = g * _pfaffian(A)
            S[ws] += pf.reshape(B.shape[:2]).sum(dim=1)
            Y = Y + pf[:, None, None] * inv
        XY = X[ws].transpose(1, 2)[:, None] @ Y.reshape(B.shape)  # (w, p, 2n, m)
        q = XY.permute(1, 2, 0, 3).reshape(B.shape[1] * 2 * n, -1)
        gp = G[ps].permute(1, 0, 2).reshape(2 * n, -1)
        z = torch.complex(gp @ q.real.contiguous(), gp @ q.imag.contiguous())
        Z[ws] += z.reshape(2 * n, -1, m).permute(1, 0, 2)
    # a rotation of orbital j into empty orbital a moves T_j by T_a and T_a's conjugate by -conj T_j
    C = T[:, ne:] @ Z[:, :, :ne] / math.sqrt(2.0)
    Zr, Zi = Z[:, :, ne::2], Z[:, :, ne + 1::2]
    Tj = T[:, :ne].conj()
    C = C + (-0.5 * (Tj @ Zr) + 0.5j * (Tj @ Zi)).transpose(1, 2)
    top = S[:, None, None] * torch.eye(ne, dtype=S.dtype, device=DEV)
    pref = _prefactor(R, n, ne) / Q.shape[0]
    g = U.conj() @ torch.cat((top, C), dim=1)
    g = torch.linalg.solve_triangular(R.transpose(1, 2), g, upper=False, left=False)
    return S * pref, g * pref[:, None, None]


def _energy64(Phi, L, h, Q, b, par):
    """First and second derivatives of O(exp(t A) Phi) at t = 0, by Cauchy's formula on a
    small circle: <hhat> and sum <Lhat^2> act on the determinant as derivatives of exp(t A)."""
    W, n, ne = Phi.shape
    K, r = 8, 0.006
    ops = torch.cat((L, h[None]))
    t = [r * complex(math.cos(2 * math.pi * k / K), math.sin(2 * math.pi * k / K)) for k in range(K)]
    E = torch.stack([torch.linalg.matrix_exp(x * ops) for x in t])  # (K, ops, n, n)
    moved = (E[:, :, None] @ Phi[None, None]).reshape(-1, n, ne)
    f = _overlap64(moved, Q, b, par)[0].reshape(K, ops.shape[0], W)
    ov = _overlap64(Phi, Q, b, par)[0]
    z = torch.tensor(t, dtype=torch.complex128, device=DEV)[:, None, None]
    e2 = 2.0 * (f[:, :-1] / z ** 2).mean(dim=0).sum(dim=0)
    e1 = (f[:, -1:] / z).mean(dim=0)[0]
    return ov, e1 / ov, e2 / ov


def _rdm64(n, Q, b, R):
    N2 = 2 * n
    X = _covariances(Q, b)
    if R is not None:
        X = R @ X @ R.T
    P = X.shape[0]
    gam2 = (math.comb(N2, 2) / math.comb(n, 1)) * X.mean(dim=0)
    # a_p^dag a_q = (g_2p - i g_2p+1)(g_2q + i g_2q+1) / 4 with <g_mu g_nu> = delta + i gam2
    M = torch.complex(torch.eye(N2, dtype=torch.float64, device=DEV), gam2)
    rdm1 = (M[0::2, 0::2] + 1j * M[0::2, 1::2] - 1j * M[1::2, 0::2] + M[1::2, 1::2]) / 4.0
    iu = torch.triu_indices(N2, N2, 1, device=DEV)
    rank = torch.full((N2, N2), -1, dtype=torch.long, device=DEV)
    rank[iu[0], iu[1]] = torch.arange(iu.shape[1], device=DEV)
    x = X[:, iu[0], iu[1]]
    S2 = x.T @ x / P
    q = torch.combinations(torch.arange(N2, device=DEV), 4)
    pair = lambda i, j: rank[q[:, i], q[:, j]]
    v = S2[pair(0, 1), pair(2, 3)] - S2[pair(0, 2), pair(1, 3)] + S2[pair(0, 3), pair(1, 2)]
    gam4 = -(math.comb(N2, 4) / math.comb(n, 2)) * v
    return dict(gam2=gam2, gam4=gam4, rdm1=rdm1, npart=torch.diagonal(rdm1).real.sum())


def _vce64(case, x):
    nc, na, nea, W = case["nc"], case["na"], case["nea"], case["W"]
    act = torch.zeros(W, 2 * na, 2 * nea, dtype=torch.complex128, device=DEV)
    f = 1.0
    for i, spin in enumerate(("up", "down")):
        V, Rc, _, _ = _frames(x[spin][:, :nc].mH.contiguous())  # core block's conjugate transpose
        act[:, i * na:(i + 1) * na, i * nea:(i + 1) * nea] = x[spin][:, nc:nc + na] @ V[:, :, nc:]
        f = f * torch.diagonal(Rc, dim1=1, dim2=2).prod(dim=1).conj() / torch.linalg.det(V)
    return (_overlap64(act, x["Q"], x["b"], x["par"])[0] * f,)


def _cost64(case):
    """Rough flops of the plain evaluation, to leave out what would take too long."""
    def pairs(n, ne, W, P):
        m = 2 * n - ne
        return W * P * (12.0 * n * m * m + 20.0 * ((n - ne) // 2 + 1) * m ** 3)
    k = case["kind"]
    if k == "batch":
        return sum(0.5 * pairs(n, ne, W, P) for n, ne, W, P in _systems(case))
    if k == "rdm":
        return 0.0
    live = 0.5 if case.get("bits", "uniform") == "uniform" else 1.0
    if k == "vce":
        return live * pairs(2 * case["na"], 2 * case["nea"], case["W"], case["P"])
    c = live * pairs(case["n"], case["ne"], case["W"], case["P"])
    if k == "energy":
        c *= 8 * (case["nchol"] + 1)
    return 6 * c if k in ("grad", "autograd") else c


def exact(case, seed):
    if _cost64(case) > 3.5e13:
        return None
    x = _inputs(case, seed)
    k = case["kind"]
    if k == "batch":
        return tuple(_overlap64(y["Phi"], y["Q"], y["b"], y["par"])[0] for y in x)
    if k == "rdm":
        return _rdm64(case["n"], x["Q"], x["b"], x["R"])
    if k == "vce":
        return _vce64(case, x)
    if k == "overlap":
        ov, pp = _overlap64(x["Phi"], x["Q"], x["b"], x["par"], case["per_pair"])
        return (ov, pp) if case["per_pair"] else (ov,)
    if k == "build":
        return x["par"].to(torch.int8), _overlap64(x["Phi"], x["Q"], x["b"], x["par"])[0]
    if k == "energy":
        return _energy64(x["Phi"], x["L"], x["h"], x["Q"], x["b"], x["par"])
    ov, g = _gradient64(x["Phi"], x["Q"], x["b"], x["par"])
    if k == "autograd":  # of sum |O|^2, in torch's convention for complex inputs
        return ov, 2.0 * ov[:, None, None] * g.conj()
    lphi = torch.einsum("gpq,wqj->wgpj", x["L"], x["Phi"])
    xb = -0.1j * torch.einsum("wgpj,wpj->wg", lphi, g) / ov[:, None]
    return ov, g, xb
