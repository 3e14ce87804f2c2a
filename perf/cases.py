"""Performance cases of the two-center multipole library: what its users have it do.

Every case goes through the public binding (``paper_0704_1672_gb300.tcm``) with the library's
default settings.  The kinds, and what each stands for:

  pair       one interaction energy of two small systems in one batched call: the smallest call a
             program makes, bound by latency and launches
  request    the plain single-request path: the moments of both systems, then their energy, one
             synchronous call after the other
  moments    the moments of one system (centre and radius computed on the device, or given)
  scan       one pair of systems at many orientations of B (Section IV of the paper): a
             protein-sized pair, or a charged shell with a ligand
  uneven     many pairs of unequal systems, each with its own degree, in one call
  gradients  energies, forces and torques of a pair at many placements (a docking step)
  serve      items of uneven degree over a pool of resident systems with cached moments, B's
             moments rotated from the cache
  surface    the energy surface over (R0, angle) at several degrees from cached moments
  direct     the exact pairwise sum for many placements

Systems are balls of uniform density (radius 1.9 N^(1/3), normal charges shifted to net zero)
or a shell of unit charges with a net excess, about a centre away from the origin.
"""
import math

import numpy as np
import torch

from paper_0704_1672_gb300 import tcm

PAD = 256  # atoms of one block in the 64-bit check


def listed():
    return [
        # the oracle-sized pair of the tests and the benchmark: one energy per call
        {"name": "pair_mixed", "kind": "pair", "n_a": 200, "n_b": 200, "lmax": 10, "precision": "mixed",
         "dtype": "f32", "rotated": False},
        # one energy of a protein-sized pair through the plain double-precision calls
        {"name": "request_fp64", "kind": "request", "n_a": 3260, "n_b": 2587, "lmax": 10, "precision": "fp64",
         "dtype": "f64"},
        # the moments of a 20,000-atom system, the binding's default precision
        {"name": "moments_mixed", "kind": "moments", "n": 20000, "lmax": 20, "precision": "mixed", "dtype": "f32",
         "given": False},
        # the moments of a large system of odd size in double, centre and radius known
        {"name": "moments_fp64", "kind": "moments", "n": 100003, "lmax": 24, "precision": "fp64", "dtype": "f64",
         "given": True},
        # the orientation scan of two 20,000-atom systems
        {"name": "scan_mixed", "kind": "scan", "shape": "ball", "n_a": 20000, "n_b": 20000, "items": 256, "lmax": 20,
         "precision": "mixed", "dtype": "f32"},
        # the same scan in double throughout (the path for ill-conditioned energies)
        {"name": "scan_fp64", "kind": "scan", "shape": "ball", "n_a": 20000, "n_b": 20000, "items": 256, "lmax": 20,
         "precision": "fp64", "dtype": "f64"},
        # the batch of uneven pairs (a quarter of the benchmark's 4,096)
        {"name": "uneven_mixed", "kind": "uneven", "pairs": 1024, "n_lo": 100, "n_hi": 100000, "precision": "mixed",
         "dtype": "f32"},
        # the large assembly: a million-charge shell and a 50,000-atom ligand
        {"name": "assembly_mixed", "kind": "scan", "shape": "shell", "n_a": 1000000, "n_b": 50000, "items": 10000,
         "lmax": 24, "precision": "mixed", "dtype": "f32"},
        # forces and torques of a ligand at many placements
        {"name": "gradients_mixed", "kind": "gradients", "n_a": 5000, "n_b": 1500, "items": 512, "lmax": 12,
         "precision": "mixed", "dtype": "f32"},
        # one iteration of the serving loop over 512 resident systems
        {"name": "serve_cached", "kind": "serve", "pool": 512, "n_lo": 500, "n_hi": 200000, "items": 2048, "l_lo": 8,
         "l_hi": 24, "precision": "mixed", "dtype": "f32"},
        # the surface scan of the paper's protein pair: 43 distances x 360 angles x 7 degrees
        {"name": "surface_cached", "kind": "surface", "n_a": 3260, "n_b": 2587, "distances": 43, "angles": 360,
         "l_max": 10, "precision": "mixed", "dtype": "f32"},
        # the exact energies of a part of that surface
        {"name": "direct_fp64", "kind": "direct", "n_a": 3260, "n_b": 2587, "items": 256, "rotated": False,
         "dtype": "f64"},
    ]


def _log(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["pair", "request", "moments", "scan", "scan", "uneven", "gradients", "serve", "surface", "direct"])
    precision = rng.choice(["mixed", "fp64"])
    dtype = rng.choice(["f32", "f64"])
    c = {"kind": kind, "precision": precision, "dtype": dtype}
    if kind in ("pair", "request"):
        c.update(n_a=_log(rng, 50, 5000), n_b=_log(rng, 50, 5000), lmax=rng.randint(2, 16))
        if kind == "pair":
            c["rotated"] = rng.random() < 0.5
    elif kind == "moments":
        c.update(n=_log(rng, 500, 1000000), lmax=rng.randint(4, 24), given=rng.random() < 0.5)
    elif kind == "scan":
        lmax = rng.randint(8, 24)
        n_b = _log(rng, 500, 50000)
        # atoms of B over all items times components: at most the assembly's, or the scan's in double
        most = 3e11 if precision == "mixed" else 3e9
        items = _log(rng, 16, max(16, min(10000, int(most / (n_b * (lmax + 1) ** 2)))))
        c.update(shape=rng.choice(["ball", "shell"]), n_a=_log(rng, 500, 200000), n_b=n_b, items=items, lmax=lmax)
    elif kind == "uneven":
        c.update(precision="mixed", dtype="f32", pairs=_log(rng, 32, 1024), n_lo=100, n_hi=_log(rng, 2000, 100000))
    elif kind == "gradients":
        lmax = rng.randint(4, 20)
        n_b = _log(rng, 200, 5000)
        most = 3e9 if precision == "mixed" else 6e8
        items = _log(rng, 16, max(16, min(2048, int(most / (n_b * (lmax + 1) ** 2)))))
        c.update(n_a=_log(rng, 500, 50000), n_b=n_b, items=items, lmax=lmax)
    elif kind == "serve":
        c.update(dtype="f32", pool=_log(rng, 32, 512), n_lo=500, n_hi=_log(rng, 5000, 200000), items=_log(rng, 64, 8192),
                 l_lo=8, l_hi=rng.randint(12, 24))
    elif kind == "surface":
        c.update(n_a=_log(rng, 500, 5000), n_b=_log(rng, 500, 5000), distances=rng.randint(5, 43),
                 angles=rng.randint(24, 360), l_max=rng.randint(3, 12))
    else:
        n_a, n_b = _log(rng, 100, 20000), _log(rng, 100, 20000)
        del c["precision"]
        c.update(n_a=n_a, n_b=n_b, items=_log(rng, 1, max(1, min(512, int(2e9 / (n_a * n_b))))),
                 rotated=rng.random() < 0.5)
    return c


# ------------------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _points(g, n, r_in, r_out):
    """n points uniform in volume between two radii."""
    v = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
    v /= v.norm(dim=1, keepdim=True)
    u = torch.rand(n, 1, generator=g, device="cuda", dtype=torch.float64)
    return v * (r_in ** 3 + u * (r_out ** 3 - r_in ** 3)) ** (1.0 / 3.0)


def _system(g, n, shape="ball"):
    """(n, 4) float64 records about a centre away from the origin, and the outer radius."""
    x = torch.empty(n, 4, device="cuda", dtype=torch.float64)
    if shape == "shell":
        r = 100.0
        x[:, :3] = _points(g, n, 0.8 * r, r)
        q = -torch.ones(n, device="cuda", dtype=torch.float64)
        q[torch.randperm(n, generator=g, device="cuda")[: (n + round(0.02 * n)) // 2]] = 1.0
    else:
        r = 1.9 * n ** (1.0 / 3.0)
        x[:, :3] = _points(g, n, 0.0, r)
        q = 0.3 * torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
        q -= q.mean()
    x[:, 3] = q
    x[:, :3] += 20.0 * torch.randn(1, 3, generator=g, device="cuda", dtype=torch.float64)
    return x, r


def _pool(g, sizes):
    """Systems of the given sizes as one (sum, 4) float64 tensor."""
    n = int(sizes.sum())
    ids = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), torch.as_tensor(sizes, device="cuda"))
    radii = torch.as_tensor(1.9 * sizes ** (1.0 / 3.0), device="cuda")
    x = torch.empty(n, 4, device="cuda", dtype=torch.float64)
    x[:, :3] = _points(g, n, 0.0, 1.0) * radii[ids][:, None]
    x[:, 3] = 0.3 * torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    mean = torch.zeros(len(sizes), device="cuda", dtype=torch.float64).index_add_(0, ids, x[:, 3])
    x[:, 3] -= (mean / torch.as_tensor(sizes, device="cuda"))[ids]
    x[:, :3] += (20.0 * torch.randn(len(sizes), 3, generator=g, device="cuda", dtype=torch.float64))[ids]
    return x


def _cast(x, case):
    return x.to(torch.float32 if case["dtype"] == "f32" else torch.float64).contiguous()


def _rotations(rng, k):
    q = rng.normal(size=(k, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    w, x, y, z = q.T
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                     2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                     2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], axis=1).reshape(k, 3, 3)


def _separations(rng, k, a_sum, lo=1.35, hi=3.0):
    v = rng.normal(size=(k, 3))
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    return v * (rng.uniform(lo, hi, k) * a_sum)[:, None]


def _inputs(case, seed):
    """Everything the case's call reads, but the library's own handles."""
    g, rng, kind = _gen(seed), np.random.default_rng(seed), case["kind"]
    if kind == "moments":
        x, r = _system(g, case["n"])
        x = _cast(x, case)
        c = x[:, :3].double().mean(0)
        a = float((x[:, :3].double() - c).norm(dim=1).max())
        return {"x": x, "lmax": case["lmax"], "center": c.cpu().numpy() if case["given"] else None,
                "radius": a if case["given"] else None}
    if kind in ("uneven", "serve"):
        count = 2 * case["pairs"] if kind == "uneven" else case["pool"]
        sizes = np.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), count)).astype(np.int64)
        radii = 1.9 * sizes ** (1.0 / 3.0)
        k = case["pairs"] if kind == "uneven" else case["items"]
        if kind == "uneven":
            a = np.arange(0, count, 2)
            b = a + 1
            lmax = rng.choice(np.array([8, 12, 16, 24]), k)
        else:
            a = rng.integers(0, count, k)
            b = (a + rng.integers(1, count, k)) % count
            lmax = rng.integers(case["l_lo"], case["l_hi"] + 1, k)
        return {"x": _cast(_pool(g, sizes), case), "sizes": sizes, "a": a, "b": b, "lmax": lmax,
                "rot": _rotations(rng, k), "R0": _separations(rng, k, radii[a] + radii[b])}
    (xa, ra), (xb, rb) = _system(g, case["n_a"], case.get("shape", "ball")), _system(g, case["n_b"])
    s = {"A": _cast(xa, case), "B": _cast(xb, case), "rot": None}
    if kind == "surface":
        r = np.linspace(1.35, 2.4, case["distances"]) * (ra + rb)
        t = np.linspace(0.0, 2.0 * np.pi, case["angles"], endpoint=False) + rng.uniform(0.0, 0.01)
        R0 = np.stack([np.outer(r, np.cos(t)), np.outer(r, np.sin(t)), np.zeros((len(r), len(t)))], axis=-1).reshape(-1, 3)
        degrees = [L for L in (1, 2, 3, 4, 6, 8, 10, 12) if L <= case["l_max"]]
        s.update(R0=np.tile(R0, (len(degrees), 1)), lmax=np.repeat(degrees, len(R0)))
        return s
    k = case.get("items", 1)
    if kind in ("scan", "gradients") or case.get("rotated"):
        s["rot"] = _rotations(rng, k)
    s["R0"] = _separations(rng, k, ra + rb)
    s["lmax"] = np.full(k, case.get("lmax", 0))
    return s


def _bounds(sizes):
    return np.concatenate([[0], np.cumsum(sizes)])


def prepare(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    s["kind"] = kind
    s["precision"] = tcm.TCM_FP64 if case.get("precision") == "fp64" else tcm.TCM_MIXED
    s["ctx"] = ctx = tcm.Context(lmax_cap=24)
    if kind in ("uneven", "serve"):  # systems resident in one buffer, each described once
        at = _bounds(s["sizes"])
        xs = [s["x"][at[i]:at[i + 1]] for i in range(len(s["sizes"]))]
        if kind == "uneven":
            s["systems"] = [tcm.make_system(x) for x in xs]
        else:  # each with its centre, radius and moment cache, as the server keeps them
            s["systems"], s["cache"] = [], []
            for x in xs:
                m = ctx.tcm_moments(x, case["l_hi"], precision=s["precision"])
                s["cache"].append(m)
                s["systems"].append(tcm.make_system(x, center=m.center, radius=m.radius, moments=m))
            ctx.tcm_ctx_set_rotate_cached(True)
    elif kind == "surface":  # fixed systems: their moments once, the grid's items marshalled once
        m = [ctx.tcm_moments(s[k], case["l_max"], precision=s["precision"]) for k in ("A", "B")]
        systems = [tcm.make_system(s[k], center=q.center, radius=q.radius, moments=q) for k, q in zip(("A", "B"), m)]
        n = len(s["R0"])
        s["cache"] = m
        s["packed"] = tcm.pack_batch(systems, np.zeros(n, int), np.ones(n, int), s["lmax"], s["R0"])
    elif kind in ("pair", "scan", "gradients"):
        n = len(s["R0"])
        s.update(systems=[(s["A"], None, None), (s["B"], None, None)], a=np.zeros(n, int), b=np.ones(n, int))
    return s


def run(s):
    ctx, kind, p = s["ctx"], s["kind"], s["precision"]
    if kind == "moments":
        m = ctx.tcm_moments(s["x"], s["lmax"], precision=p, center=s["center"], radius=s["radius"])
        return {"q": m.q, "center": m.center, "radius": m.radius}
    if kind == "request":
        L = int(s["lmax"][0])
        ma = ctx.tcm_moments(s["A"], L, precision=p)
        mb = ctx.tcm_moments(s["B"], L, precision=p)
        return {"qa": ma.q, "qb": mb.q, "E": ctx.tcm_energy(ma, mb, s["R0"][0])}
    if kind == "surface":
        E, status = ctx.tcm_energy_batch_packed(s["packed"], p)
        return {"E": E, "status": status}
    if kind == "direct":
        return {"E": ctx.tcm_direct_batch(s["A"], s["B"], s["R0"], rotB=s["rot"])}
    if kind == "gradients":
        E, G, status = ctx.tcm_gradients_batch(s["systems"], s["a"], s["b"], s["lmax"], s["R0"], rotB=s["rot"],
                                               precision=p)
        return {"E": E, "G": G, "status": status}
    E, status = ctx.tcm_energy_batch(s["systems"], s["a"], s["b"], s["lmax"], s["R0"], rotB=s["rot"], precision=p)
    return {"E": E, "status": status}


# ------------------------------------------------------------------------------ work

def _moment_flops(n, L):
    """Per atom: a recurrence step and an accumulation per component (5), the set-up (40)."""
    return n * (5.0 * (L + 1) ** 2 + 40.0)


def _energy_flops(L, sides):
    """One energy: each of ``sides`` moment sets turned into the frame of R0 (two products with
    d^l(pi/2), phases), and the contraction along the z axis."""
    s2 = sum((l + 1) ** 2 for l in range(L + 1))
    z = sum(2 * min(a, b) + 3 for a in range(L + 1) for b in range(L + 1))
    return sides * (4.0 * s2 + 12.0 * (L + 1) * (L + 2)) + 2.0 * z


def work(case):
    kind = case["kind"]
    rec = 16 if case["dtype"] == "f32" else 32
    if kind == "moments":
        return {"bytes": rec * case["n"] + 8 * (case["lmax"] + 1) ** 2, "flops": _moment_flops(case["n"], case["lmax"])}
    if kind == "direct":
        n = case["n_a"] + case["n_b"]
        return {"bytes": rec * n + case["items"] * (104 if case["rotated"] else 32),
                "flops": 20.0 * case["items"] * case["n_a"] * case["n_b"]}
    if kind == "surface":
        degrees = [L for L in (1, 2, 3, 4, 6, 8, 10, 12) if L <= case["l_max"]]
        n = case["distances"] * case["angles"]
        return {"bytes": 16 * (case["l_max"] + 1) ** 2 + 36 * n * len(degrees),
                "flops": n * sum(_energy_flops(L, 2) for L in degrees)}
    if kind == "uneven":
        mean = (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])  # of a log-uniform size
        n = 2 * case["pairs"] * mean
        return {"bytes": rec * n + 108 * case["pairs"],
                "flops": sum(_moment_flops(n / 4, L) + case["pairs"] / 4 * _energy_flops(L, 1) for L in (8, 12, 16, 24))}
    if kind == "serve":
        degrees = range(case["l_lo"], case["l_hi"] + 1)
        return {"bytes": 8 * case["pool"] * (case["l_hi"] + 1) ** 2 + 108 * case["items"],
                "flops": case["items"] * sum(_energy_flops(L, 2) for L in degrees) / len(degrees)}
    k, L = case.get("items", 1), case["lmax"]
    flops = _moment_flops(case["n_a"] + case["n_b"], L) + k * _energy_flops(L, 2)
    if kind == "gradients":
        flops += k * 4.0 * sum(12 * min(a, b) + 20 for a in range(L + 1) for b in range(L + 1))
    out = 84 if kind == "gradients" else 12
    if kind == "request":
        out += 16 * (L + 1) ** 2
    return {"bytes": rec * (case["n_a"] + case["n_b"]) + k * (96 + out), "flops": flops}


# ------------------------------------------------------------------------------ in 64 bits

def _solid_sums(x, q, L):
    """Sums over the last axis of q r^l sqrt(4 pi/(2l+1)) Y_lm at x (..., 3): {(l, m): (re, im)}."""
    X, Y, Z = x.unbind(-1)
    r2 = X * X + Y * Y + Z * Z
    out = {}
    pr, pi = q * torch.ones_like(X), torch.zeros_like(X)
    for m in range(L + 1):
        if m:
            f = -math.sqrt((2 * m - 1) / (2 * m))
            pr, pi = f * (pr * X - pi * Y), f * (pr * Y + pi * X)
        last, cur = None, (pr, pi)
        for l in range(m, L + 1):
            out[l, m] = (cur[0].sum(-1), cur[1].sum(-1))
            if l < L:
                a = (2 * l + 1) / math.sqrt((l + 1) ** 2 - m * m)
                b = math.sqrt(l * l - m * m) / math.sqrt((l + 1) ** 2 - m * m)
                nxt = tuple(a * Z * c for c in cur) if last is None else tuple(
                    a * Z * c - b * r2 * p for c, p in zip(cur, last))
                last, cur = cur, nxt
    return out


def _energies(qa, qb, R, L):
    """The energies of moment sums in the frame where R0 lies along z."""
    f = math.factorial
    E = 0.0
    for l1 in range(L + 1):
        for l2 in range(L + 1):
            t = 0.0
            for m in range(min(l1, l2) + 1):
                w = (1.0 if m == 0 else 2.0 * (-1) ** m) / math.sqrt(f(l1 + m) * f(l1 - m)) / math.sqrt(f(l2 + m) * f(l2 - m))
                t = t + w * (qa[l1, m][0] * qb[l2, m][0] + qa[l1, m][1] * qb[l2, m][1])
            E = E + (-1) ** l2 * float(f(l1 + l2)) * t / R ** (l1 + l2 + 1)
    return E


def _frames(R0):
    """Rotations (k, 3, 3) that take each R0 (k, 3) to the z axis, and the lengths."""
    x, y, z = R0.unbind(-1)
    rho, R = torch.sqrt(x * x + y * y), torch.sqrt(x * x + y * y + z * z)
    ca, sa, cb, sb, o = x / rho, y / rho, z / R, rho / R, torch.zeros_like(x)
    return torch.stack([cb * ca, cb * sa, -sb, -sa, ca, o, sb * ca, sb * sa, cb], dim=-1).reshape(-1, 3, 3), R


def _packed(Q, L):
    return torch.stack([Q[l, (j + 1) // 2][0 if j % 2 or j == 0 else 1] for l in range(L + 1) for j in range(2 * l + 1)])


def _lab_moments(x, L):
    """Moments of one system about its centroid in the lab frame, and the radius."""
    x = x.double()
    d = x[:, :3] - x[:, :3].mean(0)
    return _solid_sums(d, x[:, 3], L), d.norm(dim=1).max()


def _few_charges(Q, s, L):
    """Charges on a sphere of radius s that have the moments Q (Gauss-Legendre times equispaced
    angles: exact for products of two harmonics of degree <= L), for one system or, with sums and
    radii of shape (n,), for n at once: positions (..., p, 3), charges (..., p)."""
    z, w = np.polynomial.legendre.leggauss(L + 1)
    t = np.arange(2 * L + 1) * (2.0 * np.pi / (2 * L + 1))
    rho = np.sqrt(1.0 - z * z)
    n = np.stack([np.outer(rho, np.cos(t)), np.outer(rho, np.sin(t)), np.outer(z, np.ones_like(t))], -1).reshape(-1, 3)
    n = torch.as_tensor(n, device="cuda")
    w = torch.as_tensor(np.repeat(0.5 * w, 2 * L + 1) / (2 * L + 1), device="cuda")
    C = _solid_sums(n[:, None, :], torch.ones(len(n), 1, device="cuda", dtype=torch.float64), L)
    q = 0.0
    for (l, m), (cr, ci) in C.items():
        f = (2 * l + 1) * (1 if m == 0 else 2) * s ** -l
        q = q + (f * Q[l, m][0])[..., None] * cr + (f * Q[l, m][1])[..., None] * ci
    return s[..., None, None] * n, w * q


def _apply(M, p):
    return torch.einsum("kij,...pj->kpi", M, p) if p.dim() == 2 else torch.einsum("kij,kpj->kpi", M, p)


def _exact_scan(case, s, grad):
    L = case["lmax"]
    few = []
    for k in ("A", "B"):
        Q, a = _lab_moments(s[k], L)
        few.append(_few_charges(Q, a, L))
    (pa, qa), (pb, qb) = few
    R0 = torch.as_tensor(s["R0"], device="cuda")
    rot = None if s["rot"] is None else torch.as_tensor(s["rot"], device="cuda")
    E, G = [], []
    step = max(1, (1 << (17 if grad else 22)) // len(pa))
    for i in range(0, len(R0), step):
        r = R0[i:i + step].clone()
        xa = pa.expand(len(r), -1, -1)
        xb = pb.expand(len(r), -1, -1) if rot is None else _apply(rot[i:i + step], pb)
        if grad:
            wa, wb = torch.zeros_like(r, requires_grad=True), torch.zeros_like(r, requires_grad=True)
            r.requires_grad_(True)
            xa = xa + torch.cross(wa[:, None, :].expand_as(xa), xa, dim=-1)
            xb = xb + torch.cross(wb[:, None, :].expand_as(xb), xb, dim=-1)
        W, R = _frames(r)
        e = _energies(_solid_sums(_apply(W, xa), qa, L), _solid_sums(_apply(W, xb), qb, L), R, L)
        if grad:
            d = torch.autograd.grad(e.sum(), (r, wa, wb))
            G.append(-torch.cat(d, dim=1))
        E.append(e.detach())
    return torch.cat(E), torch.cat(G) if grad else None


def _blocks(s, which, M=None):
    """The listed systems about their centroids (turned by M, one matrix each), cut into blocks of
    PAD atoms that are filled up with zero charges: (n, PAD, 4), each block's place in the list."""
    at, blocks, owner = _bounds(s["sizes"]), [], []
    for j, k in enumerate(which):
        x = s["x"][at[k]:at[k + 1]].double()
        d = x[:, :3] - x[:, :3].mean(0)
        n = -(-len(x) // PAD)
        b = torch.zeros(n * PAD, 4, device="cuda", dtype=torch.float64)
        b[:len(x), :3], b[:len(x), 3] = d if M is None else d @ M[j].T, x[:, 3]
        blocks.append(b.reshape(n, PAD, 4))
        owner.append(np.full(n, j))
    return torch.cat(blocks), torch.as_tensor(np.concatenate(owner), device="cuda")


def _sums_of(blocks, owner, count, L):
    zero = torch.zeros(count, device="cuda", dtype=torch.float64)
    Q = _solid_sums(blocks[..., :3].contiguous(), blocks[..., 3].contiguous(), L)
    return {k: tuple(zero.index_add(0, owner, v) for v in c) for k, c in Q.items()}


def _exact_uneven(s):
    """Every pair straight from its atoms, turned into the pair's frame."""
    E = torch.zeros(len(s["a"]), device="cuda", dtype=torch.float64)
    W, R = _frames(torch.as_tensor(s["R0"], device="cuda"))
    rot = torch.as_tensor(s["rot"], device="cuda")
    for L in np.unique(s["lmax"]):
        items = np.nonzero(s["lmax"] == L)[0]
        k = torch.as_tensor(items, device="cuda")
        qa, qb = (_sums_of(*_blocks(s, side[items], M), len(items), int(L))
                  for side, M in ((s["a"], W[k]), (s["b"], W[k] @ rot[k])))
        E[k] = _energies(qa, qb, R[k], int(L))
    return E


def _exact_serve(case, s):
    """Every system replaced by few charges with its moments; the items by degree."""
    L0, n = case["l_hi"], len(s["sizes"])
    blocks, owner = _blocks(s, np.arange(n))
    radius = torch.as_tensor(1.9 * s["sizes"] ** (1.0 / 3.0), device="cuda")
    p, q = _few_charges(_sums_of(blocks, owner, n, L0), radius, L0)
    W, R = _frames(torch.as_tensor(s["R0"], device="cuda"))
    M = W @ torch.as_tensor(s["rot"], device="cuda")
    E = torch.zeros(len(s["a"]), device="cuda", dtype=torch.float64)
    for L in np.unique(s["lmax"]):
        items = np.nonzero(s["lmax"] == L)[0]
        for i in range(0, len(items), 2048):
            k = torch.as_tensor(items[i:i + 2048], device="cuda")
            a, b = (torch.as_tensor(s[side][items[i:i + 2048]], device="cuda") for side in ("a", "b"))
            E[k] = _energies(_solid_sums(_apply(W[k], p[a]), q[a], int(L)), _solid_sums(_apply(M[k], p[b]), q[b], int(L)),
                             R[k], int(L))
    return E


def _exact_surface(s):
    """Few charges for both systems at the largest degree, then every grid point once per degree."""
    L0 = int(s["lmax"].max())
    few = [_few_charges(*_lab_moments(s[k], L0), L0) for k in ("A", "B")]
    E = torch.zeros(len(s["R0"]), device="cuda", dtype=torch.float64)
    for L in np.unique(s["lmax"]):
        items = np.nonzero(s["lmax"] == L)[0]
        for i in range(0, len(items), 4096):
            k = items[i:i + 4096]
            W, R = _frames(torch.as_tensor(s["R0"][k], device="cuda"))
            qa, qb = (_solid_sums(_apply(W, p), q, int(L)) for p, q in few)
            E[torch.as_tensor(k, device="cuda")] = _energies(qa, qb, R, int(L))
    return E


def _exact_direct(s):
    A, B = s["A"].double(), s["B"].double()
    a, b = A[:, :3] - A[:, :3].mean(0), B[:, :3] - B[:, :3].mean(0)
    E = []
    for k in range(len(s["R0"])):
        x = b if s["rot"] is None else b @ torch.as_tensor(s["rot"][k], device="cuda").T
        x = x + torch.as_tensor(s["R0"][k], device="cuda")
        e = torch.zeros((), device="cuda", dtype=torch.float64)
        for i in range(0, len(a), 4096):
            d2 = sum((x[None, :, j] - a[i:i + 4096, None, j]) ** 2 for j in range(3))
            e = e + (A[i:i + 4096, 3] * (B[:, 3] / torch.sqrt(d2)).sum(1)).sum()
        E.append(e)
    return torch.stack(E)


def exact(case, seed):
    s, kind = _inputs(case, seed), case["kind"]
    with torch.no_grad() if kind != "gradients" else torch.enable_grad():
        if kind == "moments":
            x = s["x"].double()
            c = x[:, :3].mean(0) if s["center"] is None else torch.as_tensor(s["center"], device="cuda")
            d = x[:, :3] - c
            radius = float(d.norm(dim=1).max()) if s["radius"] is None else s["radius"]
            return {"q": _packed(_solid_sums(d, x[:, 3], case["lmax"]), case["lmax"]), "center": c.cpu().numpy(),
                    "radius": radius}
        if kind == "direct":
            return {"E": _exact_direct(s)}
        if kind == "uneven":
            return {"E": _exact_uneven(s), "status": None}
        if kind == "serve":
            return {"E": _exact_serve(case, s), "status": None}
        if kind == "surface":
            return {"E": _exact_surface(s), "status": None}
        E, G = _exact_scan(case, s, kind == "gradients")
        if kind == "gradients":
            return {"E": E, "G": G, "status": None}
        if kind == "request":
            return {"qa": _packed(_lab_moments(s["A"], case["lmax"])[0], case["lmax"]),
                    "qb": _packed(_lab_moments(s["B"], case["lmax"])[0], case["lmax"]), "E": float(E[0])}
        return {"E": E, "status": None}
