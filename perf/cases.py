"""Performance cases of the GPU library: the calls its users make, over the sizes they make them at.

A case is a dict of plain values; ``prepare`` builds what a program has in hand
before the call, ``run`` makes one call (or one request) through the package's
public entry points, ``work`` states the bytes and flops the result cannot do
without and ``exact`` recomputes results in 64 bits with torch alone.

Kinds of call (``kind``):
  apply     y = Z x of an assembled operator, vectors on the device
  assemble  fill and factor an operator, blocks copied out to the device
  kbar      the allocation-free Kbar of one object
  solve     GMRES for plane waves on an assembled operator, vectors on the device
  farfield  bistatic RCS of given solutions
  request   assemble + right-hand sides + solve + RCS through host arrays
Shapes (``shape``, size ``n``): "sphere" = icosphere of 20 4^n triangles; "box" =
jittered dielectric box of n x (n - 1) x (n - 3) cells; "wire" = graded copper bar of n x n/5 x n/10
cells in an oxide layer over grounded silicon; "array" / "glass" = n x n dielectric
cylinders of 240 triangles in free space / resting on a glass half-space.
Every mesh, material and frequency varies with the seed by a few per cent.
"""
import math

import numpy as np
import torch

from paper_2106_06184_gb300 import sldm

C0 = 299792458.0
ETA0 = 4e-7 * math.pi * C0
PREC = {"c128": sldm.PREC_F64, "c64": sldm.PREC_F32, "c64x2": sldm.PREC_F32X2}
# relative residual of the solves: the one the GPU tests compare solutions at
TOL = 1e-10


def listed():
    return [
        # the smallest product: a sphere of 80 triangles, one vector (launches and latency)
        dict(name="apply-sphere-fp64", kind="apply", shape="sphere", n=1, prec="c128", nrhs=1),
        # a port or sweep problem of a few excitations in complex128, Y formed by the blocked LU
        dict(name="apply-box-fp64", kind="apply", shape="box", n=9, prec="c128", nrhs=5),
        # the product inside a 32-wave lockstep solve of the 8 x 8 metasurface, complex64 (the largest operator)
        dict(name="apply-array-c64", kind="apply", shape="array", n=8, prec="c64", nrhs=32),
        # the FP64-accurate residual product of a 6 x 6 metasurface's refinement, odd number of waves
        dict(name="apply-array-c64x2", kind="apply", shape="array", n=6, prec="c64x2", nrhs=13),
        # Kbar for a caller that may not allocate
        dict(name="kbar-sphere", kind="kbar", shape="sphere", n=2, prec="c128", nrhs=1),
        # assembly of the plain FP64 sphere (fill, small LU, preconditioner)
        dict(name="assemble-sphere-fp64", kind="assemble", shape="sphere", n=2, prec="c128", nrhs=1),
        # assembly of one point of a complex64 frequency sweep (blocked LU of order 3,199)
        dict(name="assemble-sphere-c64", kind="assemble", shape="sphere", n=3, prec="c64", nrhs=1),
        # assembly of the copper wire in its stack (split fills, tables, reflected fill, inner-solve Y)
        dict(name="assemble-wire-fp64", kind="assemble", shape="wire", n=40, prec="c128", nrhs=1),
        # one plane wave on the FP64 sphere
        dict(name="solve-sphere-fp64", kind="solve", shape="sphere", n=2, prec="c128", nrhs=1),
        # a served batch: 12 plane waves in lockstep on a small catalogue model
        dict(name="solve-sphere-c64x2", kind="solve", shape="sphere", n=2, prec="c64x2", nrhs=12),
        # the metasurface's solve, 32 plane waves in lockstep
        dict(name="solve-array-c64x2", kind="solve", shape="array", n=6, prec="c64x2", nrhs=32),
        # a whole request of the metasurface on glass through host arrays, with the RCS above the glass
        dict(name="request-glass-c64x2", kind="request", shape="glass", n=5, prec="c64x2", nrhs=32),
    ]


def draw(rng):
    kind = rng.choice(["apply", "apply", "assemble", "kbar", "solve", "solve", "farfield", "request"])
    logint = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    nrhs = logint(1, 32)
    if kind == "kbar":
        shape, n = rng.choice([("sphere", 1), ("sphere", 2), ("box", 5), ("box", 6)])
        return dict(kind=kind, shape=shape, n=n, prec="c128", nrhs=1, salt=rng.randrange(1 << 16))
    if kind == "assemble":
        shape = rng.choice(["sphere", "box", "wire", "array"])
        n = {"sphere": rng.randint(1, 3), "box": rng.randint(5, 14), "wire": 10 * rng.randint(1, 3), "array": rng.randint(1, 4)}[shape]
        prec = "c128" if shape == "wire" else rng.choice(["c128", "c64", "c64x2"])
        return dict(kind=kind, shape=shape, n=n, prec=prec, nrhs=1, salt=rng.randrange(1 << 16))
    shape = rng.choice(["sphere", "box", "array", "array"]) if kind != "request" else rng.choice(["sphere", "array", "glass"])
    top = {"apply": 8, "solve": 5, "farfield": 6, "request": 4}[kind]
    n = {"sphere": rng.randint(1, 3), "box": rng.randint(5, 12)}.get(shape) or logint(1, top)
    prec = rng.choice(["c128", "c64", "c64x2"]) if kind in ("apply", "farfield") else rng.choice(["c128", "c64x2"])
    if prec == "c128" and shape in ("array", "glass"):
        n = min(n, 4)
        nrhs = min(nrhs, 8)
    return dict(kind=kind, shape=shape, n=n, prec=prec, nrhs=nrhs, salt=rng.randrange(1 << 16))


# ----------------------------------------------------------------------------- geometry
def _sphere(sub, radii):
    t = (1.0 + 5.0 ** 0.5) / 2.0
    v = np.array([[-1, t, 0], [1, t, 0], [-1, -t, 0], [1, -t, 0], [0, -1, t], [0, 1, t], [0, -1, -t], [0, 1, -t],
                  [t, 0, -1], [t, 0, 1], [-t, 0, -1], [-t, 0, 1]])
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    f = np.array([[0, 11, 5], [0, 5, 1], [0, 1, 7], [0, 7, 10], [0, 10, 11], [1, 5, 9], [5, 11, 4], [11, 10, 2], [10, 7, 6],
                  [7, 1, 8], [3, 9, 4], [3, 4, 2], [3, 2, 6], [3, 6, 8], [3, 8, 9], [4, 9, 5], [2, 4, 11], [6, 2, 10],
                  [8, 6, 7], [9, 8, 1]])
    for _ in range(sub):
        e = np.sort(np.concatenate([f[:, [0, 1]], f[:, [1, 2]], f[:, [2, 0]]]), axis=1)
        u, inv = np.unique(e, axis=0, return_inverse=True)
        mid = v[u[:, 0]] + v[u[:, 1]]
        mid /= np.linalg.norm(mid, axis=1, keepdims=True)
        m = inv.reshape(3, -1) + len(v)
        v = np.concatenate([v, mid])
        a, b, c = f.T
        ab, bc, ca = m
        f = np.concatenate([np.stack(x, 1) for x in ((a, ab, ca), (b, bc, ab), (c, ca, bc), (ab, bc, ca))])
    return v * radii, f


def _box(cells, axes, jitter, rng):
    """Closed box: one structured grid per face on the given axis coordinates, face-interior vertices jittered."""
    ids, xyz, tri = {}, [], []

    def vert(i):
        if i not in ids:
            ids[i] = len(xyz)
            p = np.array([axes[a][i[a]] for a in range(3)])
            rim = [i[a] in (0, cells[a]) for a in range(3)]
            if sum(rim) == 1:
                for a in range(3):
                    if not rim[a]:
                        h = min(axes[a][i[a]] - axes[a][i[a] - 1], axes[a][i[a] + 1] - axes[a][i[a]])
                        p[a] += jitter * h * rng.uniform(-1, 1)
            xyz.append(p)
        return ids[i]

    for a in range(3):
        b, c = (a + 1) % 3, (a + 2) % 3
        for side in (0, cells[a]):
            for i in range(cells[b]):
                for j in range(cells[c]):
                    q = []
                    for di, dj in ((0, 0), (1, 0), (1, 1), (0, 1)):
                        p = [0, 0, 0]
                        p[a], p[b], p[c] = side, i + di, j + dj
                        q.append(vert(tuple(p)))
                    two = ((0, 1, 2), (0, 2, 3)) if (i + j) % 2 == 0 else ((0, 1, 3), (1, 2, 3))
                    for t in two:
                        tri.append([q[k] for k in (t if side else t[::-1])])
    return np.array(xyz), np.array(tri)


def _cylinder(r, h):
    na, ns, m = 20, 4, 10
    ang = 2 * np.pi * np.arange(na) / na
    ang_in = 2 * np.pi * (np.arange(m) + 0.5) / m
    v = [[r * np.cos(a), r * np.sin(a), h * k / ns] for k in range(ns + 1) for a in ang]
    tri = []
    for k in range(ns):
        for i in range(na):
            a, b, c, d = k * na + i, k * na + (i + 1) % na, (k + 1) * na + (i + 1) % na, (k + 1) * na + i
            tri += [(a, b, c), (a, c, d)]
    for z, rim, up in ((h, ns * na, True), (0.0, 0, False)):
        base = len(v)
        v += [[0.5 * r * np.cos(a), 0.5 * r * np.sin(a), z] for a in ang_in] + [[0.0, 0.0, z]]
        for i in range(m):
            i0, i1 = base + (i - 1) % m, base + i
            o = [rim + (2 * i + d) % na for d in range(3)]
            for t in ((base + m, base + i, base + (i + 1) % m), (i0, o[0], o[1]), (i0, o[1], i1), (i1, o[1], o[2])):
                tri.append(t if up else t[::-1])
    return np.array(v), np.array(tri)


def _model(case, seed):
    """Mesh arrays, background, materials and frequency of a case."""
    rng = np.random.default_rng([int(seed), int(case.get("salt", 0)), 7])
    vary = lambda x, p=0.02: x * (1 + p * rng.uniform(-1, 1))  # noqa: E731
    shape, n = case["shape"], case["n"]
    air, objs, z_top, bottom, layer = [(1.0, 1.0, 0.0, 0.0)], None, 0.0, sldm.BOTTOM_HALFSPACE, 0
    if shape == "sphere":
        xyz, tri = _sphere(n, np.array([vary(0.1, 0.1), vary(0.1, 0.1), vary(0.1, 0.1)]))
        mats, freq = [(vary(4.0), 1.0, 0.002)], vary(300e6)
    elif shape == "box":
        cells = (n, n - 1, n - 3)
        xyz, tri = _box(cells, [np.linspace(-0.5, 0.5, c + 1) * vary(L) for c, L in zip(cells, (0.2, 0.18, 0.1))], 0.05, rng)
        mats, freq = [(vary(4.0), 1.0, 0.01)], vary(300e6)
    elif shape == "wire":
        cells = (n, n // 5, n // 10)
        w = 13.76 ** (np.minimum(np.arange(n), np.arange(n)[::-1]) / (n // 2 - 1))
        x = np.concatenate([[0.0], np.cumsum(w)]) / np.sum(w) - 0.5
        axes = [x * 2.5e-6 * n, np.linspace(-0.5, 0.5, cells[1] + 1) * vary(5e-8 * n),
                np.linspace(-0.5, 0.5, cells[2] + 1) * 2.5e-8 * n - 5e-6]
        xyz, tri = _box(cells, axes, 0.01, rng)
        air, bottom, layer = [(1.0, 1.0, 0.0, 0.0), (vary(3.9), 1.0, 0.0, 10e-6), (11.9, 1.0, 10.0, 200e-6)], sldm.BOTTOM_PEC, 1
        mats, freq = [(1.0, 1.0, 5.8e7, layer)], vary(3.0e9)
    else:
        v, f = _cylinder(vary(120e-9), vary(300e-9))
        p = vary(500e-9)
        at = [(p * (i - 0.5 * (n - 1)), p * (j - 0.5 * (n - 1)), 0.0) for j in range(n) for i in range(n)]
        xyz = np.concatenate([v + np.array(a) for a in at])
        tri = np.concatenate([f + k * len(v) for k in range(n * n)])
        objs = np.repeat(np.arange(n * n), len(f))
        mats, freq = [(vary(6.0), 1.0, 0.0, 0)] * (n * n), vary(C0 / 1e-6, 0.01)
        if shape == "glass":
            air = [(1.0, 1.0, 0.0, 0.0), (vary(2.25), 1.0, 0.0, 0.0)]
    # plane waves from above, up to 70 degrees off the normal, TE and TM
    th, ph = rng.uniform(0, 1.2, case["nrhs"]), rng.uniform(0, 2 * np.pi, case["nrhs"])
    khat = np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), -np.cos(th)], 1)
    te, tm = np.stack([-np.sin(ph), np.cos(ph), 0 * ph], 1), np.stack([np.cos(th) * np.cos(ph), np.cos(th) * np.sin(ph), np.sin(th)], 1)
    pol = np.where((np.arange(case["nrhs"]) % 2 == 0)[:, None], te, tm)
    return dict(xyz=xyz, tri=tri, objs=objs, layers=air, z_top=z_top, bottom=bottom, mats=mats, freq=freq, khat=khat, pol=pol,
                layered=len(air) > 1)


def _counts(case):
    """(objects, triangles and edges of one object)."""
    shape, n = case["shape"], case["n"]
    nobj = n * n if shape in ("array", "glass") else 1
    cells = {"box": (n, n - 1, n - 3), "wire": (n, n // 5, n // 10)}.get(shape)
    nt = 4 * (cells[0] * cells[1] + cells[1] * cells[2] + cells[2] * cells[0]) if cells else 20 * 4 ** n if shape == "sphere" else 240
    return nobj, nt, 3 * nt // 2


# ----------------------------------------------------------------------------- the calls
def _block_shapes(case):
    nobj, nt, ne = _counts(case)
    shapes = {sldm.BLOCK_LAM: (nobj * ne,) * 2, sldm.BLOCK_LPM: (nobj * nt,) * 2, sldm.BLOCK_LA: (ne, ne), sldm.BLOCK_LP: (nt, nt),
              sldm.BLOCK_K: (ne, ne), sldm.BLOCK_Y11: (ne, ne), sldm.BLOCK_Y21: (nt - 1, ne)}
    if case["prec"] == "c128" and ne + nt - 1 >= 2500:  # Y is applied by inner solves, not formed
        del shapes[sldm.BLOCK_Y11], shapes[sldm.BLOCK_Y21]
    return shapes


def _ell(s):
    return float(np.linalg.norm(s["xyz"][s["tri"][:, 0]] - s["xyz"][s["tri"][:, 1]], axis=1).mean())


def prepare(case, seed):
    m = _model(case, seed)
    mesh = sldm.Mesh(m["xyz"], m["tri"], m["objs"])
    stack = sldm.Stack(m["layers"], m["z_top"], m["bottom"])
    s = dict(case=case, mesh=mesh, stack=stack, xyz=m["xyz"], tri=m["tri"], mats=m["mats"], freq=m["freq"], khat=m["khat"], pol=m["pol"], prec=PREC[case["prec"]])
    kind, nrhs, N = case["kind"], case["nrhs"], mesh.n_unknowns
    if kind == "kbar":
        s["k"] = 2 * math.pi * m["freq"] / C0 * math.sqrt(m["mats"][0][0]) * (1 - 0.01j)
        s["out"] = torch.empty(mesh.ne, mesh.ne, dtype=torch.complex128, device="cuda")
        return s
    if kind == "assemble":
        s["out"] = {b: torch.empty(d, dtype=torch.complex128, device="cuda") for b, d in _block_shapes(case).items()}
        return s
    th = np.linspace(0, math.radians(89.0), 90) if m["layered"] else np.linspace(0, math.pi, 181)
    s["theta"], s["phi"] = th, np.zeros_like(th)
    if kind == "request":
        s["b"], s["x"] = np.zeros((nrhs, N), complex), np.zeros((nrhs, N), complex)
        return s
    s["op"] = sldm.Operator(mesh, stack, m["mats"], m["freq"], precision=s["prec"])
    s["x"] = torch.zeros(nrhs, N, dtype=torch.complex128, device="cuda")
    if kind == "solve":
        s["b"] = s["op"].rhs_planewave(m["khat"], m["pol"], torch.zeros_like(s["x"]))
    else:
        g = torch.Generator(device="cuda").manual_seed(int(seed))
        s["x"] = torch.randn(s["x"].shape, dtype=torch.complex128, device="cuda", generator=g)
        ell = _ell(s)
        s["x"][:, : mesh.ne] /= ell  # currents, fields and charges of one physical size
        s["x"][:, 2 * mesh.ne:] *= ell
        s["y"] = torch.empty_like(s["x"])
    return s


def _kept(case, t):
    """Results of complex64 operators are kept in complex64, the type they are computed in."""
    return t.to(torch.complex64) if case["prec"] == "c64" else t


def run(s):
    case = s["case"]
    kind, nrhs = case["kind"], case["nrhs"]
    if kind == "apply":
        return _kept(case, s["op"].apply(s["x"], s["y"], nrhs=nrhs))
    if kind == "kbar":
        return s["mesh"].kbar_noalloc(0, s["k"], s["out"])
    if kind == "solve":
        s["op"].solve(s["b"], s["x"], nrhs=nrhs, tol=TOL)
        return _kept(case, s["x"])
    if kind == "farfield":
        rcs = s["op"].farfield_n(s["x"], s["theta"], s["phi"], nrhs)
        return rcs.astype(np.float32) if case["prec"] == "c64" else rcs
    op = sldm.Operator(s["mesh"], s["stack"], s["mats"], s["freq"], precision=s["prec"])
    if kind == "assemble":
        out = [_kept(case, op.block_into(b, t)) for b, t in s["out"].items()]
        op.close()
        return out
    op.rhs_planewave(s["khat"], s["pol"], s["b"])
    op.solve(s["b"], s["x"], nrhs=nrhs, tol=TOL)
    rcs = op.farfield_n(s["x"], s["theta"], s["phi"], nrhs)
    op.close()
    return [s["x"], rcs]


# ----------------------------------------------------------------------------- what the path cannot do without
def work(case):
    nobj, nt, ne = _counts(case)
    n, N, nrhs = ne + nt - 1, nobj * (2 * ne + nt - 1), case["nrhs"]
    es = 8 if case["prec"] == "c64" else 16
    local = 3 * ne * ne + nt * nt + (nt - 1) * ne
    entries = (nobj * ne) ** 2 + (nobj * nt) ** 2 + nobj * local
    vec = 16.0 * N * nrhs
    product = dict(bytes=es * entries + 2 * vec, flops=8.0 * entries * nrhs)
    # distinct blocks of repeated cylinders: one per relative placement
    side = case["n"] if nobj > 1 else 1
    pairs = (2 * side - 1) ** 2 * nt * nt
    # 36 evaluations per pair, ~50 flops each: global L, object L, two Kbar on 6 children
    fill = 36.0 * 50.0 * (pairs + 13 * nt * nt)
    lu = 8.0 * (n ** 3 / 3.0 + float(n) * n * ne) + 8.0 * 4.0 / 3.0 * (nt - 1) ** 3
    if case["kind"] == "apply":
        return product
    if case["kind"] == "kbar":
        return dict(bytes=16.0 * ne * ne, flops=36.0 * 50.0 * 6 * nt * nt)
    if case["kind"] == "assemble":
        return dict(bytes=float(es) * entries, flops=fill + lu)
    angles = 90 if case["shape"] == "glass" else 181
    far = dict(bytes=vec, flops=8.0 * 18 * nobj * nt * angles * nrhs)
    if case["kind"] == "farfield":
        return far
    its = 30 if case["shape"] == "sphere" else 150 if case["shape"] == "box" else 60 * case["n"]  # GMRES steps, roughly
    passes = 0.5 if case["prec"] == "c64x2" else 1.0  # the cycles stream the complex64 part alone
    solve = dict(bytes=its * passes * product["bytes"], flops=its * product["flops"])
    if case["kind"] == "solve":
        return solve
    return dict(bytes=solve["bytes"] + es * entries + far["bytes"], flops=solve["flops"] + fill + lu + far["flops"])


# ----------------------------------------------------------------------------- 64-bit results by torch alone
def _operator(s):
    """Z (Eq. finalsystem) from the operator's stored blocks: a function x -> Z x on complex128 columns, and its pieces."""
    op, mesh = s["op"], s["mesh"]
    dev = dict(dtype=torch.complex128, device="cuda")
    nobj, ne, nt = mesh.nobj, mesh.ne, mesh.nt
    nq = nt - nobj
    eo, to = ne // nobj, nt // nobj
    get = lambda b, r, c, o=0: op.block_into(b, torch.empty(r, c, **dev), obj=o)  # noqa: E731
    LA, LP, IX = get(sldm.BLOCK_LAM, ne, ne), get(sldm.BLOCK_LPM, nt, nt), get(sldm.BLOCK_IX, ne, ne) if ne < 9000 else None
    if IX is None:
        return None
    loc = [{k: get(b, r, c, o) for k, b, r, c in (("A", sldm.BLOCK_LA, eo, eo), ("P", sldm.BLOCK_LP, to, to), ("K", sldm.BLOCK_K, eo, eo),
                                                 ("Y1", sldm.BLOCK_Y11, eo, eo), ("Y2", sldm.BLOCK_Y21, to - 1, eo))} for o in range(nobj)]
    _, tp, tm = mesh.edges()
    D = torch.zeros(nt, ne, **dev)
    e = torch.arange(ne, device="cuda")
    D[torch.from_numpy(tp).cuda(), e] = 1.0
    D[torch.from_numpy(tm).cuda(), e] = -1.0
    keep = torch.tensor([t for t in range(nt) if (t + 1) % to], device="cuda")
    B = torch.zeros(nt, nq, **dev)
    B[keep, torch.arange(nq, device="cuda")] = 1.0
    for o in range(nobj):
        B[(o + 1) * to - 1, o * (to - 1):(o + 1) * (to - 1)] = -1.0
    bd = lambda k: torch.block_diag(*[d[k] for d in loc])  # noqa: E731

    def mul(x):
        j, q, u = x[:ne], x[ne:2 * ne], x[2 * ne:]
        a, c = j - bd("Y1") @ q, u + bd("Y2") @ q
        return torch.cat([LA @ a + D.T @ (LP @ (B @ c)) + IX @ q, bd("A") @ j - bd("K") @ q + D.T @ (bd("P") @ (B @ u)),
                          (D @ a)[keep] + op.k0 ** 2 * c])
    return mul


def exact(case, seed):
    nobj, nt, ne = _counts(case)
    N = nobj * (2 * ne + nt - 1)
    nested = case["prec"] == "c128" and ne + nt - 1 >= 2500
    if case["kind"] in ("kbar", "assemble", "request") or nested or nobj * ne > 9000:
        return None
    if case["kind"] == "solve" and N > 6000:
        return None
    s = prepare(case, seed)
    if case["kind"] == "farfield":
        return _rcs(s, nobj, nt, ne)
    mul = _operator(s)
    if case["kind"] == "apply":
        return mul(s["x"].T).T.contiguous()
    ell = _ell(s)
    d = torch.ones(N, dtype=torch.complex128, device="cuda")
    dr, dc = d.clone(), d.clone()
    dr[2 * s["mesh"].ne:] = ell
    dc[: s["mesh"].ne] = 1 / ell
    dc[2 * s["mesh"].ne:] = ell
    Z = mul(torch.diag(dc)) * dr[:, None]
    b = s["b"].T * dr[:, None]
    x = torch.linalg.solve(Z, b)
    x = x + torch.linalg.solve(Z, b - Z @ x)
    return (x * dc[:, None]).T.contiguous()


def _rcs(s, nobj, nt, ne):
    """RCS of j - Y11 e radiating in free space: 6-point rule of degree 4 on every triangle."""
    mesh, op = s["mesh"], s["op"]
    xyz, tri = torch.from_numpy(s["xyz"]).cuda(), torch.from_numpy(s["tri"]).cuda()
    NE = nobj * ne
    x = s["x"].T
    jd = x[:NE].clone()
    for o in range(nobj):
        Y = op.block_into(sldm.BLOCK_Y11, torch.empty(ne, ne, dtype=torch.complex128, device="cuda"), obj=o)
        jd[o * ne:(o + 1) * ne] -= Y @ x[NE + o * ne: NE + (o + 1) * ne]
    uv, tp, tm = mesh.edges()
    uv = torch.from_numpy(uv).cuda()
    a1, b1, w1, a2, b2, w2 = 0.108103018168070, 0.445948490915965, 0.223381589678011, 0.816847572980459, 0.091576213509771, 0.109951743655322
    bary = torch.tensor([[a1, b1, b1], [b1, a1, b1], [b1, b1, a1], [a2, b2, b2], [b2, a2, b2], [b2, b2, a2]], dtype=torch.float64, device="cuda")
    wq = torch.tensor([w1] * 3 + [w2] * 3, dtype=torch.float64, device="cuda")
    th = torch.from_numpy(s["theta"]).cuda()
    rh = torch.stack([th.sin(), 0 * th, th.cos()], 1)
    F = torch.zeros(len(th), 3, x.shape[1], dtype=torch.complex128, device="cuda")
    for side, t in ((1.0, torch.from_numpy(tp).cuda()), (-1.0, torch.from_numpy(tm).cuda())):
        v = tri[t]
        opp = xyz[(v.sum(1) - uv.sum(1)).long()]  # the vertex opposite the edge
        r = torch.einsum("qv,evd->eqd", bary, xyz[v.long()])
        # f = +-(r - opp)/(2A): the area cancels against the weights
        g = side * 0.5 * wq[None, :, None] * (r - opp[:, None])
        for k0 in range(0, NE, 4096):
            sl = slice(k0, min(NE, k0 + 4096))
            ph = torch.exp(1j * op.k0 * torch.einsum("ad,eqd->aeq", rh, r[sl]))
            F += torch.einsum("aed,er->adr", torch.einsum("aeq,eqd->aed", ph, g[sl].to(torch.complex128)), jd[sl])
    F = F - rh[:, :, None] * (rh[:, :, None] * F).sum(1, keepdim=True)
    return (ETA0 ** 2 * (F.abs() ** 2).sum(1) / (4 * math.pi)).T.contiguous()
