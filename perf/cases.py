"""Performance cases of the solver, through its public entry points.

Each case is one call (or the calls of one step) of a program that uses the
package:

  assemble  the reduced matrix A of one scatterer, its CBFs at hand (assemble_reduced, cbfm_red_export)
  batch     the reduced matrices of a mix of scatterers at once (assemble_reduced_batch)
  solve     currents and RCS of a set of excitations on a CMP-ready reduced system (solve)
  mom       the same on the conventional MoM system in the T-diagonal arrangement (solve, PC_TDIAG)
  step      assemble_reduced, cmp_setup and solve of a scatterer whose CBFs are at hand
  cold      the first answer for a new scatterer: mesh, build_cbfs, then a step

prepare() makes what the program holds before the call; exact() states the
same answer in 64 bits with torch and numpy alone.  Inputs follow the seed:
the geometry is scaled (as a frequency sweep does, since lengths are in
wavelengths) and turned about z, the medium, the directions of the waves and
the stand-in CBFs vary.

Results of the mixed-precision path come back in the type they were computed
in: A is held as complex64 (its export widens it), the currents and the RCS are
formed in FP32 (solve widens them), so a program keeps them as complex64 and
float32.  FP64 results stay complex128 and float64.
"""
import ctypes
import math

import numpy as np
import torch

import paper_2111_11058_gb300 as P

ETA0 = 376.730313668
K0 = 2.0 * math.pi
ALPHA = 2.0            # near-pair factor (the default of mesh())
DELTA_SVD = 1e-3       # relative size of the smallest kept singular value


# ------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest assembly in use: the 960-unknown sphere, where launches and latency count
        dict(name="assemble_sphere960", path="assemble", shape="sphere", a=2, size=0.3, eps_re=4.0, eps_im=0.0,
             ncell=8, L=14, prec="mixed"),
        # the benchmark's assembly: cube of one wavelength, 9216 unknowns
        dict(name="assemble_cube9216", path="assemble", shape="cube", a=16, size=1.0, eps_re=2.5, eps_im=0.0,
             ncell=32, L=14, prec="mixed"),
        # a large lossy body whose RWG matrices are not formed in memory (the fused form)
        dict(name="assemble_spheroid32400", path="assemble", shape="spheroid", a=60, b=90, size=1.2, eps_re=3.0,
             eps_im=-0.1, ncell=96, L=8, prec="mixed"),
        # the reference-precision assembly at the size of the serving scatterers
        dict(name="assemble_cube2304_fp64", path="assemble", shape="cube", a=8, size=1.0, eps_re=2.5, eps_im=0.0,
             ncell=16, L=16, prec="fp64"),
        # many small uneven scatterers in one call (parameter studies)
        dict(name="batch_mix40", path="batch", count=40, L=16),
        # one excitation of a small sphere with a bistatic cut: the shortest solve
        dict(name="solve_sphere960_fp64", path="solve", shape="sphere", a=2, size=0.3, eps_re=4.0, eps_im=0.0, ncell=8,
             waves=12, lmax=0, prec="fp64", solver="per_rhs", nrhs=1, obs=362, tol=1e-6),
        # the benchmark's solve: 128 monostatic excitations, block GMRES with the CMP
        dict(name="solve_cube9216", path="solve", shape="cube", a=16, size=1.0, eps_re=2.5, eps_im=0.0, ncell=32,
             waves=64, lmax=0, prec="mixed", solver="block", nrhs=128, obs=0, tol=1e-6),
        # a lossy spheroid with more excitations than one block takes (a ragged second block)
        dict(name="solve_spheroid16200", path="solve", shape="spheroid", a=45, b=60, size=1.0, eps_re=3.0, eps_im=-0.1,
             ncell=64, waves=64, lmax=0, prec="mixed", solver="block", nrhs=200, obs=0, tol=1e-6),
        # the reference-precision block solve, tight tolerance, an odd number of excitations
        dict(name="solve_cube2304_fp64", path="solve", shape="cube", a=8, size=1.0, eps_re=2.5, eps_im=0.0, ncell=16,
             waves=64, lmax=0, prec="fp64", solver="block", nrhs=45, obs=0, tol=1e-8),
        # the conventional MoM the method is compared with: per-excitation GMRES, Jacobi-scaled T-diagonal system
        dict(name="mom_cube2304", path="mom", shape="cube", a=8, size=1.0, eps_re=2.5, eps_im=0.0, ncell=16,
             prec="mixed", nrhs=32, tol=1e-6),
        # the whole benchmark step
        dict(name="step_cube9216", path="step", shape="cube", a=16, size=1.0, eps_re=2.5, eps_im=0.0, ncell=32,
             waves=64, lmax=0, prec="mixed", solver="block", nrhs=128, obs=0, tol=1e-6),
        # a serving request that misses the cache: CBF generation, assembly and solve of a finite cylinder for a few
        # excitations, so the block solve takes many small block iterations
        dict(name="cold_cylinder2352", path="cold", shape="cylinder", a=28, b=10, c=2, size=0.8, eps_re=3.0, eps_im=0.0,
             ncell=16, waves=64, lmax=0, prec="mixed", solver="block", nrhs=7, obs=0, tol=1e-6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shape(rng, lo, hi, cell=180):
    """A body with lo..hi triangles (log-uniform), its size and cells of 40 to `cell` RWG functions."""
    nt = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    kind = rng.choice(("cube", "cylinder", "spheroid", "sphere"))
    d = dict(shape=kind, size=rng.uniform(0.2, 1.2), eps_re=rng.uniform(1.5, 6.0),
             eps_im=rng.choice((0.0, -0.1, -rng.uniform(0.01, 0.5))))
    if kind == "sphere":
        d["a"] = 2 if nt < 640 or hi < 1280 else 3
        d["size"] *= 0.5
    elif kind == "cube":
        d["a"] = max(3, int(math.sqrt(nt / 12.0)))
    elif kind == "cylinder":
        q = max(3.0, math.sqrt(nt / 6.0))
        d["a"] = max(7, int(1.5 * q))
        d["c"] = rng.choice((1, 2, 3))
        d["b"] = max(2, int(nt / (2.0 * d["a"])) - 2 * d["c"] + 1)
    else:
        q = max(3.0, math.sqrt(nt / 3.0))
        d["a"] = max(3, int(q))
        d["b"] = max(7, int(nt / (2.0 * d["a"])))
        d["size"] *= 0.8
    ne = 3 * _count(d) // 2
    # the electrical size follows the resolution: at least ~8 edges per wavelength in the medium
    d["size"] = min(d["size"], max(0.2, math.sqrt(ne) / 60.0))
    d["ncell"] = max(2, int(math.ceil(ne / rng.uniform(40, cell))))
    return d


def draw(rng):
    path = rng.choice(("assemble", "assemble", "solve", "solve", "solve", "batch", "mom", "step", "cold"))
    if path == "batch":
        return dict(path=path, count=rng.randint(2, 40), L=rng.randint(5, 16))
    if path == "assemble":
        prec = rng.choice(("mixed", "mixed", "mixed", "fused", "unfused", "fp64"))
        d = _shape(rng, 200, {"fp64": 1200, "fused": 4000}.get(prec, 4000))
        d.update(path=path, L=rng.randint(4, 18), prec=prec)
        return d
    if path == "mom":
        prec = rng.choice(("mixed", "fp64"))
        d = _shape(rng, 200, 500 if prec == "mixed" else 330)
        d.update(path=path, prec=prec, nrhs=_log_int(rng, 1, 12 if prec == "mixed" else 3), tol=1e-6)
        return d
    prec = rng.choice(("mixed", "mixed", "fp64"))
    solver = rng.choice(("block", "block", "per_rhs"))
    small = prec == "fp64" or path == "cold" or solver == "per_rhs"
    d = _shape(rng, 300, 1000 if small else 3000, 120 if path == "cold" else 180)
    d.update(path=path, waves=rng.choice((12, 24, 33, 64)), lmax=rng.choice((0, 0, 10)), prec=prec, solver=solver,
             nrhs=_log_int(rng, 5, 128) if solver == "block" else _log_int(rng, 1, 6), obs=rng.choice((0, 0, 181)),
             tol=1e-6 if prec == "mixed" else rng.choice((1e-6, 1e-8)))
    return d


# ----------------------------------------------------------------- meshes
def _count(c):
    """Triangles of a case's body."""
    k = c["shape"]
    if k == "sphere":
        return 20 * 4 ** c["a"]
    if k == "cube":
        return 12 * c["a"] ** 2
    if k == "cylinder":
        return 2 * c["a"] * c["b"] + 2 * c["a"] * (2 * c["c"] - 1)
    return 2 * c["a"] * c["b"]


def _rings(rings, n):
    """Triangles of a closed surface of latitude rings between two poles: vertex 0, rings * n vertices, last vertex."""
    t = []
    at = lambda r, p: 1 + r * n + p % n  # noqa: E731
    for p in range(n):
        t.append((0, at(0, p), at(0, p + 1)))
        t.append((1 + rings * n, at(rings - 1, p + 1), at(rings - 1, p)))
        for r in range(rings - 1):
            t.append((at(r, p), at(r + 1, p), at(r + 1, p + 1)))
            t.append((at(r, p), at(r + 1, p + 1), at(r, p + 1)))
    return np.array(t, np.int64)


def _revolve(rho, z, n):
    """Body of revolution through the meridian points (rho, z); the first and the last lie on the axis."""
    ph = 2.0 * np.pi * np.arange(n) / n
    v = [np.array([[0.0, 0.0, z[0]]])]
    for r, h in zip(rho[1:-1], z[1:-1]):
        v.append(np.stack([r * np.cos(ph), r * np.sin(ph), np.full(n, h)], 1))
    v.append(np.array([[0.0, 0.0, z[-1]]]))
    return np.concatenate(v), _rings(len(rho) - 2, n)


def _cube(n):
    ids, v, t = {}, [], []

    def vid(*p):
        if p not in ids:
            ids[p] = len(v)
            v.append(p)
        return ids[p]

    for ax in range(3):
        u, w = [x for x in range(3) if x != ax]
        for side in (0, n):
            for i in range(n):
                for j in range(n):
                    q = []
                    for di, dj in ((0, 0), (1, 0), (1, 1), (0, 1)):
                        p = [0, 0, 0]
                        p[ax], p[u], p[w] = side, i + di, j + dj
                        q.append(vid(*p))
                    t += [(q[0], q[1], q[2]), (q[0], q[2], q[3])]
    return np.array(v, np.float64) / n - 0.5, np.array(t, np.int64)


def _icosphere(level):
    g = (1.0 + math.sqrt(5.0)) / 2.0
    v = np.array([(-1, g, 0), (1, g, 0), (-1, -g, 0), (1, -g, 0), (0, -1, g), (0, 1, g), (0, -1, -g), (0, 1, -g),
                  (g, 0, -1), (g, 0, 1), (-g, 0, -1), (-g, 0, 1)])
    d = np.linalg.norm(v[:, None] - v[None], axis=2)
    near = np.abs(d - 2.0) < 1e-9
    t = np.array([(i, j, k) for i in range(12) for j in range(i + 1, 12) for k in range(j + 1, 12)
                  if near[i, j] and near[j, k] and near[i, k]])
    v = v / np.linalg.norm(v, axis=1)[:, None]
    for _ in range(level):
        e = np.sort(np.concatenate([t[:, [0, 1]], t[:, [1, 2]], t[:, [2, 0]]]), axis=1)
        uniq, inv = np.unique(e, axis=0, return_inverse=True)
        inv = inv.reshape(-1)
        m = v[uniq[:, 0]] + v[uniq[:, 1]]
        a, b, c = (inv[i * len(t):(i + 1) * len(t)] + len(v) for i in range(3))
        v = np.concatenate([v, m / np.linalg.norm(m, axis=1)[:, None]])
        t = np.concatenate([np.stack(x, 1) for x in ((t[:, 0], a, c), (t[:, 1], b, a), (t[:, 2], c, b), (a, b, c))])
    return v, t


def _body(c, rng):
    """(verts, tris) of a case's body: outward triangles, scaled and turned about z by the seed."""
    k, size = c["shape"], c["size"]
    if k == "sphere":
        v, t = _icosphere(c["a"])
        v = v * size
    elif k == "cube":
        v, t = _cube(c["a"])
        v = v * size
    elif k == "cylinder":
        cap = np.arange(c["c"] + 1) / c["c"] * 0.4
        side = np.linspace(0.5, -0.5, c["b"] + 1)
        v, t = _revolve(np.concatenate([cap, np.full(c["b"] - 1, 0.4), cap[::-1]]),
                        np.concatenate([np.full(c["c"] + 1, 0.5), side[1:-1], np.full(c["c"] + 1, -0.5)]), c["a"])
        v = v * size
    else:
        s = np.linspace(0.0, np.pi, c["a"] + 2)
        v, t = _revolve(0.4 * size * np.sin(s), size * np.cos(s), c["b"])
    a, b, d = v[t[:, 0]], v[t[:, 1]], v[t[:, 2]]
    flip = np.einsum("ij,ij->i", np.cross(b - a, d - a), a + b + d) < 0
    t[flip] = t[flip][:, [0, 2, 1]]
    # a cube stays aligned with the axes, as its cells are in the benchmark
    f, turn = rng.uniform(0.95, 1.05), 0.0 if k == "cube" else rng.uniform(0.0, 2.0 * np.pi)
    rot = np.array([[math.cos(turn), -math.sin(turn), 0.0], [math.sin(turn), math.cos(turn), 0.0], [0.0, 0.0, 1.0]])
    return np.ascontiguousarray(f * v @ rot.T), np.ascontiguousarray(t, np.int32)


def _waves(n, rng):
    """n directions of a Fibonacci lattice, turned about z by the seed, each with both polarisations."""
    i = np.arange(n)
    th = np.arccos(1.0 - (2.0 * i + 1.0) / n)
    ph = np.mod(i * math.pi * (3.0 - math.sqrt(5.0)) + rng.uniform(0.0, 2.0 * math.pi), 2.0 * math.pi)
    return np.stack([np.repeat(th, 2), np.repeat(ph, 2), np.tile([0.0, math.pi / 2], n)], 1)


def _mix(c):
    """A batch's scatterers: spheres, cubes and finite cylinders of 500 to 6000 unknowns, cells of about 200 RWGs."""
    rng = _rng(c["count"], 1)
    out = []
    for _ in range(c["count"]):
        k = int(rng.integers(0, 3))
        d = dict(size=float(rng.uniform(0.2, 1.2)), eps_re=float(rng.uniform(1.5, 6.0)), eps_im=0.0, L=c["L"])
        if k == 0:
            d.update(shape="sphere", a=int(rng.integers(2, 4)), size=0.5 * d["size"])
        elif k == 1:
            d.update(shape="cube", a=int(rng.integers(4, 13)))
        else:
            d.update(shape="cylinder", a=int(rng.integers(10, 25)), b=int(rng.integers(3, 10)), c=2)
        d["ncell"] = max(2, 3 * _count(d) // 2 // 200)
        out.append(d)
    return out


# -------------------------------------------------- inputs, prepare and run
def _rng(seed, stream):
    return np.random.default_rng([int(seed), stream])


def _inputs(c, seed, part=0):
    """The host inputs of one scatterer: (verts, tris, eps_r)."""
    rng = _rng(seed, 100 + part)
    v, t = _body(c, rng)
    return v, t, complex(c["eps_re"] * rng.uniform(0.97, 1.03), c["eps_im"])


def _stand_in(cell, ncell, L, seed, part=0):
    """Seeded Gaussian blocks in the place of C^M and C^J (the assembly is linear in both)."""
    rng = _rng(seed, 5000 + part)
    cm, cj = [], []
    for n in np.bincount(cell, minlength=ncell):
        k = min(int(n), L)
        for out in (cm, cj):
            out.append((rng.standard_normal((n, k)) + 1j * rng.standard_normal((n, k))) / math.sqrt(2.0 * n))
    return cm, cj


def _excitations(c, seed):
    n = (c["nrhs"] + 1) // 2
    return _waves(n, _rng(seed, 3))[:c["nrhs"]]


def _observe(c):
    """A bistatic cut over theta in the planes phi = 0 and 90 degrees, or None (monostatic)."""
    if not c.get("obs"):
        return None
    th = np.linspace(0.0, np.pi, (c["obs"] + 1) // 2)
    return np.concatenate([np.stack([th, np.full_like(th, p)], 1) for p in (0.0, np.pi / 2)])[:c["obs"]]


_PREC = {"mixed": P.MIXED, "fp64": P.FP64, "fused": P.MIXED_FUSED, "unfused": P.MIXED_UNFUSED}


def _mesh(c, v, t, eps):
    return P.mesh(v, t, c["ncell"], eps, partition="rcb")


def prepare(case, seed):
    c = case
    torch.cuda.init()
    if c["path"] == "batch":
        meshes, cbfs, outs = [], [], []
        for k, d in enumerate(_mix(c)):
            m = _mesh(d, *_inputs(d, seed, k))
            b = P.cbf_import(m, *_stand_in(m.cells(), d["ncell"], d["L"], seed, k))
            meshes.append(m)
            cbfs.append(b)
            outs.append(torch.empty((2 * int(b.L.sum()),) * 2, dtype=torch.complex128, device="cuda"))
        return dict(case=c, meshes=meshes, cbfs=cbfs, A=outs)
    v, t, eps = _inputs(c, seed)
    if c["path"] == "cold":
        s = dict(case=c, body=(v, t, eps), gen=_waves(c["waves"], _rng(seed, 2)))
    else:
        s = dict(case=c, mesh=_mesh(c, v, t, eps))
    if c["path"] == "assemble":
        s["cbf"] = P.cbf_import(s["mesh"], *_stand_in(s["mesh"].cells(), c["ncell"], c["L"], seed))
        s["A"] = torch.empty((2 * int(s["cbf"].L.sum()),) * 2, dtype=torch.complex128, device="cuda")
        return s
    exc, obs = _excitations(c, seed), _observe(c)
    s["exc"] = torch.from_numpy(exc).cuda()
    s["obs"] = None if obs is None else torch.from_numpy(obs).cuda()
    ne = 3 * t.shape[0] // 2
    s["j"] = torch.empty((2 * ne, c["nrhs"]), dtype=torch.complex128, device="cuda")
    s["rcs"] = torch.empty((c["nrhs"], 1 if obs is None else len(obs), 2), dtype=torch.float64, device="cuda")
    if c["path"] == "mom":
        s["red"] = P.assemble_mom(s["mesh"], _PREC[c["prec"]])
        P.tdiag_setup(s["red"], jacobi=True)
    elif c["path"] in ("solve", "step"):
        s["cbf"] = P.build_cbfs(s["mesh"], _waves(c["waves"], _rng(seed, 2)), DELTA_SVD, c["lmax"])
        if c["path"] == "solve":
            s["red"] = P.assemble_reduced(s["mesh"], s["cbf"], _PREC[c["prec"]])
            P.cmp_setup(s["red"])
    return s


def _export(red, out):
    st = P.cbfm.lib().cbfm_red_export(red.handle, ctypes.c_void_p(out.data_ptr()),
                                      ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    if st:
        raise P.CbfmError(st, "cbfm_red_export")
    return out


def _solve(s, red):
    c = s["case"]
    mono = s["obs"] is None
    kw = dict(tol=c["tol"], obs=s["obs"], monostatic=mono, out_j=s["j"], out_rcs=s["rcs"])
    if c["path"] == "mom":
        P.solve(red, s["exc"], restart=200, maxit=4000, solver=P.PER_RHS, precond=P.PC_TDIAG, **kw)
    else:
        # the basis may reach the order of the system, so a block solve saturates instead of restarting
        block = c["solver"] == "block"
        P.solve(red, s["exc"], restart=red.n + 256 if block else 1000, solver=P.BLOCK if block else P.PER_RHS, **kw)
    if c["prec"] == "fp64":
        return [s["j"], s["rcs"]]
    return [s["j"].to(torch.complex64), s["rcs"].float()]


def run(state):
    s, c = state, state["case"]
    if c["path"] == "batch":
        reds = P.assemble_reduced_batch(s["meshes"], s["cbfs"], P.MIXED)
        return [_export(r, a).to(torch.complex64) for r, a in zip(reds, s["A"])]
    if c["path"] == "assemble":
        a = _export(P.assemble_reduced(s["mesh"], s["cbf"], _PREC[c["prec"]]), s["A"])
        return a if c["prec"] == "fp64" else a.to(torch.complex64)
    if c["path"] in ("solve", "mom"):
        return _solve(s, s["red"])
    if c["path"] == "cold":
        mesh = _mesh(c, *s["body"])
        cbf = P.build_cbfs(mesh, s["gen"], DELTA_SVD, c["lmax"])
    else:
        mesh, cbf = s["mesh"], s["cbf"]
    red = P.assemble_reduced(mesh, cbf, _PREC[c["prec"]])
    P.cmp_setup(red)
    out = _solve(s, red)
    if c["path"] == "cold":
        out += [np.array(cbf.L), torch.from_numpy(cbf.sigma)]
    return out


# ------------------------------------------------------------------- work
def _work_assemble(nt, ncell, L, wide):
    """Half of the triangle pairs (L(s, t) is the transpose of L(t, s)), 49 point pairs of about 170 operations each
    for both media, and the projection of three ne x ne operators on the CBFs; each triangle's record and
    each CBF read once, A written once."""
    ne, nh = 1.5 * nt, ncell * L
    flops = 0.5 * nt * nt * 49 * 170 + 8.0 * 4 * (ne * ne * L + ne * L * nh)
    return 48 * 4 * wide * nt + 2 * 8 * wide * ne * L + 8 * wide * (2.0 * nh) ** 2, flops


def _work_solve(ne, n, nrhs, ndir, wide):
    """One factorisation-sized piece of work on the n x n system (8 n^3 / 3), the products for every right-hand side,
    excitations and far field by the 7-point rule; A and the CBFs read once, currents and RCS written once."""
    flops = 8.0 * n ** 3 / 3 + 8.0 * n * n * nrhs + 14.0 / 3 * ne * nrhs * (60 + 60 * ndir) + 32.0 * ne * nrhs * 8
    return 8.0 * wide * n * n + 16.0 * 2 * ne * nrhs + 16.0 * nrhs * ndir, flops


def work(case):
    c = case
    if c["path"] == "batch":   # the mix averages about 1100 triangles
        b, f = _work_assemble(1100, 8, c["L"], 1)
        return dict(bytes=b * c["count"], flops=f * c["count"])
    nt, wide = _count(c), 2 if c.get("prec") == "fp64" else 1
    ne = 3 * nt // 2
    b = f = 0.0
    L = c.get("L") or min(14, c.get("lmax") or 14)
    if c["path"] in ("assemble", "step", "cold"):
        b, f = _work_assemble(nt, c["ncell"], L, wide)
    if c["path"] != "assemble":
        n = 2 * ne if c["path"] == "mom" else 2 * c["ncell"] * L
        # an iterative solution of the conventional system needs its products alone: 200 per right-hand side
        w = _work_solve(ne, n, c["nrhs"], max(1, c.get("obs") or 1), wide)
        b, f = b + w[0], f + (8.0 * n * n * c["nrhs"] * 200 if c["path"] == "mom" else w[1])
    if c["path"] == "cold":    # per cell: the solution of its system for the generating waves, and the SVD
        nm, s = 2.0 * ne / c["ncell"], 2.0 * c["waves"]
        f += c["ncell"] * (8.0 * nm ** 3 / 3 + 8.0 * nm * nm * s + 8.0 * 20 * s ** 3)
        b += 16.0 * 2 * ne * s
    return dict(bytes=float(b), flops=float(f))


# ------------------------------------------------- the same in 64 bits
class _Geo:
    """RWG functions of a closed surface: edges (u < v) in lexicographic order, the plus triangle runs u -> v."""

    def __init__(self, v, t, dev):
        t = t.astype(np.int64)
        nt = len(t)
        u, w = t[:, [1, 2, 0]], t[:, [2, 0, 1]]          # local edge a joins vertices a+1 and a+2
        pairs = np.stack([np.minimum(u, w).ravel(), np.maximum(u, w).ravel()], 1)
        edges, inv = np.unique(pairs, axis=0, return_inverse=True)
        inv = inv.reshape(-1)
        plus = (u < w).ravel()
        self.ne, self.nt = len(edges), nt
        half = np.empty((self.ne, 2), np.int64)          # (triangle, local edge) index of both halves
        half[inv[plus], 0] = np.nonzero(plus)[0]
        half[inv[~plus], 1] = np.nonzero(~plus)[0]
        self.mid = 0.5 * (v[edges[:, 0]] + v[edges[:, 1]])
        length = np.linalg.norm(v[edges[:, 1]] - v[edges[:, 0]], axis=1)
        p = v[t]
        nrm = np.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0])
        area2 = np.linalg.norm(nrm, axis=1)
        s = math.sqrt(15.0)
        b1, b2 = (6 - s) / 21, (6 + s) / 21
        bary = np.array([[1 / 3] * 3] + [[1 - 2 * b if i == a else b for a in range(3)] for b in (b1, b2) for i in range(3)])
        wq = np.array([9 / 40] + [(155 - s) / 1200] * 3 + [(155 + s) / 1200] * 3)
        T = lambda x: torch.as_tensor(np.ascontiguousarray(x), device=dev)  # noqa: E731
        self.half, self.tri_edge, self.tris = T(half), T(inv.reshape(nt, 3)), T(t)
        self.p, self.n = T(p), T(nrm / area2[:, None])
        self.q = T(np.einsum("ka,tax->tkx", bary, p))
        self.wt = T(0.5 * area2[:, None] * wq)
        coef = np.where(plus, 1.0, -1.0).reshape(nt, 3) * length[inv].reshape(nt, 3) / area2[:, None]
        # the functions at the points of each triangle: f[t, point, a] = c_a (r - p_a)
        self.c = T(coef)
        self.f = self.c[:, None, :, None] * (self.q[:, :, None, :] - self.p[:, None, :, :])
        self.cen = self.p.mean(1)
        self.h = torch.linalg.norm(self.p - self.p[:, [1, 2, 0]], dim=2).max(1).values

    def gather(self, x, dim):
        """Half functions -> RWG functions along dim (3 nt -> ne)."""
        return x.index_select(dim, self.half[:, 0]) + x.index_select(dim, self.half[:, 1])


def _rcb(mid, ncell):
    """Recursive coordinate bisection of the edge midpoints (longest axis, ties by edge index)."""
    cell = np.zeros(len(mid), np.int64)

    def cut(ids, first, m):
        if m == 1:
            cell[ids] = first
            return
        x = mid[ids]
        ax = int(np.argmax(x.max(0) - x.min(0)))
        ids = ids[np.lexsort((ids, x[:, ax]))]
        k = int(math.floor(len(ids) * (m // 2) / m + 0.5))
        cut(ids[:k], first, m // 2)
        cut(ids[k:], first + m // 2, m - m // 2)

    cut(np.arange(len(mid)), 0, ncell)
    return cell


def _media(eps):
    n2 = complex(np.sqrt(complex(eps)))
    return ((K0 + 0j, ETA0), (K0 * n2, ETA0 / n2))


def _exp(k, R):
    """e^{-jkR} of a real R."""
    a = torch.exp(k.imag * R) if k.imag else torch.ones_like(R)
    return torch.complex(a * torch.cos(k.real * R), -a * torch.sin(k.real * R))


def _local(U, kern, W):
    """sum over points and components of U[t,p,a,x] kern[t,p,s,q] W[s,q,b,x] -> [t,a,s,b] (kern complex)."""
    t, p, s, q = kern.shape
    x = U.shape[3]
    out = []
    for part in (kern.real, kern.imag):
        y = torch.bmm(part.permute(2, 0, 1, 3).reshape(s, t * p, q), W.reshape(s, q, 3 * x))        # [s, tp, bx]
        y = y.reshape(s, t, p, 3, x).permute(1, 2, 4, 0, 3).reshape(t, p * x, s * 3)
        out.append(torch.bmm(U.permute(0, 2, 1, 3).reshape(t, 3, p * x), y))
    return torch.complex(out[0], out[1]).reshape(t, 3, s, 3)


def _near_list(g, chunk=512):
    t, s = [], []
    for t0 in range(0, g.nt, chunk):
        sl = slice(t0, min(g.nt, t0 + chunk))
        near = torch.linalg.norm(g.cen[sl, None] - g.cen[None], dim=2) < ALPHA * torch.maximum(g.h[sl, None], g.h[None])
        near |= (g.tris[sl, None, :, None] == g.tris[None, :, None, :]).any(3).any(2)
        i, j = torch.nonzero(near, as_tuple=True)
        t.append(i + t0)
        s.append(j)
    return torch.cat(t), torch.cat(s)


def _potentials(V, n, r):
    """Closed forms over triangles V [k,3,3] (normals n) at points r [k,p,3]: int 1/R, int (r'-r)/R, int (r-r')/R^3."""
    d = torch.einsum("kx,kpx->kp", n, r - V[:, None, 0])
    rho = r - d[..., None] * n[:, None]
    i1, beta_s = torch.zeros_like(d), torch.zeros_like(d)
    vr, vf = torch.zeros_like(r), torch.zeros_like(r)
    tiny = 1e-28 * torch.linalg.norm(torch.linalg.cross(V[:, 1] - V[:, 0], V[:, 2] - V[:, 0]), dim=1)[:, None]
    for i in range(3):
        A, B = V[:, i], V[:, (i + 1) % 3]
        l = (B - A) / torch.linalg.norm(B - A, dim=1, keepdim=True)
        u = torch.linalg.cross(l, n)
        dot = lambda a, b: torch.einsum("kpx,kx->kp", a, b)  # noqa: E731
        t0, lp, lm = dot(A[:, None] - rho, u), dot(B[:, None] - rho, l), dot(A[:, None] - rho, l)
        R02 = t0 * t0 + d * d
        Rp, Rm = torch.linalg.norm(r - B[:, None], dim=2), torch.linalg.norm(r - A[:, None], dim=2)
        lg = lambda x, R: torch.where(x >= 0, torch.log(R + x), torch.log(R02 / (R - x)))  # noqa: E731
        F = torch.where(R02 > tiny, lg(lp, Rp) - lg(lm, Rm), torch.zeros_like(d))
        ad = d.abs()
        beta = torch.where(ad > 0, torch.atan(t0 * lp / (R02 + ad * Rp)) - torch.atan(t0 * lm / (R02 + ad * Rm)),
                           torch.zeros_like(d))
        i1 += t0 * F
        beta_s += beta
        vr += (0.5 * (R02 * F + lp * Rp - lm * Rm))[..., None] * u[:, None]
        vf += F[..., None] * u[:, None]
    i1 = i1 - d.abs() * beta_s
    return i1, vr - (d * i1)[..., None] * n[:, None], vf + (torch.sign(d) * beta_s)[..., None] * n[:, None]


def _smooth(k, R):
    """(e^{-jkR} - 1)/(4 pi R) and g + 1/(4 pi R^3) + k^2/(8 pi R), by their series for small kR."""
    x = 1j * k * R
    small = x.abs() < 0.5
    Rs = torch.where(small, torch.ones_like(R), R)
    e = _exp(k, R)
    G = (e - 1.0) / (4 * math.pi * Rs)
    h = -(1.0 + x) * e / (4 * math.pi * Rs ** 3) + 1.0 / (4 * math.pi * Rs ** 3) + k * k / (8 * math.pi * Rs)
    sg, sh, pw = torch.zeros_like(x), torch.zeros_like(x), torch.ones_like(x)
    for m in range(0, 24):     # pw = x^m
        sg = sg + pw * ((-1.0) ** m / math.factorial(m + 1))
        sh = sh + pw * ((-1.0) ** (m + 3) * (1.0 - (m + 3)) / math.factorial(m + 3))
        pw = pw * x
    return (torch.where(small, -1j * k * sg / (4 * math.pi), G),
            torch.where(small, -((1j * k) ** 3) * sh / (4 * math.pi), h))


def _near_blocks(g, t, s, k):
    """Local blocks K, T [pair, 3, 3] of the (ordered) near pairs with the singular parts in closed form."""
    r = g.q[t]                                                           # [n, 7, 3]
    I1, Iv, I3 = _potentials(g.p[s], g.n[s], r)
    d = r[:, :, None] - g.q[s][:, None]                                  # [n, 7, 7, 3]
    G, h = _smooth(k, torch.linalg.norm(d, dim=3))
    w = g.wt[s][:, None]
    S0 = I1 / (4 * math.pi) + (w * G).sum(2)
    Sr = Iv / (4 * math.pi) - torch.einsum("npq,npqx->npx", w * G, d.to(G.dtype))
    W = (-I3 + 0.5 * k * k * Iv) / (4 * math.pi) + torch.einsum("npq,npqx->npx", w * h, d.to(h.dtype))
    ta, cb = g.f[t].to(G.dtype), g.c[s]
    rb = (cb[:, None, :, None] * (r[:, :, None] - g.p[s][:, None])).to(G.dtype)    # c_b (r - p_b)
    wt = g.wt[t].to(G.dtype)
    cc = (2 * g.c[t])[:, :, None] * (2 * cb)[:, None]                    # product of the divergences
    Sb = cb[:, None, :, None] * Sr[:, :, None] + rb * S0[..., None, None]
    T = -1j * k * (torch.einsum("np,npax,npbx->nab", wt, ta, Sb) - cc / (k * k) * (wt * S0).sum(1)[:, None, None])
    K = torch.einsum("np,npax,npbx->nab", wt, ta, torch.linalg.cross(W[:, :, None].expand_as(rb), rb))
    K[t == s] = 0
    return K, T


def _rwg(g, eps, chunk_bytes=6e8):
    """The RWG blocks Ks = K1 + K2, Ta = -(eta1 T1 + eta2 T2), Tb = T1/eta1 + T2/eta2 (ne x ne)."""
    dev = g.q.device
    Z = torch.zeros((3, g.ne, g.ne), dtype=torch.complex128, device=dev)
    nt_, ns_ = _near_list(g)
    media = _media(eps)
    scale = [(1.0, -eta, 1.0 / eta) for _, eta in media]
    near = torch.zeros((3, len(nt_), 3, 3), dtype=torch.complex128, device=dev)
    for (k, _), sc in zip(media, scale):
        for i in range(0, len(nt_), 100000):
            a, b = nt_[i:i + 100000], ns_[i:i + 100000]
            K1, T1 = _near_blocks(g, a, b, k)
            K2, T2 = _near_blocks(g, b, a, k)
            K, T = 0.5 * (K1 + K2.transpose(1, 2)), 0.5 * (T1 + T2.transpose(1, 2))
            for o, x in enumerate((K, T, T)):
                near[o, i:i + 100000] += sc[o] * x
    # components: T couples f_a . f_b and the divergences; (r - p_a) . ((r - r') x (r' - p_b)) splits into
    # (f_a x r) . f_b + f_a . (r' x c_b p_b)
    pc = g.c[:, None, :, None] * g.p[:, None]
    Ut, div = g.f, (2 * g.c)[:, None, :, None].expand(-1, 7, -1, 1)
    Uk = torch.cat([torch.linalg.cross(g.f, g.q[:, :, None].expand_as(g.f)), g.f], 3)
    Wk = torch.cat([g.f, torch.linalg.cross(g.q[:, :, None].expand_as(g.f), pc.expand_as(g.f))], 3)
    wU = g.wt[:, :, None, None]
    step = max(1, int(chunk_bytes / (49 * 16 * g.nt)))
    for t0 in range(0, g.nt, step):
        t1 = min(g.nt, t0 + step)
        sl = slice(t0, t1)
        d = g.q[sl, :, None, None] - g.q[None, None]
        R = torch.linalg.norm(d, dim=4)
        del d
        sel = (nt_ >= t0) & (nt_ < t1)
        a, b = nt_[sel] - t0, ns_[sel]
        R.permute(0, 2, 1, 3)[a, b] = 1.0         # near pairs are replaced below
        L = torch.zeros((3, t1 - t0, 3, g.nt, 3), dtype=torch.complex128, device=dev)
        for (k, _), sc in zip(media, scale):
            G = _exp(k, R) / (4 * math.pi * R)
            T = -1j * k * (_local(wU[sl] * Ut[sl], G, wU * Ut) -
                           _local(wU[sl] * div[sl], G, wU * div) / (k * k))
            G = G * (-(1.0 + 1j * k * R) / (R * R))
            K = _local(wU[sl] * Uk[sl], G, wU * Wk)
            del G
            for o, x in enumerate((K, T, T)):
                L[o] += sc[o] * x
        for o in range(3):
            L[o].permute(0, 2, 1, 3)[a, b] = near[o][sel]
            rows = g.gather(L[o].reshape(3 * (t1 - t0), 3 * g.nt), 1)
            Z[o].index_add_(0, g.tri_edge[sl].reshape(-1), rows)
    return Z


def _plane(waves, dev):
    th, ph, ps = (torch.as_tensor(waves[:, i].copy(), device=dev) for i in range(3))
    rh = torch.stack([th.sin() * ph.cos(), th.sin() * ph.sin(), th.cos()], 1)
    tv = torch.stack([th.cos() * ph.cos(), th.cos() * ph.sin(), -th.sin()], 1)
    pv = torch.stack([-ph.sin(), ph.cos(), torch.zeros_like(ph)], 1)
    return rh, tv, pv, ps


def _excite(g, waves):
    """v = [v^E; v^H] (2 ne x waves)."""
    rh, tv, pv, ps = _plane(waves, g.q.device)
    e = ps.cos()[:, None] * tv + ps.sin()[:, None] * pv
    hh = torch.linalg.cross(-rh, e) / ETA0
    ph = torch.einsum("tqx,wx->tqw", g.q, rh) * K0
    ph = torch.complex(ph.cos(), ph.sin()) * g.wt[..., None]
    fi = torch.einsum("tqax,tqw->taxw", g.f.to(ph.dtype), ph)
    out = []
    for vec in (e, -hh):
        out.append(g.gather(torch.einsum("taxw,wx->taw", fi, vec.to(ph.dtype)).reshape(3 * g.nt, -1), 0))
    return torch.cat(out)


def _rcs(g, j, waves, obs):
    """Partial RCS (nrhs, ndir, 2): every right-hand side at its own direction (obs None) or at all of obs."""
    mono = obs is None
    dirs = waves if mono else np.concatenate([obs, np.zeros((len(obs), 1))], 1)
    rh, tv, pv, _ = _plane(dirs, g.q.device)
    tj = [(x[g.tri_edge]) for x in (j[g.ne:], j[:g.ne])]                # aJ, aM: [t, a, rhs]
    nr = j.shape[1]
    out = torch.zeros((nr, 1 if mono else len(dirs), 2), dtype=torch.float64, device=j.device)
    for i in range(len(dirs)):
        ph = K0 * torch.einsum("tqx,x->tq", g.q, rh[i])
        ph = torch.complex(ph.cos(), ph.sin()) * g.wt
        fi = torch.einsum("tq,tqax->tax", ph, g.f.to(ph.dtype)).reshape(3 * g.nt, 3)
        sel = slice(i, i + 1) if mono else slice(None)
        N, L = (fi.T @ x.reshape(3 * g.nt, nr)[:, sel] for x in tj)
        dot = lambda a, b: (a[:, None] * b).sum(0)  # noqa: E731
        tvi, pvi = tv[i].to(ph.dtype), pv[i].to(ph.dtype)
        pre = 1j * K0 / (4 * math.pi)
        Ft = pre * (-ETA0 * dot(tvi, N) - dot(pvi, L))
        Fp = pre * (-ETA0 * dot(pvi, N) + dot(tvi, L))
        val = 4 * math.pi * torch.stack([Ft.abs() ** 2, Fp.abs() ** 2], 1)
        if mono:
            out[i, 0] = val[0]
        else:
            out[:, i] = val
    return out


def _project(g, Z, cell, CM, CJ):
    """A = (C^JM)^H Z C^MJ from the per-cell blocks."""
    dev = Z.device
    ncell = len(CM)
    ids = [torch.as_tensor(np.nonzero(cell == k)[0], device=dev) for k in range(ncell)]
    off = np.concatenate([[0], np.cumsum([b.shape[1] for b in CM])])
    nh = int(off[-1])
    cm = torch.zeros((g.ne, nh), dtype=torch.complex128, device=dev)
    cj = torch.zeros_like(cm)
    for k in range(ncell):
        cm[ids[k], off[k]:off[k + 1]] = torch.as_tensor(CM[k], device=dev)
        cj[ids[k], off[k]:off[k + 1]] = torch.as_tensor(CJ[k], device=dev)
    A = torch.empty((2 * nh, 2 * nh), dtype=torch.complex128, device=dev)
    A[:nh, :nh] = cj.mH @ (Z[0] @ cm)
    A[:nh, nh:] = cj.mH @ (Z[1] @ cj)
    A[nh:, :nh] = cm.mH @ (Z[2] @ cm)
    A[nh:, nh:] = cm.mH @ (Z[0] @ cj)
    return A, cm, cj


def _primary(g, Z, cell, ncell, gen, lmax):
    """Dual CBFs of every cell and its normalised singular values."""
    v = _excite(g, gen)
    # RWG Gram <f_a, n x f_b> of the half functions: the integrand is linear on every triangle
    nf = torch.linalg.cross(g.n[:, None, None].expand_as(g.f), g.f)
    gl = torch.einsum("tq,tqax,tqbx->tab", g.wt, nf, g.f)
    Gr = torch.zeros((g.ne, g.ne), dtype=torch.float64, device=v.device)
    e = g.tri_edge
    Gr.index_put_((e[:, :, None].expand(-1, 3, 3), e[:, None, :].expand(-1, 3, 3)), gl, accumulate=True)
    CM, CJ, L, sig = [], [], [], []
    for k in range(ncell):
        i = torch.as_tensor(np.nonzero(cell == k)[0], device=v.device)
        blk = [Z[o][i][:, i] for o in range(3)]
        J = torch.linalg.solve(torch.cat([torch.cat([blk[0], blk[1]], 1), torch.cat([blk[2], blk[0]], 1)]),
                               torch.cat([v[i], v[g.ne + i]]))
        n = len(i)
        JM, JJ = J[:n], J[n:]
        U, S, Vh = torch.linalg.svd(JM.mH @ (Gr[i][:, i].to(JM.dtype) @ JJ))
        S = S / S[0]
        m = min(int((S >= DELTA_SVD).sum()), n)
        m = min(m, lmax) if lmax > 0 else m
        CM.append((JM @ U[:, :m]).cpu().numpy())
        CJ.append((JJ @ Vh.mH[:, :m]).cpu().numpy())
        L.append(m)
        sig.append(S)
    return CM, CJ, np.array(L), torch.stack(sig)


def _exact_scatterer(c, v, t, eps, seed, part=0):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    g = _Geo(v, t, dev)
    Z = _rwg(g, eps)
    cell = _rcb(g.mid, c["ncell"])
    return g, Z, cell


def exact(case, seed):
    c = case
    if c["path"] == "batch":
        out = []
        for k, d in enumerate(_mix(c)):
            g, Z, cell = _exact_scatterer(d, *_inputs(d, seed, k), seed, k)
            out.append(_project(g, Z, cell, *_stand_in(cell, d["ncell"], d["L"], seed, k))[0])
        return out
    if _count(c) > 6000:      # a dense 64-bit operator of this size takes too long
        return None
    g, Z, cell = _exact_scatterer(c, *_inputs(c, seed), seed)
    if c["path"] == "assemble":
        return _project(g, Z, cell, *_stand_in(cell, c["ncell"], c["L"], seed))[0]
    exc = _excitations(c, seed)
    b = _excite(g, exc)
    extra = []
    if c["path"] == "mom":
        j = torch.linalg.solve(torch.cat([torch.cat([Z[0], Z[1]], 1), torch.cat([Z[2], Z[0]], 1)]), b)
    else:
        CM, CJ, L, sig = _primary(g, Z, cell, c["ncell"], _waves(c["waves"], _rng(seed, 2)), c["lmax"])
        A, cm, cj = _project(g, Z, cell, CM, CJ)
        x = torch.linalg.solve(A, torch.cat([cj.mH @ b[:g.ne], cm.mH @ b[g.ne:]]))
        nh = cm.shape[1]
        j = torch.cat([cm @ x[:nh], cj @ x[nh:]])
        extra = [None, sig] if c["path"] == "cold" else []
    return [j, _rcs(g, j, exc, _observe(c))] + extra
