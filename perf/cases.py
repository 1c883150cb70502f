"""What the library's speed is measured on: the calls that a user's imaging program makes, from one
small solve to a block of 64 transmitters on a shoulder mesh, each through the public binding.

A case names one family of calls ("do") and its sizes.  prepare() makes what the program holds
before the call: the mesh, the sources, a preconditioner of the background medium (kept stale, as
in an inversion) and the buffers; the permittivity iterate and the data come from the seed.  run()
makes the call.  The families:

  solve      new permittivity, then the forward solves: fields and S-matrix
  gradient   new permittivity, then cost, forward and adjoint solves and gradient (one evaluation
             of an inversion)
  setup      new background: assembly, subdomain factorisation, then a solve with it
  operator   Y = A X, a caller's own Krylov method
  apply      Z = M^-1 R without allocation, the same caller's preconditioner
  train      epochs of the learned initialiser over its training set
  infer      proposals of the learned initialiser

Solves run to a relative residual of 1e-12 (the tests' bar where fields are compared), so what
they return does not depend on where inside the last cycle they stopped.
"""
from __future__ import annotations

import numpy as np
import torch

import phantom
from paper_2311_05322_gb300 import inversion, mw

C0, MU0 = 299792458.0, 4.0e-7 * np.pi
EPS_BG = phantom.EPS_MATCHING
TOL = 1e-12
PREC = {"fp64": mw.MW_PREC_FP64, "fp32": mw.MW_PREC_FP32, "bf16": mw.MW_PREC_BF16, "sparse": mw.MW_PREC_SPARSE,
        "sparse_bf16": mw.MW_PREC_SPARSE_BF16}


def listed():
    return [
        # the smallest forward problem (sphere box, 8 dipoles): a solve of many short launches
        dict(name="sphere12_solve", do="solve", body="sphere", nx=12, ny=12, nz=12, src=8, nf=1, px=2, py=2, pz=2,
             overlap=1, prec="bf16", mode="mixed", steps=18),
        # the same problem on the plain FP64 path, the yardstick of the mixed one
        dict(name="sphere12_plain", do="solve", body="sphere", nx=12, ny=12, nz=12, src=8, nf=1, px=2, py=2, pz=2,
             overlap=1, prec="fp64", mode="fp64", steps=17),
        # waveguide ports and metal walls on a coarse shoulder: one evaluation, three guides
        dict(name="chamber24_gradient", do="gradient", body="chamber", nx=24, ny=24, nz=10, src=3, nf=1, px=4, py=4,
             pz=2, overlap=1, prec="bf16", mode="mixed", adjoint="solve", steps=36),
        # one evaluation of the inversion on its ordinary mesh, 32 dipoles
        dict(name="shoulder30_gradient", do="gradient", body="shoulder", nx=30, ny=30, nz=13, src=32, nf=1, px=6,
             py=6, pz=3, overlap=1, prec="bf16", mode="mixed", adjoint="solve", steps=22),
        # one evaluation on the full-scale inverse mesh, 64 dipoles
        dict(name="shoulder44_gradient", do="gradient", body="shoulder", nx=44, ny=44, nz=17, src=64, nf=1, px=9,
             py=9, pz=4, overlap=1, prec="bf16", mode="mixed", adjoint="solve", steps=30),
        # a data mesh's forward solves, 64 dipoles: the largest block
        dict(name="shoulder55_solve", do="solve", body="shoulder", nx=55, ny=55, nz=24, src=64, nf=1, px=11, py=11,
             pz=5, overlap=1, prec="bf16", mode="mixed", steps=40),
        # few large subdomains with two overlap layers: sparse factors, sweeps on the tensor cores
        dict(name="shoulder44_sparse16", do="solve", body="shoulder", nx=44, ny=44, nz=17, src=32, nf=1, px=4, py=4,
             pz=1, overlap=2, prec="sparse_bf16", mode="mixed", steps=15),
        # a new background medium: the factorisation and a first solve with it
        dict(name="shoulder30_setup", do="setup", body="shoulder", nx=30, ny=30, nz=13, src=8, nf=1, px=6, py=6,
             pz=3, overlap=1, prec="bf16", mode="mixed", steps=22),
        # the operator on a data mesh for a block of 32 columns in FP32
        dict(name="shoulder55_operator", do="operator", body="shoulder", nx=55, ny=55, nz=24, cols=32, xprec=1),
        # the allocation-free preconditioner on a small mesh
        dict(name="sphere12_apply", do="apply", body="sphere", nx=12, ny=12, nz=12, cols=16, px=3, py=3, pz=3),
        # the initialiser's training set at 32 transmitters, a ragged last batch
        dict(name="train_2048", do="train", n_in=2048, samples=270, batch=64, epochs=8),
        # its proposals for a test set
        dict(name="infer_2048", do="infer", n_in=2048, samples=30),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    do = rng.choice(["solve", "solve", "solve", "gradient", "gradient", "setup", "operator", "operator", "apply",
                     "train", "infer"])
    if do == "train":
        n = _log(rng, 64, 640)
        return dict(do=do, n_in=2 * rng.choice([8, 16, 23, 32, 48, 64]) ** 2, samples=n, batch=rng.choice([32, 64, 64]),
                    epochs=max(1, min(8, 1200 // n)))
    if do == "infer":
        return dict(do=do, n_in=2 * rng.choice([8, 16, 23, 32, 64]) ** 2, samples=_log(rng, 1, 300))
    if do == "apply":
        n = rng.randint(7, 13)
        return dict(do=do, body="sphere", nx=n, ny=n, nz=rng.randint(6, 13), cols=rng.randint(1, 32),
                    px=rng.randint(2, 3), py=rng.randint(2, 3), pz=rng.randint(1, 3))
    if do == "operator":
        nx = _log(rng, 12, 55)
        return dict(do=do, body="shoulder", nx=nx, ny=nx + rng.randint(-2, 0), nz=max(6, round(nx * 0.43)),
                    cols=2 * _log(rng, 1, 32) - rng.randint(0, 1), xprec=rng.choice([0, 1, 1, 5, 5, 3]))
    if do == "setup":
        nx = rng.randint(14, 30)
        nz = max(7, round(nx * 0.43))
        return dict(do=do, body="shoulder", nx=nx, ny=nx, nz=nz, src=rng.randint(4, 16), nf=rng.choice([1, 1, 2]),
                    px=max(2, round(nx / 5)), py=max(2, round(nx / 5)), pz=max(1, round(nz / 4.5)), overlap=1,
                    prec=rng.choice(["bf16", "bf16", "fp32"]), mode="mixed", steps=20)
    adjoint = {} if do == "solve" else dict(adjoint=rng.choice(["solve", "solve", "reciprocal"]))
    form = rng.choice(["sphere", "shoulder", "shoulder", "plain", "sparse"])
    if form == "plain":
        n = rng.randint(8, 13)
        return dict(do=do, body="sphere", nx=n, ny=n, nz=n, src=rng.randint(2, 12), nf=1, px=2, py=2, pz=2, overlap=1,
                    prec="fp64", mode="fp64", steps=16, **adjoint)
    if form == "sphere":
        n = rng.randint(8, 18)
        return dict(do=do, body="sphere", nx=n, ny=n, nz=n, src=rng.randint(2, 40), nf=rng.choice([1, 1, 2]),
                    px=max(2, n // 5), py=max(2, n // 5), pz=max(2, n // 6), overlap=1,
                    prec=rng.choice(["bf16", "bf16", "fp32"]), mode="mixed", steps=18, **adjoint)
    nx = _log(rng, 16, 44)
    nz = max(7, round(nx * 0.41))
    if form == "sparse":
        return dict(do=do, body="shoulder", nx=nx, ny=nx, nz=nz, src=rng.randint(6, 40), nf=1, px=rng.randint(2, 4),
                    py=rng.randint(2, 4), pz=1, overlap=rng.randint(1, 2),
                    prec=rng.choice(["sparse_bf16", "sparse_bf16", "sparse"]), mode="mixed", steps=15, **adjoint)
    return dict(do=do, body="shoulder", nx=nx, ny=nx - rng.randint(0, 2), nz=nz, src=rng.randint(5, 64),
                nf=rng.choice([1, 1, 3]) if nx < 30 else 1, px=max(2, round(nx / 5)), py=max(2, round(nx / 5)),
                pz=max(2, round(nz / 4.5)), overlap=1, prec="bf16", mode="mixed", steps=30, **adjoint)


# ---------------------------------------------------------------------------------------------
# problems
# ---------------------------------------------------------------------------------------------
def _pairs(e):
    return np.ascontiguousarray(np.stack([e.real, e.imag], 1))


def _problem(case, seed):
    """Mesh, background and iterate permittivity, frequencies, dipoles or guides."""
    rng = np.random.default_rng(seed)
    cells = (case["nx"], case["ny"], case["nz"])
    p = dict(freqs=[1.0e9] if case.get("nf", 1) == 1 else np.linspace(0.8e9, 1.2e9, case["nf"]).tolist(), ports=None)
    n_src = case.get("src", 1)
    if case["body"] == "sphere":
        m = phantom.kuhn_mesh(*cells)
        back = np.full(m.n_tet, EPS_BG, dtype=complex)
        eps, _ = phantom.sphere_phantom(m, seed)
        h = 0.12 / cells[2]
        p["pos"], p["dir"] = phantom.dipole_ring(n_src, 0.05, h / 2 if cells[2] % 2 == 0 else 0.0)
    else:
        m = phantom.kuhn_mesh(*cells, lo=phantom.SHOULDER_LO, hi=phantom.SHOULDER_HI)
        back = phantom.shoulder_eps(m)
        eps = phantom.shoulder_eps(m, phantom.random_tear(seed))
        h = (phantom.SHOULDER_HI[2] - phantom.SHOULDER_LO[2]) / cells[2]
        p["pos"], p["dir"] = phantom.dipole_ring(n_src, 0.10, h / 2 if cells[2] % 2 == 0 else 0.0, phantom.ARM_CENTER)
        if case["body"] == "chamber":
            fv, lab, ps, guide = phantom.port_chamber(m, n_per_wall=(0, 1, 1, 1))
            p["ports"] = (ps.origin, ps.u, ps.v, ps.a, ps.eps_fill, fv, lab)
            back[guide] = eps[guide] = ps.eps_fill[0]
    # an inversion's iterate: every element a little off its tissue
    eps = eps * (1.0 + 0.02 * rng.standard_normal(m.n_tet))
    p.update(mesh=m, back=back, eps=eps, rng=rng)
    return p


def _data(case, p):
    """S of the empty chamber and observed S of the right magnitudes: the dipole's field in the
    homogeneous medium (a guide's: order one), and an observation some percent away from it."""
    n, rng = case["src"], p["rng"]
    emp = np.empty((len(p["freqs"]), n, n), complex)
    for f, hz in enumerate(p["freqs"]):
        if p["ports"] is None:
            step = p["mesh"].h[2]
            r = np.linalg.norm(p["pos"][:, None] - p["pos"][None], axis=2)
            r[r < step / 2] = step / 2
            k = 2 * np.pi * hz / C0 * np.sqrt(EPS_BG)
            emp[f] = (-2j * np.pi * hz * MU0 * step ** 2 * np.exp(-1j * k * r) / (4 * np.pi * r)
                      * (1 + 1 / (1j * k * r) - 1 / (k * r) ** 2))
        else:
            emp[f] = 0.1 + 0.9 * np.eye(n)
    noise = rng.standard_normal(emp.shape) + 1j * rng.standard_normal(emp.shape)
    return emp, emp * (1.0 + 0.05 * noise)


def _opts(case):
    # inner cycles as the drivers set them: 1e-2 for the forward blocks of dense inverses, 1e-4 elsewhere
    inner = 1e-2 if case["do"] == "solve" and case["prec"] == "bf16" else inversion.INNER_TOL
    return mw.solve_opts(mode=mw.MW_MODE_FP64 if case["mode"] == "fp64" else mw.MW_MODE_MIXED, tol=TOL,
                         inner_tol=inner, max_outer=40)


def _partition(case, mesh):
    parts = (case["px"], case["py"], case["pz"])
    return int(np.prod(parts)), phantom.box_partition(mesh, parts, seed=7)


def _network(case, seed):
    rng = np.random.default_rng(seed)
    n = case["samples"]
    x = rng.standard_normal((n, case["n_in"]), dtype=np.float32)          # standardised features
    t = 0.1 * rng.standard_normal((n, 2, 32, 32, 32), dtype=np.float32)
    return x, t, inversion.he_init(case["n_in"], seed)


def prepare(case, seed):
    s = dict(case=case)
    if case["do"] in ("train", "infer"):
        s["x"], s["t"], theta = _network(case, seed)
        c = s["ctx"] = mw.Context(0)
        c.nn_init(case["n_in"], theta)
        return s
    p = _problem(case, seed)
    m = p["mesh"]
    c = s["ctx"] = mw.Context(0)
    E = c.set_mesh(m.xyz, m.tets).n_edge
    s["freqs"] = p["freqs"]
    s["eps"] = torch.from_numpy(_pairs(p["eps"])).cuda()
    if case["do"] in ("operator", "apply"):
        c.assemble(p["freqs"], _pairs(p["eps"]), EPS_BG)
        g = torch.Generator("cuda").manual_seed(seed)
        n = case["cols"]
        if case["do"] == "apply" or case["xprec"] == 1:
            s["x"] = torch.randn((E, n), dtype=torch.complex64, device="cuda", generator=g)
            s["y"] = torch.empty_like(s["x"])
        elif case["xprec"] == 5:
            s["x"] = torch.randn((E, n, 2), device="cuda", generator=g).to(torch.bfloat16)
            s["y"] = torch.empty((E, n), dtype=torch.complex64, device="cuda")
        else:
            s["x"] = torch.randn((E, n), dtype=torch.complex128, device="cuda", generator=g)
            s["y"] = torch.empty_like(s["x"])
        if case["do"] == "apply":
            c.setup_preconditioner(*_partition(case, m), 1, mw.MW_PREC_BF16)
        return s
    if p["ports"] is not None:
        c.set_ports(*p["ports"])
    else:
        c.set_sources(p["pos"], p["dir"])
    c.assemble(p["freqs"], _pairs(p["back"]), EPS_BG)
    s["part"] = _partition(case, m)
    s["opts"] = _opts(case)
    if case["do"] == "gradient":
        c.setup_preconditioner(*s["part"], case["overlap"], PREC[case["prec"]])
        c.set_adjoint_mode(case["adjoint"] == "reciprocal")
        emp, obs = _data(case, p)
        s["emp"], s["obs"] = torch.from_numpy(emp).cuda(), torch.from_numpy(obs).cuda()
        s["grad"] = torch.empty((m.n_tet, 2), dtype=torch.float64, device="cuda")
        return s
    if case["do"] == "solve":
        c.setup_preconditioner(*s["part"], case["overlap"], PREC[case["prec"]])
    s["fields"] = torch.empty((len(p["freqs"]) * c.n_src, E), dtype=torch.complex128, device="cuda")
    return s


def run(s):
    case, c = s["case"], s["ctx"]
    do = case["do"]
    if do == "train":
        losses, _ = c.nn_train(s["x"], s["t"], batch=case["batch"], epochs=case["epochs"], lr=1e-3, seed=5)
        return {"losses": losses, "theta": c.nn_get_params()}
    if do == "infer":
        return c.nn_infer(s["x"])
    if do == "operator":
        c.apply_matrix(0, case["xprec"], s["x"], s["y"], case["cols"])
        return s["y"]
    if do == "apply":
        c.apply_preconditioner_noalloc(0, s["x"], s["y"], case["cols"])
        return s["y"]
    c.assemble_dev(s["freqs"], s["eps"], EPS_BG)
    if do == "gradient":
        J = c.gradient_dev(s["obs"], s["emp"], s["grad"], 0.0, s["opts"])
        return {"J": J, "gradient": s["grad"]}
    if do == "setup":
        c.setup_preconditioner(*s["part"], case["overlap"], PREC[case["prec"]])
    S, _ = c.solve(s["opts"], fields=s["fields"])
    return {"S": S, "fields": s["fields"]}


# ---------------------------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------------------------
def _sizes(case):
    """Edges, tets, matrix entries of the Kuhn box; mean subdomain size of its partition."""
    a, b, d = case["nx"], case["ny"], case["nz"]
    V, T = (a + 1) * (b + 1) * (d + 1), 6 * a * b * d
    Fb = 4 * (a * b + b * d + a * d)
    F = (4 * T + Fb) // 2
    E = V + F - T - 1
    nnz = E + 6 * F + 6 * T
    if "px" not in case:
        return E, T, nnz, 0, 0.0, 0.0
    g = 2 * case.get("overlap", 1)
    k = case["px"] * case["py"] * case["pz"]
    own = E / k
    ns = 1.0
    for n, q in ((a, case["px"]), (b, case["py"]), (d, case["pz"])):
        ns *= min(n / q + g, n) / (n / q)
    return E, T, nnz, k, own, own * ns


def work(case):
    """Operands read once and results written once.  A solve counts its usual Arnoldi steps
    ("steps", of one block of columns): each reads the matrix and the subdomain
    inverses (the factors, for the sparse form) and a basis vector in and out."""
    do = case["do"]
    if do in ("train", "infer"):
        n, w = case["samples"], 1024
        layers = 2 * w * (case["n_in"] + w) + 2 * 64 * (16 * 16 * 64 + 16 * 8 * 512 + 8 * 2 * 4096)
        par = w * case["n_in"] + w * w
        if do == "infer":
            return {"bytes": 4 * n * (case["n_in"] + 65536) + 2 * par, "flops": n * layers}
        batches = -(-n // case["batch"]) * case["epochs"]
        return {"bytes": batches * 28 * par + case["epochs"] * 4 * n * (case["n_in"] + 65536),
                "flops": 3 * n * layers * case["epochs"]}
    E, T, nnz, k, own, ns = _sizes(case)
    if do == "operator":
        xb, yb = {0: (16, 16), 3: (16, 16), 1: (8, 8), 5: (4, 8)}[case["xprec"]]
        vb = 8 if case["xprec"] in (1, 5) else 16
        return {"bytes": nnz * (vb + 4) + 8 * E + E * case["cols"] * (xb + yb), "flops": 8 * nnz * case["cols"]}
    if do == "apply":
        R = case["cols"]
        return {"bytes": 4 * k * own * ns + 16 * E * R, "flops": 8 * k * own * ns * R}
    R, nf = case["src"], case["nf"]
    eb = 16 if case["mode"] == "fp64" else 8
    wb = {"fp64": 16, "fp32": 8, "bf16": 4, "sparse": 8, "sparse_bf16": 4}[case["prec"]]
    # factor entries of nested dissection in three dimensions grow like n^(4/3)
    w = 30.0 * k * ns ** (4 / 3) if case["prec"].startswith("sparse") else k * own * ns
    step = w * wb + nnz * (eb + 4) + 4 * eb * E * R
    twice = 2 if case.get("adjoint") == "solve" else 1
    out = 32 * T + 32 * T if do == "gradient" else 16 * E * R
    flops = case["steps"] * 8 * R * (w + nnz + 4 * E)
    if do == "setup":
        flops += 8 * k * ns ** 3
    return {"bytes": nf * (case["steps"] * step * (twice if "adjoint" in case else 1) + 24 * nnz) + out,
            "flops": nf * flops * (twice if "adjoint" in case else 1)}


# ---------------------------------------------------------------------------------------------
# 64-bit values by plain numpy and torch
# ---------------------------------------------------------------------------------------------
_EDGES = ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))


def _whitney(g, I, pairs):
    """Integrals of Whitney functions' products: g [n, p, 3] gradients, I [n, p, p] moments."""
    G = np.einsum("tpi,tqi->tpq", g, g)
    out = np.empty((g.shape[0], len(pairs), len(pairs)))
    for i, (a, b) in enumerate(pairs):
        for j, (c, d) in enumerate(pairs):
            out[:, i, j] = (I[:, a, c] * G[:, b, d] - I[:, a, d] * G[:, b, c] - I[:, b, c] * G[:, a, d]
                            + I[:, b, d] * G[:, a, c])
    return out


def _system(mesh, eps, hz):
    """Element matrices of A with their edge ids: volume [T, 6, 6] and open boundary [F, 3, 3]."""
    tets = np.sort(mesh.tets.astype(np.int64), axis=1)          # ascending vertices: every sign is +1
    P = mesh.xyz[tets]
    V = mesh.n_vert
    ekey = np.stack([tets[:, a] * V + tets[:, b] for a, b in _EDGES], 1)
    edges, te = np.unique(ekey, return_inverse=True)
    te = te.reshape(ekey.shape)
    J = P[:, 1:] - P[:, :1]
    g = np.empty((len(tets), 4, 3))
    g[:, 1:] = np.transpose(np.linalg.inv(J), (0, 2, 1))
    g[:, 0] = -g[:, 1:].sum(axis=1)
    vol = np.abs(np.linalg.det(J)) / 6
    curl = np.stack([np.cross(g[:, a], g[:, b]) for a, b in _EDGES], 1)
    K = 4 * vol[:, None, None] * np.einsum("tmi,tni->tmn", curl, curl)
    M = _whitney(g, (vol / 20)[:, None, None] * (1 + np.eye(4)), _EDGES)
    k0 = 2 * np.pi * hz / C0
    A = K - k0 ** 2 * eps[:, None, None] * M
    tri = np.concatenate([tets[:, f] for f in ((0, 1, 2), (0, 1, 3), (0, 2, 3), (1, 2, 3))])
    key, first, n = np.unique((tri[:, 0] * V + tri[:, 1]) * V + tri[:, 2], return_index=True, return_counts=True)
    tri = tri[first[n == 1]]
    Q = mesh.xyz[tri]
    cr = np.cross(Q[:, 1] - Q[:, 0], Q[:, 2] - Q[:, 0])
    area = np.linalg.norm(cr, axis=1) / 2
    nrm = cr / (2 * area)[:, None]
    opp = np.stack([Q[:, 2] - Q[:, 1], Q[:, 0] - Q[:, 2], Q[:, 1] - Q[:, 0]], 1)
    gs = np.cross(nrm[:, None], opp) / (2 * area)[:, None, None]
    pairs = ((0, 1), (0, 2), (1, 2))
    B = 1j * k0 * np.sqrt(EPS_BG) * _whitney(gs, (area / 12)[:, None, None] * (1 + np.eye(3)), pairs)
    fe = np.searchsorted(edges, np.stack([tri[:, a] * V + tri[:, b] for a, b in pairs], 1))
    return edges, te, A, fe, B


def _dipoles(mesh, edges, pos, direc):
    a, b = mesh.xyz[edges // mesh.n_vert], mesh.xyz[edges % mesh.n_vert]
    d = b - a
    z = np.nonzero((np.abs(d[:, :2]) <= 1e-9 * np.abs(d[:, 2:])).all(axis=1) & (d[:, 2] != 0))[0]
    mid = (a[z] + b[z]) / 2
    e = np.array([z[np.argmin(((mid - q) ** 2).sum(axis=1))] for q in pos])
    return e, np.where(d[e, 2] * direc[:, 2] > 0, 1.0, -1.0)


def _bf16(w):
    return w.to(torch.bfloat16).to(torch.float64)


def _exact_network(case, seed):
    """The network in 64 bits (weights of the dense layers rounded to BF16 where they are used)."""
    x, t, theta = _network(case, seed)
    x = torch.from_numpy(x).cuda().double()
    th = torch.from_numpy(theta).cuda().double()
    shapes = [(1024, case["n_in"]), (1024,), (1024, 1024), (1024,), (16, 16, 4, 4, 4), (16,), (16, 8, 4, 4, 4), (8,),
              (8, 2, 4, 4, 4), (2,)]
    cuts = np.cumsum([0] + [int(np.prod(q)) for q in shapes])

    def forward(th, x):
        w1, b1, w2, b2, k1, c1, k2, c2, k3, c3 = (th[cuts[i]:cuts[i + 1]].view(q) for i, q in enumerate(shapes))
        # the gradient passes the rounding of the weights by, as mixed-precision training does
        w1, w2 = (w + (_bf16(w) - w).detach() for w in (w1, w2))
        h = torch.relu(x @ w1.T + b1)
        h = torch.relu(h @ w2.T + b2).view(-1, 16, 4, 4, 4)
        conv = torch.nn.functional.conv_transpose3d
        h = torch.relu(conv(h, k1, c1, stride=2, padding=1))
        h = torch.relu(conv(h, k2, c2, stride=2, padding=1))
        return conv(h, k3, c3, stride=2, padding=1)

    if case["do"] == "infer":
        with torch.no_grad():
            return torch.cat([forward(th, q) for q in x.split(64)]).cpu().numpy()
    t = torch.from_numpy(t).cuda().double()
    mom, var = torch.zeros_like(th), torch.zeros_like(th)
    mask64, step, losses = (1 << 64) - 1, 0, []
    n = case["samples"]
    for ep in range(case["epochs"]):
        state = (5 + 0x632BE59BD9B4E019 * (ep + 1)) & mask64
        perm = list(range(n))
        for i in range(n - 1, 0, -1):
            state = (state + 0x9E3779B97F4A7C15) & mask64
            z = state
            z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask64
            z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask64
            j = (z ^ (z >> 31)) % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        total = 0.0
        for b in range(0, n, case["batch"]):
            idx = torch.tensor(perm[b:b + case["batch"]], device="cuda")
            th = th.detach().requires_grad_(True)
            loss = ((forward(th, x[idx]) - t[idx]) ** 2).mean()
            (gr,) = torch.autograd.grad(loss, th)
            step += 1
            mom = 0.9 * mom + 0.1 * gr
            var = 0.999 * var + 0.001 * gr * gr
            th = th.detach() - 1e-3 * (mom / (1 - 0.9 ** step)) / (torch.sqrt(var / (1 - 0.999 ** step)) + 1e-8)
            total += float(loss) * len(idx)
        losses.append(total / n)
    return {"losses": np.array(losses), "theta": th.cpu().numpy()}


def exact(case, seed):
    do = case["do"]
    if do in ("train", "infer"):
        return _exact_network(case, seed)
    if do in ("gradient", "apply"):
        return None
    E = _sizes(case)[0]
    if do != "operator" and (E > 14000 or case["nf"] > 1):
        return None                 # the direct solution takes too long
    p = _problem(case, seed)
    hz = p["freqs"][0]
    edges, te, A, fe, B = _system(p["mesh"], p["eps"], hz)
    te, fe = torch.from_numpy(te).cuda(), torch.from_numpy(fe).cuda()
    A, B = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    if do == "operator":
        g = torch.Generator("cuda").manual_seed(seed)
        n = case["cols"]
        if case["xprec"] == 1:
            x = torch.randn((E, n), dtype=torch.complex64, device="cuda", generator=g).to(torch.complex128)
        elif case["xprec"] == 5:
            x = torch.view_as_complex(torch.randn((E, n, 2), device="cuda", generator=g).to(torch.bfloat16).double())
        else:
            x = torch.randn((E, n), dtype=torch.complex128, device="cuda", generator=g)
        y = torch.zeros((E, n), dtype=torch.complex128, device="cuda")
        for idx, el in ((te, A), (fe, B)):
            for a in range(el.shape[1]):
                for b in range(el.shape[2]):
                    y.index_add_(0, idx[:, a], el[:, a, b, None] * x[idx[:, b]])
        return y
    full = torch.zeros(E * E, dtype=torch.complex128, device="cuda")
    for idx, el in ((te, A), (fe, B)):
        full.index_add_(0, (idx[:, :, None] * E + idx[:, None, :]).reshape(-1), el.reshape(-1))
    e, sign = _dipoles(p["mesh"], edges, p["pos"], p["dir"])
    rhs = np.zeros((E, len(e)), complex)
    rhs[e, np.arange(len(e))] = -2j * np.pi * hz * MU0 * sign
    X = torch.linalg.solve(full.view(E, E), torch.from_numpy(rhs).cuda()).T.contiguous()
    S = (X[:, torch.from_numpy(e).cuda()] * torch.from_numpy(sign).cuda()).T.contiguous()[None]
    return {"S": S.cpu().numpy(), "fields": X}
