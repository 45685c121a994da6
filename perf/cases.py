"""The work this library is measured on: operator products, system products, solves and operator builds.

Every case goes through the public Python binding.  A program keeps its mesh and operator handles while the vectors
change, so `prepare` keeps one handle per geometry and frequency in this process and makes the vectors from the seed; the
build cases pay for the handle in `run` itself, at a frequency of the seed.

Sizes are those of this repository's workloads (benchmark, tests, ports leg): icospheres of 80 to 20,480 triangles,
copper bars and boxes of some tens to a few thousand, grids of 7 to 63 nodes per axis, 1 to 8 right-hand sides.
"""
import math

import numpy as np
import torch

import paper_2003_11679_gb300 as sie
from synth import box, icosphere

C0 = 299792458.0
MU0 = 4e-7 * math.pi
EPS0 = 1.0 / (MU0 * C0 * C0)
COPPER = 5.8e7
WHICH = {"L0": sie.SIE_OP_L0, "K0": sie.SIE_OP_K0, "LI": sie.SIE_OP_LI, "KI": sie.SIE_OP_KI}


def _sphere(level, radius, equal_volume):
    return {"mesh": "sphere", "level": level, "radius": radius, "equal_volume": equal_volume}


def _box(size, div):
    return {"mesh": "box", "lx": size[0], "ly": size[1], "lz": size[2], "nx": div[0], "ny": div[1], "nz": div[2]}


def _medium(freq, eps_r, sigma, interior, grid_n=0, dense_pc=True):
    return {"freq": freq, "eps_r": eps_r, "sigma": sigma, "interior": interior, "grid_n": grid_n, "dense_pc": dense_pc}


def listed():
    dielectric = _medium(3e9, 4.0, 0.0, "gibc")
    lossy20480 = dict(_sphere(5, 1e-3, False), **_medium(10e9, 1.0, COPPER, "sibc", 64, False))
    lossy320 = dict(_sphere(2, 1e-3, False), **_medium(10e9, 1.0, COPPER, "gibc", 64))
    bar = dict(_box((40e-6, 4e-6, 4e-6), (20, 2, 2)), **_medium(100e9, 1.0, COPPER, "gibc"))
    return [
        # the smallest call a program makes: one L product of a coarse sphere, all launches and latency
        dict(name="L 80 tri", kind="product", which="L0", nrhs=1, **_sphere(1, 1e-2, True), **dielectric),
        # a block of right-hand sides on the dielectric sphere of the benchmark's solves
        dict(name="K 1280 tri x8", kind="product", which="K0", nrhs=8, **_sphere(3, 1e-2, True), **dielectric),
        # the largest product: 30,720 unknowns on the 128^3 transform, eight right-hand sides
        dict(name="L 20480 tri x8", kind="product", which="L0", nrhs=8, **lossy20480),
        # the benchmark's step on its coarse mesh: nested near-region interior, 128^3 transform
        dict(name="sys copper 320 tri", kind="system", precision="fp64", **lossy320),
        # an elongated conductor of the ports workload: short transforms, the nested solve and launches count
        dict(name="sys copper bar", kind="system", precision="fp64", **bar),
        # 30,720 unknowns with the surface impedance interior: transforms and the near-region product
        dict(name="sys 20480 tri", kind="system", precision="fp64", **lossy20480),
        # the same product on the complex64 grid path, as refined solves and the serving loop run it
        dict(name="sys 20480 tri mixed", kind="system", precision="mixed", **lossy20480),
        # penetrable object: interior AIM operator, nested solve with its constraint preconditioner
        dict(name="sys dielectric 320 tri", kind="system", precision="fp64", **_sphere(2, 1e-2, True), **dielectric),
        # one plane wave to the paper's tolerance, then a bistatic cut
        dict(name="solve + rcs 1280 tri", kind="solve", nrhs=1, ndir=181, **_sphere(3, 1e-2, True),
             **_medium(3e9, 1.0, COPPER, "sibc")),
        # eight excitations of the bar in lockstep, as the ports and the batching loop do
        dict(name="solve bar x8", kind="solve", nrhs=8, ndir=1, **bar),
        # operators of a new frequency, penetrable object (frequency sweeps rebuild at every point)
        dict(name="build dielectric 80 tri", kind="build", **_sphere(1, 1e-2, True), **dielectric),
        # operators of a new frequency, good conductor: the near-region-only interior
        dict(name="build copper 48 tri", kind="build", **_box((1e-3, 1e-3, 1e-3), (2, 2, 2)),
             **_medium(10e9, 1.0, COPPER, "gibc")),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["product", "product", "product", "system", "system", "system", "solve", "build"])
    # boxes of about the drawn number of triangles: 4 (ab + bc + ca) for a x b x c cells
    small = kind == "build"
    nt = _log_uniform(rng, 60, 120 if small else (600 if kind == "solve" else 4000))
    aspect = rng.uniform(1.0, 3.0 if small else 8.0)
    b = max(1, int(round(math.sqrt(nt / (4.0 * (2.0 * aspect + 1.0))))))
    div = (max(1, int(round(b * aspect))), b, max(1, b + rng.choice([-1, 0, 1])))
    cell = 1e-3 * rng.uniform(0.8, 1.2)
    m = _box([cell * d * rng.uniform(0.9, 1.1) for d in div], div)
    freq = round(_log_uniform(rng, 1e9, 8e9))
    ndiv = max(div)
    grid_n = 0 if small or rng.random() < 0.6 else rng.randint(max(16, ndiv + 8), 64)
    if kind == "product":
        return dict(kind=kind, which=rng.choice(["L0", "K0", "LI", "KI"]), nrhs=rng.randint(1, 8), **m,
                    **_medium(freq, round(rng.uniform(1.5, 6.0), 3), round(rng.choice([0.0, 0.1]), 3), "gibc", grid_n, False))
    if kind == "build":
        sigma = rng.choice([0.0, 0.1])
        return dict(kind=kind, **m, **_medium(freq, round(rng.uniform(1.5, 6.0), 3), sigma, "gibc", grid_n))
    med = _medium(freq, 1.0, round(_log_uniform(rng, 1e5, COPPER)), "sibc", grid_n, kind == "solve")
    if kind == "solve":
        return dict(kind=kind, nrhs=rng.randint(1, 8), ndir=1, **m, **med)
    return dict(kind=kind, precision=rng.choice(["fp64", "fp64", "mixed"]), **m, **med)


# ---------------------------------------------------------------- handles
_context = None
_meshes, _operators = {}, {}


def _geometry(case):
    if case["mesh"] == "sphere":
        return icosphere(case["level"], case["radius"], equal_volume=case["equal_volume"])
    return box((case["lx"], case["ly"], case["lz"]), (case["nx"], case["ny"], case["nz"]))


def _key(case, *names):
    return tuple((k, case[k]) for k in sorted(case) if k in names)


_SHAPE = ("mesh", "level", "radius", "equal_volume", "lx", "ly", "lz", "nx", "ny", "nz")
_MEDIUM = ("freq", "eps_r", "sigma", "interior", "grid_n", "dense_pc")


def _mesh(case):
    global _context
    key = _key(case, *_SHAPE)
    if key not in _meshes:
        if _context is None:
            # the stream torch's own work is on: products and torch operations stay in order
            _context = sie.Context(0, stream=torch.cuda.current_stream().cuda_stream or None)
        V, T = _geometry(case)
        _meshes[key] = (sie.Mesh(_context, V, T), V, T)
    return _meshes[key]


def _params(case):
    p = sie.params(grid_n=case["grid_n"], interior_model=sie.SIE_SIBC if case["interior"] == "sibc" else sie.SIE_GIBC)
    if not case["dense_pc"]:
        p.dense_pc_max = 0  # a program that only multiplies needs no factorised preconditioner
    return p


def _operator(case):
    key = _key(case, *_SHAPE, *_MEDIUM)
    if key not in _operators:
        _operators[key] = sie.Operator(_mesh(case)[0], case["freq"], case["eps_r"], 1.0, case["sigma"], _params(case))
    return _operators[key]


def _vectors(n, nrhs, seed):
    g = torch.Generator(device="cuda").manual_seed(1000003 * (seed % 1000003) + 17)
    v = torch.randn((nrhs, n, 2), generator=g, device="cuda", dtype=torch.float64) * math.sqrt(0.5)
    return torch.view_as_complex(v)


def _waves(nrhs, seed):
    r = np.random.Generator(np.random.PCG64(seed))
    k = r.standard_normal((nrhs, 3))
    k /= np.linalg.norm(k, axis=1, keepdims=True)
    e = np.cross(k, r.standard_normal((nrhs, 3)))
    return k, e / np.linalg.norm(e, axis=1, keepdims=True)


def prepare(case, seed):
    kind = case["kind"]
    mesh = _mesh(case)[0]
    if kind == "build":
        u = np.random.Generator(np.random.PCG64(seed)).uniform(0.95, 1.05)
        return {"case": case, "mesh": mesh, "freq": case["freq"] * u, "params": _params(case)}
    op = _operator(case)
    s = {"case": case, "op": op}
    if kind == "product":
        s["x"] = _vectors(mesh.ne, case["nrhs"], seed)
        s["y"] = torch.empty_like(s["x"])
    elif kind == "system":
        op.set_solver(precision=sie.SIE_MIXED if case["precision"] == "mixed" else sie.SIE_FP64)
        s["x"] = _vectors(mesh.ne + mesh.nt, 1, seed)[0].contiguous()
        s["y"] = torch.empty_like(s["x"])
    else:
        op.set_solver(precision=sie.SIE_FP64)
        k, e = _waves(case["nrhs"], seed)
        s["b"] = torch.zeros((case["nrhs"], mesh.ne + mesh.nt), dtype=torch.complex128, device="cuda")
        op.rhs_planewave(k, e, s["b"])
        s["x"] = torch.empty_like(s["b"])
        a = np.linspace(0.0, np.pi, case["ndir"])
        s["dirs"] = np.stack([np.sin(a), 0.0 * a, np.cos(a)], axis=1)
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "product":
        return state["op"].matvec(WHICH[case["which"]], state["x"], state["y"], case["nrhs"])
    if kind == "system":
        ne = state["op"].mesh.ne
        y = state["op"].matvec(sie.SIE_OP_SYS, state["x"], state["y"])
        if case["precision"] == "mixed":  # single-precision accuracy: kept as complex64, as its consumer would
            y = y.to(torch.complex64)
        # the two blocks of Eq. (sys) have different units
        return {"current": y[:ne], "charge": y[ne:]}
    if kind == "solve":
        x, _, _ = state["op"].solve(state["b"], state["x"], nrhs=case["nrhs"])
        return {"x": x, "rcs": state["op"].rcs(x[0], state["dirs"])}
    op = sie.Operator(state["mesh"], state["freq"], case["eps_r"], 1.0, case["sigma"], state["params"])
    out = {"L": op.near_csr(sie.SIE_OP_L0)[2], "K": op.near_csr(sie.SIE_OP_K0)[2]}
    if case["interior"] == "gibc":
        out["Li"], out["Ki"] = op.near_csr(sie.SIE_OP_LI)[2], op.near_csr(sie.SIE_OP_KI)[2]
    op.close()
    return out


# ---------------------------------------------------------------- work
def _grid_of(case):
    """(N, near triangle pairs, triangles) of a case's exterior grid, by the rules the library states."""
    V, T = _geometry(case)
    lo, hi = V.min(axis=0), V.max(axis=0)
    e = np.concatenate([V[T[:, (i + 1) % 3]] - V[T[:, i]] for i in range(3)])
    h = (hi - lo).max() / (case["grid_n"] - 7) if case["grid_n"] else 0.5 * np.linalg.norm(e, axis=1).mean()
    o = lo - (2 + 0.5 / np.sqrt([2.0, 3.0, 5.0])) * h
    N = np.floor((hi - o) / h).astype(int) + 4
    c = np.floor((V[T].mean(axis=1) - o) / h + 0.5).astype(int)
    count = np.zeros(N)
    np.add.at(count, tuple(c.T), 1.0)
    box_sum = count
    for d in range(3):
        p = np.concatenate([np.zeros_like(box_sum.take([0], d)), np.cumsum(box_sum, axis=d)], axis=d)
        i = np.arange(N[d])
        box_sum = p.take(np.minimum(i + 6, N[d]), d) - p.take(np.maximum(i - 5, 0), d)
    return N, float((count * box_sum).sum()), len(T)


def _grid_flops(N, forward, inverse):
    """Pruned transforms of the doubled box, 5 n log2 n operations per line."""
    n = 2.0 * N
    per = (5 * n[0] * np.log2(n[0]) * N[1] * N[2] + 5 * n[1] * np.log2(n[1]) * n[0] * N[2]
           + 5 * n[2] * np.log2(n[2]) * n[0] * n[1])
    return (forward + inverse) * per


def work(case):
    N, pairs, nt = _grid_of(case)
    ne = 1.5 * nt
    nnz = 2.5 * pairs  # stored edge entries per near triangle pair
    weights = 27 * 32.0 * nt
    kind = case["kind"]
    if kind == "product":
        nrhs, g = case["nrhs"], 4 if case["which"][0] == "L" else 3
        spectra = 16.0 * (1 if g == 4 else 3) * N.prod()  # the kernels are even or odd in every axis
        flops = nrhs * (_grid_flops(N, g, g) + (6.0 * 4 if g == 4 else 44.0) * 8 * N.prod() + 8 * nnz + 27 * 60.0 * nt)
        return {"bytes": 20 * nnz + weights + spectra + 32 * ne * nrhs, "flops": float(flops)}
    if kind == "build":
        # one integrand per point of the far rule (5^4 points) and pair, about 60 operations each; a conductor's
        # interior keeps only its touching pairs
        outputs = 2 if case["sigma"] > 1e3 else 4
        return {"bytes": 16 * outputs * nnz, "flops": 625 * 60.0 * pairs}
    c = 8.0 if case.get("precision") == "mixed" else 16.0
    near = nnz * (2 * c + 4) + pairs * (c + 4)
    flops = float(_grid_flops(N, 7, 4) + 76.0 * 8 * N.prod() + 16 * nnz + 8 * pairs + 27 * 100.0 * nt)
    once = near + weights * c / 16 + 4 * c * N.prod() + 32 * (ne + nt)
    if kind == "system":
        return {"bytes": once, "flops": flops}
    steps = 20  # products a converging solve needs at least
    return {"bytes": steps * once, "flops": steps * flops * case["nrhs"]}


# ---------------------------------------------------------------- the same results in plain torch
def _wavenumber(case, interior):
    w = 2 * math.pi * case["freq"]
    if not interior:
        return complex(w / C0)
    k = np.sqrt(complex(w * MU0) * complex(w * EPS0 * case["eps_r"], -case["sigma"]))
    return complex(-k if k.imag > 0 else k)


def _rwg(V, T):
    """Edge number, s l / (2 A) and c_t - p_i of every (triangle, slot); slot i is the edge opposite vertex i."""
    a, b = T[:, [1, 2, 0]].astype(np.int64), T[:, [2, 0, 1]].astype(np.int64)
    lo, hi = np.minimum(a, b), np.maximum(a, b)
    edge = np.unique(lo * len(V) + hi, return_inverse=True)[1].reshape(lo.shape)
    P = V[T]
    area = 0.5 * np.linalg.norm(np.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0]), axis=1)
    length = np.linalg.norm(V[a] - V[b], axis=2)
    coef = np.where(a < b, 1.0, -1.0) * length / (2 * area[:, None])
    cen = P.mean(axis=1)
    return edge, coef, cen[:, None, :] - P, cen, area


def _exact_product(case, seed):
    op, (mesh, V, T) = _operator(case), _mesh(case)
    x = _vectors(mesh.ne, case["nrhs"], seed)
    dev = x.device
    interior = case["which"][1] == "I"
    k = _wavenumber(case, interior)
    rp, col, val = op.near_csr(WHICH[case["which"]])
    rows = torch.from_numpy(np.repeat(np.arange(mesh.ne), np.diff(rp))).to(dev)
    col, val = torch.from_numpy(col).to(dev).long(), torch.from_numpy(val).to(dev)
    y = torch.zeros_like(x)
    for r in range(case["nrhs"]):
        y[r].index_add_(0, rows, val * x[r][col])
    if interior and op.info()[9] == 1:
        return y  # near-region only: the stored matrix is the operator
    o, h, N = op.grid()
    edge, coef, q, cen, area = _rwg(V, T)
    base = np.floor((cen - o) / h + 0.5).astype(np.int64) - 1
    g, w = np.polynomial.legendre.leggauss(5)
    g, w = 0.5 * (g + 1), 0.5 * w
    P = V[T]
    W = np.zeros((len(T), 27, 4))
    for i in range(5):
        for j in range(5):
            u, v = g[i], g[j] * (1 - g[i])
            r = P[:, 0] + u * (P[:, 1] - P[:, 0]) + v * (P[:, 2] - P[:, 0])
            t = (r - o) / h - base
            lag = [np.stack([(s - 1) * (s - 2) / 2, s * (2 - s), s * (s - 1) / 2], axis=1) for s in t.T]
            ll = (lag[2][:, :, None, None] * lag[1][:, None, :, None] * lag[0][:, None, None, :]).reshape(len(T), 27)
            ll = ll * (2 * area * (1 - u) * w[i] * w[j])[:, None]
            W[:, :, 0] += ll
            W[:, :, 1:] += ll[:, :, None] * (r - cen)[:, None, :]
    off = np.stack(np.meshgrid(np.arange(3), np.arange(3), np.arange(3), indexing="ij"), axis=-1).reshape(27, 3)[:, ::-1]
    n3 = base[:, None, :] + off[None]
    node = torch.from_numpy((n3[..., 2] * N[1] + n3[..., 1]) * N[0] + n3[..., 0]).to(dev)
    W, coef, q = (torch.from_numpy(a).to(dev) for a in (W, coef, q))
    edge = torch.from_numpy(edge).to(dev)
    shape, L = (int(N[2]), int(N[1]), int(N[0])), [2 * int(N[d]) for d in (2, 1, 0)]
    lags = [torch.from_numpy(np.where(np.arange(l) < l // 2, np.arange(l), np.arange(l) - l) * h).to(dev) for l in L]
    d = torch.meshgrid(*lags, indexing="ij")
    R = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
    R[0, 0, 0] = 1.0
    e = torch.exp(-1j * k * R) / (4 * math.pi * R)
    e[0, 0, 0] = 0
    if case["which"][0] == "L":
        spectra = [torch.fft.fftn(e)]
    else:
        e = -(1 + 1j * k * R) * e / (R * R)
        spectra = [torch.fft.fftn(e * d[2 - a]) for a in range(3)]
    del R, e, d

    def grid(values):
        f = torch.zeros(int(N.prod()), dtype=torch.complex128, device=dev)
        f.index_add_(0, node.reshape(-1), values.reshape(-1))
        return torch.fft.fftn(f.reshape(shape), s=L)

    def back(spectrum):
        return torch.fft.ifftn(spectrum)[:shape[0], :shape[1], :shape[2]].reshape(-1)[node]

    for r in range(case["nrhs"]):
        cx = coef * x[r][edge]
        alpha, beta = cx.sum(dim=1), (cx[:, :, None] * q).sum(dim=1)
        J = [grid(alpha[:, None] * W[:, :, 1 + a] + beta[:, a, None] * W[:, :, 0]) for a in range(3)]
        if case["which"][0] == "L":
            A = [back(spectra[0] * j) for j in J]
            phi = back(spectra[0] * grid(2 * alpha[:, None] * W[:, :, 0]))
            scalar = (-2.0 / (k * k)) * (phi * W[:, :, 0]).sum(dim=1)
        else:
            A = [back(spectra[(a + 1) % 3] * J[(a + 2) % 3] - spectra[(a + 2) % 3] * J[(a + 1) % 3]) for a in range(3)]
            scalar = 0.0
        s1 = sum((A[a] * W[:, :, 1 + a]).sum(dim=1) for a in range(3)) + scalar
        t0 = torch.stack([(A[a] * W[:, :, 0]).sum(dim=1) for a in range(3)], dim=1)
        out = coef * (s1[:, None] + (q * t0[:, None, :]).sum(dim=2))
        y[r].index_add_(0, edge.reshape(-1), out.reshape(-1))
    return y


def exact(case, seed):
    if case["kind"] == "product":
        return _exact_product(case, seed)
    if case["kind"] == "system":
        # the current rows need the direct integration of every near pair; the charge rows are a closed form
        mesh, V, T = _mesh(case)
        x = _vectors(mesh.ne + mesh.nt, 1, seed)[0]
        edge, coef = (torch.from_numpy(a).to(x.device) for a in _rwg(V, T)[:2])
        k0 = _wavenumber(case, False)
        return {"current": None, "charge": 2 * (coef * x[edge]).sum(dim=1) + 1j * k0 * x[mesh.ne:]}
    # solves and builds: direct integration of all near pairs again, minutes in plain torch
    return None
