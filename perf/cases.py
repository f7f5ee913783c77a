"""The charge-update workloads of the library as a calling program runs them, one pass each.

A molecular-dynamics or serving program keeps a context per electrode geometry (``CPM``) and calls it once
per time step or batch: the electrolyte potential b at every electrode site, then the electrode charges
q = S (G psi - b).  The cases cover that from the 216-site capacitor in FP64 to sixteen replicas of a
16,384-site one, the Ewald sum and P3M, the slab and wire boundaries, every S precision, and the set-up of a
new geometry.  Geometries and sizes are those of ``paper_2203_15461_gb300.systems`` and its benchmark.

The results of the single-precision paths (k_prec fp32 or f16x2) are accurate to about 1e-6; a program that
chose them passes them on as single precision, so their outputs are returned as float32.
"""
import math

import numpy as np
import torch

from paper_2203_15461_gb300 import systems
from paper_2203_15461_gb300.cpm import CPM

K_E = 14.399645   # e / (4 pi eps0 Angstrom) in volts
PSI = (0.0, 1.0)  # electrode potentials, V


# ----------------------------------------------------------------------------- the cases
def _case(name, kind, geom, cx, cy, layers, gap, alpha, m, charges, k_prec, s_prec, p3m=False, ragged=False):
    c = {"kind": kind, "geom": geom, "cx": cx, "cy": cy, "layers": layers, "gap": gap, "alpha": alpha, "m": m,
         "charges": charges, "k_prec": k_prec, "s_prec": s_prec, "p3m": p3m, "ragged": ragged}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one time step of the smallest capacitor at the library's default precision: launches and latency
        _case("tiny_fp64", "step", "gold", 6, 6, 3, 20.0, 0.3, 1, 100, "fp64", "fp64"),
        # 256 independent copies of it per captured step: many small systems at once
        _case("tiny_batch_256", "graph", "gold", 6, 6, 3, 20.0, 0.3, 256, 100, "f16x2", "fp32"),
        # a small server batch: four requests with different charge counts for a 512-site geometry
        _case("serve_512_4", "graph", "graphene", 8, 4, 2, 40.0, 0.3, 4, 1024, "f16x2", "fp32", ragged=True),
        # molecular dynamics of one 4,320-site capacitor from host buffers: copies in, step, copies out
        _case("md_host_4320", "host", "graphene", 18, 10, 3, 60.0, 0.2, 1, 5700, "f16x2", "fp32"),
        # eight replicas of it per captured step: the throughput workload of the benchmark
        _case("edl_batch_8", "graph", "graphene", 18, 10, 3, 60.0, 0.2, 8, 5700, "f16x2", "fp32"),
        # the same capacitor in FP64, one replica per step: reference runs
        _case("edl_fp64", "graph", "graphene", 18, 10, 3, 60.0, 0.2, 1, 5700, "fp64", "fp64"),
        # eight replicas with the mesh solver
        _case("edl_p3m_8", "graph", "graphene", 18, 10, 3, 60.0, 0.2, 8, 5700, "fp32", "fp32", p3m=True),
        # b for a server batch of sixteen requests on a large geometry, charge counts from 0.5 to 2 per site
        _case("serve_8192_16", "bvec", "graphene", 32, 16, 2, 40.0, 0.2, 16, 16384, "f16x2", "fp32", ragged=True),
        # the same on the largest geometry with the mesh solver
        _case("serve_p3m_16384_16", "bvec", "graphene", 32, 32, 2, 40.0, 0.15, 16, 32768, "fp32", "fp32", p3m=True,
              ragged=True),
        # co-axial nanotubes with ions between them, periodic along the axis only (wire boundary)
        _case("wire_tubes_4", "graph", "tubes", 10, 20, 10, 0.0, 0.3, 4, 96, "f16x2", "fp32"),
        # a new electrode geometry: A assembled, inverted and projected
        _case("setup_2048", "setup", "graphene", 16, 8, 2, 40.0, 0.3, 1, 0, "fp32", "fp32"),
        # the charge update alone for many replicas: S against 64 potential vectors on the tensor cores
        _case("product_4320_64", "product", "graphene", 18, 10, 3, 60.0, 0.2, 64, 0, "fp32", "bf16x3", p3m=True),
    ]


def draw(rng):
    """One more case of the ranges above: odd plate sizes, layer and replica counts, charge counts."""
    kind = rng.choice(["step", "graph", "graph", "graph", "host", "bvec", "setup", "product"])
    geom = rng.choice(["gold", "graphene", "graphene", "graphene", "tubes"])
    if geom == "gold":
        cx, cy, layers, gap, alpha = rng.randint(5, 11), 2 * rng.randint(3, 5), rng.randint(1, 4), rng.uniform(18, 40), 0.3
        n = 2 * layers * cx * cy
    elif geom == "graphene":
        cx, cy, layers, gap = rng.randint(8, 18), rng.randint(5, 10), rng.randint(1, 3), rng.uniform(30, 60)
        if kind == "setup":   # no larger than the listed one
            cx, cy, layers = min(cx, 16), min(cy, 8), min(layers, 2)
        alpha = rng.choice([0.2, 0.25, 0.3]) if cx * cy < 120 else 0.2
        n = 8 * layers * cx * cy
    else:
        cx, cy, layers, gap, alpha = 10, 20, rng.randint(5, 14), 0.0, 0.3
        n = 120 * layers
    m = int(round(math.exp(rng.uniform(0.0, math.log(24.0)))))
    if geom == "tubes":
        charges = 2 * rng.randint(8, 5 * layers)
    else:
        charges = int(n * math.exp(rng.uniform(math.log(0.3), math.log(1.5))))
        charges = 2 * (max(40, min(charges, int(0.02 * gap * _area(geom, cx, cy)))) // 2)
    k_prec, s_prec = rng.choice([("fp64", "fp64"), ("fp32", "fp32"), ("f16x2", "fp32"), ("f16x2", "fp32"),
                                 ("f16x2", "bf16x3")])
    p3m = geom != "tubes" and rng.random() < 0.25
    if kind == "setup":
        p3m = False
    if kind == "product":
        m, p3m = int(round(math.exp(rng.uniform(0.0, math.log(96.0))))), False
        s_prec = rng.choice(["fp64", "fp32", "bf16x3", "bf16x3"])
        k_prec = "fp64" if s_prec == "fp64" else "fp32"
    if k_prec == "fp64":
        m = min(m, 3)
    if p3m and k_prec == "f16x2":
        k_prec = "fp32"
    return _case(None, kind, geom, cx, cy, layers, round(gap, 2), alpha, m, 0 if kind in ("setup", "product") else charges,
                 k_prec, s_prec, p3m, ragged=kind in ("graph", "bvec") and rng.random() < 0.5)


def _area(geom, cx, cy):
    if geom == "gold":
        a = 4.08 / math.sqrt(2.0)
        return cx * a * cy * a * math.sqrt(3.0) / 2.0
    return cx * math.sqrt(3.0) * 1.42 * cy * 3.0 * 1.42


# ----------------------------------------------------------------------------- inputs
def _electrodes(case):
    if case["geom"] == "gold":
        el = systems.au111_slab(seed_layers=case["layers"], nx=case["cx"], ny=case["cy"], gap=case["gap"],
                                alpha=case["alpha"], rcut=3.6 / case["alpha"])
    elif case["geom"] == "graphene":
        el = systems.graphene_plates(case["cx"], case["cy"], case["layers"], case["gap"], alpha=case["alpha"],
                                     rcut=3.6 / case["alpha"])
    else:
        el = systems.coaxial_tubes(case["layers"], case["cx"], case["cy"], alpha=case["alpha"],
                                   rcut=3.6 / case["alpha"])
    return systems.with_p3m(el, matrix=True) if case["p3m"] else el


def _sites_of_lattice(rng, count, lx, ly, z0, z1, jitter=0.35):
    """count points of a jittered lattice that fills the box (periodic in x and y)."""
    h = (lx * ly * (z1 - z0) / count) ** (1.0 / 3.0)
    while True:
        nx, ny, nz = max(1, int(lx / h)), max(1, int(ly / h)), max(1, int((z1 - z0) / h))
        if nx * ny * nz >= count:
            break
        h *= 0.99
    at = rng.permutation(nx * ny * nz)[:count]
    p = np.stack([at % nx, (at // nx) % ny, at // (nx * ny)], axis=1) + 0.5
    cell = np.array([lx / nx, ly / ny, (z1 - z0) / nz])
    return p * cell + np.array([0.0, 0.0, z0]) + rng.uniform(-jitter, jitter, (count, 3))


def _electrolyte(case, el, rng, count):
    """count charges in the gap: rigid three-site waters and about 5 % ions (the gold capacitor and the tubes:
    ions alone)."""
    if case["geom"] == "tubes":   # on the cylinder half way between the walls
        r = 0.5 * (systems.tube_radius(case["cx"]) + systems.tube_radius(case["cy"]))
        lz = float(el.box[2])
        nth = int(2.0 * math.pi * r / 3.2)
        nz = max(1, int(lz / 3.2))
        at = rng.permutation(nth * nz)[:count]
        th = (at % nth + 0.5) * (2.0 * math.pi / nth)
        rr = r + rng.uniform(-0.6, 0.6, len(at))
        xyz = np.stack([el.box[0] / 2 + rr * np.cos(th), el.box[1] / 2 + rr * np.sin(th),
                        (at // nth + 0.5) * (lz / nz) + rng.uniform(-0.3, 0.3, len(at))], axis=1)
        return xyz, np.where(np.arange(len(at)) % 2 == 0, 1.0, -1.0)
    z0, z1 = el.z_inner[0] + 2.5, el.z_inner[1] - 2.5
    if case["geom"] == "gold":
        xyz = _sites_of_lattice(rng, count, el.box[0], el.box[1], z0, z1)
        return xyz, np.where(np.arange(count) < count // 2, 1.0, -1.0)
    ions = 2 * max(1, count // 40)
    while (count - ions) % 3 or ions % 2:
        ions += 1
    water = (count - ions) // 3
    c = _sites_of_lattice(rng, water + ions, el.box[0], el.box[1], z0, z1)
    o = c[:water]
    u = rng.normal(size=(2, water, 3))
    u[0] /= np.linalg.norm(u[0], axis=1)[:, None]
    u[1] -= np.einsum("ij,ij->i", u[1], u[0])[:, None] * u[0]
    u[1] /= np.linalg.norm(u[1], axis=1)[:, None]
    t = math.radians(109.47)
    xyz = np.concatenate([o, o + u[0], o + math.cos(t) * u[0] + math.sin(t) * u[1], c[water:]])
    q = np.concatenate([np.full(water, -0.8476), np.full(2 * water, 0.4238), np.where(np.arange(ions) % 2 == 0, 1.0, -1.0)])
    return xyz, q


def _inputs(case, seed, el):
    """Positions (m, n_e, 3) and charges (m, n_e), padded with zero charges where the counts differ, or, for the
    charge update alone, potentials b (m, n)."""
    rng = np.random.default_rng([int(seed), 7])
    m = case["m"]
    if case["kind"] == "product":
        z = (el.xyz[:, 2] - el.xyz[:, 2].mean()) / 30.0
        return rng.normal(0.0, 0.4, (m, el.n)) + rng.normal(0.0, 1.0, (m, 1)) * z
    count = [case["charges"]] * m
    if case["ragged"]:   # between a quarter of the largest and the largest
        count = [int(case["charges"] * (0.25 + 0.75 * r / max(1, m - 1))) for r in range(m)]
    got = [_electrolyte(case, el, rng, k) for k in count]
    ne = max(len(q) for _, q in got)
    xyz, q = np.zeros((m, ne, 3)), np.zeros((m, ne))
    for r, (x, c) in enumerate(got):
        xyz[r, : len(c)], q[r, : len(c)] = x, c
    return xyz, q


_stream = None


def _work_stream():
    """The one stream of the program: contexts that use captured steps need a stream of their own."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def prepare(case, seed):
    st = _work_stream()
    el = _electrodes(case)
    s = {"case": case, "el": el, "stream": st}
    dev = {"device": "cuda", "dtype": torch.float64}
    if case["kind"] == "setup":   # a geometry of its own for each seed: the plates a little strained
        rng = np.random.default_rng([int(seed), 3])
        f = 1.0 + rng.uniform(-0.005, 0.005, 2)
        xyz, box = el.xyz.copy(), el.box.copy()
        xyz[:, :2] *= f
        box[:2] *= f
        s["box"] = box
        s["xyz"] = torch.as_tensor(xyz, **dev)
        s["eta"] = torch.as_tensor(el.eta, **dev)
        s["group"] = torch.as_tensor(el.group, device="cuda")
        s["out"] = [torch.empty((el.n, el.n), **dev), torch.empty((el.n, el.n), **dev)]
        s["ctx"] = CPM(box, el.boundary, el.alpha, el.rcut, el.kcut, s_prec=case["s_prec"], k_prec=case["k_prec"], stream=st)
        return s
    m, n = case["m"], el.n
    with torch.cuda.stream(st):
        ctx = CPM.for_electrodes(el, s_prec=case["s_prec"], k_prec=case["k_prec"], stream=st)
        if case["kind"] == "bvec":
            site = torch.as_tensor(el.xyz, **dev), torch.as_tensor(el.eta, **dev), torch.as_tensor(el.group, device="cuda")
            ctx.cpm_prepare(*site, el.n_groups)
        else:
            ctx.setup(el)
            ctx.cpm_release_assembly()
        s["ctx"] = ctx
        psi = np.tile(np.asarray(PSI), (m, 1))
        if case["kind"] == "product":
            s["b"] = torch.as_tensor(_inputs(case, seed, el), **dev)
            s["psi"], s["q"] = torch.as_tensor(psi, **dev), torch.empty((m, n), **dev)
            if case["s_prec"] == "bf16x3":
                ctx.cpm_gemm_plan(m)   # tuned once per geometry and replica count
        elif case["kind"] == "host":
            xyz, q = _inputs(case, seed, el)
            s["ne"] = q.shape[1]
            for k, v in (("xyz", xyz), ("Q", q), ("psi", psi), ("q", np.zeros((m, n)))):
                s[k] = torch.as_tensor(np.ascontiguousarray(v)).pin_memory()
        else:
            xyz, q = _inputs(case, seed, el)
            s["ne"] = q.shape[1]
            s["xyz"], s["Q"] = torch.as_tensor(xyz, **dev), torch.as_tensor(q, **dev)
            s["psi"] = torch.as_tensor(psi, **dev)
            s["b"], s["q"] = torch.empty((m, n), **dev), torch.empty((m, n), **dev)
            if case["s_prec"] == "bf16x3" and case["kind"] != "bvec":
                ctx.cpm_gemm_plan(m)
    return s


# ----------------------------------------------------------------------------- one pass
def run(s):
    case, ctx, m = s["case"], s["ctx"], s["case"]["m"]
    kind = case["kind"]
    if kind == "host":
        ctx.cpm_step_host(m, s["ne"], s["xyz"], s["Q"], s["psi"], s["q"])
        return {"q": s["q"] if case["k_prec"] == "fp64" else s["q"].float()}
    with torch.cuda.stream(s["stream"]):
        if kind == "setup":
            ctx.cpm_assemble(s["xyz"], s["eta"], s["group"], s["el"].n_groups)
            ctx._check(ctx.lib.cpm_get_matrix(ctx.handle, 0, s["out"][0].data_ptr()))
            ctx.cpm_invert()
            ctx._check(ctx.lib.cpm_get_matrix(ctx.handle, 1, s["out"][1].data_ptr()))
            return {"A": s["out"][0], "S": s["out"][1]}
        if kind == "step":
            ctx.cpm_bvec(m, s["ne"], s["xyz"], s["Q"], s["b"])
            ctx.cpm_update(m, s["psi"], s["b"], s["q"])
        elif kind == "graph":
            ctx.cpm_step_graph(m, s["ne"], s["xyz"], s["Q"], s["psi"], s["b"], s["q"])
        elif kind == "bvec":
            ctx.cpm_bvec(m, s["ne"], s["xyz"], s["Q"], s["b"])
        else:
            ctx.cpm_update(m, s["psi"], s["b"], s["q"])
        out = {} if kind == "product" else {"b": s["b"]}
        if kind != "bvec":
            out["q"] = s["q"]
        return out if case["k_prec"] == "fp64" else {k: v.float() for k, v in out.items()}


# ----------------------------------------------------------------------------- the least a pass has to do
def work(case):
    """Bytes: positions, charges, potentials and sites in, b and q out, S once.  Operations: the reciprocal sum as
    two real multiply-adds per (charge, k), the pairs inside the cut-off at ten, the S product at one per entry;
    the set-up: the real-space pairs, one multiply-add per (pair of sites, column of k), factor and inverse."""
    el = _electrodes(case)
    n, m = el.n, case["m"]
    s_bytes = 8 if case["s_prec"] == "fp64" else 4
    vol = float(np.prod(el.box))
    if case["kind"] == "setup":
        cols = (el.box[0] * el.box[1] / (4.0 * math.pi ** 2)) * math.pi * el.kcut ** 2 / 2.0
        return {"bytes": 2.0 * 8 * n * n, "flops": n * n * cols + n ** 3}
    if case["kind"] == "product":
        return {"bytes": s_bytes * n * n + 2 * 8.0 * n * m, "flops": 2.0 * n * n * m}
    count = [case["charges"]] * m
    if case["ragged"]:
        count = [int(case["charges"] * (0.25 + 0.75 * r / max(1, m - 1))) for r in range(m)]
    ne = float(sum(count))
    nk = (4.0 / 3.0) * math.pi * el.kcut ** 3 * vol / (2.0 * (2.0 * math.pi) ** 3)
    gap_vol = _area(case["geom"], case["cx"], case["cy"]) * case["gap"] if case["geom"] != "tubes" else 4000.0 * case["layers"] / 10
    pairs = ne * n * min(1.0, 0.35 * (4.0 / 3.0) * math.pi * el.rcut ** 3 / max(gap_vol, 1.0))
    recip = 30.0 * 343 * (ne + n * m) if case["p3m"] else 4.0 * ne * nk
    full = case["kind"] != "bvec"
    return {"bytes": 32.0 * ne + 40.0 * n + 8.0 * n * m * (2 if full else 1) + (s_bytes * n * n if full else 0),
            "flops": recip + 10.0 * pairs + (2.0 * n * n * m if full else 0.0)}


# ----------------------------------------------------------------------------- the same in plain FP64
def _kset(el, device):
    """Half-space vectors 0 < |k| <= kcut and their Ewald weights."""
    L = [float(v) for v in el.box]
    t = [(2.0 * math.pi) / v for v in L]
    N = [int(el.kcut / v) + 1 for v in t]
    ax = [torch.arange(-v, v + 1, device=device) for v in N]
    nx, ny, nz = torch.meshgrid(*ax, indexing="ij")
    half = (nx > 0) | ((nx == 0) & (ny > 0)) | ((nx == 0) & (ny == 0) & (nz > 0))
    k = [a.double() * w for a, w in zip((nx, ny, nz), t)]
    k2 = (k[0] * k[0] + k[1] * k[1]) + k[2] * k[2]
    keep = half & (k2 <= el.kcut * el.kcut)
    k2 = k2[keep]
    V = L[0] * L[1] * L[2]
    w = (8.0 * math.pi / V) * torch.exp(-k2 / (4.0 * el.alpha ** 2)) / k2
    return torch.stack([a[keep] for a in (nx, ny, nz)], 1), w


def _phase(n, xyz, box):
    """cos and sin of 2 pi n . (x / L), the turns reduced before the product is scaled."""
    f = xyz / box
    f = f - torch.floor(f)
    turns = n.double() @ f.T
    turns = (turns - torch.round(turns)) * (2.0 * math.pi)
    return torch.cos(turns), torch.sin(turns)


def _images(el, reach):
    """Shifts by whole periods that can bring a pair whose differences are reduced to half a period within reach."""
    r = [range(-k, k + 1) for k in (int(math.floor(reach / float(v) + 0.5)) for v in el.box)]
    return [(a, b, c) for a in r[0] for b in r[1] for c in r[2]]


def _exact_b(el, xyz, Q):
    dev = xyz.device
    box = torch.as_tensor(el.box, device=dev, dtype=torch.float64)
    R = torch.as_tensor(el.xyz, device=dev, dtype=torch.float64)
    eta = torch.as_tensor(el.eta, device=dev, dtype=torch.float64)[:, None]
    V = float(np.prod(el.box))
    kn, kw = _kset(el, dev)
    shifts = _images(el, el.rcut)
    out = []
    for x, q in zip(xyz, Q):
        x, q = x[q != 0], q[q != 0]
        b = torch.zeros(el.n, device=dev, dtype=torch.float64)
        for i0 in range(0, el.n, 1024):
            Ri, acc = R[i0:i0 + 1024], 0.0
            d = [Ri[:, a:a + 1] - x[None, :, a] for a in range(3)]
            d = [v - box[a] * torch.round(v / box[a]) for a, v in enumerate(d)]
            for s in shifts:
                r = sum((d[a] + s[a] * box[a]) ** 2 for a in range(3)).sqrt()
                if not bool((r < el.rcut).any()):
                    continue
                f = (torch.erfc(el.alpha * r) - torch.erfc(eta[i0:i0 + 1024] * r)) / r
                acc = acc + torch.where(r < el.rcut, f, torch.zeros_like(f)) @ q
            b[i0:i0 + 1024] = acc
        step = max(64, int(2.5e8 / max(len(q), el.n)))
        for k0 in range(0, len(kw), step):
            c, s = _phase(kn[k0:k0 + step], x, box)
            rc, rs = (c @ q) * kw[k0:k0 + step], (s @ q) * kw[k0:k0 + step]
            c, s = _phase(kn[k0:k0 + step], R, box)
            b += rc @ c + rs @ s
        b += -math.pi * q.sum() / (V * el.alpha ** 2)
        if el.boundary == "slab":
            b += (4.0 * math.pi / V) * R[:, 2] * (q * x[:, 2]).sum()
        elif el.boundary == "wire":
            b += (2.0 * math.pi / V) * (R[:, 0] * (q * x[:, 0]).sum() + R[:, 1] * (q * x[:, 1]).sum())
        out.append(K_E * b)
    return torch.stack(out)


def _exact_A(el, xyz, dev):
    box = torch.as_tensor(el.box, device=dev, dtype=torch.float64)
    R = torch.as_tensor(xyz, device=dev, dtype=torch.float64)
    e = torch.as_tensor(el.eta, device=dev, dtype=torch.float64)
    n, V = el.n, float(np.prod(el.box))
    A = torch.zeros((n, n), device=dev, dtype=torch.float64)
    shifts = _images(el, el.rcut)
    for i0 in range(0, n, 1024):
        i1 = min(n, i0 + 1024)
        d = [R[i0:i1, a:a + 1] - R[None, :, a] for a in range(3)]
        d = [v - box[a] * torch.round(v / box[a]) for a, v in enumerate(d)]
        eij = e[i0:i1, None] * e[None, :] / torch.sqrt(e[i0:i1, None] ** 2 + e[None, :] ** 2)
        for s in shifts:
            r = sum((d[a] + s[a] * box[a]) ** 2 for a in range(3)).sqrt()
            inside = (r < el.rcut) & (r > 0)
            rr = torch.where(inside, r, torch.ones_like(r))
            f = (torch.erfc(el.alpha * rr) - torch.erfc(eij * rr)) / rr
            A[i0:i1] += torch.where(inside, f, torch.zeros_like(f))
    kn, kw = _kset(el, dev)
    step = max(64, int(1.5e8 / n))
    for k0 in range(0, len(kw), step):
        c, s = _phase(kn[k0:k0 + step], R, box)
        w = kw[k0:k0 + step, None]
        A += (c * w).T @ c + (s * w).T @ s
    A.diagonal().add_((math.sqrt(2.0) * e - 2.0 * el.alpha) / math.sqrt(math.pi))
    A += -math.pi / (V * el.alpha ** 2)
    if el.boundary == "slab":
        A += (4.0 * math.pi / V) * torch.outer(R[:, 2], R[:, 2])
    elif el.boundary == "wire":
        A += (2.0 * math.pi / V) * (torch.outer(R[:, 0], R[:, 0]) + torch.outer(R[:, 1], R[:, 1]))
    return K_E * A


def _exact_S(A):
    inv = torch.cholesky_inverse(torch.linalg.cholesky(A))
    d = inv.sum(1)
    return inv - torch.outer(d, d) / d.sum()


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    el = _electrodes(case)
    if case["kind"] == "setup":
        rng = np.random.default_rng([int(seed), 3])
        f = 1.0 + rng.uniform(-0.005, 0.005, 2)
        xyz, box = el.xyz.copy(), el.box.copy()
        xyz[:, :2] *= f
        box[:2] *= f
        el.box = box
        A = _exact_A(el, xyz, dev)
        return {"A": A, "S": _exact_S(A)}
    out = {}
    if case["kind"] == "product":
        b = torch.as_tensor(_inputs(case, seed, el), device=dev)
    else:
        xyz, Q = _inputs(case, seed, el)
        b = _exact_b(el, torch.as_tensor(xyz, device=dev), torch.as_tensor(Q, device=dev))
        if case["kind"] != "host":
            out["b"] = b
    if case["kind"] == "bvec":
        return out
    S = _exact_S(_exact_A(el, el.xyz, dev))
    v = torch.as_tensor(np.asarray(PSI)[el.group], device=dev)
    out["q"] = (v[None, :] - b) @ S
    return out
