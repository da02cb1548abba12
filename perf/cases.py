"""The work that users of this framework have it do, as measurable cases.

Every case is one call (or the few calls a program makes together) through the public
binding: operator applies in each precision and storage, solves by the solvers programs
use, and a structure taken from host coordinates to its spectrum.  Structures are the
framework's own families (graphene flakes and disks, armchair nanotubes, fcc sodium
spheres, BEM spheroids), displaced or thinned by the seed as relaxed or defective samples
are; sizes are those of its workloads, tests and serving pool.
"""
import math

import numpy as np
import torch

from paper_2103_00438_gb300 import structures as S
from paper_2103_00438_gb300 import wfq

STORES = {"fp64": wfq.STORE_FP64, "bf16": wfq.STORE_BF16X2, "pairs": wfq.STORE_F32X2,
          "sym": wfq.STORE_F32X2_SYM, "none": 0}
PRECS = {"fp64": wfq.PREC_FP64, "mixed": wfq.PREC_MIXED, "df": wfq.PREC_DF, "fmm": wfq.PREC_FMM}
# bytes of one stored entry of D
ENTRY_BYTES = {"fp64": 8, "bf16": 4, "pairs": 8, "sym": 4, "none": 0}
# Krylov steps a solve takes to 1e-8 (flakes: 1e-10), about, by family over its band
STEPS = {"flake": 50, "tube": 110, "sphere": 160, "spheroid": 30}
# frequency band of each family, eV
BANDS = {"flake": (0.3, 2.0), "tube": (0.05, 2.0), "sphere": (0.9, 1.8), "disk": (0.05, 0.20),
         "spheroid": (2.0, 4.5)}
NM = 10.0 * S.BOHR_PER_ANGSTROM


def listed():
    return [
        # One operator apply in plain FP64 of the 1014-atom flake (the smallest structure):
        # what an external FP64 Krylov code calls once per step.  Latency and launches.
        {"name": "apply_fp64_flake1k", "kind": "apply", "shape": "flake", "size": 13, "store": "fp64",
         "prec": "fp64", "cols": 1},
        # The plain method: the same flake at one frequency of its plasmon band, field along
        # x, unrestarted FP64 GMRES to 1e-10.  A chain of small dependent kernels.
        {"name": "gmres_fp64_flake1k", "kind": "gmres", "shape": "flake", "size": 13, "store": "fp64",
         "nfreq": 1, "ndir": 1, "tol": 1e-10},
        # A mixed-precision block apply of a 5046-atom flake, 8 frequencies x 3 directions:
        # one inner step of a served request on a middle-sized structure.
        {"name": "apply_mixed_flake5k", "kind": "apply", "shape": "flake", "size": 29, "store": "bf16",
         "prec": "mixed", "cols": 24},
        # The mixed block apply of the 20000-atom tube with all 64 x 3 columns: the product of
        # block GMRES and QMR.
        {"name": "apply_mixed_cnt20k", "kind": "apply", "shape": "tube", "size": 500, "store": "bf16",
         "prec": "mixed", "cols": 192},
        # The double-float apply of the same block: the true residual of every refinement
        # cycle of the mixed solvers.
        {"name": "apply_df_cnt20k", "kind": "apply", "shape": "tube", "size": 500, "store": "pairs",
         "prec": "df", "cols": 192},
        # The FP64 apply of a block of 16 columns on a 10k-atom sodium sphere (long rows of the
        # neighbour term): the product of plain FP64 block solves.
        {"name": "apply_fp64_sphere10k", "kind": "apply", "shape": "sphere", "size": 10000, "store": "fp64",
         "prec": "fp64", "cols": 16},
        # The flagship: 64 frequencies x 3 directions of the 20000-atom tube by shifted GMRES
        # to 1e-8, with the polarizabilities and cross sections.
        {"name": "shifted_cnt20k", "kind": "shifted", "shape": "tube", "size": 500, "store": "pairs",
         "nfreq": 64, "ndir": 3, "tol": 1e-8},
        # The sodium sphere's 32 x 3 columns from the symmetric tiles (the storage of the
        # largest stored structures, where the full planes do not fit beside anything else).
        {"name": "shifted_sphere15k", "kind": "shifted", "shape": "sphere", "size": 15000, "store": "sym",
         "nfreq": 32, "ndir": 3, "tol": 1e-8},
        # The matrix-free mixed apply, 16 frequencies x 1 direction, of the disk family where
        # D is no longer stored.
        {"name": "apply_mf_disk100k", "kind": "apply", "shape": "disk", "size": 58.0, "store": "none",
         "prec": "mixed", "cols": 16},
        # The fast-multipole apply of a quarter-million-atom disk, order 6, 16 columns: the
        # inner product of the largest solves.
        {"name": "apply_fmm_disk250k", "kind": "apply", "shape": "disk", "size": 92.0, "store": "none",
         "prec": "fmm", "cols": 16, "order": 6},
        # A new structure from host coordinates: geometry build, 16 frequencies x 3 directions,
        # polarizabilities.  What a program that walks over many structures pays per structure.
        {"name": "build_solve_cnt10k", "kind": "build", "shape": "tube", "size": 250, "store": "pairs",
         "nfreq": 16, "ndir": 3, "tol": 1e-8},
        # The continuum (BEM) operator on a spheroid's surface, a spectrum of 64 x 3 columns.
        {"name": "bem_spheroid12k", "kind": "shifted", "shape": "spheroid", "size": 12000, "store": "fp64+pairs",
         "nfreq": 64, "ndir": 3, "tol": 1e-8},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """A case of the same ranges: any of the listed kinds, sizes spread over their logarithm."""
    kind = rng.choice(["fp64", "gmres", "mixed", "mixed", "df", "shifted", "shifted", "mf", "fmm", "build", "bem"])
    if kind in ("fp64", "mixed", "df"):
        top = {"fp64": 10000, "mixed": 20000, "df": 20000}[kind]
        shape, size = _draw_shape(rng, 600, top)
        store = {"fp64": "fp64", "mixed": "bf16", "df": rng.choice(["pairs", "pairs", "fp64"])}[kind]
        cols = max(1, int(round(_log(rng, 1, 16 if kind == "fp64" else 192))))
        return {"kind": "apply", "shape": shape, "size": size, "store": store, "prec": kind, "cols": cols}
    if kind == "gmres":
        return {"kind": "gmres", "shape": "flake", "size": rng.randint(8, 18), "store": "fp64",
                "nfreq": rng.randint(1, 4), "ndir": rng.randint(1, 2), "tol": 1e-10}
    if kind in ("shifted", "build"):
        shape, size = _draw_shape(rng, 900, 20000 if kind == "shifted" else 10000)
        store = rng.choice(["pairs", "pairs", "sym", "fp64"]) if kind == "shifted" else "pairs"
        return {"kind": kind, "shape": shape, "size": size, "store": store,
                "nfreq": max(1, int(round(_log(rng, 1, 64 if kind == "shifted" else 16)))),
                "ndir": rng.randint(1, 2 if shape == "flake" else 3), "tol": 1e-8}
    if kind == "mf":
        return {"kind": "apply", "shape": "disk", "size": round(_log(rng, 20.0, 57.0), 1), "store": "none",
                "prec": "mixed", "cols": max(1, int(round(_log(rng, 2, 16))))}
    if kind == "fmm":
        cols = max(1, int(round(_log(rng, 1, 16))))
        if rng.random() < 0.3:
            return {"kind": "apply", "shape": "sphere", "size": int(_log(rng, 5000, 30000)), "store": "none",
                    "prec": "fmm", "cols": cols, "order": rng.randint(3, 5)}
        return {"kind": "apply", "shape": "disk", "size": round(_log(rng, 20.0, 91.0), 1), "store": "none",
                "prec": "fmm", "cols": cols, "order": rng.randint(4, 7)}
    return {"kind": "shifted", "shape": "spheroid", "size": int(_log(rng, 1500, 12000)), "store": "fp64+pairs",
            "nfreq": max(1, int(round(_log(rng, 1, 64)))), "ndir": rng.randint(1, 3), "tol": 1e-8}


def _draw_shape(rng, lo, hi):
    n = _log(rng, lo, hi)
    shape = rng.choice(["flake", "tube", "sphere"])
    if shape == "flake":
        return shape, max(10, int(math.sqrt(n / 6.0)))
    if shape == "tube":
        return shape, max(15, int(n / 40.0))
    return shape, int(n)


# ------------------------------------------------------------------ inputs

def _structure(case, seed):
    """Positions (n x 3 bohr, or a surface) and parameters of a case.  Flakes and tubes carry
    a seeded displacement of up to 0.01 A per coordinate (in the plane for flakes), spheres
    the seeded surface jitter of the sodium workload, disks 1% seeded vacancies, spheroids a
    seeded scale."""
    rng = np.random.default_rng([seed, 1])
    shape, size = case["shape"], case["size"]
    amp = 0.01 * S.BOHR_PER_ANGSTROM
    if shape == "flake":
        xyz = S.honeycomb_flake(size)
        xyz[:, :2] += rng.uniform(-amp, amp, (len(xyz), 2))
        return xyz, S.carbon_params(1.51)
    if shape == "tube":
        xyz = S.nanotube(10, 10, size)
        return xyz + rng.uniform(-amp, amp, xyz.shape), S.carbon_params(1.04)
    if shape == "sphere":
        a = 4.23
        return S.fcc_sphere(a, S.fcc_sphere_radius_for(size, a), 0.05, seed=seed), S.sodium_params()
    if shape == "disk":
        return S.graphene_disk(size, vacancy_frac=0.01, seed=seed), S.carbon_params(1.84)
    scale = rng.uniform(0.9, 1.1)
    return S.spheroid_surface(size, 20.0 * NM * scale, 10.0 * NM * scale), S.drude_metal_params()


def _atoms(case):
    """Atoms (elements) of a case, without the seed."""
    shape, size = case["shape"], case["size"]
    if shape == "flake":
        return 6 * size * size
    if shape == "tube":
        return 40 * size
    if shape == "disk":   # two atoms per cell of the honeycomb lattice, 1% removed
        a = S.GRAPHENE_A_ANG
        return int(0.99 * math.pi * (5.0 * size) ** 2 / (a * a * math.sqrt(3.0) / 4.0))
    return size


def _omega(case, seed, count):
    lo, hi = BANDS[case["shape"]]
    return S.ev(np.sort(np.random.default_rng([seed, 2]).uniform(lo, hi, count)))


def _x(case, seed, n):
    """A block of complex columns as Krylov vectors are: standard normal, made on the GPU."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 17)
    dt = torch.complex64 if case["prec"] in ("mixed", "fmm") else torch.complex128
    return torch.randn((n, case["cols"]), dtype=dt, device="cuda", generator=gen)


def _store(case):
    flags = 0
    for s in case["store"].split("+"):
        flags |= STORES[s]
    return flags


_context = []


def _ctx():
    """One context per process, as a program keeps it."""
    if not _context:
        _context.append(wfq.Context(0))
    return _context[0]


def _geometry(case, geo, params):
    if case["shape"] == "spheroid":
        return wfq.BemGeometry(_ctx(), geo["xyz"], geo["normal"], geo["area"], geo["curvature"], params,
                               store=_store(case))
    return wfq.Geometry(_ctx(), geo, params, store=_store(case))


def prepare(case, seed):
    geo, params = _structure(case, seed)
    n = len(geo["xyz"]) if isinstance(geo, dict) else len(geo)
    st = {"case": case}
    if case["kind"] == "build":
        st.update(xyz=geo, params=params)
    else:
        st["g"] = _geometry(case, geo, params)
    if case["kind"] == "apply":
        if case["prec"] == "fmm":
            st["g"].fmm_build(case["order"])
        st["x"] = _x(case, seed, n)
        st["y"] = torch.empty_like(st["x"])
        st["omega"] = _omega(case, seed, case["cols"])
    else:
        st["omega"] = _omega(case, seed, case["nfreq"])
        st["dirs"] = np.eye(3)[:case["ndir"]]
        st["E0"] = float(np.random.default_rng([seed, 3]).uniform(0.5, 2.0)) * 1e-4
        st["q"] = torch.empty((n, case["nfreq"] * case["ndir"]), dtype=torch.complex128, device="cuda")
    return st


def run(st):
    case = st["case"]
    if case["kind"] == "apply":
        stream = torch.cuda.current_stream()
        return st["g"].apply(st["omega"], st["x"], st["y"], prec=PRECS[case["prec"]], stream=stream)
    g = _geometry(case, st["xyz"], st["params"]) if case["kind"] == "build" else st["g"]
    stream = torch.cuda.current_stream()
    if case["kind"] == "gmres":
        q, _, _ = g.solve_gmres(st["omega"], st["dirs"], st["E0"], m=0, rel_tol=case["tol"], max_iter=1000,
                                prec=wfq.PREC_FP64, out=st["q"], stream=stream)
    else:
        q, _, _ = g.solve_gmres_shifted(st["omega"], st["dirs"], st["E0"], rel_tol=case["tol"],
                                        prec=wfq.PREC_FP64 if case["shape"] == "spheroid" else wfq.PREC_MIXED,
                                        out=st["q"], stream=stream)
    alpha = g.polarizability(q, st["E0"], stream=stream)
    if case["kind"] == "build":
        g.close()
        return {"q": q, "alpha": alpha}
    sigma, sigma_iso = g.cross_section(st["omega"], st["dirs"], q, st["E0"], stream=stream)
    return {"q": q, "alpha": alpha, "sigma": sigma, "sigma_iso": sigma_iso}


def work(case):
    """D read once per product that has to follow another (its stored bytes; nothing where D is
    not stored), the vectors once, 2 flops per entry and real column."""
    n = float(_atoms(case))
    stored = case["store"].split("+")[-1]
    entry = ENTRY_BYTES[stored]
    if case["kind"] == "apply":
        c = case["cols"]
        vec = 8 if case["prec"] in ("mixed", "fmm") else 16
        if case["prec"] == "fmm":
            # tree passes: neighbour pairs and about 27 (2D) or 189 (3D) interaction boxes per leaf
            nodes = case["order"] ** (2 if case["shape"] == "disk" else 3)
            leaf, near, boxes = (20, 9, 36) if case["shape"] == "disk" else (40, 27, 216)
            flops = 2.0 * 2 * c * (n * leaf * near + n / leaf * boxes * nodes ** 2 + 4.0 * n * nodes)
            return {"bytes": 2 * vec * n * c + 40 * n, "flops": flops}
        return {"bytes": entry * n * n + 2 * vec * n * c, "flops": 4.0 * n * n * c}
    nc = case["nfreq"] * case["ndir"]
    if case["kind"] == "gmres":
        return {"bytes": entry * n * n + 16 * n * nc, "flops": STEPS["flake"] * 4.0 * n * n * nc}
    steps = STEPS[case["shape"]]
    # a D that fits the cache beside the vectors is read from memory once
    reads = steps if entry * n * n > 100e6 else 1
    extra = entry * n * n if case["kind"] == "build" else 0.0
    return {"bytes": reads * entry * n * n + extra + 16 * n * nc, "flops": steps * 2.0 * n * n * case["ndir"]}


# ------------------------------------------------------------------ 64-bit values

def _z(case, params, omega):
    """The complex shift of each frequency: Eq. 12, or -Lambda of Eq. 21 for a Drude particle."""
    w = np.asarray(omega)
    if case["shape"] == "spheroid":
        eps = params["eps_inf"] - params["omega_p"] ** 2 / (w * (w + 1j * params["gamma"]))
        z = -2.0 * np.pi * (params["eps_out"] + eps) / (params["eps_out"] - eps)
    else:
        z = -(w / (2.0 * params["n0"] * params["tau"])) * (w * params["tau"] + 1j)
    return torch.from_numpy(z).cuda()


def _d_rows(xyz, params, i0, i1):
    """Rows of D (Eq. 3) and of the neighbour conductance (Eq. 9), and the distances."""
    r = torch.zeros((i1 - i0, len(xyz)), dtype=torch.float64, device="cuda")
    for k in range(3):
        r += (xyz[i0:i1, k, None] - xyz[None, :, k]) ** 2
    r.sqrt_()
    idx = torch.arange(i0, i1, device="cuda")
    r[idx - i0, idx] = 1.0
    s = math.sqrt(2.0) * math.sqrt(2.0 / math.pi) / params["eta"]
    d = torch.special.erf(r / s).div_(r)
    d[idx - i0, idx] = params["eta"]
    return d, r, idx


def _k_rows(r, idx, i0, params):
    f = torch.sigmoid(-params["d_fermi"] * (r / (params["s_fermi"] * params["r0"]) - 1.0))
    f[f < params["cutoff_eps"]] = 0.0
    k = f.mul_(params["area"]).div_(r)
    k[idx - i0, idx] = 0.0
    return k


def _chunks(n):
    step = max(1, min(n, int(3e8) // n))
    return [(i, min(n, i + step)) for i in range(0, n, step)]


def _exact_apply(case, seed):
    geo, params = _structure(case, seed)
    xyz = torch.from_numpy(geo).cuda()
    n = len(geo)
    x = _x(case, seed, n).to(torch.complex128)
    xr = torch.view_as_real(x).reshape(n, -1)
    u = torch.empty_like(xr)
    for i0, i1 in _chunks(n):
        u[i0:i1] = _d_rows(xyz, params, i0, i1)[0] @ xr
    y = torch.empty_like(xr)
    for i0, i1 in _chunks(n):
        _, r, idx = _d_rows(xyz, params, i0, i1)
        k = _k_rows(r, idx, i0, params)
        y[i0:i1] = k @ u - k.sum(dim=1, keepdim=True) * u[i0:i1]
    z = _z(case, params, _omega(case, seed, case["cols"]))
    return torch.view_as_complex(y.reshape(n, -1, 2).contiguous()) - z * x


def _system(case, seed):
    """A (dense, real), the right-hand sides per unit field along each axis, and positions."""
    geo, params = _structure(case, seed)
    if case["shape"] == "spheroid":
        xyz, nrm = torch.from_numpy(geo["xyz"]).cuda(), torch.from_numpy(geo["normal"]).cuda()
        area, curv = torch.from_numpy(geo["area"]).cuda(), torch.from_numpy(geo["curvature"]).cuda()
        n = len(xyz)
        a = torch.empty((n, n), dtype=torch.float64, device="cuda")
        for i0, i1 in _chunks(n):
            idx = torch.arange(i0, i1, device="cuda")
            r2 = torch.zeros((i1 - i0, n), dtype=torch.float64, device="cuda")
            dot = torch.zeros_like(r2)
            for k in range(3):
                diff = xyz[i0:i1, k, None] - xyz[None, :, k]
                r2 += diff * diff
                dot += nrm[i0:i1, k, None] * diff
            r2[idx - i0, idx] = 1.0
            rows = area[i0:i1, None] * dot / (r2 * r2.sqrt())
            rows[idx - i0, idx] = curv[i0:i1] * (math.pi * area[i0:i1]).sqrt()
            a[i0:i1] = rows
        return a, -area[:, None] * nrm, xyz, params
    xyz = torch.from_numpy(geo).cuda()
    n = len(geo)
    d = torch.empty((n, n), dtype=torch.float64, device="cuda")
    k = torch.empty((n, n), dtype=torch.float64, device="cuda")
    for i0, i1 in _chunks(n):
        d[i0:i1], r, idx = _d_rows(xyz, params, i0, i1)
        k[i0:i1] = _k_rows(r, idx, i0, params)
    p = k.sum(dim=1)
    rhs = k @ xyz - p[:, None] * xyz          # sum_j (V_i - V_j) K_ij with V = -r . k
    ks = k.to_sparse_csr()
    del k

    def apply(v):
        u = d @ v
        return ks @ u - p[:, None] * u

    return apply, rhs, xyz, params


def _exact_solve(case, seed):
    """q = (A - z I)^-1 R from one real Arnoldi process per direction in FP64 (twice
    orthogonalised), run far past the tolerance of the solve, and what follows from q."""
    op, rhs, xyz, params = _system(case, seed)
    apply = op if callable(op) else (lambda v: op @ v)
    omega = _omega(case, seed, case["nfreq"])
    z = _z(case, params, omega)
    e0 = float(np.random.default_rng([seed, 3]).uniform(0.5, 2.0)) * 1e-4
    n, nf, nd = len(xyz), case["nfreq"], case["ndir"]
    q = torch.empty((n, nf, nd), dtype=torch.complex128, device="cuda")
    m = min(n - 1, 420)
    for d in range(nd):
        r = e0 * rhs[:, d]
        beta = torch.linalg.vector_norm(r)
        v = torch.zeros((m + 1, n), dtype=torch.float64, device="cuda")
        h = torch.zeros((m + 1, m), dtype=torch.float64, device="cuda")
        v[0] = r / beta
        for j in range(m):
            w = apply(v[j][:, None])[:, 0]
            for _ in range(2):
                c = v[:j + 1] @ w
                w = w - c @ v[:j + 1]
                h[:j + 1, j] += c
            h[j + 1, j] = torch.linalg.vector_norm(w)
            v[j + 1] = w / h[j + 1, j]
        eye = torch.eye(m + 1, m, dtype=torch.complex128, device="cuda")
        rhs1 = torch.zeros((m + 1, 1), dtype=torch.complex128, device="cuda")
        rhs1[0, 0] = beta
        for f in range(nf):
            qm, rm = torch.linalg.qr(h.to(torch.complex128) - z[f] * eye)
            y = torch.linalg.solve_triangular(rm, qm.mH @ rhs1, upper=True)[:, 0]
            q[:, f, d] = torch.complex(y.real @ v[:m], y.imag @ v[:m])
    q = q.reshape(n, nf * nd)
    alpha = (q.mT @ xyz.to(torch.complex128)) / e0
    out = {"q": q, "alpha": alpha.cpu().numpy()}
    if case["kind"] != "build":
        im = alpha.cpu().numpy().imag.reshape(nf, nd, 3)
        sig = np.stack([4.0 * np.pi * omega / S.C_AU * im[:, d, d] for d in range(nd)], axis=1)
        out.update(sigma=sig, sigma_iso=sig.mean(axis=1))
    return out


def exact(case, seed):
    """What run() returns, in 64 bits by plain torch: the operator row by row from its
    formulas, the solves from a long Arnoldi process."""
    if case["kind"] == "apply":
        return _exact_apply(case, seed)
    return _exact_solve(case, seed)
