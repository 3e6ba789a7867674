"""Timed cases of the solver: the calls of a self-consistent-field run, each through the public entry points.

A case is a dict of plain values; `kind` names the call and the other keys its sizes:

  filter    sdft_chebyshev_filter of one real FP32 orbital block (the step that most of an SCF's time goes to)
  kpass     one k-point's CheFSI pass without the eigensolve, on complex FP32 blocks: filter, H Y, subspace
            matrices, rotation
  multi     sdft_chebyshev_filter_multi over independent cells of uneven sizes
  subspace  sdft_subspace_matrices and sdft_rotate of one real FP32 block (the Rayleigh-Ritz products)
  poisson   sdft_poisson of a mixed-precision context, from a zero potential
  features  sdft_mlp_dataset: the descriptors of the learned starting density
  mlpgrad   sdft_mlp_loss_grad: one mini-batch's loss and gradient of its network
  move      sdft_move_atoms: the set-up of the next molecular-dynamics step, with the fields and projectors it
            rebuilds read back through sdft_get_pseudocharge, sdft_get_sad_density and one H X
  scf       sdft_scf for a fixed number of iterations from the superposition of atomic densities, with its results

Cells are simple-cubic (or body-centred, `basis` 2) lattices of `m1 x m2 x m3` sites at 5.13 bohr or so with
Gaussian displacements, or random positions at least 3 bohr apart (`natom`), on a grid of `n1 x n2 x n3` points of
spacing `h`; atom positions, potentials and blocks come from the seed.  Quantities that a mixed-precision call computes
in FP32 but stores as FP64 (subspace matrices, the results of a mixed SCF) are returned as FP32, the precision
they carry.
"""
import math

import numpy as np
import torch

import paper_2005_10431_gb300 as sd

DEV = "cuda"
H_MESH = 0.2565
SPACING = 5.13
SPECIES = [dict(Z=4.0, r_loc=0.5, r_proj=0.6, E_kb=1.0, r_cut_proj=3.0, sad_width=1.0)]
MLP_PARAMS = sd.SDFT_MLP_NPARAM
R = 6
FD = [-2.0 * sum(1.0 / (r * r) for r in range(1, R + 1))] + [
    2.0 * (-1) ** (r + 1) * math.factorial(R) ** 2 / (r * r * math.factorial(R - r) * math.factorial(R + r))
    for r in range(1, R + 1)]


def listed():
    lat64 = dict(n1=80, n2=80, n3=80, h=H_MESH, m1=4, m2=4, m3=4, basis=1)
    return [
        # the smallest SCF a user runs: two atoms, all FP64, every kernel a few microseconds; launches and host
        # synchronisations count
        dict(name="scf_two_atom_fp64", kind="scf", precision="fp64", n1=24, n2=24, n3=24, h=0.25, m1=1, m2=1, m3=1,
             basis=2, states=8, buffer=0, degree=12, iterations=8),
        # the benchmark's own loop: 64 atoms, mixed precision, 154 states and 26 buffer states; the first iterations
        dict(name="scf_lattice64", kind="scf", precision="mixed", **lat64, states=154, buffer=26, degree=20,
             iterations=5),
        # one filter of a small cell on an odd, non-cubic grid with atoms at random places
        dict(name="filter_uneven", kind="filter", n1=37, n2=41, n3=45, h=H_MESH, natom=8, states=20, degree=20),
        # the filter of the benchmark's 64-atom cell
        dict(name="filter_lattice64", kind="filter", **lat64, states=180, degree=20),
        # the largest cell: 216 atoms, 520 states
        dict(name="filter_lattice216", kind="filter", n1=120, n2=120, n3=120, h=H_MESH, m1=6, m2=6, m3=6, basis=1,
             states=520, degree=24),
        # one of the many k-points of an 8-atom cell
        dict(name="kpass_kpoint8", kind="kpass", n1=40, n2=40, n3=40, h=H_MESH, m1=2, m2=2, m3=2, basis=1, states=20,
             degree=20, k1=0.375, k2=-0.125, k3=0.125),
        # a batch of independent small cells of uneven sizes, 24 to 48 points an edge, 2 to 16 atoms each
        dict(name="multi_uneven32", kind="multi", count=32, lo=24, hi=48, sizes=3, degree=20),
        # the Rayleigh-Ritz products of the 64-atom cell
        dict(name="subspace_lattice64", kind="subspace", **lat64, states=180),
        # the electrostatic potential of the 64-atom cell at the default tolerance
        dict(name="poisson_lattice64", kind="poisson", **lat64, tol=1e-10),
        # the descriptors of the learned starting density of the 64-atom cell
        dict(name="features_lattice64", kind="features", **lat64),
        # one mini-batch of the network's training set
        dict(name="mlpgrad_65536", kind="mlpgrad", points=512000, batch=65536),
        # the set-up of the next step of a 64-atom molecular-dynamics run
        dict(name="move_lattice64", kind="move", **lat64),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def lattice(lo, hi):
        n = log_int(lo, hi)
        ns = [min(hi, max(lo, n + rng.randint(-6, 6))) for _ in range(3)]
        if rng.random() < 0.4:
            ns = [n, n, n]
        if rng.random() < 0.5:
            ns = [x + x % 2 for x in ns]
        ms = [max(1, int(round(x * H_MESH / SPACING))) for x in ns]
        c = dict(n1=ns[0], n2=ns[1], n3=ns[2], h=H_MESH)
        if rng.random() < 0.3 and ms[0] * ms[1] * ms[2] <= 64:
            c["natom"] = max(2, ms[0] * ms[1] * ms[2])
        else:
            c.update(m1=ms[0], m2=ms[1], m3=ms[2], basis=1)
        return c

    def nstates(c):
        atoms = c["natom"] if "natom" in c else c["m1"] * c["m2"] * c["m3"] * c["basis"]
        s = int(math.ceil(max(2.0 * atoms + 4, 2.4 * atoms) - 1e-9))
        s += 2 * rng.randint(0, max(1, s // 10))
        return s + s % 2

    kind = rng.choice(["filter", "filter", "filter", "kpass", "multi", "subspace", "poisson", "features", "mlpgrad",
                       "move", "scf"])
    if kind == "filter":
        c = lattice(24, 112)
        return dict(kind=kind, **c, states=nstates(c), degree=rng.randint(8, 24))
    if kind == "kpass":
        c = lattice(20, 52)
        return dict(kind=kind, **c, states=nstates(c), degree=rng.randint(8, 24),
                    k1=rng.choice([0.0, 0.25, 0.375]), k2=rng.choice([-0.125, 0.5]), k3=rng.choice([0.0, 0.125]))
    if kind == "multi":
        return dict(kind=kind, count=log_int(2, 48), lo=24, hi=48, sizes=rng.randint(0, 1 << 20),
                    degree=rng.randint(8, 20))
    if kind == "subspace":
        c = lattice(40, 100)
        return dict(kind=kind, **c, states=nstates(c))
    if kind == "poisson":
        return dict(kind=kind, **lattice(24, 112), tol=rng.choice([1e-10, 1e-10, 1e-9]))
    if kind == "features" or kind == "move":
        return dict(kind=kind, **lattice(24, 96))
    if kind == "mlpgrad":
        n = log_int(4000, 800000)
        return dict(kind=kind, points=n, batch=min(n, log_int(1000, 262144)))
    n = rng.randint(20, 30)
    return dict(kind="scf", precision="fp64", n1=n, n2=n + rng.randint(0, 3), n3=n, h=0.25, m1=1, m2=1, m3=1,
                basis=rng.choice([1, 2]), states=rng.choice([6, 8, 10]), buffer=0, degree=rng.randint(8, 14),
                iterations=rng.randint(4, 8))


# ---- cells and fields --------------------------------------------------------------------------
def _cell(case, seed, sigma=0.1):
    """grid, edges and atom positions of a case."""
    n = (case["n1"], case["n2"], case["n3"])
    L = np.array([x * case["h"] for x in n])
    rng = np.random.default_rng([seed, 1])
    if "natom" in case:
        return n, L, _random_positions(L, case["natom"], rng)
    m = (case["m1"], case["m2"], case["m3"])
    ijk = np.array([(i, j, k) for k in range(m[2]) for j in range(m[1]) for i in range(m[0])], float)
    pos = (ijk + 0.5) * (L / np.array(m))
    if case["basis"] == 2:
        pos = np.concatenate([pos, pos + 0.5 * L / np.array(m)])
    return n, L, pos + rng.normal(0.0, sigma, pos.shape)


def _random_positions(L, natom, rng):
    pos = []
    for tries in range(200000):
        if len(pos) == natom:
            break
        p = rng.uniform(0.0, 1.0, 3) * L
        far = 3.0 if tries < 100000 else 1.5
        d = np.array(pos).reshape(-1, 3) - p
        d -= L * np.round(d / L)
        if (np.linalg.norm(d, axis=1) >= far).all():
            pos.append(p)
    return np.array(pos)


def _uneven_sizes(case):
    """the sizes of a `multi` case's cells, from the case alone: (points an edge, atoms, states)."""
    rng = np.random.default_rng(case["sizes"])
    for _ in range(case["count"]):
        n = int(rng.integers(case["lo"], case["hi"] + 1))
        atoms = int(min(16, max(2, round((n * H_MESH / SPACING) ** 3))))
        s = int(math.ceil(max(2.0 * atoms + 4, 2.4 * atoms) - 1e-9))
        yield n, atoms, s + s % 2


def _uneven(case, seed):
    """the cells of a `multi` case: [(n, L, pos, states)], positions from the seed."""
    rng = np.random.default_rng([seed, 2])
    out = []
    for n, atoms, states in _uneven_sizes(case):
        L = np.full(3, n * H_MESH)
        out.append(((n, n, n), L, _random_positions(L, atoms, rng), states))
    return out


def _axis(n, L, d):
    return torch.arange(n[d], device=DEV, dtype=torch.float64) * (L[d] / n[d])


def _gaussians(n, L, pos, amp, w, cut):
    """sum over atoms and periodic images of amp exp(-r^2 / (2 w^2)), r <= cut, on the grid [n3, n2, n1]."""
    out = torch.zeros((n[2], n[1], n[0]), device=DEV, dtype=torch.float64)
    for p in pos:
        near = []
        for d in range(3):
            x = _axis(n, L, d) - p[d]
            t = int(math.ceil((cut + float(x.abs().max())) / L[d]))
            near.append([y for y in (x - k * L[d] for k in range(-t, t + 1)) if float(y.abs().min()) <= cut])
        for z in near[2]:
            for y in near[1]:
                for x in near[0]:
                    r2 = (x * x)[None, None, :] + (y * y)[None, :, None] + (z * z)[:, None, None]
                    out += torch.where(r2 <= cut * cut, torch.exp(-r2 / (2 * w * w)) * amp, 0.0)
    return out.reshape(-1)


def _smooth(n, L, pos, amp, w):
    """the same sum without a cut-off, by separable factors (fields that only serve as inputs)."""
    f = []
    for d in range(3):
        x = _axis(n, L, d)[None, :] - torch.tensor(pos[:, d], device=DEV)[:, None]
        t = int(math.ceil(10 * w / L[d])) + 1
        f.append(sum(torch.exp(-((x - k * L[d]) ** 2) / (2 * w * w)) for k in range(-t, t + 1)))
    return (amp * torch.einsum("ax,ay,az->zyx", f[0], f[1], f[2])).reshape(-1)


def _charges(n, L, pos):
    s = SPECIES[0]
    b = _smooth(n, L, pos, -s["Z"] / (2 * math.pi * s["r_loc"] ** 2) ** 1.5, s["r_loc"])
    rho = _smooth(n, L, pos, s["Z"] / (2 * math.pi * s["sad_width"] ** 2) ** 1.5, s["sad_width"])
    return b, rho


def _symbol(n, L):
    """eigenvalues of -L_h on the grid [n3, n2, n1]."""
    s = []
    for d in range(3):
        k = torch.arange(n[d], device=DEV, dtype=torch.float64) * (2 * math.pi / n[d])
        s.append(-(FD[0] + sum(2 * FD[r] * torch.cos(r * k) for r in range(1, R + 1))) / (L[d] / n[d]) ** 2)
    return s[2][:, None, None] + s[1][None, :, None] + s[0][None, None, :]


def _potential_of(n, L, f):
    """zero-mean phi of -L_h phi = 4 pi (f - mean f)."""
    g = torch.fft.fftn(f.reshape(n[2], n[1], n[0]))
    sym = _symbol(n, L)
    sym[0, 0, 0] = 1.0
    g = 4 * math.pi * g / sym
    g[0, 0, 0] = 0.0
    return torch.fft.ifftn(g).real.reshape(-1).contiguous()


def _veff(n, L, pos):
    """a starting V_eff: the electrostatic potential of atomic densities and pseudocharges plus exchange."""
    b, rho = _charges(n, L, pos)
    return _potential_of(n, L, b + rho) - (3.0 / math.pi * rho.clamp_min(1e-14)) ** (1.0 / 3.0)


def _bounds(n, L, V):
    """(a, b, a0) of the filter: the wanted states lie in [a0, a], the spectrum ends below b."""
    top = -(FD[0] + sum(2 * FD[r] * (-1) ** r for r in range(1, R + 1)))
    return 1.0, 0.5 * top * sum((n[d] / L[d]) ** 2 for d in range(3)) + float(V.max()) + 1.0, -1.0


def _ctx(case, n, L, pos, states, precision, kpts=None, **more):
    return sd.sdft_create(L, n, pos, np.zeros(len(pos), int), SPECIES, dict(nstates=states, precision=precision, **more),
                          kpts=kpts)


def _gen(seed, k=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 8191 + k)
    return g


def _block(seed, k, *shape):
    return torch.rand(shape, generator=_gen(seed, k), device=DEV, dtype=torch.float32) - 0.5


# ---- preparation -------------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "mlpgrad":
        return _mlp_inputs(case, seed)
    if kind == "multi":
        cells = []
        for i, (n, L, pos, states) in enumerate(_uneven(case, seed)):
            V = _veff(n, L, pos)
            ctx = _ctx(case, n, L, pos, states, sd.SDFT_MIXED)
            sd.sdft_set_veff(ctx, 0, V)
            x = _block(seed, i, states // 2, n[0] * n[1] * n[2], 2)
            cells.append((ctx, x, torch.empty_like(x), _bounds(n, L, V)))
        return dict(case=case, cells=cells)
    n, L, pos = _cell(case, seed)
    ng = n[0] * n[1] * n[2]
    s = dict(case=case, n=n, L=L, pos=pos, ng=ng)
    if kind == "scf":
        mixed = case["precision"] == "mixed"
        s["ctx"] = _ctx(case, n, L, pos, case["states"], sd.SDFT_MIXED if mixed else sd.SDFT_FP64,
                        nbuffer=case["buffer"], cheb_degree=case["degree"], max_scf=case["iterations"], seed=seed % 65536)
        s["rho"] = torch.empty(ng, device=DEV, dtype=torch.float64)
        return s
    if kind == "poisson":
        b, rho = _charges(n, L, pos)
        s["ctx"] = _ctx(case, n, L, pos, 2 * len(pos) + 4, sd.SDFT_MIXED)
        s.update(f=b + rho, phi=torch.empty(ng, device=DEV, dtype=torch.float64))
        return s
    if kind == "features":
        s["ctx"] = _ctx(case, n, L, pos, 2 * len(pos) + 4, sd.SDFT_MIXED)
        s["feat"] = torch.empty((ng, sd.SDFT_MLP_NFEAT), device=DEV, dtype=torch.bfloat16)
        return s
    if kind == "move":
        _, _, before = _cell(case, seed + 1)
        s["ctx"] = _ctx(case, n, L, before, 2 * len(pos) + 4, sd.SDFT_FP64)
        sd.sdft_set_veff(s["ctx"], 0, _veff(n, L, pos))
        s["x"] = _block(seed, 0, 2, ng).double()
        s.update(y=torch.empty_like(s["x"]), b=torch.empty(ng, device=DEV, dtype=torch.float64),
                 sad=torch.empty(ng, device=DEV, dtype=torch.float64))
        return s
    ns = case["states"]
    V = _veff(n, L, pos)
    if kind == "subspace":
        s["ctx"] = _ctx(case, n, L, pos, ns, sd.SDFT_MIXED)
        s["y"] = _block(seed, 0, ns // 2, ng, 2) * math.sqrt(12.0 / ng)
        s["hy"] = (s["y"].double() * V[None, :, None]).float()
        q = torch.randn((ns, ns), generator=_gen(seed, 1), device=DEV, dtype=torch.float64)
        s["q"] = torch.linalg.qr(q)[0].contiguous()
        s["m"] = torch.empty((ns, ns), device=DEV, dtype=torch.float64)
        s["hs"] = torch.empty_like(s["m"])
        s["x"] = torch.empty_like(s["y"])
        return s
    kpt = [(case["k1"], case["k2"], case["k3"])] if kind == "kpass" else None
    s["ctx"] = _ctx(case, n, L, pos, ns, sd.SDFT_MIXED, kpts=kpt)
    sd.sdft_set_veff(s["ctx"], 0, V)
    s["bounds"] = _bounds(n, L, V)
    if kind == "filter":
        s["x"] = _block(seed, 0, ns // 2, ng, 2)
        s["y"] = torch.empty_like(s["x"])
        return s
    s["x"] = _block(seed, 0, ns, ng, 2)
    s["y"], s["hy"], s["z"] = (torch.empty_like(s["x"]) for _ in range(3))
    q = torch.randn((ns, ns, 2), generator=_gen(seed, 1), device=DEV, dtype=torch.float64)
    s["q"] = torch.view_as_real(torch.linalg.qr(torch.view_as_complex(q))[0].contiguous()).contiguous()
    s["m"] = torch.empty((ns, ns, 2), device=DEV, dtype=torch.float64)
    s["hs"] = torch.empty_like(s["m"])
    return s


def _mlp_inputs(case, seed):
    npts = case["points"]
    g = _gen(seed)
    # radial descriptors: non-negative, most of them a few tenths
    feat = torch.randn((npts, sd.SDFT_MLP_NFEAT), generator=g, device=DEV).abs_().mul_(0.8).to(torch.bfloat16)
    target = torch.randn(npts, generator=g, device=DEV) * 0.05
    u = torch.rand(MLP_PARAMS, generator=g, device=DEV) * 2.0 - 1.0
    scale = torch.cat([torch.full((k,), v) for k, v in ((2048, math.sqrt(6 / 96)), (64, 0.05), (4096, math.sqrt(6 / 128)),
                                                         (64, 0.05), (64, math.sqrt(6 / 65)), (1, 0.05))]).to(DEV)
    return dict(case=case, feat=feat, target=target, params=u * scale, start=seed % npts,
                grad=torch.empty(MLP_PARAMS, device=DEV), loss=torch.zeros(1, device=DEV, dtype=torch.float64))


# ---- one pass ----------------------------------------------------------------------------------
def run(state):
    s, case = state, state["case"]
    kind = case["kind"]
    if kind == "filter":
        a, b, a0 = s["bounds"]
        return sd.sdft_chebyshev_filter(s["ctx"], 0, 0, sd.SDFT_MIXED, s["x"], s["y"], case["states"], case["degree"],
                                        a, b, a0)
    if kind == "kpass":
        a, b, a0 = s["bounds"]
        ctx, ns = s["ctx"], case["states"]
        sd.sdft_chebyshev_filter(ctx, 0, 0, sd.SDFT_MIXED, s["x"], s["y"], ns, case["degree"], a, b, a0)
        sd.sdft_apply_h(ctx, 0, 0, sd.SDFT_MIXED, s["y"], s["hy"], ns)
        sd.sdft_subspace_matrices(ctx, 0, sd.SDFT_MIXED, s["y"], s["hy"], s["m"], s["hs"], ns)
        sd.sdft_rotate(ctx, 0, sd.SDFT_MIXED, s["y"], s["q"], s["z"], ns)
        return s["y"], s["hy"], s["m"].float(), s["hs"].float(), s["z"]
    if kind == "multi":
        cells = s["cells"]
        return sd.sdft_chebyshev_filter_multi([c[0] for c in cells], [c[1] for c in cells], [c[2] for c in cells],
                                              case["degree"], [c[3][0] for c in cells], [c[3][1] for c in cells],
                                              [c[3][2] for c in cells])
    if kind == "subspace":
        ctx, ns = s["ctx"], case["states"]
        sd.sdft_subspace_matrices(ctx, 0, sd.SDFT_MIXED, s["y"], s["hy"], s["m"], s["hs"], ns)
        sd.sdft_rotate(ctx, 0, sd.SDFT_MIXED, s["y"], s["q"], s["x"], ns)
        return s["m"].float(), s["hs"].float(), s["x"]
    if kind == "poisson":
        s["phi"].zero_()
        sd.sdft_poisson(s["ctx"], s["f"], s["phi"], tol=case["tol"])
        return s["phi"]
    if kind == "features":
        return sd.sdft_mlp_dataset(s["ctx"], s["feat"])[0]
    if kind == "mlpgrad":
        s["loss"].zero_()
        sd.sdft_mlp_loss_grad(s["feat"], s["target"], case["points"], case["batch"], s["start"], s["params"], s["grad"],
                              s["loss"])
        return s["grad"], s["loss"].float()
    if kind == "move":
        sd.sdft_move_atoms(s["ctx"], s["pos"], guess=0)
        sd.sdft_apply_h(s["ctx"], 0, 0, sd.SDFT_FP64, s["x"], s["y"], 2)
        return (sd.sdft_get_pseudocharge(s["ctx"], s["b"]), sd.sdft_get_sad_density(s["ctx"], s["sad"]), s["y"])
    # scf
    ctx = s["ctx"]
    sd.sdft_reset(ctx)
    r = sd.sdft_scf(ctx)
    sd.sdft_get_density(ctx, s["rho"])
    eig, forces = sd.sdft_get_eigenvalues(ctx), sd.sdft_get_forces(ctx)
    if case["precision"] == "mixed":
        return r["energy"], s["rho"].float(), eig.astype(np.float32)
    return np.float64(r["energy"]), s["rho"], eig, forces


# ---- what a pass cannot do without ---------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "mlpgrad":
        return dict(bytes=float(case["batch"]) * (64 + 4) + 8.0 * MLP_PARAMS,
                    flops=6.0 * case["batch"] * (32 * 64 + 64 * 64 + 64))
    if kind == "multi":
        by = fl = 0.0
        for n, _, states in _uneven_sizes(case):
            by += 8.0 * n ** 3 * states
            fl += 76.0 * n ** 3 * states * case["degree"]
        return dict(bytes=by, flops=fl)
    ng = float(case["n1"] * case["n2"] * case["n3"])
    ns = case.get("states", 0)
    if kind == "filter":   # x in, y out; 19 multiply-adds and 18 additions of the stencil, 10 more of the step
        return dict(bytes=8.0 * ng * ns, flops=76.0 * ng * ns * case["degree"])
    if kind == "kpass":
        return dict(bytes=4 * 8.0 * ng * ns, flops=2 * 76.0 * ng * ns * (case["degree"] + 1) + 24.0 * ng * ns * ns)
    if kind == "subspace":
        return dict(bytes=3 * 4.0 * ng * ns, flops=6.0 * ng * ns * ns)
    if kind == "poisson":
        return dict(bytes=16.0 * ng, flops=76.0 * ng)
    if kind == "features":
        atoms = case["natom"] if "natom" in case else case["m1"] * case["m2"] * case["m3"] * case["basis"]
        vol = ng * case["h"] ** 3
        return dict(bytes=64.0 * ng, flops=ng * (atoms * 4 / 3 * math.pi * 6.5 ** 3 / vol) * 32 * 4)
    if kind == "move":
        return dict(bytes=16.0 * ng + 4 * 8.0 * ng, flops=76.0 * 2 * ng)
    b = 4.0 if case["precision"] == "mixed" else 8.0
    nf, passes = ns + case["buffer"], case["iterations"] + 3
    return dict(bytes=passes * (case["degree"] + 3) * b * ng * nf,
                flops=passes * ((case["degree"] + 1) * 76.0 * ng * nf + 6.0 * ng * nf * nf))


# ---- the same in 64 bits, by plain torch ---------------------------------------------------------
def _projectors(n, L, pos, kred=None):
    """per atom: grid indices [atoms, cap] and chi (with Bloch phases) [atoms, cap], padded with zeros."""
    sp = SPECIES[0]
    h = L / np.array(n)
    norm = (math.pi ** 1.5 * sp["r_proj"] ** 3) ** -0.5
    lists = []
    for p in pos:
        lo = np.ceil((p - sp["r_cut_proj"]) / h).astype(int)
        hi = np.floor((p + sp["r_cut_proj"]) / h).astype(int)
        ax = [np.arange(lo[d], hi[d] + 1) for d in range(3)]
        I, J, K = np.meshgrid(*ax, indexing="ij")
        I, J, K = I.ravel(), J.ravel(), K.ravel()
        r2 = (I * h[0] - p[0]) ** 2 + (J * h[1] - p[1]) ** 2 + (K * h[2] - p[2]) ** 2
        keep = r2 < sp["r_cut_proj"] ** 2
        I, J, K, r2 = I[keep], J[keep], K[keep], r2[keep]
        v = norm * np.exp(-r2 / (2 * sp["r_proj"] ** 2))
        if kred is not None:
            t = [np.floor_divide(x, n[d]) for d, x in enumerate((I, J, K))]
            v = v * np.exp(-2j * np.pi * sum(kred[d] * t[d] for d in range(3)))
        lists.append((((K % n[2]) * n[1] + J % n[1]) * n[0] + I % n[0], v))
    cap = max(len(i) for i, _ in lists)
    idx = np.zeros((len(lists), cap), np.int64)
    val = np.zeros((len(lists), cap), np.complex128 if kred is not None else np.float64)
    for a, (i, v) in enumerate(lists):
        idx[a, :len(i)], val[a, :len(i)] = i, v
    return torch.from_numpy(idx).to(DEV), torch.from_numpy(val).to(DEV), sp["E_kb"] * float(np.prod(h))


def _apply_h(X, n, L, V, proj, kred=None):
    """H X of [cols, ng] in 64 bits."""
    idx, val, gamma = proj
    u = X.reshape(-1, n[2], n[1], n[0])
    out = (V * X).reshape(u.shape)
    for d in range(3):
        ax, c = 3 - d, -0.5 / (L[d] / n[d]) ** 2
        ph = complex(np.exp(2j * np.pi * kred[d])) if kred is not None else 1.0
        reach = [torch.arange(-R, n[d] + R, device=DEV)]
        t = torch.div(reach[0], n[d], rounding_mode="floor")
        pad = u.index_select(ax, reach[0] % n[d])
        if kred is not None:
            shape = [1, 1, 1, 1]
            shape[ax] = -1
            pad = pad * torch.tensor([ph ** int(k) for k in t.tolist()], device=DEV, dtype=X.dtype).reshape(shape)
        out = out.add_(u, alpha=c * FD[0])
        for r in range(1, R + 1):
            out.add_(pad.narrow(ax, R + r, n[d]), alpha=c * FD[r]).add_(pad.narrow(ax, R - r, n[d]), alpha=c * FD[r])
        del pad
    out = out.reshape(X.shape)
    C = (X[:, idx.reshape(-1)].reshape(X.shape[0], *idx.shape) * val.conj()).sum(-1) * gamma
    out.index_add_(1, idx.reshape(-1), (C[:, :, None] * val).reshape(X.shape[0], -1))
    return out


def _filter(X, n, L, V, proj, m, a, b, a0, kred=None):
    e, c = 0.5 * (b - a), 0.5 * (b + a)
    s1 = e / (a0 - c)
    s, prev = s1, X
    cur = (_apply_h(X, n, L, V, proj, kred) - c * X) * (s1 / e)
    for _ in range(2, m + 1):
        s2 = 1.0 / (2.0 / s1 - s)
        nxt = _apply_h(cur, n, L, V, proj, kred).add_(cur, alpha=-c).mul_(2.0 * s2 / e).add_(prev, alpha=-s * s2)
        prev, cur, s = cur, nxt, s2
    return cur


def _filter_paired(x, n, L, pos, V, m, bounds):
    """the filter of a paired FP32 block [pairs, ng, 2] in 64 bits, a few columns at a time."""
    proj = _projectors(n, L, pos)
    out = torch.empty(x.shape, device=DEV, dtype=torch.float64)
    step = max(1, int(3e7 // x.shape[1]))
    for p in range(0, x.shape[0], step):
        X = x[p:p + step].double().permute(0, 2, 1).reshape(-1, x.shape[1]).contiguous()
        Y = _filter(X, n, L, V, proj, m, *bounds)
        out[p:p + step] = Y.reshape(-1, 2, x.shape[1]).permute(0, 2, 1)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "scf":
        return None
    if kind == "mlpgrad":
        return _mlp_exact(case, seed)
    if kind == "multi":
        out = []
        for i, (n, L, pos, states) in enumerate(_uneven(case, seed)):
            V = _veff(n, L, pos)
            x = _block(seed, i, states // 2, n[0] * n[1] * n[2], 2)
            out.append(_filter_paired(x, n, L, pos, V, case["degree"], _bounds(n, L, V)))
        return out
    n, L, pos = _cell(case, seed)
    ng = n[0] * n[1] * n[2]
    if kind == "poisson":
        b, rho = _charges(n, L, pos)
        return _potential_of(n, L, b + rho)
    if kind == "features":
        return _features(n, L, pos)
    if kind == "move":
        sp = SPECIES[0]
        x = _block(seed, 0, 2, ng).double()
        return (_gaussians(n, L, pos, -sp["Z"] / (2 * math.pi * sp["r_loc"] ** 2) ** 1.5, sp["r_loc"], 10 * sp["r_loc"]),
                _gaussians(n, L, pos, sp["Z"] / (2 * math.pi * sp["sad_width"] ** 2) ** 1.5, sp["sad_width"],
                           10 * sp["sad_width"]),
                _apply_h(x, n, L, _veff(n, L, pos), _projectors(n, L, pos)))
    ns = case["states"]
    V = _veff(n, L, pos)
    if kind == "subspace":
        y = _block(seed, 0, ns // 2, ng, 2) * math.sqrt(12.0 / ng)
        hy = (y.double() * V[None, :, None]).float()
        Y = y.double().permute(0, 2, 1).reshape(ns, ng)
        HY = hy.double().permute(0, 2, 1).reshape(ns, ng)
        q = torch.randn((ns, ns), generator=_gen(seed, 1), device=DEV, dtype=torch.float64)
        q = torch.linalg.qr(q)[0].contiguous()       # column-major: row j holds output column j
        X = (q @ Y).reshape(ns // 2, 2, ng).permute(0, 2, 1).contiguous()
        return Y @ Y.T, Y @ HY.T, X
    if kind == "filter":
        return _filter_paired(_block(seed, 0, ns // 2, ng, 2), n, L, pos, V, case["degree"], _bounds(n, L, V))
    kred = (case["k1"], case["k2"], case["k3"])
    X = torch.view_as_complex(_block(seed, 0, ns, ng, 2).double())
    proj = _projectors(n, L, pos, kred)
    Y = _filter(X, n, L, V, proj, case["degree"], *_bounds(n, L, V), kred)
    HY = _apply_h(Y, n, L, V, proj, kred)
    q = torch.randn((ns, ns, 2), generator=_gen(seed, 1), device=DEV, dtype=torch.float64)
    q = torch.linalg.qr(torch.view_as_complex(q))[0].contiguous()
    parts = Y, HY, (Y.conj() @ Y.T).T.contiguous(), (Y.conj() @ HY.T).T.contiguous(), q @ Y
    return tuple(torch.view_as_real(v) for v in parts)


def _features(n, L, pos):
    nf, rc = sd.SDFT_MLP_NFEAT, 6.5
    out = torch.zeros((n[0] * n[1] * n[2], nf), device=DEV, dtype=torch.float64)
    mu = 6.0 * torch.arange(nf, device=DEV, dtype=torch.float64) / 31.0
    for p in pos:
        near = []
        for d in range(3):
            x = _axis(n, L, d) - p[d]
            t = int(math.ceil((rc + float(x.abs().max())) / L[d]))
            near.append([y for y in (x - k * L[d] for k in range(-t, t + 1)) if float(y.abs().min()) <= rc])
        for z in near[2]:
            for y in near[1]:
                for x in near[0]:
                    r = ((x * x)[None, None, :] + (y * y)[None, :, None] + (z * z)[:, None, None]).sqrt().reshape(-1)
                    at = torch.nonzero(r <= rc).reshape(-1)
                    r = r[at][:, None]
                    fc = 0.5 * (torch.cos(math.pi * r / rc) + 1.0)
                    out.index_add_(0, at, torch.exp(-(r - mu) ** 2 / (2 * (6.0 / 31.0) ** 2)) * fc)
    return out


def _mlp_exact(case, seed):
    s = _mlp_inputs(case, seed)
    npts, nb = case["points"], case["batch"]
    mult = 999983 if npts % 1000003 == 0 else 1000003
    at = ((s["start"] + torch.arange(nb, device=DEV, dtype=torch.int64)) % npts) * mult % npts
    p = s["params"].to(torch.bfloat16).double()
    W1, b1, W2, b2, w3, b3 = torch.split(p, [2048, 64, 4096, 64, 64, 1])
    W1, W2 = W1.reshape(64, 32), W2.reshape(64, 64)
    X, t = s["feat"][at].double(), s["target"][at].double()
    z1 = X @ W1.T + b1
    s1 = torch.sigmoid(z1)
    h1 = z1 * s1
    z2 = h1 @ W2.T + b2
    s2 = torch.sigmoid(z2)
    h2 = z2 * s2
    e = h2 @ w3 + b3 - t
    dy = 2.0 * e / nb
    d2 = dy[:, None] * w3 * (s2 * (1 + z2 * (1 - s2)))
    d1 = (d2 @ W2) * (s1 * (1 + z1 * (1 - s1)))
    grad = torch.cat([(d1.T @ X).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0), h2.T @ dy, dy.sum().reshape(1)])
    return grad, (e * e).mean().reshape(1)
