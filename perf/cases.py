"""Performance cases: what users of this library have it do, through the Python binding.

A case is a dict of plain values; `listed()` names twelve, `draw(rng)` gives more of the same
ranges.  `prepare` makes what a program holds before a call (a context with its molecule, points
and weights on the GPU), `run` is one call (or the forward and backward pair), `work` its
unavoidable bytes and operations, and `exact` the same outputs from plain torch in FP64.

Kinds:
  forward   new points, then the MO vgl [walk][elec][5][mo] (optionally cusp-corrected)
  backward  new points, the MO vgl and dL/dC, dL/dR of L = sum W * vgl
  move      one electron of every walker proposed, its MO vgl [walk][5][mo]
  density   new grid points, then sum_i w_i phi_i^2
  batch     new points in several molecules of uneven sizes, their MO vgl in one run
Systems: water; organic (C:N:O:H chain, s to f shells); chain (C/H, s to d); cluster (C:O:H, packed
at 10 A^3 per atom); peptide (C:N:O:H:Cu, packed).
"""
import math
import random

import numpy as np
import torch

from paper_2512_16677_gb300 import qmckl, synth

# element ratios, basis recipe, screening (bits B or cutoff eps) of each system
SYSTEMS = {
    "water": ({"O": 1, "H": 2}, synth.RECIPE_SMALL, {"bits": 53}),
    "organic": ({"C": 56, "N": 10, "O": 9, "H": 75}, synth.RECIPE_TZ, {"eps": 1e-10}),
    "chain": ({"C": 1, "H": 1}, synth.RECIPE_SMALL, {"bits": 53}),
    "cluster": ({"C": 4, "O": 1, "H": 5}, synth.RECIPE_SMALL, {"eps": 1e-10}),
    "peptide": ({"C": 34, "N": 11, "O": 10, "H": 48, "Cu": 1}, synth.RECIPE_SMALL, {"eps": 1e-10}),
}
# Cartesian AOs per nucleus of each system, for sizing draws (the recipes' averages)
AO_PER_NUCLEUS = {"water": 8.4, "organic": 11.0, "chain": 10.0, "cluster": 10.0, "peptide": 10.5}


def listed():
    def case(name, kind, system, nuclei, electrons, walkers, mos, mode, **more):
        return dict(name=name, kind=kind, system=system, nuclei=nuclei, electrons=electrons,
                    walkers=walkers, mos=mos, mode=mode, **more)

    return [
        # a small molecule in the library's default mode: launches and latency count
        case("water_fp64", "forward", "water", 3, 10, 64, 5, "fp64"),
        # the inner step of a Monte Carlo walk: one electron of every walker moves
        case("move_organic_bf16x3", "move", "organic", 150, 600, 256, 300, "bf16x3"),
        # the same in double precision
        case("move_organic_fp64", "move", "organic", 150, 600, 256, 300, "fp64"),
        # a whole configuration of a walker population: the headline workload
        case("organic_bf16x3", "forward", "organic", 150, 600, 256, 300, "bf16x3"),
        # all-electron orbitals with the nuclear cusp, an odd population and electron count
        case("organic_cusp_bf16x3", "forward", "organic", 150, 599, 37, 299, "bf16x3", cusp=True),
        # the headline workload in plain single precision
        case("organic_fp32", "forward", "organic", 150, 600, 256, 300, "fp32"),
        # and in double precision, the accuracy anchor
        case("organic_fp64", "forward", "organic", 150, 600, 256, 300, "fp64"),
        # orbital and geometry optimisation: values, then gradients in C and the nuclei
        case("backward_chain_bf16x3", "backward", "chain", 50, 200, 128, 100, "bf16x3"),
        case("backward_chain_fp64", "backward", "chain", 50, 200, 128, 100, "fp64"),
        # a data set of molecules of uneven sizes
        dict(name="batch_bf16x3", kind="batch", system="organic", molecules=12, sizes=4,
             mode="bf16x3"),
        # a large system
        case("cluster_bf16x3", "forward", "cluster", 1000, 4000, 16, 2000, "bf16x3"),
        # a density grid for visualisation
        dict(name="density_tf32", kind="density", system="peptide", nuclei=104, mos=218, nx=100,
             ny=100, nz=100, mode="tf32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["forward", "move", "backward", "density", "batch"], [6, 2, 2, 1, 1])[0]
    mode = rng.choice(["fp64", "fp32", "tf32", "bf16x3"])
    if kind == "batch":
        return dict(kind=kind, system="organic", molecules=rng.randint(2, 12),
                    sizes=rng.randrange(1 << 20), mode=rng.choice(["tf32", "bf16x3"]))
    if kind == "density":
        nuclei = _log_int(rng, 20, 150)
        # points x MOs x AOs of the 100^3 grid in the reduced modes, a tenth of it otherwise
        side = 100 if mode in ("tf32", "bf16x3") else 46
        n = [_log_int(rng, 12, side) for _ in range(3)]
        return dict(kind=kind, system="peptide", nuclei=nuclei, mos=rng.randint(nuclei, 2 * nuclei),
                    nx=n[0], ny=n[1], nz=n[2], mode=mode)
    system = rng.choice(["water", "organic", "chain", "cluster"] if kind == "forward"
                        else ["organic", "chain"])
    nuclei = {"water": 3, "organic": _log_int(rng, 20, 200), "chain": _log_int(rng, 10, 100),
              "cluster": _log_int(rng, 100, 1000)}[system]
    electrons = 10 if system == "water" else rng.randint(3 * nuclei, 4 * nuclei)
    mos = 5 if system == "water" else rng.randint(nuclei, 2 * nuclei)
    # no more work than the largest listed case of the mode (points x MOs x AOs)
    most = {"forward": {"fp64": 7e10, "fp32": 1.2e11, "tf32": 1.2e12, "bf16x3": 1.2e12},
            "backward": {"fp64": 3e9, "fp32": 1e10, "tf32": 1e10, "bf16x3": 5e10},
            "move": {"fp64": 7e10, "fp32": 7e10, "tf32": 7e10, "bf16x3": 7e10}}[kind][mode]
    per_walker = electrons * mos * AO_PER_NUCLEUS[system] * nuclei
    walkers = _log_int(rng, 1, max(1, min(256, int(most / per_walker))))
    case = dict(kind=kind, system=system, nuclei=nuclei, electrons=electrons, walkers=walkers,
                mos=mos, mode=mode)
    if kind == "forward" and rng.random() < 0.2:
        case["cusp"] = True
    return case


# ----------------------------------------------------------------------------- inputs


def _molecule(case, seed, mos):
    """The case's molecule: geometry, basis, MO coefficients and electron positions."""
    ratio, recipe, screening = SYSTEMS[case["system"]]
    rng = np.random.default_rng([2512, seed])
    n = case["nuclei"]
    elements = synth.element_counts(ratio, n)
    if case["system"] == "water":
        pos = np.array([[0.0, 0.0, 0.0], [0.76, 0.0, 0.59], [-0.76, 0.0, 0.59]])
    elif case["system"] in ("cluster", "peptide"):
        elements = [elements[i] for i in rng.permutation(n)]
        pos = synth.packed_cluster(rng, n, (3.0 * 10.0 * n / (4.0 * math.pi)) ** (1.0 / 3.0))
    else:
        elements = [("C", "H")[i % 2] for i in range(n)] if case["system"] == "chain" else \
            [elements[i] for i in rng.permutation(n)]
        pos = synth.self_avoiding_chain(rng, n)
    return synth.make_molecule(case["system"], rng, elements, pos, recipe, mos,
                               case.get("electrons", 1), case.get("walkers", 1), **screening)


def _batch_cases(case):
    """The forward cases of a batch: chains of 20-200 nuclei, 16-256 walkers."""
    rng = random.Random(case["sizes"])
    out = []
    for _ in range(case["molecules"]):
        n, w = _log_int(rng, 20, 200), _log_int(rng, 16, 256)
        out.append(dict(kind="forward", system=case["system"], nuclei=n, electrons=4 * n,
                        walkers=w, mos=2 * n, mode=case["mode"]))
    return out


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _proposals(case, mol, seed):
    """(electron, [walk][3] proposed positions): a Gaussian step of 0.5 bohr."""
    rng = np.random.default_rng([166, seed])
    e = int(rng.integers(case["electrons"]))
    return e, mol.coord[:, e] + 0.5 * rng.normal(size=(case["walkers"], 3))


def _grid(case, mol):
    """[nx * ny * nz][3] points over the nuclei +- 4 bohr, z fastest."""
    lo, hi = mol.nucl_coord.min(axis=0) - 4.0, mol.nucl_coord.max(axis=0) + 4.0
    axes = [torch.linspace(lo[k], hi[k], case[c], dtype=torch.float64, device="cuda")
            for k, c in enumerate(("nx", "ny", "nz"))]
    return torch.stack(torch.meshgrid(*axes, indexing="ij"), dim=-1).reshape(-1, 3).contiguous()


def _loss_weights(case, seed):
    """W [walk][elec][5][mo] of L = sum W * vgl, U(-1, 1) in the mode's type."""
    dt = torch.float64 if case["mode"] == "fp64" else torch.float32
    w = torch.rand((case["walkers"], case["electrons"], 5, case["mos"]), dtype=dt, device="cuda",
                   generator=_generator(seed))
    return w.mul_(2.0).sub_(1.0)


def _context(case, seed):
    mol = _molecule(case, seed, case["mos"])
    ctx = qmckl.Context(case["mode"])
    ctx.set_molecule(mol)
    if case.get("cusp"):
        ctx.set_mo_cusp(synth.cusp_radii(mol))
    return mol, ctx


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        parts = [_context(c, seed * 64 + i) for i, c in enumerate(_batch_cases(case))]
        coords = [torch.from_numpy(m.coord).cuda() for m, _ in parts]
        ctxs = [c for _, c in parts]
        for ctx, coord in zip(ctxs, coords):
            ctx.set_points_device(coord)
        return dict(kind=kind, ctxs=ctxs, coords=coords, batch=qmckl.Batch(ctxs))
    mol, ctx = _context(case, seed)
    state = dict(kind=kind, ctx=ctx)
    if kind == "density":
        state.update(coord=_grid(case, mol), occupation=synth.occupations(mol))
        return state
    state["coord"] = torch.from_numpy(mol.coord).cuda()
    if kind == "backward":
        state["dW"] = _loss_weights(case, seed)
    elif kind == "move":
        e, pos = _proposals(case, mol, seed)
        state.update(electron=e, proposed=torch.from_numpy(pos).cuda())
        ctx.set_points_device(state["coord"])
    return state


def run(state):
    kind = state["kind"]
    if kind == "batch":
        for ctx, coord in zip(state["ctxs"], state["coords"]):
            ctx.set_points_device(coord)
        return state["batch"].run()
    ctx = state["ctx"]
    if kind == "move":
        ctx.set_single_point_device(state["electron"], state["proposed"])
        return ctx.mo_vgl_single_device()
    ctx.set_points_device(state["coord"])
    if kind == "density":
        return ctx.density_device(state["occupation"])
    out = ctx.mo_vgl_device()
    if kind == "backward":
        dC, dR = ctx.backward_device(state["dW"])
        return out, dC, dR
    return out


# ------------------------------------------------------------------------------- work


def _nonzero_aos(case, mol):
    """Mean count of AOs per point that screening keeps, on a sample of the points."""
    rng = np.random.default_rng(1)
    if case["kind"] == "density":
        lo, hi = mol.nucl_coord.min(axis=0) - 4.0, mol.nucl_coord.max(axis=0) + 4.0
        pts = rng.uniform(lo, hi, size=(64, 3))
    else:
        pts = mol.points[rng.integers(mol.point_num, size=64)]
    first = np.concatenate([[0], np.cumsum(mol.shell_prim_num)[:-1]])
    r2_max = _threshold(mol) / np.minimum.reduceat(mol.exponent, first)
    d = pts[:, None, :] - mol.nucl_coord[None, :, :]
    hit = ((d * d).sum(-1))[:, mol.shell_nucleus] < r2_max
    size = (mol.shell_ang_mom + 1) * (mol.shell_ang_mom + 2) // 2
    return float((hit * size).sum(1).mean())


def work(case):
    if case["kind"] == "batch":
        parts = [work(c) for c in _batch_cases(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    mol = _molecule(dict(case, walkers=1), 0, 1)
    es = 8 if case["mode"] == "fp64" else 4
    n_mo, n_ao, nnz = case["mos"], mol.ao_num, _nonzero_aos(case, mol)
    read = es * n_mo * n_ao
    if case["kind"] == "density":
        n = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": float(n * (24 + es) + read), "flops": n * n_mo * (2.0 * nnz + 3.0)}
    n = case["walkers"] * (1 if case["kind"] == "move" else case["electrons"])
    out = es * n * 5 * n_mo
    flops = 2.0 * 5 * n_mo * nnz * n
    if case["kind"] == "backward":
        return {"bytes": float(24 * n + read + 2 * out + 8 * n_mo * n_ao + 24 * mol.nucl_num),
                "flops": 3 * flops}
    return {"bytes": float(24 * n + read + out), "flops": flops}


# ------------------------------------------------------------------------------ exact


def _threshold(mol):
    """T of Eq. 3: a primitive counts where gamma r^2 < T."""
    return (mol.bits - 1) * math.log(2.0) if mol.eps is None else -math.log(mol.eps)


class _Aos:
    """AO vgl of a molecule in FP64 torch, by shells of one angular momentum at a time."""

    def __init__(self, mol):
        def dev(a):
            return torch.as_tensor(a, device="cuda")

        self.T = _threshold(mol)
        self.l = np.asarray(mol.shell_ang_mom)
        size = (self.l + 1) * (self.l + 2) // 2
        self.ao0 = np.concatenate([[0], np.cumsum(size)[:-1]])
        first = np.concatenate([[0], np.cumsum(mol.shell_prim_num)[:-1]])
        width = int(mol.shell_prim_num.max())
        g, c = np.full((mol.shell_num, width), 1e300), np.zeros((mol.shell_num, width))
        for s in range(mol.shell_num):
            p = slice(first[s], first[s] + mol.shell_prim_num[s])
            g[s, :mol.shell_prim_num[s]] = mol.exponent[p]
            c[s, :mol.shell_prim_num[s]] = mol.shell_factor[s] * mol.coefficient[p] * mol.prim_factor[p]
        self.r2_max = dev(self.T / g.min(axis=1))
        self.nucleus, self.gamma, self.coef = dev(mol.shell_nucleus), dev(g), dev(c)
        self.factor = dev(mol.ao_factor)
        self.R = dev(mol.nucl_coord)

    def near(self, pts):
        """The shells that screening keeps at any of the points (numpy indices)."""
        d = pts[:, None, :] - self.R[None, :, :]
        r2 = (d * d).sum(-1)[:, self.nucleus]
        return (r2 < self.r2_max).any(0).nonzero()[:, 0].cpu().numpy()

    def radial(self, shells, r2):
        """S_m = sum_k c_k gamma_k^m exp(-gamma_k r2), m = 0, 1, 2, for r2 [n][shells]."""
        g, c = self.gamma[shells], self.coef[shells]
        t = r2[..., None] * g
        e = torch.where(t < self.T, c * torch.exp(-t), torch.zeros_like(t))
        g = torch.where(c != 0, g, torch.zeros_like(g))
        return e.sum(-1), (e * g).sum(-1), (e * g * g).sum(-1)

    def vgl(self, pts, R, shells, components=5):
        """([n][components][columns], the AO of each column) of the given shells."""
        parts, cols = [], []
        for l in range(4):
            s = shells[self.l[shells] == l]
            if s.size == 0:
                continue
            si = torch.as_tensor(s, device="cuda")
            d = pts[:, None, :] - R[self.nucleus[si]][None, :, :]
            r2 = (d * d).sum(-1)
            s0, s1, s2 = self.radial(si, r2)

            def power(k, n, d=d):
                return d[..., k] ** n if n > 0 else torch.full_like(d[..., k], 1.0 if n == 0 else 0.0)

            for j, abc in enumerate(synth.cartesian_powers(l)):
                ao = self.ao0[s] + j
                m = self.factor[torch.as_tensor(ao, device="cuda")]
                f = [power(k, abc[k]) for k in range(3)]
                rest = [f[1] * f[2], f[0] * f[2], f[0] * f[1]]
                p = f[0] * rest[0]
                v = [p * s0]
                if components == 5:
                    v += [abc[k] * power(k, abc[k] - 1) * rest[k] * s0 - 2.0 * d[..., k] * p * s1
                          for k in range(3)]
                    lap = sum(abc[k] * (abc[k] - 1) * power(k, abc[k] - 2) * rest[k]
                              for k in range(3))
                    v.append(lap * s0 - 2.0 * (2 * l + 3) * p * s1 + 4.0 * r2 * p * s2)
                parts.append(torch.stack(v, dim=1) * m)
                cols.append(ao)
        if not parts:
            return torch.zeros((pts.shape[0], components, 0), dtype=torch.float64, device="cuda"), \
                torch.zeros(0, dtype=torch.int64, device="cuda")
        return torch.cat(parts, dim=-1), torch.as_tensor(np.concatenate(cols), device="cuda")


def _blocks(n, size):
    return [(i, min(n, i + size)) for i in range(0, n, size)]


def _exact_vgl(mol, aos, coord):
    """MO vgl [walk][elec][5][mo] in FP64, electrons of one place together."""
    C = torch.as_tensor(mol.mo_coef, device="cuda")
    w, e = coord.shape[:2]
    out = torch.empty((w, e, 5, C.shape[0]), dtype=torch.float64, device="cuda")
    for a, b in _blocks(e, max(1, 256 // w)):
        pts = coord[:, a:b].reshape(-1, 3)
        chi, cols = aos.vgl(pts, aos.R, aos.near(pts))
        out[:, a:b] = (chi.reshape(-1, cols.numel()) @ C[:, cols].T).reshape(w, b - a, 5, -1)
    return out


def _add_cusp(mol, aos, coord, out):
    """Adds the cusp correction to out: inside radius rc of nucleus A the s part of A gives way
    to a cubic in rho that joins it in value, slope and curvature at rc and has Kato's slope
    at the nucleus."""
    rc, n_mo = synth.cusp_radii(mol), mol.mo_num
    C = torch.as_tensor(mol.mo_coef, device="cuda")
    at_nuclei = _exact_vgl(mol, aos, aos.R[None])[0, :, 0]
    pts, flat = coord.reshape(-1, 3), out.reshape(-1, 5, n_mo)
    for A in range(mol.nucl_num):
        s = np.nonzero((mol.shell_nucleus == A) & (mol.shell_ang_mom == 0))[0]
        ao, si = torch.as_tensor(aos.ao0[s], device="cuda"), torch.as_tensor(s, device="cuda")
        cs = C[:, ao] * aos.factor[ao]

        def s_part(rho, cs=cs, si=si):
            return [S @ cs.T for S in aos.radial(si, (rho * rho)[:, None].expand(-1, len(si)))]

        r, Z = float(rc[A]), float(mol.nucl_charge[A])
        g0, g1, g2 = (x[0] for x in s_part(torch.tensor([r], dtype=torch.float64, device="cuda")))
        q = at_nuclei[A] - s_part(torch.zeros(1, dtype=torch.float64, device="cuda"))[0][0]
        lhs = torch.tensor([[1, r, r * r, r ** 3], [0, 1, 2 * r, 3 * r * r], [0, 0, 2, 6 * r],
                            [Z, 1, 0, 0]], dtype=torch.float64, device="cuda")
        f = torch.linalg.solve(lhs, torch.stack([g0, -2 * r * g1, 4 * r * r * g2 - 2 * g1, -Z * q]))
        d = pts - aos.R[A]
        rho = d.square().sum(-1).sqrt()
        hit = (rho < r).nonzero()[:, 0]
        if hit.numel() == 0:
            continue
        d, rho = d[hit], rho[hit][:, None]
        g0, g1, g2 = s_part(rho[:, 0])
        slope = f[1] / rho + 2 * f[2] + 3 * f[3] * rho + 2 * g1
        add = [f[0] + f[1] * rho + f[2] * rho ** 2 + f[3] * rho ** 3 - g0]
        add += [slope * d[:, k:k + 1] for k in range(3)]
        add.append(2 * f[1] / rho + 6 * f[2] + 12 * f[3] * rho - (4 * rho ** 2 * g2 - 6 * g1))
        flat[hit] += torch.stack(add, dim=1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [exact(c, seed * 64 + i) for i, c in enumerate(_batch_cases(case))]
    mol = _molecule(case, seed, case["mos"])
    aos = _Aos(mol)
    if kind == "density":
        C = torch.as_tensor(mol.mo_coef, device="cuda")
        grid, occ = _grid(case, mol), torch.as_tensor(synth.occupations(mol), device="cuda")
        rho = torch.empty(grid.shape[0], dtype=torch.float64, device="cuda")
        for a, b in _blocks(grid.shape[0], 4096):
            chi, cols = aos.vgl(grid[a:b], aos.R, aos.near(grid[a:b]), components=1)
            rho[a:b] = (chi[:, 0] @ C[:, cols].T).square() @ occ
        return rho
    if kind == "move":
        pos = torch.from_numpy(_proposals(case, mol, seed)[1]).cuda()
        return _exact_vgl(mol, aos, pos[:, None])[:, 0]
    coord = torch.from_numpy(mol.coord).cuda()
    out = _exact_vgl(mol, aos, coord)
    if case.get("cusp"):
        _add_cusp(mol, aos, coord, out)
    if kind == "forward":
        return out
    C = torch.as_tensor(mol.mo_coef, device="cuda")
    dW = _loss_weights(case, seed).double()
    R = aos.R.clone().requires_grad_(True)
    dC = torch.zeros_like(C)
    w, e = coord.shape[:2]
    for a, b in _blocks(e, max(1, 1024 // w)):
        pts = coord[:, a:b].reshape(-1, 3)
        chi, cols = aos.vgl(pts, R, aos.near(pts))
        if cols.numel() == 0:
            continue
        W = dW[:, a:b].reshape(-1, C.shape[0])
        dC[:, cols] += W.T @ chi.detach().reshape(W.shape[0], -1)
        ((W @ C[:, cols]).reshape(chi.shape) * chi).sum().backward()
    return out, dC, R.grad if R.grad is not None else torch.zeros_like(R)
