"""The calls this library is used for, at the sizes of its own workloads, as cases to measure.

A case is one pass of a user's program on the GPU: positions (or caller matrices) in hand, through
the public entry points of `paper_1210_1531_gb300`, to the results such a program keeps. The
kinds of pass:

    md        a molecular-dynamics step: rebuild at the positions, energy and forces
    rho       the stages one by one: columns, mu, density matrix, energies, ICOHP
    caller    the caller's own H and S (a self-consistent loop): set_hs, columns, mu, density matrix
    green     G(z) of every column on the pattern at complex energies
    spectrum  energy-resolved COHP and density of states on a contour

An "md" pass takes new positions from the seed. The others return arrays over the pattern of H
and S, so their structure is the case's own and the model's hoppings (or the caller's matrices)
come from the seed, as when a model is fitted.

mu itself is not among the outputs: in a gap N(mu) is flat to rounding, so that mu is not
determined there, while what is formed from it (energies, density matrix, forces) is.
"""
import dataclasses
import functools
import math

import numpy as np
import torch

import paper_1210_1531_gb300 as eg
import workloads as wl

KT = 0.1


def listed():
    return [
        # the smallest system in use: 64 atoms, every cluster the whole system, library defaults;
        # a call whose launches and latency count
        dict(name="md 64 whole-system", kind="md", system="diamond", nx=2, ny=2, nz=2, sigma=0.05,
             r_cluster=0.0, nu=30, form="default"),
        # an odd size (vacancies), a whole-system cluster of 211 atoms, the options an MD run sets
        dict(name="md 211 ragged", kind="md", system="diamond", nx=3, ny=3, nz=3, sigma=0.08, keep=211,
             r_cluster=0.0, nu=30, form="production"),
        # staged calls on a middle-sized system, library defaults (two classical passes)
        dict(name="rho 512", kind="rho", system="diamond", nx=4, ny=4, nz=4, sigma=0.1, r_cluster=6.0,
             nu=30, form="default"),
        # caller H and S as dense 4x4 blocks
        dict(name="caller 512", kind="caller", system="diamond", nx=4, ny=4, nz=4, sigma=0.1,
             r_cluster=6.0, nu=30, form="default"),
        # the Green's function itself at a few energies
        dict(name="green 512", kind="green", system="diamond", nx=4, ny=4, nz=4, sigma=0.1, r_cluster=6.0,
             nu=30, n_z=8, form="default"),
        # forces that are the exact gradient of the truncated method, 1000 atoms
        dict(name="exact forces 1000", kind="md", system="diamond", nx=5, ny=5, nz=5, sigma=0.1,
             r_cluster=6.0, nu=30, form="exact"),
        # the benchmark's system and form: 4096 atoms, work queue, autotuned, captured step
        dict(name="md 4096", kind="md", system="diamond", nx=8, ny=8, nz=8, sigma=0.1, r_cluster=6.0,
             nu=30, form="production"),
        # the same system in the library's default form, and in the memory-saving workflow
        dict(name="md 4096 default", kind="md", system="diamond", nx=8, ny=8, nz=8, sigma=0.1,
             r_cluster=6.0, nu=30, form="default"),
        dict(name="spectrum 4096 two-pass", kind="spectrum", system="diamond", nx=8, ny=8, nz=8, sigma=0.1,
             r_cluster=6.0, nu=30, n_z=32, form="two_pass"),
        # sp2-sp3 composite: uneven clusters, nu by size class
        dict(name="md composite 32768", kind="md", system="composite", n=32768, r_cluster=6.0, nu=30,
             classes=True, form="production"),
        # the dense disordered carbon streamed in batches with the eigen-factors kept: the
        # 10^6-atom workload at a sixteenth of its size
        dict(name="md amorphous 65536", kind="md", system="amorphous", nx=32, ny=16, nz=16, r_cluster=5.0,
             nu=30, batch_atoms=16384, keep_factors=1100, form="production"),
    ]


COMPOSITES = (6000, 8192, 10000, 14000, 16384)      # atom counts that the generator reaches


def draw(rng):
    def cells(lo, hi):
        n = math.exp(rng.uniform(math.log(lo), math.log(hi)))       # atoms
        side = (n / 8.0) ** (1.0 / 3.0)
        return [max(4, round(side * rng.uniform(0.8, 1.25))) for _ in range(3)]

    kind = rng.choice(["md", "md", "md", "rho", "caller", "green", "spectrum"])
    c = dict(kind=kind, nu=rng.randint(16, 40), r_cluster=round(rng.uniform(4.6, 6.4), 2))
    system = rng.choice(["diamond", "diamond", "composite", "amorphous"] if kind in ("md", "rho") else
                        ["diamond", "diamond", "amorphous"])
    hi = {"md": 16000, "rho": 8000, "caller": 2000, "green": 1500, "spectrum": 3000}[kind]
    if system == "composite":
        n = rng.choice(COMPOSITES)
        c.update(system="composite", n=n, keep=int(n * rng.uniform(0.9, 1.0)), classes=rng.random() < 0.5)
    else:
        nx, ny, nz = cells(512, hi)
        c.update(system=system, nx=nx, ny=ny, nz=nz)
        if system == "diamond":
            c.update(sigma=round(rng.uniform(0.05, 0.1), 3))
            if rng.random() < 0.5:      # vacancies: odd atom counts
                c.update(keep=int(8 * nx * ny * nz * rng.uniform(0.9, 0.995)))
    if kind in ("green", "spectrum"):
        c.update(n_z=rng.randint(3, 24))
    forms = {"md": ["production", "production", "default", "two_pass"], "rho": ["default", "production"],
             "caller": ["default", "production"], "green": ["default"], "spectrum": ["default", "two_pass"]}[kind]
    if kind == "md" and c["system"] == "diamond" and c.get("keep", 8 * c["nx"] * c["ny"] * c["nz"]) < 1500:
        forms = forms + ["exact"]
    c.update(form=rng.choice(forms))
    return c


# ---------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=None)
def grains(n):
    """The composite's lattice sites (diamond grains in graphite, one fixed arrangement)."""
    pos, box, _ = wl.composite(n, sigma=0.0)
    return pos, box


def model(case, seed):
    """The two-centre model: the workloads' own, for the analysis calls with hoppings from the seed."""
    sk = wl.sk_params()
    if case["kind"] != "md":
        g = np.random.default_rng(seed + 29)
        sk = dataclasses.replace(sk, Es=sk.Es + g.normal(0.0, 0.1), V0=tuple(v * g.uniform(0.95, 1.0) for v in sk.V0))
    return sk


def structure(case, seed):
    """Positions and box of the case's system, from the seed where the results' shapes allow it."""
    if case["kind"] != "md":
        seed = 1210
    if case["system"] == "composite":
        pos, box = grains(case["n"])
        pos = pos + np.random.default_rng(seed).normal(0.0, 0.05, pos.shape)
        pos -= box * np.floor(pos / box)
    elif case["system"] == "amorphous":
        pos, box = wl.amorphous((case["nx"], case["ny"], case["nz"]), seed=seed)
    else:
        pos, box = wl.diamond((case["nx"], case["ny"], case["nz"]), sigma=case["sigma"], seed=seed)
    if case.get("keep"):        # vacancies
        kept = np.sort(np.random.default_rng(seed + 5).choice(len(pos), case["keep"], replace=False))
        pos = pos[kept]
    return np.ascontiguousarray(pos), box


def energies(case):
    """A contour across the band, 0.2 eV above the real axis."""
    n = case["n_z"]
    return [complex(-20.0 + 30.0 * (i + 0.5) / n, 0.2) for i in range(n)]


FORMS = {
    "default": {},
    "production": dict(schedule=1, autotune=True, graph=True, reorth=1),
    "two_pass": dict(two_pass=True, schedule=1, reorth=1),
    "exact": dict(exact_forces=True, schedule=1, reorth=1),
}


def prepare(case, seed):
    pos, box = structure(case, seed)
    options = dict(FORMS[case["form"]])
    for k in ("batch_atoms", "keep_factors"):
        if k in case:
            options[k] = case[k]
    if case.get("classes"):
        options["nu_classes"] = ((100, 20), (140, 30), (1 << 30, 40))
    pos = torch.as_tensor(pos, dtype=torch.float64).cuda()
    system = eg.System(pos, box, model(case, seed), case["r_cluster"], case["nu"], KT, 4.0 * len(pos), **options)
    state = dict(case=case, pos=pos, box=box, system=system)
    if case["kind"] in ("green", "spectrum"):
        state["z"] = energies(case)
    if case["kind"] == "caller":    # the caller's matrices: the model's, with its own on-site shifts
        H, S = system.hs()
        rp, ci = system.pattern()
        rows = torch.repeat_interleave(torch.arange(len(pos), device="cuda"), (rp[1:] - rp[:-1]).long())
        g = torch.Generator(device="cuda").manual_seed(seed + 17)
        shift = 0.3 * torch.randn(len(pos), generator=g, device="cuda", dtype=torch.float64)
        own = torch.nonzero(rows == ci.long()).squeeze(1)
        H[own] += shift[rows[own], None, None] * torch.eye(4, device="cuda", dtype=torch.float64)
        state.update(H=H, S=S, shift=shift)
    return state


def run(state):
    case, s = state["case"], state["system"]
    if case["kind"] == "md":
        s.rebuild(state["pos"])
        _, e_band, f_free, forces = s.energy_force()
        return dict(e_band=e_band, f_free=f_free, forces=forces)
    if case["kind"] == "green":
        s.rebuild(state["pos"])
        return dict(G=s.green_columns(z=state["z"]))
    if case["kind"] == "spectrum":
        s.rebuild(state["pos"])
        s.green_columns()
        c, c_sigma, c_pi, dos = s.cohp_spectrum(state["z"])
        return dict(c=c, c_sigma=c_sigma, c_pi=c_pi, dos=dos)
    if case["kind"] == "rho":
        s.rebuild(state["pos"])
    else:
        s.set_hs(state["H"], state["S"])
    s.green_columns()
    mu, n_at_mu = s.find_mu()
    rho, rho_e = s.density_matrix(mu)
    e = s.energies(mu)
    out = dict(rho=rho, rho_e=rho_e, n=n_at_mu, e_band=e["E_band"], f_free=e["F_free"])
    if case["kind"] == "rho":
        out["icohp"], out["icohp_sigma"], out["icohp_pi"] = s.icohp(rho)
    return out


# ---------------------------------------------------------------- what a pass cannot do without
def counts(case):
    """Atoms, mean cluster size and mean pattern row, from the density."""
    if case["system"] == "composite":
        n = case.get("keep") or case["n"]
        density = 0.125 * n / case["n"]
    else:
        a = wl.DIAMOND_A * ((3.515 / 3.0) ** (1.0 / 3.0) if case["system"] == "amorphous" else 1.0)
        full = 8 * case["nx"] * case["ny"] * case["nz"]
        n = case.get("keep") or full
        density = 8.0 / a ** 3 * n / full
    ball = lambda r: 4.0 / 3.0 * math.pi * r ** 3 * density  # noqa: E731
    return n, float(n) if case["r_cluster"] <= 0 else min(n, ball(case["r_cluster"])), min(n, ball(2.6))


def work(case):
    n, cluster, row = counts(case)
    nu = 25 if case.get("classes") else case["nu"]
    nc, columns = 4.0 * cluster, 4.0 * n
    # per column: nu sparse products with H and with S (64 flops per block pair, three quarters of a
    # row inside the cluster), three projections and one update per step, the projected problem
    flops = columns * (nu * 64 * 0.75 * row * cluster + nc * (6 + 2) * nu * nu / 2 + 20 * nu ** 3)
    block = 16 * 8.0 * n * row
    if case["form"] == "exact":
        flops *= 3
    if case["form"] == "two_pass":
        flops *= 2
    size = 24.0 * n + 24.0 * n + 16.0
    if case["kind"] == "rho":
        size = 24.0 * n + 2 * block + 3 * block / 16
    elif case["kind"] == "caller":
        size = 4 * block
    elif case["kind"] == "green":
        size = 24.0 * n + 2 * block * case["n_z"]
    elif case["kind"] == "spectrum":
        size = 24.0 * n + 3 * block / 16 * case["n_z"]
    return dict(bytes=size, flops=flops)


# ---------------------------------------------------------------- the same in plain torch, 64 bits
def dense_blocks(pos, box, sk):
    """Dense H and S as [n, 4, n, 4], the pattern mask [n, n]; differentiable in pos."""
    n, dev = len(pos), pos.device
    d = pos[None, :, :] - pos[:, None, :]
    d = d - box * torch.round(d / box).detach()
    eye = torch.eye(n, dtype=torch.bool, device=dev)
    r = torch.sqrt(torch.where(eye, torch.ones_like(d[..., 0]), (d * d).sum(-1)))
    mask = (r <= sk.r_cut) & ~eye
    u = d / r[..., None]
    x = (r - sk.r_on) / (sk.r_cut - sk.r_on)
    t = torch.where(r <= sk.r_on, torch.ones_like(r), 1 - 10 * x ** 3 + 15 * x ** 4 - 6 * x ** 5)
    t = torch.where(mask, t, torch.zeros_like(t))
    outs = []
    for v0, q, onsite in ((sk.V0, sk.qH, (sk.Es, sk.Ep)), (sk.S0, sk.qS, (1.0, 1.0))):
        ss, sp, pps, ppp = (v0[k] * torch.exp(-q[k] * (r - sk.r0)) * t for k in range(4))
        pp = u[..., :, None] * u[..., None, :] * (pps - ppp)[..., None, None]
        pp = pp + torch.eye(3, dtype=pos.dtype, device=dev) * ppp[..., None, None]
        top = torch.cat([ss[..., None], u * sp[..., None]], -1)
        low = torch.cat([-(u * sp[..., None])[..., None], pp], -1)
        b = torch.cat([top[..., None, :], low], -2)
        diag = torch.diag(torch.tensor([onsite[0]] + [onsite[1]] * 3, dtype=pos.dtype, device=dev))
        outs.append((b + eye[..., None, None] * diag).permute(0, 2, 1, 3))
    return outs[0], outs[1], mask | eye, r


def exact(case, seed):
    """The pass in plain torch: dense matrices, every column's Krylov space by two classical
    Gram-Schmidt passes, LAPACK for the projected problems, forces by autograd."""
    n = case.get("keep") or (8 * case["nx"] * case["ny"] * case["nz"] if "nx" in case else case["n"])
    if n > 512 or case["system"] == "composite" or case["form"] == "exact" or case["kind"] == "spectrum":
        return None
    dev = "cuda"
    pos, box = structure(case, seed)
    pos = torch.as_tensor(pos, dtype=torch.float64, device=dev)
    box = torch.as_tensor(box, dtype=torch.float64, device=dev)
    sk, nu, m = model(case, seed), case["nu"], 4 * n
    pos.requires_grad_(True)
    H4, S4, mask, r = dense_blocks(pos, box, sk)
    H, S = H4.detach().reshape(m, m), S4.detach().reshape(m, m)
    if case["kind"] == "caller":
        g = torch.Generator(device="cuda").manual_seed(seed + 17)
        shift = 0.3 * torch.randn(n, generator=g, device=dev, dtype=torch.float64)
        H = H + torch.diag(shift.repeat_interleave(4))
    if case["r_cluster"] > 0:
        near = (r <= case["r_cluster"]) | torch.eye(n, dtype=torch.bool, device=dev)
    else:
        near = torch.ones_like(mask)
    inside = near.repeat_interleave(4, 0).repeat_interleave(4, 1).to(H.dtype)     # [column, row]
    # every column at once: rows of the batch are columns j, vectors masked to the cluster
    U = torch.zeros(m, nu, m, dtype=H.dtype, device=dev)
    SU, HU = torch.zeros_like(U), torch.zeros_like(U)
    u = torch.diag(1.0 / torch.sqrt(torch.diagonal(S)))
    for k in range(nu):
        U[:, k] = u
        HU[:, k], SU[:, k] = (u @ H) * inside, (u @ S) * inside
        if k + 1 == nu:
            break
        w = HU[:, k].clone()
        for _ in range(2):
            h = torch.bmm(SU[:, :k + 1], w[:, :, None])
            w = w - torch.bmm(U[:, :k + 1].transpose(1, 2), h)[:, :, 0]
        beta2 = (w * ((w @ S) * inside)).sum(1)
        if float(beta2.min()) <= 1e-20:
            return None     # a space that is exhausted: the recursion stops there
        u = w / torch.sqrt(beta2)[:, None]
    Hp, Sp = torch.bmm(U, HU.transpose(1, 2)), torch.bmm(U, SU.transpose(1, 2))
    Hp, Sp = (0.5 * (x + x.transpose(1, 2)).cpu() for x in (Hp, Sp))
    L = torch.linalg.cholesky(Sp)
    A = torch.linalg.solve_triangular(L, Hp, upper=False)
    A = torch.linalg.solve_triangular(L, A.transpose(1, 2), upper=False)
    eps, Q = torch.linalg.eigh(0.5 * (A + A.transpose(1, 2)))
    V = torch.linalg.solve_triangular(L.transpose(1, 2), Q, upper=True).to(dev)
    eps, at = eps.to(dev), torch.arange(m, device=dev)
    c, d, gg = (torch.einsum("jk,jkl->jl", X[at, :, at], V) for X in (U, SU, HU))
    block, col = torch.nonzero(mask, as_tuple=True)     # e = (I, J), rows ascending

    def on_pattern(X):      # X[j, i] of column j to [e, a, b] of (I, a), (J, b)
        return X.reshape(n, 4, n, 4).permute(2, 3, 0, 1)[block, :, col, :]

    if case["kind"] == "green":
        out = []
        for z in energies(case):
            w = torch.einsum("jkl,jl->jk", V.to(torch.complex128), c / (z - eps))
            out.append(on_pattern(torch.einsum("jki,jk->ji", U.to(torch.complex128), w)))
        return dict(G=torch.stack(out, -1))

    def fermi(mu):
        return 2.0 / (1.0 + torch.exp(torch.clamp((eps - mu) / KT, max=700.0)))

    lo, hi = float(eps.min()) - 40 * KT, float(eps.max()) + 40 * KT
    while hi - lo >= 1e-13:
        mid = 0.5 * (lo + hi)
        if mid in (lo, hi):
            break
        lo, hi = (mid, hi) if float((fermi(mid) * c * d).sum()) < 4.0 * n else (lo, mid)
    mu = 0.5 * (lo + hi)
    f = fermi(mu)
    x = (eps - mu) / KT
    omega = float((c * d * (-2 * KT) * (torch.clamp(-x, min=0.0) + torch.log1p(torch.exp(-x.abs())))).sum())
    e_band, f_free = float((f * gg * c).sum()), omega + mu * 4.0 * n
    rho, rho_e = (torch.einsum("jki,jk->ji", U, torch.einsum("jkl,jl->jk", V, y)) for y in (f * c, f * eps * c))
    if case["kind"] == "md":
        keep = mask.repeat_interleave(4, 0).repeat_interleave(4, 1).to(H.dtype)
        total = (H4.reshape(m, m) * (rho.T * keep)).sum() - (S4.reshape(m, m) * (rho_e.T * keep)).sum()
        total.backward()
        return dict(e_band=e_band, f_free=f_free, forces=-pos.grad)
    out = dict(rho=on_pattern(rho), rho_e=on_pattern(rho_e), n=float((f * c * d).sum()), e_band=e_band, f_free=f_free)
    if case["kind"] == "rho":
        Hb = H.reshape(n, 4, n, 4)[block, :, col, :]
        out["icohp"] = (Hb * out["rho"]).sum((1, 2))
        out["icohp_sigma"] = out["icohp_pi"] = None
    return out
