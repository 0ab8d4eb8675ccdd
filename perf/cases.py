"""The work that is measured: passes through the public entry points of the GW+C library.

A case is one call, or the few calls in a row, that a program makes on a molecule it has in hand: polarizability
builds, screened interactions, self-energy grids, quasiparticle energies, spectrum requests and cumulant spectra, in
the split-BF16 mode (the library's default) and in the FP64 mode that checks it. Molecules are synthetic with the sizes
of the acene study and of the serving recipe (n_occ = n_states / 18, n_aux = 3.5 n_states, n_core = 0.3 n_occ): 1s
cores near -10.4 Ha, valence states in [-1, -0.25] Ha, virtual states in [0, 3] Ha with a tenth of them up to 40 Ha,
normal RI coefficients with amplified core rows, scaled so that the largest eigenvalue of -Pi(0) is 2.
"""
import math

import numpy as np
import torch

from paper_2412_17132_gb300 import gwc

EV = 27.211386245988
ETA = 1e-3
N_IM = 32
XI0 = 1.0
T_MAX = 2000.0


def recipe(n_states):
    """(n_occ, n_core, n_aux) of the serving recipe for a molecule of n_states orbitals."""
    n_occ = max(2, round(n_states / 18))
    return n_occ, max(1, round(0.3 * n_occ)), round(3.5 * n_states)


def sized(kind, n_states, n_occ, n_core, n_aux, **more):
    return dict(kind=kind, n_states=n_states, n_occ=n_occ, n_core=n_core, n_aux=n_aux, **more)


def listed():
    tiny = (60, 8, 1, 200)
    benzene = (300, 21, 6, 1100)
    pentacene = (1300, 73, 22, 4500)
    small = (100, *recipe(100))
    middle = (340, *recipe(340))
    large = (700, *recipe(700))
    return [
        # the smallest call: W at one frequency of the tiny molecule, all launches and latency
        sized("screen", *tiny, prec="bf16x3", freqs=1, rhs=1, name="screen tiny 1 frequency"),
        # a chunk of residue frequencies with a right-hand side per core: the loop of every self-energy grid
        sized("screen", *benzene, prec="bf16x3", freqs=64, rhs=6, name="screen benzene 64"),
        # few frequencies of a large molecule: one QP iterate, a probe of W at chosen points
        sized("screen", *large, prec="bf16x3", freqs=8, rhs=12, name="screen 700 states 8"),
        # the largest polarizabilities, read back whole
        sized("chi0", *pentacene, prec="bf16x3", freqs=2, name="chi0 pentacene 2"),
        # the G0W0 self-energy of a small molecule on its whole satellite window, one dielectric build per residue
        sized("sigma", *tiny, prec="bf16x3", points=400, name="sigma tiny 400 points"),
        # the same grid in the mode that checks the others
        sized("sigma", *tiny, prec="fp64", points=400, name="sigma tiny fp64"),
        # FP64 check of W at a few frequencies of a middle-sized molecule
        sized("screen", *benzene, prec="fp64", freqs=8, rhs=6, name="screen benzene fp64 8"),
        # quasiparticle energies of a molecule just received: load, imaginary-axis table, secant iteration
        sized("qp", *benzene, prec="bf16x3", name="qp benzene"),
        # spectrum requests as the server runs them: load into a resident context, plan, step, results
        sized("request", *small, prec="bf16x3", capacity=150, points=200, name="request 100 states"),
        sized("request", *middle, prec="bf16x3", capacity=340, points=200, name="request 340 states"),
        # spectra from a self-energy in hand: one core, and every core of the largest molecule
        dict(kind="cumulant", n_core=1, points=400, n_t=1 << 16, name="cumulant 1 core"),
        dict(kind="cumulant", n_core=22, points=800, n_t=1 << 16, name="cumulant 22 cores"),
    ]


def draw(rng):
    def span(lo, hi):
        return round(math.exp(rng.uniform(math.log(lo), math.log(hi))))

    kind = rng.choice(("screen", "screen", "chi0", "sigma", "qp", "request", "cumulant", "cumulant"))
    if kind == "cumulant":
        return dict(kind=kind, n_core=span(1, 22), points=span(50, 1600), n_t=1 << rng.randint(12, 16))
    prec = "fp64" if kind in ("screen", "sigma") and rng.random() < 0.35 else "bf16x3"
    if prec == "fp64":
        n = span(24, 120 if kind == "sigma" else 260)
    else:
        n = span(24, {"screen": 700, "chi0": 700, "sigma": 120, "qp": 260, "request": 300}[kind])
    n_occ = max(2, round(n / rng.uniform(7, 20)))
    n_core = max(1, round(n_occ * rng.uniform(0.1, 0.4)))
    n_aux = max(8, round(n * rng.uniform(2.5, 4.2)))
    if kind == "screen":
        return sized(kind, n, n_occ, n_core, n_aux, prec=prec, freqs=span(1, 8 if prec == "fp64" or n > 300 else 64),
                     rhs=span(1, 30))
    if kind == "chi0":
        return sized(kind, n, n_occ, n_core, n_aux, prec=prec, freqs=span(1, 16))
    if kind == "sigma":
        return sized(kind, n, n_occ, n_core, n_aux, prec=prec, points=span(20, 400 if n <= 60 else 60))
    if kind == "request":
        return sized(kind, n, n_occ, n_core, n_aux, prec=prec, capacity=rng.choice((n, n + n // 3)),
                     points=span(40, 300))
    return sized(kind, n, n_occ, n_core, n_aux, prec=prec)


# -- inputs ---------------------------------------------------------------------------------------------------------
def system(case, seed):
    """Orbital energies and RI coefficients of a synthetic molecule, on the GPU."""
    n, n_occ, n_core, n_aux = (case[k] for k in ("n_states", "n_occ", "n_core", "n_aux"))
    r = np.random.default_rng([seed, 11])
    n_virt = n - n_occ
    high = round(n_virt * 5 / 52)
    eps = np.concatenate([np.sort(r.uniform(-10.41, -10.39, n_core)), np.sort(r.uniform(-1.0, -0.25, n_occ - n_core)),
                          np.sort(np.concatenate([r.uniform(0.0, 3.0, n_virt - high), r.uniform(3.0, 40.0, high)]))])
    g = torch.Generator(device="cuda").manual_seed(seed)
    amp = 1.0 + 4.0 * (torch.rand((n_core, n_aux), generator=g, device="cuda") < 0.1).double()  # [core][P]
    o_ov = torch.empty((n_aux, n_occ, n_virt), dtype=torch.float64, device="cuda").normal_(0.0, 0.02, generator=g)
    o_ov[:, :n_core] *= amp.t()[:, :, None]
    o_core = torch.empty((n, n_core, n_aux), dtype=torch.float64, device="cuda").normal_(0.0, 0.02, generator=g)
    o_core[:n_core] = 0.5 ** 0.5 * (o_core[:n_core] + o_core[:n_core].transpose(0, 1))
    o_core[n_occ:] = o_ov[:, :n_core].permute(2, 1, 0)  # O^P_{a c} = O^P_{c a}
    o_core[:n_occ] *= amp[None]
    o_core[:n_core] *= amp[:, None]
    o_ov = o_ov.reshape(n_aux, n_occ * n_virt)
    e = torch.as_tensor(eps, device="cuda")
    w = 4.0 / (e[None, n_occ:] - e[:n_occ, None]).reshape(-1)
    v = torch.ones(n_aux, dtype=torch.float64, device="cuda")
    for _ in range(20):  # largest eigenvalue of sum_ia w O O^T
        u = o_ov @ (w * (o_ov.t() @ v))
        lam = torch.linalg.vector_norm(u) / torch.linalg.vector_norm(v)
        v = u / torch.linalg.vector_norm(u)
    s = torch.sqrt(2.0 / lam)
    return dict(eps=eps, eps_d=e, n_occ=n_occ, core=np.arange(n_core), o_ov=o_ov.mul_(s), o_core=o_core.mul_(s))


def frequencies(case, seed):
    """Residue positions |eps_m - w| + i eta: core ones within the 30 eV window, valence ones near 9.5 Ha."""
    r = np.random.default_rng([seed, 12])
    f = case["freqs"]
    x = np.where(r.random(f) < 0.7, r.uniform(0.0, 25.0 / EV, f), r.uniform(8.5, 10.3, f))
    return torch.as_tensor(np.stack([x, np.full(f, ETA)], 1), device="cuda").contiguous()


def right_hand_sides(case, seed, mol):
    """Rows O^._{m c} of the residue states, one set per frequency."""
    r = np.random.default_rng([seed, 13])
    m = torch.as_tensor(r.integers(0, mol["n_occ"], (case["freqs"], case["rhs"])), device="cuda")
    c = torch.as_tensor(r.integers(0, case["n_core"], (case["freqs"], case["rhs"])), device="cuda")
    return mol["o_core"][m, c].contiguous()


def window(mol, points):
    c = float(np.mean(mol["eps"][mol["core"]]))
    return np.linspace(c - 25.0 / EV, c + 5.0 / EV, points)


def relative(points):
    return np.linspace(-25.0 / EV, 5.0 / EV, points)


def self_energies(case, seed):
    """Relative grids and Im Sigma of every core: satellite peaks of width eta and above on a small background."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    nc, nw = case["n_core"], case["points"]
    w = torch.as_tensor(relative(nw), device="cuda")[None].repeat(nc, 1)
    w = w + (torch.rand((nc, 1), generator=g, device="cuda", dtype=torch.float64) - 0.5) * 0.02
    pos = -0.92 * torch.rand((nc, 40), generator=g, device="cuda", dtype=torch.float64)
    wid = 0.002 + 0.02 * torch.rand((nc, 40), generator=g, device="cuda", dtype=torch.float64)
    s = 0.02 * torch.rand((nc, 40), generator=g, device="cuda", dtype=torch.float64) * (0.05 - pos).square()
    im = (s[:, :, None] * wid[:, :, None] / ((w[:, None] - pos[:, :, None]).square() + wid[:, :, None].square())).sum(1)
    return w.contiguous(), torch.where(w < 0, im, torch.zeros_like(im)).contiguous()


def options(case):
    return dict(eta=ETA, n_im=N_IM, xi0=XI0, t_max=T_MAX)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "cumulant":
        w, im = self_energies(case, seed)
        # the context of the molecule whose cores these are; its own size does not enter the spectrum
        mol = system(dict(n_states=3 * case["n_core"] + 8, n_occ=case["n_core"] + 2, n_core=case["n_core"], n_aux=32), seed)
        ctx = gwc.Context(mol["eps_d"], mol["n_occ"], mol["core"], mol["o_ov"], mol["o_core"], prec="bf16x3",
                          n_t=case["n_t"], batch=1, **options(case))
        return dict(kind=kind, ctx=ctx, w=w, im=im)
    mol = system(case, seed)
    if kind == "request":
        n = case["capacity"]
        occ = max(case["n_occ"], round(case["n_occ"] * n / case["n_states"]))
        core = max(case["n_core"], round(case["n_core"] * n / case["n_states"]))
        aux = max(case["n_aux"], round(case["n_aux"] * n / case["n_states"]))
        ctx = gwc.Context.with_capacity(n, occ, aux, core, prec=case["prec"], qp_mode="hedin", batch=64, **options(case))
        return dict(kind=kind, ctx=ctx, mol=mol, grid=relative(case["points"]))
    ctx = gwc.Context(mol["eps_d"], mol["n_occ"], mol["core"], mol["o_ov"], mol["o_core"], prec=case["prec"],
                      **options(case))
    if kind == "qp":
        return dict(kind=kind, ctx=ctx, mol=mol)
    if kind == "sigma":
        return dict(kind=kind, ctx=ctx, grid=window(mol, case["points"]))
    z = frequencies(case, seed)
    if kind == "chi0":
        return dict(kind=kind, ctx=ctx, z=z)
    return dict(kind=kind, ctx=ctx, z=z, rhs=right_hand_sides(case, seed, mol))


def load(ctx, mol):
    ctx.load(mol["eps_d"], mol["o_ov"], mol["o_core"], core_idx=mol["core"], n_occ=mol["n_occ"])


def run(state):
    kind, ctx = state["kind"], state["ctx"]
    if kind == "cumulant":
        return ctx.cumulant_spectrum(state["w"], state["im"])
    if kind == "chi0":
        return ctx.build_chi0(state["z"])
    if kind == "screen":
        return ctx.screen(state["z"], state["rhs"])
    if kind == "sigma":
        return ctx.sigma_core(state["grid"])
    load(ctx, state["mol"])
    if kind == "qp":
        return ctx.qp_solve()
    ctx.request_plan(state["grid"])
    ctx.request_step()
    return ctx.request_results()


# -- the work of one pass -------------------------------------------------------------------------------------------
def work(case):
    if case["kind"] == "cumulant":
        nc, nw, nt = case["n_core"], case["points"], case["n_t"]
        # one transform and one complex exponential per time; the grid enters once
        return dict(bytes=8.0 * (2 * nc * nw + nc * nt + nt), flops=nc * nt * (5.0 * math.log2(nt) + 20.0))
    n, n_occ, nc, na = (case[k] for k in ("n_states", "n_occ", "n_core", "n_aux"))
    n_ov = n_occ * (n - n_occ)
    build = 2.0 * na * (na + 1) * n_ov    # lower triangle, real and imaginary part
    factor = 8.0 * na ** 3 / 3
    solve = 8.0 * na * na / 2             # one right-hand side
    o_ov, o_core = 8.0 * na * n_ov, 8.0 * n * nc * na
    if case["kind"] == "chi0":
        f = case["freqs"]
        return dict(bytes=o_ov + 16.0 * f * na * na, flops=f * build)
    if case["kind"] == "screen":
        f, r = case["freqs"], case["rhs"]
        return dict(bytes=o_ov + f * r * (8.0 * na + 16), flops=f * (build + factor + r * solve))
    if case["kind"] == "sigma":
        nw = case["points"]
        pairs = nw * (n_occ - nc) + round(nw * 25 / 30) * nc
        return dict(bytes=o_ov + o_core + 32.0 * nc * nw, flops=pairs * (build + factor + nc * solve))
    table = (N_IM + 1) * (build / 2 + factor / 4 + n * nc * solve / 4)
    if case["kind"] == "qp":
        evals = 4.0  # dH and the secant's self-energies at least, with a build per core and occupied state each
        pairs = nc * (n_occ - nc + 1)
        return dict(bytes=o_ov + o_core, flops=table + evals * pairs * (build + factor + solve))
    nw = case["points"]
    pairs = nc * (n_occ - nc + (nc + 1) / 2)
    return dict(bytes=o_ov + o_core + 8.0 * nc * (nw + (1 << 16)),
                flops=table + pairs * (build + factor + solve) + round(nw * 25 / 30) * (build + factor + nc * solve))


# -- the same in 64 bits, in plain torch ----------------------------------------------------------------------------
def pi_of(mol, z):
    """Pi(z) = O diag(2[1/(z - D) - 1/(z + D)]) O^T for one complex z."""
    e, o, n_occ = mol["eps_d"], mol["o_ov"], mol["n_occ"]
    d = (e[None, n_occ:] - e[:n_occ, None]).reshape(-1)
    f = 2.0 * (1.0 / (z - d) - 1.0 / (z + d))

    def part(s):
        n = o.shape[0]
        step = max(512, -(-n // 4))
        p = torch.empty((n, n), dtype=torch.float64, device=o.device)
        for q in range(0, n, step):  # blocks on and below the diagonal
            p[q:, q : q + step] = o[q:] @ (o[q : q + step] * s).t()
            p[q : q + step, q + step :] = p[q + step :, q : q + step].t()
        return p

    re = part(f.real)
    return torch.complex(re, part(f.imag) if complex(z).real != 0.0 else torch.zeros_like(re))


def w_of(mol, z, b):
    """b^T (eps(z)^-1 - 1) b for the rows of b."""
    eps = -pi_of(mol, z)
    eps.diagonal().add_(1.0)
    bc = b.to(torch.complex128)
    x = torch.linalg.solve(eps, bc.t())
    return (bc * x.t()).sum(1) - (b * b).sum(1)


def theta(x):
    return 1.0 if x > 0 else (0.0 if x < 0 else 0.5)


def prefactor(em, w, ef):
    return -theta(ef - em) * theta(em - w) + theta(em - ef) * theta(w - em)


def imaginary_axis(mol):
    """Nodes, weights and W(i xi) of every state and core; the last plane is W(0)."""
    x, g = np.polynomial.legendre.leggauss(N_IM)
    xi, wx = XI0 * (1 + x) / (1 - x), 2 * XI0 * g / (1 - x) ** 2
    n, nc, na = mol["o_core"].shape
    b = mol["o_core"].reshape(n * nc, na)
    tab = torch.stack([w_of(mol, complex(0.0, k), b).real.reshape(n, nc) for k in [*xi, 0.0]])
    return torch.as_tensor(xi, device="cuda"), torch.as_tensor(wx, device="cuda"), tab


def imaginary_term(mol, axis, c, w):
    """I_n(w) = (1/pi) sum_m int a / (a^2 + xi^2) W(i xi), with W(0) taken out and integrated exactly."""
    xi, wx, tab = axis
    a = (w - mol["eps_d"])[:, None]
    k = wx[None] * a / (a * a + (xi * xi)[None]) / math.pi
    t = tab[:, :, c].t()
    return float(((k * (t[:, :-1] - t[:, -1:])).sum(1) + 0.5 * torch.sign(a[:, 0]) * t[:, -1]).sum())


def exact_cumulant(w, im, n_t):
    nc, nw = w.shape
    q = torch.zeros_like(w)
    q[:, 1:] += 0.5 * (w[:, 1:] - w[:, :-1])
    q[:, :-1] += 0.5 * (w[:, 1:] - w[:, :-1])
    coef = torch.where(w == 0, torch.zeros_like(w), q * im.abs() / math.pi / (w * w))
    dt = T_MAX / n_t
    t = dt * torch.arange(n_t, device="cuda", dtype=torch.float64)
    a = []
    for c in range(nc):
        re, ph = torch.zeros_like(t), torch.zeros_like(t)
        for j in range(0, nw, 64):
            x = w[c, j : j + 64, None] * t[None]
            k = coef[c, j : j + 64, None]
            re -= (2.0 * k * torch.sin(0.5 * x).square()).sum(0)
            ph -= (k * torch.sin(x)).sum(0)
        g = torch.polar(torch.exp(re - ETA * t), ph)
        g[0] *= 0.5
        a.append(torch.fft.fftshift(torch.fft.ifft(g).real * (n_t * dt / math.pi)))
    nu = 2.0 * math.pi / T_MAX * torch.arange(-(n_t // 2), n_t // 2, device="cuda", dtype=torch.float64)
    return torch.stack(a), nu


def exact_dh(mol, axis, cores):
    """Hedin shifts Re Sigma^c_n(eps_n), v^xc being the exchange."""
    eps, ef = mol["eps"], 0.5 * (mol["eps"][mol["n_occ"] - 1] + mol["eps"][mol["n_occ"]])
    dh = []
    for c in range(cores):
        w = float(eps[c])
        s = -imaginary_term(mol, axis, c, w)
        for m in range(mol["n_occ"]):
            f = prefactor(eps[m], w, ef)
            if f:
                s += f * float(w_of(mol, complex(abs(eps[m] - w), ETA), mol["o_core"][m, c : c + 1])[0].real)
        dh.append(s)
    return torch.tensor(dh, dtype=torch.float64, device="cuda")


def exact(case, seed):
    kind = case["kind"]
    if kind == "cumulant":
        return exact_cumulant(*self_energies(case, seed), case["n_t"])
    if work(case)["flops"] > 1.5e13:  # a device does about 1e12 of these a second in 64 bits
        return None
    mol = system(case, seed)
    if kind == "chi0":
        z = frequencies(case, seed).cpu().tolist()
        return torch.stack([torch.view_as_real(pi_of(mol, complex(*f))) for f in z])
    if kind == "screen":
        z, rhs = frequencies(case, seed).cpu().tolist(), right_hand_sides(case, seed, mol)
        return torch.stack([torch.view_as_real(w_of(mol, complex(*f), b)) for f, b in zip(z, rhs)])
    axis = imaginary_axis(mol)
    eps, n_occ, nc = mol["eps"], mol["n_occ"], case["n_core"]
    ef = 0.5 * (eps[n_occ - 1] + eps[n_occ])
    if kind == "sigma":
        grid = window(mol, case["points"])
        sig = np.zeros((nc, len(grid)), dtype=complex)
        dec = np.zeros((nc, len(grid)))
        for j, w in enumerate(grid):
            for c in range(nc):
                sig[c, j] = -imaginary_term(mol, axis, c, float(w))
            for m in range(case["n_states"]):
                f = prefactor(eps[m], w, ef)
                if f:
                    v = f * w_of(mol, complex(abs(eps[m] - w), ETA), mol["o_core"][m]).cpu().numpy()
                    sig[:, j] += v
                    if m < nc:
                        dec[m, j] += v[m].imag
        sx = -mol["o_core"][:n_occ].square().sum((0, 2))
        return np.stack([sig.real, sig.imag], -1), dec, sx
    dh = exact_dh(mol, axis, nc)
    qp = mol["eps_d"][:nc] + dh  # the fixed point of the shifted equation
    if kind == "qp":
        return qp, dh, None
    grid = relative(case["points"])
    im = torch.zeros((nc, len(grid)), dtype=torch.float64, device="cuda")
    core = torch.stack([mol["o_core"][c, c] for c in range(nc)])
    for j, x in enumerate(grid):
        f = [prefactor(eps[c], eps[c] + x, ef) for c in range(nc)]
        if any(f):
            im[:, j] = torch.tensor(f, device="cuda", dtype=torch.float64) * w_of(mol, complex(abs(x), ETA), core).imag
    a, nu = exact_cumulant(torch.as_tensor(grid, device="cuda")[None].repeat(nc, 1), im, 1 << 16)
    return qp, dh, None, im, a, nu
