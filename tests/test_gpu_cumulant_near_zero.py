"""Cumulant spectrum with grid points next to zero against the oracle: c_j = q_j beta_j / w_j^2 is huge there, while its term
c_j (e^{-i w_j t} - 1) need not be. A window such as linspace(-25 eV, 5 eV, 181) passes 1.1e-16 where 0 is meant.

Tolerance: 1e-10 of the peak, as for any other grid, plus what the rounding of the points next to zero does to either side:
an error of k 2^-53 in cos and sin moves C~(t) by at most k 2^-53 sum_j |c_j| (|sin w_j t| + [cos w_j t != 1]), with k = 4 where
they are evaluated at every time and k = 64 where 32 times share a rotation, and the spectrum by dt / pi sum_k |g_k| of that."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EV = 27.211386245988
N_T, T_MAX, ETA = 1 << 14, 2000.0, 1e-3


def _context(n_core):
    from paper_2412_17132_gb300 import gwc

    eps = torch.linspace(-10.5, 3.0, 12, dtype=torch.float64, device="cuda")
    o_ov = torch.zeros((8, (n_core + 1) * (11 - n_core)), dtype=torch.float64, device="cuda")
    o_core = torch.zeros((12, n_core, 8), dtype=torch.float64, device="cuda")
    return gwc.Context(eps, n_core + 1, list(range(n_core)), o_ov, o_core, prec="fp64", n_t=N_T, t_max=T_MAX, eta=ETA)


def _rounding(w, im, k):
    from oracle import gwc_oracle as G

    near = (np.abs(w) * T_MAX <= 2.0 ** -10) & (w != 0.0) & (im != 0.0)
    beta = np.abs(im) / np.pi
    t = T_MAX / N_T * np.arange(N_T)
    x = np.outer(t, w[near])
    c = (G.trapezoid_weights(w) * beta)[near] / w[near] ** 2
    dc = k * 2.0 ** -53 * (np.abs(np.sin(x)) + (np.cos(x) != 1.0)) @ c
    g = np.exp(G.cumulant_ct(w, beta, t).real - ETA * t)
    return T_MAX / N_T / np.pi * float(np.sum(g * dc))


def _check(ws, ims, k=4, rel=1e-10):
    from oracle import gwc_oracle as G

    ctx = _context(len(ws))
    a, _ = ctx.cumulant_spectrum(torch.as_tensor(np.stack(ws), device="cuda"), torch.as_tensor(np.stack(ims), device="cuda"))
    ctx.sync()
    for c, (w, im) in enumerate(zip(ws, ims)):
        ref = G.gwc_spectrum(w, im, ETA, N_T, T_MAX)[1]
        assert np.all(np.isfinite(ref))
        err = np.max(np.abs(a[c].cpu().numpy() - ref))
        assert err <= rel * np.max(np.abs(ref)) + _rounding(w, im, k), c
    ctx.close()


def _window(n, seed):
    w = np.linspace(-25.0 / EV, 5.0 / EV, n)
    im = np.random.default_rng(seed).uniform(0.0, 0.02, n) * np.minimum(1.0, (w / 0.3) ** 2)
    return w, np.where(w < -1e-6, im, 0.0)


@pytest.mark.parametrize("n", [181, 901])
@pytest.mark.parametrize("near", [1.1102230246251565e-16, -1e-15, 1e-9])
def test_a_point_next_to_zero(n, near):
    ws, ims = [], []
    for value in (0.0, 7e-20, 1e-12, 1e-5):
        w, im = _window(n, n)
        j = int(np.argmin(np.abs(w)))
        w[j], im[j] = near, value
        ws.append(w)
        ims.append(im)
    _check(ws, ims)


@pytest.mark.parametrize("points", [8, 9])  # as many as are taken out of the blocks, and one more (the direct sum)
def test_several_points_next_to_zero_in_any_order(points):
    w, im = _window(300, 5)
    j = np.random.default_rng(1).choice(300, points, replace=False)
    w[j] = 1e-8 * (np.arange(points) - 3.5)
    im[j] = 1e-13
    _check([w, _window(300, 6)[0]], [im, _window(300, 6)[1]], k=4 if points == 8 else 64)


def test_large_coefficients_that_are_not_next_to_zero():
    """sum |c_j| on both sides of the largest that goes by blocks (2^14)."""
    ws, ims = [], []
    for total in (1.5e4, 1.8e4):
        w, im = _window(400, 7)
        j = int(np.argmin(np.abs(w)))
        w[j] = -2e-6
        q = 0.5 * (w[j + 1] - w[j - 1])
        im[j] = total * np.pi * w[j] ** 2 / q
        ws.append(w)
        ims.append(im)
    # (not next to zero, which ends at 2^-10 / t_max = 4.9e-7; 64 2^-53 sum |c_j| = 1.3e-10)
    _check(ws, ims, rel=2.3e-10)
