"""Cumulant spectrum against the oracle at the edges of the blocks of times: grids around the largest frequency that a
block takes (w_max dt = 1/2, beyond it the direct sum), times too few for one block, and grid sizes around a chunk."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _context(n_core, n_t, t_max, eta):
    from paper_2412_17132_gb300 import gwc

    eps = torch.linspace(-10.5, 3.0, 12, dtype=torch.float64, device="cuda")
    o_ov = torch.zeros((8, (n_core + 1) * (11 - n_core)), dtype=torch.float64, device="cuda")
    o_core = torch.zeros((12, n_core, 8), dtype=torch.float64, device="cuda")
    return gwc.Context(eps, n_core + 1, list(range(n_core)), o_ov, o_core, prec="fp64", n_t=n_t, t_max=t_max, eta=eta)


# (n_core, n_w, n_t, t_max, largest frequency of each core)
CASES = [
    (1, 1, 16, 30.0, [0.9]),                       # fewer times than one block, one grid point
    (1, 2, 32, 60.0, [0.2]),                       # one block
    (2, 255, 4096, 2000.0, [0.95, 1.0239]),        # blocks of 32 times, just inside w_max dt = 1/2
    (2, 256, 4096, 2000.0, [0.95, 1.0241]),        # one core on blocks, the other just beyond
    (3, 257, 4096, 500.0, [0.95, 5.0, 0.01]),      # a block size of its own per core, one direct
    (1, 1025, 1 << 16, 2000.0, [0.9]),             # long blocks, several chunks of the grid
    (9, 40, 1 << 16, 2000.0, [0.9] * 9),           # several blocks per item
]


@pytest.mark.parametrize("n_core,n_w,n_t,t_max,top", CASES)
def test_spectrum_at_block_edges_matches_the_oracle(n_core, n_w, n_t, t_max, top):
    from oracle import gwc_oracle as G

    eta = 1e-3
    rng = np.random.default_rng(n_w + n_t)
    w = np.stack([np.linspace(-top[c], 0.2 * top[c], n_w) for c in range(n_core)])
    im = np.where(w < 0, rng.uniform(0.0, 0.02, w.shape) * np.minimum(1.0, (w / 0.3) ** 2), 0.0)
    ctx = _context(n_core, n_t, t_max, eta)
    a, nu = ctx.cumulant_spectrum(torch.as_tensor(w, device="cuda"), torch.as_tensor(im, device="cuda"))
    ctx.sync()
    for c in range(n_core):
        nu_ref, a_ref = G.gwc_spectrum(w[c], im[c], eta, n_t, t_max)
        assert np.max(np.abs(a[c].cpu().numpy() - a_ref)) <= 1e-10 * np.max(np.abs(a_ref))
        assert np.max(np.abs(nu.cpu().numpy() - nu_ref)) <= 1e-12 * np.max(np.abs(nu_ref))
    ctx.close()


def test_a_grid_that_is_not_finite_gives_no_finite_spectrum():
    ctx = _context(1, 4096, 2000.0, 1e-3)
    w = torch.linspace(-0.9, 0.2, 100, dtype=torch.float64, device="cuda")[None].repeat(1, 1)
    w[0, 3] = float("nan")
    a, _ = ctx.cumulant_spectrum(w, torch.full((1, 100), 0.01, dtype=torch.float64, device="cuda"))
    ctx.sync()
    assert torch.isnan(a).all()
    ctx.close()
