"""gwc_screen for few right-hand sides (the cluster form of the forward substitution) and for more of them (one CTA per 64): in
FP64 against the oracle's LU solve at 1e-9 of the largest value, the bound of the other FP64 W tests, at panel edges,
with a lone right-hand side, at the last size of the few and beyond it, and over several frequency chunks."""
import numpy as np
import pytest

from oracle import gwc_oracle as G
from paper_2412_17132_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_aux,r,batch", [(1, 1, 0), (63, 3, 0), (64, 8, 2), (65, 9, 0), (130, 16, 3), (193, 17, 0), (320, 32, 0),
                                           (200, 33, 0), (641, 5, 2)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_screen_matches_the_oracle(n_aux, r, batch, prec):
    from paper_2412_17132_gb300 import gwc

    mol = synth.small(n_states=44, n_occ=6, n_core=2, n_aux=n_aux, seed=40 + n_aux)
    zs = [complex(0.0, 0.7), complex(2.5, 0.3), complex(0.4, 1e-2), complex(9.0, 0.5), complex(1.0, 0.2)]
    rng = np.random.default_rng(n_aux)
    rhs = np.stack([mol.o_core[rng.integers(0, 44, r), rng.integers(0, 2, r)] for _ in zs])
    ctx = gwc.Context.from_molecule(mol, prec=prec, batch=batch)
    z = torch.tensor([[v.real, v.imag] for v in zs], dtype=torch.float64, device="cuda")
    delta = G.transition_energies(mol.eps, mol.n_occ)
    ref = np.stack([G.screened_wc(G.chi0(mol.o_ov, delta, v), b.T) for v, b in zip(zs, rhs)])
    tol = 1e-9 if prec == "fp64" else 2e-3
    for _ in range(2):  # the second call finds its scratch
        w = ctx.screen(z, torch.as_tensor(rhs, device="cuda")).cpu().numpy()
        assert np.max(np.abs(w[..., 0] + 1j * w[..., 1] - ref)) <= tol * np.max(np.abs(ref))
    assert ctx.sync_status() == 0
    ctx.close()
