"""SIMT factorisations on both sides of the rule that chooses one CTA per matrix or launches over all of them (sizes, matrices at
once, appended rows): W from either equals the other's, and the oracle's LU solve at 1e-9 of the largest value in FP64."""
import numpy as np
import pytest

from oracle import gwc_oracle as G
from paper_2412_17132_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_aux", [64, 65, 128, 129, 193, 257, 321])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_batches_on_both_sides_agree(n_aux, prec):
    from paper_2412_17132_gb300 import gwc

    f = 310
    mol = synth.small(n_states=40, n_occ=5, n_core=2, n_aux=n_aux, seed=n_aux)
    rng = np.random.default_rng(n_aux)
    zs = np.stack([rng.uniform(0.0, 10.0, f), rng.uniform(0.05, 0.5, f)], 1)
    rhs = mol.o_core[rng.integers(0, 40, (f, 2)), rng.integers(0, 2, (f, 2))]
    z, b = torch.as_tensor(zs, device="cuda"), torch.as_tensor(rhs, device="cuda")
    delta = G.transition_energies(mol.eps, mol.n_occ)
    some = [0, 100, 309]
    ref = np.stack([G.screened_wc(G.chi0(mol.o_ov, delta, complex(*zs[i])), rhs[i].T) for i in some])
    tol = (1e-9 if prec == "fp64" else 2e-3) * np.max(np.abs(ref))
    outs, sig = [], []
    for batch in (7, 140, 152, 300, 310):
        ctx = gwc.Context.from_molecule(mol, prec=prec, batch=batch)
        w = ctx.screen(z, b).cpu().numpy()
        sig.append(ctx.sigma_core(np.linspace(-10.8, -10.2, 5))[0].cpu().numpy())  # rows appended to the matrices
        assert ctx.sync_status() == 0
        ctx.close()
        outs.append(w[..., 0] + 1j * w[..., 1])
        assert np.max(np.abs(outs[-1][some] - ref)) <= tol
    for o, s in zip(outs[1:], sig[1:]):
        assert np.max(np.abs(o - outs[0])) <= tol
        assert np.max(np.abs(s - sig[0])) <= (1e-8 if prec == "fp64" else 2e-3) * np.max(np.abs(sig[0]))
