"""gwc_screen on both sides of the rule that chooses between the cluster forms of the forward substitution and the one-CTA
kernel (panels, right-hand sides, matrices at once): in FP64 against the oracle's LU solve at 1e-9 of the largest value,
and every way of splitting the same frequencies into batches within it of the others."""
import numpy as np
import pytest

from oracle import gwc_oracle as G
from paper_2412_17132_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_aux", [65, 128, 129, 257])
@pytest.mark.parametrize("r", [9, 17, 32])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_batches_of_any_size_agree(n_aux, r, prec):
    from paper_2412_17132_gb300 import gwc

    f = 160
    mol = synth.small(n_states=40, n_occ=5, n_core=2, n_aux=n_aux, seed=n_aux)
    rng = np.random.default_rng(n_aux + r)
    zs = np.stack([rng.uniform(0.0, 10.0, f), rng.uniform(0.05, 0.5, f)], 1)
    rhs = mol.o_core[rng.integers(0, 40, (f, r)), rng.integers(0, 2, (f, r))]
    z, b = torch.as_tensor(zs, device="cuda"), torch.as_tensor(rhs, device="cuda")
    delta = G.transition_energies(mol.eps, mol.n_occ)
    some = [0, 3, 77, 159]
    ref = np.stack([G.screened_wc(G.chi0(mol.o_ov, delta, complex(*zs[i])), rhs[i].T) for i in some])
    tol = (1e-9 if prec == "fp64" else 2e-3) * np.max(np.abs(ref))
    outs = []
    for batch in (5, 33, 100, 160):
        ctx = gwc.Context.from_molecule(mol, prec=prec, batch=batch)
        w = ctx.screen(z, b).cpu().numpy()
        assert ctx.sync_status() == 0
        ctx.close()
        outs.append(w[..., 0] + 1j * w[..., 1])
        assert np.max(np.abs(outs[-1][some] - ref)) <= tol
    for o in outs[1:]:
        assert np.max(np.abs(o - outs[0])) <= tol
