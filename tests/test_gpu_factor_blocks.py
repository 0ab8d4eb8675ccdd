"""The 16-column blocks inside a factorisation panel and its rows below, at the sizes where a block is ragged (through the C
ABI): W and Sigma^c of both tensor-core forms against the FP64 oracle. The frequencies lie away from the RPA poles (2e-3 of the
largest value is the bound that the other factorisation tests use there), with 3 right-hand sides appended as rows."""
import os

import numpy as np
import pytest

from oracle import gwc_oracle as G
from paper_2412_17132_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ZS = [complex(0.0, 0.9), complex(2.9, 0.5), complex(6.0, 1.0)]


@pytest.mark.parametrize("factor", ["tc", "split"])
@pytest.mark.parametrize("n_aux", [2, 15, 16, 17, 31, 33, 47, 49, 66, 79, 81, 111, 129, 143, 177])
def test_blocks_of_a_panel_against_the_oracle(n_aux, factor, monkeypatch):
    from paper_2412_17132_gb300 import gwc

    monkeypatch.setenv("GWC_FACTOR", factor)
    mol = synth.small(n_states=40, n_occ=6, n_core=3, n_aux=n_aux, seed=300 + n_aux)
    ctx = gwc.Context.from_molecule(mol, prec="bf16x3")
    z = torch.tensor([[v.real, v.imag] for v in ZS], dtype=torch.float64, device="cuda")
    rhs = np.stack([mol.o_core[[0, 5, 20, 39], 0, :] for _ in ZS])
    got = ctx.screen(z, torch.as_tensor(rhs, device="cuda")).cpu().numpy()
    assert ctx.sync_status() == 0
    delta = G.transition_energies(mol.eps, mol.n_occ)
    for f, v in enumerate(ZS):
        ref = G.screened_wc(G.chi0(mol.o_ov, delta, v), rhs[f].T)
        assert np.max(np.abs(got[f, :, 0] + 1j * got[f, :, 1] - ref)) <= 2e-3 * np.max(np.abs(ref))
    # the appended rows: Sigma^c above the valence residues, every matrix with 3 rows below the last panel
    w = float(mol.eps[5]) + 0.01
    sig, _, _ = ctx.sigma_core([w])
    ref = np.array(G.System.from_molecule(mol).sigma_c(w)[0])
    s = sig[:, 0].cpu().numpy()
    assert np.max(np.abs(s[:, 0] + 1j * s[:, 1] - ref)) <= 2e-2 * np.max(np.abs(ref)) + 2e-3
    ctx.close()
