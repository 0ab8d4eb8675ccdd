"""Right-hand sides of the imaginary-axis table: one conversion written for several nodes.

Each node of the table takes the same N_states N_core rows; a CTA converts a row once for as many nodes as leave the chip
full (one of 33, groups of 8 with a last group of one, and all of them). The table enters Sigma^c, which is compared
with the FP64 oracle within the bounds of the other Sigma^c tests: FP64 1e-8 Ha, split BF16 2e-2 relative plus 2e-3 Ha.
"""
import numpy as np
import pytest

from oracle import gwc_oracle as G
from paper_2412_17132_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,rel,ab", [("fp64", 0.0, 1e-8), ("bf16x3", 2e-2, 2e-3)])
@pytest.mark.parametrize("n_states,n_core", [(37, 1), (100, 6), (250, 10)])
def test_table_right_hand_sides_vs_oracle(n_states, n_core, prec, rel, ab):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_17132_gb300 import gwc

    mol = synth.small(n_states=n_states, n_occ=n_core + 3, n_core=n_core, n_aux=21, seed=n_states)
    omega = mol.eps[0] + np.array([-0.7, -0.1, 0.2])
    ctx = gwc.Context.from_molecule(mol, prec=prec)
    sig, _, _ = ctx.sigma_core(omega, want_dec=False)
    assert ctx.sync_status() == 0
    got = sig.cpu().numpy()
    got = got[..., 0] + 1j * got[..., 1]
    ctx.close()
    ref, _ = G.System.from_molecule(mol).sigma_c_grid(omega)
    assert np.all(np.abs(got - ref) <= rel * np.abs(ref) + ab), np.max(np.abs(got - ref))
