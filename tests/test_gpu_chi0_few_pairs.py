"""FP64 polarizability on both sides of the shortest contraction that goes by digits, against an extended-precision sum. Bound: the
rounding of the scaled operand (a few 2^-53 per term, D_ia's own included) and that of a sum of N_ov terms, in units of the
sum of the terms' magnitudes."""
import numpy as np
import pytest

from oracle import gwc_oracle as G
from paper_2412_17132_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_states,n_occ", [(3, 1), (20, 5), (44, 3), (32, 4), (31, 4), (117, 1)])  # N_ov 2, 75, 123, 112, 108, 116
@pytest.mark.parametrize("n_aux", [64, 130])
def test_against_extended_precision(n_states, n_occ, n_aux):
    from paper_2412_17132_gb300 import gwc

    mol = synth.small(n_states=n_states, n_occ=n_occ, n_core=1, n_aux=n_aux, seed=n_states)
    zs = [complex(0.0, 0.8), complex(0.9, 0.05), complex(11.5, 1e-3)]
    ctx = gwc.Context.from_molecule(mol, prec="fp64")
    got = ctx.build_chi0(torch.tensor([[v.real, v.imag] for v in zs], dtype=torch.float64, device="cuda")).cpu().numpy()
    assert ctx.sync_status() == 0
    ctx.close()
    d = G.transition_energies(mol.eps, mol.n_occ).astype(np.longdouble)
    o = mol.o_ov.astype(np.longdouble)
    for f, z in enumerate(zs):
        x, y = np.longdouble(z.real), np.longdouble(z.imag)
        a, b = (x - d) * (x + d) - y * y, 2 * x * y
        s = 4 * d / (a * a + b * b)
        for part, c in ((0, s * a), (1, -s * b)):
            size = np.abs(o * c) @ np.abs(o).T
            # d and z^2 - d^2 each to a few 2^-53 of (|z| + d)^2, which they may be far below
            near = float(np.max((abs(z) + d) ** 2 / np.sqrt(a * a + b * b)))
            assert np.all(np.abs(got[f, :, :, part] - (o * c) @ o.T) <= (o.shape[1] + 16 * near) * 2.0 ** -53 * size + 1e-300)
