"""FP64 polarizability from 8-bit digits on the tensor cores (fixed-point rows, exact integer sums), through the C ABI, at the
edges of its tiles, chunks and segments, against an extended-precision sum. Derived bound: the scaled operand's own
rounding and that of D_ia (a few 2^-53 per term) and the digits dropped (2^-63 of the product of the row maxima, which
exceed the typical |O| and |D O| by at most about 1e3 here) keep the error below 1e-15 of the largest |Pi|."""
import numpy as np
import pytest

from oracle import gwc_oracle as G
from paper_2412_17132_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _ext(mol, z):
    d = G.transition_energies(mol.eps, mol.n_occ).astype(np.longdouble)
    x, y = np.longdouble(z.real), np.longdouble(z.imag)
    a, b = (x - d) * (x + d) - y * y, 2 * x * y
    s = 4 * d / (a * a + b * b)
    o = mol.o_ov.astype(np.longdouble)
    return (o * (s * a)) @ o.T, (o * (-s * b)) @ o.T


# N_ov = n_occ (n_states - n_occ): 1 to 17 chunks of 64, multiples of 64 and ragged; N_aux around 64 and 128-row tiles
@pytest.mark.parametrize("n_aux,n_states,n_occ", [(64, 20, 4), (65, 21, 5), (127, 33, 1), (128, 34, 2), (129, 40, 8), (200, 73, 16),
                                                  (256, 43, 11), (257, 48, 23), (70, 68, 34), (66, 3, 1)])
def test_chi0_fixed_point_against_extended_precision(n_aux, n_states, n_occ):
    from paper_2412_17132_gb300 import gwc

    mol = synth.small(n_states=n_states, n_occ=n_occ, n_core=1, n_aux=n_aux, seed=n_aux)
    zs = [complex(0.0, 0.8), complex(0.0, 0.0), complex(0.1, 1e-3), complex(0.9, 0.05), complex(11.5, 1e-3)]
    ctx = gwc.Context.from_molecule(mol, prec="fp64", batch=2)
    got = ctx.build_chi0(torch.tensor([[v.real, v.imag] for v in zs], dtype=torch.float64, device="cuda")).cpu().numpy()
    assert ctx.sync_status() == 0
    for f, z in enumerate(zs):
        re, im = _ext(mol, z)
        for part, ref in ((0, re), (1, im)):
            assert np.max(np.abs(got[f, :, :, part] - ref)) <= 1e-15 * float(np.max(np.abs(re))), (z, part)
    ctx.close()


def test_rows_of_very_different_size_and_of_zeros():
    from paper_2412_17132_gb300 import gwc

    mol = synth.small(n_states=30, n_occ=5, n_core=1, n_aux=90, seed=2)
    mol.o_ov *= np.logspace(-150, 3, 90)[:, None]
    mol.o_ov[17] = 0.0
    ctx = gwc.Context.from_molecule(mol, prec="fp64")
    z = complex(0.2, 0.1)
    got = ctx.build_chi0(torch.tensor([[z.real, z.imag]], dtype=torch.float64, device="cuda")).cpu().numpy()[0]
    s = np.sqrt(np.sum(mol.o_ov.astype(np.longdouble) ** 2, axis=1))
    s[17] = 1
    for part, ref in enumerate(_ext(mol, z)):
        assert np.max(np.abs((got[:, :, part] - ref) / s[:, None] / s[None, :])) <= 1e-14  # per row and column
        assert np.all(got[17, :, part] == 0.0) and np.all(got[:, 17, part] == 0.0)
    ctx.close()


def test_a_frequency_on_a_pole_gives_what_the_sum_gives():
    from paper_2412_17132_gb300 import gwc

    mol = synth.small(n_states=30, n_occ=5, n_core=1, n_aux=80, seed=3)
    d = G.transition_energies(mol.eps, mol.n_occ)
    ctx = gwc.Context.from_molecule(mol, prec="fp64")
    z = torch.tensor([[float(d[7]), 0.0], [0.3, 0.2]], dtype=torch.float64, device="cuda")
    got = ctx.build_chi0(z).cpu().numpy()
    assert np.isnan(got[0]).all() and np.isfinite(got[1]).all()  # D = inf * 0 there
    ctx.close()
