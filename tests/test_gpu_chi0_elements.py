"""FP64 polarizability element by element, where the largest entry of one row meets a zero or a small entry of the other: the
error of an element is bounded by the sum S of the magnitudes of its own terms, not by the rows' maxima.

Bound: the product D O is rounded once (2^-53 S); digits and fixed point leave at most 0.64 sqrt(N_ov) 2^-54 S, or the element is
summed in FP64 by 32 lanes (at most N_ov / 256 + 7 + 8 additions in a chain); the sums of the digit orders up to a cut are at
most 3.1 S and three of them are rounded. The reference takes D as the library computes it, read
from polarizabilities of unit vectors (one exact product each)."""
import numpy as np
import pytest

from oracle import gwc_oracle as G
from paper_2412_17132_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _chi0(eps, n_occ, o, zs):
    from paper_2412_17132_gb300 import gwc

    o_core = np.zeros((len(eps), 1, o.shape[0]))
    ctx = gwc.Context(torch.as_tensor(eps, device="cuda"), n_occ, [0], torch.as_tensor(o, device="cuda"),
                      torch.as_tensor(o_core, device="cuda"), prec="fp64")
    got = ctx.build_chi0(torch.tensor([[z.real, z.imag] for z in zs], dtype=torch.float64, device="cuda")).cpu().numpy()
    assert ctx.sync_status() == 0
    ctx.close()
    return got


def _check(mol, o, zs):
    n_ov = o.shape[1]
    eye = np.eye(n_ov)
    d = np.concatenate([np.diagonal(_chi0(mol.eps, mol.n_occ, eye, [z])[0]).T[:, None] for z in zs], 1).reshape(n_ov, len(zs), 2)
    got = _chi0(mol.eps, mol.n_occ, o, zs)
    bound = max(10.3 + 0.32 * np.sqrt(n_ov), n_ov / 256 + 16) * 2.0 ** -53
    ol = o.astype(np.longdouble)
    for f, z in enumerate(zs):
        for part in (0, 1):
            b = ol * d[:, f, part].astype(np.longdouble)
            ref, s = ol @ b.T, np.abs(ol) @ np.abs(b).T
            assert np.all(np.abs(got[f, :, :, part] - ref) <= bound * s), (z, part, float(np.max(np.abs(got[f, :, :, part] - ref) / s)))


def _molecule(n_states=73, n_occ=16, seed=1):
    return synth.small(n_states=n_states, n_occ=n_occ, n_core=1, n_aux=8, seed=seed)


@pytest.mark.parametrize("eta", [1e-3, 1e-5, 1e-8])
@pytest.mark.parametrize("n_aux", [64, 130, 257])
def test_a_pole_that_some_rows_do_not_see(n_aux, eta):
    mol = _molecule()
    d = G.transition_energies(mol.eps, mol.n_occ)
    k = 137
    o = np.random.default_rng(n_aux).normal(0.0, 0.02, (n_aux, len(d)))
    o[0::3, k] = 0.0
    o[1::3, k] *= 1e-9
    _check(mol, o, [complex(d[k], eta), complex(d[k] + 2e-3, eta), complex(0.0, 0.7)])


def test_rows_that_hardly_overlap():
    mol = _molecule(seed=2)
    n_ov = 16 * 57
    o = np.random.default_rng(3).normal(0.0, 0.02, (150, n_ov))
    o[:70, n_ov // 2 :] *= 1e-14
    o[70:140, : n_ov // 2] = 0.0
    o[149] = 0.0
    _check(mol, o, [complex(0.4, 1e-3), complex(9.6, 1e-3)])


def test_columns_and_rows_of_very_different_size():
    mol = _molecule(n_states=40, n_occ=7, seed=4)
    r = np.random.default_rng(5)
    o = r.normal(0.0, 1.0, (100, 7 * 33)) * 10.0 ** r.uniform(-13, 0, 7 * 33)
    _check(mol, o * 10.0 ** r.uniform(-120, 20, 100)[:, None], [complex(0.3, 1e-3), complex(0.2, 0.1)])


def test_rows_of_the_largest_and_smallest_digits():
    """Entries next to powers of two (digits of -128 and 127, carries through all of them) and rows of one value."""
    mol = _molecule(n_states=34, n_occ=4, seed=6)
    n_ov = 4 * 30
    r = np.random.default_rng(7)
    o = 2.0 ** r.integers(-40, 1, (80, n_ov)) * (1.0 + r.choice([-1.0, 0.0, 1.0], (80, n_ov)) * 2.0 ** -52) * r.choice([-1, 1], (80, n_ov))
    o[3] = 1.0 - 2.0 ** -53
    o[4] = -1.0
    o[5] = np.where(np.arange(n_ov) == 9, 1.0, 2.0 ** -60)
    _check(mol, o, [complex(0.3, 1e-3), complex(0.0, 0.5)])
