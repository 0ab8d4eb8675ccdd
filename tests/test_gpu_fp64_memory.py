"""FP64 contexts on a device whose memory is nearly taken: what fits without the digits of the tensor-core polarizability is
created, and computes with the SIMT build."""
import numpy as np
import pytest

from oracle import gwc_oracle as G
from paper_2412_17132_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _build(ctx, mol, z):
    ctx.load(torch.as_tensor(mol.eps, device="cuda"), torch.as_tensor(mol.o_ov, device="cuda"),
             torch.as_tensor(mol.o_core, device="cuda"), core_idx=np.arange(mol.o_core.shape[1]), n_occ=mol.n_occ)
    p = ctx.build_chi0(torch.tensor([[z.real, z.imag]], dtype=torch.float64, device="cuda"))
    assert ctx.sync_status() == 0
    return p.cpu().numpy()[0]


def test_a_context_that_fits_without_the_digits():
    from paper_2412_17132_gb300 import gwc

    mol = synth.small(n_states=60, n_occ=8, n_core=1, n_aux=150, seed=4)
    z = complex(0.4, 1e-3)
    # O of 3000 x 100 000: 2.4 GB, its digits 6.6 GB
    shape = dict(n_states=1100, n_occ=100, n_aux=3000, n_core=1)
    free = torch.cuda.mem_get_info()[0]
    if free < 16 << 30:
        pytest.skip("the device's memory is taken already")
    hold = torch.empty(free - (6 << 30), dtype=torch.uint8, device="cuda")
    try:
        left = torch.cuda.mem_get_info()[0]
        ctx = gwc.Context.with_capacity(shape["n_states"], shape["n_occ"], shape["n_aux"], shape["n_core"], prec="fp64", batch=1)
        taken = left - torch.cuda.mem_get_info()[0]
        assert taken < 4 << 30
        short = _build(ctx, mol, z)
        ctx.close()
    finally:
        del hold
        torch.cuda.empty_cache()
    ctx = gwc.Context.with_capacity(shape["n_states"], shape["n_occ"], shape["n_aux"], shape["n_core"], prec="fp64", batch=1)
    ample = _build(ctx, mol, z)
    ctx.close()
    ref = G.chi0(mol.o_ov, G.transition_energies(mol.eps, mol.n_occ), z)
    for got in (short, ample):
        assert np.max(np.abs(got[..., 0] + 1j * got[..., 1] - ref)) <= 1e-13 * np.max(np.abs(ref))
    assert not np.array_equal(short, ample)  # two kernels: sequential sums and digits


def test_the_variable_keeps_the_simt_build(monkeypatch):
    from paper_2412_17132_gb300 import gwc

    mol = synth.small(n_states=60, n_occ=8, n_core=1, n_aux=150, seed=5)
    z = torch.tensor([[0.4, 1e-3]], dtype=torch.float64, device="cuda")
    out = []
    for value in (None, "simt"):
        if value:
            monkeypatch.setenv("GWC_CHI0_FP64", value)
        ctx = gwc.Context.from_molecule(mol, prec="fp64")
        out.append(ctx.build_chi0(z).cpu().numpy())
        assert ctx.sync_status() == 0
        ctx.close()
    assert not np.array_equal(*out)
    assert np.max(np.abs(out[0] - out[1])) <= 1e-13 * np.max(np.abs(out[1]))
