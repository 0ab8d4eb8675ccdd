"""gwc_build_chi0's full matrix at the edges of the 32 x 32 output tiles: equal on both sides of the diagonal, and the same
doubles into an output that is not 16-byte aligned."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_aux", [1, 31, 32, 33, 64, 97])
@pytest.mark.parametrize("prec", ["bf16x3", "fp64", "fp32"])
def test_both_triangles_and_an_odd_output_address(n_aux, prec):
    from paper_2412_17132_gb300 import gwc, synth

    mol = synth.small(n_states=30, n_occ=5, n_core=1, n_aux=n_aux, seed=n_aux)
    ctx = gwc.Context.from_molecule(mol, prec=prec)
    z = torch.tensor([[0.2, 0.1], [3.0, 0.4]], dtype=torch.float64, device="cuda")
    a = ctx.build_chi0(z)
    assert torch.equal(a, a.transpose(1, 2)) and torch.isfinite(a).all()
    odd = torch.full((2 * n_aux * n_aux * 2 + 2,), 7.0, dtype=torch.float64, device="cuda")
    gwc._check(gwc.lib().gwc_build_chi0(ctx._ctx, z.data_ptr(), 2, odd.data_ptr() + 8, torch.cuda.current_stream().cuda_stream),
               ctx._ctx)
    ctx.sync()
    assert torch.equal(odd[1:-1].reshape(a.shape), a) and odd[0] == 7.0 and odd[-1] == 7.0
    ctx.close()
