"""FP64 contexts compute with every wait bound, however short: the bound is the mixed-precision kernels' (the FP64
polarizability had no waits before it ran on the tensor cores)."""
import pytest

from paper_2412_17132_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_aux", [48, 300])
def test_a_short_bound_changes_nothing(n_aux):
    from paper_2412_17132_gb300 import gwc

    mol = synth.small(n_states=60, n_occ=9, n_core=2, n_aux=n_aux, seed=61)
    z = torch.tensor([[0.0, 0.6], [0.41, 1e-3], [3.3, 1e-3]], dtype=torch.float64, device="cuda")
    out = []
    for wait_us in (0, 1):
        ctx = gwc.Context.from_molecule(mol, prec="fp64", wait_us=wait_us)
        p, (eqp, _, _) = ctx.build_chi0(z), ctx.qp_solve()
        assert ctx.sync_status() == 0
        out.append((p.cpu(), eqp.cpu()))
        ctx.close()
    assert all(torch.equal(a, b) for a, b in zip(*out))
