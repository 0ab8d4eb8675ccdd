"""The launch shapes of the tensor-core polarizability: chosen by size, one CTA pair per item, persistent, and what the autotuner
leaves behind give the same matrices."""
import numpy as np
import pytest

from paper_2412_17132_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_aux", [90, 300])
def test_launch_shapes_agree(n_aux):
    from paper_2412_17132_gb300 import gwc

    mol = synth.small(n_states=60, n_occ=9, n_core=2, n_aux=n_aux, seed=59)
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    z = torch.tensor([[0.0, 0.6], [0.41, 1e-3], [3.3, 1e-3]], dtype=torch.float64, device="cuda")
    outs = []
    for ctas in (0, n_sm, 1 << 30, "tuned"):
        tuned = ctas == "tuned"
        ctx = gwc.Context.from_molecule(mol, prec="bf16x3", qp_mode="hedin", batch=32, chi0_ctas=0 if tuned else ctas)
        if tuned:
            ctx.request_plan(np.linspace(-1.0, 0.2, 61))
            ctx.autotune()
            if ctx.chi0_tile():  # (the one-CTA tiles sum in another order)
                ctx.close()
                continue
        outs.append(ctx.build_chi0(z))
        assert ctx.sync_status() == 0
        ctx.close()
    assert all(torch.equal(outs[0], o) for o in outs[1:])
