"""The adjoint with an odd number of particles per side: the second derivatives of the initial
conditions' chain are rows of an odd number of floats each."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth_inputs  # noqa: E402
from gpu_common import oracle_cfg  # noqa: E402
from oracle import adjoint  # noqa: E402
from test_gpu_adjoint import _gpu_loss_grad, _pkg, _sim, _target  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


# Seeds and bounds of the even case (FP32 against the FP64 adjoint: a particle at a kink of its CIC
# weights may take the other one-sided derivative, a wrong term moves every seed).
@pytest.mark.parametrize("lpt_order", [1, 2])
@pytest.mark.parametrize("ntiles,nbuf", [(1, 0), (3, 2)])
def test_backward_with_odd_sides_matches_fp64_oracle_adjoint(ntiles, nbuf, lpt_order):
    kw = dict(L=45.0, Np=15, Ntiles=ntiles, Nbuf=nbuf, mesh_ratio=1, nsteps=3, a_i=0.05, a_f=1.0, lpt_order=lpt_order)
    cfg = oracle_cfg(kw)
    target = _target(kw, 22)
    sim = _sim(kw, "simt")
    rels = []
    for seed in (21, 23, 24):
        w = synth_inputs.white_noise(15, seed)
        val, g = _gpu_loss_grad(sim, w, target)
        _pkg().scola_device_status(sim.ctx)
        val_o, g_o = adjoint.loss_and_grad(w.astype(np.float64), cfg, target)
        assert abs(val / val_o - 1) < 1e-4
        rels.append(np.linalg.norm(g - g_o) / np.linalg.norm(g_o))
    sim.close()
    print("gradient vs FP64 oracle, 15 a side: %s" % rels)
    assert np.median(rels) < 1e-3 and max(rels) < 5e-3, rels
