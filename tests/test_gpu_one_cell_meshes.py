"""Boxes of one cell (no buffer around a tile of one particle) in the dense FP32 solve: the
elimination along x has a single row there and no second half, alone and beside larger boxes."""
import pytest

torch = pytest.importorskip("torch")

from test_gpu_parity import _check_pm_force  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


# The tolerances of every force test.  Meshes of 1 and 3 cells, of 1 alone, of 2 and 4.
@pytest.mark.parametrize("ntiles,buffers", [(4, [0, 1] * 32), (4, [0] * 64), (2, [0, 1] * 4)])
def test_force_of_boxes_of_one_cell(ntiles, buffers):
    _check_pm_force(dict(L=16.0, Np=4, Ntiles=ntiles, Nbuf=0, buffers=buffers, mesh_ratio=1, nsteps=1, a_i=0.05,
                         a_f=1.0), "simt", False)
