"""The order-2 Poisson solve with elimination along x (z and y transforms, recursions along x) at
the edges of its kernels: the smallest meshes, meshes whose columns leave a partial tile, the
largest planes of the FP32 form and the first mesh beyond them, the folded and ragged tensor-core
passes, and boxes of several sizes in one launch."""
import pytest

torch = pytest.importorskip("torch")

from test_gpu_parity import CASES_PM, _check_pm_force  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def _one_box(n, ng):
    return dict(L=4.0 * n, Np=n, Ntiles=1, Nbuf=0, Ng=ng, nsteps=1, a_i=0.05, a_f=1.0)


# A force evaluation per mesh size and form; the tolerances are those of every force test
# (maximum 2e-4 and RMS 2e-5 of the largest force: FP32 transforms of length Ng carry
# ~sqrt(Ng) 2^-24 relative error, the recursions ~sqrt(Ng) 2^-24 as well, and the gradient
# amplifies it by ~10-100).
@pytest.mark.parametrize("ng,variant", [(3, "tc"), (8, "tc3"), (8, "simt"), (11, "simt"), (12, "tc3"), (47, "tc"), (64, "tc3"),
                                        (65, "simt"), (92, "tc3"), (96, "simt"), (113, "simt"), (128, "simt"),
                                        (129, "simt"), (132, "tc"), (160, "tc"), (191, "tc")])
def test_force_at_mesh_edges(ng, variant):
    _check_pm_force(_one_box(min(ng, 24) // 2 * 2 if ng > 3 else 2, ng), variant, False)


@pytest.mark.parametrize("variant", ["simt", "tc", "tc3"])
def test_force_of_boxes_of_several_sizes(variant):
    _check_pm_force(CASES_PM["uneven"], variant, False)
