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


# The interpolation's texture gathers against plain loads, bit for bit: the same box with a mesh
# whose padded rows allow a texture (a multiple of 4 cells) is evaluated at order 2 through
# scola_pm_force and its forces are recomputed on the host from the returned potential with the
# kernel's formula in FP32 order (three products and sums a corner pair, within 4 roundings).
# Displacements reach every face and leave the box, so the uppermost corner's plain-load form and
# the clamps are taken; 48 and 40 sites a side take the two block shapes, 50 a partial block.
@pytest.mark.parametrize("n,ng", [(48, 48), (40, 80), (50, 52), (24, 240)])
def test_texture_gathers_match_the_returned_potential(n, ng):
    import numpy as np
    import paper_2003_04925_gb300 as sc
    kw = dict(L=4.0 * n, Np=n, Ntiles=1, Nbuf=0, Ng=ng, nsteps=1, a_i=0.05, a_f=1.0)
    sim = sc.Scola(**kw)
    g = torch.Generator("cuda").manual_seed(n)
    sim.lpt_fields(torch.randn(n, n, n, generator=g, device="cuda"))
    sim.setup_boxes()
    s = 12.0 * torch.randn(3, n**3, generator=g, device="cuda")
    s[:, -8:] = 4.0 * n                                    # beyond the upper corner
    F, _, phi = sim.pm_force(s, 1.0, want_phi=True)
    off = int(sim.box_offsets()[1][0])
    S = ng + 4
    P = phi[off:off + S**3].cpu().numpy().astype(np.float64)
    dg = np.float64(np.float32(4.0 * n / ng))
    b = np.indices((n, n, n)).reshape(3, -1)
    inv = np.float32(1.0 / (4.0 * n / ng))
    q2u = np.float32(ng / n)
    u = (s.cpu().numpy().astype(np.float64) * np.float64(inv)
         + (b * np.float64(q2u) + np.float64(np.float32(0.5) * q2u - np.float32(0.5))).astype(np.float32)).astype(np.float32)
    u = np.clip(u, np.float32(-1.0), np.float32(ng))
    i0 = np.minimum(np.floor(u), ng - 1).astype(np.int64)
    f = (u - i0).astype(np.float64)
    ref = np.zeros((3, n**3))
    for e in np.ndindex(2, 2, 2):
        w = np.prod([f[a] if e[a] else 1.0 - f[a] for a in range(3)], axis=0)
        at = ((i0[0] + e[0] + 2) * S + i0[1] + e[1] + 2) * S + i0[2] + e[2] + 2
        for a, st in enumerate((S * S, S, 1)):
            ref[a] += w * (P[at + st] - P[at - st]) * 0.5 / dg
    # FP32 sums of eight differences of neighbouring potentials (a few roundings of the largest);
    # where u rounds to the other side of a cell face both forms interpolate the same piecewise
    # linear function, so the difference stays at that level
    err = np.abs(F.cpu().numpy() - ref).max()
    assert err <= 16 * 2.0**-24 * np.abs(P).max() / dg, (err, np.abs(P).max() / dg)
    sc.scola_device_status(sim.ctx)
    sim.close()
