"""The atomic deposit's scratch counts are left at zero by the kernel that reads them: an
evaluation after one with other positions gives the bits of a context's first evaluation."""
import pytest

torch = pytest.importorskip("torch")

import paper_2003_04925_gb300 as sc  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


# rows of a multiple of 4 cells (pairs of counts a load) and not, a last thread with 1 to 3 cells
# (Ng odd: Ng^3 mod 4 is 1 or 3), and boxes of 192^3 cells, which are groups of their own
@pytest.mark.parametrize("ntiles,nbuf,ng", [(2, 1, 11), (2, 1, 13), (2, 1, 16), (2, 1, 18), (2, 1, 192), (1, 0, 191)])
def test_scratch_counts_are_cleared(ntiles, nbuf, ng):
    kw = dict(L=64.0, Np=16, Ntiles=ntiles, Nbuf=nbuf, Ng=ng, nsteps=1, a_i=0.05, a_f=1.0,
              deposit_form=sc.binding.SCOLA_DEPOSIT_ATOMIC)
    g = torch.Generator("cuda").manual_seed(ng)
    w = torch.randn(16, 16, 16, generator=g, device="cuda")
    out = []
    for warm in (False, True):
        sim = sc.Scola(**kw)
        sim.lpt_fields(w)
        sim.setup_boxes()
        gs = torch.Generator("cuda").manual_seed(1)
        s = 3.0 * torch.randn(3, sim.P, generator=gs, device="cuda")
        if warm:
            sim.pm_force(20.0 * torch.randn(3, sim.P, generator=gs, device="cuda"), 1.0)
        F, delta, _ = sim.pm_force(s, 1.0, want_delta=True)
        cells = torch.cat([delta[o:o + ng**3] for o in sim.box_offsets()[0]])     # (not the gaps between boxes)
        out.append((F.clone(), cells.clone()))
        sim.close()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
