"""The deposit autotuner times its candidates at the mean growth of a run's force evaluations, also
where a run has two of them."""
import pytest

torch = pytest.importorskip("torch")

import paper_2003_04925_gb300 as sc  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


# The atomic form slows down steadily with the displacements: on these boxes 0.76 ms on the initial
# lattice, 1.03 half way and 1.28 at a = 1.  A run of one step from a = 0.02 to 1 is tuned
# between two runs that stay at either end (by more than the few per cent that timings differ).
def test_two_evaluations_are_tuned_half_way():
    def atomic_ms(a_i, a_f):
        sim = sc.Scola(L=500.0, Np=256, Ntiles=4, Nbuf=8, mesh_ratio=1, nsteps=1, a_i=a_i, a_f=a_f)
        g = torch.Generator("cuda").manual_seed(2)
        sim.lpt_fields(torch.randn(256, 256, 256, generator=g, device="cuda"))
        sim.setup_boxes()
        ms = sim.stats()["ms_deposit_candidates"][4]
        sim.close()
        return ms

    early, run, late = atomic_ms(0.02, 0.021), atomic_ms(0.02, 1.0), atomic_ms(0.99, 1.0)
    print("atomic deposit, tuned early / one step / late: %.3f / %.3f / %.3f ms" % (early, run, late))
    assert 1.08 * early < run < late / 1.08
