"""The atomic deposit's scratch is cleared by the kernel that reads it in small groups of boxes and by
a memset in large ones: the same bits on both sides of that line, and a clearing that is cheap next to
the deposit itself."""
import pytest

torch = pytest.importorskip("torch")

import paper_2003_04925_gb300 as sc  # noqa: E402
from test_gpu_launch_counts import recorded  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


# 8 boxes of 40^3 cells are 512,000 counts (of 524,288), of 41^3 and 42^3 551,368 and 592,704
@pytest.mark.parametrize("ng", [40, 41, 42])
def test_evaluations_repeat_bit_for_bit(ng):
    sim = sc.Scola(L=64.0, Np=16, Ntiles=2, Nbuf=1, Ng=ng, nsteps=1, a_i=0.05, a_f=1.0,
                   deposit_form=sc.binding.SCOLA_DEPOSIT_ATOMIC)
    g = torch.Generator("cuda").manual_seed(ng)
    sim.lpt_fields(torch.randn(16, 16, 16, generator=g, device="cuda"))
    sim.setup_boxes()
    s = 3.0 * torch.randn(3, sim.P, generator=g, device="cuda")
    first = sim.pm_force(s, 1.0)[0].clone()
    sim.pm_force(20.0 * torch.randn(3, sim.P, generator=g, device="cuda"), 1.0)
    assert torch.equal(first, sim.pm_force(s, 1.0)[0])
    sim.close()


# 64 boxes of 64^3 cells, one per particle: the source kernel and the clearing stream 28 bytes a cell
# and take a fifth of the deposit's eight scattered weights a particle; twice that is a fault
def test_clearing_is_cheap_next_to_the_deposit():
    sim = sc.Scola(L=300.0, Np=192, Ntiles=4, Nbuf=8, mesh_ratio=1, nsteps=1, a_i=0.02, a_f=1.0,
                   deposit_form=sc.binding.SCOLA_DEPOSIT_ATOMIC)
    g = torch.Generator("cuda").manual_seed(1)
    sim.lpt_fields(torch.randn(192, 192, 192, generator=g, device="cuda"))
    sim.setup_boxes()
    s = 2.0 * torch.randn(3, sim.P, generator=g, device="cuda")
    sim.pm_force(s, 1.0)
    ev = recorded(lambda: [sim.pm_force(s, 1.0) for _ in range(5)])
    us = {"k_deposit(": 0.0, "k_density_source": 0.0, "memset": 0.0}
    for e in ev:
        if e.device_type == torch.autograd.DeviceType.CUDA:
            for k in us:
                if k in e.name or (k == "memset" and k in e.name.lower()):
                    us[k] += e.device_time_total / 5
    print("deposit %.0f us, source %.0f us, memset %.0f us" % tuple(us.values()))
    assert 0.0 < us["k_density_source"] + us["memset"] < 0.3 * us["k_deposit("]
    sim.close()
