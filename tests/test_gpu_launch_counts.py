"""The launch counters of a context against the kernels that the profiler records."""
import pytest

torch = pytest.importorskip("torch")

import paper_2003_04925_gb300 as sc  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def recorded(fn):
    """The profiler's events during fn."""
    from torch.profiler import ProfilerActivity, profile
    acts = [ProfilerActivity.CPU, ProfilerActivity.CUDA]
    with profile(activities=acts):                          # (the first session loses its first events)
        torch.zeros(8, device="cuda").sum().item()
    with profile(activities=acts) as pr:
        fn()
        torch.cuda.synchronize()
    return list(pr.events())


def _kernels(fn):
    names = [e.name for e in recorded(fn) if e.device_type == torch.autograd.DeviceType.CUDA]
    names = [n for n in names if not n.lower().startswith(("memcpy", "memset"))]    # (copies and fills)
    return sum("scola::" in n for n in names), len(names)


# Own kernels, and all of them, of a run (the second, whose initial conditions are captured as a
# graph, and the third) with each order of the initial conditions, and of a periodic run.  The dense
# FP32 form launches fewest: 8 boxes of 24^3, 11 evaluations, 97 own kernels with the sorted deposit.
@pytest.mark.parametrize("lpt_order,variant", [(2, "SIMT"), (1, "SIMT"), (2, "TC_3PASS")])
def test_launch_counts_of_a_run(lpt_order, variant):
    sim = sc.Scola(L=100.0, Np=32, Ntiles=2, Nbuf=4, mesh_ratio=1, nsteps=10, a_i=0.02, a_f=1.0, lpt_order=lpt_order,
                   dst_variant=getattr(sc, "SCOLA_DST_" + variant), deposit_form=sc.binding.SCOLA_DEPOSIT_SORTED)
    g = torch.Generator("cuda").manual_seed(1)
    w = torch.randn(32, 32, 32, generator=g, device="cuda")
    sim.forward(w)
    for _ in range(2):
        own, every = _kernels(lambda: sim.forward(w))
        st = sim.stats()
        assert (st["own_kernel_launches"], st["kernel_launches"]) == (own, every)
        assert every > own > 0
    if lpt_order == 2 and variant == "SIMT":
        assert own == 97
    sim.tcola(w)
    own, every = _kernels(lambda: sim.tcola(w))
    st = sim.stats()
    assert (st["own_kernel_launches"], st["kernel_launches"]) == (own, every)
    sim.close()
