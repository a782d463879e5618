"""The full-box stages (initial conditions, periodic tCOLA) run launch by launch on a context's
first call and as a graph from the second on: every call gives the first call's bits, for each
call's own noise and output buffers, on the default stream and on another one."""
import pytest

torch = pytest.importorskip("torch")

import paper_2003_04925_gb300 as sc  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

KW = dict(L=64.0, Np=16, Ntiles=2, Nbuf=4, mesh_ratio=1, nsteps=2, a_i=0.05, a_f=1.0)


def _calls(sim, w):
    f = sim.lpt_fields(w)
    x, p = sim.tcola(w)
    xf, pf = sim.forward(w)
    torch.cuda.synchronize()
    return [f["delta"], f["phi1"], f["phi2"], f["psi1"], f["psi2"], x, p, xf, pf]


@pytest.mark.parametrize("lpt_order", [1, 2])
@pytest.mark.parametrize("own_stream", [False, True])
def test_replayed_stages_repeat_the_first_call(lpt_order, own_stream):
    g = torch.Generator("cuda").manual_seed(4)
    noise = [torch.randn(16, 16, 16, generator=g, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    first = []
    for w in noise:                                      # one context per noise: its first calls
        sim = sc.Scola(lpt_order=lpt_order, **KW)
        first.append(_calls(sim, w))
        sim.close()
    sim = sc.Scola(lpt_order=lpt_order, stream=torch.cuda.Stream() if own_stream else None, **KW)
    for k in (0, 1, 0, 1, 1):                            # first, captured, replayed
        kept = noise[k].clone()
        for got, want in zip(_calls(sim, noise[k]), first[k]):
            assert torch.equal(got, want)
        assert torch.equal(noise[k], kept)               # the caller's noise stays as it was
    sim.close()
