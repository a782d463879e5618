"""Host calls of a context, as the profiler records them."""
import pytest

torch = pytest.importorskip("torch")

import paper_2003_04925_gb300 as sc  # noqa: E402
from test_gpu_launch_counts import recorded  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def _texture_calls(names):
    return {n for n in names if "TextureObject" in n or "DeviceProperties" in n}


# Textures serve scola_pm_force, which takes contexts of one batch: a streamed run whose batches
# differ in shape (every change rebinds the work lists) makes none.
def test_streamed_runs_make_no_textures():
    kw = dict(L=200.0, Np=64, Ntiles=2, Nbuf=0, buffers=[4, 8, 16, 4, 8, 4, 16, 8], mesh_ratio=1, nsteps=2, a_i=0.05,
              a_f=1.0)
    g = torch.Generator("cuda").manual_seed(1)
    w = torch.randn(64, 64, 64, generator=g, device="cuda")
    sims = []
    one = [e.name for e in recorded(lambda: sims.append(sc.Scola(**kw)))]
    if not any("CreateTextureObject" in k for k in one):
        pytest.skip("the profiler does not record the runtime's texture calls")
    sim = sc.Scola(batch_boxes=3, **kw)
    assert sim.stats()["batches"] > 1
    sim.forward(w)
    streamed = [e.name for e in recorded(lambda: sim.forward(w))]
    assert any("GraphLaunch" in k for k in streamed)
    assert not _texture_calls(streamed), _texture_calls(streamed)
    sim.close()
    sims[0].close()
