"""The force interpolation of boxes whose lattice leaves idle lanes in its blocks of sites (sides that
are not a multiple of the block's and still fill eight ninths of it), with texture gathers (padded rows
of a multiple of 4 cells) and without."""
import pytest

torch = pytest.importorskip("torch")

from test_gpu_elimination import test_texture_gathers_match_the_returned_potential as _check  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def _blocks(n):
    """Extents of a block of 256 sites and the sites it would cover, or None where runs are taken."""
    bz = 16 if n % 16 == 0 else 8
    ext = (4, 64 // bz, bz)
    cover = 256
    for e in ext:
        cover *= -(-n // e)
    return ext if 8 * cover <= 9 * n**3 else None


# against the formula in 64 bits on the returned potential, within 16 roundings of its largest value
# over the cell size, as for the sides that fill their blocks
@pytest.mark.parametrize("n,ng", [(31, 32), (47, 48), (55, 56), (63, 64), (47, 47), (63, 66)])
def test_partial_blocks_match_the_returned_potential(n, ng):
    ext = _blocks(n)
    assert ext is not None and any(n % e for e in ext)
    _check(n, ng)
