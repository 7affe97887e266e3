"""gs_gather_attrs at the edges of its 128-row tiles, with and without rows that
keep what they held, and with the small groups (xyz, scale, opacity) 16-B aligned
or 4-B aligned only, on either side.  Copies: no tolerance."""
import numpy as np
import pytest

from harness import GpuScene
from paper_2601_16736_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)


@pytest.fixture(scope="module")
def G():
    from paper_2601_16736_gb300 import build
    build.build()
    from paper_2601_16736_gb300 import gsopt
    return gsopt


def _at(x, offset):
    """x on the device; the small groups `offset` floats past an aligned address."""
    off = offset if x.shape[1] in (1, 3) else 0
    out = torch.zeros(x.size + off, device="cuda")[off:].view(x.shape)
    out.copy_(torch.from_numpy(x))
    return out


@pytest.mark.parametrize("holes", [False, True])
@pytest.mark.parametrize("off_in,off_out", [(0, 0), (1, 0), (0, 1), (3, 2)])
@pytest.mark.parametrize("n_new", [1, 127, 128, 129, 257, 1023])
def test_gather_at_tile_edges(G, n_new, off_in, off_out, holes):
    n = 1009
    groups = synth.scene_uniform(n, 1301)
    run = GpuScene(groups)
    src = np.random.default_rng(1302 + n_new).integers(0, n, n_new).astype(np.int32)
    src[-1] = n - 1
    if holes:
        src[::5] = -1
        src[:min(n_new, 129)][-1] = -1             # the only one of a tile, or its last
    held = {k: np.full((n_new, x.shape[1]), -7.5, np.float32) for k, x in groups.items()}
    attrs = {k: _at(x, off_in) for k, x in groups.items()}
    out = {k: _at(x, off_out) for k, x in held.items()}
    G.gs_gather_attrs(run.h, G.make_attrs(attrs), n, G.make_attrs(out), torch.from_numpy(src).cuda(), n_new)
    torch.cuda.synchronize()
    for k, x in groups.items():
        want = np.where((src >= 0)[:, None], x[np.maximum(src, 0)], held[k])
        assert np.array_equal(out[k].cpu().numpy(), want)
    assert G.gs_opt_sync_errors(run.h) == G.GS_OK
    run.close()
