"""FP8 moments in a scene of more than one wave of blocks (4 CTAs of 256 rows to
an SM): every block on its full pass in some step, blocks in the CTAs beyond the
first wave among them, and the step followed at once by a launch that reads the
state.  What a block becomes depends on its rows, its number and the iteration
alone, so the first blocks are bit for bit those of a scene of one wave; all of
them follow the FP32 path in the first step."""
import numpy as np
import pytest

from harness import GpuScene
from paper_2601_16736_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

LR = synth.lr_for_step(1, 10)
BLOCK = 256


@pytest.fixture(scope="module")
def G():
    from paper_2601_16736_gb300 import build
    build.build()
    from paper_2601_16736_gb300 import gsopt
    return gsopt


def _wave():
    return 4 * torch.cuda.get_device_properties(0).multi_processor_count


def _iterations(tiles):
    """The first step; one with the last block on its full pass; one with an StSS
    event; one with block 0 on its full pass (iteration + block a multiple of 128)."""
    return 1, 128 - (tiles - 1) % 128, 77, 128


@pytest.mark.parametrize("extra", [1, BLOCK + 1])
def test_blocks_beyond_one_wave(G, extra):
    n0 = _wave() * BLOCK
    n = n0 + extra
    groups = synth.scene_blobs(n, 1101, 12.5)
    grads = synth.grads_rows(n, 1102)
    one = GpuScene({k: x[:n0] for k, x in groups.items()}, prec=G.GS_MOM_FP8E4M3)
    large = GpuScene(groups, prec=G.GS_MOM_FP8E4M3)
    fp32 = GpuScene(groups)
    one.set_grads(grads[:n0])
    for r in (large, fp32):
        r.set_grads(grads)
    cams = synth.ring_cameras(10, (0.0,))
    t_want = np.zeros(n, np.uint32)
    src = np.arange(n, dtype=np.int32)
    src[:n0] ^= 1                                # neighbours change places: the same rows in every block
    src = torch.from_numpy(src).cuda()
    for i, k in enumerate(_iterations((n + BLOCK - 1) // BLOCK)):
        p = G.make_params(LR, k, restate=(k == 77), restate_ratio=0.3, seed=5)
        one.step_camera(cams[i], p)
        large.step_camera(cams[i], p)
        if i == 0:
            fp32.step_camera(cams[i], p)
            assert large.rows().tobytes() == fp32.rows().tobytes()
            assert torch.equal(large.mask, fp32.mask)
            _, _, t = fp32.state()
            assert np.array_equal(large.state()[2], t)
        G.gs_reindex_state(one.h, src[:n0], None, n0)
        G.gs_reindex_state(large.h, src, None, n)
        assert torch.equal(large.mask[:n0], one.mask)
        assert int(large.nvis.item()) == int(large.mask.sum().item())
        t_want = (t_want + large.mask.cpu().numpy())[src.cpu().numpy()]
        state = large.state()
        assert np.array_equal(state[2], t_want)
        for a, b in zip(one.state(), state):
            assert a.tobytes() == b[:n0].tobytes()
        assert large.rows()[:n0].tobytes() == one.rows().tobytes()
    for r in (one, large, fp32):
        r.close()


def test_captured_steps_beyond_one_wave(G):
    n = _wave() * BLOCK + BLOCK + 1
    groups = synth.scene_blobs(n, 1103, 12.5)
    grads = synth.grads_rows(n, 1104)
    cams = synth.ring_cameras(10, (0.0,))
    steps = [(cams[i], G.make_params(LR, k)) for i, k in enumerate(_iterations((n + BLOCK - 1) // BLOCK))]
    got = []
    for captured in (False, True):
        r = GpuScene(groups, prec=G.GS_MOM_FP8E4M3)
        r.set_grads(grads)
        torch.cuda.synchronize()

        def iterate():
            for cam, p in steps:
                r.step_camera(cam, p)

        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                iterate()
            iterate = g.replay
        for _ in range(2):
            iterate()
        got.append([r.rows().tobytes(), r.mask.cpu().numpy().tobytes(), int(r.nvis.item())] +
                   [x.tobytes() for x in r.state()])
        r.close()
    assert got[0] == got[1]
