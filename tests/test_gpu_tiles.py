"""The step's tile sizes change with the number of rows (64, 128 or 256 rows to
a CTA, and smaller tiles at the end of a large grid; FP8: 256 or 512 threads to
a block).  The tiling must not show in the results: bit for bit those of the
batched step, which cuts a scene into whole tiles, at sizes on both sides of
every edge."""
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


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _state_bytes(run):
    return [run.rows().tobytes()] + [x.tobytes() for x in run.state()]


# rows: waves of 5 CTAs an SM times the tile, on both sides of the edge, and a large ragged size
@pytest.mark.parametrize("waves,tile,extra", [(1, 64, 0), (1, 64, 1), (1, 256, 0), (1, 256, 1), (2, 256, -63)])
@pytest.mark.parametrize("prec", ["FP32", "BF16", "BF16_HYBRID", "FP16_BLOCK"])
def test_tiling_does_not_change_the_step(G, prec, waves, tile, extra):
    n = 5 * _sms() * waves * tile + extra
    groups = synth.scene_blobs(n, 77, 12.5)
    grads = synth.grads_rows(n, 78)
    one, cut, terms = (GpuScene(groups, prec=getattr(G, "GS_MOM_" + prec)) for _ in range(3))
    for r in (one, cut, terms):
        r.set_grads(grads)
    cams = synth.ring_cameras(10, (0.0,))
    batch = G.gs_batch_create([cut.h])
    nvis = torch.zeros(1, dtype=torch.int64, device="cuda")
    active = torch.zeros(1, dtype=torch.int64, device="cuda")
    for k in range(1, 4):
        kw = dict(restate=(k == 2), restate_ratio=0.3, seed=5)
        p = G.make_params(synth.lr_for_step(k, 10), k, **kw)
        one.step_camera(cams[k], p)
        nvis.zero_()
        batch.set(0, G.make_attrs(cut.attrs), G.make_attrs(cut.grads), G.make_camera(cams[k]), p)
        G.gs_batch_step(batch, nvis)
        assert int(nvis.item()) == int(one.nvis.item()) == int(one.mask.sum().item())
        active.zero_()
        terms.step_camera(cams[k], G.make_params(synth.lr_for_step(k, 10), k, noise=2, noise_lr=0.0, n_active=active,
                                                 **kw))
        op = terms.attrs["opacity"]
        assert int(active.item()) == int((op > np.float32(-np.log(254.0))).sum().item())
    want = _state_bytes(one)
    assert _state_bytes(cut) == want
    assert _state_bytes(terms) == want
    batch.close()
    for r in (one, cut, terms):
        r.close()


@pytest.mark.parametrize("prec", ["FP32", "BF16", "BF16_HYBRID"])
def test_large_sparse_scene(G, prec):
    """From 1.5 Mi rows on (hybrid: 3 Mi), the sparse tiles of a step, and of its
    forms with the optional terms, read their gradients another way: same results."""
    n = (3 << (20 if prec == "BF16_HYBRID" else 19)) + 17
    groups = synth.scene_blobs(n, 81, 40.0)
    grads = synth.grads_rows(n, 82)
    one, cut, terms = (GpuScene(groups, prec=getattr(G, "GS_MOM_" + prec)) for _ in range(3))
    for r in (one, cut, terms):
        r.set_grads(grads)
    cam = synth.ring_cameras(10, (0.0,))[3]
    batch = G.gs_batch_create([cut.h])
    nvis = torch.zeros(1, dtype=torch.int64, device="cuda")
    active = torch.zeros(1, dtype=torch.int64, device="cuda")
    kw = dict(restate=True, restate_ratio=0.3, seed=5)
    p = G.make_params(synth.lr_for_step(1, 10), 1, **kw)
    one.step_camera(cam, p)
    batch.set(0, G.make_attrs(cut.attrs), G.make_attrs(cut.grads), G.make_camera(cam), p)
    G.gs_batch_step(batch, nvis)
    terms.step_camera(cam, G.make_params(synth.lr_for_step(1, 10), 1, n_active=active, **kw))
    assert 0 < int(nvis.item()) == int(one.nvis.item()) < n // 4
    assert int(active.item()) == int((terms.attrs["opacity"] > np.float32(-np.log(254.0))).sum().item())
    def same(r):
        assert all(torch.equal(r.attrs[k], one.attrs[k]) for k in one.attrs)
        assert all(a.tobytes() == b.tobytes() for a, b in zip(r.state(), one.state()))

    same(cut)
    same(terms)
    # the form with noise on every row, here of size zero
    one.step_camera(cam, G.make_params(synth.lr_for_step(2, 10), 2))
    terms.step_camera(cam, G.make_params(synth.lr_for_step(2, 10), 2, noise=2, noise_lr=0.0))
    same(terms)
    batch.close()
    for r in (one, cut, terms):
        r.close()


def test_fp8_block_width_does_not_change_the_step(G):
    """The same blocks in a scene small enough for 512 threads a block and in
    one with a block more, which takes 256."""
    n = 2 * _sms() * 256
    groups = synth.scene_blobs(n + 256, 79, 12.5)
    grads = synth.grads_rows(n + 256, 80)
    small = GpuScene({k: x[:n] for k, x in groups.items()}, prec=G.GS_MOM_FP8E4M3)
    large = GpuScene(groups, prec=G.GS_MOM_FP8E4M3)
    small.set_grads(grads[:n])
    large.set_grads(grads)
    cams = synth.ring_cameras(10, (0.0,))
    for k in range(1, 5):
        p = G.make_params(synth.lr_for_step(k, 10), k, restate=(k == 2), restate_ratio=0.3, seed=5)
        small.step_camera(cams[k], p)
        large.step_camera(cams[k], p)
    assert large.rows()[:n].tobytes() == small.rows().tobytes()
    for a, b in zip(small.state(), large.state()):
        assert a.tobytes() == b[:n].tobytes()
    small.close()
    large.close()
