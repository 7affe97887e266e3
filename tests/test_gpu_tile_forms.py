"""The forms of the step (plain; count and noise on visible rows; noise on every
row with AIU) at sizes in every part of the tiling rule: tiles of 64 and 128
rows, one wave of tiles of 144 to 256 rows, whole tiles with 128-row ones at the
end, and the kernels of large scenes.  Rows against the oracle, counts and step counters exactly; the plain
step bit for bit that of the batched one, which cuts whole tiles."""
import numpy as np
import pytest

from harness import GpuScene, assert_close
from paper_2601_16736_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

# CTAs of the kernels with optional terms resident on an SM (plain step: 5)
TERMS_CTAS = {"FP32": 5, "BF16": 5, "BF16_HYBRID": 4, "FP16_BLOCK": 4}


@pytest.fixture(scope="module")
def G():
    from paper_2601_16736_gb300 import build
    build.build()
    from paper_2601_16736_gb300 import gsopt
    return gsopt


def _wave(ctas):
    return ctas * torch.cuda.get_device_properties(0).multi_processor_count


# rows a resident CTA has, in tenths, and extra rows
@pytest.mark.parametrize("tenths,extra", [(1280, 0), (1280, 1), (1600, 0), (1600, 17), (2400, 1), (2560, -15)])
@pytest.mark.parametrize("prec", list(TERMS_CTAS))
def test_plain_step_in_one_wave(G, prec, tenths, extra):
    n = _wave(5) * tenths // 10 + extra
    groups = synth.scene_blobs(n, 1201, 12.5)
    grads = synth.grads_rows(n, 1202)
    one, cut = (GpuScene(groups, prec=getattr(G, "GS_MOM_" + prec)) for _ in range(2))
    for r in (one, cut):
        r.set_grads(grads)
    cams = synth.ring_cameras(10, (0.0,))
    batch = G.gs_batch_create([cut.h])
    nvis = torch.zeros(1, dtype=torch.int64, device="cuda")
    for k in (1, 2):
        p = G.make_params(synth.lr_for_step(k, 10), k, restate=(k == 2), restate_ratio=0.3, seed=5)
        one.step_camera(cams[k], p)
        nvis.zero_()
        batch.set(0, G.make_attrs(cut.attrs), G.make_attrs(cut.grads), G.make_camera(cams[k]), p)
        G.gs_batch_step(batch, nvis)
        assert int(nvis.item()) == int(one.nvis.item()) == int(one.mask.sum().item())
    assert one.rows().tobytes() == cut.rows().tobytes()
    for a, b in zip(one.state(), cut.state()):
        assert a.tobytes() == b.tobytes()
    batch.close()
    one.close()
    cut.close()


def _check(G, orc, prec, n, form, density, steps):
    """Noise far above the rounding, so that a row with another row's noise shows."""
    groups = synth.scene_uniform(n, 1211)
    rng = np.random.default_rng(1212)
    groups["scale"] = rng.normal(-1.2, 0.3, (n, 3)).astype(np.float32)
    groups["opacity"][::3] = rng.normal(-5.537, 0.05, (len(groups["opacity"][::3]), 1))     # near -ln 254
    run = GpuScene(groups, prec=getattr(G, "GS_MOM_" + prec))
    st = orc.State(synth.to_rows(groups))
    cfg = orc.Config(n_i=orc.dar_normaliser(800 * 800))
    g = synth.grads_rows(n, 1213)
    active = torch.zeros(1, dtype=torch.int64, device="cuda")
    for k in range(1, steps + 1):
        mask = (rng.random(n) < density).astype(np.uint8)
        gk = np.roll(g, 7 * k, axis=0)
        lr = synth.lr_for_step(k, steps)
        aiu = form == "all" and k > 1
        ext = orc.Ext(noise_mode=1 if form == "visible" else 2, aiu=aiu, noise_lr=400.0, noise_k=3.0, noise_t=0.5,
                      aiu_prob=0.35, aiu_scale=0.5, seed=79)
        run.set_grads(gk)
        active.zero_()
        run.step_mask(torch.from_numpy(mask).cuda(),
                      G.make_params(lr, k, restate=(k == 2), restate_ratio=0.3, seed=79, n_active=active,
                                    noise=ext.noise_mode, noise_lr=400.0, noise_k=3.0, noise_t=0.5, aiu=aiu,
                                    aiu_prob=0.35, aiu_scale=0.5))
        orc.step_ext(cfg, st, gk, mask, lr, True, True, k, ext)
        if k == 2:
            orc.restate(cfg, st, 79, k, 0.3)
        assert int(active.item()) == orc.active_rows(run.attrs["opacity"].cpu().numpy().ravel()).size
    got = run.rows()
    assert np.abs(got[:, 0:3] - synth.to_rows(groups)[:, 0:3]).max() > 1e-3
    assert_close(got, st.theta, 1e-5 if prec == "FP32" else 2e-3, what=f"{form}, {n} rows")
    assert np.array_equal(run.state()[2], st.t)
    run.close()


@pytest.mark.parametrize("density", [0.15, 0.9])
@pytest.mark.parametrize("form", ["visible", "all"])
@pytest.mark.parametrize("tenths,extra", [(640, 1), (1280, 1), (2400, 1), (2560, 0), (2560, 65), (5120, 300)])
@pytest.mark.parametrize("prec", ["FP32", "BF16_HYBRID", "FP16_BLOCK"])
def test_terms_at_every_tiling(G, orc, prec, tenths, extra, form, density):
    """FP32 tiles of more and of fewer than two groups of 64 visible rows."""
    _check(G, orc, prec, _wave(TERMS_CTAS[prec]) * tenths // 10 + extra, form, density, 3)


@pytest.mark.parametrize("prec,n,form", [("FP32", (3 << 19) + 17, "visible"), ("FP32", (3 << 19) + 17, "all"),
                                         ("BF16_HYBRID", (3 << 20) + 17, "all")])
def test_terms_in_a_large_sparse_scene(G, orc, prec, n, form):
    """Sparse tiles that read their gradients as ordinary lines, with noise and AIU."""
    _check(G, orc, prec, n, form, 0.15, 2)
