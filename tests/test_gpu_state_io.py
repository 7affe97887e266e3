"""Export and import of the optimizer state at the edges of the 64-row tiles
(and of FP8's 256-row blocks), from and to arrays that are 16-B aligned and
ones that are 4-B aligned only, whole and in parts.  Every value must be
exactly the format's encoding of the imported one: no tolerance."""
import numpy as np
import pytest

from harness import GpuScene
from paper_2601_16736_gb300 import synth
from test_gpu_fp8 import _encode as _fp8
from test_gpu_mixed import _bf16, _f16b

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


def _hybrid(x):
    out = _bf16(x)
    out[:, :14] = x[:, :14]                       # FP32: all but the SH rest
    return out


ENCODE = {"FP32": (lambda x: x, lambda x: x), "BF16": (_bf16, _bf16), "BF16_HYBRID": (_hybrid, _hybrid),
          "FP16_BLOCK": (_f16b, lambda x: _f16b(x, second_moment=True)),
          "FP8E4M3": (_fp8, lambda x: _fp8(x, second_moment=True))}


def _values(n, seed):
    rng = np.random.default_rng(seed)
    m = (rng.normal(size=(n, 59)) * np.exp(rng.normal(0, 3, (n, 1)))).astype(np.float32)
    v = (rng.random((n, 59)) ** 4 * np.exp(rng.normal(0, 5, (n, 1)))).astype(np.float32)
    m[::7, 3] = 0.0
    v[n // 2:, 40] = 0.0
    return m, v, rng.integers(0, 60000, n).astype(np.int32)


def _device(x, offset):
    """x on the device, `offset` elements past an aligned address."""
    buf = torch.zeros(x.size + offset, dtype=torch.int32 if x.dtype == np.int32 else torch.float32, device="cuda")
    out = buf[offset:].view(x.shape)
    out.copy_(torch.from_numpy(x))
    return out


def _export(G, run, n, offset):
    m, v, t = _device(np.full((n, 59), 7.0, np.float32), offset), _device(np.full((n, 59), 7.0, np.float32), offset), \
        _device(np.full(n, 7, np.int32), offset)
    G.gs_opt_export_state(run.h, m, v, t)
    torch.cuda.synchronize()
    return m.cpu().numpy(), v.cpu().numpy(), t.cpu().numpy()


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("n", [1, 63, 64, 65, 255, 256, 257, 1345])
@pytest.mark.parametrize("prec", list(ENCODE))
def test_import_and_export_at_tile_edges(G, prec, n, offset):
    enc_m, enc_v = ENCODE[prec]
    run = GpuScene(synth.scene_uniform(n, 40), prec=getattr(G, "GS_MOM_" + prec))
    m, v, t = _values(n, 41 + n)
    G.gs_opt_import_state(run.h, _device(m, offset), _device(v, offset), _device(t, offset))
    got = _export(G, run, n, offset)
    want = [enc_m(m), enc_v(v), t]
    for g, w in zip(got, want):
        assert np.array_equal(g, w)
    # parts: the others keep what they held, and a part alone can be exported
    m2, v2, t2 = _values(n, 941 + n)
    for part, x in (("m", m2), ("v", v2), ("t", t2)):
        G.gs_opt_import_state(run.h, **{part: _device(x, offset)})
        want["mvt".index(part)] = enc_m(x) if part == "m" else enc_v(x) if part == "v" else x
        for g, w in zip(_export(G, run, n, offset), want):
            assert np.array_equal(g, w)
        alone = _device(np.full(x.shape, 7, x.dtype), offset)
        G.gs_opt_export_state(run.h, **{part: alone})
        torch.cuda.synchronize()
        assert np.array_equal(alone.cpu().numpy(), want["mvt".index(part)])
    run.close()
