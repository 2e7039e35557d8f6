"""Integer LayerNorm at the row counts and widths where its dispatch changes (rows per warp, words per lane, pieces of a short
row), with rows whose constants need the wide form (small standard deviation), constant rows and extremes.  Bit-exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2511_15369_b200 import api as _api
    _api.lib()
    return _api


def _rows(g, rows, dim):
    x = g.normal(0.0, 1.0, size=(rows, dim)) * g.choice([0.4, 2.0, 30.0], size=(rows, 1))
    x[0] = 7
    if rows > 5:
        x[1], x[2] = 0, -128
        x[3] = np.where(np.arange(dim) % 2, 127, -128)
        x[4] = 0
        x[4, 0] = 1
    return np.clip(np.round(x), -128, 127).astype(np.int8)


@pytest.mark.parametrize("variant", [0, 1, 2])
@pytest.mark.parametrize("rows,dim", [(1, 16), (63, 32), (64, 32), (65, 48), (1000, 64), (4737, 96), (77, 112), (4099, 128), (70, 132),
                                      (4736, 192), (4737, 256), (18945, 128 + 4), (18949, 192), (4739, 640), (18951, 768), (3, 1024), (4745, 1100),
                                      (18946, 1536), (37, 2048), (4741, 2052), (9, 3072)])
def test_rows_and_widths(api, orc, variant, rows, dim):
    import torch
    g = np.random.default_rng(rows * 7 + dim)
    x = _rows(g, rows, dim)
    gamma = g.normal(1.0, 0.2, dim).astype(np.float32)
    beta = g.normal(0.0, 0.2, dim).astype(np.float32)
    ptf = g.integers(0, 4, dim).astype(np.uint8) if variant == 2 else None
    for zp, out_bits in ((0, 8), (-11, 6)):
        gq, bq, c = orc.layernorm_prepare(gamma, beta, 8.0 / (1 << (out_bits - 1)), zp, out_bits, variant)
        gq2, bq2, ca = api.layernorm_prepare(gamma, beta, 8.0 / (1 << (out_bits - 1)), zp, out_bits, variant)
        cu = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()
        got = api.layernorm(cu(x), cu(gq2), cu(bq2), ca, cu(ptf)).cpu().numpy()
        want = orc.layernorm(x, gq, bq, c, ptf)
        bad = np.argwhere(got != want)
        assert bad.size == 0, (len(bad), bad[:3].tolist())
