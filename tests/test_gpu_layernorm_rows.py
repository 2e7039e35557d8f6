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


# the remaining kernels of the dispatch: one to four rows per warp at 52 .. 112, 384, 512, 1024 and 2048 channels, rows that fill their
# words exactly and rows that do not
@pytest.mark.parametrize("variant", [0, 1, 2])
@pytest.mark.parametrize("rows,dim", [(4740, 52), (18947, 80), (18946, 112), (4743, 384), (18945, 384), (18950, 260), (4738, 512), (18947, 512),
                                      (18946, 388), (4737, 1024), (18945, 1024), (18946, 900), (4738, 2048), (4737, 1540)])
def test_the_remaining_rows_per_warp(api, orc, variant, rows, dim):
    test_rows_and_widths(api, orc, variant, rows, dim)


def _general(api, orc, g, dim, variant):
    """Parameters whose zero point does not fit into the rounding constant (outputs coarser than gamma); beta as large as its 32 bits allow."""
    gamma = g.normal(0.2, 0.02, dim).astype(np.float32)
    top = float(np.abs(gamma).max())
    beta = (g.uniform(-1, 1, dim) * top * min(30.0, 0.9 * (64 - 1.125 * np.sqrt(dim)))).astype(np.float32)
    for zp, out_scale in ((100, 2.05 * top), (-100, 3 * top), (-128, 9 * top), (0, 200 * top)):
        gq, bq, c = orc.layernorm_prepare(gamma, beta, out_scale, zp, 8, variant)
        _, _, ca = api.layernorm_prepare(gamma, beta, out_scale, zp, 8, variant)
        assert abs((1 << (ca.out.shift - 1)) + (zp << ca.out.shift)) >= 1 << 30
        yield gq, bq, c, ca


@pytest.mark.parametrize("variant", [0, 1, 2])
@pytest.mark.parametrize("rows,dim", [(1, 4), (70, 96), (333, 128), (65, 200), (9, 3072)])
def test_zero_points_beyond_the_rounding_constant(api, orc, variant, rows, dim):
    import torch
    g = np.random.default_rng(rows + dim)
    x = _rows(g, rows, dim)
    ptf = g.integers(0, 4, dim).astype(np.uint8) if variant == 2 else None
    cu = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()
    kinds = 0
    for gq, bq, c, ca in _general(api, orc, g, dim, variant):
        want = orc.layernorm(x, gq, bq, c, ptf)
        kinds = max(kinds, len(np.unique(want)))
        assert (api.layernorm(cu(x), cu(gq), cu(bq), ca, cu(ptf)).cpu().numpy() == want).all()
    assert kinds > (20 if dim in (96, 128, 200) else 3)


@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("variant", [1, 2])
@pytest.mark.parametrize("rows,C,parts", [(70, 96, 1), (5, 64, 1), (301, 48, 4), (4740, 96, 4), (19000, 24, 3), (90, 768, 4)])
def test_gathered_rows_of_every_kind(api, orc, general, variant, rows, C, parts):
    """Gathered LayerNorm with power-of-two factors, a zero point, and a zero point beyond the rounding constant."""
    import torch
    g = np.random.default_rng(rows + C)
    x = _rows(g, 500, C)
    idx = g.integers(-1, 500, size=(rows, parts)).astype(np.int32)
    dim = C * parts
    src = np.ascontiguousarray(np.where((idx >= 0)[:, :, None], x[np.maximum(idx, 0)], 0).reshape(rows, dim).astype(np.int8))
    ptf = g.integers(0, 4, dim).astype(np.uint8) if variant == 2 else None
    if general:
        gq, bq, c, ca = next(_general(api, orc, g, dim, variant))
    else:
        gamma, beta = g.normal(1.0, 0.2, dim).astype(np.float32), g.normal(0.0, 0.2, dim).astype(np.float32)
        gq, bq, c = orc.layernorm_prepare(gamma, beta, 8 / 127, -9, 8, variant)
        _, _, ca = api.layernorm_prepare(gamma, beta, 8 / 127, -9, 8, variant)
    cu = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()
    got = api.layernorm_gather(cu(x), cu(idx), cu(gq), cu(bq), ca, cu(ptf)).cpu().numpy()
    assert (got == orc.layernorm(src, gq, bq, c, ptf)).all()
