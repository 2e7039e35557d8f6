"""The one-launch-per-layer analysis (iptq_analyze_*) against the numpy oracle of the Unified Metric at the sizes where its
kernels can go wrong: rows shorter than a warp step, at and past a step's end, element counts that are no multiple of a
vector, the widest rows.  Tolerance as for iptq_metric_*: fp64 sums in another order and another exp / erf move them by
about 1e-13; 1e-9 relative leaves four orders of margin."""
import numpy as np
import pytest

from paper_2511_15369_b200 import synth

pytestmark = pytest.mark.gpu
REL = 1e-9


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from oracle import metric
    from paper_2511_15369_b200 import api, assign
    api.lib()
    return api, assign, metric


def _cu(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _same(cand, want):
    assert abs(cand.sum_x2 - want[0]) <= REL * abs(want[0]), (cand, want)
    assert abs(cand.sum_err2 - want[1]) <= REL * abs(want[1]), (cand, want)


@pytest.mark.parametrize("rows,n", [(1, 1), (3, 32), (9, 33), (70, 64), (11, 65), (300, 129), (591, 197), (40, 256), (17, 257), (5, 512), (9, 1000)])
def test_softmax_candidates(env, orc, rows, n):
    api, assign, metric = env
    S = synth.SOFTMAX_SCALE_ACC
    s = synth.quantize_scores(synth.softmax_logits(rows, n, seed=rows + n), S)
    an = assign.Analyzer()
    layer = an.softmax_layer("x", _cu(s), S)
    an.finish()
    X = metric.softmax_float(s, S)
    assert [c.variant for c in layer.candidates] == [0, 1, 2, 3]
    for c in layer.candidates:
        p = orc.softmax(s, orc.softmax_prepare(S, n, 4 if c.variant == orc.SM_LOG2 else 8, c.variant))
        _same(c, metric.error_sums(X, metric.log2_deq(p) if c.variant == orc.SM_LOG2 else metric.softmax_deq(p, 8)))
        assert c.op_count == api.op_count(api.LAYER_SOFTMAX, c.variant, rows, n)


@pytest.mark.parametrize("n", [1, 3, 4, 1023, 4097, 1 << 18])
def test_gelu_candidates(env, orc, n):
    api, assign, metric = env
    S = 2.5e-4
    xq = np.clip(np.round(synth.gelu_values(n, seed=n) / S), -32768, 32767).astype(np.int32)
    So, zp = 8.2 / 255, -123
    an = assign.Analyzer()
    layer = an.gelu_layer("x", _cu(xq), S, 16, So, zp)
    an.finish()
    assert [c.variant for c in layer.candidates] == [0, 1, 2]
    for c in layer.candidates:
        y = orc.gelu(xq, orc.gelu_prepare(S, 16, So, zp, 8, c.variant))
        _same(c, metric.error_sums(metric.gelu_float(xq, S), metric.affine_deq(y, So, zp)))


@pytest.mark.parametrize("n,constant", [((1 << 21) - 1, False), ((1 << 21) + 3, False), (10_000_003, False), (10_000_000, True)])
def test_gelu_counted_codes(env, orc, n, constant):
    """Layers large enough for the kernel that counts codes: every code of the range, a tail that fills no vector, more elements
    than a counter of one CTA can hold (it is emptied on the way), all of them on one code."""
    api, assign, metric = env
    S, So, zp = 2.5e-4, 8.2 / 255, -123
    xq = np.full(n, -77, np.int32) if constant else np.random.default_rng(n).integers(-32768, 32768, n).astype(np.int32)
    an = assign.Analyzer()
    layer = an.gelu_layer("x", _cu(xq), S, 16, So, zp)
    an.finish()
    codes, counts = np.unique(xq, return_counts=True)
    X = metric.gelu_float(codes, S)
    for c in layer.candidates:
        d = X - metric.affine_deq(orc.gelu(codes, orc.gelu_prepare(S, 16, So, zp, 8, c.variant)), So, zp)
        _same(c, (float((counts * X * X).sum()), float((counts * d * d).sum())))


@pytest.mark.parametrize("rows,dim", [(1, 4), (9, 100), (33, 128), (197, 192), (50, 768), (7, 3072)])
def test_layernorm_candidates(env, orc, rows, dim):
    api, assign, metric = env
    xf, gamma, beta, _ = synth.ln_values(rows, dim, seed=dim)
    x, _ = synth.quantize_sym(xf, 8, np.int8)
    if rows > 2:
        x[2] = 5                                               # a constant row
    ptf = (np.arange(dim) % 4).astype(np.uint8)
    So, zp = 8.0 / 127, 3
    an = assign.Analyzer()
    layer = an.layernorm_layer("x", _cu(x), gamma, beta, So, zp, ptf_shift=_cu(ptf))
    an.finish()
    assert [c.variant for c in layer.candidates] == [0, 1, 2]
    for c in layer.candidates:
        gq, bq, oc = orc.layernorm_prepare(gamma, beta, So, zp, 8, c.variant)
        sh = ptf if c.variant == orc.LN_PTF else None
        y = orc.layernorm(x, gq, bq, oc, sh)
        _same(c, metric.error_sums(metric.layernorm_float(x, gamma, beta, sh), metric.affine_deq(y, So, zp)))


def test_sums_are_the_same_bits_twice_and_the_capacity_is_kept(env):
    api, assign, metric = env
    S = synth.SOFTMAX_SCALE_ACC
    s = _cu(synth.quantize_scores(synth.softmax_logits(1000, 197, seed=1), S))
    an = assign.Analyzer(max_evaluations=8)
    for _ in range(2):
        an.softmax_layer("x", s, S)
    with pytest.raises(RuntimeError):
        an.softmax_layer("x", s, S)
    a, b = an.layers
    an.finish()
    assert [(c.sum_x2, c.sum_err2) for c in a.candidates] == [(c.sum_x2, c.sum_err2) for c in b.candidates]


@pytest.mark.parametrize("n", [1 << 18, (1 << 21) + 3])
def test_scratch_at_every_alignment_the_header_admits(env, n):
    """Scratch on a 16-byte boundary that is no 32-byte boundary: the terms of the codes are read 32 bytes at a time."""
    import ctypes as C

    import torch
    api, assign, metric = env
    x = _cu(np.random.default_rng(n).integers(-32768, 32768, n).astype(np.int32))
    consts = (api.GeluConsts * 2)(api.gelu_prepare(2.5e-4, 16, 8.2 / 255, -123), api.gelu_prepare(2.5e-4, 16, 8.2 / 255, -123, 8, 1))
    got = []
    for off in (0, 16):
        buf = torch.zeros(api.ANALYZE_WORK_BYTES + 64, dtype=torch.uint8, device="cuda")
        guard = off + api.ANALYZE_WORK_BYTES
        buf[:off] = 0xAB
        buf[guard:] = 0xAB
        sums = torch.zeros(4, dtype=torch.float64, device="cuda")
        assert buf.data_ptr() % 32 == 0
        assert api.lib().iptq_analyze_gelu(x.data_ptr(), n, 2.5e-4, 8.2 / 255, -123, C.cast(consts, C.c_void_p), 2, sums.data_ptr(),
                                           buf.data_ptr() + off, torch.cuda.current_stream().cuda_stream) == api.OK
        got.append(sums.cpu().numpy())
        assert (buf[:off] == 0xAB).all() and (buf[guard:] == 0xAB).all()
    assert (got[0] == got[1]).all() and (got[0] > 0).all()


@pytest.mark.parametrize("n", [9, 4097, (1 << 18) + 2, (1 << 21) + 1])
def test_codes_beyond_the_table(env, orc, n):
    """Inputs wider than 16 bits among the others, in vectors and in the tail, with and without a table of terms."""
    api, assign, metric = env
    S, So, zp = 2.5e-4, 8.2 / 255, -123
    x = np.random.default_rng(n).integers(-32768, 32768, n).astype(np.int32)
    x[::3] = np.tile([-32769, 32768, 1 << 20, -(1 << 22)], n)[:x[::3].size]
    x[-1] = 70000
    an = assign.Analyzer()
    layer = an.gelu_layer("x", _cu(x), S, 16, So, zp)
    an.finish()
    X = metric.gelu_float(x, S)
    for c in layer.candidates:
        _same(c, metric.error_sums(X, metric.affine_deq(orc.gelu(x, orc.gelu_prepare(S, 16, So, zp, 8, c.variant)), So, zp)))


@pytest.mark.parametrize("dim", [1028, 1536, 1540, 3072])
def test_wide_layernorms_can_be_recorded(env, dim):
    """A layer too wide for the launch's parameters, recorded into a graph and replayed after the caller's host arrays have changed."""
    import torch
    api, assign, metric = env
    xf, gamma, beta, _ = synth.ln_values(20, dim, seed=dim)
    x = _cu(synth.quantize_sym(xf, 8, np.int8)[0])
    plain = assign.Analyzer()
    plain.layernorm_layer("x", x, gamma, beta, 8.0 / 127, 3)
    want = plain.finish()[0][0].candidates
    an = assign.Analyzer()
    graph, g, b = torch.cuda.CUDAGraph(), gamma.copy(), beta.copy()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        an.layernorm_layer("x", x, g, b, 8.0 / 127, 3)
    g[:], b[:] = np.nan, np.nan
    for _ in range(2):
        graph.replay()
    got = an.finish()[0][0].candidates
    assert [(c.sum_x2, c.sum_err2) for c in got] == [(c.sum_x2, c.sum_err2) for c in want]
