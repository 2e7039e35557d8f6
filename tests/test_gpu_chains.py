"""Chains of dependent launches, run back to back many times: every launch may start while the one before it is still running,
and each of these chains writes buffers that an earlier pass of it has read.  The last outputs have to be the first ones."""
import numpy as np
import pytest

from paper_2511_15369_b200 import synth

pytestmark = pytest.mark.gpu
PASSES = 20


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2511_15369_b200 import api as _api
    _api.lib()
    return _api


def _cu(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def test_gathers_and_patches_of_a_buffer_that_every_pass_rewrites(api):
    """The readers of int8 activations that do not go through the copy engine, right behind the launch that writes them."""
    import torch
    g = np.random.default_rng(5)
    src = [_cu(g.integers(-128, 128, size=(3136, 96)).astype(np.int8)) for _ in range(2)]
    perm = _cu(g.permutation(3136).astype(np.int32).reshape(-1, 1))
    four = _cu(g.integers(-1, 3136, size=(784, 4)).astype(np.int32))
    gq, bq, c = api.layernorm_prepare(g.normal(1, 0.1, 384), g.normal(0, 0.1, 384), 8 / 127)
    gq, bq = _cu(gq), _cu(bq)
    buf, rows = torch.empty_like(src[0]), torch.empty((784, 384), dtype=torch.int8, device="cuda")

    def one(x):
        api.gather_rows(x, perm, out=buf)
        n = api.layernorm_gather(buf, four, gq, bq, c)
        api.gather_rows(buf, four, out=rows)
        return n, api.layernorm(rows, gq, bq, c), api.patchify(buf.view(1, 3, 224, 448))
    want = []
    for x in src:
        want.append(one(x))
        torch.cuda.synchronize()
    for i in range(PASSES):
        got = [one(x) for x in src]
    torch.cuda.synchronize()
    for a, b in zip(want, got):
        assert torch.equal(a[0], a[1])
        assert all(torch.equal(p, q) for p, q in zip(a, b))
    assert not torch.equal(want[0][0], want[1][0])


def _passes(api, run, check):
    """run() PASSES times eagerly and PASSES times as a recorded graph; every pass's launches follow the last one's at once."""
    import torch
    first = run().clone()
    torch.cuda.synchronize()
    check()
    for _ in range(PASSES):
        last = run()
    torch.cuda.synchronize()
    assert torch.equal(first, last)
    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=side):
        out = run()
    for _ in range(PASSES):
        graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(first, out)
    check()
    assert len(torch.unique(first)) > 30


@pytest.mark.parametrize("table", [(0, 0, 0, 0), (3, 1, 2, 1)])
@pytest.mark.parametrize("shape", [synth.BlockShape("DeiT-T b1", 1, 197, 192, 3, 64, 768), synth.BlockShape("DeiT-S b64", 64, 197, 384, 6, 64, 1536),
                                   synth.BlockShape("50 tokens", 40, 50, 384, 6, 64, 1536)])
def test_encoder_blocks(api, shape, table):
    spec = synth.make_block(shape, seed=1, calib_images=1)
    blk, x = api.EncoderBlock(spec, table), _cu(spec.x)
    _passes(api, lambda: blk(x), blk.ws.check)


def test_a_small_backbone(api):
    from paper_2511_15369_b200 import swin
    spec = synth.make_swin(1, [dict(dim=96, heads=3, depth=2, grid=(20, 31)), dict(dim=192, heads=6, depth=2, grid=(10, 16)),
                               dict(dim=384, heads=12, depth=2, grid=(5, 8))], seed=3)
    net, x = swin.SwinBackbone(spec), _cu(spec.x)
    _passes(api, lambda: net(x), net.check)


def test_a_whole_model(api):
    from paper_2511_15369_b200 import vit
    spec = synth.make_vit("DeiT-T", 2, 1)
    model, image = vit.VitModel(spec), _cu(spec.image)
    _passes(api, lambda: model(image), model.check)


@pytest.mark.parametrize("table", [(0, 0, 0, 0), (3, 1, 2, 1)])
def test_fresh_states(api, table):
    """First passes of one block state after the other, each in memory of its own that goes back to the device in between: every first pass and
    every replay gives the same bytes, and nothing reaches for memory that is no longer there."""
    import gc

    import torch
    spec = synth.make_block(synth.BlockShape("DeiT-S b64", 64, 197, 384, 6, 64, 1536), seed=1, calib_images=1)
    rng, want = np.random.default_rng(0), None
    for n in range(60):
        pad = torch.empty(int(rng.integers(1, 40)) << 20, dtype=torch.uint8, device="cuda")
        blk, x = api.EncoderBlock(spec, table), _cu(spec.x)
        torch.cuda.synchronize()
        y = blk(x)
        torch.cuda.synchronize()
        got = y.cpu()
        want = got if want is None else want
        assert torch.equal(got, want), n
        if n % 3 == 0:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                out = blk(x)
            for _ in range(5):
                graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(out, y), n
            del graph, out
        del pad, blk, x, y
        gc.collect()
        torch.cuda.empty_cache()
