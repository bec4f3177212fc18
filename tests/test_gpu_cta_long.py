"""The compressor over streams of several blocks per CTA (slots swapped, the
next block loaded into the buffer in use, look-back by the idle warp) and on
both sides of the rule that gives a shortened last block its own launch,
against the general compressor byte for byte, index included."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# (element size, block elements): one to sixteen warps, the fixed block sizes and
# others, whose streams never take two launches
SHAPES = [(1, 2048), (1, 8192), (1, 12288), (2, 1024), (2, 4096), (4, 256), (4, 512), (4, 1024),
          (4, 2048), (4, 3072), (4, 4096), (4, 16384), (8, 256), (8, 512), (8, 1024), (8, 4096),
          (8, 8192)]


def _same(bsgpu, d, es, B, level):
    c = bsgpu.compress(d, B, es, level=level)
    assert bsgpu.status(c.ws) == 0
    out, nb, offs = bsgpu.compress_noalloc(d, B, elem_size=es, offsets=torch.zeros_like(c.offsets),
                                           level=level)
    torch.cuda.synchronize()
    assert c.nbytes == int(nb.item())
    assert torch.equal(c.buf[:c.nbytes], out[:c.nbytes]) and torch.equal(c.offsets, offs)


@pytest.mark.parametrize("level", [0, 1])
@pytest.mark.parametrize("es,B", SHAPES)
def test_several_blocks_per_cta(es, B, level):
    from paper_1503_00638_gb300 import bsgpu, synth
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    per = min(32, 228 * 1024 // (B * es + 1024))            # at least the CTAs an SM can hold
    n = 3 * sms * per * B + B // 2 // 8 * 8 + 3
    _same(bsgpu, synth.random_walk_device(n, es, seed=B + es), es, B, level)


@pytest.mark.parametrize("es,B", [(1, 8192), (2, 2048), (4, 512), (4, 2048), (4, 4096), (8, 1024), (8, 4096)])
@pytest.mark.parametrize("blocks", [-1, 0])
def test_shortened_last_block_around_the_two_launch_rule(es, B, blocks):
    from paper_1503_00638_gb300 import bsgpu, synth
    full = ((64 if B * es <= 8192 else 128) << 20) // (B * es) + blocks
    _same(bsgpu, synth.random_walk_device(full * B + 8, es, seed=es), es, B, 0)


@pytest.mark.parametrize("tslow", [False, True])
@pytest.mark.parametrize("es,B", [(4, 2048), (4, 1024), (8, 1024), (8, 512)])
def test_cube_of_several_blocks_per_cta_with_a_shortened_last_block(es, B, tslow):
    from paper_1503_00638_gb300 import bsgpu, synth
    cfg = synth.VisConfig(151, 64, 29, 2 ** 16, 0.01, seed=3)      # 73 MB: two launches
    v = synth.visibilities_torch(cfg)
    src = v.permute(2, 0, 1).contiguous() if tslow else v
    c = bsgpu.compress_vis_ex(src, cfg.n_samp, cfg.f, elem_size=es, block_elems=B, time_slowest=tslow)
    assert bsgpu.status(c.ws) == 0 and c.n_elem % B != 0
    bits = torch.view_as_real(bsgpu.reduce_precision(v, cfg.n_samp, cfg.f)).contiguous()
    out, nb, offs = bsgpu.compress_noalloc(bits, B, elem_size=es, offsets=torch.zeros_like(c.offsets))
    torch.cuda.synchronize()
    assert c.nbytes == int(nb.item())
    assert torch.equal(c.buf[:c.nbytes], out[:c.nbytes]) and torch.equal(c.offsets, offs)
