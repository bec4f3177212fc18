"""The compressor (a CTA per block) against the general compressor:
`compress_noalloc` takes the general kernel for every shape, and both must
write the same bytes; the oracle decodes them.  Sizes: one block and many,
block sizes of one to sixteen warps and in between, shortened last blocks
whose bit-rows are no whole words, verbatim tails, more blocks than CTAs."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# (element size, block elements); (4, 3072) takes three warps, (8, 96) a part
# of one, (4, 2048) / (8, 512) / (2, 4096) / (1, 8192) the kernels of a fixed
# block size
SHAPES = [(4, 2048), (4, 1024), (4, 32), (4, 3072), (4, 16384), (8, 1024), (8, 512), (8, 96),
          (8, 8192), (2, 4096), (2, 2048), (2, 64), (2, 16384), (1, 8192), (1, 4096), (1, 128),
          (1, 65536)]


def _walk(n, es, seed, noisy):
    g = np.random.Generator(np.random.PCG64([seed, es]))
    w = np.cumsum((g.integers(0, 2, n) * 2 - 1) << g.integers(0, 7, n))
    if noisy:       # stretches of zeros and of noise: matches of every length
        cut = g.integers(0, n, 1 + n // 300)
        for k, a in enumerate(cut):
            w[a:a + int(g.integers(1, 400))] = 0 if k % 2 else g.integers(-2 ** 31, 2 ** 31)
    return w.astype(np.int64).view(np.uint64).astype({1: np.uint8, 2: np.uint16, 4: np.uint32,
                                                      8: np.uint64}[es])


@pytest.mark.parametrize("level", [0, 1])
@pytest.mark.parametrize("noisy", [False, True])
@pytest.mark.parametrize("es,B", SHAPES)
def test_streams_equal_the_general_compressors(orc, es, B, noisy, level):
    from paper_1503_00638_gb300 import bsgpu
    many = max(2, 40_000_000 // (B * es * 10))       # more blocks than CTAs for the small blocks
    for n in (8, B - 8 if B > 8 else 8, B, B + 8, 3 * B + 40 + 5, many * B, many * B + B // 2 + 3):
        x = _walk(n, es, n % 1009, noisy)
        d = torch.from_numpy(x.view({1: np.uint8, 2: np.int16, 4: np.int32, 8: np.int64}[es])).cuda()
        c = bsgpu.compress(d, B, level=level)
        assert bsgpu.status(c.ws) == 0
        out, nb, offs = bsgpu.compress_noalloc(d, B, offsets=torch.zeros_like(c.offsets), level=level)
        torch.cuda.synchronize()
        assert c.nbytes == int(nb.item())
        assert torch.equal(c.buf[:c.nbytes], out[:c.nbytes])
        if bsgpu.num_blocks(n, es, B):
            assert torch.equal(c.offsets, offs)
        if n <= 4 * B:
            rc, back = orc.decompress(c.buf[:c.nbytes].cpu().numpy().tobytes(), n, x.dtype, B)
            assert rc == 0 and np.array_equal(back, x)


@pytest.mark.parametrize("tslow", [False, True])
@pytest.mark.parametrize("dtype", ["f32", "i32"])
@pytest.mark.parametrize("shape", [(3, 5, 16), (7, 16, 48), (2, 9, 40), (5, 4, 7), (1, 3, 1000)])
def test_cube_streams_equal_rounding_then_compressing(shape, dtype, tslow):
    """Fused rounding, by groups and by samples, every order and element
    size, against bsgpu_reduce_precision and the general compressor; samples
    the group rounding cannot take (huge values, NaN, infinities, an autos
    row that is zero) among them."""
    from paper_1503_00638_gb300 import bsgpu, synth
    F, n, T = shape
    cfg = synth.VisConfig(F, n, T, 2 ** 16, 0.01, seed=F * n + T)
    if dtype == "f32":
        v = synth.visibilities(cfg)
        flat = v.reshape(-1).view(np.float32)
        g = np.random.Generator(np.random.PCG64(5))
        k = g.integers(0, flat.size, 12)
        flat[k] = np.array([np.nan, np.inf, -np.inf, 3e38, -1e30, 1e-40, -0.0, 1e9, 7.5e8, -2e12,
                            0.0, 1e20], np.float32)
        v[0, synth.auto_product_index(1, n)] = 0
        d = torch.from_numpy(v).cuda()
    else:
        d = torch.from_numpy(synth.visibilities_int(cfg, 2.0 ** 22)).cuda()
    src = d.permute(2, 0, 1, *range(3, d.dim())).contiguous() if tslow else d
    for comp in (False, True):
        want = bsgpu.reduce_precision(d, cfg.n_samp, cfg.f, compensate=comp)
        bits = torch.view_as_real(want) if dtype == "f32" else want
        for es, B in ((4, 2048), (4, 1024), (4, 96), (8, 1024), (8, 512), (8, 64)):
            c = bsgpu.compress_vis_ex(src, cfg.n_samp, cfg.f, compensate=comp, elem_size=es,
                                      block_elems=B, time_slowest=tslow)
            assert bsgpu.status(c.ws) == 0
            out, nb, _ = bsgpu.compress_noalloc(bits.contiguous(), B, elem_size=es)
            torch.cuda.synchronize()
            assert c.nbytes == int(nb.item())
            assert torch.equal(c.buf[:c.nbytes], out[:c.nbytes])
        c = bsgpu.compress_vis_ex(src, cfg.n_samp, cfg.f, compensate=comp, block_elems=2048,
                                  time_slowest=tslow, level=1)
        out, nb, _ = bsgpu.compress_noalloc(bits.contiguous(), 2048, elem_size=4, level=1)
        assert c.nbytes == int(nb.item()) and torch.equal(c.buf[:c.nbytes], out[:c.nbytes])


@pytest.mark.parametrize("shape", [(1, 40, 300), (2, 128, 1), (3, 24, 1100), (1, 90, 33)])
def test_compensated_f_over_slices_of_the_products(orc, shape):
    """The minimum over the products taken slice by slice, in both orders and
    over time axes longer than a CTA, bit for bit the oracle's."""
    from paper_1503_00638_gb300 import bsgpu, synth
    F, n, T = shape
    cfg = synth.VisConfig(F, n, T, 2 ** 14, 0.05, seed=n, rho=0.6)
    v = synth.visibilities(cfg)
    v[0, 5] = np.complex64(complex(np.nan, 1.0)) if T > 1000 else v[0, 5]
    want = orc.reduce_precision(v, cfg.n_samp, cfg.f, True).view(np.uint32)
    d = torch.from_numpy(v).cuda()
    for tslow in (False, True):
        x = d.permute(2, 0, 1).contiguous() if tslow else d
        got = bsgpu.reduce_precision(x, cfg.n_samp, cfg.f, True, time_slowest=tslow)
        assert np.array_equal(got.cpu().numpy().view(np.uint32), want)
