"""The compensated f at the sizes where its kernel changes form (a few lanes
to a sample for few inputs, a CTA or slices of one per frequency for more),
bit for bit the oracle's, in both orders and for both data types."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


# one input (no cross product), two, the largest of the first rule with one and
# with many samples, both sides of the second (16 n^2 samples), and more inputs
# with few times (several warps to a time in the time-slowest order)
@pytest.mark.parametrize("shape", [(3, 1, 5), (700, 2, 33), (1, 12, 1), (2100, 12, 3), (5, 13, 9),
                                   (1, 16, 4095), (1, 16, 4097), (16, 32, 1024), (2, 33, 3),
                                   (3, 40, 7), (2, 64, 1)])
@pytest.mark.parametrize("dtype", ["f32", "i32"])
def test_compensated_rounding_equals_the_oracles(orc, shape, dtype):
    from paper_1503_00638_gb300 import bsgpu, synth
    F, n, T = shape
    cfg = synth.VisConfig(F, n, T, 2 ** 14, 0.05, seed=F + n + T, rho=0.6)
    if dtype == "f32":
        v = synth.visibilities(cfg)
        if n > 1:       # a product that is no number, an autos row of zeros
            v[0, 1, 0] = np.complex64(complex(np.nan, 1.0))
            v[F - 1, synth.auto_product_index(1, n), T - 1] = 0
    else:
        v = synth.visibilities_int(cfg, 2.0 ** 16)
    want = orc.reduce_precision(v, cfg.n_samp, cfg.f, True).view(np.uint32)
    d = torch.from_numpy(v).cuda()
    for tslow in (False, True):
        x = d.permute(2, 0, 1, *range(3, d.dim())).contiguous() if tslow else d
        got = bsgpu.reduce_precision(x, cfg.n_samp, cfg.f, True, time_slowest=tslow)
        assert np.array_equal(got.cpu().numpy().view(np.uint32), want)
