"""Decoding around the block sizes where the decoder changes (8 and 16 KiB),
every element size, with and without a block index, shortened last blocks, and
the verdict on a damaged stream; against the data and the oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("es", [1, 2, 4, 8])
@pytest.mark.parametrize("size", [8192, 8256, 12288, 16320, 16384, 16448, 32768, 65536])
def test_blocks_around_the_decoders_limits(orc, es, size):
    from paper_1503_00638_gb300 import bsgpu, synth
    B = size // es
    for n in (B, 3 * B + 8, 700 * B + B // 2 // 8 * 8 + 5):
        d = synth.random_walk_device(n, es, seed=n % 997)
        c = bsgpu.compress(d, B, es)
        for offs in (c.offsets, None):
            ws = bsgpu.new_workspace(bsgpu.workspace_size(bsgpu.OP_DECOMPRESS, n, es, B))
            back = bsgpu.decompress(c.buf, c.nbytes, n, es, B, offsets=offs, ws=ws)
            assert bsgpu.status(ws) == 0 and torch.equal(back, d)
    # another first token in block 1: 15 literals and more, a match of 19 and more
    bad = c.stream_bytes().clone()
    first = int(c.offsets[1].item())
    bad[first + 4] = 0xFF
    want, _ = orc.decompress(bad.cpu().numpy().tobytes(), n, {1: np.uint8, 2: np.uint16, 4: np.uint32,
                                                             8: np.uint64}[es], B)
    ws = bsgpu.new_workspace(bsgpu.workspace_size(bsgpu.OP_DECOMPRESS, n, es, B))
    bsgpu.decompress(bad, bad.numel(), n, es, B, offsets=c.offsets, ws=ws)
    assert (bsgpu.status(ws) == 0) == (want == 0)
