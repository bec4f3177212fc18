"""A look-back that runs out in the main compressor: a test build of the
library in which predecessors never look ready (a flag that nothing sets).
The bounded wait gives up, the status word says so, no block is placed at an
offset that nobody knows, and one limit is all that a call waits, however many
blocks a CTA has; nothing faults or hangs."""
import ctypes
import time

import pytest
import torch

from paper_1503_00638_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bs():
    from paper_1503_00638_gb300 import build
    build.build()
    from paper_1503_00638_gb300 import bsgpu
    return bsgpu


@pytest.fixture(scope="module")
def stalled(bs, tmp_path_factory):
    from paper_1503_00638_gb300 import build
    path = build.build(force=True, extra_flags=("-DBSG_TEST_LOOKBACK_STALL",),
                       lib=str(tmp_path_factory.mktemp("stall") / "libbsgpu_stall.so"))
    fn = ctypes.CDLL(path).bsgpu_compress
    fn.argtypes, fn.restype = bs._SIGS["bsgpu_compress"]
    return fn


def _call(bs, fn, d, B, level):
    n = d.numel()
    cap = bs.compress_bound(n, 4, B)
    out = torch.full((cap,), 0xAB, dtype=torch.uint8, device="cuda")
    nbytes = torch.full((1,), 12345, dtype=torch.int64, device="cuda")
    ws = bs.new_workspace(bs.workspace_size(bs.OP_COMPRESS, n, 4, B))
    torch.cuda.synchronize()
    t = time.monotonic()
    rc = fn(d.data_ptr(), n, 4, B, level, out.data_ptr(), cap, nbytes.data_ptr(), None,
            ws.data_ptr(), ws.numel(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    t = time.monotonic() - t
    assert rc == 0
    return out, int(nbytes.item()), bs.status(ws), t


@pytest.mark.parametrize("B,level", [(2048, 0), (1024, 0), (3072, 0), (2048, 1)])
def test_compress_reports_a_look_back_that_ran_out(bs, stalled, B, level):
    d = torch.from_numpy(synth.random_walk(2 * B, "int32", seed=5)).cuda()
    ref = bs.compress(d, B, level=level)
    first = int(ref.offsets[1].item())              # block 0 ends here
    out, nbytes, status, t_two = _call(bs, stalled, d, B, level)
    assert status == bs.ERR_TIMEOUT and nbytes == 0
    assert torch.equal(out[12:first], ref.buf[12:first])
    assert bool((out[first:] == 0xAB).all())        # block 1 was not placed
    # many blocks per CTA, after one another: still one limit
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    d = torch.zeros(6 * 32 * sms * B, dtype=torch.int32, device="cuda")
    _, nbytes, status, t_many = _call(bs, stalled, d, B, level)
    assert status == bs.ERR_TIMEOUT and nbytes == 0
    assert t_many < 2.5 * t_two + 0.5, (t_two, t_many)
    # the regular library still works
    d = torch.from_numpy(synth.random_walk(2 * B, "int32", seed=6)).cuda()
    c = bs.compress(d, B, level=level)
    back = bs.decompress(c.buf, c.nbytes, 2 * B, 4, B, offsets=c.offsets)
    assert torch.equal(back, d.view(torch.uint8))
