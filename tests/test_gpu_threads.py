"""Threads with different block sizes share the kernels: no call is refused,
and each stream stays its own."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


def test_threads_with_different_block_sizes():
    from paper_1503_00638_gb300 import bsgpu, synth
    errors = []

    def work(es, B, level):
        try:
            torch.cuda.set_device(0)
            with torch.cuda.stream(torch.cuda.Stream()):
                n = 5 * B + 13
                d = synth.random_walk_device(n, es, seed=B)
                want = bsgpu.compress(d, B, es, level=level)
                torch.cuda.current_stream().synchronize()
                ws = bsgpu.new_workspace(bsgpu.workspace_size(bsgpu.OP_DECOMPRESS, n, es, B))
                for _ in range(400):
                    c = bsgpu.compress(d, B, es, level=level, ws=want.ws)
                    back = bsgpu.decompress(want.buf, want.nbytes, n, es, B, offsets=want.offsets, ws=ws)
                torch.cuda.current_stream().synchronize()
                assert c.nbytes == want.nbytes and torch.equal(c.buf[:c.nbytes], want.buf[:want.nbytes])
                assert torch.equal(back, d) and bsgpu.status(ws) == 0
        except Exception as e:      # noqa: BLE001 - reported by the main thread
            errors.append(f"{es} {B} {level}: {e!r}")
    # shared memory of one kernel just over 48 KiB to its most
    threads = [threading.Thread(target=work, args=a) for a in
               [(4, 16384, 0), (4, 12288, 0), (8, 8192, 0), (8, 6400, 0), (4, 16384, 1), (4, 13312, 1)]]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
