"""A served one-leaf tree is done only once all four words of its root are stored.

With four threads per state (batches of at most four leaf tasks per SM) the words
of a root come from four warps, so the flag that completes the request has to wait
for all of them.  One-leaf requests run beside a longer tree that keeps their batch
running; each is read the moment it is done and released, so that a later request
gets its buffer with other words in it.  Against the oracle, word for word.
"""
import time

import numpy as np
import pytest

import oracle
import pg_synth

torch = pytest.importorskip("torch")
pg = pytest.importorskip("paper_2506_09505_gb300")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def ready():
    pg.load(build_if_missing=True)
    pg.init(0)
    yield


@pytest.mark.parametrize("width", [1, 8, 13])
def test_one_leaf_roots_are_whole_when_done(width):
    host = [pg_synth.matrix(0xEE00 + 64 * width + k, 1, width) for k in range(32)]
    want = [oracle.hash_rows(h).view(np.int64) for h in host]
    rows = [torch.from_numpy(h.view(np.int64)).cuda() for h in host]
    long_host = pg_synth.matrix(0xEEF0 + width, 1 << 13, 64)
    long_rows = torch.from_numpy(long_host.view(np.int64)).cuda()
    long_root = oracle.merkle_build(long_host, nthreads=8)[-1].view(np.int64)
    torch.cuda.synchronize()
    srv = pg.Server(pool_bytes=1 << 24, max_inflight=2, schedule={"engine": pg.BATCH_ENGINE_TENSOR})
    try:
        for _ in range(4):
            long_id = srv.submit(long_rows)
            waiting = {srv.submit(r): k for k, r in enumerate(rows)}
            t0 = time.time()
            while waiting and time.time() - t0 < 30:
                for rid in [r for r in waiting if srv.query(r)["state"] == pg.REQ_DONE]:
                    got = srv.nodes(rid, 1).cpu().numpy()
                    srv.release(rid)
                    assert (got == want[waiting.pop(rid)]).all()
            assert not waiting
            srv.drain(30.0)
            assert (srv.nodes(long_id, 1 << 13)[-1].cpu().numpy() == long_root).all()
            srv.release(long_id)
    finally:
        srv.close()
