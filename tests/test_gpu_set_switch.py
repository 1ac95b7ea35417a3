"""The first launch after a change of parameter set reads the new tables.

On a stream that does not wait for the legacy stream, right after the switch;
permutations, row digests and a small tree (all three table copies) in both sets,
against the oracle.
"""
import numpy as np
import pytest

import oracle
import pg_synth

torch = pytest.importorskip("torch")
pg = pytest.importorskip("paper_2506_09505_gb300")

pytestmark = pytest.mark.gpu


def test_first_launches_after_a_switch_use_the_new_set():
    pg.load(build_if_missing=True)
    pg.init(0)
    st = pg_synth.matrix(0xB500, 200, 12)
    rows = pg_synth.matrix(0xB501, 64, 9)
    t0, r0 = (torch.from_numpy(a.view(np.int64)).cuda() for a in (st, rows))
    side = torch.cuda.Stream()
    got = []
    try:
        for k in range(12):
            t = t0.clone()
            torch.cuda.synchronize()
            pg.params_select("pg12_small" if k % 2 == 0 else None)
            with torch.cuda.stream(side):
                got.append((pg.permute_batch(t), pg.hash_rows(r0), pg.merkle_build(r0)))
            side.synchronize()
    finally:
        pg.params_select(None)
    for k, (t, digests, nodes) in enumerate(got):
        rc, mds = (oracle.params_small() if k % 2 == 0 else oracle.params())[:2]
        want = oracle.permute(st, rc=rc, mds=mds)
        assert (t.cpu().numpy().view(np.uint64) == want).all(), k
        leaves = oracle.hash_rows(rows, rc=rc, mds=mds)
        assert (digests.cpu().numpy().view(np.uint64) == leaves).all(), k
        assert (nodes[:64].cpu().numpy().view(np.uint64) == leaves).all(), k
