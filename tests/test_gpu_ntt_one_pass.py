"""Transforms on both sides of the line up to which all stages are one pass.

2^11 words in a tile (rows times the columns of a tile, csrc/ntt.cu plan_shape):
a transform within it is one launch of the pass kernel, an extension two; above
it the passes split.  Values against the oracle, word for word.
"""
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


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int64)).cuda()


def host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy().view(np.uint64)


def passes(call):
    pg.profile_enable()
    call()
    torch.cuda.synchronize()
    got = pg.profile_read()
    pg.profile_enable(False)
    return got["k_ntt_pass"]["launches"]


@pytest.mark.parametrize("log_n,cols,one", [(6, 8, True), (7, 1, True), (7, 3, True), (7, 64, True), (8, 8, True), (8, 13, True),
                                            (9, 3, True), (10, 2, True), (11, 1, True), (9, 8, False), (10, 3, False),
                                            (11, 2, False), (12, 1, False)])
def test_one_pass_up_to_2e11_words(log_n, cols, one):
    x = pg_synth.matrix(0x7A00 + 32 * log_n + cols, 1 << log_n, cols)
    t = dev(x)
    n = passes(lambda: pg.ntt(t))
    want = oracle.ntt_columns(x)
    assert (host(t) == want).all()
    assert (n == 1) == one
    pg.ntt(t, inverse=True)
    assert (host(t) == x).all()
    for b in (0, 1, 3, 7):
        e = dev(x)
        out = []
        n = passes(lambda: out.append(pg.lde(e, b)))
        assert (host(out[0]) == oracle.lde_columns(x, b)).all(), b
        assert (n == 2) == one, b
