"""Transforms on both sides of every line of the pass plan (csrc/ntt.cu, plan_shape).

Below 2^19 rows (times chunks of eight columns) a transform runs on blocks of
256 threads whose tiles shrink with the size; from there on blocks of 128
threads.  Every column-chunk width, the smallest tile, the last and first size
of each kind, and row counts that leave passes of one and two bits, against
the oracle, word for word.
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


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int64)).cuda()


def _host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy().view(np.uint64)


@pytest.mark.parametrize("log_n,cols", [(6, 1), (7, 3), (8, 8), (12, 2), (14, 5), (15, 20), (16, 3), (16, 63), (16, 64),
                                        (18, 1), (18, 2), (18, 4), (18, 8), (19, 1), (19, 2), (19, 3), (19, 8)])
def test_transform_matches_the_oracle(log_n, cols):
    x = pg_synth.matrix(0x9A00 + 64 * log_n + cols, 1 << log_n, cols)
    want = oracle.ntt_columns(x)
    t = pg.ntt(_dev(x))
    assert (_host(t) == want).all()
    assert (_host(pg.ntt(t, inverse=True)) == x).all()


@pytest.mark.parametrize("log_n,log_b,cols", [(5, 1, 8), (9, 3, 1), (16, 1, 8), (16, 3, 3), (17, 1, 8), (17, 2, 8),
                                              (18, 1, 1), (17, 2, 2)])
def test_extension_matches_the_oracle(log_n, log_b, cols):
    ev = pg_synth.matrix(0x9B00 + 64 * log_n + 8 * log_b + cols, 1 << log_n, cols)
    assert (_host(pg.lde(_dev(ev), log_b)) == oracle.lde_columns(ev, log_b)).all()
