"""Transforms of 2^9 and 2^10 rows with so many columns that one pass fills the GPU.

Both sides of the lines (csrc/ntt.cu plan_shape): 9 bits with more column chunks
than SMs, 10 bits from 2^18 rows times chunks on.  Launches counted, values against
the oracle on the first, some middle and the last columns, and a round trip.
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


@pytest.mark.parametrize("log_n,cols,want", [(9, 1216, 2), (9, 1217, 1), (9, 2003, 1), (10, 2040, 2), (10, 2041, 1), (10, 4100, 1),
                                             (11, 2050, 2)])
def test_one_pass_when_the_columns_fill_the_gpu(log_n, cols, want):
    x = pg_synth.matrix_torch(0x7C00 + 32 * log_n + cols, 1 << log_n, cols, device="cuda")
    pick = [0, 1, 7, 8, cols // 2, cols - 9, cols - 2, cols - 1]
    xs = np.ascontiguousarray(host(x[:, pick].contiguous()))
    t = x.clone()
    n = passes(lambda: pg.ntt(t))
    assert n == want
    assert (host(t[:, pick].contiguous()) == oracle.ntt_columns(xs)).all()
    pg.ntt(t, inverse=True)
    assert torch.equal(t, x)
    for b in (0, 2):
        assert (host(pg.lde(x, b)[:, pick].contiguous()) == oracle.lde_columns(xs, b)).all(), b


@pytest.mark.parametrize("cols,b", [(3, 8), (4, 9), (8, 9)])
def test_wide_extension_of_ten_bits(cols, b):
    x = pg_synth.matrix(0x7C80 + cols, 1 << 10, cols)
    t = torch.from_numpy(x.view(np.int64)).cuda()
    assert (host(pg.lde(t, b)) == oracle.lde_columns(x, b)).all()
