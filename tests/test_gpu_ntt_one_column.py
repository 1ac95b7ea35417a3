"""Large transforms of one column, on both sides of the line between two and three passes.

Up to 20 bits in two passes on tiles of 2^11 rows, above in three (csrc/ntt.cu
plan_shape).  Values against the oracle; and an extension of one column, which
moves half the words of two, may not come near the time of two.
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


@pytest.mark.parametrize("log_n", [19, 20, 21])
def test_one_column_transform(log_n):
    x = pg_synth.matrix(0x7B00 + log_n, 1 << log_n, 1)
    t = dev(x)
    pg.ntt(t)
    assert (host(t) == oracle.ntt_columns(x)).all()
    pg.ntt(t, inverse=True)
    assert (host(t) == x).all()


@pytest.mark.parametrize("log_n,b", [(3, 16), (11, 8), (12, 7), (16, 3), (18, 1), (18, 2), (19, 0), (19, 1), (20, 1), (21, 1)])
def test_one_column_extension(log_n, b):
    x = pg_synth.matrix(0x7B40 + 32 * log_n + b, 1 << log_n, 1)
    assert (host(pg.lde(dev(x), b)) == oracle.lde_columns(x, b)).all()


@pytest.mark.parametrize("log_n,b", [(19, 0), (20, 3)])
def test_one_column_takes_well_under_the_time_of_two(log_n, b):
    def best(cols):
        e = pg_synth.matrix_torch(0x7B90 + cols, 1 << log_n, cols, device="cuda")
        out = torch.empty((1 << (log_n + b), cols), dtype=torch.int64, device="cuda")
        scratch = torch.empty_like(e)
        times = []
        for k in range(12):
            a, z = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(8):
                pg.lde(e, b, out=out, scratch=scratch)
            z.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(z))
        return min(times[2:])
    assert best(1) < 0.75 * best(2)
