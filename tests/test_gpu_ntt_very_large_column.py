"""One column of 2^26 and 2^27 rows: both sides of the line at which the tiles grow again.

The oracle's transform of such a column takes minutes, so the input is one whose
transform is known in closed form: a polynomial of a few terms.  Its values on the
subgroup and on the coset are checked at random positions with Python integers.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pg = pytest.importorskip("paper_2506_09505_gb300")

pytestmark = pytest.mark.gpu
P = oracle.P


@pytest.fixture(scope="module", autouse=True)
def ready():
    pg.load(build_if_missing=True)
    pg.init(0)
    yield


def sparse(log_n, seed):
    """{exponent: coefficient} of a few terms, and the coefficient column on the device."""
    rng = np.random.default_rng(seed)
    n = 1 << log_n
    terms = {int(j): int(a) for j, a in zip([1, n - 1, *rng.integers(0, n, 4)], rng.integers(1, P, 6, dtype=np.uint64))}
    col = torch.zeros((n, 1), dtype=torch.int64, device="cuda")
    for j, a in terms.items():
        col[j, 0] = int(np.array(a, dtype=np.uint64).view(np.int64))
    return terms, col


def check(values, terms, log_n, shift, seed):
    n, w = 1 << log_n, oracle.two_adic_root(log_n)
    where = np.concatenate([[0, 1, n - 1, n // 2], np.random.default_rng(seed).integers(0, n, 400)])
    got = values[torch.from_numpy(where).cuda(), 0].cpu().numpy().view(np.uint64)
    for k, v in zip(where, got):
        x = shift * pow(w, int(k), P) % P
        assert int(v) == sum(a * pow(x, j, P) for j, a in terms.items()) % P, int(k)


@pytest.mark.parametrize("log_n,b", [(26, 1), (27, 0), (27, 2)])
def test_transform_and_extension_of_a_sparse_polynomial(log_n, b):
    terms, col = sparse(log_n, log_n)
    evals = pg.ntt(col.clone())
    check(evals, terms, log_n, 1, 1)
    check(pg.lde(evals, b), terms, log_n + b, oracle.LDE_SHIFT, 2)
    assert torch.equal(pg.ntt(evals, inverse=True), col)


def test_one_very_large_column_takes_well_under_the_time_of_two():
    def best(cols):
        e = torch.randint(-2**63, 2**63 - 1, (1 << 27, cols), dtype=torch.int64, device="cuda")
        out = torch.empty((1 << 29, cols), dtype=torch.int64, device="cuda")
        scratch = torch.empty_like(e)
        times = []
        for _ in range(4):
            a, z = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            pg.lde(e, 2, out=out, scratch=scratch)
            z.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(z))
        return min(times[1:])
    assert best(1) < 0.8 * best(2)
