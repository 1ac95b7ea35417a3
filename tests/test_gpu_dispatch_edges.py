"""Both sides of each line at which a launch changes kernel form (csrc/pg12.cu).

Four threads per state up to one unit of 128 states per SM, one above
(permutations, row digests, path checks); batches up to four leaf tasks per SM;
path checks on 32 lanes, 16 lanes and the tensor cores.  Against the oracle, word
for word.
"""
import numpy as np
import pytest

import oracle
import pg_synth

torch = pytest.importorskip("torch")
pg = pytest.importorskip("paper_2506_09505_gb300")

pytestmark = pytest.mark.gpu
UNIT = 128


@pytest.fixture(scope="module", autouse=True)
def ready():
    pg.load(build_if_missing=True)
    pg.init(0)
    yield


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int64)).cuda()


def _host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy().view(np.uint64)


@pytest.mark.parametrize("extra", [-1, 0, 1])
def test_permutations_around_one_unit_per_sm(extra):
    st = pg_synth.matrix(0x9C00 + extra, _sms() * UNIT + extra, 12)
    st[-1] = np.uint64((1 << 64) - 1)
    t = _dev(st)
    pg.permute_batch(t)
    assert (_host(t) == oracle.permute(st, nthreads=8)).all()


@pytest.mark.parametrize("extra,width", [(0, 13), (1, 13), (0, 8), (1, 8)])
def test_row_digests_around_one_unit_per_sm(extra, width):
    rows = pg_synth.matrix(0x9C10 + 2 * width + extra, _sms() * UNIT + extra, width)
    assert (_host(pg.hash_rows(_dev(rows))) == oracle.hash_rows(rows)).all()


@pytest.mark.parametrize("log_n", [0, 1, 9])
def test_path_checks_around_every_line(log_n):
    n, sms = 1 << log_n, _sms()
    nodes_h = oracle.merkle_build(pg_synth.matrix(0x9C40 + log_n, n, 8), nthreads=8)
    nodes, root = _dev(nodes_h), _dev(nodes_h[-1])
    for k in (1, 2, 4 * sms, 4 * sms + 1, 5120, 5121, sms * UNIT, sms * UNIT + 1):
        rng = np.random.default_rng(k)
        idx_h = rng.integers(0, n, k)
        idx = torch.from_numpy(idx_h).cuda()
        paths = pg.merkle_open(nodes, n, idx) if log_n else torch.empty((k, 0, 4), dtype=torch.int64, device="cuda")
        leaves = nodes[idx].contiguous()
        want = np.ones(k, dtype=bool)
        for q in {0, k // 2, k - 1}:  # one word of a leaf or of a path, or the position, is wrong
            what = rng.integers(0, 3)
            if what == 0:
                leaves[q, int(rng.integers(0, 4))] ^= 1 << 40
            elif what == 1 and log_n:
                paths[q, int(rng.integers(0, log_n)), int(rng.integers(0, 4))] ^= 1
            else:
                idx[q] += n
            want[q] = False
        ok = pg.merkle_verify(root, n, leaves, idx, paths)
        assert (ok.cpu().numpy().astype(bool) == want).all(), k


@pytest.mark.parametrize("extra", [0, 1])
def test_batches_around_four_tasks_per_sm(extra):
    tasks = 4 * _sms()
    sizes = [(7 + b, 8 + 5 * (b % 2)) for b in range(tasks.bit_length()) if tasks >> b & 1]
    sizes += [(4, 3)] * extra  # one more task: a tree of less than a unit
    host_rows = [pg_synth.matrix(0x9C80 + i, 1 << lg, w) for i, (lg, w) in enumerate(sizes)]
    nodes = pg.merkle_build_batch([_dev(r) for r in host_rows], schedule={"engine": pg.BATCH_ENGINE_TENSOR})
    for rows, got in zip(host_rows, nodes):
        assert (_host(got) == oracle.merkle_build(rows, nthreads=8)).all()
