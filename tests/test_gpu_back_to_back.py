"""Calls that follow each other on a stream with no synchronisation between them.

Every launch here may be resident while the one before it still writes what it
reads (programmatic dependent launch), on buffers whose old words would be taken
for new ones if a read came too early or from a stale line.  The prover's sequence
-- extension, commitment, openings, path checks -- and permutations in place, run
eagerly and as a captured graph, against the oracle word for word.
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


def shifted(a, words):
    """The words of `a` on the device, `words` words past a 256-byte boundary."""
    buf = torch.empty(a.size + words, dtype=torch.int64, device="cuda")
    view = buf[words:].view(a.shape)
    view.copy_(dev(a))
    return view


@pytest.mark.parametrize("n,off", [(1, 0), (129, 1), (300, 2), (19457, 0), (19457, 2), (80003, 1), (80003, 2)])
def test_permutations_in_place_back_to_back(n, off):
    st = pg_synth.matrix(0xB2B0 + n + off, n, 12)
    t = shifted(st, off)
    for _ in range(3):
        pg.permute_batch(t)
    want = st
    for _ in range(3):
        want = oracle.permute(want, nthreads=8)
    assert (host(t) == want).all()


def _commit(evals, b, out, scratch, nodes, idx):
    """Extension, commitment, openings and their check; no synchronisation."""
    n = out.shape[0]
    pg.lde(evals, b, out=out, scratch=scratch)
    pg.merkle_build(out, nodes)
    paths = pg.merkle_open(nodes, n, idx)
    ok = pg.merkle_verify(nodes[-1], n, nodes[idx].contiguous(), idx, paths)
    return paths, ok


def _paths(nodes, n, idx):
    off = pg.level_offsets(n)
    return np.stack([nodes[off[l] + ((idx >> l) ^ 1)] for l in range(len(off) - 1)], axis=1)


# widths that read rows 8 and 16 bytes at a time; leaves in the latency form, at
# one unit per SM and above it; openings checked on lanes and on the tensor cores
@pytest.mark.parametrize("log_n,b,cols,k", [(9, 1, 3, 33), (12, 2, 8, 700), (13, 2, 3, 6000), (15, 1, 5, 20000),
                                            (16, 1, 8, 1021)])
def test_extension_commitment_openings_on_reused_buffers(log_n, b, cols, k):
    n, big = 1 << log_n, 1 << (log_n + b)
    inputs = [pg_synth.matrix(0xB300 + 16 * log_n + i, n, cols) for i in range(2)]
    device_inputs = [dev(x) for x in inputs]
    idx_h = np.random.default_rng(log_n).integers(0, big, k)
    idx = torch.from_numpy(idx_h).cuda()
    evals = torch.empty((n, cols), dtype=torch.int64, device="cuda")
    scratch = torch.empty_like(evals)
    out = torch.empty((big, cols), dtype=torch.int64, device="cuda")
    nodes = torch.empty((2 * big - 1, 4), dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    got = []
    for r in range(4):
        evals.copy_(device_inputs[r % 2])
        paths, ok = _commit(evals, b, out, scratch, nodes, idx)
        got.append((nodes.clone(), paths, ok))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        gpaths, gok = _commit(evals, b, out, scratch, nodes, idx)
    for r in range(4):
        evals.copy_(device_inputs[r % 2])
        graph.replay()
        got.append((nodes.clone(), gpaths.clone(), gok.clone()))
    trees = [oracle.merkle_build(oracle.lde_columns(x, b), nthreads=8) for x in inputs]
    for r, (nd, paths, ok) in enumerate(got):
        assert (host(nd) == trees[r % 2]).all(), r
        assert (host(paths) == _paths(trees[r % 2], big, idx_h)).all(), r
        assert ok.all().item(), r


@pytest.mark.parametrize("log_n,cols", [(4, 3), (16, 3)])
def test_captured_transforms_and_permutations_after_copies(log_n, cols):
    """A captured dependent launch whose predecessor is a copy, and replays back to back."""
    x = pg_synth.matrix(0xB400 + log_n, 1 << log_n, cols)
    st = pg_synth.matrix(0xB410 + log_n, 257, 12)
    src, states = dev(x), dev(st)
    t, u = torch.empty_like(src), torch.empty_like(states)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        t.copy_(src)
        pg.ntt(t)
        u.copy_(states)
        pg.permute_batch(u)
        digests = pg.hash_rows(t)
    for _ in range(3):
        graph.replay()
    want = oracle.ntt_columns(x)
    assert (host(t) == want).all()
    assert (host(u) == oracle.permute(st)).all()
    assert (host(digests) == oracle.hash_rows(want)).all()
