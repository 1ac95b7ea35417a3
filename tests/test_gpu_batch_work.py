"""Batches on both sides of the line between four threads per state and one.

The line weighs a batch's units against its longest chain (csrc/pg12.cu
tc_small_batch): narrow and wide rows, few large and many small trees, fused levels
and handed-off tops, against the oracle word for word.  And a batch of wide rows
may not take longer than a larger one.
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


# (log2 leaves, width, trees): units a chain and SM of 0.6, 1.2, 1.9, 1.8, 4.0 and, fused, 1.1 and 2
@pytest.mark.parametrize("log_n,width,trees,fuse,top", [(12, 8, 10, 0, 1), (10, 8, 76, 0, 1), (10, 64, 57, 0, 1),
                                                        (8, 8, 152, 0, 16), (5, 24, 608, 0, 1), (10, 8, 152, 1, 16),
                                                        (10, 16, 152, 2, 1)])
def test_batches_on_both_sides_of_the_line(log_n, width, trees, fuse, top):
    hosts = [pg_synth.matrix(0x9D00 + k, 1 << log_n, width) for k in range(trees)]
    nodes = pg.merkle_build_batch([dev(h) for h in hosts], schedule={"engine": pg.BATCH_ENGINE_TENSOR, "fuse_levels": fuse,
                                                                     "top_lanes": top})
    for h, got in zip(hosts, nodes):
        assert (got.cpu().numpy().view(np.uint64) == oracle.merkle_build(h, nthreads=8)).all()


def test_a_batch_of_wide_rows_takes_no_longer_than_a_larger_one():
    tasks_per_sm = torch.cuda.get_device_properties(0).multi_processor_count * 4

    def best(trees):
        rows = [torch.randint(-2**63, 2**63 - 1, (1 << 10, 256), dtype=torch.int64, device="cuda") for _ in range(trees)]
        graph = pg.BatchGraph(rows, schedule={"engine": pg.BATCH_ENGINE_TENSOR})
        times = []
        for _ in range(6):
            a, z = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            graph.launch()
            z.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(z))
        graph.close()
        return min(times[1:])
    assert best(tasks_per_sm // 8) < 1.2 * best(tasks_per_sm // 8 + 1)
