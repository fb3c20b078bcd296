"""Which form of a chain runs on either side of the lines between forms, as the graph or the kernel itself reports it, and that the
results on both sides are the same."""
import numpy as np
import pytest
import torch

from paper_2607_08973_b200 import binding as sf
from paper_2607_08973_b200 import synth

from gpu_util import BF16, F32, Ctx, assert_bits_equal
from test_gpu_chains import _oracle_w, _ring, _rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,n,dtype,mode,by_tags", [
    (8, 1, BF16, sf.SPECULATIVE, 1), (8, 73_728, BF16, sf.SPECULATIVE, 1), (8, 73_729, BF16, sf.SPECULATIVE, 0),   # 48 and 49 tiles
    (4, 73_728, F32, sf.SPECULATIVE, 1), (4, 73_729, F32, sf.SPECULATIVE, 0),
    (2, 294_912, BF16, sf.SPECULATIVE, 1), (2, 294_913, BF16, sf.SPECULATIVE, 0),
    (8, 4096, BF16, sf.DUALBUF, 0), (8, 4096, BF16, sf.BARRIER_ONESHOT, 0)])
def test_graphs_by_tags_up_to_the_line(oracle, P, n, dtype, mode, by_tags):
    steps = 4
    d = synth.chain_workload("llama", P)
    with Ctx(P, n, dtype) as ctx:
        ring, stride = _ring(n, dtype, steps)
        ch = sf.sifar_chain_create(ctx.h, sf.make_workload(**d), n, mode, sf.CHAIN_GRAPH, ring.data_ptr(), steps, steps)
        try:
            g = sf.sifar_chain_graph_shape(ch)
            sf.sifar_chain_run(ch, 0)
            torch.cuda.synchronize()
        finally:
            sf.sifar_chain_destroy(ch)
        assert sf.sifar_status(ctx.h) == 0
    assert g["kernels"] == 2 * steps and g["tagged_producers"] == by_tags * steps
    want = oracle.chain(_oracle_w(oracle, d), P, n, dtype, steps)
    for t, row in enumerate(_rows(ring, stride, steps, n, dtype)):
        assert_bits_equal(row, want[t], dtype, f"step {t + 1}")


@pytest.mark.parametrize("P,dtype,pairs,above", [(1, BF16, 40_000, None), (1, F32, 30_000, None), (2, BF16, 37_000, 1),
                                                 (3, BF16, 52_000, 0), (3, F32, 65_000, 0), (5, F32, 75_000, 0), (6, F32, 60_000, 0)])
def test_speculative_clusters_end_by_ranks_and_type(monkeypatch, P, dtype, pairs, above):
    """The largest payload whose chunks are clusters and the first above it (there: for placement only, or none; where no line is
    given, one well inside), against chunks spread over the machine; two runs, the second from the first."""
    steps = 6
    d = synth.chain_workload("sweep", P)
    per_unit = 6 if dtype == BF16 else 3
    for n, clustered in ((pairs // P * per_unit, 1), (pairs // P * per_unit + 1, 1 if above is None else above)):
        results = []
        for env in ("1", "0"):
            monkeypatch.setenv("SIFAR_CHAIN_CLUSTER", env)
            with Ctx(P, n, dtype) as ctx:
                ring, stride = _ring(n, dtype, steps)
                ch = sf.sifar_chain_create(ctx.h, sf.make_workload(**d), n, sf.SPECULATIVE, sf.CHAIN_PERSISTENT,
                                           ring.data_ptr(), steps, steps)
                for _ in range(2):
                    sf.sifar_chain_run(ch, 0)
                torch.cuda.synchronize()
                assert sf.sifar_status(ctx.h) == 0
                g = sf.sifar_chain_geometry(ch)
                sf.sifar_chain_destroy(ch)
                assert g["clustered"] == g["kernel_clustered"] == (clustered if env == "1" else 0)
                results.append(_rows(ring, stride, steps, n, dtype))
        assert results[0][-1].any() and np.array_equal(results[0].view(np.uint8), results[1].view(np.uint8))
