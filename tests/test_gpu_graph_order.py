"""Graph chains in tagged words: a step's producers have no place on the GPU before the reducer that they poll for has its own,
so however many such chains run at once, what waits never holds the place of what it waits for."""
import pytest
import torch

from paper_2607_08973_b200 import binding as sf
from paper_2607_08973_b200 import synth

from gpu_util import BF16, F32, Ctx, assert_bits_equal
from test_gpu_chains import _oracle_w, _ring, _rows

pytestmark = pytest.mark.gpu


def _create(ctx, d, n, dtype, steps, mode=sf.SPECULATIVE):
    ring, stride = _ring(n, dtype, steps)
    return sf.sifar_chain_create(ctx.h, sf.make_workload(**d), n, mode, sf.CHAIN_GRAPH, ring.data_ptr(), steps, steps), ring, stride


@pytest.mark.parametrize("P,n,dtype,steps", [(8, 1, BF16, 2), (8, 4096, BF16, 8), (3, 50_001, F32, 6), (8, 73_727, BF16, 4)])
def test_producers_follow_the_reducer_they_poll_for(P, n, dtype, steps):
    with Ctx(P, n, dtype) as ctx:
        ch, _, _ = _create(ctx, synth.chain_workload("llama", P), n, dtype, steps)
        try:
            g = sf.sifar_chain_graph_shape(ch)
        finally:
            sf.sifar_chain_destroy(ch)
    # per step after the first: the reducer behind the reducer's end, the producers let in by both kernels before them
    assert g == {"kernels": 2 * steps, "tagged_producers": steps, "end_edges": steps - 1, "let_in_edges": 2 * (steps - 1)}


@pytest.mark.parametrize("chains,P,n,dtype", [(3, 8, 4099, BF16), (5, 8, 73_727, BF16), (4, 2, 250_007, BF16)])
def test_several_chains_at_once(oracle, chains, P, n, dtype):
    """A stream each, enqueued without waiting; their producers alone could fill the GPU more than once."""
    steps, runs = 16, 4
    ctxs = [Ctx(P, n, dtype) for _ in range(chains)]
    streams = [torch.cuda.Stream() for _ in range(chains)]
    ds = [dict(synth.chain_workload("llama", P), seed=11 + i) for i in range(chains)]
    try:
        made = [_create(ctx, d, n, dtype, steps) for ctx, d in zip(ctxs, ds)]
        torch.cuda.synchronize()
        for _ in range(runs):
            for (ch, _, _), s in zip(made, streams):
                sf.sifar_chain_run(ch, s.cuda_stream)
        torch.cuda.synchronize()
        got = []
        for (ch, ring, stride), ctx in zip(made, ctxs):
            assert sf.sifar_status(ctx.h) == 0
            got.append(_rows(ring, stride, steps, n, dtype))
            sf.sifar_chain_destroy(ch)
    finally:
        for ctx in ctxs:
            ctx.__exit__()
    for i, d in enumerate(ds):
        want = oracle.chain(_oracle_w(oracle, d), P, n, dtype, steps * runs)
        for t in range(steps):
            assert_bits_equal(got[i][t], want[(runs - 1) * steps + t], dtype, f"chain {i} step {(runs - 1) * steps + t + 1}")


def test_the_environment_is_read_once(monkeypatch):
    """SIFAR_CHAIN_PDL, set after the first chain, changes neither the form nor the order of a later one."""
    P, n, steps = 8, 4096, 6
    shapes = []
    with Ctx(P, n, BF16) as ctx:
        for env in (None, "0"):
            if env is not None:
                monkeypatch.setenv("SIFAR_CHAIN_PDL", env)
            ch, _, _ = _create(ctx, synth.chain_workload("llama", P), n, BF16, steps)
            shapes.append(sf.sifar_chain_graph_shape(ch))
            sf.sifar_chain_destroy(ch)
    assert shapes[0] == shapes[1] and shapes[0]["tagged_producers"] == steps
