"""A chain is ready when its creation returns, whatever the caller's default stream still has to do."""
import pytest
import torch

from paper_2607_08973_b200 import binding as sf
from paper_2607_08973_b200 import synth

from gpu_util import BF16, F32, Ctx, assert_bits_equal
from test_gpu_chains import _oracle_w, _ring, _rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,n,dtype,mode", [
    ("graph", 4099, BF16, sf.SPECULATIVE), ("graph", 16384, BF16, sf.BARRIER_ONESHOT),
    ("persistent", 4099, BF16, sf.SPECULATIVE), ("persistent", 65_536, BF16, sf.DUALBUF),
    ("persistent", 98_305, BF16, sf.SPECULATIVE), ("persistent", 30_001, F32, sf.BARRIER_ONESHOT),
    ("readers", 4099, BF16, sf.SPECULATIVE), ("readers", 65_536, F32, sf.DUALBUF)])
def test_the_default_stream_may_be_busy_while_a_chain_is_created(oracle, kind, n, dtype, mode):
    """A chain of the same size is destroyed first, so that its memory, call numbers in it, is there to be given out again.
    The first run ends while the default stream is still busy, the second starts when that is over: state that were zeroed in
    the default stream's turn would be old in the first and wiped between the two."""
    P, steps = 8, 6
    d = synth.chain_workload("llama", P)
    copies = P if kind == "readers" else 1

    def create(ctx, ring, seed):
        w = sf.make_workload(**dict(d, seed=seed))
        if kind == "readers":
            return sf.sifar_symchain_create(ctx.h, w, n, mode, ring.data_ptr(), steps, steps)
        impl = sf.CHAIN_GRAPH if kind == "graph" else sf.CHAIN_PERSISTENT
        return sf.sifar_chain_create(ctx.h, w, n, mode, impl, ring.data_ptr(), steps, steps)

    run, destroy = ((sf.sifar_symchain_run, sf.sifar_symchain_destroy) if kind == "readers" else
                    (sf.sifar_chain_run, sf.sifar_chain_destroy))
    ring, stride = _ring(n, dtype, copies * steps)
    other = torch.cuda.Stream()                       # a stream that the default one does not hold back
    with Ctx(P, n, dtype) as old, Ctx(P, n, dtype) as ctx:
        ch = create(old, ring, 77)
        for _ in range(2):
            run(ch, 0)
        torch.cuda.synchronize()
        destroy(ch)
        for _ in range(4):
            sf.sifar_spin(50_000_000, 0)
        ch = create(ctx, ring, d["seed"])
        try:
            run(ch, other.cuda_stream)
            other.synchronize()
            assert not torch.cuda.default_stream().query(), "the default stream was not busy long enough to show anything"
            torch.cuda.synchronize()
            first = _rows(ring, stride, copies * steps, n, dtype)
            run(ch, other.cuda_stream)
            torch.cuda.synchronize()
            second = _rows(ring, stride, copies * steps, n, dtype)
            assert sf.sifar_status(ctx.h) == 0
            st = sf.sifar_get_stats(ctx.h)
        finally:
            destroy(ch)
    assert st["calls"] == st["epoch"] == 2 * steps and st["timeouts"] == 0
    want = oracle.chain(_oracle_w(oracle, d), P, n, dtype, 2 * steps)
    for t in range(2 * steps):
        for r in range(copies):
            got = (first if t < steps else second)[r * steps + t % steps]
            assert_bits_equal(got, want[t], dtype, f"{kind} n={n} mode={mode} copy {r} step {t + 1}")
