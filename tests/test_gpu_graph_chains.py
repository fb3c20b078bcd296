"""The graph chain whose kernels wait for tagged words only: one slot to several per thread, ragged sizes, the hand-over from
replay to replay, seeded delays, forced retries, and a wait that runs out."""
import pytest
import torch

from paper_2607_08973_b200 import binding as sf
from paper_2607_08973_b200 import synth

from gpu_util import BF16, F32, Ctx, assert_bits_equal
from test_gpu_chains import _oracle_w, _ring, _rows

pytestmark = pytest.mark.gpu


def _run(ctx, d, n, dtype, steps, runs):
    ring, stride = _ring(n, dtype, steps)
    ch = sf.sifar_chain_create(ctx.h, sf.make_workload(**d), n, sf.SPECULATIVE, sf.CHAIN_GRAPH, ring.data_ptr(), steps, steps)
    got = []
    try:
        for _ in range(runs):
            sf.sifar_chain_run(ch, 0)
            torch.cuda.synchronize()
            got.append(_rows(ring, stride, steps, n, dtype))
    finally:
        sf.sifar_chain_destroy(ch)
    return got


@pytest.mark.parametrize("forced", [0, 1])
@pytest.mark.parametrize("P,n,dtype,workload", [
    (8, 1, BF16, "llama"), (8, 767, BF16, "moe"), (3, 769, F32, "sweep"), (8, 4099, BF16, "skew"),
    (8, 73_727, BF16, "llama"),           # the largest reducer grid that is left unordered
    (2, 250_007, BF16, "sweep"),          # more slots than the producers have threads
    (1, 100_003, F32, "token")])
def test_replays_of_a_chain_in_tagged_words(oracle, P, n, dtype, workload, forced):
    steps, runs = 6, 3
    d = synth.chain_workload(workload, P)
    with Ctx(P, n, dtype) as ctx:
        sf.sifar_debug_force_retries(ctx.h, forced)
        got = _run(ctx, d, n, dtype, steps, runs)
        assert sf.sifar_status(ctx.h) == 0
        st = sf.sifar_get_stats(ctx.h)
    assert st["calls"] == st["epoch"] == steps * runs and st["timeouts"] == 0
    want = oracle.chain(_oracle_w(oracle, d), P, n, dtype, steps * runs)
    for t in range(steps * runs):
        assert_bits_equal(got[t // steps][t % steps], want[t], dtype, f"step {t + 1}")


def test_replays_back_to_back_and_then_a_single_call(oracle):
    """Twenty replays enqueued without waiting, then an ordinary call on the same context."""
    P, n, steps = 8, 4096, 8
    d = synth.chain_workload("llama", P)
    with Ctx(P, n, BF16) as ctx:
        ring, stride = _ring(n, BF16, steps)
        ch = sf.sifar_chain_create(ctx.h, sf.make_workload(**d), n, sf.SPECULATIVE, sf.CHAIN_GRAPH, ring.data_ptr(), steps, steps)
        for _ in range(20):
            sf.sifar_chain_run(ch, 0)
        torch.cuda.synchronize()
        got = _rows(ring, stride, steps, n, BF16)
        sf.sifar_chain_destroy(ch)
        want = oracle.chain(_oracle_w(oracle, d), P, n, BF16, 20 * steps)
        for t in range(steps):
            assert_bits_equal(got[t], want[19 * steps + t], BF16, f"step {19 * steps + t + 1}")
        x = [torch.full((n,), 1.0, dtype=torch.bfloat16, device="cuda") for _ in range(P)]
        out = torch.zeros(n, dtype=torch.bfloat16, device="cuda")
        torch.cuda.synchronize()
        for r in range(P):
            sf.sifar_pack(ctx.h, r, x[r].data_ptr(), n, sf.SPECULATIVE, 0)
        sf.sifar_allreduce(ctx.h, None, out.data_ptr(), n, sf.SPECULATIVE, 0)
        torch.cuda.synchronize()
        assert sf.sifar_status(ctx.h) == 0 and bool((out == P).all())


def test_a_wait_that_runs_out_ends_the_replay(oracle):
    """Ranks delayed by up to 1 ms against a 50 us limit: the kernels end by themselves, and after a reset the context runs
    the same chain without delays."""
    P, n, steps = 8, 4096, 8
    d = synth.chain_workload("llama", P)
    with Ctx(P, n, BF16, timeout_us=50) as ctx:
        _run(ctx, dict(d, delay_max_ns=1_000_000), n, BF16, steps, 1)
        assert sf.sifar_status(ctx.h) == sf.ERR_TIMEOUT
        sf.sifar_reset(ctx.h, 0)
        sf.sifar_set_timeout_us(ctx.h, 2_000_000)
        got = _run(ctx, d, n, BF16, steps, 1)[0]
        assert sf.sifar_status(ctx.h) == 0
    want = oracle.chain(_oracle_w(oracle, d), P, n, BF16, steps)
    for t in range(steps):
        assert_bits_equal(got[t], want[t], BF16, f"step {t + 1}")
