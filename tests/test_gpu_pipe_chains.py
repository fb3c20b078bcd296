"""The persistent speculative chain whose threads take several units in turn: ragged last chunks and warps, one, two and more
units per thread on either side, the hand-over from run to run, forced retries, and a wait that runs out."""
import pytest
import torch

from paper_2607_08973_b200 import binding as sf
from paper_2607_08973_b200 import synth

from gpu_util import BF16, F32, Ctx, assert_bits_equal
from test_gpu_chains import _oracle_w, _ring, _rows


def _expected_units(P, n, dtype):
    """Units per producer thread: as many chunks of 128 units per rank as six CTAs per SM hold beside a reader each."""
    units = -(-n // (6 if dtype == BF16 else 3))
    room = 6 * torch.cuda.get_device_properties(0).multi_processor_count
    k = 1
    while -(-units // (128 * k)) * (P + 1) > room:
        k += 1
    return k


@pytest.mark.gpu
@pytest.mark.parametrize("forced", [0, 2])
@pytest.mark.parametrize("P,n,dtype,workload", [
    (8, 76_801, BF16, "llama"),           # two units per thread, a last chunk of one warp
    (8, 98_304, BF16, "moe"),             # whole chunks only; outliers in the first step
    (8, 160_003, BF16, "skew"),           # integers, seeded delays before the first store of a step
    (8, 262_139, BF16, "llama"),          # four units, readers with two, sentinel polling
    (5, 100_007, F32, "sweep"),           # a scale that is no power of two
    (2, 1_000_003, BF16, "sweep")])
def test_units_taken_in_turn(oracle, P, n, dtype, workload, forced):
    steps, runs = 4, 3
    d = synth.chain_workload(workload, P)
    with Ctx(P, n, dtype) as ctx:
        sf.sifar_debug_force_retries(ctx.h, forced)
        ring, stride = _ring(n, dtype, steps)
        ch = sf.sifar_chain_create(ctx.h, sf.make_workload(**d), n, sf.SPECULATIVE, sf.CHAIN_PERSISTENT, ring.data_ptr(),
                                   steps, steps)
        got = []
        try:
            for _ in range(runs):
                sf.sifar_chain_run(ch, 0)
                torch.cuda.synchronize()
                got.append(_rows(ring, stride, steps, n, dtype))
            g = sf.sifar_chain_geometry(ch)
        finally:
            sf.sifar_chain_destroy(ch)
        assert sf.sifar_status(ctx.h) == 0
        st = sf.sifar_get_stats(ctx.h)
    assert st["calls"] == st["epoch"] == steps * runs and st["timeouts"] == 0
    if forced:
        assert st["calls_with_retry"] == steps * runs and st["slot_reloads"] >= forced * steps * runs * P * (n // 6)
    assert g["kernel_tagged"] == 1 and g["kernel_clustered"] == 0 and _expected_units(P, n, dtype) > 1
    assert 2 <= g["units_per_thread"] <= _expected_units(P, n, dtype)
    want = oracle.chain(_oracle_w(oracle, d), P, n, dtype, steps * runs)
    for t in range(steps * runs):
        assert_bits_equal(got[t // steps][t % steps], want[t], dtype, f"step {t + 1}")


@pytest.mark.gpu
@pytest.mark.parametrize("n", [98_305, 262_139])
def test_a_wait_that_runs_out_ends_the_chain(oracle, n):
    """Ranks delayed by up to 1 ms against a 50 us limit: whoever waits gives up, the kernel ends by itself, and after a
    reset the context runs the same chain without delays."""
    P, steps = 8, 4
    d = synth.chain_workload("llama", P)
    with Ctx(P, n, BF16, timeout_us=50) as ctx:
        ring, stride = _ring(n, BF16, steps)
        ch = sf.sifar_chain_create(ctx.h, sf.make_workload(**dict(d, delay_max_ns=1_000_000)), n, sf.SPECULATIVE,
                                   sf.CHAIN_PERSISTENT, ring.data_ptr(), steps, steps)
        sf.sifar_chain_run(ch, 0)
        torch.cuda.synchronize()
        assert sf.sifar_status(ctx.h) == sf.ERR_TIMEOUT
        sf.sifar_chain_destroy(ch)
        sf.sifar_reset(ctx.h, 0)
        sf.sifar_set_timeout_us(ctx.h, 2_000_000)
        ch = sf.sifar_chain_create(ctx.h, sf.make_workload(**d), n, sf.SPECULATIVE, sf.CHAIN_PERSISTENT, ring.data_ptr(),
                                   steps, steps)
        sf.sifar_chain_run(ch, 0)
        torch.cuda.synchronize()
        assert sf.sifar_status(ctx.h) == 0
        sf.sifar_chain_destroy(ch)
        want = oracle.chain(_oracle_w(oracle, d), P, n, BF16, steps)
        for t, row in enumerate(_rows(ring, stride, steps, n, BF16)):
            assert_bits_equal(row, want[t], BF16, f"step {t + 1}")
