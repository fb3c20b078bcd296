"""Which speculative chains of several units per thread take them in turn: every rank count and type, on both sides of the lines
where the two kernels cross, as the kernel of the run reports it, and the results of either."""
import pytest
import torch

from paper_2607_08973_b200 import binding as sf
from paper_2607_08973_b200 import synth

from gpu_util import BF16, F32, Ctx, assert_bits_equal
from test_gpu_chains import _oracle_w, _ring, _rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,n,dtype,in_turn", [
    (1, 360_001, BF16, 0), (2, 240_001, BF16, 0), (2, 760_003, BF16, 1), (3, 210_011, BF16, 1), (4, 170_003, BF16, 1),
    (5, 140_009, BF16, 1), (6, 100_003, BF16, 1), (7, 100_003, BF16, 1), (8, 100_003, BF16, 1),
    (1, 250_007, F32, 0), (2, 160_001, F32, 0), (3, 110_017, F32, 0), (3, 180_001, F32, 1), (4, 90_001, F32, 1),
    (5, 64_001, F32, 0), (5, 67_001, F32, 1), (6, 60_013, F32, 1), (7, 60_013, F32, 1), (8, 60_013, F32, 1),
    (8, 4099, BF16, 0), (4, 70_001, BF16, 0)])          # one unit per thread
def test_units_are_taken_in_turn_where_that_is_faster(oracle, P, n, dtype, in_turn):
    steps, runs = 4, 2
    d = synth.chain_workload("sweep", P)
    with Ctx(P, n, dtype) as ctx:
        ring, stride = _ring(n, dtype, steps)
        ch = sf.sifar_chain_create(ctx.h, sf.make_workload(**d), n, sf.SPECULATIVE, sf.CHAIN_PERSISTENT, ring.data_ptr(),
                                   steps, steps)
        got = []
        try:
            assert sf.sifar_chain_in_turn(ch) is False               # nothing has run yet
            for _ in range(runs):
                sf.sifar_chain_run(ch, 0)
                torch.cuda.synchronize()
                got.append(_rows(ring, stride, steps, n, dtype))
            ran = sf.sifar_chain_in_turn(ch)
        finally:
            sf.sifar_chain_destroy(ch)
        assert sf.sifar_status(ctx.h) == 0
    assert ran is bool(in_turn)
    want = oracle.chain(_oracle_w(oracle, d), P, n, dtype, steps * runs)
    for t in range(steps * runs):
        assert_bits_equal(got[t // steps][t % steps], want[t], dtype, f"step {t + 1}")
