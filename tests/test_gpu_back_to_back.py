"""Large calls enqueued back to back, a stream per rank, the reducer of the next call right behind that of the last: the
next reducer must not take the machine from producers that the last one still waits for."""
import pytest
import torch

from paper_2607_08973_b200 import binding as sf
from paper_2607_08973_b200 import synth

from gpu_util import BF16, F32, MODES, Ctx, assert_bits_equal, empty_out, out_to_numpy, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("P,n,dtype", [(2, 9_000_000, BF16), (4, 3_798_784, BF16), (3, 3_578_624, F32), (8, 200_003, F32)])
def test_calls_of_three_contexts_in_a_row_without_waiting(oracle, P, n, dtype, mode):
    streams, main, done = [torch.cuda.Stream() for _ in range(P)], torch.cuda.Stream(), torch.cuda.Event()
    xs = synth.rank_inputs(P, n, dtype, 17, "uniform")
    xd = [to_device(x) for x in xs]
    ctxs = [Ctx(P, n, dtype) for _ in range(3)]                       # 2 s limit: far more than all calls take
    outs = [empty_out(n, dtype) for _ in ctxs]
    torch.cuda.synchronize()
    try:
        for call in range(60):
            ctx, out = ctxs[call % 3], outs[call % 3]
            for r in range(P):
                streams[r].wait_event(done)
                sf.sifar_pack(ctx.h, r, xd[r].data_ptr(), n, mode, streams[r].cuda_stream)
            sf.sifar_allreduce(ctx.h, None, out.data_ptr(), n, mode, main.cuda_stream)
            done.record(main)
        torch.cuda.synchronize()
        assert [sf.sifar_status(c.h) for c in ctxs] == [0, 0, 0]
        assert [sf.sifar_get_stats(c.h)["calls"] for c in ctxs] == [20, 20, 20]
        want = oracle.allreduce(xs, dtype)
        for out in outs:
            assert_bits_equal(out_to_numpy(out, n, dtype)[0], want, dtype, f"P={P} n={n} mode={mode}")
    finally:
        for c in ctxs:
            c.__exit__()
