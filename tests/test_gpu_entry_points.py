"""Calls that need no protocol between streams: partials in host memory, caller buffers and packs on one stream, and
the allocation-free call on two streams at once."""
import os
import subprocess
import sys
import textwrap

import numpy as np
import pytest
import torch

from paper_2607_08973_b200 import binding as sf
from paper_2607_08973_b200 import synth

from gpu_util import BF16, F32, MODES, Ctx, assert_bits_equal, canary_ok, empty_out, out_to_numpy, to_device

pytestmark = pytest.mark.gpu

# elements around one 16-byte vector, one CTA (256 vectors) and the 32 KiB up to which pageable partials are bounced
EDGES = {BF16: [1, 7, 8, 9, 2047, 2048, 2049, 16383, 16384, 16385, 50_001],
         F32: [1, 3, 4, 5, 1023, 1024, 1025, 8191, 8192, 8193, 50_001]}



@pytest.mark.parametrize("memory", ["pinned", "pageable", "mixed"])
@pytest.mark.parametrize("P,dtype", [(1, F32), (3, BF16), (8, BF16), (8, F32)])
def test_host_partials_at_the_edges(oracle, P, dtype, memory):
    with Ctx(P, 50_001, dtype) as ctx:
        calls = 0
        for n in EDGES[dtype]:
            for mode in MODES:
                xs = synth.rank_inputs(P, n, dtype, 31 + n + mode, "gauss")
                hx = [torch.from_numpy(x.view(np.int16) if dtype == BF16 else x) for x in xs]
                if memory != "pageable":
                    hx = [t.pin_memory() if memory == "pinned" or r % 2 else t for r, t in enumerate(hx)]
                out = torch.zeros(n + 8, dtype=hx[0].dtype)
                out = out.pin_memory() if memory == "pinned" else out
                sf.sifar_allreduce_host(ctx.h, [t.data_ptr() for t in hx], out.data_ptr(), n, mode)
                calls += 1
                got = out.numpy().view(np.uint16) if dtype == BF16 else out.numpy()
                assert not got[n:].any(), "wrote past n"
                assert_bits_equal(got[:n], oracle.allreduce(xs, dtype), dtype, f"P={P} n={n} mode={mode} {memory}")
        st = sf.sifar_get_stats(ctx.h)
        assert st["calls"] == st["epoch"] == calls and st["timeouts"] == 0


@pytest.mark.parametrize("pinned", [False, True])
@pytest.mark.parametrize("shift", [0, 8, -8])
def test_a_host_result_may_lie_on_a_partial(oracle, pinned, shift):
    """In place of rank 1's partial, and straddling it by 16 bytes: the result is that of the values before the call."""
    P, n = 4, 20_011
    with Ctx(P, n, BF16) as ctx:
        xs = synth.rank_inputs(P, n, BF16, 5, "gauss")
        flat = torch.zeros(P * (n + 5) + 64, dtype=torch.int16)
        flat = flat.pin_memory() if pinned else flat
        base = [32 + r * 20_016 for r in range(P)]                       # 16-byte aligned rows
        for r in range(P):
            flat[base[r]: base[r] + n] = torch.from_numpy(xs[r].view(np.int16))
        at = base[1] + shift
        sf.sifar_allreduce_host(ctx.h, [flat.data_ptr() + 2 * b for b in base], flat.data_ptr() + 2 * at, n, sf.SPECULATIVE)
        assert_bits_equal(flat.numpy()[at: at + n].view(np.uint16), oracle.allreduce(xs, BF16), BF16, f"shift {shift}")


def _in_a_process_of_its_own(code, **env):
    """Loaded kernels and the switches that are read at load time belong to a process."""
    here = os.path.dirname(os.path.abspath(__file__))
    out = subprocess.run([sys.executable, "-c", textwrap.dedent(code)], capture_output=True, text=True, timeout=300,
                         cwd=os.path.dirname(here),
                         env=dict(os.environ, PYTHONPATH=os.pathsep.join([os.path.dirname(here), here]), **env))
    assert out.returncode == 0, out.stdout + out.stderr
    return out.stdout


@pytest.mark.parametrize("mode", MODES)
def test_the_first_host_call_beside_a_reducer_that_waits_for_a_late_rank(mode):
    """The process's first host call is made while another context's reducer polls for a rank whose store the same thread
    launches afterwards: it may not wait for the device to become idle (its kernel is loaded with the context)."""
    _in_a_process_of_its_own(f"""
        import time
        import torch
        from paper_2607_08973_b200 import binding as sf
        n = 4096
        sf.sifar_workload_preload()
        waiting, host = sf.sifar_create(2, n, sf.BF16), sf.sifar_create(3, n, sf.F32)
        sf.sifar_set_timeout_us(waiting, 2_000_000)
        x = [torch.ones(n, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        out = torch.zeros(n, dtype=torch.bfloat16, device="cuda")
        hx = [torch.full((n,), float(r + 1)).pin_memory() for r in range(3)]
        hout = torch.zeros(n).pin_memory()
        ranks, red = [torch.cuda.Stream() for _ in range(2)], torch.cuda.Stream()
        torch.cuda.synchronize()
        sf.sifar_pack(waiting, 0, x[0].data_ptr(), n, sf.SPECULATIVE, ranks[0].cuda_stream)
        late, epoch = sf.sifar_rank_buffer(waiting, 1, sf.SPECULATIVE)
        sf.sifar_allreduce(waiting, None, out.data_ptr(), n, sf.SPECULATIVE, red.cuda_stream)
        t0 = time.perf_counter()
        sf.sifar_allreduce_host(host, [t.data_ptr() for t in hx], hout.data_ptr(), n, {mode})
        assert time.perf_counter() - t0 < 1.0, "the call waited for the reducer's time limit"
        sf.sifar_store_slots(x[1].data_ptr(), late, 0, sf.sifar_slot_count(sf.BF16, n), n, sf.BF16, epoch, ranks[1].cuda_stream)
        torch.cuda.synchronize()
        assert sf.sifar_status(waiting) == 0 and sf.sifar_get_stats(waiting)["timeouts"] == 0
        assert bool((out == 2).all()) and bool((hout == 6).all())
        """, CUDA_DEVICE_MAX_CONNECTIONS="32")                    # no two of the streams in one hardware queue


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("P,dtype", [(1, BF16), (8, BF16), (5, F32)])
def test_packs_and_reducer_on_one_stream(oracle, P, dtype, mode):
    """Each small pack may become resident while the one before it runs; its inputs come from the stream as well."""
    sizes = [1, 5, 6, 7, 8, 9, 1535, 1536, 1537, 2048, 2049, 65_549, 300_007]
    with Ctx(P, max(sizes), dtype) as ctx:
        s = torch.cuda.Stream()
        for n in sizes:
            for rep in range(3):                                          # calls back to back, without waiting
                xs = synth.rank_inputs(P, n, dtype, 7 * rep + n, "gauss")
                hx = [torch.from_numpy(x.view(np.int16) if dtype == BF16 else x).pin_memory() for x in xs]
                out = empty_out(n, dtype)
                torch.cuda.synchronize()
                with torch.cuda.stream(s):
                    for r in range(P):
                        xd = hx[r].to("cuda", non_blocking=True)
                        sf.sifar_pack(ctx.h, r, xd.data_ptr(), n, mode, s.cuda_stream)
                    sf.sifar_allreduce(ctx.h, None, out.data_ptr(), n, mode, s.cuda_stream)
                    again = empty_out(n, dtype)
                    for r in range(P):
                        sf.sifar_pack(ctx.h, r, out.data_ptr(), n, mode, s.cuda_stream)
                    sf.sifar_allreduce(ctx.h, None, again.data_ptr(), n, mode, s.cuda_stream)
                torch.cuda.synchronize()
                assert sf.sifar_status(ctx.h) == 0
                got, tail = out_to_numpy(out, n, dtype)
                want = oracle.allreduce(xs, dtype)
                assert canary_ok(tail, dtype)
                assert_bits_equal(got, want, dtype, f"P={P} n={n} mode={mode}")
                assert_bits_equal(out_to_numpy(again, n, dtype)[0], oracle.allreduce([want] * P, dtype), dtype, "second call")


@pytest.mark.parametrize("other_stream", [False, True])
def test_caller_buffers_on_one_stream_and_across_streams(oracle, other_stream):
    """sifar_wait_writable behind a reducer of the same stream, and on a stream that has to wait for it."""
    P, n = 8, 40_003
    with Ctx(P, n, BF16) as ctx:
        s, q = torch.cuda.Stream(), torch.cuda.Stream()
        bufs = [torch.zeros(n + 8, dtype=torch.int16, device="cuda") for _ in range(P)]
        outs, wants = [], []
        done = torch.cuda.Event()
        torch.cuda.synchronize()
        for call in range(4):
            xs = synth.rank_inputs(P, n, BF16, 60 + call, "gauss")
            w = q if (other_stream and call % 2) else s
            w.wait_event(done)
            xd = [torch.from_numpy(x.view(np.int16)).pin_memory() for x in xs]
            with torch.cuda.stream(w):
                for r in range(P):
                    sf.sifar_wait_writable(ctx.h, r, w.cuda_stream)
                    bufs[r][:n].copy_(xd[r], non_blocking=True)
                    sf.sifar_arrive(ctx.h, r, sf.BARRIER_ONESHOT, w.cuda_stream)
            out = empty_out(n, BF16)
            s.wait_stream(torch.cuda.current_stream())
            sf.sifar_allreduce(ctx.h, [b.data_ptr() for b in bufs], out.data_ptr(), n, sf.BARRIER_ONESHOT, s.cuda_stream)
            done.record(s)
            outs.append(out)
            wants.append((xd, oracle.allreduce(xs, BF16)))
        torch.cuda.synchronize()
        assert sf.sifar_status(ctx.h) == 0
        for call in range(4):
            got, tail = out_to_numpy(outs[call], n, BF16)
            assert canary_ok(tail, BF16)
            assert_bits_equal(got, wants[call][1], BF16, f"call {call}")


def test_noalloc_calls_on_two_streams_are_both_booked(oracle):
    P, n = 8, 1 << 20
    xs = synth.rank_inputs(P, n, BF16, 3, "gauss")
    xd = [to_device(x) for x in xs]
    want = oracle.allreduce(xs, BF16)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    outs = [empty_out(n, BF16) for _ in range(2)]
    torch.cuda.synchronize()
    before = sf.sifar_noalloc_counters()["calls"]
    for _ in range(20):
        for s, out in zip(streams, outs):
            sf.sifar_allreduce_noalloc([x.data_ptr() for x in xd], out.data_ptr(), n, BF16, s.cuda_stream)
    torch.cuda.synchronize()
    now = sf.sifar_noalloc_counters()
    assert (now["calls"], now["elements"]) == (before + 40, n)
    for out in outs:
        assert_bits_equal(out_to_numpy(out, n, BF16)[0], want, BF16, "two streams")


@pytest.mark.parametrize("n,mode,policy", [(4096, sf.SPECULATIVE, None), (262_144, sf.SPECULATIVE, None),
                                           (1 << 20, sf.SPECULATIVE, None), (1 << 20, sf.DUALBUF, None)] +
                         [(4 << 20, mode, sf.SWEEP_NEVER) for mode in MODES] +
                         [(4 << 20, mode, sf.SWEEP_ALWAYS) for mode in MODES])
def test_producer_streams_may_go_once_their_packs_are_enqueued(oracle, n, mode, policy):
    """Slots, block flags below 8 tiles per SM, and any size where the policy says that the streams are not asked."""
    from cuda.bindings import runtime as rt
    P = 8
    xs = synth.rank_inputs(P, n, BF16, 77, "gauss")
    xd, out = [to_device(x) for x in xs], empty_out(n, BF16)
    red = torch.cuda.Stream()
    with Ctx(P, n, BF16) as ctx:
        if policy is not None:
            sf.sifar_debug_sweep_policy(ctx.h, policy)
        torch.cuda.synchronize()
        for _ in range(2):
            for r in range(P):
                err, s = rt.cudaStreamCreateWithFlags(rt.cudaStreamNonBlocking)
                assert err == rt.cudaError_t.cudaSuccess
                sf.sifar_pack(ctx.h, r, xd[r].data_ptr(), n, mode, int(s))
                assert rt.cudaStreamDestroy(s)[0] == rt.cudaError_t.cudaSuccess       # its work goes on
            sf.sifar_allreduce(ctx.h, None, out.data_ptr(), n, mode, red.cuda_stream)
            torch.cuda.synchronize()
            assert sf.sifar_status(ctx.h) == 0
            assert_bits_equal(out_to_numpy(out, n, BF16)[0], oracle.allreduce(xs, BF16), BF16, f"n={n} mode={mode}")


@pytest.mark.parametrize("entry", ["noalloc", "pack", "arrive"])
def test_a_launch_that_cuda_refuses_leaves_no_error_for_the_next_call(oracle, entry):
    """The legacy stream may not be used while a blocking stream is being captured.  The call reports that, once."""
    from cuda.bindings import runtime as rt
    n = 4096
    xs = synth.rank_inputs(1, n, BF16, 3, "gauss")
    x, out = to_device(xs[0]), empty_out(n, BF16)
    sf.sifar_allreduce_noalloc([x.data_ptr()], out.data_ptr(), n, BF16, 0)            # resolves its array
    s = torch.cuda.Stream()
    err, capturing = rt.cudaStreamCreate()
    assert err == rt.cudaError_t.cudaSuccess
    with Ctx(1, n, BF16) as ctx:
        torch.cuda.synchronize()
        assert rt.cudaStreamBeginCapture(capturing, rt.cudaStreamCaptureMode.cudaStreamCaptureModeRelaxed)[0] == 0
        try:
            with pytest.raises(sf.SifarError) as ei:
                if entry == "noalloc":
                    sf.sifar_allreduce_noalloc([x.data_ptr()], out.data_ptr(), n, BF16, 0)
                elif entry == "pack":
                    sf.sifar_pack(ctx.h, 0, x.data_ptr(), n, sf.SPECULATIVE, 0)
                else:
                    sf.sifar_arrive(ctx.h, 0, sf.DUALBUF, 0)
            assert ei.value.code == sf.ERR_CUDA
        finally:
            rt.cudaStreamEndCapture(capturing)                                        # invalidated by then
            rt.cudaStreamDestroy(capturing)
        sf.sifar_allreduce(ctx.h, None, out.data_ptr(), 0, sf.SPECULATIVE, s.cuda_stream)      # nothing to add: a plain launch
        sf.sifar_pack(ctx.h, 0, x.data_ptr(), n, sf.SPECULATIVE, s.cuda_stream)
        sf.sifar_allreduce(ctx.h, None, out.data_ptr(), n, sf.SPECULATIVE, s.cuda_stream)
        torch.cuda.synchronize()
        assert sf.sifar_status(ctx.h) == 0
        assert_bits_equal(out_to_numpy(out, n, BF16)[0], xs[0], BF16, entry)


@pytest.mark.parametrize("pdl", ["1", "0"])
@pytest.mark.parametrize("entry", ["noalloc", "packs", "arrivals"])
def test_dependent_launches_follow_the_switch(entry, pdl):
    """A captured row of launches shows how each was launched: a programmatic edge to the kernel before it, or a full
    one.  With SIFAR_PDL=0 the plain stream order is back in all of them."""
    out = _in_a_process_of_its_own(f"""
        import ctypes
        import torch
        from cuda.bindings import runtime as rt
        from paper_2607_08973_b200 import binding as sf
        P, n, entry = 4, 4096, "{entry}"
        x = [torch.ones(n, dtype=torch.bfloat16, device="cuda") for _ in range(P)]
        out = torch.zeros(n, dtype=torch.bfloat16, device="cuda")
        ptrs, s = [t.data_ptr() for t in x], torch.cuda.Stream().cuda_stream
        ctx = sf.sifar_create(P, n, sf.BF16)
        sf.sifar_allreduce_noalloc(ptrs, out.data_ptr(), n, sf.BF16, s)
        torch.cuda.synchronize()
        assert rt.cudaStreamBeginCapture(s, rt.cudaStreamCaptureMode.cudaStreamCaptureModeRelaxed)[0] == 0
        if entry == "noalloc":
            for _ in range(3):
                sf.sifar_allreduce_noalloc(ptrs, out.data_ptr(), n, sf.BF16, s)
        else:
            for call in range(2):
                for r in range(P):
                    if entry == "packs":
                        sf.sifar_pack(ctx, r, ptrs[r], n, sf.SPECULATIVE, s)
                    else:
                        sf.sifar_wait_writable(ctx, r, s)
                        sf.sifar_arrive(ctx, r, sf.BARRIER_ONESHOT, s)
                sf.sifar_allreduce(ctx, ptrs if entry == "arrivals" else None, out.data_ptr(), n,
                                   sf.BARRIER_ONESHOT if entry == "arrivals" else sf.SPECULATIVE, s)
        err, graph = rt.cudaStreamEndCapture(s)
        assert err == 0
        k = ctypes.c_size_t(64)
        ends, data = [(ctypes.c_void_p * 64)() for _ in range(2)], (ctypes.c_uint8 * 8 * 64)()
        assert ctypes.CDLL("libcudart.so.12").cudaGraphGetEdges_v2(ctypes.c_void_p(int(graph)), *ends, data, ctypes.byref(k)) == 0
        kinds = [d[2] for d in data[:k.value]]                    # from port, to port, type
        err, ex = rt.cudaGraphInstantiate(graph, 0)
        assert err == 0
        for _ in range(3):                                        # the call number advances on the device
            out.zero_()
            torch.cuda.synchronize()
            assert rt.cudaGraphLaunch(ex, s)[0] == 0
            torch.cuda.synchronize()
            assert bool((out == P).all()) and sf.sifar_status(ctx) == 0
        rt.cudaGraphExecDestroy(ex)
        print(len(kinds), sum(k == int(rt.cudaGraphDependencyType.cudaGraphDependencyTypeProgrammatic) for k in kinds))
        """, SIFAR_PDL=pdl)
    edges, programmatic = map(int, out.split()[-2:])
    assert edges > 0 and programmatic == (edges if pdl == "1" else 0)


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("dtype", [BF16, F32])
def test_packs_around_the_size_from_which_threads_take_several_units(oracle, dtype, mode):
    """Two CTAs of 256 threads per SM: up to there a thread has one unit, whose words travel ahead of the call number."""
    P, threads = 2, 2 * 256 * torch.cuda.get_device_properties(0).multi_processor_count
    per_unit = (3 if mode == sf.SPECULATIVE else 4) * (2 if dtype == BF16 else 1)
    edge = threads * per_unit
    sizes = [edge - per_unit, edge - 1, edge, edge + 1, edge + per_unit, edge + per_unit * 256 + 1]
    assert sf.sifar_spec_format(P, dtype, max(sizes)) == sf.FORMAT_SLOTS
    s = torch.cuda.Stream()
    with Ctx(P, max(sizes), dtype) as ctx:
        for n in sizes:
            xs = synth.rank_inputs(P, n, dtype, 11 + n % 97, "gauss")
            xd, out = [to_device(x) for x in xs], empty_out(n, dtype)
            torch.cuda.synchronize()
            for r in range(P):
                sf.sifar_pack(ctx.h, r, xd[r].data_ptr(), n, mode, s.cuda_stream)
            sf.sifar_allreduce(ctx.h, None, out.data_ptr(), n, mode, s.cuda_stream)
            torch.cuda.synchronize()
            assert sf.sifar_status(ctx.h) == 0
            got, tail = out_to_numpy(out, n, dtype)
            assert canary_ok(tail, dtype)
            assert_bits_equal(got, oracle.allreduce(xs, dtype), dtype, f"n={n} mode={mode}")
