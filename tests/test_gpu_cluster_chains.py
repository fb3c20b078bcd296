"""The persistent chains whose ranks meet in a cluster's shared memory: edges of warps and chunks, one rank to eight,
the hand-over from run to run, and the same results as the kernels that spread a chunk over the machine."""
import numpy as np
import pytest
import torch

from paper_2607_08973_b200 import binding as sf
from paper_2607_08973_b200 import synth

from gpu_util import BF16, F32, MODES, Ctx, assert_bits_equal
from test_gpu_chains import _oracle_w, _ring, _rows, run_chain
from test_gpu_symmetric import run_sym

pytestmark = pytest.mark.gpu

# one element; a warp of 12-byte units and of 16-byte vectors, and one element on either side; a chunk of either
EDGES = [1, 191, 192, 193, 255, 256, 257, 767, 768, 769, 1023, 1024, 1025, 3 * 1024 + 5]


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("P,dtype", [(1, BF16), (2, F32), (5, BF16), (8, BF16), (8, F32)])
def test_one_reader_at_the_edges_of_warps_and_chunks(oracle, P, dtype, mode):
    d = synth.chain_workload("moe", P)
    steps, runs = 4, 3                                # three runs: both ways a result crosses from step to step
    for n in EDGES:
        got, st = run_chain(P, n, dtype, d, mode, sf.CHAIN_PERSISTENT, steps, runs=runs)
        want = oracle.chain(_oracle_w(oracle, d), P, n, dtype, steps * runs)
        for t in range(steps * runs):
            assert_bits_equal(got[t], want[t], dtype, f"P={P} n={n} mode={mode} step {t + 1}")
        assert st["calls"] == st["epoch"] == steps * runs and st["timeouts"] == 0


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("P,dtype", [(1, F32), (3, BF16), (8, BF16)])
def test_every_reader_at_the_edges_of_warps_and_chunks(oracle, P, dtype, mode):
    d = synth.chain_workload("sweep", P)
    steps, runs = 4, 3
    for n in EDGES:
        got, _, _, _, st = run_sym(P, n, dtype, d, mode, steps, runs=runs)
        want = oracle.chain(_oracle_w(oracle, d), P, n, dtype, steps * runs)
        for r in range(P):
            for t in range(steps * runs):
                assert_bits_equal(got[r, t], want[t], dtype, f"P={P} n={n} mode={mode} rank {r} step {t + 1}")
        assert st["calls"] == steps * runs and st["timeouts"] == 0


@pytest.mark.parametrize("mode", MODES)
def test_clusters_and_spread_chunks_agree_up_to_the_size_where_clusters_end(monkeypatch, mode):
    """P = 8: the largest bf16 payload below the limit, and the first above it, in both layouts."""
    P, steps = 8, 6
    d = synth.chain_workload("llama", P)
    per_unit, pairs = (6, 50_000) if mode == sf.SPECULATIVE else (8, 65_000)
    for n, clustered in ((pairs // P * per_unit, 1), (pairs // P * per_unit + 1, 0)):
        results = []
        for env in ("1", "0"):
            monkeypatch.setenv("SIFAR_CHAIN_CLUSTER", env)
            with Ctx(P, n, BF16) as ctx:
                ring, stride = _ring(n, BF16, steps)
                ch = sf.sifar_chain_create(ctx.h, sf.make_workload(**d), n, mode, sf.CHAIN_PERSISTENT, ring.data_ptr(),
                                           steps, steps)
                sf.sifar_chain_run(ch, 0)
                torch.cuda.synchronize()
                assert sf.sifar_status(ctx.h) == 0
                assert sf.sifar_chain_geometry(ch)["kernel_clustered"] == (clustered if env == "1" else 0)
                sf.sifar_chain_destroy(ch)
                results.append(_rows(ring, stride, steps, n, BF16))
        assert np.array_equal(results[0], results[1])


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("readers", ["one", "all"])
@pytest.mark.parametrize("P,n", [(8, 4096), (8, 1025), (3, 2049), (2, 70)])
def test_a_cluster_that_gives_up_waits_for_the_stores_on_their_way(oracle, P, n, mode, readers):
    """Ranks delayed by up to 1 ms against a 50 us limit, so warps give up with stores of others still to come.  Every
    CTA waits for what comes to it and for no more: had one of those waits run out it would be counted as a second
    time-out.  The context then runs the same chain without delays."""
    steps = 8
    create, run, destroy = ((sf.sifar_chain_create, sf.sifar_chain_run, sf.sifar_chain_destroy) if readers == "one" else
                            (sf.sifar_symchain_create, sf.sifar_symchain_run, sf.sifar_symchain_destroy))
    impl = (sf.CHAIN_PERSISTENT,) if readers == "one" else ()
    d = synth.chain_workload("llama", P)
    copies = 1 if readers == "one" else P
    with Ctx(P, n, BF16) as ctx:
        for seed in range(4):
            late = dict(d, seed=100 + seed, delay_max_ns=1_000_000)
            sf.sifar_set_timeout_us(ctx.h, 50)
            rings, stride = _ring(n, BF16, copies * steps)
            ch = create(ctx.h, sf.make_workload(**late), n, mode, *impl, rings.data_ptr(), steps, steps)
            run(ch, 0)
            torch.cuda.synchronize()
            assert sf.sifar_status(ctx.h) == sf.ERR_TIMEOUT
            assert sf.sifar_get_stats(ctx.h)["timeouts"] == 1
            destroy(ch)
            sf.sifar_reset(ctx.h, 0)
        sf.sifar_set_timeout_us(ctx.h, 2_000_000)
        ch = create(ctx.h, sf.make_workload(**d), n, mode, *impl, rings.data_ptr(), steps, steps)
        run(ch, 0)
        torch.cuda.synchronize()
        assert sf.sifar_status(ctx.h) == 0
        destroy(ch)
        want = oracle.chain(_oracle_w(oracle, d), P, n, BF16, steps)
        got = _rows(rings, stride, copies * steps, n, BF16)
        for i in range(copies * steps):
            assert_bits_equal(got[i], want[i % steps], BF16, f"row {i}")


@pytest.mark.parametrize("P,dtype,pairs", [(8, BF16, 25_000), (8, F32, 25_000), (7, BF16, 40_000), (7, F32, 40_000), (8, F32, 49_000)])
def test_speculative_chunks_meet_in_shared_memory_or_through_the_l2(monkeypatch, P, dtype, pairs):
    """Seven and eight ranks: the largest payload whose chunks meet in shared memory and the first whose clusters are there
    for placement only, against chunks spread over the machine; the results of two runs, the second from the first."""
    steps = 6
    d = synth.chain_workload("moe", P)
    per_unit = 6 if dtype == BF16 else 3
    for n in (pairs // P * per_unit, pairs // P * per_unit + 1):
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
                assert (g["clustered"], g["kernel_clustered"]) == ((1, 1) if env == "1" else (0, 0))
                sf.sifar_chain_destroy(ch)
                results.append(_rows(ring, stride, steps, n, dtype))
        assert results[0][-1].any() and np.array_equal(results[0].view(np.uint8), results[1].view(np.uint8))


@pytest.mark.parametrize("P,n,dtype,mode", [
    (8, 65_537, BF16, sf.DUALBUF), (8, 73_729, BF16, sf.BARRIER_ONESHOT), (7, 78_001, BF16, sf.DUALBUF),
    (4, 131_072, BF16, sf.BARRIER_ONESHOT), (2, 131_071, F32, sf.DUALBUF), (4, 131_069, BF16, sf.SPECULATIVE),
    (4, 66_001, F32, sf.SPECULATIVE), (6, 84_001, BF16, sf.SPECULATIVE), (5, 44_999, F32, sf.SPECULATIVE)])
def test_the_largest_grids_in_clusters_agree_with_spread_ones(monkeypatch, P, n, dtype, mode):
    """Grids that nearly fill the machine with clusters, whole and ragged last chunks: two runs, the second from the first."""
    steps = 6
    d = synth.chain_workload("moe", P)
    results = []
    for env in ("1", "0"):
        monkeypatch.setenv("SIFAR_CHAIN_CLUSTER", env)
        with Ctx(P, n, dtype) as ctx:
            ring, stride = _ring(n, dtype, steps)
            ch = sf.sifar_chain_create(ctx.h, sf.make_workload(**d), n, mode, sf.CHAIN_PERSISTENT, ring.data_ptr(), steps, steps)
            for _ in range(2):
                sf.sifar_chain_run(ch, 0)
            torch.cuda.synchronize()
            assert sf.sifar_status(ctx.h) == 0
            g = sf.sifar_chain_geometry(ch)
            assert g["kernel_clustered"] == int(env) and g["units_per_thread"] >= 1
            sf.sifar_chain_destroy(ch)
            results.append(_rows(ring, stride, steps, n, dtype))
    assert results[0][-1].any() and np.array_equal(results[0].view(np.uint8), results[1].view(np.uint8))


@pytest.mark.parametrize("P,n,dtype,mode", [
    (8, 65_537, BF16, sf.DUALBUF), (8, 73_729, BF16, sf.BARRIER_ONESHOT), (4, 131_072, BF16, sf.BARRIER_ONESHOT),
    (2, 131_071, F32, sf.DUALBUF), (6, 84_001, BF16, sf.SPECULATIVE), (5, 36_864, F32, sf.DUALBUF)])
def test_all_clusters_of_a_grid_run_at_once(P, n, dtype, mode):
    """Grids near the largest that go in clusters, placed by load and not: every chunk has started before any has ended."""
    steps = 64
    d = synth.chain_workload("llama", P)
    with Ctx(P, n, dtype) as ctx:
        ring, _ = _ring(n, dtype, steps)
        ch = sf.sifar_chain_create(ctx.h, sf.make_workload(**d), n, mode, sf.CHAIN_PERSISTENT, ring.data_ptr(), steps, steps)
        try:
            for _ in range(2):
                sf.sifar_chain_run(ch, 0)
                torch.cuda.synchronize()
            stamps = [sf.sifar_chain_chunk_stamps(ch, c, steps) for c in range(sf.sifar_chain_chunks(ch))]
            assert sf.sifar_chain_geometry(ch)["kernel_clustered"] == 1
        finally:
            sf.sifar_chain_destroy(ch)
        assert sf.sifar_status(ctx.h) == 0
    assert len(stamps) > 1 and max(s[0] for s in stamps) < min(s[-1] for s in stamps)
