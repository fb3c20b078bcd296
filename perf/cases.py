"""The work that users of this library have it do, as cases that can be timed and compared.

Six paths through the public entry points (``paper_2607_08973_b200.binding``):

* ``chain``    a decode step: dependent {P producers -> all-reduce} steps with one reader, as one persistent
               kernel or as a replayed CUDA graph (``sifar_chain_run``);
* ``readers``  the same decode step with every rank reducing for itself (``sifar_symchain_run``);
* ``call``     one all-reduce of P partials: ``sifar_pack`` for every rank, then ``sifar_allreduce``, on one
               stream (a simple client) or with a stream per rank;
* ``buffers``  one all-reduce of partials that the caller's own kernels have stored: ``sifar_wait_writable`` and
               ``sifar_arrive`` for every rank, then ``sifar_allreduce`` on the caller's buffers;
* ``host``     one all-reduce from host memory to host memory (``sifar_allreduce_host``);
* ``noalloc``  one all-reduce of ready partials by a caller that must not allocate (``sifar_allreduce_noalloc``).

Sizes are those of ``synth.CONFIGS`` and of the tests: 2 KB to 64 MiB per rank for single calls, decode payloads
of 8 KB to 512 KB per rank for the chains, ragged sizes among them, bf16 and fp32, every mode.  The chain whose
producers are held back by seeded delays is left out: it times the delays.
"""
from __future__ import annotations

import torch

from paper_2607_08973_b200 import binding as sf
from paper_2607_08973_b200 import synth

_ELEM = {"bf16": 2, "f32": 4}
_TORCH = {"bf16": torch.bfloat16, "f32": torch.float32}
_DTYPE = {"bf16": sf.BF16, "f32": sf.F32}
_MODE = {"barrier": sf.BARRIER_ONESHOT, "dualbuf": sf.DUALBUF, "speculative": sf.SPECULATIVE}
_IMPL = {"graph": sf.CHAIN_GRAPH, "persistent": sf.CHAIN_PERSISTENT}
_LARGEST_BYTES = 8 << 26                # all partials of the largest listed call: 8 ranks of 64 MiB


def listed() -> list[dict]:
    return [
        # one token of the dense model's decode step at batch 1, the headline of the benchmark: 64 all-reduces of 8 KB
        {"name": "decode-8k", "path": "chain", "impl": "persistent", "workload": "llama", "P": 8, "n": 4096,
         "dtype": "bf16", "mode": "speculative", "steps": 64},
        # the same at batch 16, for a caller that keeps plain partials
        {"name": "decode-128k-dualbuf", "path": "chain", "impl": "persistent", "workload": "llama", "P": 8,
         "n": 65536, "dtype": "bf16", "mode": "dualbuf", "steps": 64},
        # the mixture-of-experts decode step at its largest batch: 120 all-reduces of 512 KB, outliers among the values
        {"name": "decode-512k-moe", "path": "chain", "impl": "persistent", "workload": "moe", "P": 8, "n": 262144,
         "dtype": "bf16", "mode": "speculative", "steps": 120},
        # an engine that replays its decode step as a CUDA graph, batch 4
        {"name": "graph-32k", "path": "chain", "impl": "graph", "workload": "llama", "P": 8, "n": 16384,
         "dtype": "bf16", "mode": "speculative", "steps": 64},
        # four ranks that each reduce for themselves, a hidden size that fills no tile
        {"name": "readers-ragged", "path": "readers", "workload": "llama", "P": 4, "n": 12291, "dtype": "bf16",
         "mode": "speculative", "steps": 64},
        # the conventional design as a baseline: both barriers, eight readers
        {"name": "readers-8k-barrier", "path": "readers", "workload": "llama", "P": 8, "n": 4096, "dtype": "bf16",
         "mode": "barrier", "steps": 64},
        # a decode-sized all-reduce by a simple client: pack the ranks one after another, reduce, all on one stream
        {"name": "call-8k", "path": "call", "streams": "one", "P": 8, "n": 4096, "dtype": "bf16",
         "mode": "speculative"},
        # a prefill chunk in fp32 on four ranks with a stream per rank, ragged
        {"name": "call-4m-f32-ragged", "path": "call", "streams": "per rank", "P": 4, "n": 1000003, "dtype": "f32",
         "mode": "dualbuf"},
        # prefill: 16 MiB per rank, a stream per rank, the reducer enqueued while they pack
        {"name": "call-16m", "path": "call", "streams": "per rank", "P": 8, "n": 8 << 20, "dtype": "bf16",
         "mode": "speculative"},
        # the largest: partials that the caller's own kernels left in its own buffers, both barriers
        {"name": "buffers-64m", "path": "buffers", "P": 8, "n": 32 << 20, "dtype": "bf16", "mode": "barrier"},
        # the end-to-end call of a host program, pinned buffers, decode payload
        {"name": "host-8k", "path": "host", "memory": "pinned", "P": 8, "n": 4096, "dtype": "bf16",
         "mode": "speculative"},
        # an engine that owns all device memory
        {"name": "noalloc-128k-ragged", "path": "noalloc", "P": 8, "n": 65549, "dtype": "bf16"},
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    """Log-uniform on [lo, hi]; half of them odd sizes, half multiples of 256 where there is room for one."""
    v = int(round(lo * (hi / lo) ** rng.random()))
    if rng.random() < 0.5 and v >= 512:
        v -= v % 256
    else:
        v |= 1
    return max(lo, min(hi, v))


def draw(rng) -> dict:
    path = rng.choice(["chain", "chain", "readers", "call", "call", "buffers", "host", "noalloc"])
    P = rng.choice([2, 4, 8, 8, rng.randint(1, 8)])
    dtype = rng.choice(["bf16", "bf16", "f32"])
    mode = rng.choice(["barrier", "dualbuf", "speculative", "speculative"])
    es = _ELEM[dtype]
    case = {"path": path, "P": P, "dtype": dtype}
    if path in ("chain", "readers"):
        top = (512 << 10) // es                       # 512 KB per rank, the largest decode payload
        case.update(workload=rng.choice(["token", "llama", "moe", "sweep"] if P == 1 else ["llama", "moe", "sweep"]),
                    n=_log_int(rng, 1024, top if path == "chain" else top // 4), mode=mode,
                    steps=rng.choice([64, 100, 120]))
        if path == "chain":
            case["impl"] = rng.choice(["persistent", "persistent", "graph"])
    elif path == "call":
        case.update(n=_log_int(rng, 1024, min(1 << 25, _LARGEST_BYTES // (3 * P * es))), mode=mode,
                    streams=rng.choice(["one", "per rank"]))
    elif path == "buffers":
        case.update(n=_log_int(rng, 1024, min(1 << 25, _LARGEST_BYTES // (P * es))), mode="barrier")
    elif path == "host":
        case.update(n=_log_int(rng, 1024, (4 << 20) // es), mode=mode,
                    memory=rng.choice(["pinned", "pinned", "pageable"]))
    else:
        case.update(n=_log_int(rng, 1024, 1 << 20))
    return case


_streams: dict = {}
_reduced: dict = {}


def _stream(name) -> torch.cuda.Stream:
    """The streams of the user's program: one for the reducer ("main"), one per rank."""
    if name not in _streams:
        _streams[name] = torch.cuda.Stream()
    return _streams[name]


def _last_reduced() -> torch.cuda.Event:
    """Recorded behind every reducer of the program: the next layer's producers consume its result."""
    if not _reduced:
        _reduced["event"] = torch.cuda.Event()
    return _reduced["event"]


class _State:
    """What the program holds between calls.  Handles are released with it."""

    def __init__(self):
        self.ctx = self.chain = 0
        self.free_chain = None

    def __del__(self):
        if self.chain:
            self.free_chain(self.chain)
        if self.ctx:
            sf.sifar_destroy(self.ctx)


def _partials(case: dict, seed: int, device: str) -> list[torch.Tensor]:
    """Partial sums of a layer: N(0, 1), one element in a hundred an outlier of a hundred times that."""
    g = torch.Generator(device=device)
    g.manual_seed(seed)
    xs = []
    for _ in range(case["P"]):
        x = torch.randn(case["n"], generator=g, device=device)
        x *= 1.0 + 99.0 * (torch.rand(case["n"], generator=g, device=device) < 0.01)
        xs.append(x.to(_TORCH[case["dtype"]]))
    return xs


def prepare(case: dict, seed: int):
    st = _State()
    path, P, n = case["path"], case["P"], case["n"]
    dtype, torch_dtype = _DTYPE[case["dtype"]], _TORCH[case["dtype"]]
    st.case, st.main = case, _stream("main").cuda_stream
    st.P, st.n, st.dtype, st.mode = P, n, dtype, _MODE.get(case.get("mode", ""), 0)
    if path in ("chain", "readers"):
        steps = case["steps"]
        rows = steps if path == "chain" else P * steps
        stride = sf.sifar_chain_ring_stride(dtype, n)
        st.ring = torch.zeros(rows, stride // _ELEM[case["dtype"]], dtype=torch_dtype, device="cuda")
        st.out = st.ring[:, :n]                           # every result of the decode step, P copies with P readers
        d = dict(synth.chain_workload(case["workload"], P), seed=seed & 0x7FFFFFFF)
        torch.cuda.synchronize()                          # the library's streams do not wait for torch's
        st.ctx = sf.sifar_create(P, n, dtype)
        if path == "chain":
            st.chain = sf.sifar_chain_create(st.ctx, sf.make_workload(**d), n, st.mode, _IMPL[case["impl"]],
                                             st.ring.data_ptr(), steps, steps)
            st.free_chain, st.run_chain = sf.sifar_chain_destroy, sf.sifar_chain_run
        else:
            st.chain = sf.sifar_symchain_create(st.ctx, sf.make_workload(**d), n, st.mode, st.ring.data_ptr(), steps,
                                                steps)
            st.free_chain, st.run_chain = sf.sifar_symchain_destroy, sf.sifar_symchain_run
        return st
    if path == "host":
        pin = (lambda t: t.pin_memory()) if case["memory"] == "pinned" else (lambda t: t)
        st.x = [pin(x.cpu()) for x in _partials(case, seed, "cuda")]
        st.out = pin(torch.empty(n, dtype=torch_dtype))
    else:
        st.x = _partials(case, seed, "cuda")
        st.out = torch.empty(n, dtype=torch_dtype, device="cuda")
    st.ptrs = [x.data_ptr() for x in st.x]
    st.out_ptr = st.out.data_ptr()
    if path != "noalloc":
        st.ctx = sf.sifar_create(P, n, dtype)
    if path in ("call", "buffers"):
        st.streams = [_stream(r) if case.get("streams") == "per rank" else _stream("main") for r in range(P)]
        st.done = _last_reduced() if case.get("streams") == "per rank" else None
    torch.cuda.synchronize()
    return st


def run(st):
    path = st.case["path"]
    if path in ("chain", "readers"):
        st.run_chain(st.chain, st.main)
    elif path == "call":
        if st.done is None:
            for r in range(st.P):
                sf.sifar_pack(st.ctx, r, st.ptrs[r], st.n, st.mode, st.main)
            sf.sifar_allreduce(st.ctx, None, st.out_ptr, st.n, st.mode, st.main)
        else:
            # the producers of this call come after the program's all-reduce before it, whose result they consume;
            # nothing orders the reducer of this call behind them but the mode's own flags or tags
            for r in range(st.P):
                st.streams[r].wait_event(st.done)
                sf.sifar_pack(st.ctx, r, st.ptrs[r], st.n, st.mode, st.streams[r].cuda_stream)
            sf.sifar_allreduce(st.ctx, None, st.out_ptr, st.n, st.mode, st.main)
            st.done.record(_stream("main"))
    elif path == "buffers":
        for r in range(st.P):
            sf.sifar_wait_writable(st.ctx, r, st.main)
            sf.sifar_arrive(st.ctx, r, st.mode, st.main)
        sf.sifar_allreduce(st.ctx, st.ptrs, st.out_ptr, st.n, st.mode, st.main)
    elif path == "host":
        sf.sifar_allreduce_host(st.ctx, st.ptrs, st.out_ptr, st.n, st.mode)
    else:
        sf.sifar_allreduce_noalloc(st.ptrs, st.out_ptr, st.n, st.dtype, st.main)
    return st.out


def work(case: dict) -> dict:
    P, n, es = case["P"], case["n"], _ELEM[case["dtype"]]
    if case["path"] in ("chain", "readers"):
        # every result is written once (by every reader); per step and element each rank scales, adds its noise
        # and is summed
        copies = P if case["path"] == "readers" else 1
        return {"bytes": copies * case["steps"] * n * es,
                "flops": case["steps"] * n * (4 * P + copies * (P - 1))}
    return {"bytes": (P + 1) * n * es, "flops": (P - 1) * n}


def tolerance(case: dict):
    """The order of the adds and the one rounding are part of the contract, so there is one right answer per bit."""
    return "exact"
