"""The work a user of this library has it do, as cases that can be timed.

A case is one pass over collectives of P virtual ranks through the public
entry points: ``hiccl.Comm`` (compose, init, start, wait, group) and
``collectives``.  Communicators are persistent, as the paper's are: a program
composes and initializes them once over buffers it keeps, fills the send
buffers and starts them again and again.  Four forms of use:

* ``start``   one collective, started and waited for from the host;
* ``graph``   several starts, each on a stream of its own, captured once in a
              CUDA graph and replayed (a training or inference step);
* ``group``   many small and middle-sized collectives as one grouped
              communicator, started and waited for;
* ``request`` a shape that has not been seen before: compose, init, start,
              wait and destroy (what a service does for a new request).

Sizes, hierarchies, stripes and pipeline depths are those of the
configurations, the benchmark and the tests of this repository, or round
numbers; ``d`` is the chunk length in elements (a rank's largest buffer holds
``d * P``), and odd values of it give rows and chunks that no 16-byte
boundary meets.
"""
from __future__ import annotations

import torch

import synth
from paper_2408_05962_gb300 import collectives as C
from paper_2408_05962_gb300 import hiccl as H

_TORCH = {"f32": torch.float32, "i32": torch.int32, "bf16": torch.bfloat16, "fp8": torch.uint8}
_REDUCING = ("reduce", "reducescatter", "allreduce", "allreduce_via_bcast_reduce")
_SEVEN = "broadcast,scatter,gather,allgather,reducescatter,allreduce,alltoall"


def _case(form, kinds, P, h, s, m, d, dtype="f32", op="sum", ring=1, root=0, name=None):
    c = {"form": form, "kinds": kinds, "P": P, "h": "x".join(map(str, h)), "s": s, "m": m, "d": d, "dtype": dtype,
         "op": op, "ring": ring, "root": root}
    return {"name": name, **c} if name else c


def _mix(n, mix_seed, min_bytes, max_bytes, name=None):
    c = {"form": "group", "n": n, "mix_seed": mix_seed, "min_bytes": min_bytes, "max_bytes": max_bytes}
    return {"name": name, **c} if name else c


def _elems(nbytes, P, dtype):
    """Chunk length of a per-rank buffer of ``nbytes`` in whole 16-byte (FP8: block) chunks."""
    if dtype == "fp8":
        return max(1, nbytes // P // 128) * 128            # bytes of values, before the scales
    e = H.ESIZE[H.DTYPES[dtype]]
    return max(16, nbytes // P // 16 * 16) // e


def listed():
    return [
        # the smallest call: a few parameters or a control block to eight ranks
        _case("start", "broadcast", 8, (2, 4), 1, 1, _elems(16 << 10, 8, "f32"), name="bcast_16k"),
        # one token's activations summed over a tensor-parallel group while decoding, inside a captured step
        _case("graph", "allreduce", 8, (2, 4), 1, 1, _elems(64 << 10, 8, "bf16"), "bf16", name="decode_allreduce"),
        # sharded training: a layer's parameters gathered and its gradients scattered, in BF16
        _case("graph", "allgather,reducescatter", 16, (4, 4), 4, 2, _elems(16 << 20, 16, "bf16"), "bf16",
              name="shard_layer_bf16"),
        # the benchmark's step: seven collectives of 64 ranks, 4 MiB per rank
        _case("graph", _SEVEN, 64, (4, 4, 4), 4, 8, _elems(4 << 20, 64, "f32"), name="seven_p64"),
        # data-parallel gradients, 64 MiB per rank (the largest case)
        _case("start", "allreduce", 32, (4, 8), 1, 4, 1 << 19, name="grads_f32_64m"),
        # the same gradients (as many values) as block-scaled FP8
        _case("start", "allreduce", 32, (4, 8), 1, 4, 1 << 19, "fp8", name="grads_fp8"),
        # gradients of a parameter list whose length nothing divides: every row and chunk lies off 16 bytes
        _case("start", "allreduce", 16, (4, 4), 4, 2, 98_311, name="grads_ragged"),
        # expert dispatch: every rank sends every other one an odd number of BF16 values
        _case("start", "alltoall", 64, (4, 4, 4), 4, 1, 8_203, "bf16", name="dispatch_ragged"),
        # per-row maxima of counters over a machine without levels (one 64-way fold)
        _case("start", "reduce", 64, (64,), 1, 1, _elems(1 << 20, 64, "i32"), "i32", "max", name="counters_max"),
        # parameter server: reduce to one rank, then broadcast, nodes chained as a ring
        _case("start", "allreduce_via_bcast_reduce", 16, (4, 4), 4, 4, _elems(8 << 20, 16, "f32"), ring=4,
              name="server_ring"),
        # a bucketed step: many collectives of mixed kinds, sizes and payloads in one launch
        _mix(48, 0, 4 << 10, 16 << 20, name="buckets"),
        # a request of a new shape, planned, run and dropped
        _case("request", "allreduce", 16, (4, 4), 1, 1, _elems(1 << 20, 16, "bf16"), "bf16", name="new_request"),
    ]


_HIER = {8: [(2, 4), (4, 2), (2, 2, 2), (8,)], 12: [(2, 2, 3), (3, 4)], 16: [(4, 4), (2, 8), (16,)],
         32: [(4, 8), (8, 4), (2, 4, 4)], 64: [(4, 4, 4), (8, 8), (64,)]}


def _log(rng, lo, hi):
    return int(lo * (hi / lo) ** rng.random())


def draw(rng):
    form = rng.choice(["start", "start", "start", "graph", "group", "request"])
    if form == "group":
        return _mix(rng.randint(8, 60), rng.randint(1, 1 << 20), 4 << 10, _log(rng, 256 << 10, 16 << 20))
    P = rng.choice([8, 12, 16, 32, 64])
    h = rng.choice(_HIER[P])
    dtype = rng.choice(["f32", "f32", "bf16", "bf16", "i32", "fp8"])
    s = rng.choice([1, h[-1] if len(h) > 1 else 1])
    m = rng.choice([1, 2, 4, 8])
    ring = h[0] if len(h) > 1 and s <= P // h[0] and rng.random() < 0.15 else 1
    if form == "graph":
        kinds = ",".join(rng.sample(_SEVEN.split(","), rng.randint(1, 4)))
        nbytes = _log(rng, 16 << 10, 8 << 20)
    elif form == "request":
        kinds = rng.choice(_SEVEN.split(","))
        nbytes = _log(rng, 1 << 10, 16 << 20)
    else:
        kinds = rng.choice(_SEVEN.split(",") + ["reduce", "allreduce", "allreduce", "allreduce_via_bcast_reduce"])
        nbytes = _log(rng, 4 << 10, min(64 << 20, (2 << 30) // P))
    d = _elems(nbytes, P, dtype)
    if dtype != "fp8" and rng.random() < 0.4:              # a count that no 16-byte boundary divides
        d = max(1, min(d, (16 << 20) // P) - rng.randint(1, 3))
    op = rng.choice(["sum", "sum", "max", "min"]) if dtype != "fp8" else "sum"
    if kinds == "allreduce_via_bcast_reduce":
        op = "sum"                                         # composed from primitives that sum
    return _case(form, kinds, P, h, s, m, d, dtype, op, ring, rng.randrange(P) if "reduce" != kinds else 0)


# ---- inputs --------------------------------------------------------------------


def _members(case):
    """(kind, P, hierarchy, stripe, pipeline, d, dtype, op, ring, root) of every collective of the case."""
    if case["form"] == "group":
        out = []
        for q in synth.batch_mix(case["n"], case["mix_seed"], case["min_bytes"], case["max_bytes"]):
            e = H.ESIZE[H.DTYPES[q["dtype"]]]
            out.append((q["kind"], q["P"], tuple(q["hierarchy"]), 1, 1, q["bytes_per_rank"] // e // q["P"], q["dtype"],
                        "sum", 1, 0))
        return out
    h = tuple(int(f) for f in case["h"].split("x"))
    return [(k, case["P"], h, case["s"], case["m"], case["d"], case["dtype"], case["op"], case["ring"], case["root"])
            for k in case["kinds"].split(",")]


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _fill(t, P, dtype, g):
    """Send rows as the path meets them: gradients of ranks whose scales differ, activations, full-range integers."""
    if dtype == "i32":
        t.copy_(torch.randint(-(2**31), 2**31 - 1, t.shape, generator=g, device=t.device, dtype=torch.int64))
        return
    scale = 10.0 ** (2 * torch.rand((P, 1), generator=g, device=t.device) - 1)
    if dtype != "fp8":
        for r in range(P):                                  # row by row: no second copy of the largest inputs
            t[r].copy_(torch.randn(t.shape[1], generator=g, device=t.device) * scale[r])
        return
    for r in range(P):                                      # 128 codes, the block's scale amax / 448, 12 zero bytes
        x = (torch.randn(t.shape[1] // 144 * 128, generator=g, device=t.device) * scale[r]).reshape(-1, 128)
        amax = x.abs().amax(1, keepdim=True)
        b = t[r].reshape(-1, 144)
        b[:, :128] = (x * (448.0 / amax)).clamp(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8)
        b[:, 128:132] = (amax / 448.0).view(torch.uint8)
        b[:, 132:] = 0


def _buffers(case, seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed))
    bufs = []
    for kind, P, h, s, m, d, dtype, op, ring, root in _members(case):
        b = C.Buffers(kind, P, d, _TORCH[dtype], _device())
        _fill(b.send, P, dtype, g)
        b.recv.zero_()
        bufs.append(b)
    return bufs


def _composed(member, b):
    kind, P, h, s, m, d, dtype, op, ring, root = member
    c = H.Comm(P, dtype)
    if ring > 1:
        c.set_option(H.OPT_RING, ring)
    if kind in H.COLLECTIVES:
        c.add_collective(kind, d, b.send_ptrs(), b.recv_ptrs(), root, op)
    else:
        C.compose(c, kind, d, b.send_ptrs(), b.recv_ptrs(), root)
    return c


# ---- passes ----------------------------------------------------------------------


def prepare(case, seed):
    members = _members(case)
    bufs = _buffers(case, seed)
    torch.cuda.synchronize()
    st = {"form": case["form"], "members": members, "bufs": bufs, "out": [b.recv for b in bufs]}
    if case["form"] == "request":
        return st
    comms = [_composed(q, b) for q, b in zip(members, bufs)]
    if case["form"] == "group":
        for q, c in zip(members, comms):
            c.plan(q[2], q[3], q[4])
        st["comms"] = comms
        st["comm"] = H.Comm.group(comms)
        return st
    for q, c in zip(members, comms):
        c.init(q[2], q[3], q[4])
    st["comms"] = comms
    if case["form"] == "start":
        st["comm"] = comms[0]
        return st
    for c in comms:                                         # one direct start before the capture
        c.start()
        c.wait()
    main = torch.cuda.Stream()
    side = [main] + [torch.cuda.Stream() for _ in comms[1:]]
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=main):
        fork = torch.cuda.Event()
        fork.record(main)
        for c, s in zip(comms, side):
            if s is not main:
                s.wait_event(fork)
            c.start(s)
        for s in side[1:]:
            join = torch.cuda.Event()
            join.record(s)
            main.wait_event(join)
    st["graph"], st["streams"] = graph, side
    return st


def run(state):
    form = state["form"]
    if form == "graph":
        state["graph"].replay()
    elif form == "request":
        q = state["members"][0]
        c = _composed(q, state["bufs"][0])
        c.init(q[2], q[3], q[4])
        c.start()
        c.wait()
        c.destroy()
    else:
        state["comm"].start()
        state["comm"].wait()
    return state["out"]


def work(case):
    """Bytes with every input read once and every output written once; one operation per folded value."""
    total = flops = 0
    for kind, P, h, s, m, d, dtype, op, ring, root in _members(case):
        one = H.nbytes(H.DTYPES[dtype], d)
        chunk, full = P * one, P * P * one                  # a chunk per rank, a whole buffer per rank
        total += {"broadcast": chunk + full, "reduce": full + chunk, "allgather": chunk + full,
                  "reducescatter": full + chunk, "scatter": 2 * chunk, "gather": 2 * chunk}.get(kind, 2 * full)
        if kind in _REDUCING:
            flops += (P - 1) * P * d
    return {"bytes": total, "flops": flops}


# ---- the values in 64 bits ---------------------------------------------------------


def _wide(row, dtype):
    return row.to(torch.int64) if dtype == "i32" else row.to(torch.float64)


def _reduced(send, dtype, op):
    acc = _wide(send[0], dtype)
    for r in range(1, send.shape[0]):
        x = _wide(send[r], dtype)
        acc = acc + x if op == "sum" else torch.maximum(acc, x) if op == "max" else torch.minimum(acc, x)
    if dtype == "i32":                                      # 32-bit sums wrap
        acc = acc.to(torch.int32).to(torch.int64)
    return acc


def exact(case, seed):
    out = []
    for (kind, P, h, s, m, d, dtype, op, ring, root), b in zip(_members(case), _buffers(case, seed)):
        if dtype == "fp8":                                  # bytes of codes and scales: no 64-bit counterpart
            out.append(None)
            continue
        x = b.send
        zero = torch.zeros(b.recv.shape, dtype=torch.int64 if dtype == "i32" else torch.float64, device=x.device)
        if kind == "broadcast":
            y = _wide(x[root], dtype).expand(P, -1)
        elif kind == "scatter":
            y = _wide(x[root], dtype).reshape(P, d)
        elif kind == "gather":
            y = zero
            y[root] = _wide(x, dtype).reshape(-1)
        elif kind == "allgather":
            y = _wide(x, dtype).reshape(-1).expand(P, -1)
        elif kind == "alltoall":
            y = _wide(x, dtype).reshape(P, P, d).transpose(0, 1).reshape(P, P * d)
        elif kind == "reduce":
            y = zero
            y[root] = _reduced(x, dtype, op)
        elif kind == "reducescatter":
            y = _reduced(x, dtype, op).reshape(P, d)
        else:
            y = _reduced(x, dtype, op).expand(P, -1)
        out.append(y)
    return out if any(y is not None for y in out) else None
