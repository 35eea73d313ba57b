"""Sweep kernels on the GPU at the sizes where their tiling can go wrong, bit
for bit against the step executor on the same buffers (a traced communicator
runs its schedule step by step), whose results the parity tests compare with
the oracle; and the step executor's own data paths against the oracle."""
import numpy as np
import pytest

from oracle import programs as PR
from oracle import semantics as S
from tests._cases import fill
from tests._gpu import assert_bit_equal, run_on_gpu

pytestmark = pytest.mark.gpu
REDUCING = ("reduce", "reducescatter", "allreduce")


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def _buffers(kind, P, d, dtype, seed, pad=0):
    import torch
    from paper_2408_05962_gb300 import collectives as C
    tdt = {"f32": torch.float32, "i32": torch.int32, "bf16": torch.bfloat16, "fp8": torch.uint8}[dtype]
    b = C.Buffers(kind, P, d, tdt, "cuda", pad)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if dtype == "i32":
        b.send.copy_(torch.randint(-2**31, 2**31 - 1, b.send.shape, generator=g, device="cuda"))
    elif dtype == "fp8":                                   # any finite codes, scales of several decades
        b.send.random_(0, 0x7f, generator=g)
        blk = b.send.reshape(P, -1, 144)
        blk[:, :, :64] |= 0x80
        scale = 10.0 ** (4 * torch.rand(blk.shape[:2] + (1,), generator=g, device="cuda") - 2)
        blk[:, :, 128:132] = scale.view(torch.uint8)
        blk[:, :, 132:] = 0
    else:
        b.send.copy_(torch.randn(b.send.shape, generator=g, device="cuda"))
    return b


def _both(kind, P, h, s, m, d, dtype, op="sum", ring=1, seed=0, pad=0):
    """The sweep's result equals the step executor's."""
    import torch
    from paper_2408_05962_gb300 import hiccl as H
    b = _buffers(kind, P, d, dtype, seed, pad)
    got = []
    for trace in (0, 1):
        c = H.Comm(P, dtype)
        c.set_option(H.OPT_TRACE, trace)
        if ring > 1:
            c.set_option(H.OPT_RING, ring)
        c.add_collective(kind, d, b.send_ptrs(), b.recv_ptrs(), P - 1, op if kind in REDUCING else "sum")
        c.init(h, s, m)
        assert c.sweep()
        for _ in range(2):
            b.recv.view(torch.uint8).fill_(0xa5)
            c.start()
            c.wait()
        got.append(b.recv.clone())
        c.destroy()
    assert torch.equal(got[0].view(torch.uint8), got[1].view(torch.uint8))


# chunk lengths around one lane, one row of lanes (512 bytes) and several
# vectors a lane, whole and with element tails; the last ones take the widest units
@pytest.mark.parametrize("d", [1, 3, 4, 127, 128, 129, 511, 1030, 4096, 131072 + 64, 131072 + 67])
@pytest.mark.parametrize("dtype", ["f32", "bf16", "i32"])
@pytest.mark.parametrize("kind", ["allreduce", "alltoall"])
def test_chunk_edges(kind, dtype, d):
    _both(kind, 8, [2, 4], 1, 1, d, dtype, seed=d)


# rows `pad` elements longer than their data: chunks of every rank lie
# differently off a 16-byte boundary, and the padding is not written
@pytest.mark.parametrize("d", [1, 7, 9, 15, 16, 23, 247, 248, 249, 255, 991, 993, 1000, 66000, 262147])
@pytest.mark.parametrize("dtype,pad", [("f32", 1), ("f32", 3), ("bf16", 1), ("bf16", 2), ("bf16", 7)])
@pytest.mark.parametrize("kind", ["allreduce", "alltoall", "broadcast"])
def test_operands_off_each_other(kind, dtype, pad, d):
    _both(kind, 6, [2, 3], 1, 1, d, dtype, seed=d, pad=pad)


@pytest.mark.parametrize("dtype,op", [("f32", "max"), ("i32", "min"), ("i32", "lor"), ("bf16", "min"), ("bf16", "sum")])
@pytest.mark.parametrize("d", [77, 65536, 65537])
def test_operators_and_fan_ins(dtype, op, d):
    _both("reducescatter", 12, [2, 2, 3], 3, 2, d, dtype, op, seed=d)
    _both("reduce", 16, [16], 1, 1, d, dtype, op, seed=d + 1)
    _both("allreduce", 9, [9], 1, 1, d, dtype, op, seed=d + 2)


# folds whose plain combines fill, straddle or miss a group of four, in the first
# 32 sources and after them; enough units for a warp, not a block, to own each
@pytest.mark.parametrize("dtype,op", [("f32", "max"), ("i32", "max"), ("bf16", "max"), ("i32", "sum")])
@pytest.mark.parametrize("P,h", [(3, [3]), (5, [5]), (8, [8]), (9, [9]), (24, [4, 6]), (35, [35]), (36, [3, 12]), (70, [7, 10])])
def test_groups_of_plain_combines(P, h, dtype, op):
    d = 330000 // P + 3                                    # 2600 units, 1300 of BF16
    _both("reduce", P, h, 1, 1, d, dtype, op, seed=P, pad=-(P * d) % 8)


@pytest.mark.parametrize("blocks", [1, 3, 4, 5, 64, 2051])
@pytest.mark.parametrize("P,h,ring", [(8, [2, 4], 1), (12, [2, 2, 3], 1), (16, [16], 1), (12, [4, 3], 4)])
def test_fp8_blocks(P, h, ring, blocks):
    for kind in ("allreduce", "allgather"):
        _both(kind, P, h, 1, 1, 128 * blocks, "fp8", ring=ring, seed=blocks)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("P,h,ring,d", [(64, [2] * 6, 1, 70), (64, [2] * 6, 1, 9000), (64, [4, 4, 4], 16, 515),
                                        (32, [4, 8], 32, 4096), (1024, [32, 32], 1, 5)])
def test_deep_and_wide_expressions(P, h, ring, d, dtype):
    """As many saved values as the kernels hold, chains, and 1024 sources."""
    _both("reducescatter" if P < 1024 else "reduce", P, h, 1, 1, d, dtype, ring=ring, seed=d)


@pytest.mark.parametrize("name", ["broadcast", "scatter", "gather", "allgather", "reducescatter", "allreduce", "alltoall"])
@pytest.mark.parametrize("dtype,d,mis", [("f32", 2053, 0), ("f32", 8192, 0), ("i32", 999, 1), ("bf16", 4099, 0),
                                         ("bf16", 2048, 3), ("fp8", 61, 0)])
def test_step_executor(name, dtype, d, mis):
    """The step executor, where a sweep would otherwise run: bulk copies,
    shared-memory folds, wide and misaligned operands."""
    from paper_2408_05962_gb300 import hiccl as H
    prog = PR.BUILDERS[name](12, d, dtype=dtype)
    mem0 = fill(prog, d)
    ref = {k: v.copy() for k, v in mem0.items()}
    S.run_program(prog, ref, [4, 3])
    for h in ([4, 3], [12]):
        ref = {k: v.copy() for k, v in mem0.items()}
        S.run_program(prog, ref, h)
        outs, _ = run_on_gpu(prog, h, 3, 2, mem0, repeats=2, misalign_elems=mis, options={H.OPT_TRACE: 1})
        for out in outs:
            assert_bit_equal(ref, out)


def test_current_stream_of_a_start():
    """A start without a stream goes to PyTorch's current one, as it changes."""
    import torch
    from paper_2408_05962_gb300 import hiccl as H
    streams = [torch.cuda.default_stream(), torch.cuda.Stream(), torch.cuda.Stream(priority=-1)]
    for s in streams + streams:
        with torch.cuda.stream(s):
            assert H._stream_handle(None) == torch.cuda.current_stream().cuda_stream == s.cuda_stream
    b = _buffers("allreduce", 8, 50000, "f32", 3)
    c = H.Comm(8, "f32")
    c.add_collective("allreduce", 50000, b.send_ptrs(), b.recv_ptrs())
    c.init([2, 4], 1, 1)
    c.start()
    c.wait()
    want = b.recv.clone()
    torch.cuda.synchronize()
    with torch.cuda.stream(streams[1]):
        torch.cuda._sleep(20_000_000)                      # the fill is still queued when the start is issued
        b.recv.zero_()
        c.start()
        c.wait()
    assert torch.equal(b.recv, want)


def test_sweep_replayed_and_restarted():
    """Captured starts of two communicators on forked streams, replayed beside
    direct starts; one CTA per SM (CTAS_PER_SM = 1) gives the same result."""
    import torch
    from paper_2408_05962_gb300 import hiccl as H
    P, d = 16, 30000
    want, comms, bufs = [], [], []
    for kind in ("allreduce", "reducescatter"):
        b = _buffers(kind, P, d, "f32", 7)
        c = H.Comm(P, "f32")
        c.add_collective(kind, d, b.send_ptrs(), b.recv_ptrs())
        c.init([4, 4], 4, 2)
        c.start()
        c.wait()
        want.append(b.recv.clone())
        comms.append(c)
        bufs.append(b)
    main, side = torch.cuda.Stream(), torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=main):
        fork, join = torch.cuda.Event(), torch.cuda.Event()
        fork.record(main)
        side.wait_event(fork)
        comms[0].start(main)
        comms[1].start(side)
        join.record(side)
        main.wait_event(join)
    for ctas in (2, 1):
        for c in comms:
            c.set_option(H.OPT_CTAS_PER_SM, ctas)
        for _ in range(3):
            for b in bufs:
                b.recv.zero_()
            torch.cuda.synchronize()
            graph.replay()
            torch.cuda.synchronize()
            assert all(torch.equal(b.recv, w) for b, w in zip(bufs, want))
            for b, c in zip(bufs, comms):
                b.recv.zero_()
                torch.cuda.synchronize()
                c.start()
                c.wait()
            assert all(torch.equal(b.recv, w) for b, w in zip(bufs, want))


def test_many_classes():
    """A program of 300 primitives of different lengths: copies and folds whose
    classes are found through hints."""
    from oracle.model import Program
    prog = Program(4)
    n = [1 + 13 * k % 2200 for k in range(300)]
    a = [prog.buffer(("send", r), sum(n)) for r in range(4)]
    b = [prog.buffer(("recv", r), sum(n)) for r in range(4)]
    o = 0
    for k, m in enumerate(n):
        if k % 3:
            prog.multicast(k % 4, [0, 1, 2, 3], m, a[k % 4].shift(o), {j: b[j].shift(o) for j in range(4)})
        else:
            prog.reduction([0, 1, 2, 3], k % 4, m, {j: a[j].shift(o) for j in range(4)}, b[k % 4].shift(o))
        o += m
    mem0 = fill(prog, 11)
    ref = {k: v.copy() for k, v in mem0.items()}
    S.run_program(prog, ref, [2, 2])
    outs, comm = run_on_gpu(prog, [2, 2], 1, 1, mem0, repeats=2)
    assert comm.sweep()
    for out in outs:
        assert_bit_equal(ref, out)
