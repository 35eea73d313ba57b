"""The step executor where starts would otherwise run a sweep: traced
communicators, and groups with a member whose program has no sweep.  Its
ticket counter across grid changes and replays, stream order, work-item
options, and the tickets of grouped members, all against the oracle.  And
sweeps on several streams, which share the device."""
import numpy as np
import pytest

from oracle import programs as PR
from oracle import semantics as S
from tests._cases import fill
from tests.test_gpu_group import MEMBERS, _check, _reset

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def _allreduce(P, h, d, s, m, options=()):
    """A traced All-reduce communicator over new buffers."""
    import torch
    from paper_2408_05962_gb300 import collectives as C
    from paper_2408_05962_gb300 import hiccl as H
    b = C.Buffers("allreduce", P, d, torch.float32)
    comm = H.Comm(P, "f32")
    comm.set_option(H.OPT_TRACE, 1)
    for opt, value in options:
        comm.set_option(opt, value)
    C.compose(comm, "allreduce", d, b.send_ptrs(), b.recv_ptrs())
    comm.init(h, s, m)
    return comm, b


def _inputs(P, h, d, seed):
    prog = PR.allreduce(P, d)
    mem0 = fill(prog, seed)
    ref = {k: v.copy() for k, v in mem0.items()}
    S.run_program(prog, ref, h)
    return (np.stack([mem0[("send", r)] for r in range(P)]), np.stack([ref[("recv", r)] for r in range(P)]))


def _same(t, want):
    return np.array_equal(t.cpu().numpy().view(np.uint32), want.view(np.uint32))


def test_grid_changes_and_replays_number_items_from_one_counter():
    """CTAs per SM and threads change between starts, and a graph captured with
    the last grid is replayed between further starts."""
    import torch
    from paper_2408_05962_gb300 import hiccl as H
    P, h, d = 16, [4, 4], 8195
    comm, b = _allreduce(P, h, d, 2, 4)
    graph = None
    plan = [(2, 256, False), (1, 256, False), (1, 256, False), (2, 128, False), (2, 256, False), (2, 256, True),
            (2, 256, False), (2, 256, True), (2, 256, True)]
    for it, (per_sm, threads, replay) in enumerate(plan):
        x, want = _inputs(P, h, d, 700 + it)
        b.send.copy_(torch.from_numpy(x))
        b.recv.fill_(-1.0)
        torch.cuda.synchronize()
        comm.set_option(H.OPT_CTAS_PER_SM, per_sm)
        comm.set_option(H.OPT_THREADS, threads)
        if replay:
            if graph is None:
                gs = torch.cuda.Stream()
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=gs):
                    comm.start(gs)
            graph.replay()
            torch.cuda.synchronize()
        else:
            comm.start()
            comm.wait()
        assert _same(b.recv, want), it
    assert len(comm.trace()) == comm.plan_info()["items"]          # one record an item: it ran step by step
    comm.destroy()


def test_stream_order():
    """Inputs written by the kernel before a start, results read by the kernel
    after it, and a second start right behind the first."""
    import torch
    P, h, d = 16, [4, 4], 4099
    comm, b = _allreduce(P, h, d, 4, 4)
    twin, b2 = _allreduce(P, h, d, 2, 2)
    s = torch.cuda.current_stream()
    for it in range(4):
        x, want = _inputs(P, h, d, 500 + it)
        staged = torch.from_numpy(x).cuda()
        torch.cuda.synchronize()
        b.recv.fill_(float(it))
        b2.recv.fill_(float(it))
        b.send.copy_(staged)
        b2.send.copy_(staged)
        comm.start(s)
        twin.start(s)
        out = b.recv.clone()
        out2 = b2.recv.clone()
        comm.wait()
        twin.wait()
        assert _same(out, want) and _same(out2, want), it
    comm.destroy()
    twin.destroy()


def test_work_item_options_do_not_change_results():
    import torch
    from paper_2408_05962_gb300 import hiccl as H
    P, h, d = 16, [4, 4], 5000
    x, want = _inputs(P, h, d, 3)
    items = set()
    for opts in ([], [(H.OPT_ORDER, 0)], [(H.OPT_ITEM_BYTES, 4096)], [(H.OPT_ITEM_BYTES, 1 << 20), (H.OPT_SLOT_ITEMS, 8)],
                 [(H.OPT_CTAS_PER_SM, 1)], [(H.OPT_THREADS, 512)]):
        comm, b = _allreduce(P, h, d, 4, 4, opts)
        b.send.copy_(torch.from_numpy(x))
        comm.start()
        comm.wait()
        items.add(comm.plan_info()["items"])
        assert _same(b.recv, want), opts
        comm.destroy()
    assert len(items) > 1


def test_grouped_members_share_the_tickets():
    """A group runs step by step when one member has no sweep (All-gather as
    Gather and Broadcast): directly, from a graph, and directly again."""
    import torch
    from paper_2408_05962_gb300 import hiccl as H
    from tests._bridge import register
    progs, refs, dev, comms = [], [], [], []
    for i, (name, P, h, s, m, dt, d) in enumerate(MEMBERS + [("allgather_bcast_gather", 8, [2, 4], 2, 2, "f32", 513)]):
        prog = PR.BUILDERS[name](P, d, dtype=dt)
        mem0 = fill(prog, 200 + i)
        ref = {k: v.copy() for k, v in mem0.items()}
        S.run_program(prog, ref, h)
        bufs = {k: torch.from_numpy(v.view(np.uint8).copy()).cuda() for k, v in mem0.items()}
        es = np.dtype(next(iter(mem0.values())).dtype).itemsize
        comm = register(prog, lambda r, b=bufs, es=es: int(b[r.key].data_ptr()) + es * r.off)
        comm.plan(h, s, m)
        progs.append((prog, mem0))
        refs.append(ref)
        dev.append(bufs)
        comms.append(comm)
    assert not comms[-1].sweep()
    g = H.Comm.group(comms)
    assert not g.sweep()
    for _ in range(2):
        _reset(progs, dev)
        g.start()
        g.wait()
        _check(progs, refs, dev)
    s = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=s):
        g.start(s)
    for _ in range(3):
        _reset(progs, dev)
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        _check(progs, refs, dev)
    _reset(progs, dev)
    g.start()
    g.wait()
    _check(progs, refs, dev)
    g.destroy()


def test_sweeps_on_several_streams_overlap():
    """Eight flat sums of 512 ranks, a few warps each and tens of microseconds
    long, captured on one stream and on eight: side by side they take less than
    half as long."""
    import torch
    from paper_2408_05962_gb300 import collectives as C
    from paper_2408_05962_gb300 import hiccl as H
    P, d, n = 512, 4, 8
    comms, bufs = [], []
    for _ in range(n):
        b = C.Buffers("reduce", P, d, torch.float32)
        b.send.normal_()
        c = H.Comm(P, "f32")
        c.add_collective("reduce", d, b.send_ptrs(), b.recv_ptrs(), 0)
        c.init([P], 1, 1)
        assert c.sweep()
        c.start()
        c.wait()
        comms.append(c)
        bufs.append(b)
    ms = {}
    for width in (1, n):
        main = torch.cuda.Stream()
        side = [main] + [torch.cuda.Stream() for _ in range(width - 1)]
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=main):
            fork = torch.cuda.Event()
            fork.record(main)
            for s in side[1:]:
                s.wait_event(fork)
            for k, c in enumerate(comms):
                c.start(side[k % width])
            for s in side[1:]:
                join = torch.cuda.Event()
                join.record(s)
                main.wait_event(join)
        times = []
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            graph.replay()
            e1.record()
            torch.cuda.synchronize()
            times.append(e0.elapsed_time(e1))
        ms[width] = sorted(times)[1]
    assert ms[n] < 0.5 * ms[1], ms
    for c in comms:
        c.destroy()
