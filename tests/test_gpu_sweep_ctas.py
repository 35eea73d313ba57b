"""Sweeps limited to one CTA an SM (CTAS_PER_SM = 1) give the same bits as
unlimited ones, in passes of a few units and of several waves."""
import pytest

from tests.test_gpu_sweep import _buffers

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


# 2432 warps in a wave: copies of 2 KiB, folds and FP8 folds of 512 and 576
# bytes a unit; operands off each other (pad) take the shifted copies and the
# narrow folds
@pytest.mark.parametrize("kind,P,h,d,dtype,pad", [
    ("broadcast", 4, [4], 9, "f32", 0), ("broadcast", 4, [4], 1 << 19, "f32", 0), ("alltoall", 16, [4, 4], 32771, "bf16", 1),
    ("alltoall", 16, [4, 4], 7, "bf16", 1), ("allreduce", 8, [2, 4], 200003, "f32", 0), ("allreduce", 8, [2, 4], 131075, "bf16", 0),
    ("reduce", 64, [2] * 6, 30000, "bf16", 0), ("reducescatter", 12, [2, 2, 3], 40001, "f32", 1),
    ("reducescatter", 12, [2, 2, 3], 5, "bf16", 1), ("allreduce", 16, [4, 4], 128 * 700, "fp8", 0),
    ("reducescatter", 8, [8], 128 * 3, "fp8", 0), ("reduce", 64, [64], 3000, "i32", 0)])
def test_one_cta_an_sm(kind, P, h, d, dtype, pad):
    import torch
    from paper_2408_05962_gb300 import hiccl as H
    b = _buffers(kind, P, d, dtype, d, pad)
    c = H.Comm(P, dtype)
    c.add_collective(kind, d, b.send_ptrs(), b.recv_ptrs(), P - 1)
    c.init(h, 1, 1)
    got = []
    for ctas in (2, 1):
        c.set_option(H.OPT_CTAS_PER_SM, ctas)
        for _ in range(2):
            b.recv.view(torch.uint8).fill_(0xa5)
            c.start()
            c.wait()
        got.append(b.recv.clone())
    c.destroy()
    c = H.Comm(P, dtype)                                   # limited from the start, and under capture
    c.set_option(H.OPT_CTAS_PER_SM, 1)
    c.add_collective(kind, d, b.send_ptrs(), b.recv_ptrs(), P - 1)
    c.init(h, 1, 1)
    b.recv.view(torch.uint8).fill_(0xa5)
    s, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=s):
        c.start(s)
    graph.replay()
    torch.cuda.synchronize()
    c.destroy()
    assert torch.equal(got[0].view(torch.uint8), b.recv.view(torch.uint8))
    assert torch.equal(got[0].view(torch.uint8), got[1].view(torch.uint8))
