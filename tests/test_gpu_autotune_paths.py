"""The autotuner on both execution paths: a sweep does not depend on what is
tuned, so the communicator keeps its configuration (and with it the schedule's
byte counts); a communicator that runs step by step is tuned as ever."""
import numpy as np
import pytest

from oracle import programs as PR
from oracle import semantics as S
from tests._cases import fill

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("tune_method", [False, True])
@pytest.mark.parametrize("trace", [0, 1])
@pytest.mark.parametrize("s,m", [(4, 8), (2, 3)])
def test_autotune(s, m, trace, tune_method):
    import torch
    from paper_2408_05962_gb300 import hiccl as H
    from tests._bridge import register
    prog = PR.allreduce(16, 2048)
    h = [4, 4]
    mem0 = fill(prog, 11)
    ref = {k: v.copy() for k, v in mem0.items()}
    S.run_program(prog, ref, h)
    bufs = {k: torch.from_numpy(v).cuda() for k, v in mem0.items()}
    comm = register(prog, lambda r: int(bufs[r.key].data_ptr()) + 4 * r.off)
    comm.set_option(H.OPT_TRACE, trace)
    comm.init(h, s, m)
    image, info, traffic = comm.image(), comm.plan_info(), comm.hbm_bytes()
    best = comm.autotune(tune_method=tune_method)
    assert best["us"] > 0 and best["trials"] >= (15 if tune_method else 8)
    if trace:
        assert best["order"] in (0, 1) and (tune_method or (best["stripe"], best["pipeline"]) == (s, m))
    else:
        assert (best["stripe"], best["pipeline"]) == (s, m)
        assert comm.plan_info() == info and comm.hbm_bytes() == traffic
        assert comm.image()[0] == image[0] and np.array_equal(comm.image()[1], image[1])
    for k, v in mem0.items():
        bufs[k].copy_(torch.from_numpy(v))
    comm.start()
    comm.wait()
    for k in ref:
        assert np.array_equal(bufs[k].cpu().numpy().view(np.uint32), ref[k].view(np.uint32)), k
    comm.destroy()
