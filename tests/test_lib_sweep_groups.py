"""Two-step forms of sums over many groups: the sections are the groups, as far
as a CTA holds their values, and both steps give the plain expression's bits."""
import numpy as np
import pytest

from oracle import programs as PR
from oracle import semantics as S
from oracle.model import DTYPES
from paper_2408_05962_gb300 import build as B
from tests._bridge import FakeAddresses, register
from tests._cases import fill
from tests.test_lib_sweep import FP8_TEAM, TEAM, decode, evaluate


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


@pytest.mark.parametrize("P,h,T", [(64, [32, 2], 32), (66, [33, 2], 33), (512, [64, 8], 64), (1024, [128, 8], 128),
                                   (258, [129, 2], 0), (256, [2, 32, 4], 64)])
@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
def test_sections_are_the_groups(P, h, T, dtype):
    if dtype == "fp8" and h[0] == 2:                         # FP8 values are no cheaper than sources: the fewer groups
        T = 2
    prog = PR.reduce(P, 1, dtype=dtype)
    fake = FakeAddresses(prog)
    comm = register(prog, fake.addr)
    comm.plan(h, 1, 1)
    cls, lau, ptrs, toks = decode(comm.sweep())
    (c,), (L,) = cls, lau
    assert c["team"] == T and (L["kernel"] == (FP8_TEAM if dtype == "fp8" else TEAM)) == (T > 0)
    mem = fill(prog, P)
    views = {k: v.view(np.uint8) for k, v in mem.items()}
    vals = []
    for a in ptrs[:P]:
        key, off = fake.resolve(a)
        vals.append(views[key][off:off + c["nbytes"]].copy().view(DTYPES[dtype]))
    out, _ = evaluate(vals, toks[c["tok"]:c["tok"] + P], "sum", dtype)
    if T:
        lower, bounds, upper = np.split(np.array(toks[c["ttok"]:c["ttok"] + P + 2 * T + 1]), [P, P + T + 1])
        parts = [evaluate(vals[a:z], lower[a:z].tolist(), "sum", dtype)[0] if z - a > 1 else vals[a]
                 for a, z in zip(bounds, bounds[1:])]
        two, _ = evaluate(parts, upper.tolist(), "sum", dtype)
        assert np.array_equal(two.view(np.uint8), out.view(np.uint8))
    S.run_program(prog, mem, h)
    key, off = fake.resolve(ptrs[P])
    assert np.array_equal(mem[key].view(np.uint8)[off:off + c["nbytes"]], out.view(np.uint8))
