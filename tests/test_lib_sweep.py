"""The sweep of a plan (one pass of independent expressions), decoded on the
host and evaluated on NumPy buffers with its members in a random order, gives
the oracle's plain semantics bit for bit -- and so the result of the step
table, which the other tests of the factorizer compare with the same oracle."""
import struct

import numpy as np
import pytest

from oracle import programs as PR
from oracle import semantics as S
from oracle.hierarchy import all_factorizations
from oracle.lowprec import from_acc, to_acc
from oracle.model import DTYPES, Program
from oracle.semantics import combine
from paper_2408_05962_gb300 import build as B
from paper_2408_05962_gb300 import hiccl as H
from tests._bridge import FakeAddresses, register
from tests._cases import fill, random_program

START, PUSH, ROUND, POP, JOIN = 1, 2, 1, 2, 3
COPY, FOLD, FP8, NARROW, SHIFT, TEAM, FP8_TEAM = range(7)


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def decode(blob):
    """(classes, launches, pointers, tokens) of a sweep's inspection blob."""
    nc, nl, npt, nt, nh = struct.unpack_from("<5Q", blob, 0)
    o = 40
    cls = [dict(zip(("nbytes", "ptr", "unit0", "upm", "nmem", "nsrc", "ndst", "tok", "meta", "group",
                     "team", "ttok"),
                    struct.unpack_from("<2Q10I", blob, o + 64 * k))) for k in range(nc)]
    o += 64 * nc
    lau = [dict(zip(("kernel", "lo", "hi", "units", "threads", "words", "hint"), struct.unpack_from("<7I", blob, o + 32 * k)))
           for k in range(nl)]
    o += 32 * nl
    ptrs = np.frombuffer(blob, np.uint64, npt, o).tolist()
    toks = np.frombuffer(blob, np.uint32, nt, o + 8 * npt).tolist()
    assert len(blob) == o + 8 * npt + 4 * (nt + nh)
    hints = np.frombuffer(blob, np.uint32, nh, o + 8 * npt + 4 * nt)
    for L in lau:                                        # the class of every unit lies between two hints
        first = [c["unit0"] for c in cls[L["lo"]:L["hi"]]]
        if len(first) > 96:
            at = np.searchsorted(first, np.arange(L["units"]), side="right") - 1
            h = hints[L["hint"]:]
            i = np.arange(L["units"]) >> 7
            assert (h[i] <= at).all() and (at <= h[i + 1]).all() and (h[i + 1] < len(first)).all()
    for c in cls:
        m = c["meta"]
        c.update(dtype=m & 15, rop=(m >> 4) & 7, width=1 << ((m >> 7) & 7), v=(m >> 10) & 31, kernel=(m >> 15) & 7)
    return cls, lau, ptrs, toks


def evaluate(vals, toks, op, dtype):
    """One expression by its tokens, on the payload's accumulators."""
    lp = dtype in ("bf16", "fp8")
    wide = (lambda v: to_acc(v, dtype).copy()) if lp else (lambda v: v.copy())
    comb = (lambda a, b: combine(a, b, op).astype(np.float32)) if lp else (lambda a, b: combine(a, b, op))
    acc, saved, most = None, [], 0
    for v, t in zip(vals, toks):
        if t & START:
            if t & PUSH:
                saved.append(acc)
                most = max(most, len(saved))
            acc = wide(v)
        else:
            acc = comb(acc, wide(v))
        o = t >> 8
        while o:
            if o & 3 == ROUND:
                acc = wide(from_acc(acc, dtype))
            elif o & 3 == POP:
                acc = comb(saved.pop(), acc)
            else:
                acc = comb(acc, saved.pop())
            o >>= 2
    assert not saved
    return (from_acc(acc, dtype) if lp else acc), most


def run_sweep(comm, fake, mem, dtype, seed=0):
    """Evaluate every member of the plan's sweep, in a random order; None if
    the plan has no sweep.  Checks the launch data on the way."""
    blob = comm.sweep()
    if not blob:
        return None
    cls, lau, ptrs, toks = decode(blob)
    views = {k: v.view(np.uint8) for k, v in mem.items()}
    dt = DTYPES[dtype]

    def view(a, n):
        key, off = fake.resolve(a)
        return views[key][off:off + n]

    assert [x for L in lau for x in range(L["lo"], L["hi"])] == list(range(len(cls)))
    members = []
    for L in lau:
        units = 0
        for c in cls[L["lo"]:L["hi"]]:
            assert c["kernel"] == L["kernel"] and c["unit0"] == units
            unit = {FP8: 4 * 144, FP8_TEAM: 4 * 144, SHIFT: 31 * 16}.get(L["kernel"], 32 * min(c["width"], 16)) * c["v"]
            assert (c["upm"] - 1) * unit < c["nbytes"] <= c["upm"] * unit        # units tile a member
            assert c["v"] in (1, 2, 4, 8, 16)
            assert c["group"] == (c["ndst"] if c["nsrc"] > 1 else 2)
            units += c["upm"] * c["nmem"] * -(-c["ndst"] // c["group"])
            for i in range(c["nmem"]):
                p = ptrs[c["ptr"] + i * (c["nsrc"] + c["ndst"]):][:c["nsrc"] + c["ndst"]]
                assert all((a - p[0]) % c["width"] == 0 for a in p) and (c["width"] >= 16 or p[0] % c["width"] == 0)
                assert (L["kernel"] in (NARROW, SHIFT)) == (c["width"] < 16)
                assert L["kernel"] == FOLD or (c["nsrc"] > 1) == (L["kernel"] not in (COPY, SHIFT))
                members.append((c, p))
        assert L["units"] == units and L["threads"] in (32, 64, 128, 256, 512)
    rng = np.random.Generator(np.random.PCG64(seed))
    for k in rng.permutation(len(members)):
        c, p = members[k]
        vals = [view(a, c["nbytes"]).copy().view(dt) for a in p[:c["nsrc"]]]
        out = vals[0]
        if c["nsrc"] > 1:
            op, n, T = H.OP_NAMES[c["rop"]], c["nsrc"], c["team"]
            out, most = evaluate(vals, toks[c["tok"]:c["tok"] + n], op, dtype)
            assert T > 1 or c["kernel"] not in (TEAM, FP8_TEAM)
            if T:                                        # in two steps, whichever the launch takes
                lower, bounds, upper = np.split(np.array(toks[c["ttok"]:c["ttok"] + n + 2 * T + 1]), [n, n + T + 1])
                assert bounds[0] == 0 and bounds[-1] == n and T <= 32 and n >= 8
                parts = [evaluate(vals[a:z], lower[a:z].tolist(), op, dtype) if z - a > 1 else (vals[a], 0)
                         for a, z in zip(bounds, bounds[1:])]
                two, m2 = evaluate([p for p, _ in parts], upper.tolist(), op, dtype)
                assert np.array_equal(two.view(np.uint8), out.view(np.uint8))
                most = max([most, m2] + [m for _, m in parts])
            acc = 16 if dtype == "fp8" else (min(c["width"], 16) // (2 if dtype == "bf16" else 4))
            L = next(x for x in lau if x["kernel"] == c["kernel"])
            assert most * max(acc, 1) * c["v"] <= L["words"]   # saved values fit
        for a in p[c["nsrc"]:]:
            view(a, c["nbytes"])[...] = out.view(np.uint8)
    return mem


def check(prog, h, s, m, seed=0, ring=1, zero_frac=0.0, fake=None):
    fake = fake or FakeAddresses(prog)
    comm = register(prog, fake.addr)
    if ring > 1:
        comm.set_option(H.OPT_RING, ring)
    comm.plan(h, s, m)
    mem0 = fill(prog, seed, zero_frac)
    ref = {k: v.copy() for k, v in mem0.items()}
    S.run_program(prog, ref, h, ring)
    got = run_sweep(comm, fake, {k: v.copy() for k, v in mem0.items()}, prog.dtype, seed)
    if got is not None:
        for k in ref:
            assert np.array_equal(ref[k].view(np.uint8), got[k].view(np.uint8)), k
    return got is not None


TABLE2 = PR.SEVEN + ("reduce", "allreduce_single", "allreduce_bcast_reduce", "reduce_gather_rs", "broadcast_ag_scatter")


@pytest.mark.parametrize("name", TABLE2)
@pytest.mark.parametrize("dtype", ["f32", "i32", "bf16", "fp8"])
@pytest.mark.parametrize("P,h,s,m,ring", [(8, [2, 4], 1, 1, 1), (12, [2, 2, 3], 3, 2, 1), (16, [16], 2, 3, 1),
                                          (12, [4, 3], 3, 2, 4), (8, [2, 2, 2], 1, 2, 8), (12, [2, 2, 3], 2, 1, 4)])
def test_collectives_have_sweeps_equal_to_the_oracle(name, dtype, P, h, s, m, ring):
    assert check(PR.BUILDERS[name](P, 3 if dtype == "fp8" else 37, dtype=dtype), h, s, m, seed=P + s, ring=ring)


@pytest.mark.parametrize("op,dtype", [(o, d) for o in ("max", "min") for d in ("f32", "i32", "bf16")] + [("lor", "i32")])
def test_operators(op, dtype):
    for name in ("allreduce", "reducescatter"):
        assert check(PR.BUILDERS[name](12, 29, dtype=dtype, op=op), [2, 2, 3], 3, 2, seed=5, zero_frac=0.25)


def test_random_programs_and_hierarchies():
    """Random leaf sets, roots and fences over every hierarchy: a sweep, where
    the plan has one, equals the oracle; both outcomes occur."""
    seen = set()
    for P in (2, 3, 4, 6, 8, 12):
        for h in all_factorizations(P):
            for seed in range(4):
                prog = random_program(P, P * 100 + seed + len(h), ("f32", "i32", "bf16")[seed % 3])
                if S.find_race(prog) is None:
                    seen.add(check(prog, h, 1 + seed % P, 1 + seed % 2, seed=seed))
    assert seen == {True, False}


@pytest.mark.parametrize("dtype,shift", [("f32", 1), ("f32", 4), ("bf16", 1), ("bf16", 2), ("bf16", 8)])
def test_operands_off_a_vector_boundary(dtype, shift):
    """Every buffer `shift` elements off its boundary, odd chunk lengths: the
    accesses are as wide as all operands of a member allow."""
    for name in ("allreduce", "alltoall", "broadcast"):
        prog = PR.BUILDERS[name](8, 131, dtype=dtype)
        fake = FakeAddresses(prog)
        fake.base = {k: a + shift * DTYPES[dtype].itemsize for k, a in fake.base.items()}
        assert check(prog, [2, 4], 2, 2, seed=shift, fake=fake)


def two_epochs(build):
    """A 4-rank program over buffers a and b of 64 values per rank."""
    prog = Program(4)
    a = [prog.buffer(("send", r), 64) for r in range(4)]
    b = [prog.buffer(("recv", r), 64) for r in range(4)]
    build(prog, a, b)
    return prog


def test_in_place_allreduce_is_one_sweep():
    """Listing 2 with receive buffers equal to the send buffers: the gathered
    chunk overwrites sources of its own expression at the same offsets."""
    P, d = 8, 48
    base = [0x7f0000000000 + r * 0x10000 for r in range(P)]
    c = H.Comm(P, "f32")
    c.add_collective("allreduce", d, base, base)
    c.plan([2, 4], 2, 2)
    cls, _, ptrs, _ = decode(c.sweep())
    assert sum(k["nmem"] for k in cls) == P
    for k in cls:
        for i in range(k["nmem"]):
            p = ptrs[k["ptr"] + i * (k["nsrc"] + k["ndst"]):][:k["nsrc"] + k["ndst"]]
            assert k["nsrc"] == P and sorted(p[:P]) == sorted(p[P:])


def _all(r):
    return {j: r[j] for j in range(4)}


@pytest.mark.parametrize("case", ["sum_of_sums", "overwritten_source", "part", "other_offset", "two_values"])
def test_other_conflicts_across_a_fence_stay_with_the_steps(case):
    """A program whose later epoch is not a copy of one expression has no sweep."""
    def build(prog, a, b):
        prog.reduction([0, 1, 2, 3], 0, 32, _all(a), b[0])
        if case == "two_values":
            prog.multicast(1, [0], 32, a[1], {0: b[0].shift(32)})
        prog.fence()
        if case == "sum_of_sums":
            prog.reduction([0, 1], 2, 32, {0: b[0], 1: a[1]}, b[2])
        elif case == "overwritten_source":
            prog.multicast(3, [2], 32, a[3].shift(32), {2: a[2]})
        elif case == "part":
            prog.multicast(0, [2], 16, b[0].shift(8), {2: b[2]})
        elif case == "other_offset":
            prog.multicast(0, [2], 32, b[0], {2: a[2].shift(16)})
        else:
            prog.multicast(0, [2], 64, b[0], {2: b[2]})
    prog = two_epochs(build)
    assert S.find_race(prog) is None
    assert not check(prog, [2, 2], 1, 1)


def test_a_repeated_copy_and_a_disjoint_one_are_swept():
    def build(prog, a, b):
        prog.multicast(0, [1, 2], 32, a[0], {1: b[1], 2: b[2]})
        prog.fence()
        prog.multicast(1, [2, 3], 32, b[1], {2: b[2], 3: b[3]})       # b[2] again, with the same value
        prog.multicast(3, [0], 32, a[3], {0: b[0].shift(32)})         # touches nothing of the first epoch
    assert check(two_epochs(build), [2, 2], 1, 1)


@pytest.mark.parametrize("P,h,dtype,op,ring,T", [(64, [4, 4, 4], "f32", "sum", 1, 4), (64, [8, 8], "bf16", "sum", 1, 8),
                                                 (12, [2, 2, 3], "bf16", "sum", 1, 4), (8, [2, 4], "f32", "sum", 1, 2),
                                                 (16, [16], "f32", "sum", 1, 0), (16, [16], "i32", "sum", 1, 4),
                                                 (64, [64], "i32", "max", 1, 8), (16, [4, 4], "f32", "min", 4, 4),
                                                 (16, [4, 4], "f32", "sum", 4, 0), (6, [2, 3], "f32", "sum", 1, 0),
                                                 (16, [4, 4], "fp8", "sum", 1, 4)])
def test_two_step_forms(P, h, dtype, op, ring, T):
    """Sections at a level's groups, or anywhere for exact operators; none for
    chains and one-level sums, whose order is sequential, nor for few sources."""
    prog = PR.reducescatter(P, 2 if dtype == "fp8" else 37, dtype=dtype, op=op)
    assert check(prog, h, 1, 1, seed=P, ring=ring, zero_frac=0.25)
    fake = FakeAddresses(prog)
    comm = register(prog, fake.addr)
    comm.set_option(H.OPT_RING, ring)
    comm.plan(h, 1, 1)
    cls, lau, _, _ = decode(comm.sweep())
    assert {c["team"] for c in cls} == {T}
    if T and all(c["width"] >= 16 for c in cls):
        assert [x["kernel"] for x in lau] == [FP8_TEAM if dtype == "fp8" else TEAM]


def test_many_classes_have_hints():
    """A program of 150 multicasts of different lengths: classes beyond the
    argument prefix are found through hints, and the sweep is the oracle's."""
    prog = Program(4)
    n = [3 + 7 * k % 1500 for k in range(150)]
    a = [prog.buffer(("send", r), sum(n)) for r in range(4)]
    b = [prog.buffer(("recv", r), sum(n)) for r in range(4)]
    o = 0
    for k, m in enumerate(n):
        prog.multicast(k % 4, [0, 1, 2, 3], m, a[k % 4].shift(o), {j: b[j].shift(o) for j in range(4)})
        o += m
    assert check(prog, [2, 2], 1, 1, seed=3)


def test_deep_hierarchies_fall_back():
    """Eight levels of two need seven saved values, more than the kernels hold."""
    assert check(PR.reduce(64, 8), [2] * 6, 1, 1)
    assert not check(PR.reduce(256, 4), [2] * 8, 1, 1)


def test_group_sweep_is_the_union():
    shapes = [("allreduce", [4, 4], 2, 3, "f32"), ("allgather", [2, 8], 4, 2, "bf16"), ("reducescatter", [16], 1, 1, "bf16")]
    members, total = [], 0
    base = 0x7f0000000000
    for name, h, s, m, dt in shapes:
        prog = PR.BUILDERS[name](16, 40, dtype=dt)
        fake = FakeAddresses(prog, base=base)
        base = (fake.end + (1 << 20)) & ~255
        c = register(prog, fake.addr)
        c.plan(h, s, m)
        members.append(c)
        total += sum(k["nmem"] for k in decode(c.sweep())[0])
    g = H.Comm.group_plan(members)
    cls, lau, ptrs, _ = decode(g.sweep())
    assert sum(k["nmem"] for k in cls) == total
    assert sorted(ptrs) == sorted(p for c in members for p in decode(c.sweep())[2])
    assert [x["kernel"] for x in lau] == [FOLD, TEAM]         # the flat sum is sequential


@pytest.mark.parametrize("what,needle", [(3, "outside the primitives' buffers"), (4, "do not tile"),
                                         (5, "not an expression"), (6, "two steps")])
def test_corrupted_sweeps_are_caught_on_the_host(what, needle):
    """What a start launches is checked as the step table is: an operand outside
    the buffers, a missing unit, an unbalanced expression, an empty section."""
    prog = PR.reducescatter(16, 37)
    comm = register(prog, FakeAddresses(prog).addr)
    comm.plan([4, 4], 2, 2)
    comm.validate()
    comm.corrupt(what)
    with pytest.raises(H.HicclError) as e:
        comm.validate()
    assert e.value.status == H.ERR_INVALID
    assert needle in H.hiccl_last_error(comm.handle)


@pytest.mark.parametrize("what", range(7))
def test_corrupted_plans_do_not_run(what):
    """A corrupted plan is refused before any CUDA call, by itself and in a group."""
    prog = PR.allreduce(16, 37)
    comm = register(prog, FakeAddresses(prog).addr)
    comm.plan([4, 4], 2, 2)
    comm.corrupt(what)
    for run in (lambda: comm.init([4, 4], 2, 2), comm.run_static, lambda: H.Comm.group_plan([comm])):
        with pytest.raises(H.HicclError) as e:
            run()
        assert e.value.status == H.ERR_INVALID
