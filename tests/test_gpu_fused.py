"""Fused entries (runs of instructions decoded when programs are loaded)
against the oracle, at the sizes and forms where they can go wrong: programs
around the 64 instructions of a mask record, jumps back to earlier records,
jumps on constants, wide constants, program words read and written as data,
operands at the end of memory, runs stopped inside an entry and resumed, and
programs shared by machines of different memories. Needs a GPU."""
import numpy as np
import pytest

from paper_2604_12902_gb300 import workloads as W
from tests.helpers import assert_same_state, oracle_state

pytestmark = pytest.mark.gpu
LOD, ADD, MUL, STO, BNZ, RD, PRI = 1, 2, 3, 4, 5, 6, 7


@pytest.fixture(scope="module")
def rasp():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_12902_gb300 import rasp as R
    R.lib()
    return R


def machines(V, m, w, seed, extra=24, p_code=0.02, shared=0, huge=False):
    """V machines of m instructions: opcodes weighted to the fused form, small
    and wide constants, data words mostly behind the program, jump targets
    mostly even; a few operands in the program or past the memory."""
    rng = np.random.default_rng(seed)
    P = shared or V
    n = 2 * m + extra
    op = rng.choice([LOD, ADD, MUL, STO, BNZ, RD, PRI, 0, 9], size=(P, m),
                    p=[.30, .24, .08, .17, .12, .04, .03, .01, .01])
    data = rng.integers(2 * m, n, (P, m))
    near = rng.integers(2 * m, 2 * m + 4, (P, m))                 # the same few words: stores that are read at once
    arg = np.where(rng.random((P, m)) < .5, near, data)
    arg = np.where(rng.random((P, m)) < p_code, rng.integers(0, 2 * m, (P, m)), arg)
    arg = np.where(rng.random((P, m)) < .01, rng.integers(n, n + 3, (P, m)), arg)
    target = 2 * rng.integers(0, m, (P, m)) + (rng.random((P, m)) < .03)
    wide = rng.choice([-1, 1, 0, 2, -32768, 32767, 32768, 70000, -(1 << 31), (1 << 31) - 1], size=(P, m))
    if huge:                                                      # words of 8 bytes only
        far = [1 << 31, (1 << 32) - 1, (1 << 32) + 1, 1 << 62, -(1 << 63), -(1 << 40) + 4, (1 << 48) - 1]
        wide = np.where(rng.random((P, m)) < .5, wide, rng.choice(far, size=(P, m)))
        op = np.where(rng.random((P, m)) < .01, (1 << 32) + op, op)
    const = np.where(rng.random((P, m)) < .1, wide, rng.integers(-3, 4, (P, m)))
    arg = np.where(op == BNZ, target, np.where(op == LOD, const, arg))
    if huge:
        arg = np.where(rng.random((P, m)) < .02, wide, arg)
    prog = np.empty((P, 2 * m), np.int64)
    prog[:, 0::2], prog[:, 1::2] = op, arg
    ell, s = 5, 3
    tape = rng.integers(-1000, 1000, V * ell)
    caps = rng.integers(1, 900, V).astype(np.uint64)
    pvm = rng.integers(0, P, V).astype(np.uint32) if shared else None
    mem = (n + rng.integers(0, 9, V) if shared else np.full(V, n)).astype(np.uint32)
    return W.Workload("fused", prog.reshape(-1), np.arange(P + 1, dtype=np.uint64) * np.uint64(2 * m), mem, tape,
                      np.arange(V + 1, dtype=np.uint64) * np.uint64(ell), caps, ell, s, w, pvm)


def check(rasp, wl, budgets, what, classic=False, i32=True, **kw):
    flags = kw.pop("flags", 0) | (rasp.ISA_CLASSIC if classic else 0)
    with rasp.Batch(wl.mem_words, wl.ell, wl.s, word_bits=wl.w, flags=flags, **kw) as b:
        if i32:
            rasp.rasp_load_programs_i32(b.h, wl.programs, wl.prog_off, wl.prog_of_vm)
            b.load_inputs(wl.tapes, wl.tape_off, wl.caps)
        else:
            b.load_workload(wl)
        for _ in range(2):                                        # from c_0 twice: a reset forgets written programs
            for t in budgets:
                b.run(t)
                st, _ = oracle_state(wl, budget=t, threads=8, classic=classic)
                assert_same_state(b.read_state(), st, wl.ell, wl.s, what="%s, budget %d" % (what, t))
            b.reset()


@pytest.mark.parametrize("w", [64, 48, 32, 20, 6])
@pytest.mark.parametrize("m", [1, 2, 31, 64, 65, 130])
def test_entries_match_the_oracle(rasp, m, w):
    wl = machines(700, m, w, seed=1000 * m + w)
    check(rasp, wl, [3, 20, 21, 200, 1000], "m=%d w=%d" % (m, w), i32=(m + w) % 2 == 0)


@pytest.mark.parametrize("w", [64, 48, 33, 32, 31])
@pytest.mark.parametrize("classic", [False, True])
def test_words_beyond_32_bits(rasp, w, classic):
    wl = machines(1500, 40, w, seed=40 + w, huge=True)
    check(rasp, wl, [9, 60, 1000], "huge words w=%d" % w, classic=classic, i32=False)


@pytest.mark.parametrize("w", [64, 32])
def test_classic_set(rasp, w):
    check(rasp, machines(700, 70, w, seed=5), [7, 64, 1000], "classic w=%d" % w, classic=True)


@pytest.mark.parametrize("p_code", [0.0, 0.3])
def test_long_programs_and_code_words(rasp, p_code):
    check(rasp, machines(150, 513, 64, seed=6, p_code=p_code), [100, 1000], "m=513 code %.1f" % p_code)
    check(rasp, machines(300, 64, 64, seed=7, p_code=p_code, extra=2), [50, 1000], "no room beside the program")


@pytest.mark.parametrize("first,count", [(0, 1), (0, 8), (3, 30), (8, 16), (5, 2), (61, 3), (0, 64)])
def test_reading_ranges_of_padded_slabs(rasp, first, count):
    wl = machines(64, 20, 64, seed=60, shared=5)
    wl.mem_words[:] = int(wl.mem_words.max()) + 1 & ~1
    with rasp.Batch(wl.mem_words, wl.ell, wl.s, flags=rasp.SCHED_SHARED) as b:
        b.load_workload(wl)
        b.run(300)
        whole = b.read_state()["mem"].reshape(64, -1)
        st, _ = oracle_state(wl, budget=300)
        assert np.array_equal(whole.reshape(-1).view(np.uint64), st.mem)
        assert np.array_equal(b.read_state(first, count)["mem"].reshape(count, -1), whole[first:first + count])


@pytest.mark.parametrize("w", [64, 32])
def test_many_short_programs(rasp, w):
    """Enough instructions (over 2^21) for the decoder that takes a program per
    lane and keeps only the entries it reaches."""
    wl = machines(33_000, 65, w, seed=50 + w)
    check(rasp, wl, [40, 1000], "per lane w=%d" % w, i32=w == 64)


def test_shared_programs_on_several_memory_sizes(rasp):
    wl = machines(1500, 40, 64, seed=8, shared=37)
    check(rasp, wl, [30, 1000], "prog_of_vm", i32=False)
    check(rasp, wl, [30, 1000], "prog_of_vm int32")


@pytest.mark.parametrize("w", [64, 20])
@pytest.mark.parametrize("m", [1, 40, 64, 129])
def test_shared_program_schedule(rasp, m, w):
    """Entries in shared memory beside the program, VMs that read and write
    program words, memories read back midway (which fills the slabs)."""
    for p_code in (0.0, 0.1):
        wl = machines(900, m, w, seed=20 + m + w, shared=11, p_code=p_code)
        check(rasp, wl, [30, 31, 1000], "shared m=%d w=%d code %.1f" % (m, w, p_code), flags=rasp.SCHED_SHARED,
              i32=m != 40)


@pytest.mark.parametrize("classic", [False, True])
@pytest.mark.parametrize("m", [8, 64])
def test_checked_loop(rasp, m, classic):
    """The epoch loop under CHECKED semantics: overflows of large data at every
    step of a run, faulting addresses and fetches, runs stopped and resumed."""
    wl = machines(900, m, 64, seed=30 + m)
    rng = np.random.default_rng(m)
    big = rng.integers(-(1 << 31), 1 << 31, wl.tapes.size) << rng.choice([0, 16, 32], wl.tapes.size)
    wl.tapes = big.astype(np.int64)
    prog = wl.programs.reshape(900, -1)
    prog[:, 0:2 * min(4, m // 2):2], prog[:, 1:2 * min(4, m // 2):2] = RD, 2 * m + np.arange(min(4, m // 2))
    flags = rasp.ISA_CLASSIC if classic else 0
    with rasp.Batch(wl.mem_words, wl.ell, wl.s, semantics=rasp.CHECKED, flags=flags) as b:
        b.load_workload(wl)
        for t in (5, 6, 100, 1000):
            b.run(t)
            st, _ = oracle_state(wl, budget=t, threads=8, checked=True, classic=classic)
            assert_same_state(b.read_state(), st, wl.ell, wl.s, what="checked, budget %d" % t)
    assert {3, 4} <= set(st.status.tolist()) and (st.steps[st.status == 3] > 6).any()


def test_self_writing_programs(rasp):
    """Batches in which all, some or few programs mostly write into themselves."""
    a = W.random_programs(num_vms=512, seed=3, mem_words=200)
    check(rasp, a, [20, 256], "all")
    c = machines(512, 32, 64, seed=13, extra=136)
    for every in (2, 9):
        own = (np.arange(512) % every == 0)[:, None]
        prog = np.where(own, a.programs.reshape(512, -1), c.programs.reshape(512, -1))
        wl = W.Workload("mixed", prog.reshape(-1), a.prog_off, c.mem_words, c.tapes, c.tape_off, c.caps, c.ell, c.s)
        check(rasp, wl, [20, 1000], "every %d" % every)


def test_reloading_other_programs_under_a_graph(rasp):
    """A captured run must not keep the entries of the programs loaded before."""
    a, c = machines(600, 20, 64, seed=9, extra=120), machines(600, 60, 64, seed=10, extra=40)
    assert np.array_equal(a.mem_words, c.mem_words)
    with rasp.Batch(a.mem_words, a.ell, a.s, flags=rasp.CUDA_GRAPH) as b:
        for wl in (a, c, a):
            b.load_workload(wl)
            b.run(400)
            st, _ = oracle_state(wl, budget=400, threads=8)
            assert_same_state(b.read_state(), st, wl.ell, wl.s, what="reload")


def test_restored_memories_run_from_memory(rasp):
    """A checkpoint whose memory differs from the loaded program's words."""
    a, c = machines(300, 30, 64, seed=11), machines(300, 30, 64, seed=12)
    with rasp.Batch(a.mem_words, a.ell, a.s) as b:
        b.load_workload(a)
        with rasp.Batch(c.mem_words, c.ell, c.s) as d:
            d.load_workload(c)
            st = d.read_state()
        b.load_inputs(c.tapes, c.tape_off, c.caps)
        b.load_state(st)
        b.run(500)
        want, _ = oracle_state(c, budget=500, threads=8)
        assert_same_state(b.read_state(), want, c.ell, c.s, what="restored")
