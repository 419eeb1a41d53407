"""Machines with fused entries (runs of instructions decoded when programs are
loaded; every test here asks rasp_describe whether they were), against the
oracle: programs of one to many mask records, the limits of 16 bits in an
entry, memories that differ from the loaded program, code read behind the
program that runs off the end of memory, and launch settings at the ends of
their range. Needs a GPU."""
import numpy as np
import pytest

from paper_2604_12902_gb300 import workloads as W
from tests.helpers import assert_same_state, oracle_state
from tests.test_gpu_fused import machines

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


def flat(progs, n, tapes, w=64, s=3, cap=3000, pvm=None):
    """A workload of the given programs (rows of equal or unequal length)."""
    V, ell = tapes.shape
    off = np.zeros(len(progs) + 1, np.uint64)
    off[1:] = np.cumsum([len(p) for p in progs])
    return W.Workload("entries", np.concatenate(progs).astype(np.int64), off, np.full(V, n, np.uint32),
                      tapes.astype(np.int64).reshape(-1), np.arange(V + 1, dtype=np.uint64) * np.uint64(ell),
                      np.full(V, cap, np.uint64), ell, s, w, pvm)


def check(rasp, wl, budgets, what, classic=False, i32=True, entries=True, **kw):
    """From c_0 twice through the budgets; `entries`: the programs have them."""
    flags = kw.pop("flags", 0) | (rasp.ISA_CLASSIC if classic else 0)
    with rasp.Batch(wl.mem_words, wl.ell, wl.s, word_bits=wl.w, flags=flags, **kw) as b:
        if i32:
            rasp.rasp_load_programs_i32(b.h, wl.programs, wl.prog_off, wl.prog_of_vm)
            b.load_inputs(wl.tapes, wl.tape_off, wl.caps)
        else:
            b.load_workload(wl)
        assert b.describe()["entries"] is entries, what
        for _ in range(2):
            for t in budgets:
                b.run(t)
                st, _ = oracle_state(wl, budget=t, threads=8, classic=classic)
                assert_same_state(b.read_state(), st, wl.ell, wl.s, what="%s, budget %d" % (what, t))
            b.reset()


@pytest.mark.parametrize("w", [64, 48, 32, 20, 11])
@pytest.mark.parametrize("m", [31, 64, 65, 130])
def test_programs_of_one_to_three_records(rasp, m, w):
    check(rasp, machines(700, m, w, seed=2000 * m + w, extra=2 * m + 8), [3, 20, 21, 200, 1000], "m=%d w=%d" % (m, w),
          i32=(m + w) % 2 == 0)


@pytest.mark.parametrize("w", [64, 48, 33, 32, 31])
@pytest.mark.parametrize("classic", [False, True])
def test_words_beyond_32_bits(rasp, w, classic):
    wl = machines(1500, 40, w, seed=140 + w, extra=90, huge=True)
    check(rasp, wl, [9, 60, 1000], "huge words w=%d" % w, classic=classic, i32=False)
    check(rasp, machines(700, 70, w, seed=105, extra=150), [7, 64, 1000], "classic %s w=%d" % (classic, w), classic=classic)


@pytest.mark.parametrize("p_code", [0.0, 0.3])
def test_long_programs_and_code_words(rasp, p_code):
    check(rasp, machines(150, 513, 64, seed=106, p_code=p_code, extra=1030), [100, 1000], "m=513 code %.1f" % p_code)


@pytest.mark.parametrize("w", [64, 32])
@pytest.mark.parametrize("V,m", [(33_000, 65), (25_000, 150)])
def test_programs_decoded_per_lane(rasp, V, m, w):
    """More than 24,000 machines: the decoder that takes a program per lane and
    keeps only the entries it reaches, over two and three mask records."""
    check(rasp, machines(V, m, w, seed=150 + w + m, extra=2 * m + 8), [40, 1000], "per lane m=%d w=%d" % (m, w), i32=w == 64)


def test_some_programs_write_into_themselves(rasp):
    """Half of the programs: the batch has entries, those programs run from memory."""
    a, c = W.random_programs(num_vms=512, seed=103, mem_words=200), machines(512, 32, 64, seed=113, extra=136)
    own = (np.arange(512) % 16 < 8)[:, None]
    prog = np.where(own, a.programs.reshape(512, -1), c.programs.reshape(512, -1))
    check(rasp, W.Workload("mixed", prog.reshape(-1), a.prog_off, c.mem_words, c.tapes, c.tape_off, c.caps, c.ell, c.s),
          [20, 1000], "half")


@pytest.mark.parametrize("w", [64, 32])
def test_restored_memories_run_from_memory(rasp, w):
    """A checkpoint whose memory differs from the loaded program's words; the
    next reset runs the loaded program again."""
    a, c = machines(300, 30, w, seed=111, extra=64), machines(300, 30, w, seed=112, extra=64)
    with rasp.Batch(a.mem_words, a.ell, a.s, word_bits=w) as b:
        b.load_workload(a)
        assert b.describe()["entries"]
        with rasp.Batch(c.mem_words, c.ell, c.s, word_bits=w) as d:
            d.load_workload(c)
            st = d.read_state()
        b.load_inputs(c.tapes, c.tape_off, c.caps)
        b.load_state(st)
        for t in (60, 500):
            b.run(t)
            assert_same_state(b.read_state(), oracle_state(c, budget=t, threads=8)[0], c.ell, c.s, what="restored")
        b.load_inputs(a.tapes, a.tape_off, a.caps)
        b.reset()
        b.run(500)
        assert_same_state(b.read_state(), oracle_state(a, budget=500, threads=8)[0], a.ell, a.s, what="reset")


# ---- the 16-bit fields of an entry
@pytest.mark.parametrize("w", [64, 32, 17])
@pytest.mark.parametrize("classic", [False, True])
def test_operands_around_65535(rasp, w, classic):
    wl = machines(120, 24, w, seed=160 + w, extra=70_000)
    n = int(wl.mem_words[0])
    rng = np.random.default_rng(w)
    prog = wl.programs.reshape(120, -1, 2)
    edge = rng.choice([65533, 65534, 65535, 65536, 65537, 65538, n - 2, n - 1, 60, 61], size=prog.shape[:2])
    mem = np.isin(prog[:, :, 0], (ADD, MUL, STO, RD, PRI)) & (rng.random(prog.shape[:2]) < .25)
    prog[:, :, 1] = np.where(mem, edge, prog[:, :, 1])
    check(rasp, wl, [25, 500], "operands at 2^16, w=%d" % w, classic=classic, i32=w != 17)


@pytest.mark.parametrize("m,entries", [(65_535, True), (65_536, False)])
@pytest.mark.parametrize("w", [64, 32])
def test_longest_programs(rasp, m, entries, w):
    """Jumps between the first and the last records of 65,535 instructions (one
    more has no entries), operands and wide constants (a + the program word at
    2p + 1) on both sides of word 65,535."""
    V, rng = 24, np.random.default_rng(m + w)
    op = rng.choice([LOD, ADD, BNZ, PRI, STO], size=(V, m), p=[.32, .34, .25, .05, .04])
    edge = lambda at, width: np.clip(at + rng.integers(-width, width, (V, m)), 0, None)
    pick = rng.integers(0, 4, (V, m))
    target = 2 * np.where(pick == 0, edge(40, 40), np.where(pick == 1, m - 1 - rng.integers(0, 70, (V, m)),
                          np.where(pick == 2, edge(32_767, 60), rng.integers(0, m, (V, m)))))
    word = np.where(pick == 0, edge(65_535, 4), rng.integers(0, 65_530, (V, m)))
    word = np.where(rng.random((V, m)) < .05, 2 * m - 1 - rng.integers(0, 9, (V, m)), word)
    const = np.where(pick == 0, rng.integers(40_000, 1 << 30, (V, m)), rng.integers(-2, 3, (V, m)))
    arg = np.where(op == BNZ, target, np.where(op == LOD, const, np.where(op == STO, 2 * m + 7 + pick, word)))
    prog = np.stack([op, arg], axis=2).reshape(V, 2 * m)
    wl = flat(list(prog), 4 * m + 40, np.zeros((V, 4)), w=w, s=40, cap=20_000)
    check(rasp, wl, [100, 20_000], "m=%d w=%d" % (m, w), entries=entries, i32=w == 32)


def code_from_the_tape(w, seed, V=224, programs=7, k=36):
    """Shared programs that read k instructions from the tape into the last
    2k words before n (w = 64) or 2^w, jump there and run on past the end,
    where i (+) 2 is reduced: the program starts again with i >= n (or i = 0)
    and reads the next k instructions, and the third time it halts."""
    rng = np.random.default_rng(seed)
    m = 2 * k + 3
    n = 4 * m + 10
    end = min(n, 1 << w)
    assert 2 * m <= end - 2 * k and n % 2 == 0
    progs = []
    for p in range(programs):
        ops = [(RD, end - 2 * k + q) for q in range(2 * k)]
        ops += [(LOD, p + 1), (BNZ, end - 2 * k + 2 * (p % 3)), (LOD, 5)]
        progs.append(np.array(ops).reshape(-1))
    data = np.arange(2 * m, end - 2 * k) if end < n else np.arange(2 * m, n - 2 * k)
    ops = rng.choice([LOD, ADD, MUL, STO, PRI], size=(V, 2 * k), p=[.3, .3, .1, .2, .1])
    arg = np.where(ops == LOD, rng.integers(0, 6, (V, 2 * k)), rng.choice(data, size=(V, 2 * k)))
    tapes = np.stack([ops, arg], axis=2).reshape(V, 4 * k)
    return flat(progs, n, tapes, w=w, pvm=rng.integers(0, programs, V).astype(np.uint32))


@pytest.mark.parametrize("epoch", [1, 7, 128])
@pytest.mark.parametrize("w", [64, 8])
def test_shared_machines_run_off_the_end_of_memory(rasp, w, epoch):
    """A machine of a shared program that runs code of its own over an odd
    number of steps ends an epoch at i (+) 2 = n (or 2^w): the next fetch is
    M[0], not the word behind the memory."""
    wl = code_from_the_tape(w, seed=70 + w)
    with rasp.Batch(wl.mem_words, wl.ell, wl.s, word_bits=w, flags=rasp.SCHED_SHARED, epoch=epoch) as b:
        b.load_workload(wl)
        assert b.describe()["entries"]
        for t in (90, 111, 112, 113, 250, 3000):
            b.run(t)
            st, _ = oracle_state(wl, budget=t, threads=8)
            assert_same_state(b.read_state(), st, wl.ell, wl.s, what="w %d epoch %d budget %d" % (w, epoch, t))
    assert (st.steps > 2 * (2 * 36 + 30)).all() and (st.status == 1).all()


@pytest.mark.parametrize("epoch", [1, (1 << 32) - 2, (1 << 32) - 1])
@pytest.mark.parametrize("shared", [False, True])
def test_smallest_and_largest_epochs(rasp, shared, epoch):
    """Every epoch takes a step: entries go in pairs, and the largest count of
    them must not round up to none."""
    wl = W.shared_programs(num_programs=4, vms_per_program=64) if shared else W.template_programs(num_vms=256, seed=7)
    flags = rasp.SCHED_SHARED if shared else rasp.SCHED_AUTO
    with rasp.Batch(wl.mem_words, wl.ell, wl.s, flags=flags, epoch=epoch) as b:
        b.load_workload(wl)
        assert b.describe()["entries"]
        for t in (50, 4096):
            b.run(t)
            st, _ = oracle_state(wl, budget=t, threads=8)
            assert_same_state(b.read_state(), st, wl.ell, wl.s, what="epoch %d budget %d" % (epoch, t))


def test_staged_buckets_keep_their_resident_warps(rasp):
    """Beside entries the SMEM-staged kernel is launched at its own occupancy."""
    small, large = (W.template_programs(num_vms=1 << 14, seed=s, mem_words=n) for s, n in ((3, 256), (4, 512)))
    V = 1 << 14
    wl = W.Workload("two sizes", np.concatenate([small.programs, large.programs]),
                    np.concatenate([small.prog_off, large.prog_off[1:] + small.prog_off[-1]]),
                    np.concatenate([small.mem_words, large.mem_words]), np.concatenate([small.tapes, large.tapes]),
                    np.concatenate([small.tape_off, large.tape_off[1:] + small.tape_off[-1]]),
                    np.concatenate([small.caps, large.caps]), small.ell, small.s)
    with rasp.Batch(wl.mem_words, wl.ell, wl.s) as b:
        b.load_workload(wl)
        k = b.describe()["buckets"][0]
        b.plan_bucket(k["index"], rasp.SCHED_PERSIST)
        d = b.describe()
        assert d["entries"] and [x["schedule"] for x in d["launches"]] == ["persist", "persist_gl"]
        k = d["buckets"][0]
        assert k["ctas_per_sm"] >= 3 and d["launches"][0]["grid"] == min(k["grid"], V // 32)
        b.run()
        st, _ = oracle_state(wl, threads=8)
        assert_same_state(b.read_state(), st, wl.ell, wl.s, what="staged beside entries")


def test_reading_the_largest_padded_slabs(rasp):
    """Equal memories of 2^27 words on the shared-program schedule: two of them
    are more bytes than a strided copy takes as a pitch."""
    n, V = 1 << 27, 3
    prog = np.array([LOD, 7, STO, n - 1, LOD, 9, STO, 100, RD, 101, 0, 0])
    wl = flat([prog], n, np.arange(1, V + 1).reshape(V, 1), pvm=np.zeros(V, np.uint32))
    want = {1: 7, 2: STO, 0: LOD, 3: n - 1, 4: LOD, 5: 9, 6: STO, 7: 100, 8: RD, 9: 101, 100: 9, n - 1: 7}
    with rasp.Batch(wl.mem_words, wl.ell, wl.s, flags=rasp.SCHED_SHARED) as b:
        b.load_workload(wl)
        b.run()
        for first, count in ((0, 3), (1, 2)):
            got = b.read_state(first, count)
            assert (got["steps"] == 5).all() and (got["status"] == 1).all()
            for k, slab in enumerate(got.pop("mem").reshape(count, n)):
                at = np.flatnonzero(slab)
                assert dict(zip(at.tolist(), slab[at].tolist())) == {**want, 101: first + k + 1}


def test_autotune_after_a_run_that_wrote_code(rasp):
    """The plain schedule has written HALT over the first instruction of an
    endless loop: the autotuner's trials must run that memory, where every
    machine halts at once, and not the loaded program's entries."""
    at = 14
    prog = [LOD, 0, STO, 2 * at] + [LOD, 1] * (at - 2) + [LOD, 1, ADD, 60, STO, 60, BNZ, 2 * at]
    wl = flat([np.array(prog)] * 64, 96, np.zeros((64, 2)), cap=1 << 40)
    with rasp.Batch(wl.mem_words, wl.ell, wl.s) as b:
        b.load_workload(wl)
        assert b.describe()["entries"]
        k = b.describe()["buckets"][0]["index"]
        b.plan_bucket(k, rasp.SCHED_PLAIN)
        b.run(5)
        rep = b.autotune(max_steps=10_000_000, reps=1)
        ms = {t["schedule"]: t["ms"] for t in rep["trials"]}
        assert max(v for name, v in ms.items() if name.startswith("persist_gl")) < 20, ms   # the loop takes seconds
        b.run()
        st, _ = oracle_state(wl, threads=8)
        assert_same_state(b.read_state(), st, wl.ell, wl.s, what="after autotune")


# ---- operands that no entry holds: words behind 65,535, wide constants of shared programs
def stalling(V, n, far, every, shared=False, turns=300):
    """Counter loops of 10 steps; in every `every`-th program the loop reads
    and writes word `far` (or, of shared programs, loads a wide constant)."""
    near = [LOD, turns, STO, 100, LOD, 1, ADD, 101, STO, 101, LOD, 3, ADD, 102, STO, 102, LOD, -1, ADD, 100, STO, 100,
            BNZ, 4, PRI, 101, 0, 0]
    prog = np.tile(np.array(near), (V // 32 if shared else V, 1))
    if shared:
        prog[::every, 5], prog[::every, 11] = 100_000, 70_000
    else:
        prog[::every, 7] = prog[::every, 9] = prog[::every, 25] = far
    wl = flat(list(prog), n, np.zeros((V, 2)), cap=10 ** 6, pvm=np.repeat(np.arange(len(prog)), 32).astype(np.uint32) if shared else None)
    return wl


@pytest.mark.parametrize("w", [64, 32, 18])
@pytest.mark.parametrize("every", [3, 33])
def test_machines_that_leave_their_entries(rasp, w, every):
    wl = stalling(384, 70_000, 66_000, every)
    wl.w = w
    check(rasp, wl, [17, 100, 1000, 10_000], "far operands in one of %d, w=%d" % (every, w))
    wl = stalling(768, 256, 0, every, shared=True)
    wl.w = w
    for flags in (rasp.SCHED_SHARED, rasp.SCHED_AUTO):
        check(rasp, wl, [17, 100, 1000, 10_000], "wide constants in one of %d, w=%d" % (every, w), flags=flags)


def test_most_machines_stall(rasp):
    """No entries where most programs would leave them."""
    wl = stalling(256, 70_000, 66_000, 1)
    check(rasp, wl, [1000, 10_000], "far operands", entries=False)
    wl = stalling(512, 256, 0, 1, shared=True)
    for flags in (rasp.SCHED_SHARED, rasp.SCHED_AUTO):
        check(rasp, wl, [1000, 10_000], "wide constants", flags=flags, entries=False)


def test_stalls_do_not_hold_the_warp(rasp):
    """Half of the programs load two wide constants in 12 instructions: machines
    that stall all the time run on from memory (2 times the time of small
    constants; 9 times if they stay)."""
    import torch
    stream, ms = torch.cuda.current_stream(), []
    for every in (1 << 20, 2):
        wl = stalling(65_536, 256, 0, every, shared=True, turns=2000)
        wl.programs.reshape(2048, -1)[0] = wl.programs.reshape(2048, -1)[1]
        with rasp.Batch(wl.mem_words, wl.ell, wl.s, flags=rasp.SCHED_SHARED) as b:
            b.load_workload(wl)
            assert b.describe()["entries"]
            took = []
            for _ in range(4):
                b.reset()
                e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
                e[0].record(stream)
                b.run()
                e[1].record(stream)
                torch.cuda.synchronize()
                took.append(e[0].elapsed_time(e[1]))
            ms.append(min(took))
    assert ms[1] < 4.5 * ms[0], ms


@pytest.mark.parametrize("i32", [False, True])
@pytest.mark.parametrize("sched", [0x10, 0x20], ids=["plain", "staged"])
def test_entries_only_where_a_plan_runs_from_them(rasp, sched, i32):
    """The plain and SMEM-staged schedules load without decoding; a plan that
    moves to the HBM-slab schedule (pinned or autotuned, also midway, under a
    graph, with programs shared) decodes before it runs."""
    for shared in (0, 9):
        wl = machines(600, 40, 64, seed=170 + shared, extra=100, shared=shared)
        part, full = (oracle_state(wl, budget=t, threads=8)[0] for t in (33, 1000))
        for how in ("pinned", "midway", "autotuned"):
            with rasp.Batch(wl.mem_words, wl.ell, wl.s, flags=sched | rasp.CUDA_GRAPH) as b:
                load = rasp.rasp_load_programs_i32 if i32 else rasp.rasp_load_programs
                load(b.h, wl.programs, wl.prog_off, wl.prog_of_vm)
                b.load_inputs(wl.tapes, wl.tape_off, wl.caps)
                assert not b.describe()["entries"]
                if how != "pinned":
                    b.run(33)
                    assert_same_state(b.read_state(), part, wl.ell, wl.s, what=how)
                    assert not b.describe()["entries"]
                if how == "autotuned":
                    b.autotune(max_steps=1000, reps=1)
                    assert b.describe()["entries"]
                else:
                    for k in b.describe()["buckets"]:
                        b.plan_bucket(k["index"], rasp.SCHED_PERSIST_GL)
                for _ in range(2):
                    b.run(1000)
                    assert b.describe()["entries"]
                    assert_same_state(b.read_state(), full, wl.ell, wl.s, what=how)
                    b.reset()


def test_launch_settings_hold_for_few_machines(rasp):
    """Few VMs spread over one-warp CTAs only where neither warps_per_cta nor
    ctas_per_sm is set, in the configuration or for a bucket."""
    wl = W.template_programs(num_vms=2048, seed=5)
    st, _ = oracle_state(wl, threads=8)
    for kw, want in (({}, None), (dict(warps_per_cta=4), (16, 4, 32)), (dict(warps_per_cta=2), (32, 2, 32)),
                     (dict(ctas_per_sm=5), (16, 4, 32))):
        for pin in (False, True):
            with rasp.Batch(wl.mem_words, wl.ell, wl.s, **({} if pin else kw)) as b:
                b.load_workload(wl)
                if pin:
                    b.plan_bucket(b.describe()["buckets"][0]["index"], rasp.SCHED_PERSIST_GL, **kw)
                got = b.describe()["launches"][0]
                got = got["grid"], got["warps_per_cta"], got["lanes_per_warp"]
                if want is None:
                    assert got[1] == 1 and got[2] < 32 and got[0] * got[2] >= 2048, got
                else:
                    assert got == want
                b.run()
                assert_same_state(b.read_state(), st, wl.ell, wl.s, what=str(kw))


@pytest.mark.parametrize("V", [1, 33, 6100, 8192, 9800])
def test_lanes_of_few_machines(rasp, V):
    """One-warp CTAs of as many lanes as eight warps per SM take, at their
    edges; programs that write into themselves run on four lanes in place of
    five to eight."""
    import torch
    spread = 8 * torch.cuda.get_device_properties(0).multi_processor_count
    lanes = -(-V // spread)
    for wl, own in ((W.template_programs(num_vms=V, seed=6), False), (W.random_programs(num_vms=V, seed=6), True)):
        st, _ = oracle_state(wl, threads=8)
        with rasp.Batch(wl.mem_words, wl.ell, wl.s) as b:
            b.load_workload(wl)
            got, want = b.describe()["launches"][0], 4 if own and 4 < lanes <= 8 else lanes
            assert (got["warps_per_cta"], got["lanes_per_warp"], got["grid"]) == (1, want, -(-V // want))
            b.run()
            assert_same_state(b.read_state(), st, wl.ell, wl.s, what="%s %d" % (wl.name, V))


def test_budget_rounds_by_kind(rasp):
    """Between half and all of the resident lanes, batches run in budget rounds
    unless their programs write into themselves."""
    import torch
    V = 152 * 7 * 128 * 3 // 4 if torch.cuda.get_device_properties(0).multi_processor_count == 152 else 100_000
    for wl, rounds in ((W.template_programs(num_vms=V, seed=8, cap=5000), True),
                       (W.random_programs(num_vms=V, seed=8, cap=5000), False)):
        st, _ = oracle_state(wl, threads=8)
        with rasp.Batch(wl.mem_words, wl.ell, wl.s) as b:
            b.load_workload(wl)
            b.run()
            assert (b.stats()["launches"] > 1) is rounds, wl.name
            assert_same_state(b.read_state(), st, wl.ell, wl.s, what=wl.name)


@pytest.mark.parametrize("w", [32, 20])
def test_pools_of_small_words(rasp, w):
    """A pool's requests hold 8-byte words at every w: their size is asked for so."""
    from paper_2604_12902_gb300 import serving
    wl = machines(900, 40, w, seed=180 + w, extra=100)
    st, _ = oracle_state(wl, threads=8)
    with serving.Pool(1 << 26, wl.ell, wl.s, word_bits=w) as pool:
        tickets = [pool.submit(wl) for _ in range(3)]
        for t in tickets:
            assert_same_state(pool.read(t), st, wl.ell, wl.s, what="pool, w = %d" % w)


@pytest.mark.parametrize("sched,w", [(0x00, 64), (0x00, 32), (0x40, 64), (0x20, 64)])
def test_arenas_without_room_for_entries(rasp, sched, w):
    """A caller's arena that lacks only the room for entries and between slabs
    (16 bytes per 128 words and per VM, 32 bytes after every second slab) holds
    the batch without them; a smaller one is refused."""
    import ctypes
    import torch
    V = 999
    wl = machines(V, 30, w, seed=190 + w + sched, extra=90, shared=40 if sched == 0x40 else 0)
    st, _ = oracle_state(wl, threads=8)
    cfg = rasp.rasp_config(w, 0, wl.ell, wl.s, sched, 0, 0, 0, 0, 0, None, None, 0)
    pad = (V - 1) // 2 * 4
    words = int((wl.mem_words.astype(np.int64) + 1 & ~1).sum()) + pad
    lean = rasp.rasp_batch_bytes(cfg, wl.mem_words) - 16 * (words // 128 + V + 1) - (8 + (4 if w == 32 else 8)) * pad
    arena = torch.empty(lean + 1024, dtype=torch.uint8, device="cuda")
    cfg.arena = ctypes.c_void_p(arena.data_ptr())
    for size, ok in ((lean + 1024, True), (lean - 2048, False)):
        cfg.arena_bytes = size
        if not ok:
            with pytest.raises(rasp.RaspError):
                rasp.rasp_batch_create(cfg, wl.mem_words)
            continue
        b = rasp.Batch.__new__(rasp.Batch)
        b.mem_words, b.V, b.ell, b.s, b.w, b.cfg, b._arena = wl.mem_words, V, wl.ell, wl.s, w, cfg, arena
        b.h, b.n_total = rasp.rasp_batch_create(cfg, wl.mem_words), int(wl.mem_words.sum())
        with b:
            b.load_workload(wl)
            assert not b.describe()["entries"]
            for _ in range(2):
                b.run()
                assert_same_state(b.read_state(), st, wl.ell, wl.s, what="lean arena")
                b.reset()


def test_pools_without_room_for_entries(rasp):
    from paper_2604_12902_gb300 import serving
    V = 20_000
    wl = W.template_programs(num_vms=V, seed=12)
    st, _ = oracle_state(wl, threads=8)
    cfg = rasp.rasp_config(64, 0, wl.ell, wl.s, 0, 0, 0, 0, 0, 0, None, None, 0)
    with serving.Pool(rasp.rasp_batch_bytes(cfg, wl.mem_words) - 32 * V, wl.ell, wl.s) as pool:
        for _ in range(2):
            assert_same_state(pool.read(pool.submit(wl)), st, wl.ell, wl.s, what="lean pool")


@pytest.mark.parametrize("flags", [0x0, 0x4000], ids=["eager", "cuda-graph"])
@pytest.mark.parametrize("w", [64, 32])
def test_short_runs_of_new_programs(rasp, w, flags):
    """Programs loaded after inputs with small caps are decoded by the second
    run, whether it starts from c_0 or goes on from memories that the first
    has written code into; with larger caps or steps by the load or the run."""
    wl = machines(700, 60, w, seed=200 + w, extra=130, p_code=0.2)
    short = np.minimum(wl.caps, 250)
    with rasp.Batch(wl.mem_words, wl.ell, wl.s, word_bits=w, flags=flags) as b:
        def load(caps):
            wl.caps = caps
            b.load_inputs(wl.tapes, wl.tape_off, caps)
            b.load_programs(wl.programs, wl.prog_off)

        def run(t, entries):
            b.run(t)
            assert b.describe()["entries"] is entries
            assert_same_state(b.read_state(), oracle_state(wl, budget=t, threads=8)[0], wl.ell, wl.s, what="%d" % t)

        long = wl.caps.copy()
        for _ in range(2):
            load(short)
            run(1000, False)
            b.reset()
            run(30, True)
            run(1000, True)
            load(short)
            run(40, False)
            run(90, True)                     # from memories without marks
            run(1000, True)
            b.reset()
            run(1000, True)
            load(long)
            run(30, True)
            run(1000, True)
            load(short)
            wl.caps = long
            b.load_inputs(wl.tapes, wl.tape_off, long)
            run(1000, True)


@pytest.mark.parametrize("shared", [0, 40])
@pytest.mark.parametrize("warm", [False, True])
def test_short_runs_in_the_callers_graph(rasp, shared, warm):
    """A run that the caller captures decodes nothing; its replays, which keep
    no marks, mix with later runs."""
    import torch
    wl = machines(600, 60, 64, seed=210 + shared, extra=130, p_code=0.2, shared=shared)
    wl.caps = np.minimum(wl.caps, 250)
    part, full = (oracle_state(wl, budget=t, threads=8)[0] for t in (60, 1000))
    side = torch.cuda.Stream()
    with torch.cuda.stream(side), rasp.Batch(wl.mem_words, wl.ell, wl.s) as b:
        b.load_inputs(wl.tapes, wl.tape_off, wl.caps)
        for _ in range(2):
            b.load_programs(wl.programs, wl.prog_off, wl.prog_of_vm)
            assert b.describe()["entries"] is bool(shared)   # (shared: few instructions for each machine)
            if warm:
                b.run(60)
                b.reset()
            side.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=side):
                b.run(60)
            for _ in range(2):
                g.replay()
                assert_same_state(b.read_state(), part, wl.ell, wl.s, what="replay")
                b.run(1000)
                assert_same_state(b.read_state(), full, wl.ell, wl.s, what="run on")
                b.reset()
            assert b.describe()["entries"]


@pytest.mark.parametrize("w", [64, 32])
def test_callers_graphs_and_the_marks(rasp, w):
    """Replays of a run captured on the plain schedule write program words
    without marks; marks set inside a capture are not there before its replay."""
    import torch
    wl = machines(600, 60, w, seed=220 + w, extra=130, p_code=0.2)
    full = oracle_state(wl, threads=8)[0]
    side = torch.cuda.Stream()

    def batch():
        b = rasp.Batch(wl.mem_words, wl.ell, wl.s, word_bits=w)
        b.load_workload(wl)
        assert b.describe()["entries"]
        return b, b.describe()["buckets"][0]["index"]

    def capture(b, t):
        side.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            b.run(t)
        return g

    with torch.cuda.stream(side):
        b, k = batch()
        b.plan_bucket(k, rasp.SCHED_PLAIN)
        g = capture(b, 60)
        b.plan_bucket(k, rasp.SCHED_PERSIST_GL)
        for rep in range(3):
            if rep == 2:
                b.load_inputs(wl.tapes, wl.tape_off, wl.caps)
                b.load_programs(wl.programs, wl.prog_off)
            g.replay()
            b.run()
            assert_same_state(b.read_state(), full, wl.ell, wl.s, what="replayed on the plain schedule, %d" % rep)
            b.reset()
        b.close()

        b, k = batch()
        h = capture(b, 1 << 62)
        for rep in range(2):
            b.plan_bucket(k, rasp.SCHED_PLAIN)
            if rep == 0:
                b.run(60)
                g = capture(b, 60)
            else:
                g.replay()
            h.replay()
            assert_same_state(b.read_state(), full, wl.ell, wl.s, what="entries replayed after the plain schedule")
            b.reset()
        b.close()

        b, k = batch()
        b.plan_bucket(k, rasp.SCHED_PLAIN)
        b.run(60)
        b.plan_bucket(k, rasp.SCHED_PERSIST_GL)
        g = capture(b, 200)
        b.run()
        assert_same_state(b.read_state(), full, wl.ell, wl.s, what="marks captured, not replayed")
        b.reset()
        g.replay()
        b.run()
        assert_same_state(b.read_state(), full, wl.ell, wl.s, what="replayed after a reset")
        b.close()


def test_new_inputs_of_a_callers_graph(rasp):
    """u_0 = 0 of new inputs is not owed until after the replay that reads them."""
    import torch
    side = torch.cuda.Stream()
    a, c = (machines(600, 60, 64, seed=seed, extra=130) for seed in (230, 231))
    with torch.cuda.stream(side), rasp.Batch(a.mem_words, a.ell, a.s) as b:
        b.load_workload(a)
        b.run()
        side.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            b.run()
        for wl in (c, a):
            b.load_workload(wl)
            g.replay()
            assert_same_state(b.read_state(), oracle_state(wl, threads=8)[0], wl.ell, wl.s, what="new inputs")


def test_a_first_run_in_a_callers_graph(rasp):
    """A graph captured right after the loads does not reset u_0: nothing has
    moved it since the pack."""
    import torch
    side = torch.cuda.Stream()
    wl = machines(600, 60, 64, seed=232, extra=130)
    full = oracle_state(wl, threads=8)[0]
    with torch.cuda.stream(side), rasp.Batch(wl.mem_words, wl.ell, wl.s) as b:
        b.load_workload(wl)
        side.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            b.run()
        for t in (0, 40, 90):
            if t:
                b.run(t)
            g.replay()
            assert_same_state(b.read_state(), full, wl.ell, wl.s, what="after %d steps" % t)
            b.reset()
        g.replay()
        b.load_inputs(wl.tapes, wl.tape_off, wl.caps)
        assert not b.read_state()["uhead"].any()


def test_new_programs_under_a_callers_graph(rasp):
    """A graph that the caller has captured holds the place of the entries:
    loads that move them, have none or fail leave its replays right."""
    import torch
    side = torch.cuda.Stream()
    n = 250
    kinds = [machines(500, m, 64, seed=240 + m, extra=n - 2 * m, p_code=0.05) for m in (60, 20, 41)]
    kinds.append(W.random_programs(num_vms=500, seed=244, mem_words=n, tape_len=5, s=3, cap=600))
    kinds.append(kinds[0])
    full = [oracle_state(wl, threads=8)[0] for wl in kinds]
    for i32 in (False, True):
        with torch.cuda.stream(side), rasp.Batch(kinds[0].mem_words, 5, 3) as b:
            def load(wl):
                b.load_inputs(wl.tapes, wl.tape_off, wl.caps)
                (rasp.rasp_load_programs_i32 if i32 else rasp.rasp_load_programs)(b.h, wl.programs, wl.prog_off)

            load(kinds[0])
            assert b.describe()["entries"]
            b.run()
            side.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=side):
                b.run()
            for k, (wl, st) in enumerate(zip(kinds, full)):
                load(wl)
                assert b.describe()["entries"] is (k < 3 if i32 else k == 0)   # int32 words: one place for all
                g.replay()
                assert_same_state(b.read_state(), st, wl.ell, wl.s, what="kind %d" % k)
                b.reset()
                b.run(40)
                g.replay()
                assert_same_state(b.read_state(), st, wl.ell, wl.s, what="kind %d, after a run" % k)


def test_a_failed_load_under_a_callers_graph(rasp):
    import torch
    side = torch.cuda.Stream()
    wl = machines(500, 60, 64, seed=250, extra=130)
    full = oracle_state(wl, threads=8)[0]
    bad = np.arange(501, dtype=np.uint64) * np.uint64(220)       # words over the entries of those before
    bad[7] += 1                                                  # an odd length
    with torch.cuda.stream(side), rasp.Batch(wl.mem_words, wl.ell, wl.s) as b:
        b.load_workload(wl)
        b.run()
        side.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            b.run()
        b.reset()
        b.run(25)
        junk = np.full(500 * 220, 0x4444444444444444, np.int64)
        with pytest.raises(rasp.RaspError):
            b.load_programs(junk, bad)
        g.replay()
        assert_same_state(b.read_state(), full, wl.ell, wl.s, what="after a failed load")
        b.load_workload(wl)
        g.replay()
        assert_same_state(b.read_state(), full, wl.ell, wl.s, what="loaded again")


@pytest.mark.parametrize("flags", [0x40, 0x4040], ids=["shared", "shared, own graph too"])
def test_shared_programs_under_a_callers_graph(rasp, flags):
    import torch
    side = torch.cuda.Stream()
    kinds = [machines(700, m, 64, seed=260 + m, extra=240 - 2 * m, shared=30, p_code=0.05) for m in (60, 25)]
    for wl in kinds:
        wl.mem_words[:] = 240
    full = [oracle_state(wl, threads=8)[0] for wl in kinds]
    with torch.cuda.stream(side), rasp.Batch(kinds[0].mem_words, 5, 3, flags=flags) as b:
        b.load_workload(kinds[0])
        b.run()
        side.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            b.run()
        for k in (0, 1, 0):
            wl = kinds[k]
            b.load_inputs(wl.tapes, wl.tape_off, wl.caps)
            b.load_programs(wl.programs, wl.prog_off, wl.prog_of_vm)
            for _ in range(2):
                g.replay()
                assert_same_state(b.read_state(), full[k], wl.ell, wl.s, what="kind %d" % k)
                b.reset()
                b.run()
                assert_same_state(b.read_state(), full[k], wl.ell, wl.s, what="kind %d, run" % k)
                b.reset()
