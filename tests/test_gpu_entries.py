"""Machines beside their fused entries (runs of instructions decoded when
programs are loaded), against the oracle: code stored or read behind the
program that runs off the end of memory, and launch settings at the ends of
their range. Needs a GPU."""
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


def flat(progs, n, tapes, w=64, s=3, cap=3000, pvm=None):
    """A workload of the given programs (rows of equal or unequal length)."""
    V, ell = tapes.shape
    off = np.zeros(len(progs) + 1, np.uint64)
    off[1:] = np.cumsum([len(p) for p in progs])
    return W.Workload("entries", np.concatenate(progs).astype(np.int64), off, np.full(V, n, np.uint32),
                      tapes.astype(np.int64).reshape(-1), np.arange(V + 1, dtype=np.uint64) * np.uint64(ell),
                      np.full(V, cap, np.uint64), ell, s, w, pvm)


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
        for t in (50, 4096):
            b.run(t)
            st, _ = oracle_state(wl, budget=t, threads=8)
            assert_same_state(b.read_state(), st, wl.ell, wl.s, what="epoch %d budget %d" % (epoch, t))
