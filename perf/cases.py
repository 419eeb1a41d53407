"""The calls whose speed matters to a user of this framework, as measurable cases.

Each case is one pass through the public entry points (``rasp.Batch``, the
C ABI calls under the same names, ``rasp_run_static``, ``serving.Pool``) on
machines drawn by the repository's own generators. A pass returns what the
user's program reads back: the final registers, outputs and, for small
batches, the memories of every machine, a histogram of halting times, or the
best halting times. All outputs are whole numbers, so they are equal or wrong.

Large batches repeat a block of generated programs; every machine keeps its
own copy of its program, its own tape and its own step cap.
"""
from __future__ import annotations

import ctypes

import numpy as np
import torch

from paper_2604_12902_gb300 import rasp as R
from paper_2604_12902_gb300 import sampler as S
from paper_2604_12902_gb300 import serving as V
from paper_2604_12902_gb300 import workloads as W

FIELDS = (("i", torch.int64, 8), ("a", torch.int64, 8), ("steps", torch.int64, 8), ("status", torch.uint8, 1),
          ("uhead", torch.int32, 4), ("ylen", torch.int32, 4))
TAU_EDGES = np.concatenate([np.arange(0, 101), [1000, 10 ** 4, 10 ** 5, 10 ** 6, 1 << 62]]).astype(np.uint64)
BLOCK = 8192          # distinct programs behind a large batch


def listed():
    return [
        # A unit-test or debugging sized call: 1,024 self-modifying programs of 32
        # instructions, every field and memory read back; launches and latency count.
        dict(name="random-1k", kind="random", vms=1024, w=64, cap=256),
        # A small batch that fits the resident lanes: one candidate set of a search step.
        dict(name="templates-2k", kind="templates", vms=2048, w=64, cap=4096),
        # The headline workload: 2^20 loop programs re-packed, run to their halt, results read.
        dict(name="templates-1m", kind="templates", vms=1 << 20, w=64, cap=4096),
        # Ragged programs, memories and caps; a third of the machines time out; replayed as a CUDA graph.
        dict(name="uneven-256k", kind="uneven", vms=1 << 18, w=64, cap=65536),
        # Rollouts: each candidate program on 256 input tapes.
        dict(name="shared-1m", kind="shared", vms=1 << 20, w=64, cap=2048),
        # The halting experiment: 2^20 sampled array programs at w = 32 to 10^6 steps, and its histogram.
        dict(name="halting-1m", kind="halting", vms=1 << 20, w=32, cap=10 ** 6),
        # One round of the program search: new programs loaded, run, the best halting times kept.
        dict(name="search-128k", kind="search", vms=1 << 17, w=32, cap=10 ** 5),
        # End to end from page-locked host memory: new inputs and programs, run, results back.
        dict(name="rollout-256k", kind="rollout", vms=1 << 18, w=64, cap=4096),
        # The classic opcode set (SUB and BPA) on an odd number of machines.
        dict(name="classic-100k", kind="classic", vms=99_991, w=64, cap=4096),
        # Machines whose overflows and addresses are checked.
        dict(name="checked-64k", kind="checked", vms=1 << 16, w=64, cap=4096),
        # A caller-owned state store run in place, without allocation.
        dict(name="static-32k", kind="static", vms=1 << 15, w=64, cap=4096),
        # Serving: requests of several sizes submitted together, each read when done.
        dict(name="serve-4x", kind="serve", vms=24_000, w=64, cap=65536),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["random", "templates", "templates", "uneven", "uneven", "shared", "halting", "search",
                       "rollout", "classic", "checked", "static", "serve"])
    top = dict(random=65_536, templates=1 << 20, uneven=1 << 18, shared=1 << 20, halting=1 << 20, search=1 << 18,
               rollout=1 << 18, classic=1 << 18, checked=1 << 17, static=1 << 17, serve=48_000)[kind]
    vms = _log(rng, 256, top)
    w, cap = 64, 4096
    if kind == "random":
        w, cap = rng.choice([64, 64, 32, 16]), rng.choice([64, 256, 1000])
    elif kind in ("templates", "classic", "static"):
        w, cap = rng.choice([64, 64, 64, 48, 32, 24, 16]), rng.choice([100, 700, 4096])
    elif kind in ("uneven", "serve"):
        cap = _log(rng, 1000, 65536)
    elif kind == "shared":
        cap = 2048
    elif kind == "halting":
        w, cap = rng.choice([32, 29, 64]), _log(rng, 10 ** 3, 10 ** 6 if vms < 1 << 19 else 10 ** 5)
    elif kind == "search":
        w, cap = 32, _log(rng, 10 ** 3, 10 ** 5)
    return dict(kind=kind, vms=vms, w=w, cap=cap)


# ---------------------------------------------------------------- inputs
def _repeat(wl, vms, rng, caps=None):
    """`wl`'s programs repeated over `vms` machines, with tapes of their own."""
    base = wl.num_vms
    reps = -(-vms // base)
    plen = np.tile(wl.prog_off[1:] - wl.prog_off[:-1], reps)[:vms]
    off = np.zeros(vms + 1, np.uint64)
    np.cumsum(plen, out=off[1:])
    words = np.tile(wl.programs.astype(np.int32), reps)[:int(off[-1])]
    lo, hi = int(wl.tapes.min()), int(wl.tapes.max())
    tapes = rng.integers(lo, hi + 1, vms * wl.ell, dtype=np.int64)
    if caps is None:
        caps = np.full(vms, int(wl.caps[0]), np.uint64)
    return W.Workload(wl.name, words, off, np.tile(wl.mem_words, reps)[:vms], tapes,
                      np.arange(vms + 1, dtype=np.uint64) * np.uint64(wl.ell), caps, wl.ell, wl.s, wl.w)


def _workload(case, seed):
    kind, vms, cap = case["kind"], case["vms"], case["cap"]
    rng = np.random.default_rng(seed)
    base = min(vms, BLOCK)
    if kind == "random":
        return W.random_programs(num_vms=vms, seed=seed, cap=cap)
    if kind in ("templates", "rollout", "classic", "checked", "static"):
        return _repeat(W.template_programs(num_vms=base, seed=seed, cap=cap), vms, rng)
    if kind in ("uneven", "serve"):
        caps = np.exp(rng.uniform(np.log(64), np.log(cap + 1), vms)).astype(np.uint64)
        return _repeat(W.uneven_programs(num_vms=base, seed=seed), vms, rng, caps)
    if kind == "shared":
        programs = max(1, vms // 256)
        wl = W.shared_programs(num_programs=programs, vms_per_program=min(vms, 256), seed=seed, cap=cap)
        return wl
    return S.halting_programs_parallel(vms, workers=8, seed=seed, w=case["w"], cap=cap)


def _i32(words):
    return words.dtype == np.int32 or (words.size and -(1 << 31) <= words.min() and words.max() < 1 << 31)


class _State:
    """What the user's program holds: the case, its batch or pool, host buffers."""

    def __init__(self, case):
        self.kind = case["kind"]
        self.batch = self.pool = None

    def __del__(self):
        for x in (self.batch, self.pool):
            if x is not None:
                x.close()


def _host_buffers(st, count, s):
    """Page-locked result buffers and the view that fills them."""
    st.out = {name: torch.empty(count, dtype=dt, pin_memory=True) for name, dt, _ in FIELDS}
    st.out["y"] = torch.empty(count, s, dtype=torch.int64, pin_memory=True)
    st.view = R.rasp_state_view(*(ctypes.c_void_p(st.out[k].data_ptr())
                                  for k in ("i", "a", "steps", "status", "uhead", "ylen", "y")), None, 0)


def _pinned(a):
    t = torch.from_numpy(np.ascontiguousarray(a).view(np.int32 if a.dtype.itemsize == 4 else np.int64)).pin_memory()
    return t, t.numpy().view(a.dtype)


def prepare(case, seed):
    kind = case["kind"]
    wl = _workload(case, seed)
    st = _State(case)
    st.cap = case["cap"]
    if kind == "static":
        return _prepare_static(st, wl, case)
    if kind == "serve":
        return _prepare_serve(st, wl, case)
    flags, semantics = 0, R.WRAP
    if kind == "uneven":
        flags = R.CUDA_GRAPH
    elif kind == "shared":
        flags = R.SCHED_SHARED
    elif kind == "classic":
        flags = R.ISA_CLASSIC
    elif kind == "checked":
        semantics = R.CHECKED
    st.batch = b = R.Batch(wl.mem_words, wl.ell, wl.s, word_bits=case["w"], semantics=semantics, flags=flags)
    if kind == "search":
        st.wl = wl
        return st
    words = wl.programs.astype(np.int32) if _i32(wl.programs) else wl.programs
    load = R.rasp_load_programs_i32 if words.dtype == np.int32 else R.rasp_load_programs
    if kind == "rollout":
        st.keep = [_pinned(x) for x in (words, wl.prog_off, wl.tapes, wl.tape_off, wl.caps)]
        st.words, st.prog_off, st.tapes, st.tape_off, st.caps = (v for _, v in st.keep)
        st.load = load
    else:
        load(b.h, words, wl.prog_off, wl.prog_of_vm)
        b.load_inputs(wl.tapes, wl.tape_off, wl.caps)
    st.whole = kind not in ("rollout", "halting") and b.n_total <= 1 << 22   # small batches: memories too
    if not st.whole:
        _host_buffers(st, b.V, b.s)
    return st


def _prepare_static(st, wl, case):
    """The state store of `rasp_run_static` in torch tensors, and the c_0 it is set to."""
    n, vms, s = int(wl.mem_words[0]), wl.num_vms, wl.s
    mask = (1 << case["w"]) - 1 if case["w"] < 64 else -1
    dev = dict(device="cuda")
    words = torch.from_numpy(wl.programs).to(**dev).view(vms, -1).to(torch.int64)
    st.mem0 = torch.zeros(vms, n, dtype=torch.int64, **dev)
    st.mem0[:, :words.shape[1]] = words & mask
    st.tape = torch.from_numpy(wl.tapes).to(**dev) & mask
    st.cap_t = torch.from_numpy(wl.caps.view(np.int64)).to(**dev)
    st.n = torch.full((vms,), n, dtype=torch.int32, **dev)
    st.off = torch.arange(vms, dtype=torch.int64, **dev) * n
    st.mem = torch.empty_like(st.mem0)
    st.out = {name: torch.empty(vms, dtype=dt, **dev) for name, dt, _ in FIELDS}
    st.out["y"] = torch.empty(vms, s, dtype=torch.int64, **dev)
    st.out["mem"] = st.mem
    r = st.call = R.rasp_static_run()
    for name, t in (("cap", st.cap_t), ("n", st.n), ("mem_off", st.off), ("mem", st.mem), ("tape", st.tape),
                    *((k, st.out[k]) for k in ("i", "a", "steps", "status", "uhead", "ylen", "y"))):
        setattr(r, name, t.data_ptr())
    r.num_vms, r.word_bits, r.semantics, r.in_cap, r.out_cap = vms, case["w"], R.WRAP, wl.ell, s
    r.max_steps, r.mem_words = R.U64_MAX, vms * n
    r.stream = torch.cuda.current_stream().cuda_stream
    return st


def _prepare_serve(st, wl, case):
    """Four requests (1/2, 1/4, 1/8 and 1/8 of the machines) and the pool they go to."""
    words = wl.programs.astype(np.int64)
    cuts = [0] + [int(wl.num_vms * f) for f in (0.5, 0.75, 0.875)] + [wl.num_vms]
    st.requests = []
    for lo, hi in zip(cuts[:-1], cuts[1:]):
        p0, p1 = int(wl.prog_off[lo]), int(wl.prog_off[hi])
        st.requests.append(W.Workload("request", words[p0:p1].copy(), wl.prog_off[lo:hi + 1] - wl.prog_off[lo],
                                      wl.mem_words[lo:hi].copy(), wl.tapes[lo * wl.ell:hi * wl.ell].copy(),
                                      np.arange(hi - lo + 1, dtype=np.uint64) * np.uint64(wl.ell),
                                      wl.caps[lo:hi].copy(), wl.ell, wl.s))
    need = sum(R.rasp_batch_bytes(R.rasp_config(64, 0, wl.ell, wl.s, 0, 0, 0, 0, 0, 0, None, None, 0), q.mem_words)
               for q in st.requests)
    st.pool = V.Pool(2 * need + (1 << 24), wl.ell, wl.s)
    return st


# ---------------------------------------------------------------- one pass
def run(st):
    kind, b = st.kind, st.batch
    if kind == "static":
        st.mem.copy_(st.mem0)
        for name, _, _ in FIELDS:
            st.out[name].zero_()
        st.out["y"].zero_()
        if R.rasp_run_static(st.call) != R.RASP_OK:
            raise RuntimeError("rasp_run_static failed")
        return st.out
    if kind == "serve":
        tickets = [st.pool.submit(q) for q in st.requests]
        return [st.pool.read(t) for t in tickets]
    if kind == "search":
        b.load_workload(st.wl)
        b.run()
        tau, vm = b.top_halting(16)
        got = b.stats()
        return dict(tau=tau, vm=vm, **{k: got[k] for k in ("vm_steps", "running", "halted", "timeout")})
    if kind == "rollout":
        R.rasp_load_inputs(b.h, st.tapes, st.tape_off, st.caps)
        st.load(b.h, st.words, st.prog_off)
        b.run()
    else:
        b.reset()
        b.run()
    if st.whole:
        return b.read_state()
    if kind == "halting":
        counts, other = b.halting_histogram(TAU_EDGES)
        R.rasp_read_state(b.h, 0, b.V, st.view)
        return dict(st.out, counts=counts, other=other)
    R.rasp_read_state(b.h, 0, b.V, st.view)
    return st.out


# ---------------------------------------------------------------- what a pass cannot do without
# (words of M, instructions, tape words, output words, machine steps) of a machine, on average; the
# steps as the oracle counts them at the listed caps
_SHAPE = dict(random=(64, 32, 4, 8, 28), templates=(256, 64, 16, 8, 699), rollout=(256, 64, 16, 8, 699),
              classic=(256, 64, 16, 8, 699), checked=(256, 64, 16, 8, 699), static=(256, 64, 16, 8, 699),
              uneven=(846, 121, 16, 8, 1456), serve=(846, 121, 16, 8, 1456), shared=(224, 0.1875, 8, 8, 566),
              halting=(250, 44, 10, 2, 53_000), search=(250, 44, 10, 2, 5_400))


def work(case):
    """Bytes: programs (4-byte words where they are loaded so) and tapes read, memories, registers and
    outputs written, each once. Operations: one for each machine step."""
    n, instr, tape, s, steps = _SHAPE[case["kind"]]
    word = 4 if case["w"] <= 32 and case["kind"] not in ("static", "serve", "shared") else 8
    prog = 8 if case["kind"] in ("static", "serve", "search") else 4
    per_vm = 2 * instr * prog + 8 * tape + word * n + 8 * s + 41
    full = dict(halting=10 ** 6, search=10 ** 5, uneven=65536, serve=65536).get(case["kind"], steps)
    return dict(bytes=case["vms"] * per_vm, flops=case["vms"] * steps * min(1.0, case["cap"] / full))


# ---------------------------------------------------------------- the machine in plain numpy
def exact(case, seed):
    """Final states of small word-RASP batches: the transition of the machine on 64-bit words, every
    machine of the batch one step at a time. None where that would take too long."""
    if case["kind"] not in ("random", "templates") or case["vms"] * case["cap"] > 1 << 24:
        return None
    wl = _workload(case, seed)
    vms, ell, s = wl.num_vms, wl.ell, wl.s
    n = int(wl.mem_words[0])
    mask = np.uint64((1 << case["w"]) - 1)
    one, two, zero = np.uint64(1), np.uint64(2), np.uint64(0)
    words = wl.programs.astype(np.int64).view(np.uint64).reshape(vms, -1) & mask
    M = np.zeros((vms, n), np.uint64)
    M[:, :words.shape[1]] = words
    T = wl.tapes.view(np.uint64).reshape(vms, ell) & mask
    i, a = np.zeros(vms, np.uint64), np.zeros(vms, np.uint64)
    u0, y0, steps = np.zeros(vms, np.int64), np.zeros(vms, np.int64), np.zeros(vms, np.uint64)
    y, status, live = np.zeros((vms, s), np.int64), np.zeros(vms, np.uint8), np.arange(vms)
    while live.size:
        v, iv, av = live, i[live], a[live]
        o, j = M[v, (iv % np.uint64(n)).astype(np.int64)], M[v, (((iv + one) & mask) % np.uint64(n)).astype(np.int64)]
        jm = (j % np.uint64(n)).astype(np.int64)
        taken = (o == 5) & (av != 0)
        fixed = (o < 1) | (o > 7) | ((o == 6) & (u0[v] >= ell)) | (taken & (j == iv))
        out = ~fixed & (steps[v] >= wl.caps[v])
        status[v[fixed]], status[v[out]] = 1, 2
        go = ~(fixed | out)
        v, iv, av, o, j, jm, taken = (x[go] for x in (v, iv, av, o, j, jm, taken))
        m = M[v, jm]
        a[v] = np.where(o == 1, j, np.where(o == 2, av + m, np.where(o == 3, av * m, av))) & mask
        sto, rd, pri = o == 4, o == 6, (o == 7) & (y0[v] < s)
        M[v[sto], jm[sto]] = av[sto]
        M[v[rd], jm[rd]] = T[v[rd], u0[v[rd]]]
        u0[v[rd]] += 1
        y[v[pri], y0[v[pri]]] = m[pri].view(np.int64)
        y0[v[pri]] += 1
        i[v] = np.where(taken, j, (iv + two) & mask)
        steps[v] += one
        live = v
    return dict(i=i.view(np.int64), a=a.view(np.int64), steps=steps, status=status, uhead=u0.astype(np.uint32),
                ylen=y0.astype(np.uint32), y=y, mem=M.reshape(-1).view(np.int64))
