"""The calls that stand for this library's use, for timing and for comparing results.

A case is one call of a workload entry point, made as a program makes it: the object, the
device buffers and (where the program keeps one) the CUDA graph exist already, and a pass
clears what the workload asks to be cleared and launches.  Every family of the library is
here: grid barriers, mutexes (from device and from host buffers), counting semaphores, the
condition-variable queue, the batched many-mutex kernel and the persistent serving loop.

Results that the order of the grants decides (the grant log, tickets, which consumer took an
item, the running maximum of a semaphore's holders, latencies) are not outputs: two runs of
one build differ in them.  Everything else is, and is exact.
"""
import math

import numpy as np
import torch

from paper_1110_4623_gb300 import autotune, gsync as G, inputs, runner

MASK64 = (1 << 64) - 1
# Sleep of a waiting block (min_ns, max_ns) by kind, and the blocks per cluster of the cluster locks.
MUTEX_BACKOFF = {"cas_backoff": (16, 512), "ticket": (128, 4000), "cohort": (128, 4000), "cluster": (128, 4000),
                 "cluster_mcs": (128, 4000)}
MUTEX_CLUSTER = {"cluster": 4, "cluster_mcs": 8}
SEM_BACKOFF = {"window": (16, 2000), "ticket": (16, 2000), "spin_backoff": (64, 4096)}
# Policies of the batched kernel's hot, warm and cold keys: untuned, tuned without clusters,
# and tuned with them.
BATCHED_POLICY = {
    "untuned": autotune.DEFAULT_POLICY,
    "carry": [("cohort_carry", 0, 0), ("ticket_carry", 64, 2000), ("cas_backoff", 128, 4096)],
    "tuned": [("cluster_die_carry", 0, 0), ("cluster", 128, 4000), ("ticket_carry", 64, 2000)],
}
SERVE_POOL = 256 << 20  # int32 values (1 GiB: a request's values come from DRAM)


def listed():
    return [
        # The paper's barrier test: 16 blocks, 10,000 rounds, every block folds every slot.
        dict(name="barrier 16 full", family="barrier", kind="count", param=8, nblocks=16, threads=128, rounds=10000,
             full=True),
        # A persistent kernel that fills the GPU, one exchange with a partner per crossing.
        dict(name="barrier 1184", family="barrier", kind="count", param=8, nblocks=1184, threads=128, rounds=1000,
             full=False),
        # A short kernel with a few global steps, one block per SM: the launch counts.
        dict(name="barrier 148 short", family="barrier", kind="count", param=8, nblocks=148, threads=128, rounds=16,
             full=False),
        # The default mutex on a full grid, a critical section wider than the block.
        dict(name="mutex mcs 1184", family="mutex", kind="cluster_mcs", nblocks=1184, threads=256, acq=100,
             cs_words=1024, host=False),
        # The paper's spin lock at the grid where its contention is worst.
        dict(name="mutex spin 1184", family="mutex", kind="cas_spin", nblocks=1184, threads=256, acq=100, cs_words=64,
             host=False),
        # A small locked job from host buffers to host buffers.
        dict(name="mutex host 16", family="mutex", kind="ticket", nblocks=16, threads=256, acq=10, cs_words=64,
             host=True),
        # The default semaphore on a full grid.
        dict(name="sem window 1184", family="sem", kind="window", nblocks=1184, threads=128, pairs=200, n=16,
             hold_hi=5000),
        # The paper's spin-lock semaphore with backoff.
        dict(name="sem spin 296", family="sem", kind="spin_backoff", nblocks=296, threads=128, pairs=20, n=4,
             hold_hi=5000),
        # A producer/consumer queue under a mutex and two condition variables.
        dict(name="condvar 592+592", family="condvar", kind="ticket", producers=592, consumers=592, items=10,
             capacity=16, threads=128),
        # Many mutexes under one launch, tuned and replayed from a graph.
        dict(name="batched 1e6 tuned", family="batched", policy="tuned", nacq=1_000_000, nkeys=4096, s=1.1,
             nblocks=1184, threads=128, ngroups=64, rounds=100, cluster=8, graph=True),
        # The same kernel untuned, on keys of milder skew and without clusters.
        dict(name="batched 2e5 untuned", family="batched", policy="untuned", nacq=200_000, nkeys=4096, s=0.6,
             nblocks=592, threads=128, ngroups=16, rounds=20, cluster=1, graph=False),
        # A backlog of requests drained by the serving loop.
        dict(name="serve backlog", family="serve", nreq=8192, len_hi=1 << 20, nslots=64, nblocks=304, admitters=16,
             chunk=8192, ring="host"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    family = rng.choice(["barrier", "barrier", "mutex", "mutex", "mutex", "sem", "sem", "condvar", "batched", "batched",
                         "serve"])
    if family == "barrier":
        kind, param = rng.choice([("count", 8), ("count", 8), ("count", 0), ("exchange", 8), ("atomic", 0), ("flag", 0),
                                  ("tree", 8), ("cluster", 8 | 2 << 4), ("cluster", 4)])
        full = rng.random() < 0.4
        nblocks = _log_int(rng, 2, 296 if full else 1184)
        if kind == "cluster":
            nblocks = max(1, nblocks // (param & 0xF)) * (param & 0xF)
        threads = rng.choice([32, 64, 128] if nblocks > 592 else [32, 64, 128, 256])
        return dict(family=family, kind=kind, param=param, nblocks=nblocks, threads=threads,
                    rounds=_log_int(rng, 10, 1000), full=full)
    if family == "mutex":
        kind = rng.choice(["cluster_mcs", "cluster_mcs", "cluster", "cohort", "ticket", "sleep_queue", "cas_backoff",
                           "cas_spin", "ring"])
        nblocks, c = _log_int(rng, 8, 1184), MUTEX_CLUSTER.get(kind, 1)
        return dict(family=family, kind=kind, nblocks=nblocks // c * c, threads=rng.choice([64, 128, 256]),
                    acq=_log_int(rng, 5, 60), cs_words=rng.choice([0, _log_int(rng, 1, 2048), _log_int(rng, 1, 2048)]),
                    host=rng.random() < 0.3)
    if family == "sem":
        kind = rng.choice(["window", "window", "ticket", "spin_backoff"])
        spin = kind == "spin_backoff"
        return dict(family=family, kind=kind, nblocks=_log_int(rng, 2, 296 if spin else 1184),
                    threads=rng.choice([32, 128, 256]), pairs=_log_int(rng, 5, 20 if spin else 100),
                    n=_log_int(rng, 4 if spin else 1, 64), hold_hi=_log_int(rng, 100, 5000))
    if family == "condvar":
        consumers = 8 * _log_int(rng, 1, 48)
        return dict(family=family, kind=rng.choice(["ticket", "ticket", "cohort", "cluster", "cluster_mcs"]),
                    producers=consumers * rng.choice([1, 2]), consumers=consumers, items=_log_int(rng, 2, 20),
                    capacity=_log_int(rng, 1, 256), threads=rng.choice([32, 128]))
    if family == "batched":
        policy = rng.choice(["untuned", "carry", "tuned"])
        cluster = rng.choice([2, 4, 8]) if policy == "tuned" else 1
        nblocks = 8 * _log_int(rng, 8, 148)
        return dict(family=family, policy=policy, nacq=_log_int(rng, 10_000, 300_000), nkeys=_log_int(rng, 64, 8192),
                    s=round(rng.uniform(0.4, 1.2), 2), nblocks=nblocks, threads=128, ngroups=nblocks // 32,
                    rounds=_log_int(rng, 5, 100), cluster=cluster, graph=rng.random() < 0.5)
    return dict(family=family, nreq=_log_int(rng, 64, 8192), len_hi=_log_int(rng, 1 << 13, 1 << 20),
                nslots=rng.choice([16, 64]), nblocks=304, admitters=rng.choice([8, 16]),
                chunk=rng.choice([8192, 32768]), ring="host")


def _backoff(table, kind):
    return runner.backoff(min_ns=table[kind][0], max_ns=table[kind][1]) if kind in table else None


# ---------------------------------------------------------------------------------------
# What a program has in hand before the call
# ---------------------------------------------------------------------------------------

def prepare(case, seed):
    return globals()["_prepare_" + case["family"]](case, seed & MASK64)


def _rounds(case, seed):
    """The barrier workload's only input is its length: one round more for every other seed."""
    return case["rounds"] + seed % 2


def _prepare_barrier(case, seed):
    run = runner.BarrierRun(case["kind"], case["nblocks"], case["threads"], case["rounds"] + 1, case["full"],
                            param=case["param"])
    run.work.rounds = _rounds(case, seed)  # chk has room for the longer run
    return case, run


def _mutex_inputs(case, seed):
    return inputs.mutex_inputs(case["nblocks"], case["acq"], seed)


def _prepare_mutex(case, seed):
    delay, add = _mutex_inputs(case, seed)
    kind, bo, cluster = case["kind"], _backoff(MUTEX_BACKOFF, case["kind"]), MUTEX_CLUSTER.get(case["kind"], 0)
    if not case["host"]:
        return case, runner.MutexRun(kind, case["nblocks"], case["threads"], case["acq"], case["cs_words"], delay, add,
                                     bo=bo, cluster=cluster)
    n, k = case["nblocks"] * case["acq"], case["cs_words"]
    host = {"delay": torch.from_numpy(delay.view(np.int32)).pin_memory(),
            "addend": torch.from_numpy(add.view(np.int32)).pin_memory()}
    for name, size in (("data", max(k, 1)), ("total", 1), ("log", n), ("ticket", n), ("count", case["nblocks"]),
                       ("status", 1)):
        host[name] = torch.zeros(size, dtype=torch.int32).pin_memory()
    work = G.gsync_mutex_work(G.MUTEX_KINDS[kind], case["nblocks"], case["threads"], case["acq"], k, cluster,
                              *(host[x].data_ptr() for x in ("delay", "addend", "data", "total", "log", "ticket",
                                                             "count", "status")))
    nbytes = G.gsync_bench_mutex_workspace_bytes(work.kind, work.nblocks, work.acq, k)
    return case, (work, bo, torch.empty(nbytes, dtype=torch.uint8, device="cuda"), nbytes, host)


def _sem_inputs(case, seed):
    return inputs.sem_inputs(case["nblocks"], case["pairs"], seed, hold_hi=case["hold_hi"])


def _prepare_sem(case, seed):
    hold, add = _sem_inputs(case, seed)
    return case, runner.SemRun(case["kind"], case["nblocks"], case["threads"], case["pairs"], case["n"], hold, add,
                               bo=_backoff(SEM_BACKOFF, case["kind"]), timeout_ns=30_000_000_000)


def _prepare_condvar(case, seed):
    value = inputs.condvar_inputs(case["producers"] * case["items"], seed)
    bo = runner.backoff(min_ns=64 if case["kind"] == "ticket" else 128, max_ns=2000 if case["kind"] == "ticket" else 4000)
    return case, runner.CondVarRun(case["producers"], case["consumers"], case["items"], case["capacity"], value,
                                   block_threads=case["threads"], bo=bo, mutex=case["kind"],
                                   cluster=MUTEX_CLUSTER.get(case["kind"], 0))


def _batched_inputs(case, seed):
    return inputs.batched_inputs(case["nacq"], case["nkeys"], case["s"], seed)[:2]


def _prepare_batched(case, seed):
    keys, adds = _batched_inputs(case, seed)
    run = autotune.make_run(keys, adds, case["nkeys"], case["nblocks"], case["ngroups"], case["rounds"],
                            case["cluster"], autotune.classify_keys(keys, case["nkeys"], case["nblocks"]),
                            block_threads=case["threads"], plain_launch=case["graph"] and case["cluster"] == 1)
    run.set_policy(BATCHED_POLICY[case["policy"]])
    if case["graph"]:
        run.capture()
    return case, run


def _serve_requests(case, seed):
    length = inputs.log_uniform_int(seed, case["nreq"], 256, case["len_hi"])
    offset = np.floor(inputs.unit_f64(seed ^ 0x0FF5E7, case["nreq"]) * (SERVE_POOL - length + 1)).astype(np.int64)
    return offset, length


def _serve_pool(seed):
    gen = torch.Generator(device="cuda").manual_seed(seed % (1 << 62))
    return torch.randint(-(1 << 20), (1 << 20) + 1, (SERVE_POOL,), dtype=torch.int32, device="cuda", generator=gen)


def _prepare_serve(case, seed):
    offset, length = _serve_requests(case, seed)
    # a backlog: every request has arrived when the loop starts
    return case, runner.ServeRun(offset, length, np.zeros(case["nreq"], dtype=np.int64), _serve_pool(seed),
                                 nslots=case["nslots"], nblocks=case["nblocks"], admitters=case["admitters"],
                                 chunk_elems=case["chunk"], ring=case["ring"])


# ---------------------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------------------

def run(state):
    case, r = state
    return globals()["_run_" + case["family"]](case, r)


def _run_barrier(case, r):
    G.check("gsync_bench_barrier", r.launch())
    out = {"mix": r.mix, "bad": r.bad, "status": r.status}
    return {**out, "chk": r.chk} if case["full"] else out


def _run_mutex(case, r):
    if case["host"]:
        work, bo, ws, nbytes, host = r
        G.check("gsync_bench_mutex_host", G.gsync_bench_mutex_host(work, bo, ws, nbytes))
        return {k: host[k] for k in ("data", "total", "count", "status")}
    r.reset()
    G.check("gsync_bench_mutex", r.launch())
    return {"data": r.data, "total": r.total, "count": r.count, "status": r.status}


def _run_sem(case, r):
    r.reset()
    G.check("gsync_bench_sem", r.launch())
    s = r.scalars  # occupancy, the running maximum, total, tally and status, each on a line of its own
    return {"occupancy": s[0:1], "total": s[64:65], "tally": s[96:97], "status": s[128:129], "count": r.count}


def _run_condvar(case, r):
    r.reset()
    G.check("gsync_bench_condvar", r.launch())
    # which consumer took an item is the scheduler's choice: the consumers' sums add up
    return {"seen": r.seen, "sum": r.sum.sum(), "count": r.count, "status": r.status}


def _run_batched(case, r):
    if case["graph"]:
        r.replay()
    else:
        r.reset()
        G.check("gsync_bench_batched", r.launch())
    return {"sum": r.sum, "count": r.count, "mix": r.mix, "bad": r.bad, "status": r.status}


def _run_serve(case, r):
    out = r.run()
    G.check("gsync_serve_run", out["rc"])
    return {"res": out["res"], "stats": np.array(out["stats"], dtype=np.int64)}


# ---------------------------------------------------------------------------------------
# What a pass has to read and write, and what it has to return
# ---------------------------------------------------------------------------------------

def work(case):
    f = case["family"]
    if f == "barrier":
        # a slot written per block and round, and read by a partner or by every block
        per = case["nblocks"] if case["full"] else 1
        n = case["nblocks"] * case["rounds"] * (4 + 4 * per + (4 if case["full"] else 0)) + 8 * case["nblocks"]
    elif f == "mutex":
        # delay, addend, log and ticket per acquisition; data and total read and written
        n = case["nblocks"] * case["acq"] * (16 + 8 + 8 * case["cs_words"]) + 4 * case["nblocks"]
    elif f == "sem":
        n = case["nblocks"] * case["pairs"] * (8 + 8) + 4 * case["nblocks"]
    elif f == "condvar":
        # an item's id put and taken, its value read and its take counted
        n = case["producers"] * case["items"] * 20 + 12 * case["consumers"]
    elif f == "batched":
        n = case["nacq"] * (4 + 8 + 2 * 12) + case["nkeys"] * 12 + case["nblocks"] * case["rounds"] * 8
    else:
        mean = (case["len_hi"] - 256) / math.log(case["len_hi"] / 256)  # log-uniform lengths
        n = case["nreq"] * (4 * mean + 16 + 12)
    return {"bytes": n, "flops": 0}


def _lowbias32(x):
    x = np.asarray(x, dtype=np.uint32).copy()
    with np.errstate(over="ignore"):
        x ^= x >> np.uint32(16)
        x *= np.uint32(0x7FEB352D)
        x ^= x >> np.uint32(15)
        x *= np.uint32(0x846CA68B)
        x ^= x >> np.uint32(16)
    return x


def _i32(x):
    return np.ascontiguousarray(np.asarray(x, dtype=np.uint32)).view(np.int32)


def _rotl5(x):
    return (x << np.uint32(5)) | (x >> np.uint32(27))


def _sampled_mix(nblocks, rounds):
    b, mix = np.arange(nblocks), np.zeros(nblocks, dtype=np.uint32)
    for r in range(rounds):
        mix = _rotl5(mix) ^ _lowbias32((r * nblocks + (b + r + 1) % nblocks).astype(np.uint32))
    return mix


def exact(case, seed):
    seed &= MASK64
    f, none = case["family"], np.zeros(1, dtype=np.int32)
    if f == "barrier":
        n, rounds = case["nblocks"], _rounds(case, seed)
        bad = np.zeros(n, dtype=np.int32)
        if not case["full"]:
            return {"mix": _i32(_sampled_mix(n, rounds)), "bad": bad, "status": none}
        mix, chk = np.uint32(0), np.zeros((case["rounds"] + 1, n), dtype=np.uint32)
        for r in range(rounds):
            slots = np.arange(r * n, (r + 1) * n, dtype=np.uint32)
            chk[r] = np.bitwise_xor.reduce(slots)
            mix = _rotl5(mix) ^ np.uint32(_lowbias32(slots).astype(np.uint64).sum() & np.uint64(0xFFFFFFFF))
        return {"mix": _i32(np.full(n, mix)), "bad": bad, "status": none, "chk": _i32(chk.reshape(-1))}
    if f == "mutex":
        add, k = _mutex_inputs(case, seed)[1].astype(np.uint64), case["cs_words"]
        data = np.zeros(max(k, 1), dtype=np.uint64)
        for i in range(k):
            data[i] = (add ^ np.uint64(i * 0x9E3779B1 & 0xFFFFFFFF)).sum() & np.uint64(0xFFFFFFFF)
        return {"data": _i32(data), "total": _i32([case["nblocks"] * case["acq"]]),
                "count": _i32(np.full(case["nblocks"], case["acq"])), "status": none}
    if f == "sem":
        add, pairs = _sem_inputs(case, seed)[1].astype(np.uint64), case["nblocks"] * case["pairs"]
        return {"occupancy": none, "total": _i32([pairs if case["n"] == 1 else 0]),
                "tally": _i32([add.sum() & np.uint64(0xFFFFFFFF)]), "status": none,
                "count": _i32(np.full(case["nblocks"], case["pairs"]))}
    if f == "condvar":
        n = case["producers"] * case["items"]
        return {"seen": np.ones(n, dtype=np.int32),
                "sum": np.int64(inputs.condvar_inputs(n, seed).view(np.int32).astype(np.int64).sum()),
                "count": _i32(np.full(case["consumers"], n // case["consumers"])), "status": none}
    if f == "batched":
        keys, adds = _batched_inputs(case, seed)
        total = np.zeros(case["nkeys"], dtype=np.int64)
        with np.errstate(over="ignore"):
            np.add.at(total, keys, adds)
        sizes = inputs.barrier_group_sizes(case["ngroups"], 2, 256, case["nblocks"], multiple=case["cluster"])[1]
        mix, at = np.zeros(case["nblocks"], dtype=np.uint32), 0
        for size in sizes:  # consecutive groups, each with slots of its own
            mix[at:at + size] = _sampled_mix(int(size), case["rounds"])
            at += size
        return {"sum": total, "count": _i32(np.bincount(keys, minlength=case["nkeys"])), "mix": _i32(mix),
                "bad": np.zeros(case["nblocks"], dtype=np.int32), "status": none}
    offset, length = _serve_requests(case, seed)
    pool = _serve_pool(seed).cpu().numpy()
    res = np.array([pool[o:o + n].sum(dtype=np.int64) for o, n in zip(offset, length)])
    chunks = int((-(-length // case["chunk"])).sum())
    return {"res": res, "stats": np.array([case["nreq"], chunks, case["nreq"], 0], dtype=np.int64)}
