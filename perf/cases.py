"""The work that users have this checker do, as cases that can be timed and compared.

Every case builds seeded access traces on the GPU, in the shapes of the package's own
generators (``tracegen``: tree reduction in shared memory, owned tiles with random shared
words in global memory, power-law graph push, uneven batches), and checks them through the
package's binding: ``Checker.check_trace``, ``check_trace_host``, ``check_batch`` and the
hand-instrumented kernels.

A pass is what a program does with one trace: put the region back to INIT, check, wait for
the report, and put the races in an order of their own (the checker appends them in no fixed
order).  It returns the ordered race keys (zeros where a report ring has room left), the race
count, the status and the whole shadow, which the next chunk or the next launch would continue
from; all of it is whole numbers and does not depend on the order in which accesses of one wave
were applied.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2401_04701_gb300 import hirace

R, W, A, ST, SW = 0, 1, 2, 3, 4      # record ops: read, write, atomic, __syncthreads, __syncwarp


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # The smallest request of the batch and serving mixes: a 10,000-record trace of a
        # 64-thread block, on a checker as it comes.  Launches and waits, hardly any work.
        tree("tree_10k", block=64, segments=16, length=10_000),
        # A shared-memory reduction of one block (12,288 words, 8 barrier epochs, 1.03M
        # records): the plain single-block check, tuned once as a program would.
        tree("tree_1x256", block=256, segments=48, length=1_028_160, tuned=True),
        # A kernel of a few blocks, checked without tuning and in three calls, as a tracer
        # hands its buffers over: the later calls continue in the middle of a kernel.
        mix("mix_64x256_chunks", blocks=64, block_dim=256, chunks=3),
        # Sizes that are no powers of two: 3-warp blocks, an odd tile, selective monitoring
        # of a window of the words.
        mix("mix_301x96_window", blocks=301, block_dim=96, tile=50_021, window=True, tuned=True),
        # The benchmark workload: 1024 x 256 threads over 2^26 words, 75.2M records.
        mix("mix_1024x256", blocks=1024, block_dim=256, tuned=True),
        # The same kind of trace on the 4-byte shadow (half the shadow memory).
        mix("mix_509x256_compact", blocks=509, block_dim=256, compact=True, tuned=True),
        # Every racy epoch reported instead of the first one.
        mix("mix_256x256_every_epoch", blocks=256, block_dim=256, every=True),
        # A recorded trace in page-locked host memory, copied in while it is checked.
        mix("mix_256x256_host", blocks=256, block_dim=256, host=True),
        # Graph relaxation: irregular atomics on a shadow that fits L2, hub vertices that
        # many threads touch; a small graph untuned, and 2^22 vertices with 537M records.
        push("push_40k", vertices=40_000, degree=16, sweeps=2),
        push("push_4m", vertices=1 << 22, degree=16, sweeps=4, tuned=True),
        # Many traces of uneven length in one launch, replayed from a CUDA graph.
        batch("batch_64", traces=64, min_len=10_000, max_len=10_000_000, shape=1),
        # Source-level instrumentation: stencil, histogram and two reductions, each with
        # hr_access() beside every monitored access.
        inline("inline_4096x256", grid=4096),
    ]


def draw(rng):
    """One more case of the same ranges, sizes spread over their logarithm."""
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    tuned = rng.random() < 0.5
    kind = rng.choice(["tree", "mix", "mix", "mix", "push", "batch", "inline"])
    if kind == "tree":
        block = 32 * rng.randint(2, 32)
        segments = max(1, rng.randint(4, 48) * 256 // block)
        c = tree("", block=block, segments=segments, length=log(10_000, 10_000_000), tuned=tuned)
    elif kind == "mix":
        form = rng.choice(["plain", "plain", "plain", "compact", "every", "host", "window", "chunks"])
        c = mix("", blocks=log(16, 512 if form in ("every", "host") else 1024),
                block_dim=rng.choice([64, 96, 128, 192, 256]),
                tile=rng.choice([65_536, 32_768, rng.randint(20_000, 65_535)]),
                compact=form == "compact", every=form == "every", host=form == "host", window=form == "window",
                chunks=rng.randint(2, 4) if form == "chunks" else 1, tuned=tuned and form != "every")
    elif kind == "push":
        c = push("", vertices=log(5_000, 1 << 21), degree=rng.randint(4, 16), sweeps=rng.randint(1, 4), tuned=tuned)
    elif kind == "batch":
        c = batch("", traces=log(4, 64), min_len=10_000, max_len=rng.choice([1_000_000, 3_000_000, 10_000_000]),
                  shape=rng.randint(2, 1_000_000))
    else:
        c = inline("", grid=log(64, 4096))
    del c["name"]
    return c


def tree(name, block, segments, length, tuned=False):
    return dict(name=name, kind="tree", block=block, segments=segments, length=length, tuned=tuned)


def mix(name, blocks, block_dim, tile=65_536, compact=False, every=False, host=False, window=False, chunks=1,
        tuned=False):
    return dict(name=name, kind="mix", blocks=blocks, block_dim=block_dim, tile=tile, compact=compact, every=every,
                host=host, window=window, chunks=chunks, tuned=tuned)


def push(name, vertices, degree, sweeps, tuned=False):
    return dict(name=name, kind="push", vertices=vertices, degree=degree, sweeps=sweeps, tuned=tuned)


def batch(name, traces, min_len, max_len, shape):
    return dict(name=name, kind="batch", traces=traces, min_len=min_len, max_len=max_len, shape=shape)


def inline(name, grid):
    return dict(name=name, kind="inline", grid=grid)


# ------------------------------------------------------------------ traces

def records(word, tid, bc, wc, kernel, op, flags=0):
    """16-byte records (word, tid, wc | bc << 16, kernel | op << 16 | flags << 24), as int32 [n, 4]."""
    out = torch.empty((word.numel(), 4), dtype=torch.int32, device="cuda")
    out[:, 0] = word.reshape(-1)
    out[:, 1] = tid.reshape(-1) if torch.is_tensor(tid) else tid
    out[:, 2] = (wc | (bc << 16)).reshape(-1) if torch.is_tensor(wc | (bc << 16)) else wc | (bc << 16)
    last = kernel | (op << 16) | (flags << 24)
    out[:, 3] = last.reshape(-1) if torch.is_tensor(last) else last
    return out


def arange(n, *shape):
    return torch.arange(n, dtype=torch.int32, device="cuda").reshape(shape)


def tree_epochs(block):
    return int(math.log2(block))


def tree_reps(c):
    per_rep = c["segments"] * 3 * sum((c["block"] // 2) >> k for k in range(tree_epochs(c["block"])))
    return max(1, c["length"] // max(1, per_rep)), per_rep


def tree_trace(c, rng):
    """One block reduces `segments` arrays of `block` words: in epoch k, thread t < s = block/2 >> k
    reads words t and t+s and writes word t, again and again; barriers between epochs.  Races: a few
    (segment, epoch) units run with twice the threads, and one barrier in a hundred is missing."""
    block, seg = c["block"], c["segments"]
    reps, _ = tree_reps(c)
    epochs = tree_epochs(block)
    doubled = rng.random((seg, epochs)) < 0.01
    doubled[rng.integers(seg), rng.integers(epochs)] = True
    dropped = rng.random(epochs) < 0.01
    nwarp = -(-block // 32)
    t = arange(nwarp * 32, nwarp, 1, 1, 1, 32)
    sg = arange(seg, 1, 1, seg, 1, 1)
    j = arange(3, 1, 1, 1, 3, 1)
    parts, bc = [], 0
    for k in range(epochs):
        s = (block // 2) >> k
        if k > 0 and not dropped[k]:
            bc += 1
            every = arange(block, block)
            parts.append(records(every * 0, every, bc, 0, 0, ST))
        bound = torch.from_numpy(np.where(doubled[:, k], 2 * s, s).astype(np.int32)).cuda().reshape(1, 1, seg, 1, 1)
        shape = (nwarp, reps, seg, 3, 32)
        keep = ((t < bound) & (t < block)).expand(shape)
        word = (sg * block + torch.where(j == 1, (t + s) % block, t)).expand(shape)[keep]
        op = torch.where(j == 2, W, R).to(torch.int32).expand(shape)[keep]
        parts.append(records(word, t.expand(shape)[keep], bc, 0, 0, op))
    return torch.cat(parts)


def mix_shape(c):
    """(epochs, sub-epochs, accesses between two barriers) that a tile of c["tile"] words holds."""
    slots = c.get("slots", 8)
    epochs = min(c.get("epochs", 8), max(1, (c["tile"] // 4) // (slots * c["block_dim"])))
    return epochs, 4, slots


def mix_trace(c, gen, rate=0.001):
    """Blocks of `block_dim` threads, each with a tile of `tile` words: 45% reads and 5% atomics of
    random words anywhere (the upper part of every tile is read-only, a sixteenth atomic-only), 25%
    reads and 25% writes of the block's own rows, which move between threads over barriers only.
    Races: as many random accesses as `rate` of the words become writes of words others touch."""
    blocks, bd, tile = c["blocks"], c["block_dim"], c["tile"]
    epochs, subs, slots = mix_shape(c)
    nwarp = bd // 32
    own, at = tile // 4, tile // 16
    shape = (epochs, subs, blocks, nwarp, slots + 1, 32)
    e, w = arange(epochs, -1, 1, 1, 1, 1, 1), arange(subs, -1, 1, 1, 1, 1)
    b, v = arange(blocks, -1, 1, 1, 1), arange(nwarp, -1, 1, 1)
    i, ln = arange(slots + 1, -1, 1), arange(32, 32)
    n = math.prod(shape)

    def rand(hi):
        return torch.randint(hi, (n,), dtype=torch.int32, device="cuda", generator=gen)

    u = rand(100)
    own_word = (b * tile + (e * slots + (i - 1)) * bd + ((v + e) % nwarp) * 32 + (ln + w) % 32).expand(shape).reshape(-1)
    any_tile = rand(blocks) * tile
    word = torch.where(u < 45, any_tile + own + at + rand(tile - own - at),
                       torch.where(u < 50, any_tile + own + rand(at), own_word))
    del any_tile, own_word
    op = torch.where(u < 45, R, torch.where(u < 50, A, torch.where(u < 75, R, W))).to(torch.int32)
    sync = (i == 0).expand(shape).reshape(-1)
    n_inj = int(rate * blocks * tile)
    if n_inj:  # carriers: random-class accesses; targets: what some other access touches
        pick = torch.randint(n, (2, 4 * n_inj), device="cuda", generator=gen)
        ok = ~sync[pick[0]] & (u[pick[0]] < 50) & ~sync[pick[1]] & ((u[pick[1]] < 45) | (u[pick[1]] >= 50))
        first = torch.cumsum(ok, 0) <= n_inj
        src = word[pick[1][ok & first]]
        into = pick[0][ok & first]
        # several picks of one carrier: the last of them by place, not by the order of the writes
        into, where = torch.sort(into, stable=True)
        last = torch.ones_like(into, dtype=torch.bool)
        last[:-1] = into[1:] != into[:-1]
        word[into[last]] = src[where][last]
        op[into[last]] = W
    del u
    word[sync] = 0
    op = torch.where(sync, torch.where(w == 0, ST, SW).to(torch.int32).expand(shape).reshape(-1), op)
    tid = (b * bd + v * 32 + ln).expand(shape).reshape(-1)
    rec = records(word, tid, e.expand(shape).reshape(-1), w.expand(shape).reshape(-1), 0, op)
    keep = ~(sync & ((e == 0) & (w == 0)).expand(shape).reshape(-1))  # no barrier before the first accesses
    return rec[keep]


def push_trace(c, gen):
    """Thread v of each sweep (a launch each) visits its out-edges: an atomic load of dist[v], an
    atomicMin of dist[u]; both ends of an edge are drawn by power-law weights.  Races: one atomicMin
    in two thousand is a plain write."""
    n, m, sweeps = c["vertices"], c["vertices"] * c["degree"], c["sweeps"]
    weight = torch.arange(1, n + 1, dtype=torch.float64, device="cuda") ** (-1.0 / 1.1)
    cdf = torch.cumsum(weight, 0)
    cdf /= cdf[-1].clone()

    def ends():
        x = torch.searchsorted(cdf, torch.rand(m, dtype=torch.float64, device="cuda", generator=gen), right=True)
        return x.clamp_(max=n - 1).to(torch.int32)

    src, dst = torch.sort(ends()).values, ends()
    rec = torch.empty((sweeps, m, 2, 4), dtype=torch.int32, device="cuda")
    rec[:, :, 0, 0] = src
    rec[:, :, 1, 0] = dst
    rec[:, :, :, 1] = src[:, None]
    rec[:, :, :, 2] = 0
    del src, dst
    kernel = torch.arange(sweeps, dtype=torch.int32, device="cuda")
    rec[:, :, 0, 3] = (kernel | (A << 16) | (1 << 24))[:, None]
    rec[:, :, 1, 3] = (kernel | (A << 16))[:, None]
    hit = torch.randint(m, (sweeps, max(1, m // 2000)), device="cuda", generator=gen)
    for k in range(sweeps):
        rec[k, hit[k], 1, 3] = k | (W << 16)
    return rec.reshape(-1, 4)


def batch_plan(c):
    """The traces of a batch: 60% single-block reductions of 64 to 1024 threads on 4 to 48 KB, the
    rest global-memory traces over 1 to 64 MB, lengths spread over their logarithm."""
    rng = np.random.default_rng(c["shape"])
    plan = []
    for _ in range(c["traces"]):
        target = int(np.exp(rng.uniform(np.log(c["min_len"]), np.log(c["max_len"]))))
        if rng.random() < 0.6:
            block = int(rng.integers(2, 33)) * 32
            plan.append(tree("", block, max(1, int(rng.integers(4, 49)) * 256 // block), target))
        else:
            blocks = max(1, int(float(np.exp(rng.uniform(0.0, np.log(64.0)))) * 262_144) // 65_536)
            per_thread = max(1, target // (blocks * 256))
            epochs = int(np.clip(per_thread // 32, 1, 8))
            p = mix("", blocks, 256)
            p.update(epochs=epochs, slots=int(np.clip(per_thread // (4 * epochs), 1, 8)))
            plan.append(p)
    return plan


def words_of(c):
    if c["kind"] == "tree":
        return c["segments"] * c["block"]
    return c["vertices"] if c["kind"] == "push" else c["blocks"] * c["tile"]


def length_of(c):
    """Records of a case's trace, near enough for the bytes it has to read."""
    if c["kind"] == "tree":
        reps, per_rep = tree_reps(c)
        return reps * per_rep + c["block"] * (tree_epochs(c["block"]) - 1)
    if c["kind"] == "push":
        return c["vertices"] * c["degree"] * 2 * c["sweeps"]
    epochs, subs, slots = mix_shape(c)
    return (epochs * subs * (slots + 1) - 1) * c["blocks"] * c["block_dim"]


def trace_of(c, rng, gen, rate=0.001):
    t = tree_trace(c, rng) if c["kind"] == "tree" else push_trace(c, gen) if c["kind"] == "push" \
        else mix_trace(c, gen, rate)
    return t.reshape(-1).view(torch.uint8)


def region_of(c):
    reg = dict(n_words=words_of(c), block_dim=c.get("block") or c.get("block_dim") or 256)
    if c.get("compact"):
        reg.update(shadow_bytes=4, tid_bits=max(4, (c["blocks"] * c["block_dim"] - 1).bit_length()))
    if c.get("every"):
        reg.update(report_mode=hirace.REPORT_EVERY_EPOCH)
    if c.get("window"):  # the middle half of the words
        reg.update(n_words=window_of(c)[1] - window_of(c)[0])
    return reg


def window_of(c):
    return words_of(c) // 4, words_of(c) // 4 + words_of(c) // 2


def ring_room(c, rate=0.001):
    """Race records a region keeps: room for twice the races its trace was given."""
    if c["kind"] == "tree":
        return 2 * words_of(c)
    if c["kind"] == "push":
        return 1024 + 2 * c["sweeps"] * (c["vertices"] * c["degree"] // 2000)
    return 1024 + int(2 * rate * words_of(c))


def shadow_bytes(c):
    reg = region_of(c)
    return reg["n_words"] * (24 if c.get("every") else 4 if c.get("compact") else 8)


# ------------------------------------------------------------------ a program's state, and one pass

def prepare(case, seed):
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if case["kind"] == "inline":
        return prepare_inline(case, gen)
    if case["kind"] == "batch":
        return prepare_batch(case, rng, gen)
    trace = trace_of(case, rng, gen)
    shadow = torch.zeros(shadow_bytes(case) // 4, dtype=torch.int32, device="cuda")
    room = ring_room(case)
    ring = torch.zeros((room, 4), dtype=torch.int32, device="cuda")
    ck = hirace.Checker([region_of(case)], report_capacity=room, buffers=[(shadow, ring)])
    if case.get("window"):
        ck.set_filter(0, word_lo=window_of(case)[0], word_hi=window_of(case)[1])
    if case["tuned"]:
        ck.autotune(0, trace)
    if case.get("host"):
        host = torch.empty(trace.numel(), dtype=torch.uint8, pin_memory=True)
        trace = host.copy_(trace)
    n, k = trace.numel() // 16, case.get("chunks", 1)
    cuts = [(n * x // k + (x % k) * 7) * 16 for x in range(k)] + [n * 16]
    return dict(kind="trace", ck=ck, shadow=shadow, ring=ring, host=bool(case.get("host")),
                pieces=[trace[a:b] for a, b in zip(cuts[:-1], cuts[1:])])


def prepare_batch(case, rng, gen):
    plan = batch_plan(case)
    at = np.cumsum([0] + [-(-shadow_bytes(c) // 256) * 64 for c in plan])
    shadow = torch.zeros(int(at[-1]), dtype=torch.int32, device="cuda")
    room = [ring_room(c, rate=0.01) for c in plan]
    end = np.cumsum(room)
    ring = torch.zeros((int(end[-1]), 4), dtype=torch.int32, device="cuda")
    ck = hirace.Checker([dict(region_of(c), report_capacity=k) for c, k in zip(plan, room)], report_capacity=1,
                        buffers=[(shadow[at[i]:at[i + 1]], ring[end[i] - room[i]:end[i]]) for i in range(len(plan))])
    jobs = [(i, trace_of(c, rng, gen, rate=float(rng.uniform(0.0, 0.01)))) for i, c in enumerate(plan)]
    ck.batch_reserve(len(jobs), 1 << 16)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        ck.check_batch(jobs, stream=side)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        for i in range(len(jobs)):
            ck.reset(i, stream=side)
        ck.check_batch(jobs, stream=side)
    return dict(kind="batch", ck=ck, shadow=shadow, ring=ring, jobs=jobs, graph=graph)


def prepare_inline(case, gen):
    n = case["grid"] * 256
    x = torch.rand(n, device="cuda", generator=gen)
    keys = torch.randint(0, 4096, (n,), device="cuda", dtype=torch.int32, generator=gen)
    regions = [dict(n_words=w, block_dim=256) for w in (2 * n, 4096, n, n)]
    shadows = [torch.zeros(r["n_words"], dtype=torch.int64, device="cuda") for r in regions]
    ck = hirace.Checker(regions, report_capacity=1 << 16, buffers=shadows)
    hirace.load_workloads()
    return dict(kind="inline", ck=ck, shadows=shadows, x=x, keys=keys, out=torch.zeros_like(x),
                bins=torch.zeros(4096, dtype=torch.int32, device="cuda"), data=torch.zeros_like(x),
                sums=torch.zeros(case["grid"], device="cuda"))


def race_keys(ring):
    """Race records (four 32-bit words each) as sorted keys epoch << 48 | kernel << 32 | word (whose
    thread reported a race first is left to the order of the accesses)."""
    return torch.sort(ring[:, ::2].contiguous().view(torch.int64).reshape(-1)).values


def run(state):
    ck = state["ck"]
    if state["kind"] == "trace":
        state["ring"].zero_()
        ck.reset(0)
        for piece in state["pieces"]:
            if state["host"]:
                ck.check_trace_host(0, piece)
            else:
                ck.check_trace(0, piece)
        _, status, n, _ = ck.report(0, cap=0)
        return dict(status=status, n=n, races=race_keys(state["ring"]), shadow=state["shadow"])
    if state["kind"] == "batch":
        state["ring"].zero_()
        state["graph"].replay()
        told = [ck.report(i, cap=0)[1:3] for i in range(len(state["jobs"]))]
        return dict(told=np.array(told), races=race_keys(state["ring"]), shadow=state["shadow"])
    for i in range(4):
        ck.reset(i)
    hirace.run_stencil(ck.device_view(0), state["x"], state["out"])
    state["bins"].zero_()
    hirace.run_histogram(ck.device_view(1), state["keys"], state["bins"])
    state["data"].copy_(state["x"])
    hirace.run_reduce(ck.device_view(2), state["data"])
    hirace.run_smem_reduce(ck.device_view(3), state["x"], state["sums"], 1)
    for i in range(4):
        ck.sync(i)
    told = [ck.report(i, cap=0)[1:3] for i in range(4)]
    return dict(told=np.array(told), out=state["out"], bins=state["bins"], data=state["data"], sums=state["sums"],
                shadows=state["shadows"])


def work(case):
    """The trace read once and the shadow written once (inline: the kernels' own arrays and the shadow)."""
    if case["kind"] == "inline":
        n = case["grid"] * 256
        return dict(bytes=n * 4 * 7 + (4 * n + 4096) * 8, flops=n * 4)
    plan = batch_plan(case) if case["kind"] == "batch" else [case]
    return dict(bytes=sum(length_of(c) * 16 + shadow_bytes(c) for c in plan), flops=0)


def exact(case, seed):
    """The instrumented kernels' float results in 64 bits.  Checks return whole numbers only."""
    if case["kind"] != "inline":
        return None
    n = case["grid"] * 256
    x = torch.rand(n, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed)).double()
    out = x.clone()
    out[1:] += x[:-1]
    out[:-1] += x[1:]
    data = torch.nn.functional.pad(x, (0, -n % 512)).reshape(-1, 512).clone()
    s = 256
    while s:
        data[:, :s] += data[:, s:2 * s]
        s //= 2
    return dict(told=None, out=out, bins=None, data=data.reshape(-1)[:n], sums=x.reshape(-1, 256).sum(1), shadows=None)
