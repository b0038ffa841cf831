"""What a user of this framework has it do, as measurable cases.

Three kinds of work, each through the public entry points:

* ``batch``: gp_eval_small_noalloc on a batch of small trees whose arrays the
  caller owns on the device (a service, a real-time loop);
* ``full``: one full evaluation of a resident population (``eval_full``) and
  the read of its fitness;
* ``run``: a whole run -- new trees loaded, evaluated in full, then a number
  of generations (selection, crossover, incremental evaluation), the fitness
  read as it goes and the best tree at the end.

The tree shapes are those of this repository's workloads: ramped
half-and-half trees of depths 2..12 (``ramped``), trees grown by grafting
such trees onto leaves (``grafted``), and uniform random binary trees with
sizes log-uniform in [lo, hi] (``uneven``), over the binary32, 32-bit integer
and Boolean multiplexer sets.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2205_03251_gb300 as gp

DEPTHS = (2, 12)             # ramped half-and-half depths
CHUNK = 1 << 26              # most nodes of a forest built at once


def listed():
    return [
        # a handful of candidate formulas on few samples, as a real-time loop evaluates them: launch latency
        {"name": "batch-tiny", "kind": "batch", "set": "f32", "shape": "uneven", "trees": 8, "lo": 15, "hi": 127,
         "cases": 16},
        # a service's batch of small trees on an odd number of cases: the whole size range of the entry point
        {"name": "batch-service", "kind": "batch", "set": "f32", "shape": "uneven", "trees": 3000, "lo": 15, "hi": 1023,
         "cases": 100},
        # the first generation of an ordinary run: ramped half-and-half trees
        {"name": "full-ramped", "kind": "full", "set": "f32", "shape": "ramped", "trees": 500, "lo": 0, "hi": 0,
         "cases": 48},
        # the benchmark's population of huge trees
        {"name": "full-huge", "kind": "full", "set": "f32", "shape": "grafted", "trees": 500, "lo": 1000000, "hi": 1000000,
         "cases": 48},
        # trees of very different sizes on many cases, the last block of them ragged
        {"name": "full-cases", "kind": "full", "set": "f32", "shape": "uneven", "trees": 600, "lo": 10, "hi": 100000,
         "cases": 1000},
        # the 11-multiplexer: 2,048 cases packed in words
        {"name": "full-mux11", "kind": "full", "set": "mux11", "shape": "uneven", "trees": 1500, "lo": 10, "hi": 200000,
         "cases": 2048},
        # integer regression
        {"name": "full-int", "kind": "full", "set": "i32", "shape": "uneven", "trees": 2001, "lo": 10, "hi": 100000,
         "cases": 48},
        # the benchmark's run: huge trees, fitness first, learned work order, captured generations
        {"name": "run-huge", "kind": "run", "set": "f32", "shape": "grafted", "trees": 500, "lo": 1000000, "hi": 1000000,
         "cases": 48, "order": "first", "graph": 10, "launches": 6},
        # a population of very uneven trees, fitness first, captured generations
        {"name": "run-uneven", "kind": "run", "set": "f32", "shape": "uneven", "trees": 4096, "lo": 10, "hi": 100000,
         "cases": 48, "order": "first", "graph": 10, "launches": 3},
        # the same over the 6-multiplexer
        {"name": "run-mux6", "kind": "run", "set": "mux6", "shape": "uneven", "trees": 2048, "lo": 10, "hi": 100000,
         "cases": 64, "order": "first", "graph": 10, "launches": 3},
        # an ordinary run of moderate trees, every child built at crossover, generations called one by one
        {"name": "run-built", "kind": "run", "set": "f32", "shape": "grafted", "trees": 200, "lo": 20000, "hi": 20000,
         "cases": 48, "order": "built", "graph": 0, "launches": 30},
        # the smallest run: ramped half-and-half trees, generations called one by one
        {"name": "run-ramped", "kind": "run", "set": "f32", "shape": "ramped", "trees": 500, "lo": 0, "hi": 0,
         "cases": 48, "order": "built", "graph": 0, "launches": 30},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["batch", "full", "full", "run"])
    if kind == "batch":
        hi = _log(rng, 63, 1023)
        return {"kind": kind, "set": "f32", "shape": "uneven", "trees": _log(rng, 4, 4000), "lo": rng.randint(3, 31),
                "hi": hi, "cases": _log(rng, 8, 200)}
    funcs = rng.choice(["f32", "f32", "f32", "i32", "mux6", "mux11"])
    cases = {"mux6": 64, "mux11": 2048, "i32": rng.randint(20, 100)}.get(funcs) or \
        rng.choice([rng.randint(20, 64), _log(rng, 20, 1100)])
    shape = rng.choice(["ramped", "grafted", "uneven", "uneven"])
    c = {"kind": kind, "set": funcs, "shape": shape, "cases": cases}
    # nodes of the whole population so that no drawn case costs more than the largest listed ones
    most = 200_000_000 * 48 // max(48, {"mux11": 64, "mux6": 48}.get(funcs, cases))
    if shape == "ramped":
        c.update(trees=rng.randint(100, 1200), lo=0, hi=0)
    elif shape == "grafted":
        size = _log(rng, 20_000, 1_000_000)
        c.update(trees=max(20, min(_log(rng, 60, 500), most // size)), lo=size, hi=size)
    else:
        hi = _log(rng, 5_000, 200_000)
        c.update(trees=max(50, min(_log(rng, 300, 4096), int(most / (hi / math.log(hi / 10)) / 2))), lo=10, hi=hi)
    if kind == "run":
        graph = rng.choice([0, 4, 10])
        c.update(order=rng.choice(["first", "first", "built"]), graph=graph, launches=3 if graph else rng.randint(10, 30))
    return c


# ---------------------------------------------------------------- inputs

class _Source:
    """Random numbers on the GPU from one seed."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed) & (2**62 - 1))

    def below(self, n, size):
        return torch.randint(0, int(n), (int(size),), generator=self.g, device="cuda")

    def rand(self, size):
        return torch.rand(int(size), generator=self.g, device="cuda", dtype=torch.float64)


def _leaf_ops(src, n, funcs):
    """Opcodes of n leaves: x or a table constant with p = 0.5; Boolean: an input."""
    if funcs == "mux6":
        return 4 + src.below(6, n)
    if funcs == "mux11":
        return 4 + src.below(11, n)
    return torch.where(src.rand(n) < 0.5, 4, 5 + src.below(251, n))


def _label(src, is_func, funcs):
    """One byte per node: a random function or leaf for each."""
    n = is_func.numel()
    return torch.where(is_func, src.below(4, n), _leaf_ops(src, n, funcs)).to(torch.uint8)


def _splice(values, tree, lens, fill):
    """Each element repeated lens times: (values, tree, offset within, first) where fill(rep, within) gives the bytes."""
    start = torch.cumsum(lens, 0) - lens
    rep = torch.repeat_interleave(torch.arange(values.numel(), device=values.device), lens)
    within = torch.arange(rep.numel(), device=values.device) - start[rep]
    return fill(rep, within), tree[rep]


def _ramped(src, n):
    """(is_func, tree) of n ramped half-and-half trees: depths 2..12 in turn, full for even indices, grow for odd ones
    (a non-root node is a function with p = 0.5)."""
    idx = torch.arange(n, device="cuda")
    span = DEPTHS[1] - DEPTHS[0] + 1
    left = DEPTHS[0] + (idx // 2) % span            # edges still allowed below a placeholder; -1: a leaf, -2: a function
    tree, full = idx, idx % 2 == 0
    for level in range(DEPTHS[1] + 1):
        open_ = left >= 0
        func = open_ & (left > 0) & (full[tree] | (level == 0) | (src.rand(left.numel()) < 0.5))
        lens = torch.where(func, 3, 1)
        now = torch.where(func, -2, torch.where(open_, -1, left))

        def fill(rep, within, now=now, left=left):
            return torch.where(within > 0, left[rep] - 1, now[rep])
        left, tree = _splice(now, tree, lens, fill)
    return left == -2, tree


def _grafted(src, n, target):
    """(is_func, tree) of n trees grown from ramped half-and-half trees to about `target` nodes by grafting such trees
    onto uniformly chosen leaves."""
    bank_f, bank_t = _ramped(src, 220)
    bank_n = torch.bincount(bank_t, minlength=220)
    bank_o = torch.cumsum(bank_n, 0) - bank_n
    mean = float(bank_n.double().mean())

    def copies(pick):
        lens = bank_n[pick]
        first = torch.cumsum(lens, 0) - lens
        rep = torch.repeat_interleave(torch.arange(pick.numel(), device="cuda"), lens)
        return bank_f[bank_o[pick][rep] + torch.arange(rep.numel(), device="cuda") - first[rep]], rep
    func, tree = copies(src.below(220, n))
    for _ in range(60):
        size = torch.bincount(tree, minlength=n).double()
        if bool((size >= 0.97 * target).all()):
            break
        # grafts for each tree: at most twice its size, and about what is missing
        want = torch.minimum((target - size).clamp(min=0) / mean, 2 * size / mean + 1)
        leaves = (size + 1) / 2
        q = (want / leaves).clamp(max=1.0)
        graft = ~func & (src.rand(func.numel()) < q[tree])
        pick = src.below(220, func.numel())
        lens = torch.where(graft, bank_n[pick], 1)

        def fill(rep, within, func=func, graft=graft, pick=pick):
            return torch.where(graft[rep], bank_f[(bank_o[pick][rep] + within).clamp(max=bank_f.numel() - 1)], func[rep])
        func, tree = _splice(func, tree, lens, fill)
    return func, tree


def _uneven(src, n, lo, hi):
    """(is_func, tree) of n uniform random binary trees with odd sizes log-uniform in [lo, hi]: a uniform order of the
    functions and leaves, rotated to the one start that makes it a complete prefix expression (the cycle lemma)."""
    u = src.rand(n).cpu().numpy()
    inner = np.maximum(1, ((np.exp(np.log(lo) + u * (np.log(hi) - np.log(lo))) - 1) / 2).astype(np.int64))
    size = torch.from_numpy(2 * inner + 1).cuda()
    tree = torch.repeat_interleave(torch.arange(n, device="cuda"), size)
    first = torch.cumsum(size, 0) - size
    at = torch.arange(tree.numel(), device="cuda") - first[tree]
    order = torch.argsort(src.rand(tree.numel()) + tree)
    func = torch.empty(tree.numel(), dtype=torch.bool, device="cuda")
    func[order] = at < torch.from_numpy(inner).cuda()[tree]
    # balance before each position, within its tree; the start follows the first position of the lowest one after it
    step = torch.where(func, 1, -1)
    bal = torch.cumsum(step, 0)
    bal = bal - (bal - step)[first][tree]
    low = torch.full((n,), 1 << 40, device="cuda").scatter_reduce(0, tree, bal, "amin")
    place = torch.where(bal == low[tree], at, 1 << 40)
    rot = torch.full((n,), 1 << 40, device="cuda").scatter_reduce(0, tree, place, "amin") + 1
    return func[first[tree] + (at + rot[tree]) % size[tree]], tree


def _forest(case, seed):
    """(opcodes on the GPU, offsets): the case's trees."""
    src = _Source(seed * 7919 + 1)
    n, shape = case["trees"], case["shape"]
    each = {"ramped": 800, "grafted": case["hi"], "uneven": max(1, int(case["hi"] / math.log(max(3, case["hi"] / case["lo"])))
                                                                if shape == "uneven" else 1)}[shape]
    step = max(1, CHUNK // each)
    if shape == "ramped":
        step = max(22, step // 22 * 22)
    ops, sizes = [], []
    for a in range(0, n, step):
        k = min(step, n - a)
        if shape == "ramped":
            func, tree = _ramped(src, k)
        elif shape == "grafted":
            func, tree = _grafted(src, k, case["hi"])
        else:
            func, tree = _uneven(src, k, case["lo"], case["hi"])
        ops.append(_label(src, func, case["set"]))
        sizes.append(torch.bincount(tree, minlength=k))
        del func, tree
    ops, sizes = torch.cat(ops), torch.cat(sizes)
    off = np.zeros(n + 1, np.int64)
    off[1:] = np.cumsum(sizes.cpu().numpy())
    return ops, off


def _samples(case, seed):
    """Test cases, targets and the constant table, as the sextic regression uses them."""
    r = np.random.RandomState((seed * 104729 + 17) % (2**32))
    n = case["cases"]
    if case["set"] == "i32":
        x = r.randint(-8, 9, n)
        return x.astype(np.int32), (x * x * (x * x - 1) ** 2).astype(np.int32), r.randint(-8, 9, 251).astype(np.int32)
    grid = 1.0 / 8388608.0
    x = (r.randint(0, 1 << 24, n) * grid - 1.0).astype(np.float32)
    k = (r.randint(0, 1 << 24, 251) * grid - 1.0).astype(np.float32)
    d = x.astype(np.float64) ** 2
    return x, (d * (d - 1) ** 2).astype(np.float32), k


def _most(case):
    """The bound on a tree's nodes that the user sets: about twice the largest tree of the start."""
    return 2 * case["hi"] + (65536 if case["shape"] == "grafted" else 16384)


def prepare(case, seed):
    ops, off = _forest(case, seed)
    x, t, k = _samples(case, seed)
    if case["kind"] == "batch":
        pad = (-ops.numel()) % 16
        s = {"kind": "batch", "ops": torch.cat([ops, torch.zeros(pad, dtype=torch.uint8, device="cuda")]),
             "off": torch.from_numpy(off).cuda(), "x": torch.from_numpy(x).cuda(), "t": torch.from_numpy(t).cuda(),
             "k": torch.from_numpy(k).cuda(), "values": torch.empty((case["trees"], case["cases"]), device="cuda"),
             "fitness": torch.empty(case["trees"], device="cuda")}
        return s
    host = torch.empty(ops.numel(), dtype=torch.uint8, pin_memory=True)      # where the user's trees are
    host.copy_(ops)
    torch.cuda.synchronize()
    del ops
    torch.cuda.empty_cache()                     # the population takes its memory from the device, not from PyTorch
    boolean = case["set"].startswith("mux")
    first = case.get("order") == "first"
    most = _most(case)
    pop = gp.Population(x, t, k, host.numpy(), off.astype(np.uint64), max_nodes=most, boolean=boolean,
                        mux_k=3 if case["set"] == "mux11" else 2, integer=case["set"] == "i32", seed=seed,
                        lazy=first, packing=gp.GP_PACK_MLP if first else gp.GP_PACK_STATIC)
    s = {"kind": case["kind"], "pop": pop, "ops": host.numpy(), "keep": host, "off": off.astype(np.uint64)}
    if case["kind"] == "run":
        s.update(graph=case["graph"], launches=case["launches"], tree=np.zeros(most, np.uint8))
        pop.eval_full()
        if case["graph"]:
            # a population that starts uneven may end with the largest trees only: about one node in 40 of such a tree
            # heads a subtree of the cache's size
            pop.set_graph_mode(True, case["trees"] * most // 40 if case["shape"] == "uneven" else 0)
            pop.eval_full()
            _first_generations(pop)
            pop.graph_capture(2, case["graph"])
    return s


def _first_generations(pop):
    # two, because the buffers of parents and children change places with each: a graph captured after an even number
    # of generations is replayed after an even number
    for g in range(2):
        pop.crossover(g)
        pop.eval_incremental(want_stats=False)


def run(s):
    if s["kind"] == "batch":
        gp.gp_eval_small_noalloc(s["ops"], s["off"], s["x"], s["t"], s["k"], s["values"], s["fitness"])
        return {"values": s["values"], "fitness": s["fitness"]}
    pop = s["pop"]
    if s["kind"] == "full":
        pop.eval_full()
        return {"fitness": pop.fitness()}
    pop.load_trees(s["ops"], s["off"])
    pop.eval_full()
    _first_generations(pop)
    fits = [pop.fitness()]
    for g in range(s["launches"]):
        if s["graph"]:
            pop.graph_launch()
        else:
            pop.crossover(g + 2)
            pop.eval_incremental(want_stats=False)
        fits.append(pop.fitness())
    last = np.where(np.isnan(fits[-1]), np.inf, fits[-1])
    tree = pop.tree(int(np.argmin(last)))
    s["tree"][:tree.size] = tree
    s["tree"][tree.size:] = 0
    return {"fitness": np.stack(fits), "tree": s["tree"]}


def _nodes(case):
    if case["shape"] == "ramped":
        return case["trees"] * 733
    if case["shape"] == "grafted" or case["lo"] == case["hi"]:
        return case["trees"] * case["hi"]
    return int(case["trees"] * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"]))


def work(case):
    """One pass: each opcode read once and one operation per function node and case (Boolean: per 32-case word); a run
    besides moves the trees of a generation and evaluates what its crossovers disrupt, of which only the bytes of the
    children that become parents (about 0.4 of them) are counted."""
    n = _nodes(case)
    width = case["cases"] / 32 if case["set"].startswith("mux") else case["cases"]
    out = 4 * case["trees"] * (1 + (case["cases"] if case["kind"] == "batch" else 0))
    w = {"bytes": n + out, "flops": n / 2 * width}
    if case["kind"] == "run":
        gens = 2 + case["launches"] * max(1, case["graph"])
        w["bytes"] += int(n + gens * 0.8 * n + 4 * case["trees"] * case["launches"])
    return w


# ---------------------------------------------------------------- 64 bits

def _exact_tree(ops, leaf, C):
    """One tree on all cases in binary64, right to left with a stack; None where a value is not finite in binary32."""
    stack = []
    for o in ops[::-1]:
        if o >= 4:
            stack.append(leaf[o])
            continue
        a = stack.pop()
        b = stack.pop()
        if o == 0:
            stack.append(a + b)
        elif o == 1:
            stack.append(a - b)
        elif o == 2:
            stack.append(a * b)
        else:
            stack.append(np.where(b == 0, 1.0, a / np.where(b == 0, 1.0, b)))
    return stack[0]


def exact(case, seed):
    # evaluations of small trees; a deep tree's value is chaotic (a quotient by a near-cancelled difference amplifies
    # the rounding of its operands without bound), and a run's selections are decisions, so larger cases have none
    if case["set"] != "f32" or case["kind"] == "run" or _nodes(case) * case["cases"] > 100_000_000:
        return None
    ops, off = _forest(case, seed)
    ops = ops.cpu().numpy()
    x, t, k = (v.astype(np.float64) for v in _samples(case, seed))
    leaf = [None] * 4 + [x] + [np.full(case["cases"], c) for c in k]
    with np.errstate(all="ignore"):
        values = np.stack([_exact_tree(ops[off[i]:off[i + 1]], leaf, case["cases"]) for i in range(case["trees"])])
        fitness = np.abs(values - t).sum(1)
    return {"values": values, "fitness": fitness} if case["kind"] == "batch" else {"fitness": fitness}
