"""The calls that programs make of this evaluator, from the smallest to the
largest, as cases that can be timed and compared.

A pass is what a program does with a batch of nets it has as text: empty the
context (inet_reset), load the nets, reduce them to normal form in one of the
loop forms and read the results back (numerals with their interaction counts,
or whole normal forms as text), or admit requests to a server and run its
epochs until all have finished.  The context, its workspace, its rule set and
the kernel compiled for the rules are kept by such a program and belong to the
prepared state.

    listed()            the cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) the state of a case: nets drawn from the seed
    run(state)          one pass
    work(case)          the bytes and operations a pass cannot do without
    exact(case, seed)   the numerals by their closed forms
"""
from __future__ import annotations

import functools
import math
import time
from dataclasses import dataclass

import numpy as np

# Unary arithmetic: the rules of the arithmetic workloads.
ARITH = """\
Add(y, r) = Z -> r = y;
Add(y, r) = S(x) -> Add(y, w) = x, r = S(w);
Dup(a, b) = Z -> a = Z, b = Z;
Dup(a, b) = S(x) -> Dup(p, q) = x, a = S(p), b = S(q);
Era = Z -> ;
Era = S(x) -> Era = x;
Mul(y, r) = Z -> Era = y, r = Z;
Mul(y, r) = S(x) -> Dup(y1, y2) = y, Mul(y1, w) = x, Add(y2, r) = w;
A(n, r) = Z -> r = S(n);
A(n, r) = S(m) -> A2(m, r) = n;
A2(m, r) = Z -> A(S(Z), r) = m;
A2(m, r) = S(n) -> Dup(m1, m2) = m, A(n, w) = S(m2), A(w, r) = m1;
Pred(r) = Z -> r = Z;
Pred(r) = S(x) -> r = x;
Fib(r) = Z -> r = Z;
Fib(r) = S(x) -> Fib2(r) = x;
Fib2(r) = Z -> r = S(Z);
Fib2(r) = S(x) -> Dup(a, b) = x, Fib(w1) = S(a), Fib(w2) = b, Add(w2, r) = w1;
"""

# The algae L-System A -> AB, B -> A.
LSYS = """\
SymA(r) = Z -> r = LeafA;
SymA(r) = S(k) -> Dup(k1, k2) = k, SymA(x) = k1, SymB(y) = k2, r = Cat(x, y);
SymB(r) = Z -> r = LeafB;
SymB(r) = S(k) -> SymA(r) = k;
Dup(a, b) = Z -> a = Z, b = Z;
Dup(a, b) = S(x) -> Dup(p, q) = x, a = S(p), b = S(q);
"""

# Binary trees, with constructors of two ports.
TREE = """\
Mirror(r) = Leaf -> r = Leaf;
Mirror(r) = Node(a, b) -> r = Node(y, x), Mirror(x) = a, Mirror(y) = b;
Leaves(r) = Leaf -> r = S(Z);
Leaves(r) = Node(a, b) -> Leaves(x) = a, Leaves(y) = b, Add(y, r) = x;
Drop = Leaf -> ;
Drop = Node(a, b) -> Drop = a, Drop = b;
Copy(p, q) = Leaf -> p = Leaf, q = Leaf;
Copy(p, q) = Node(a, b) -> Copy(a1, a2) = a, Copy(b1, b2) = b, p = Node(a1, b1), q = Node(a2, b2);
Left(r) = Leaf -> r = Leaf;
Left(r) = Node(a, b) -> r = a, Drop = b;
Swap(r) = Leaf -> r = Leaf;
Swap(r) = Node(a, b) -> r = Node(b, a);
Add(y, r) = Z -> r = y;
Add(y, r) = S(x) -> Add(y, w) = x, r = S(w);
"""

RULES = {"add": ARITH, "mul": ARITH, "ack": ARITH, "fib": ARITH, "lsys": LSYS, "tree": TREE, "serve": ARITH}


def listed():
    return [
        # the smallest call: one sum of two small numbers, as an interactive program asks for it
        {"name": "add_one", "kind": "add", "count": 1, "lo": 0, "hi": 16, "second": 16, "mode": "async"},
        # many short independent sums in one batch
        {"name": "add4096", "kind": "add", "count": 4096, "lo": 0, "hi": 256, "second": 256, "mode": "async"},
        # one long sum: a single chain of dependent interactions, no parallelism at all
        {"name": "chain20k", "kind": "add", "count": 1, "lo": 19000, "hi": 21000, "second": 64, "mode": "async"},
        # the benchmark's batch of products
        {"name": "mul2048", "kind": "mul", "count": 2048, "hi": 64, "mode": "async"},
        # a smaller batch of products of odd sizes, in the loop form that reduce() takes by default
        {"name": "mul333_default", "kind": "mul", "count": 333, "hi": 37, "mode": "persistent"},
        # Ackermann: few pairs at a time, of many rules
        {"name": "ack3", "kind": "ack", "first": 3, "lo": 4, "hi": 8, "count": 5, "mode": "async"},
        # Fibonacci, single nets: narrow at first and at the end
        {"name": "fib20_25", "kind": "fib", "lo": 20, "hi": 25, "count": 6, "mode": "async"},
        # Fibonacci, a batch that fills the device: the largest call
        {"name": "fib25x64", "kind": "fib", "lo": 22, "hi": 25, "count": 64, "mode": "async"},
        # the L-System word of half a million symbols, its normal form read back as text
        {"name": "lsys27", "kind": "lsys", "n": 27, "mode": "persistent"},
        # random binary trees copied, mirrored and counted: another rule set, constructors with two ports
        {"name": "tree512", "kind": "tree", "count": 512, "depth": 10, "mode": "async"},
        # the server: requests of every family, sizes spread over orders of magnitude
        {"name": "serve2000", "kind": "serve", "requests": 2000, "median": 1000, "cap": 100000, "epoch_us": 250},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["add", "add", "mul", "mul", "ack", "fib", "lsys", "tree", "serve"])
    mode = rng.choice(["async", "async", "persistent"])
    if kind == "add":
        if rng.random() < 0.4:  # few long sums
            lo = _log_int(rng, 300, 10000)
            return {"kind": kind, "count": rng.randint(1, 8), "lo": lo, "hi": lo + lo // 8 + 1, "second": rng.randint(1, 64),
                    "mode": "async"}
        return {"kind": kind, "count": _log_int(rng, 1, 4096), "lo": 0, "hi": _log_int(rng, 8, 256),
                "second": _log_int(rng, 8, 256), "mode": mode}
    if kind == "mul":
        return {"kind": kind, "count": _log_int(rng, 1, 2048), "hi": _log_int(rng, 8, 64), "mode": mode}
    if kind == "ack":
        hi = rng.randint(4, 8)
        return {"kind": kind, "first": rng.randint(2, 3), "lo": rng.randint(1, hi), "hi": hi, "count": rng.randint(1, 5),
                "mode": "async"}
    if kind == "fib":
        hi = rng.randint(10, 25)
        return {"kind": kind, "lo": max(1, hi - rng.randint(0, 6)), "hi": hi, "count": _log_int(rng, 1, 64), "mode": "async"}
    if kind == "lsys":
        return {"kind": kind, "n": rng.randint(13, 27), "mode": mode}
    if kind == "tree":
        return {"kind": kind, "count": _log_int(rng, 1, 512), "depth": rng.randint(5, 10), "mode": mode}
    return {"kind": kind, "requests": _log_int(rng, 64, 2000), "median": _log_int(rng, 100, 1000),
            "cap": _log_int(rng, 10000, 100000), "epoch_us": rng.choice([250, 500, 1000])}


# --- sizes: numbers of interactions, values ------------------------------------------

def _numeral(k):
    return "S(" * k + "Z" + ")" * k


def _add_count(m):
    return m + 1


def _mul_count(m, n):
    return n + 2 + m * (n + 3) + n * m * (m - 1) // 2


def _ack(m, n):
    return n + 1 if m == 0 else n + 2 if m == 1 else 2 * n + 3 if m == 2 else 2 ** (n + 3) - 3


@functools.lru_cache(maxsize=None)
def _ack_count(m, n):
    if m == 0:
        return 1
    if n == 0:
        return 2 + _ack_count(m - 1, 1)
    total = 2 + _ack_count(m - 1, 1)
    for k in range(1, n + 1):
        total += 2 + m + _ack_count(m - 1, _ack(m, k - 1))
    return total


@functools.lru_cache(maxsize=None)
def _fib(n):
    return n if n < 2 else _fib(n - 1) + _fib(n - 2)


@functools.lru_cache(maxsize=None)
def _fib_count(n):
    if n < 2:
        return n + 1
    return 2 + (n - 2 + 1) + _fib_count(n - 1) + _fib_count(n - 2) + _fib(n - 1) + 1


def _tree(rng, depth):
    """A random binary tree as (text, leaves, leaves below each node summed): full near the root, ragged below."""
    if depth == 0 or (depth < 8 and rng.random() < 0.2):
        return "Leaf", 1, 0
    a, x, i = _tree(rng, depth - 1)
    b, y, j = _tree(rng, depth - 1)
    return "Node(%s,%s)" % (a, b), x + y, x + y + i + j


@dataclass
class Request:
    arrival_s: float
    net: str
    size: int
    value: int


def _requests(case, rng):
    """Sums, products, Ackermann and Fibonacci in equal parts, sizes lognormal."""
    acks = sorted((_ack_count(a, b), a, b) for a in range(4) for b in range(8) if a < 3 or b < 7)
    fibs = sorted((_fib_count(n), n) for n in range(26))
    out = []
    for _ in range(case["requests"]):
        t = min(max(1.0, float(rng.lognormal(math.log(case["median"]), 2.16))), float(case["cap"]))
        fam = int(rng.integers(0, 4))
        if fam == 0:
            m, n = max(0, int(round(t)) - 1), int(rng.integers(0, 65))
            out.append(Request(0.0, "< r | Add(%s, r) = %s >" % (_numeral(n), _numeral(m)), _add_count(m), m + n))
        elif fam == 1:
            k = max(1, int((2 * t) ** (1 / 3)))
            m, n = int(rng.integers(max(0, k - 2), k + 1)), int(rng.integers(max(0, k - 2), k + 1))
            out.append(Request(0.0, "< r | Mul(%s, r) = %s >" % (_numeral(n), _numeral(m)), _mul_count(m, n), m * n))
        elif fam == 2:
            c, a, b = min(acks, key=lambda r: abs(math.log(r[0] / t)) if r[0] <= case["cap"] else math.inf)
            out.append(Request(0.0, "< r | A(%s, r) = %s >" % (_numeral(b), _numeral(a)), c, _ack(a, b)))
        else:
            c, n = min(fibs, key=lambda r: abs(math.log(r[0] / t)) if r[0] <= case["cap"] else math.inf)
            out.append(Request(0.0, "< r | Fib(r) = %s >" % _numeral(n), c, _fib(n)))
    return out


def _nets(case, seed):
    """The nets of a case: (text, value of its numeral, interactions), value -1 where the result is no numeral."""
    rng = np.random.default_rng(seed)
    kind, out = case["kind"], []
    if kind == "add":
        for _ in range(case["count"]):
            m, n = int(rng.integers(case["lo"], case["hi"] + 1)), int(rng.integers(0, case["second"] + 1))
            out.append(("< r | Add(%s, r) = %s >" % (_numeral(n), _numeral(m)), m + n, _add_count(m)))
    elif kind == "mul":
        for _ in range(case["count"]):
            m, n = (int(v) for v in rng.integers(0, case["hi"] + 1, 2))
            out.append(("< r | Mul(%s, r) = %s >" % (_numeral(n), _numeral(m)), m * n, _mul_count(m, n)))
    elif kind == "ack":
        # ack(a, b) + k, for each b of the range in turn
        span = case["hi"] - case["lo"] + 1
        for i in range(case["count"]):
            a, b, k = case["first"], case["hi"] - i % span, int(rng.integers(0, 1000))
            v = _ack(a, b)
            out.append(("< r | A(%s, w) = %s, Add(%s, r) = w >" % (_numeral(b), _numeral(a), _numeral(k)), v + k,
                        _ack_count(a, b) + _add_count(v)))
    elif kind == "fib":
        # fib(n) + k, for each n of the range in turn
        span = case["hi"] - case["lo"] + 1
        for i in range(case["count"]):
            n, k = case["hi"] - i % span, int(rng.integers(0, 1000))
            v = _fib(n)
            out.append(("< r | Fib(w) = %s, Add(%s, r) = w >" % (_numeral(n), _numeral(k)), v + k,
                        _fib_count(n) + _add_count(v)))
    elif kind == "lsys":
        # the word after n steps, and eight short ones in an order drawn from the seed
        for n in [case["n"]] + [int(v) for v in rng.permutation(np.arange(4, 12))]:
            out.append(("< r | SymA(r) = %s >" % _numeral(n), -1, -1))
    elif kind == "tree":
        # the leaves of a tree and of its mirror image, added
        for _ in range(case["count"]):
            text, leaves, below = _tree(rng, case["depth"])
            # copied, mirrored, counted twice; at each node the left count added to the right one, in both images
            steps = 4 * (2 * leaves - 1) + below + 2 * (leaves - 1) + _add_count(leaves)
            out.append(("< r | Copy(p, q) = %s, Mirror(u) = p, Leaves(a) = u, Leaves(b) = q, Add(b, r) = a >" % text,
                        2 * leaves, steps))
    return out


# --- capacities of a context, as a program sizes it for its batches -----------------------

def _pow2(n):
    return 1 << max(0, int(math.ceil(math.log2(max(1, n)))))


def _caps(case):
    kind = case["kind"]
    if kind == "add" and case["count"] == 1 and case["hi"] <= 64:
        return {}  # the defaults
    if kind == "add":
        slots = case["count"] * (case["hi"] + case["second"] + 4) * 2
        nets = 2 * case["count"]
    elif kind == "mul":
        slots, nets = case["count"] * (2 * case["hi"] ** 2 + 64), 2 * case["count"]
    elif kind == "ack":
        slots, nets = 1 << 22, 64
    elif kind == "fib":
        slots, nets = case["count"] * _fib_count(case["hi"]) // 4, 2 * case["count"]
    elif kind == "lsys":
        slots, nets = 1 << 22, 64
    else:
        slots, nets = case["count"] * (1 << case["depth"]) * 16, 2 * case["count"]
    slots = max(1 << 20, _pow2(slots))
    return dict(max_agents=slots, max_vars=slots, max_pairs=max(1 << 20, slots // 2 if kind == "lsys" else slots // 8),
                max_nets=max(64, _pow2(nets)))


@dataclass
class State:
    case: dict
    nets: list
    engine: object


def prepare(case, seed):
    import paper_1404_0076_gb300 as pkg
    from paper_1404_0076_gb300.serve import Server
    if case["kind"] == "serve":
        srv = Server(ARITH, device=0, budget_bytes=4 << 30, epoch_us=case["epoch_us"])
        return State(case, _requests(case, np.random.default_rng(seed)), srv)
    ev = pkg.Evaluator(device=0, **_caps(case))
    ev.load_rules(RULES[case["kind"]])
    if case["mode"] == "async":
        ev.build_jit()  # otherwise part of the first reduction
    return State(case, [t for t, _, _ in _nets(case, seed)], ev)


def run(state):
    case, ev = state.case, state.engine
    if case["kind"] == "serve":
        # a request loop: admit what has come in, run an epoch, collect what finished
        reqs = [(rid, r.net, r.size, 0.0) for rid, r in enumerate(state.nets)]
        done, admitted, t0 = [], 0, time.perf_counter()
        while admitted < len(reqs) or ev.busy():
            if admitted < len(reqs):
                admitted += ev.admit_many(reqs[admitted:admitted + 256], time.perf_counter() - t0)
            done.extend(ev.epoch(lambda: time.perf_counter() - t0))
        done.sort(key=lambda f: f.rid)
        return {"values": np.array([-1 if f.value is None else f.value for f in done], dtype=np.int64),
                "interactions": np.array([f.interactions for f in done], dtype=np.int64)}
    ev.reset()
    ids = ev.load_nets(state.nets)
    st = ev.reduce(ids, mode=case["mode"])
    total = np.array([st["interactions"]] + st["per_rule"], dtype=np.int64)
    if case["kind"] == "lsys":
        text = "".join(ev.readback(i) for i in ids)
        return {"text": np.frombuffer(text.encode(), dtype=np.uint8), "total": total}
    values, interactions = ev.readback_nats(ids)
    return {"values": np.array([-1 if v is None else v for v in values], dtype=np.int64),
            "interactions": np.array(interactions, dtype=np.int64), "total": total}


def _lsys_counts(n):
    """(symbols, characters of the normal form) after n steps from A, and from B."""
    a, b = (1, 5), (1, 5)
    for _ in range(n):
        a, b = (a[0] + b[0], len("Cat(, )") + a[1] + b[1]), a
    return a


def work(case):
    """Texts in, results out; one operation for each interaction."""
    if case["kind"] == "serve":
        reqs = _requests(case, np.random.default_rng(1))
        return {"bytes": sum(len(r.net) for r in reqs) + 16 * len(reqs), "flops": sum(r.size for r in reqs)}
    nets = _nets(case, 1)
    text = sum(len(t) for t, _, _ in nets)
    if case["kind"] == "lsys":
        sizes = [_lsys_counts(n) for n in [case["n"]] + list(range(4, 12))]
        # a symbol step for every Cat node and SymB, a duplication for every step count copied
        return {"bytes": text + sum(c for _, c in sizes), "flops": sum(5 * s for s, _ in sizes)}
    return {"bytes": text + 16 * len(nets), "flops": sum(c for _, _, c in nets)}


def exact(case, seed):
    if case["kind"] == "lsys":
        return None
    if case["kind"] == "serve":
        reqs = _requests(case, np.random.default_rng(seed))
        return {"values": np.array([r.value for r in reqs], dtype=np.int64),
                "interactions": np.array([r.size for r in reqs], dtype=np.int64)}
    nets = _nets(case, seed)
    return {"values": np.array([v for _, v, _ in nets], dtype=np.int64),
            "interactions": np.array([c for _, _, c in nets], dtype=np.int64), "total": None}
