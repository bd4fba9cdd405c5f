"""Random rule sets of walkers over constructor terms, all of whose nets end:
each rule goes on to a smaller term, or to a later walker over one as large.
Constructors have up to three ports; walkers up to three, each an accumulator
that takes a term or an output that gives one, so the rules have any number of
output streams, of names and of agents, pass, rebuild, drop and copy what they
meet, and hold active pairs in their right-hand sides.  Drop and Copy are
there for every constructor."""
import random


class RuleSet:
    def __init__(self, seed: int, walkers: int = 4, constructors: int = 3):
        rng = self.rng = random.Random(seed)
        self.cons = [("N", 0)] + [(f"C{i}", rng.choice((1, 1, 2, 3))) for i in range(constructors)]
        self.tail = {c: rng.randrange(a) for c, a in self.cons if a}
        # a walker's ports: 'a' takes a term, 'o' gives one; at least one output
        self.walk = [(f"W{i}", "".join(rng.choice("ao") for _ in range(rng.randint(0, 2))) + "o") for i in range(walkers)]
        self.walk = [(w, "".join(rng.sample(s, len(s)))) for w, s in self.walk]
        rules = [f"Drop = {c}" + (f"({', '.join(f't{i}' for i in range(a))})" if a else "") + " -> " +
                 ", ".join(f"Drop = t{i}" for i in range(a)) + ";" for c, a in self.cons]
        for c, a in self.cons:
            t = [f"t{i}" for i in range(a)]
            kids = ["(" + ", ".join(f"{x}{i}" for i in range(a)) + ")" if a else "" for x in "ab"]
            rules.append(f"Copy(p, q) = {c}" + (f"({', '.join(t)})" if a else "") + " -> " +
                         ", ".join([f"Copy(a{i}, b{i}) = t{i}" for i in range(a)] + [f"p = {c}{kids[0]}", f"q = {c}{kids[1]}"]) + ";")
        for i in range(walkers):
            for c, a in self.cons:
                rules.append(self._rule(i, c, a))
        self.text = "\n".join(rules) + "\n"

    def _build(self, have, depth=1):
        """A term of constructors over the terms in `have` (each used at most once)."""
        rng = self.rng
        if depth == 0 or (have and rng.random() < 0.5):
            return have.pop(rng.randrange(len(have))) if have else "N"
        c, a = rng.choice(self.cons)
        return c if a == 0 else f"{c}({', '.join(self._build(have, depth - 1) for _ in range(a))})"

    def _rule(self, i, c, a):
        rng = self.rng
        w, sig = self.walk[i]
        ports = [f"p{k}" for k in range(len(sig))]
        lhs = f"{w}({', '.join(ports)}) = {c}" + (f"({', '.join(f't{k}' for k in range(a))})" if a else "")
        have = [p for p, s in zip(ports, sig) if s == "a"]
        outs = [p for p, s in zip(ports, sig) if s == "o"]
        eqs = []
        if a:
            tail = f"t{self.tail[c]}"
            have += [f"t{k}" for k in range(a) if f"t{k}" != tail]
            # the walker itself, mostly; a later one; or a later one over a new constructor
            j = i if rng.random() < 0.6 else rng.randrange(i, len(self.walk))
            v, vsig = self.walk[j]
            cons1 = [x for x in self.cons if x[1]]
            wrap = j > i and rng.random() < 0.5
            fresh = iter(f"w{k}" for k in range(8))
            args, given = [], []
            for k, s in enumerate(vsig):
                if s == "a":
                    # what the walker has in that port stays there, mostly
                    same = ports[k] if j == i and ports[k] in have and rng.random() < 0.7 else None
                    if same:
                        have.remove(same)
                    args.append(same or self._build(have, rng.randint(0, 1)))
                else:
                    own = ports[k] if j == i and ports[k] in outs and rng.random() < 0.35 else None
                    if own:
                        outs.remove(own)
                    args.append(own or next(fresh))
                    if not own:
                        given.append((args[-1], ports[k] if j == i else None))
            over = tail
            if wrap:
                cc, ca = rng.choice(cons1)
                kids = ["N" if not have else have.pop() for _ in range(ca)]
                if kids[self.tail[cc]] != "N":
                    have.append(kids[self.tail[cc]])
                kids[self.tail[cc]] = tail
                over = f"{cc}({', '.join(kids)})"
            eqs.append((f"{v}({', '.join(args)})" if args else v, over))
            # each new output goes, inside a constructor mostly, to one of the rule's
            for x, back in given:
                out = back if back in outs else (outs[0] if outs else None)
                if out is None:
                    eqs.append(("Drop", x))
                    continue
                outs.remove(out)
                term = x
                if rng.random() < 0.8:
                    cc, ca = rng.choice(cons1)
                    kids = [self._build(have, 0) for _ in range(ca)]
                    at = self.tail[cc]
                    if kids[at] != "N":
                        have.append(kids[at])
                    kids[at] = x
                    term = f"{cc}({', '.join(kids)})"
                eqs.append((out, term))
        for out in outs:
            eqs.append((out, self._build(have, 1)))
        eqs += [("Drop", x) for x in have]
        rng.shuffle(eqs)
        return f"{lhs} -> {', '.join(f'{x} = {y}' for x, y in eqs)};"

    def term(self, n: int) -> str:
        """A term of n constructors along the tails, in stretches of one."""
        rng = self.rng
        cons1 = [x for x in self.cons if x[1]]
        head, foot, c = [], [], rng.choice(cons1)
        for _ in range(n):
            if rng.random() < 0.15:
                c = rng.choice(cons1)
            kids = ["N" if rng.random() < 0.8 else self._build([], 1) for _ in range(c[1])]
            at = self.tail[c[0]]
            head.append(f"{c[0]}(" + "".join(k + ", " for k in kids[:at]))
            foot.append("".join(", " + k for k in kids[at + 1:]) + ")")
        return "".join(head) + "N" + "".join(reversed(foot))

    def net(self, n: int) -> str:
        """One to three walkers, each over the last one's output or a term of its own."""
        rng = self.rng
        eqs, results, over = [], [], self.term(n)
        k = 0
        for _ in range(rng.randint(1, 3)):
            w, sig = rng.choice(self.walk + [("Copy", "oo")])
            args, outs = [], []
            for s in sig:
                if s == "a":
                    args.append(self.term(rng.randint(0, 3)) if rng.random() < 0.7 else f"x{k}")
                    if args[-1] == f"x{k}":
                        eqs.append(f"x{k} = {self.term(rng.randint(0, 3))}")
                else:
                    args.append(f"x{k}")
                    outs.append(f"x{k}")
                k += 1
            eqs.append(f"{w}({', '.join(args)}) = {over}")
            over = outs[0]
            results += outs[1:]
        results.append(over)
        rng.shuffle(eqs)
        return f"< {', '.join(results)} | {', '.join(eqs)} >"
