"""Runs along lists (csrc/inet_async.cuh: chain_info, run_rule, pass_rule) and
the active pairs a right-hand side contains (csrc/inet_jit.cpp: inside_rules):
the specialised kernel against the oracle at the lengths where a run, a block
of neighbouring slots or a lane's slots end, for rules of every form that
runs take.  Everything compared is exact: normal form, interactions, rule
histogram, live agents."""
import os
import subprocess

import pytest

import workloads as W
from tests import oracle_runner

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

LENGTHS = [0, 1, 2, 7, 8, 9, 16, 17, 31, 32, 33, 40, 41, 65, 130]

LIST_RULES = """\
Append(y, r) = Nil -> r = y;
Append(y, r) = Cons(h, t) -> Append(y, w) = t, r = Cons(h, w);
Rev(acc, r) = Nil -> r = acc;
Rev(acc, r) = Cons(h, t) -> Rev(Cons(h, acc), r) = t;
Wrap(r) = Nil -> r = Nil;
Wrap(r) = Cons(h, t) -> r = Cons(S(h), w), Wrap(w) = t;
Snoc(u, r) = Snil -> r = Cons(u, Nil);
Scons(t, h) = Snoc(u, r) -> Snoc(u, w) = t, r = Cons(h, w);
Len(r) = Nil -> r = Z;
Len(r) = Cons(h, t) -> r = S(w), Len(w) = t, Drop = h;
Drop = E -> ;
Drop = S(x) -> Drop = x;
Turn(p, q) = Z -> p = Z, q = S(Z);
Turn(p, q) = S(x) -> Turn(q, p) = x;
Mix(r) = Z -> r = Z;
Mix(r) = S(x) -> r = S(w), Mix(w) = x;
Mix(r) = T(x) -> Mix(r) = x;
Odd(r) = S(x) -> Go(r) = Hop(x);
Odd(r) = Z -> r = Z;
Go(r) = Hop(x) -> Even(r) = x;
Even(r) = S(x) -> Odd(w) = x, r = T(w);
Even(r) = Z -> r = Z;
"""


def cons(n, elem="E"):
    return f"Cons({elem}, " * n + "Nil" + ")" * n


def snoc(n):
    return "Scons(" * n + "Snil" + ", E)" * n


def mixed(n):
    """S and T alternating in stretches of 1, 2, 3, .."""
    out, k, lab = [], 1, "S"
    while len(out) < n:
        out += [lab] * min(k, n - len(out))
        k, lab = k + 1, "T" if lab == "S" else "S"
    return "".join(x + "(" for x in out) + "Z" + ")" * n


def list_nets(n):
    half = n // 2
    return [
        f"< r | Append({cons(3)}, r) = {cons(n)} >",
        # the list is bound to a name, and is itself being produced
        f"< r | Append({cons(2)}, r) = x, Append({cons(n)}, x) = {cons(half)} >",
        f"< r | Append(Nil, r) = x, Append(y, x) = {cons(half)}, Append(Nil, y) = {cons(n - half)} >",
        f"< r | Rev(Nil, r) = {cons(n)} >",
        f"< r | Rev(Nil, x) = {cons(n, 'S(E)')}, Append({cons(1)}, r) = x >",
        f"< r | Wrap(x) = {cons(n)}, Wrap(r) = x >",
        f"< r | Snoc(E, r) = {snoc(n)} >",
        f"< r | Len(r) = x, Wrap(x) = {cons(n)} >",
        f"< p, q | Turn(p, q) = {W.numeral(n)} >",
        f"< r | Mix(r) = {mixed(n)} >",
        f"< r | Odd(r) = {W.numeral(n)} >",
        f"< a, r | Append(a, r) = {cons(n)} >",          # a free name at the end of the list
        f"< r | Mix(r) = x, Mix(x) = {W.numeral(half)} >",
    ]


def arith_nets(n):
    m = n % 19
    return [
        W.add_net(n, 3), W.mul_net(3, n), W.mul_net(n % 13, m), W.ack_net(2, m), W.fib_net(m % 13),
        f"< r | Add({W.numeral(n)}, r) = x, Add(Z, x) = {W.numeral(n)} >",
        f"< a, b | Dup(a, c) = {W.numeral(n)}, Dup(b, d) = c, Era = d >",
        f"< r | Era = {W.numeral(n)}, r = Z >",
        f"< r | Mul(y, r) = {W.numeral(m)}, Dup(y, z) = {W.numeral(n)}, Era = z >",
    ]


@pytest.mark.gpu
@pytest.mark.parametrize("free_nets", [False, True])
@pytest.mark.parametrize("slice_us", [0, 30])
@pytest.mark.parametrize("rules,family", [(LIST_RULES, list_nets), (W.ARITH_RULES, arith_nets)], ids=["lists", "arith"])
def test_runs_equal_the_oracle(rules, family, slice_us, free_nets):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a GPU"
    from paper_1404_0076_gb300 import Evaluator
    oracle_runner.build()
    nets = [t for n in LENGTHS for t in family(n)]
    exp = oracle_runner.run(rules, nets)
    assert all(o["status"] == "ok" for o in exp)
    with Evaluator(device=0, jit=True, free_nets=free_nets, max_agents=1 << 20, max_vars=1 << 20, max_pairs=1 << 16,
                   max_nets=1024) as ev:
        ev.load_rules(rules)
        for _ in range(2):  # the second time on slots that the first one freed and on a context in use
            ids = ev.load_nets(nets)
            ev.stage(ids)
            hist = [0] * len(ev.rules())
            for k in range(10000):
                st = ev.reduce([], mode="async", slice_us=slice_us, check=False)
                hist = [a + b for a, b in zip(hist, st["per_rule"])]
                if st["status"] != "STEP_LIMIT":
                    break
            assert st["status"] == "OK" and st["pending_pairs"] == 0
            assert ev.jit_info()["state"] == 1
            assert hist == [sum(o["per_rule"][r] for o in exp) for r in range(len(hist))]
            for i, net, o in zip(ids, nets, exp):
                info = ev.net_info(i)
                assert (ev.readback(i), info["interactions"], info["live_agents"]) == \
                    (o["result"], o["interactions"], o["live"]), net
            assert st["live_agents"] == sum(o["live"] for o in exp)
            if not free_nets:
                break
            ev.free(ids)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 9, 40])
def test_runs_in_an_arena_with_little_room(n):
    # far fewer slots than the grid's lanes could keep for themselves
    from paper_1404_0076_gb300 import Evaluator
    nets = arith_nets(n) * 4
    exp = oracle_runner.run(W.ARITH_RULES, nets)
    with Evaluator(device=0, jit=True, max_agents=1 << 15, max_vars=1 << 15, max_pairs=1 << 12, max_nets=64) as ev:
        ev.load_rules(W.ARITH_RULES)
        ids = ev.load_nets(nets)
        ev.reduce(ids, mode="async")
        for i, o in zip(ids, exp):
            assert ev.readback(i) == o["result"] and ev.net_info(i)["interactions"] == o["interactions"]


def test_rules_inside_a_right_hand_side(tmp_path):
    # on the CPU: the templates with reduced pairs, interpreted, against the
    # loaded ones, on nets that reach every rule
    exe = str(tmp_path / "inside_check")
    csrc = os.path.join(ROOT, "paper_1404_0076_gb300", "csrc")
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", os.path.join(ROOT, "include"), "-I", csrc,
                    os.path.join(ROOT, "tests", "inside_check.cpp"), os.path.join(csrc, "inet_text.cpp"), "-o", exe],
                   check=True)
    for rules, nets in ((LIST_RULES, [t for n in (0, 1, 2, 9) for t in list_nets(n)]),
                        (W.ARITH_RULES, [t for n in (0, 1, 5, 11) for t in arith_nets(n)])):
        rp, np_ = tmp_path / "rules.txt", tmp_path / "nets.txt"
        rp.write_text(rules)
        np_.write_text("\n".join(nets) + "\n")
        r = subprocess.run([exe, str(rp), str(np_)], capture_output=True, text=True)
        assert r.returncode == 0, r.stdout + r.stderr
        # some rule had a pair to reduce, and the nets applied it
        assert int(r.stdout.split()[0]) > 0 and int(r.stdout.split()[1]) > 0, r.stdout
