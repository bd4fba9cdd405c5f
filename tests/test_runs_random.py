"""Runs along lists and the active pairs inside right-hand sides, on rule sets
drawn at random (tests/random_walkers.py) and on lists as long as the longest
runs: the specialised kernel and the compiled pairs (csrc/inet_inside.h) against
the oracle and the loaded rules.  Everything compared is exact: normal form,
interactions, rule histogram, live agents."""
import os
import subprocess

import pytest

import workloads as W
from tests import oracle_runner
from tests.random_walkers import RuleSet

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def rule_set(seed):
    return RuleSet(seed, walkers=(2, 3, 4, 8)[seed % 4], constructors=(2, 3, 4)[seed // 2 % 3])


def test_random_rules_inside_a_right_hand_side(tmp_path):
    # on the CPU, with the sequential interpreter of tests/inside_check.cpp
    exe = str(tmp_path / "inside_check")
    csrc = os.path.join(ROOT, "paper_1404_0076_gb300", "csrc")
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", os.path.join(ROOT, "include"), "-I", csrc,
                    os.path.join(ROOT, "tests", "inside_check.cpp"), os.path.join(csrc, "inet_text.cpp"), "-o", exe],
                   check=True)
    sets = rules = applied = 0
    for seed in range(60):
        rs = rule_set(seed)
        rp, np_ = tmp_path / "rules.txt", tmp_path / "nets.txt"
        rp.write_text(rs.text)
        np_.write_text("\n".join(rs.net(n) for n in (0, 1, 2, 3, 9, 40)) + "\n")
        r = subprocess.run([exe, str(rp), str(np_)], capture_output=True, text=True)
        if "more than 8 agents" in r.stdout:
            continue    # no template: the rule set does not load
        assert r.returncode == 0, (seed, r.stdout + r.stderr)
        sets += 1
        rules += int(r.stdout.split()[0])
        applied += int(r.stdout.split()[1])
    assert sets > 40 and rules > 20 and applied > 20


def compare(ev, nets, exp, mode="async", slice_us=0):
    ev.reset()
    ids = ev.load_nets(nets)
    ev.stage(ids)
    hist = [0] * len(ev.rules())
    for _ in range(20000):
        st = ev.reduce([], mode=mode, slice_us=slice_us, check=False)
        hist = [a + b for a, b in zip(hist, st["per_rule"])]
        if st["status"] != "STEP_LIMIT":
            break
    assert st["status"] == "OK" and st["pending_pairs"] == 0
    assert hist == [sum(o["per_rule"][r] for o in exp) for r in range(len(hist))]
    for i, net, o in zip(ids, nets, exp):
        info = ev.net_info(i)
        assert (ev.readback(i), info["interactions"], info["live_agents"]) == \
            (o["result"], o["interactions"], o["live"]), net


# 15, 30, 20 and 50 rules; constructors and walkers of one to three ports
@pytest.mark.gpu
@pytest.mark.parametrize("seed", [61, 67, 69, 71])
def test_random_rules_equal_the_oracle(seed):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a GPU"
    from paper_1404_0076_gb300 import Evaluator
    oracle_runner.build()
    rs = rule_set(seed)
    nets = [rs.net(n) for n in (0, 1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 33, 40, 63, 64, 65, 130) for _ in range(3)]
    lone = [rs.net(n) for n in (515, 1030)]
    exp = oracle_runner.run(rs.text, nets + lone)
    assert all(o["status"] == "ok" for o in exp)
    exp, exp_lone = exp[:len(nets)], exp[len(nets):]
    with Evaluator(device=0, jit=True, free_nets=bool(seed // 2 % 2), max_agents=1 << 20, max_vars=1 << 20,
                   max_pairs=1 << 16, max_nets=1024) as ev:
        ev.load_rules(rs.text)
        ev.build_jit()
        compare(ev, nets, exp)
        compare(ev, nets, exp, slice_us=30)
        compare(ev, nets * 8, exp * 8)      # warps of many lanes
        compare(ev, nets, exp, mode="persistent")
        for net, o in zip(lone, exp_lone):       # a warp's only lane
            compare(ev, [net], [o])
        assert ev.jit_info()["state"] == 1


@pytest.mark.gpu
def test_lists_longer_than_a_run():
    # around the most interactions of one run of a warp's only lane (512), and
    # lists whose links go through names, each and one after another
    import torch
    assert torch.cuda.is_available(), "GPU tests need a GPU"
    from paper_1404_0076_gb300 import Evaluator
    oracle_runner.build()
    nets = [f(n) for n in (509, 510, 511, 512, 513, 514, 515, 516, 1023, 1024, 1025, 1026, 1029)
            for f in (lambda n: W.add_net(n, 2), lambda n: f"< a, b | Dup(a, b) = {W.numeral(n)} >",
                      lambda n: f"< r | Era = {W.numeral(n)}, r = Z >", lambda n: W.mul_net(n, 0))]
    for n in (600, 1100):
        links = ", ".join(f"x{i} = S(x{i + 1})" for i in range(n))
        nets += [f"< r | Add(Z, r) = x0, {links}, x{n} = Z >", f"< a, b | Dup(a, b) = x0, {links}, x{n} = Z >"]
    for n in (1023, 1025, 3000):
        names = ", ".join(f"x{i} = x{i + 1}" for i in range(n))
        nets += [f"< r | Add(Z, r) = S(x0), {names}, x{n} = S(Z) >", f"< a, b | Dup(a, b) = S(x0), {names}, x{n} = S(Z) >",
                 f"< r | Add(Z, r) = S(x0), {names} >"]
    exp = oracle_runner.run(W.ARITH_RULES, nets)
    assert all(o["status"] == "ok" for o in exp)
    with Evaluator(device=0, jit=True, max_agents=1 << 20, max_vars=1 << 20, max_pairs=1 << 16, max_nets=1024) as ev:
        ev.load_rules(W.ARITH_RULES)
        ev.build_jit()
        for net, o in zip(nets, exp):
            compare(ev, [net], [o])
        compare(ev, nets, exp)
        compare(ev, nets, exp, slice_us=30)
        assert ev.jit_info()["state"] == 1
