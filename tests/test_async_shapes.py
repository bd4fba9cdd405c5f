"""Where the asynchronous kernel's time must not depend on what a batch does not
use (csrc/inet_async.cuh)."""
import pytest

import workloads as W


def device_ms(ev, nets, times):
    out, got = [], []
    for _ in range(times):
        ev.reset()
        ids = ev.load_nets(nets)
        st = ev.reduce(ids, mode="async")
        out.append(st["device_ms"])
        got.append((st["interactions"], ev.readback(ids[0])))
    assert all(g == got[0] for g in got)
    return min(out), got[0]


@pytest.mark.gpu
def test_general_kernel_keeps_its_blocks_with_the_largest_rule_sets():
    # 64 rules and 57 symbols fill the tables in shared memory: still two
    # blocks an SM (with one, the batch takes 1.28 times as long)
    import torch
    assert torch.cuda.is_available(), "GPU tests need a GPU"
    from paper_1404_0076_gb300 import Evaluator
    pads = "".join(f"Pad{i}(a, b) = Z -> a = b;\n" for i in range(64 - W.ARITH_RULES.count("->")))
    nets = W.config1().nets
    got = []
    for rules in (W.ARITH_RULES, W.ARITH_RULES + pads):
        with Evaluator(device=0, jit=False, max_agents=1 << 24, max_vars=1 << 24, max_pairs=1 << 20, max_nets=4096) as ev:
            ev.load_rules(rules)
            got.append(device_ms(ev, nets, 5))
    assert got[0][1] == got[1][1]
    assert got[1][0] < 1.15 * got[0][0], got


@pytest.mark.gpu
def test_a_list_taken_one_agent_at_a_time_is_not_made_in_runs():
    # the L-System's Dup copies numerals that only SymA and SymB take, one S at
    # a time; with a rule that walks such lists Dup is reduced in runs, which
    # hold the copies back (measured: 1.6 times as long)
    import torch
    assert torch.cuda.is_available(), "GPU tests need a GPU"
    from paper_1404_0076_gb300 import Evaluator
    walker = "Walk(r) = Z -> r = Z;\nWalk(r) = S(x) -> Walk(w) = x, r = S(w);\n"
    got = []
    for rules in (W.LSYS_RULES, W.LSYS_RULES + walker):
        with Evaluator(device=0, jit=True, max_agents=1 << 22, max_vars=1 << 22, max_pairs=1 << 20, max_nets=64) as ev:
            ev.load_rules(rules)
            ev.build_jit()
            got.append(device_ms(ev, [W.lsys_net(16)], 12))
            assert ev.jit_info()["state"] == 1
    assert got[0][1] == got[1][1]
    assert got[0][0] < 0.85 * got[1][0], got
