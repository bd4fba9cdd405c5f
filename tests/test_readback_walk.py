"""Numeral readback by warps (csrc/inet_readback.cuh, k_nat_walk): lengths
around the 32 slots of a round trip and around the budget beyond which a
numeral is ranked, laid out in order, in reverse, scattered and through names,
against the closed forms."""
import pytest

import workloads as W

LENGTHS = [0, 1, 30, 31, 32, 33, 63, 64, 65, 255, 256, 257, 1000, 8160, 8191, 8192, 8193, 8225]


@pytest.mark.gpu
@pytest.mark.parametrize("begin_end", [False, True])
def test_numerals_of_every_layout(begin_end):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a GPU"
    from paper_1404_0076_gb300 import Evaluator
    fib = [0, 1]
    while len(fib) < 20:
        fib.append(fib[-1] + fib[-2])
    nets, values = [], []
    for n in LENGTHS:
        nets += [f"< {W.numeral(n)} | >", W.add_net(n, 5), W.add_net(5, n),
                 f"< r | Dup(r, e) = {W.numeral(n)}, Era = e >", f"< r | Dup(e, r) = {W.numeral(n)}, Era = e >",
                 f"< r | r = {W.numeral(n)} >"]
        values += [n, n + 5, n + 5, n, n, n]
    nets += [W.fib_net(k) for k in range(20)] + ["< S(S(x)), x | >", "< r | r = Era >", "< S(Era) | >"]
    values += fib + [None, None, None]
    with Evaluator(device=0, max_agents=1 << 21, max_vars=1 << 21, max_pairs=1 << 16, max_nets=512) as ev:
        ev.load_rules(W.ARITH_RULES)
        ids = ev.load_nets(nets)
        ev.reduce(ids, mode="async")
        for order in (ids, ids[::-1], ids[:1], ids[-1:]):
            if begin_end:
                ev.readback_nats_begin(order)
                got = ev.readback_nats_end(True)[0]
            else:
                got = ev.readback_nats(order)[0]
            assert list(got) == [values[i] for i in order]
