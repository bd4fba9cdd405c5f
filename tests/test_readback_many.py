"""Numeral readback of more nets than the device holds warps for, where a few
lanes walk each net (csrc/inet_readback.cuh, k_nat_walk): lengths around their
window and around the budget beyond which a numeral is ranked, in slot order,
scattered and through names, against the closed forms."""
import pytest

import workloads as W


@pytest.mark.gpu
@pytest.mark.parametrize("begin_end", [False, True])
def test_numerals_of_many_nets(begin_end):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a GPU"
    from paper_1404_0076_gb300 import Evaluator
    fib = [0, 1]
    while len(fib) < 17:
        fib.append(fib[-1] + fib[-2])
    nets = [f"< {W.numeral(n)} | >" for n in (0, 1, 2, 3, 4, 5, 7, 8, 9)] + [W.add_net(n, 3) for n in (0, 1, 3, 4, 5)] + \
        [W.fib_net(k) for k in range(12)] + [f"< r | Dup(r, e) = {W.numeral(6)}, Era = e >", "< S(x) | >", "< S(Era) | >"]
    values = [0, 1, 2, 3, 4, 5, 7, 8, 9] + [3, 4, 6, 7, 8] + fib[:12] + [6, None, None]
    many = 24000
    nets, values = (nets * (many // len(nets) + 1))[:many], (values * (many // len(values) + 1))[:many]
    # beyond the budget of 256 round trips of 4 slots, or of one scattered agent each
    nets += [f"< {W.numeral(n)} | >" for n in (1019, 1020, 1021, 1025, 3000)] + [W.fib_net(k) for k in (13, 14, 16)]
    values += [1019, 1020, 1021, 1025, 3000] + [fib[k] for k in (13, 14, 16)]
    with Evaluator(device=0, max_agents=1 << 21, max_vars=1 << 21, max_pairs=1 << 17, max_nets=1 << 15) as ev:
        ev.load_rules(W.ARITH_RULES)
        ids = ev.load_nets(nets)
        ev.reduce(ids, mode="async")
        if begin_end:
            ev.readback_nats_begin(ids)
            got = ev.readback_nats_end(True)[0]
        else:
            got = ev.readback_nats(ids)[0]
    assert list(got) == values
