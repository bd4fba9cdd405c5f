"""A context that runs on recycled slots (csrc/inet_async.cuh, fill_stacks): the
same batch loaded, reduced and freed again and again in an arena a little
larger than its peak, where the bump pointer soon stands near the end and every
slot comes from the ring.  The results stay exact, and a batch takes about as
long as the first one did, whose slots came from the bump pointer."""
import pytest

import workloads as W


@pytest.mark.gpu
@pytest.mark.parametrize("count", [256, 2048])
def test_batches_on_recycled_slots(count):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a GPU"
    from paper_1404_0076_gb300 import Evaluator
    w = W.config1(count=count)
    expect = [(m * n, n + 2 + m * (n + 3) + n * m * (m - 1) // 2) for m, n in w.params]

    def rounds(max_agents, k):
        ms = []
        with Evaluator(device=0, jit=True, free_nets=True, max_agents=max_agents, max_vars=1 << 22, max_pairs=1 << 19,
                       max_nets=4096) as ev:
            ev.load_rules(W.ARITH_RULES)
            ev.build_jit()
            for _ in range(k):
                ids = ev.load_nets(w.nets)
                ms.append(ev.reduce(ids, mode="async")["device_ms"])
                assert list(zip(*ev.readback_nats(ids))) == expect
                ev.free(ids)
            usage = ev.arena_usage()
        assert usage["free_agent_slots"] == usage["agent_slots"] and usage["free_name_slots"] == usage["name_slots"]
        return usage["agent_slots"], ms

    used, _ = rounds(1 << 24, 2)
    # room for the next batch's records above the slots in use, and a little more
    ms = rounds(int(used * 1.12), 20)[1]
    assert sorted(ms[10:])[5] < 1.4 * ms[0], ms
