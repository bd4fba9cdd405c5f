"""A record that holds a word which is neither an agent nor a name: whichever
equation of a right-hand side the word ends up in, every loop form reports
INET_ERR_STATE instead of dropping the equation."""
import pytest

# one equation per argument: the k-th port of F and G is a side of equation k
RULES = """\
F(a, b, c) = G(d, e) -> P = a, P = b, P = c, P = d, P = e;
P = Z -> ;
"""


@pytest.mark.gpu
@pytest.mark.parametrize("mode,jit", [("plain", False), ("graph", False), ("persistent", False), ("async", False),
                                      ("async", True)])
@pytest.mark.parametrize("word", [0, 7])  # EMPTY; a tag that no word carries
def test_corrupt_word_is_reported(mode, jit, word):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a GPU"
    from paper_1404_0076_gb300 import Evaluator
    for port in range(5):
        with Evaluator(device=0, jit=jit, max_agents=1 << 12, max_vars=1 << 12, max_pairs=1 << 10, max_nets=64) as ev:
            ev.load_rules(RULES)
            ids = [ev.load_net("< | F(Z, Z, Z) = G(Z, Z) >")]
            ev.stage(ids)
            # F's record is followed by those of its arguments, then G's
            ws = ev._ws[(-ev._ws.data_ptr()) % 256:]
            w = ws[:ws.numel() // 4 * 4].view(torch.int32)
            f = [(1 << 2) | 1, (2 << 2) | 1, (3 << 2) | 1]
            at = torch.nonzero((w[1:-20] == f[0]) & (w[2:-19] == f[1]) & (w[3:-18] == f[2]) &
                               (w[17:-4] == (5 << 2 | 1)) & (w[18:-3] == (6 << 2 | 1))).flatten().tolist()
            assert len(at) == 1
            w[at[0] + (1 + port if port < 3 else 17 + port - 3)] = word
            st = ev.reduce([], mode=mode, check=False)
            assert st["status"] == "STATE", (port, st["status"])
            # the context is usable again after a reset
            ev.reset()
            ids = [ev.load_net("< | F(Z, Z, Z) = G(Z, Z) >")]
            st = ev.reduce(ids, mode=mode)
            assert st["interactions"] == 6 and st["live_agents"] == 0
