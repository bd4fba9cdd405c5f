"""serve() while its parser thread still holds the only requests left (CPU)."""
import time

from paper_1404_0076_gb300.serve import Server
from tests.test_serving import FakeEvaluator, Req


class SlowParser(FakeEvaluator):
    def parse(self, texts):
        time.sleep(0.05)
        return super().parse(texts)


def test_requests_being_parsed_are_served():
    srv = Server("", budget_bytes=64 << 20, max_pairs=1 << 10, make_evaluator=SlowParser)
    for count in (1, 40):
        done = srv.serve([Req(0.0, f"n:{k % 3 + 1}", k % 3 + 1) for k in range(count)], time_scale=0.0)
        assert sorted(f.rid for f in done) == list(range(count))
