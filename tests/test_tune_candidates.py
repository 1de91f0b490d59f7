"""The autotuner's default candidates hold every number of threads per atom that
the library can choose by itself, so that a tuned layout is no worse."""
import inspect

import paper_2603_07321_gb300 as P
from paper_2603_07321_gb300.tune import tune


def test_default_candidates_hold_every_lane_count():
    lanes = inspect.signature(tune).parameters["lanes"].default
    accepted = [n for n in range(1, 33)
                if P.pta_footprint_bytes(P.make_specimen(4), P.default_params(lanes=n))]
    assert sorted(lanes) == accepted == [1, 2, 4, 8, 16]
