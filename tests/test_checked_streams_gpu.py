"""The bounds-checked build on the streaming passes of a step (source, limiter,
closing statistics, displacements): blocks that take parts of several tiles'
columns, the 16-wide tile, and grids that no tile fits; and the cluster's stores
into its neighbours with every form of the schedule."""
import pytest

import test_checked_gpu as T

pytestmark = pytest.mark.gpu

CASES = [
    ((16, 1024, 16), "mixed", {}),       # 16-wide tiles, 2.2 planes a block
    ((8, 256, 256), "mixed", {}),        # 32-wide tiles, 4.5 planes a block
    ((256, 8, 32), "fp64", {}),          # pieces of one plane
    ((8, 16, 16), "fp64", {}),           # one tile, fewer planes than blocks
    ((64, 32, 8), "mixed", {}),          # no tile fits
    ((32, 32, 32), "mixed", {"nu1": 0, "nu2": 2}),
    ((32, 32, 32), "mixed", {"nu1": 2, "nu2": 0}),
    ((64, 64, 64), "mixed", {"nu1": 0, "nu2": 1, "coarse_faces": 0}),
]


def test_streaming_passes_stay_within_their_arrays(tmp_path, monkeypatch):
    monkeypatch.setattr(T, "CASES", CASES)
    T.test_checked_build_reports_no_failed_check_and_gives_the_same_bits(tmp_path)
