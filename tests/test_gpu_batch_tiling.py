"""SWBatch.get_tiling reports the tiling in use: set explicitly, the same one
does the same."""
import numpy as np
import pytest

from paper_1711_04471_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_get_tiling_reports_what_runs(tmp_path):
    import paper_1711_04471_gb300 as P
    P.build()
    from paper_1711_04471_gb300.sw import SWBatch
    ms = [inputs.sw_ensemble_member(n, 77, k) for k, n in enumerate((64, 90, 130, 201))]
    cache = str(tmp_path / "tune.txt")
    with SWBatch(ms) as a, SWBatch(ms) as b, SWBatch(ms) as c:
        T, rows = a.get_tiling()
        # a few grids of one strip or two: 128 rows would leave most blocks without an item
        assert T == 3 and 8 <= rows < 128 and rows % 8 == 0
        b.set_tiling(T, rows)
        assert b.get_tiling() == (T, rows)
        for x in (a, b):
            x.step(20)
        sa, sb = ([x.get_state(m) for m in range(4)] for x in (a, b))
        pair = b.autotune(trial_steps=12, cache_path=cache)
        automatic = open(cache).read().split()[-1] == "auto"
        assert b.get_tiling() == ((T, rows) if automatic else pair)
        c.autotune(trial_steps=12, cache_path=cache)       # from the file
        assert c.get_tiling() == b.get_tiling()
        b.set_tiling(2, 64)
        assert b.get_tiling() == (2, 64)
    for m in range(4):
        for f in ("eta", "u", "v"):
            assert np.array_equal(sa[m][f], sb[m][f])
