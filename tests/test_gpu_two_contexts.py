"""Contexts on streams and host threads of their own, all with kernels that want
every SM (cooperative launches): they take turns and give the same bits as one
after the other."""
import threading

import numpy as np
import pytest

from paper_1711_04471_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_contexts_side_by_side():
    import torch
    import paper_1711_04471_gb300 as P
    P.build()
    from paper_1711_04471_gb300.les import LES
    from paper_1711_04471_gb300.sw import SW
    inp = inputs.sw_hump(n=500)

    def sw(stream):
        with SW(inp.params(), inp.H, inp.eta0, stream=stream) as g:
            assert g.chip_plan() is not None
            for _ in range(20):
                g.step(37)
            return list(g.get_state().values()) + [np.array(g.volume())]

    def les(stream):
        with LES(72, 48, 40, stream=stream) as s:
            stats = s.step(4)
            return [s.get(f) for f in ("u", "v", "w", "p")] + [np.array([x["iters"] for x in stats])]

    jobs = [sw, les, sw, les]
    want = [job(None) for job in jobs]
    got = [None] * len(jobs)

    def run(k):
        got[k] = jobs[k](torch.cuda.Stream())

    threads = [threading.Thread(target=run, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for a, b in zip(want, got):
        assert b is not None
        for x, y in zip(a, b):
            assert np.array_equal(x, y)
