"""The stopping rule as the host watches it: a solve that reports to its caller enqueues no steps behind
the stop, and more solves at once than there are slots for that give the same results."""
import os
import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2301_06384_gb300 import kb as _kb
    if not os.path.exists(_kb.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    return _kb


KW = dict(t=0.5, tol=1e-4)


def test_steps_behind_the_stop_are_not_enqueued(kb):
    import torch
    g = synth.random_geometric_graph(6000, 10, seed=8)
    nodes = np.random.default_rng(0).choice(np.nonzero(np.diff(g.rowptr) > 6)[0], size=9, replace=False).astype(np.int32)
    with kb.Graph.from_csr(g) as G:
        counts = []
        for info in (True, False):
            a = kb.kb_launch_counter()
            r = kb.kernel_columns(G, "cbl", "exp", nodes, 100, info=info, **KW)
            torch.cuda.synchronize()
            counts.append(kb.kb_launch_counter() - a)
            if info:
                Y, steps = r[0], r[1]["steps_done"]
        assert torch.equal(Y, r)
        assert 8 <= steps <= 48
        # ten launches a step; two steps run on behind a check, a check and the end take some 20
        assert counts[0] < counts[1] * (steps + 10) / 100


def test_more_solves_than_slots(kb):
    import torch
    g = synth.random_geometric_graph(3000, 10, seed=9)
    rng = np.random.default_rng(1)
    cand = np.nonzero(np.diff(g.rowptr) > 6)[0]
    sets = [rng.choice(cand, size=1 + i % 7, replace=False).astype(np.int32) for i in range(80)]   # (64 slots)
    with kb.Graph.from_csr(g) as G:
        want = [kb.kernel_columns(G, "cbl", "exp", s, 100, info=True, **KW) for s in sets]
        torch.cuda.synchronize()
        got, start = [None] * len(sets), threading.Barrier(len(sets))

        def work(i, Y, stream):
            start.wait()
            for _ in range(3):
                got[i] = kb.kb_krylov_apply(G, "cbl", "exp", kb.make_params(**KW), sets[i], sets[i].size, 100, Y,
                                            stream=stream, info=True)

        Ys = [torch.zeros(g.n, s.size, device="cuda") for s in sets]
        streams = [torch.cuda.Stream() for _ in sets]
        torch.cuda.synchronize()
        threads = [threading.Thread(target=work, args=(i, Ys[i], streams[i])) for i in range(len(sets))]
        for t in threads:
            t.start()
        for t in threads:
            t.join(120)
        torch.cuda.synchronize()
        for i, (Y, info) in enumerate(want):
            assert got[i] == info and torch.equal(Ys[i], Y)
