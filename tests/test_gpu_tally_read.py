"""mc_tally_read from several threads of one context: each gets its own tally."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("slots", [1, 1 << 16, (1 << 16) + 1])
def test_reads_side_by_side(slots):
    import torch

    import paper_2403_06362_gb300 as mc
    from paper_2403_06362_gb300 import workloads as W

    ctx = mc.Context(0)
    prob = W.to_mc_problem(W.slab_problem(10.0, 1.0, 0.5, 100, slots, 1, 0), mc)
    probs = mc.problem_array([prob])
    tallies = [mc.Tally(slots, 1) for _ in range(4)]
    for i, t in enumerate(tallies):
        t.bins.copy_(torch.arange(slots, device="cuda") * 8 + i)
        t.counts.fill_(100 + i)
    torch.cuda.synchronize()
    want = [t.bins.cpu().numpy().reshape(1, slots) for t in tallies]
    bad = []

    def read(i):
        stream = torch.cuda.Stream()
        for _ in range(20):
            r = mc.mc_tally_read(ctx, probs, 0, tallies[i].c, stream, check=False)
            if not np.array_equal(r.raw, want[i]) or set(r.counts.values()) != {100 + i}:
                bad.append(i)

    threads = [threading.Thread(target=read, args=(i,)) for i in range(len(tallies))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
