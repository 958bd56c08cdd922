"""GPU: what a call keeps for later calls, and what stays apart inside a call:
captured step graphs against fields set anew, waits that run out, non-finite
particles, one order of the sums whatever a kernel outputs beside u."""
import math

import numpy as np
import pytest
import torch

import paper_2107_01104_gb300 as trk
import synth

pytestmark = pytest.mark.gpu
L = 2 * math.pi
F64, F32, BF16 = trk.TRK_F64, trk.TRK_F32, trk.TRK_BF16X2


def velocity(N, seed):
    return torch.from_numpy(synth.velocity_field_np(N, min(10, N // 3), seed)).cuda()


def points(n, seed=0, lo=0.0, hi=L):
    return torch.from_numpy(np.random.default_rng(seed).uniform(lo, hi, (3, n))).cuda()


# dense sets (slab launches, captured with the field's address and tensor maps by
# value) and a set of the descriptors' route, stepped again after the field was
# re-allocated while something else took the memory it had
@pytest.mark.parametrize("storage", [F32, BF16])
def test_batched_graph_after_the_field_moved(storage):
    N, n, steps = 32, 40000, 7
    specs = [(n, 6, 1), (n, 8, 0), (300, 4, 0)]

    def run(t):
        sets = []
        for k, (m, I, deriv) in enumerate(specs):
            pos = points(m, seed=k)
            sets.append(dict(pos=pos, rhs=0.1 * torch.cos(pos.float()), I=I, m=I // 2 - 1, family=trk.TRK_SPLINE,
                             out=outs[k], deriv=deriv))
        t.advance_batched(sets, 4e-3, steps, history_valid=True)
        t.sync()
        return [s["pos"] for s in sets] + [s["rhs"] for s in sets] + [o.clone() for o in outs]

    outs = [torch.zeros((9 if d else 3, m), device="cuda") for m, _, d in specs]
    a, b = velocity(N, 1), velocity(N, 2)
    t = trk.Tracker(N, storage=storage)
    t.set_field(a)
    run(t)
    t.set_field(torch.cat([a, a, a, a]))      # another size: the three-component field is freed
    taker = trk.Tracker(N, storage=storage)
    taker.set_field(torch.full_like(a, 1e3))  # ... and its memory taken
    t.set_field(b)
    got = run(t)
    fresh = trk.Tracker(N, storage=storage)
    fresh.set_field(b)
    for x, y in zip(got, run(fresh)):
        assert torch.equal(x, y)
    for x in (t, taker, fresh):
        x.close()
