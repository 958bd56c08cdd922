"""GPU: what a call keeps for later calls, and what stays apart inside a call:
captured step graphs against fields set anew, waits that run out, non-finite
particles."""
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


# A wait limit of no polls: every wait for a copy of the field gives up, so nothing
# moves and nothing is written; of one poll: some do, and a particle has either made
# the step or stayed.  Either way every particle is there once, and the tracker says so.
def stopped(t):
    with pytest.raises(trk.TrackerError) as e:
        t.sync()
    assert e.value.status == trk.TRK_ECUDA and "did not complete" in str(e.value)


@pytest.mark.parametrize("storage,I,kind", [(F32, 4, trk.TRK_STEP_COLUMN), (F32, 6, trk.TRK_STEP_COLUMN),
                                            (F32, 8, trk.TRK_STEP_BLOCK), (BF16, 6, trk.TRK_STEP_BLOCK),
                                            (F64, 6, trk.TRK_STEP_BLOCK)])
@pytest.mark.parametrize("scheme", [trk.TRK_RK2, trk.TRK_AB3])
def test_waits_that_run_out(monkeypatch, storage, I, kind, scheme):
    N, n, dt = 64, 70001, 4e-3
    u, pos = velocity(N, 3), points(n)
    rhs = 0.1 * torch.cos(pos.float()).repeat(2, 1, 1)

    def tracker(limit):
        monkeypatch.delenv("TRK_WAIT_LIMIT", raising=False)
        if limit is not None:
            monkeypatch.setenv("TRK_WAIT_LIMIT", str(limit))
        t = trk.Tracker(N, I=I, m=I // 2 - 1, storage=storage)
        t.set_field(u)
        t.set_step_kernel(kind)
        return t

    def advance(t, steps):
        p, r = pos.clone(), rhs.clone()
        if scheme == trk.TRK_RK2:
            t.advance(p, dt, steps)
            return p, p
        t.advance(p, dt, steps, scheme, rhs=r, history_valid=2)
        return p, r

    t = tracker(0)
    p, r = advance(t, 6)
    stopped(t)
    assert torch.equal(p, pos) and (scheme == trk.TRK_RK2 or torch.equal(r, rhs))
    out = torch.full((3, n), 7.0, dtype=torch.float64 if storage == F64 else torch.float32, device="cuda")
    t.interpolate(pos, out_dtype=out.dtype, out=out)
    stopped(t)
    assert (out == 7).all()
    t.close()

    whole = tracker(None)
    want, _ = advance(whole, 1)
    whole.sync()
    t = tracker(1)
    for _ in range(3):
        p, _ = advance(t, 1)
        try:
            t.sync()
        except trk.TrackerError as e:
            assert e.status == trk.TRK_ECUDA
        assert ((p == want).all(0) | (p == pos).all(0)).all()
    t.close()
    whole.close()


@pytest.mark.parametrize("I", [4, 6, 8])
def test_adjoint_and_batched_waits_that_run_out(monkeypatch, I):
    monkeypatch.setenv("TRK_WAIT_LIMIT", "0")
    N, n = 64, 70001
    t = trk.Tracker(N, I=I, m=I // 2 - 1, storage=F32)
    t.set_field(velocity(N, 3))
    t.set_step_kernel(trk.TRK_STEP_BLOCK)
    pos = points(n)
    lam = torch.sin(3 * pos)
    gf = torch.zeros((3, N, N, N), dtype=torch.float64, device="cuda")
    gpos, _ = t.adjoint(pos, lam, 4e-3, 3, 2, grad_field=gf)
    stopped(t)
    assert torch.equal(gpos, lam) and not gf.any()
    for deriv in (0, 1):
        s = dict(pos=pos.clone(), rhs=torch.cos(pos.float()), I=I, m=I // 2 - 1, family=trk.TRK_SPLINE, deriv=deriv,
                 out=torch.full((9 if deriv else 3, n), 7.0, device="cuda"))
        t.advance_batched([s], 4e-3, 5, history_valid=True)
        stopped(t)
        assert torch.equal(s["pos"], pos) and torch.equal(s["rhs"], torch.cos(pos.float())) and (s["out"] == 7).all()
    t.close()


# A non-finite lambda, and a non-finite node of the field, reach the nodes of the
# stencils they belong to and no others, whichever way the gradient is scattered.
@pytest.mark.parametrize("I", [4, 6, 8])
@pytest.mark.parametrize("what", ["lambda", "field"])
def test_nonfinite_field_gradient_stays_in_its_stencils(monkeypatch, I, what):
    N, n = 32, 4099
    u, pos = velocity(N, 4).float(), points(n)
    lam = torch.cos(pos)
    if what == "lambda":
        lam[1, 17], lam[0, 1234] = math.nan, math.inf
    else:
        u[2, 3, 4, 5], u[0, 20, 21, 22] = math.nan, math.inf
    got = {}
    for name, kind, scratch in (("gathers", trk.TRK_STEP_DIRECT, None), ("slabs", trk.TRK_STEP_BLOCK, None),
                                ("atomics", trk.TRK_STEP_BLOCK, "0")):
        monkeypatch.delenv("TRK_ADJ_SCRATCH_BYTES", raising=False)
        if scratch is not None:
            monkeypatch.setenv("TRK_ADJ_SCRATCH_BYTES", scratch)
        t = trk.Tracker(N, I=I, m=I // 2 - 1, storage=F32)
        t.set_field(u)
        t.set_step_kernel(kind)
        gf = torch.zeros((3, N, N, N), dtype=torch.float64, device="cuda")
        t.adjoint(pos, lam, 5e-3, 1, 1, grad_field=gf)
        torch.cuda.synchronize()
        got[name] = gf
        t.close()
    ref = got.pop("gathers")
    bad = ~torch.isfinite(ref)
    assert 0 < bad.sum().item() < 0.2 * bad.numel()
    top = ref[~bad].abs().max().item()
    for gf in got.values():
        assert torch.equal(~torch.isfinite(gf), bad)
        assert (gf - ref)[~bad].abs().max().item() <= 1e-6 * top   # float32 sums within a block


# Tuning lines that an earlier library wrote, whose numbers meant other launch shapes,
# are not taken over: the workload is timed again.
def test_tunings_of_earlier_kernels_are_not_used(tmp_path, monkeypatch):
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("TRK_TUNE_CACHE", str(cache))
    N, n = 64, 40000

    def source():
        t = trk.Tracker(N, storage=F32)
        t.set_field(velocity(N, 8))
        t.advance(points(n), 4e-3, 20)
        s = t.tuning()["source"]
        t.close()
        return s

    assert source() == trk.TRK_TUNE_TIMED and source() == trk.TRK_TUNE_CACHED
    key = cache.read_text().split("|")[0]
    old = key[:key.index(" order=") + len(" order=2")]   # the fields the earlier keys had
    cache.write_text(old + f"|{trk.TRK_STEP_BLOCK} 8 8 0 256\n")
    assert source() == trk.TRK_TUNE_TIMED


# The launch shape an untimed call reports is one that can be fixed: the one by size.
@pytest.mark.parametrize("n", [5000, 40000])
def test_reported_launch_shape_is_the_one_by_size(n):
    t = trk.Tracker(64, storage=F32)
    t.set_field(velocity(64, 8))
    t.advance(points(n), 4e-3, 2)
    info = t.tuning()
    assert info.pop("source") == trk.TRK_TUNE_DEFAULT and info["direct_particles"] == 256
    t.set_tuning(**info)
    t.advance(points(n), 4e-3, 2)
    assert t.tuning() == dict(info, source=trk.TRK_TUNE_FIXED)
    t.close()


# Steps replayed from a graph bin in the block shape of now, not of the capture.
def test_step_graph_after_the_block_shape_changed():
    N, n, steps = 64, 40000, 8
    u, pos = velocity(N, 9), points(n)

    def run(t, edge):
        trk.tracker_set_block(t.h, edge, edge, edge)
        p = pos.clone()
        t.advance(p, 4e-3, steps)
        t.sync()
        return p

    t, want = trk.Tracker(N, storage=F32), None
    t.set_field(u)
    t.set_step_kernel(trk.TRK_STEP_DIRECT)
    for edge in (4, 16, 4, 8, 2):
        fresh = trk.Tracker(N, storage=F32)
        fresh.set_field(u)
        fresh.set_step_kernel(trk.TRK_STEP_DIRECT)
        want = run(fresh, edge)
        fresh.close()
        assert torch.equal(run(t, edge), want), edge
    t.close()


# Positions and history in overlapping memory: a step starts from both as they were, and
# the history is written last, in small sets (which step in place) as in large ones.
def test_history_that_overlaps_the_positions():
    n = 3000
    rng = np.random.default_rng(3)
    bits = (np.int64(0x3FF00000) + rng.integers(0, 1 << 20, 3 * n)) << 32 | 0x3DCCCCCD   # 1 <= x < 2, low word 0.1f
    buf = torch.from_numpy(bits.view(np.float64)).cuda()
    pos, rhs = buf.view(3, n), buf.view(torch.float32)[1001:1001 + 3 * n].view(3, n)
    t = trk.Tracker(32, I=4, m=1, storage=F32)
    t.set_field(velocity(32, 2))
    p, r = pos.clone(), rhs.clone()
    t.advance(p, 4e-3, 2, trk.TRK_AB2, rhs=r, history_valid=1)
    t.advance(pos, 4e-3, 2, trk.TRK_AB2, rhs=rhs, history_valid=1)
    t.sync()
    want = p.clone().reshape(-1)
    want.view(torch.float32)[1001:1001 + 3 * n] = r.reshape(-1)
    assert torch.equal(buf.view(torch.int64), want.view(torch.int64))
    t.close()


@pytest.mark.parametrize("shift", [-64, 0, 1000])
def test_adjoint_into_memory_that_overlaps_lambda(shift):
    n = 5000
    pos = points(n)
    buf = torch.cos(torch.arange(3 * n + 2000, dtype=torch.float64, device="cuda"))
    lam, grad = buf[1000:1000 + 3 * n].view(3, n), buf[1000 + shift:1000 + shift + 3 * n].view(3, n)
    t = trk.Tracker(32, I=6, m=2, storage=F32)
    t.set_field(velocity(32, 2))
    want = trk.tracker_adjoint(t.h, pos, lam.clone(), 4e-3, 3, 2)[0].clone()
    trk.tracker_adjoint(t.h, pos, lam, 4e-3, 3, 2, grad_pos0=grad)
    t.sync()
    assert torch.equal(grad, want)
    t.close()


# A step captured by the caller, on a tracker whose buffers a larger set has sized, allocates
# nothing whatever the density.
def test_captured_step_after_a_larger_set():
    N = 256
    t = trk.Tracker(N, I=8, m=3, storage=F32)
    t.set_field(synth.velocity_field_torch(N, 20, 5))
    big, pos = points(1100000), points(500000)       # bins of 8^3 and, outside a capture, 4^3 cells
    t.advance(big, 1e-3, 1)
    p = pos.clone()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        t.advance(p, 1e-3, 1)
    p.copy_(pos)
    g.replay()
    torch.cuda.synchronize()
    want = pos.clone()
    t.advance(want, 1e-3, 1)
    t.sync()
    assert torch.equal(p, want)
    t.close()


@pytest.mark.parametrize("value", ["", "none", "12x"])
def test_wait_limit_that_is_no_number(monkeypatch, value):
    monkeypatch.setenv("TRK_WAIT_LIMIT", value)
    t = trk.Tracker(32, storage=F32)
    t.set_field(velocity(32, 2))
    p = points(40000)
    t.advance(p, 4e-3, 2)
    t.sync()
    t.close()
