"""GPU: the kernels' edges.  Every step and interpolation kernel performs the
same floating-point operations in the same order per particle, whatever the
lanes per particle (6, 8, 16 or 32), the launch shape, the grouping and where
the stencil comes from (global memory, halos, slabs), so results are compared
bit for bit; binning is compared with the oracle's."""
import math

import numpy as np
import pytest
import torch

import oracle
import paper_2107_01104_gb300 as trk
import synth

pytestmark = pytest.mark.gpu
L = 2 * math.pi
F64, F32, BF16 = trk.TRK_F64, trk.TRK_F32, trk.TRK_BF16X2


def tracker(N, I, m, storage, seed=5, scale=1.0):
    t = trk.Tracker(N, family=trk.TRK_SPLINE, I=I, m=m, storage=storage)
    t.set_field(torch.from_numpy(scale * synth.velocity_field_np(N, min(10, N // 3), seed)).cuda())
    return t


def points(n, seed=0, lo=-L, hi=2 * L):
    return torch.from_numpy(np.random.default_rng(seed).uniform(lo, hi, (3, n))).cuda()


def sync(t, cfl=False):
    try:
        t.sync()
    except trk.TrackerError as e:
        assert cfl and e.status == trk.TRK_ECFL


def steps_of(t, pos, scheme, steps=3, hist=0, dt=4e-3):
    p = pos.clone()
    rhs = 0.1 * torch.cos(pos.float()).repeat(max(scheme, 1), 1, 1)   # [order - 1][3][n]
    if scheme == trk.TRK_RK2:
        t.advance(p, dt, steps)
        return [p]
    t.advance(p, dt, steps, scheme, rhs=rhs, history_valid=hist)
    return [p, rhs]


# Sets below 32768 particles step and interpolate in the caller's order; the
# same particles in a set one larger are grouped first.
@pytest.mark.parametrize("storage,I,m", [(F64, 4, 1), (F64, 6, 2), (F32, 4, 1), (F32, 6, 2), (F32, 8, 3), (BF16, 8, 3)])
@pytest.mark.parametrize("scheme,hist", [(trk.TRK_RK2, 0), (trk.TRK_AB2, 1), (trk.TRK_AB4, 2)])
def test_small_sets_in_the_callers_order_match_grouped(storage, I, m, scheme, hist):
    n = 32768
    t = tracker(64, I, m, storage)
    t.set_step_kernel(trk.TRK_STEP_DIRECT)
    pos = points(n)
    big, small = steps_of(t, pos, scheme, hist=hist), steps_of(t, pos[:, :n - 1].contiguous(), scheme, hist=hist)
    for a, b in zip(big, small):
        assert torch.equal(a[..., :n - 1], b)
    out = torch.float64 if storage == F64 else torch.float32
    for deriv in (False, True):
        a = t.interpolate(pos, out_dtype=out, deriv=deriv)
        assert torch.equal(a[..., :n - 1], t.interpolate(pos[:, :n - 1].contiguous(), out_dtype=out, deriv=deriv))
    t.sync()


def test_small_set_interpolated_over_its_own_positions():
    """Values written over the positions: the positions are read before (float64) or
    the set is grouped first."""
    t = tracker(32, 4, 1, F64)
    pos = points(3001)
    ref = t.interpolate(pos, out_dtype=torch.float64).clone()
    buf = pos.clone()
    trk.tracker_interpolate(t.h, buf, 3, out=buf)
    t.sync()
    assert torch.equal(buf, ref)


# direct gathers: sizes around a CTA's and a wave's, each launch shape, against
# the block kernel (float32: the slab pipeline)
@pytest.mark.parametrize("storage,I,m", [(F64, 6, 2), (F64, 8, 3), (F32, 4, 1), (F32, 6, 2), (F32, 6, 3), (F32, 8, 3), (BF16, 6, 2)])
@pytest.mark.parametrize("scheme", [trk.TRK_RK2, trk.TRK_AB2])
def test_direct_launch_shapes_match_block(storage, I, m, scheme):
    t = tracker(64, I, m, storage)
    for n in (32768, 38911, 38913, 160001):
        pos = points(n, seed=n)
        t.set_step_kernel(trk.TRK_STEP_BLOCK)
        ref = steps_of(t, pos, scheme, steps=2, hist=int(scheme != trk.TRK_RK2))
        for P in (64, 128, 256):
            t.set_tuning(step_kernel=trk.TRK_STEP_DIRECT, direct_block=16, direct_particles=P)
            for a, b in zip(ref, steps_of(t, pos, scheme, steps=2, hist=int(scheme != trk.TRK_RK2))):
                assert torch.equal(a, b), (n, P)
    t.sync()


# the slab pipeline: empty blocks, rounds that span blocks far apart, remainders,
# the smallest grid, X* beyond the halo (scale 40)
@pytest.mark.parametrize("I,m", [(4, 1), (6, 2), (8, 3)])
@pytest.mark.parametrize("N,n,layout", [(16, 1, "any"), (16, 5, "any"), (32, 63, "corners"), (64, 65, "corners"),
                                        (64, 609, "any"), (64, 2433, "corners"), (128, 40007, "any")])
@pytest.mark.parametrize("scale", [1.0, 40.0])
def test_slab_pipeline_matches_direct(I, m, N, n, layout, scale):
    t = tracker(N, I, m, F32, scale=scale)
    pos = points(n, seed=N + n)
    if layout == "corners":   # two opposite corners of the box: every group of four may span both
        pos = points(n, seed=n, lo=-8 * L / N, hi=8 * L / N)
    got = {}
    others = [trk.TRK_STEP_BLOCK] + ([trk.TRK_STEP_COLUMN] if I < 8 else [])
    for kind in [trk.TRK_STEP_DIRECT] + others:
        t.set_step_kernel(kind)
        got[kind] = steps_of(t, pos, trk.TRK_RK2, steps=2) + steps_of(t, pos, trk.TRK_AB3, steps=2, hist=1)
        if kind != trk.TRK_STEP_COLUMN:
            got[kind] += [t.interpolate(pos), t.interpolate(pos, deriv=True)]
        sync(t, cfl=scale > 1)
    for kind in others:
        for a, b in zip(got[trk.TRK_STEP_DIRECT], got[kind]):
            assert torch.equal(a, b), kind


@pytest.mark.parametrize("segment", [1, 2, 8])
def test_column_order_segments_match(segment):
    t = tracker(64, 6, 2, F32)
    pos = points(20011)
    t.set_step_kernel(trk.TRK_STEP_DIRECT)
    ref = steps_of(t, pos, trk.TRK_RK2)
    t.set_tuning(step_kernel=trk.TRK_STEP_COLUMN, column_segment=segment)
    assert torch.equal(ref[0], steps_of(t, pos, trk.TRK_RK2)[0])
    t.sync()


# batched sets: in the caller's order (32767), grouped gathers (40000 for I = 4 at
# 64^3: below 1/4 per cell), slabs (70001), against the same set on its own
@pytest.mark.parametrize("storage", [F32, BF16])
def test_batched_routes_match_single_sets(storage):
    N, dt, steps = 64, 4e-3, 3
    specs = [(n, I, deriv) for n in (1, 130, 32767, 40000, 70001) for I in (4, 6, 8) for deriv in (0, 1)]
    t = tracker(N, 6, 2, storage)
    sets = []
    for k, (n, I, deriv) in enumerate(specs):
        pos = points(n, seed=k)
        sets.append(dict(pos=pos, rhs=0.1 * torch.cos(pos.float()), I=I, m=I // 2 - 1, family=trk.TRK_SPLINE,
                         out=torch.zeros((9 if deriv else 3, n), device="cuda"), deriv=deriv))
    start = [dict(s, pos=s["pos"].clone(), rhs=s["rhs"].clone()) for s in sets]
    t.advance_batched(sets, dt, steps, history_valid=True)
    t.sync()
    for I in (4, 6, 8):
        one = tracker(N, I, I // 2 - 1, storage)
        one.set_step_kernel(trk.TRK_STEP_DIRECT)
        for s, b in zip(start, sets):
            if s["I"] != I or s["deriv"]:
                continue
            one.advance(s["pos"], dt, steps, trk.TRK_AB2, rhs=s["rhs"], history_valid=1)
            assert torch.equal(s["pos"], b["pos"]) and torch.equal(s["rhs"], b["rhs"]), (I, s["pos"].shape)
        # with gradients the sums have their own order: float32 values of u in two orders
        # differ by up to about 100 x 2^-24 (|u| <= 4, about 20 roundings each), positions by
        # at most 2 dt times that per step
        for s, b in zip(start, sets):
            if s["I"] != I or not s["deriv"]:
                continue
            one.advance(s["pos"], dt, steps - 1, trk.TRK_AB2, rhs=s["rhs"], history_valid=1)
            at = s["pos"].clone()
            one.advance(s["pos"], dt, 1, trk.TRK_AB2, rhs=s["rhs"], history_valid=1)
            assert (s["pos"] - b["pos"]).abs().max().item() <= steps * dt * 256 * 2.0 ** -24
            g = one.interpolate(at, deriv=True)
            assert (g - b["out"]).abs().max().item() <= 2e-5 * g.abs().max().item()
        one.sync()
        one.close()


def test_batched_sets_that_share_arrays():
    """Each set starts from the arrays as they were; the last one's results stay."""
    t = tracker(32, 6, 2, F32)
    pos, rhs = points(3000), torch.zeros((3, 3000), device="cuda")
    alone = [dict(pos=pos.clone(), rhs=rhs.clone(), I=I, m=I // 2 - 1, family=trk.TRK_SPLINE, deriv=0,
                  out=torch.zeros((3, 3000), device="cuda")) for I in (4, 8)]
    shared = [dict(s, pos=pos, rhs=rhs, out=torch.zeros((3, 3000), device="cuda")) for s in alone]
    t.advance_batched(alone, 4e-3, 2, history_valid=False)
    t.advance_batched(shared, 4e-3, 2, history_valid=False)
    t.sync()
    assert torch.equal(pos, alone[1]["pos"]) and torch.equal(rhs, alone[1]["rhs"])
    for a, b in zip(alone, shared):
        assert torch.equal(a["out"], b["out"])


# stable binning: tiles of 4096 keys, warps' runs of 512, one digit only
@pytest.mark.parametrize("n", [1, 31, 511, 513, 4095, 4096, 4097, 12289])
@pytest.mark.parametrize("width", [1.0, 1.0 / 64])
def test_binning_tiles(n, width):
    N = 128
    pos = np.random.default_rng(n).uniform(0, L * width, (3, n))
    t = trk.Tracker(N, family=trk.TRK_LAGRANGE, I=4, storage=F32)
    keys, perm, offsets = t.bin(torch.from_numpy(pos).cuda())
    t.sync()
    for got, want in zip((keys, perm, offsets), oracle.bin_particles(pos, N, (8, 8, 8))):
        np.testing.assert_array_equal(got.cpu().numpy(), want)


# the adjoint of float32 fields: odd counts, more than 128 particles in a block,
# X* cells away (scale 40), through slabs and through gathers.  The position
# gradient is the same arithmetic; the field gradient is summed in two orders
# (float32 sums within a block: 1e-6 relative, the adjoint's bar)
@pytest.mark.parametrize("I,m", [(4, 1), (6, 2), (8, 3)])
@pytest.mark.parametrize("N,n,width", [(16, 1, 1.0), (32, 129, 0.25), (32, 1001, 0.25), (32, 4099, 1.0)])
@pytest.mark.parametrize("scale", [1.0, 40.0])
def test_adjoint_paths_agree(I, m, N, n, width, scale):
    out = []
    pos = points(n, seed=n, lo=0.01, hi=0.01 + (L - 0.02) * width)
    for kind in (trk.TRK_STEP_DIRECT, trk.TRK_STEP_BLOCK):
        t = tracker(N, I, m, F32, scale=scale)
        t.set_step_kernel(kind)
        gf = torch.zeros((3, N, N, N), dtype=torch.float64, device="cuda")
        gpos, _ = t.adjoint(pos, torch.cos(pos), 5e-3, 3, 2, grad_field=gf)
        sync(t, cfl=scale > 1)
        out.append((gpos.clone(), gf))
        t.close()
    assert torch.equal(out[0][0], out[1][0])
    assert (out[0][1] - out[1][1]).norm().item() <= 1e-6 * out[1][1].norm().item()


# the sparse scatter: a CTA's round is 20 particles (I = 6) or 16, one round or two per CTA
# (at 256^3 one below 50000 particles), X* in another cell for all, some and none of them;
# against the dense form (float32 sums within a block: 1e-6 relative, the adjoint's bar)
@pytest.mark.parametrize("I,m", [(4, 1), (6, 2), (8, 3)])
@pytest.mark.parametrize("N,n", [(256, 1), (256, 21), (256, 643), (64, 41), (64, 5001)])
@pytest.mark.parametrize("dt", [1e-6, 5e-3, 0.2])
def test_sparse_field_gradient_rounds(I, m, N, n, dt):
    pos, gf = points(n, seed=n), []
    u = 0.2 * synth.velocity_field_torch(N, 10, 5)
    for kind in (trk.TRK_STEP_DIRECT, trk.TRK_STEP_BLOCK):
        t = trk.Tracker(N, I=I, m=m, storage=F32)
        t.set_field(u)
        t.set_step_kernel(kind)
        gf.append(torch.zeros((3, N, N, N), dtype=torch.float64, device="cuda"))
        t.adjoint(pos, torch.cos(pos), dt, 1, 1, grad_field=gf[-1])
        sync(t, cfl=dt > 0.1)
        t.close()
    assert (gf[0] - gf[1]).abs().max().item() <= 1e-6 * gf[1].abs().max().item()


# untimed calls bin by 4^3 or 8^3 cells (256^3: 4^3 from 0.02 to 0.06 per cell for I = 6 and 8):
# the same steps, and AB history, on either side of the rule and with the edge fixed
@pytest.mark.parametrize("storage,I,m", [(F32, 6, 2), (BF16, 8, 3)])
def test_untimed_binning_edge(storage, I, m):
    N = 256
    t = trk.Tracker(N, I=I, m=m, storage=storage)
    t.set_field(synth.velocity_field_torch(N, 20, 5))
    for n, edge in ((335544, 8), (335545, 4), (400001, 4)):
        t.set_tuning()
        pos = points(n)
        got = steps_of(t, pos, trk.TRK_AB2, steps=5, hist=1)
        assert t.tuning()["direct_block"] == edge and t.tuning()["source"] == trk.TRK_TUNE_DEFAULT
        t.set_tuning(step_kernel=trk.TRK_STEP_DIRECT, direct_block=12 - edge)
        for a, b in zip(got, steps_of(t, pos, trk.TRK_AB2, steps=5, hist=1)):
            assert torch.equal(a, b)
    sync(t, cfl=True)
    t.close()
