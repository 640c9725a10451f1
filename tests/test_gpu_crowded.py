"""Encode, decode and largest momentum of stores with much of their mass in few
cells: the values of the oracle, and no slower than a crowd has to be."""
import numpy as np
import pytest

from oracle import pm

from gpu_util import assert_store_equal, oracle_params, read_store

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def cube():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from conftest import build_lib
    build_lib()
    import paper_1712_06121_gb300 as c
    torch.cuda.set_device(0)
    return c


def _us(fn, calls=5):
    """Median device time of a call."""
    fn()
    t = []
    for _ in range(calls):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        torch.cuda.synchronize()
        t.append(1e3 * a.elapsed_time(b))
    return sorted(t)[calls // 2]


def _crowd(n, nf, seed, crowds):
    """n particles anywhere but the first few thousands: `crowds` (particles,
    corner, side in fine cells)."""
    rng = np.random.default_rng(seed)
    pos = rng.random((3, n)) * nf
    at = 0
    for m, corner, side in crowds:
        pos[:, at:at + m] = corner + side * rng.random((3, m))
        at += m
    pos = pos.astype(np.float32)
    pos[pos >= nf] = 0.0
    vel = rng.normal(0.0, 0.3, (3, n)).astype(np.float32) + np.float32(0.2) * np.sin(pos[::-1])
    return np.ascontiguousarray(pos[:, rng.permutation(n)]), vel.astype(np.float32), np.arange(n, dtype=np.uint32)


# groups of 64 cells on either side of 16384 particles, the most that one CTA
# takes, cut into runs at the multiples of 8192: one crowded cell, crowds of
# several cells and groups, all particles in one cell; every code width and
# brick; scales given and measured.  Whole numbers, exact.
@pytest.mark.parametrize("n,nf,ratio,brick,xb,vb,sigma,crowds", [
    (16384, 48, 4, 4, 1, 1, 0.0, [(16384, 5.0, 0.9)]),
    (16385, 48, 4, 4, 2, 2, 0.0, [(16385, 5.0, 0.9)]),
    (60001, 48, 4, 1, 1, 2, 0.0, [(24577, 9.0, 0.9), (17000, 30.0, 3.0)]),
    (120011, 64, 4, 2, 2, 1, 0.5, [(50000, 16.5, 7.0), (40000, 33.0, 14.0)]),
    (200003, 32, 8, 1, 1, 1, 0.0, []),
])
def test_encode_of_crowded_groups_is_bit_exact(cube, n, nf, ratio, brick, xb, vb, sigma, crowds):
    pos, vel, ids = _crowd(n, nf, 1712214, crowds)
    prm = cube.make_params(nf, n, ratio=ratio, brick=brick, x_bytes=xb, v_bytes=vb, box=50.0, omega_m=0.3, omega_l=0.7)
    ctx = cube.cube_create(prm, torch.cuda.current_stream())
    try:
        for _ in range(2):                                    # the second time over the first one's scratch
            cube.cube_encode(ctx, pos, vel, ids, 0.02, sigma)
            g = read_store(cube, ctx)
            ref = pm.encode(oracle_params(pm, prm, brick), pos, vel, ids, 0.02, g["sigma"], snap=False)
            assert_store_equal(g, ref, f"encode of {n}")
            if sigma == 0.0:
                free = pm.encode(oracle_params(pm, prm, brick), pos, vel, ids, 0.02, 0.0)
                assert g["sigma"] == pytest.approx(free.sigma, rel=1e-12)
            cube.cube_pm_step(ctx, 0.02, 0.0200001)           # (the step's crowded-brick words, the batch's lists)
            assert cube.cube_stats_get(ctx).error_flags == 0
    finally:
        cube.cube_destroy(ctx)


# a fifth of 128^3 particles in one cell: the encode that added momenta up by
# 64-bit global atomics took 1.9 times as long as for particles anywhere, one
# CTA for the crowd 17 times
def test_encode_does_not_wait_for_a_crowd(cube):
    n, nf = 128 ** 3, 256
    prm = cube.make_params(nf, n, box=50.0)
    ctx = cube.cube_create(prm, torch.cuda.current_stream())
    try:
        t = []
        for crowds in ([], [(n // 5, 41.0, 0.9)]):
            x, v, i = (torch.from_numpy(a.view(np.int32) if a.dtype == np.uint32 else a).cuda()
                       for a in _crowd(n, nf, 1712215, crowds))
            t.append(_us(lambda: cube.cube_encode(ctx, x, v, i, 0.02, 0.0)))
        assert t[1] < 6 * t[0], t
    finally:
        cube.cube_destroy(ctx)


# cells on either side of the 2048 particles that a warp finishes alone, several
# of them in one CTA's share, the largest momentum anywhere in a crowd; every
# code width, alone and in a batch.  The decoded values' own maximum, exactly.
@pytest.mark.parametrize("vb", [1, 2])
@pytest.mark.parametrize("crowds", [[(2048, 5.0, 0.9)], [(2049, 5.0, 0.9)],
                                    [(30000, 4.1, 3.8), (2500, 8.1, 3.8), (2040, 20.1, 3.8), (9000, 40.1, 7.8)]])
def test_largest_momentum_of_crowded_cells(cube, vb, crowds):
    n, nf = 60000, 48
    prm = cube.make_params(nf, n, v_bytes=vb, box=50.0)
    batch = cube.cube_batch_create([prm] * 2, torch.cuda.current_stream())
    ctx = cube.cube_create(prm, torch.cuda.current_stream())
    try:
        pos, vel, ids = _crowd(n, nf, 1712216, crowds)
        crowd = np.flatnonzero((np.abs(pos - 5.5) < 2.0).all(axis=0))
        members = [ctx, cube.cube_batch_member(batch, 0), cube.cube_batch_member(batch, 1)]
        for k, c in enumerate(members):
            v = vel.copy()
            v[k, crowd[(k + 1) * len(crowd) // 4]] = (3.0, -2.5, 2.75)[k]
            cube.cube_encode(c, pos, v, ids, 0.02, 0.5)
            out = [np.empty((3, n), np.float32) for _ in range(2)]
            cube.cube_decode(c, *out)
            assert cube.cube_max_speed(c) == np.abs(out[1]).max()
    finally:
        cube.cube_destroy(ctx)
        cube.cube_batch_destroy(batch)


# a fifth of 128^3 particles in one cell, against particles anywhere: 16 times
# with a CTA a brick, 47 times with a warp for the crowd
def test_largest_momentum_does_not_wait_for_a_warp(cube):
    n, nf = 128 ** 3, 256
    prm = cube.make_params(nf, n, box=50.0)
    ctx = cube.cube_create(prm, torch.cuda.current_stream())
    try:
        t = []
        for crowds in ([], [(n // 5, 41.0, 0.9)]):
            cube.cube_encode(ctx, *_crowd(n, nf, 1712215, crowds), 0.02, 0.0)
            t.append(_us(lambda: cube.cube_max_speed(ctx)))
        assert t[1] < 24 * t[0], t
    finally:
        cube.cube_destroy(ctx)


# decode of bricks of one, 8 and 64 cells, 64 cells a CTA: a last CTA of 24
# cells, crowds within and across its shares, every code width
@pytest.mark.parametrize("nf,ratio,brick,xb,vb", [(24, 4, 1, 1, 1), (24, 4, 1, 2, 2), (48, 4, 2, 1, 2), (64, 2, 2, 2, 1),
                                                  (48, 4, 4, 2, 2), (32, 8, 1, 1, 1)])
def test_decode_of_any_brick_matches_oracle(cube, nf, ratio, brick, xb, vb):
    n = 30011
    pos, vel, ids = _crowd(n, nf, 1712217, [(12000, 5.0, 0.9), (5000, 8.0, 9.0)])
    prm = cube.make_params(nf, n, ratio=ratio, brick=brick, x_bytes=xb, v_bytes=vb, box=50.0, omega_m=0.3, omega_l=0.7)
    ctx = cube.cube_create(prm, torch.cuda.current_stream())
    try:
        cube.cube_encode(ctx, pos, vel, ids, 0.02, 0.5)
        g = read_store(cube, ctx)
        ref = pm.encode(oracle_params(pm, prm, brick), pos, vel, ids, 0.02, g["sigma"], snap=False)
        out = [np.empty((3, n), np.float32) for _ in range(2)] + [np.empty(n, np.uint32)]
        cube.cube_decode(ctx, *out)
        rp, rv = pm.decode(ref)[:2]
        assert np.array_equal(out[0], rp.astype(np.float32))
        assert np.array_equal(out[2], ref.ids)
        # v_c and the FP32 table entry are each rounded once, and their sum
        assert np.all(np.abs(out[1] - rv) <= 2.0 ** -23 * (np.abs(ref.vc).max() + np.abs(rv)))
    finally:
        cube.cube_destroy(ctx)


# a fifth of 128^3 particles in one cell: bricks of one cell take as long as
# bricks of 64 (one warp for the crowd took 7 times as long)
def test_decode_of_a_crowd_does_not_depend_on_the_brick(cube):
    n, nf = 128 ** 3, 256
    t = []
    for brick in (4, 2, 1):
        prm = cube.make_params(nf, n, brick=brick, box=50.0)
        ctx = cube.cube_create(prm, torch.cuda.current_stream())
        try:
            cube.cube_encode(ctx, *_crowd(n, nf, 1712215, [(n // 5, 41.0, 0.9)]), 0.02, 0.0)
            p, v = torch.empty((3, n), device="cuda"), torch.empty((3, n), device="cuda")
            t.append(_us(lambda: cube.cube_decode(ctx, p, v, None)))
        finally:
            cube.cube_destroy(ctx)
    assert max(t) < 2.5 * t[0], t
