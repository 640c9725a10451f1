"""Kernels at the sizes where their work split changes: edges of tiles,
remainders and the smallest and largest of their ranges, against the oracle."""
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


def _random_particles(n, nf, seed):
    rng = np.random.default_rng(seed)
    pos = (rng.random((3, n)) * nf).astype(np.float32)
    pos[pos >= nf] = 0.0
    return pos, rng.normal(0.0, 0.3, (3, n)).astype(np.float32), np.arange(n, dtype=np.uint32)


# ---------------------------------------------------------------- power spectrum
# rows of 9 to 129 kx (one lane to several rounds of 32, a last round of one
# lane), one bin, bins beyond the mesh's corner (empty: NaN).  Mode counts are
# exact; |k| sums in pairs of floats (2^-46 per addition, fewer than 2^10
# additions in a chain) stay within 1e-12; P carries the FP32 transform (1e-4).
@pytest.mark.parametrize("nf,n_bins", [(16, 2048), (24, 21), (48, 1), (64, 60), (96, 84), (256, 128)])
def test_power_spectrum_bins_at_the_edges(cube, nf, n_bins):
    n = 5001
    pos, vel, ids = _random_particles(n, nf, 1712201)
    prm = cube.make_params(nf, n, x_bytes=2, v_bytes=1, box=50.0, omega_m=0.3, omega_l=0.7)
    ctx = cube.cube_create(prm, torch.cuda.current_stream())
    try:
        cube.cube_encode(ctx, pos, vel, ids, 0.02, 0.5)
        g = read_store(cube, ctx)
        ref = pm.encode(oracle_params(pm, prm, g["brick"]), pos, vel, ids, 0.02, g["sigma"], snap=False)
        k, p, m = (np.empty(n_bins) for _ in range(3))
        cube.cube_power_spectrum(ctx, n_bins, k, p, m)
        rk, rp, rm = pm.power_spectrum(ref, n_bins)
        assert np.array_equal(m, rm)
        full = rm > 0
        assert np.all(np.isnan(k[~full])) and np.all(np.isnan(p[~full]))
        assert np.allclose(k[full], rk[full], rtol=1e-12, atol=0.0)
        assert np.allclose(p[full], rp[full], rtol=1e-4, atol=0.0)
    finally:
        cube.cube_destroy(ctx)


# ---------------------------------------------------------------- decode and largest momentum
def _blob(n, nf, seed):
    """n particles, half of them in one coarse cell, the rest anywhere."""
    pos, vel, ids = _random_particles(n, nf, seed)
    pos[:, : n // 2] = 5.0 + 0.9 * (pos[:, : n // 2] / nf)
    return pos, vel, ids


# one particle, a round's edges and a crowded brick, every code width, bricks
# of 4 to 16 fine cells, 2-byte positions at 256 coarse cells per side (25-bit
# q: rounded); the decoded values are the oracle's rounded once
@pytest.mark.parametrize("n,nf,ratio,xb,vb", [(1, 16, 4, 1, 1), (33, 16, 4, 2, 2), (257, 32, 8, 1, 2), (4099, 32, 2, 2, 1),
                                              (3001, 48, 1, 1, 1), (9000, 256, 1, 2, 2)])
def test_decode_and_max_speed_match_oracle(cube, n, nf, ratio, xb, vb):
    pos, vel, ids = _blob(n, nf, 1712202)
    prm = cube.make_params(nf, n, ratio=ratio, x_bytes=xb, v_bytes=vb, box=50.0, omega_m=0.3, omega_l=0.7)
    ctx = cube.cube_create(prm, torch.cuda.current_stream())
    try:
        cube.cube_encode(ctx, pos, vel, ids, 0.02, 0.5)
        g = read_store(cube, ctx)
        ref = pm.encode(oracle_params(pm, prm, g["brick"]), pos, vel, ids, 0.02, g["sigma"], snap=False)
        dp, dv = torch.zeros((3, n), device="cuda"), torch.zeros((3, n), device="cuda")
        di = torch.zeros(n, device="cuda", dtype=torch.int32)
        cube.cube_decode(ctx, dp, dv, di)
        rp, rv = pm.decode(ref)[:2]
        assert np.array_equal(dp.cpu().numpy(), rp.astype(np.float32))
        assert np.array_equal(di.cpu().numpy().astype(np.uint32), ref.ids)
        v = dv.cpu().numpy()
        # v_c and the FP32 table entry are each rounded once, and their sum
        assert np.all(np.abs(v - rv) <= 2.0 ** -23 * (np.abs(ref.vc).max() + np.abs(rv)))
        assert cube.cube_max_speed(ctx) == np.abs(v).max()
    finally:
        cube.cube_destroy(ctx)


# packed meshes into 16-byte aligned and unaligned device memory and into host memory
@pytest.mark.parametrize("nf", [16, 24, 96])
def test_packed_meshes_do_not_depend_on_alignment(cube, nf):
    n = 3000
    pos, vel, ids = _random_particles(n, nf, 1712203)
    prm = cube.make_params(nf, n, x_bytes=1, v_bytes=1, box=50.0, omega_m=0.3, omega_l=0.7)
    ctx = cube.cube_create(prm, torch.cuda.current_stream())
    try:
        cube.cube_encode(ctx, pos, vel, ids, 0.02, 0.5)
        for call in (cube.cube_density, cube.cube_potential):
            host = np.empty((nf, nf, nf), dtype=np.float32)
            call(ctx, host)
            for shift in (0, 1, 2):
                buf = torch.full((nf ** 3 + 8,), -1.0, device="cuda")
                call(ctx, buf[shift:shift + nf ** 3])
                got = buf.cpu().numpy()
                assert np.array_equal(got[shift:shift + nf ** 3].reshape(nf, nf, nf), host)
                assert np.all(got[:shift] == -1.0) and np.all(got[shift + nf ** 3:] == -1.0)
    finally:
        cube.cube_destroy(ctx)


# ---------------------------------------------------------------- pass B's split
# epochs so close that the clump's force moves nothing, and momenta that cross
# 0.7 fine cells (rms) in a step
_EPOCHS = [0.5, 0.50005, 0.5001]
_SPEED = 0.7 / (0.00005 / (0.5 ** 3 * 0.5 ** -1.5))


def _mixed_particles(n, nf, seed, speed=_SPEED):
    """Uniform random particles with 3000 of them in one brick."""
    rng = np.random.default_rng(seed)
    pos = rng.uniform(0.0, nf, (3, n))
    pos[:, :3000] = 9.0 + 1.5 * rng.standard_normal((3, 3000))
    vel = speed * rng.standard_normal((3, n))
    return np.mod(pos, nf).astype(np.float32) % np.float32(nf), vel.astype(np.float32), np.arange(n, dtype=np.uint32)


# more than 16 bricks per SM, 1-byte velocities: a warp per brick, crowded
# bricks by whole CTAs, empty bricks, bricks of one cell; whole numbers, exact
@pytest.mark.parametrize("nf,ratio,brick,n,xb,idb", [(256, 4, 4, 40000, 1, 4), (128, 4, 2, 33000, 2, 1),
                                                     (64, 4, 1, 20001, 1, 2)])
def test_resort_of_many_bricks_is_bit_exact(cube, nf, ratio, brick, n, xb, idb):
    bricks = (nf // ratio // brick) ** 3
    assert bricks > 16 * torch.cuda.get_device_properties(0).multi_processor_count
    pos, vel, ids = _mixed_particles(n, nf, 1712204)
    prm = cube.make_params(nf, n, ratio=ratio, x_bytes=xb, v_bytes=1, id_bytes=idb, brick=brick, box=50.0)
    ctx = cube.cube_create(prm, torch.cuda.current_stream())
    try:
        a = _EPOCHS
        cube.cube_encode(ctx, pos, vel, ids, a[0], 0.0)
        cube.cube_keep_drifted(ctx, True)
        for i in range(2):
            before = read_store(cube, ctx)
            cube.cube_pm_step(ctx, a[i], a[i + 1])
            cell, u, p = np.empty((3, n), np.int32), np.empty((3, n), np.float32), np.empty((3, n), np.float32)
            sig = cube.cube_debug_drifted(ctx, cell, u, p)
            g = read_store(cube, ctx)
            ref = pm.encode_drifted(oracle_params(pm, prm, g["brick"]), cell, u, p, before["ids"], sig, g["a"],
                                    g["a_p"])
            assert_store_equal(g, ref, f"step {i}")
    finally:
        cube.cube_destroy(ctx)


# a batch whose members' bricks together pass the split gives each member's own run
@pytest.mark.parametrize("vb", [1, 2])
def test_batch_past_the_split_equals_members_alone(cube, vb):
    nf, n, members = 128, 30000, 5
    prm = cube.make_params(nf, n, v_bytes=vb, box=50.0)
    batch = cube.cube_batch_create([prm] * members, torch.cuda.current_stream())
    one = cube.cube_create(prm, torch.cuda.current_stream())
    try:
        sets = [_mixed_particles(n, nf, 1712205 + i) for i in range(members)]
        ctxs = [cube.cube_batch_member(batch, i) for i in range(members)]
        for c, s in zip(ctxs, sets):
            cube.cube_encode(c, *s, _EPOCHS[0], 0.0)
        for a0, a1 in zip(_EPOCHS, _EPOCHS[1:]):
            cube.cube_batch_step(batch, [a0] * members, [a1] * members)
        for c, s in zip(ctxs, sets):
            cube.cube_encode(one, *s, _EPOCHS[0], 0.0)
            for a0, a1 in zip(_EPOCHS, _EPOCHS[1:]):
                cube.cube_pm_step(one, a0, a1)
            x, y = read_store(cube, c), read_store(cube, one)
            for k in ("counts", "offsets", "vc", "chi", "nu", "ids", "sigma"):
                assert np.array_equal(x[k], y[k]), k
            assert cube.cube_stats_get(c).max_migration == 1
    finally:
        cube.cube_destroy(one)
        cube.cube_batch_destroy(batch)


# ---------------------------------------------------------------- encode
# the sort's tiles (4096 items, 512 a warp) and their remainders, one to three
# passes of 8 bits, scales given and measured, particles outside the box;
# whole numbers, exact
@pytest.mark.parametrize("n,nf,ratio,xb,vb,sigma", [(1, 16, 4, 1, 1, 0.5), (511, 16, 4, 2, 2, 0.0), (4096, 64, 4, 1, 2, 0.0),
                                                    (4097, 64, 4, 2, 1, 0.3), (12801, 96, 1, 1, 1, 0.0),
                                                    (40001, 256, 2, 1, 2, 0.0)])
def test_encode_at_tile_edges(cube, n, nf, ratio, xb, vb, sigma):
    pos, vel, ids = _blob(n, nf, 1712207)
    rng = np.random.default_rng(n)
    pos = pos[:, rng.permutation(n)] + np.float32(nf) * rng.integers(-2, 3, (3, n)).astype(np.float32)
    prm = cube.make_params(nf, n, ratio=ratio, x_bytes=xb, v_bytes=vb, box=50.0, omega_m=0.3, omega_l=0.7)
    ctx = cube.cube_create(prm, torch.cuda.current_stream())
    try:
        for host in (True, False):
            put = (lambda a: a) if host else (lambda a: torch.from_numpy(a.copy()).cuda())
            cube.cube_encode(ctx, put(pos), put(vel), put(ids.view(np.int32)), 0.02, sigma)
            g = read_store(cube, ctx)
            ref = pm.encode(oracle_params(pm, prm, g["brick"]), pos, vel, ids, 0.02, g["sigma"], snap=False)
            assert_store_equal(g, ref, f"encode {n} host {host}")
            if sigma == 0.0:
                free = pm.encode(oracle_params(pm, prm, g["brick"]), pos, vel, ids, 0.02, 0.0)
                assert g["sigma"] == pytest.approx(free.sigma, rel=1e-12)
    finally:
        cube.cube_destroy(ctx)


# ---------------------------------------------------------------- checkpoint sections
# section lengths with every remainder of 16 bytes, buffers the copy kernel
# takes (aligned, on the device) and those it does not: the same bytes, and the
# same store from each of them
@pytest.mark.parametrize("n,xb,vb,idb", [(1, 1, 1, 1), (1003, 2, 1, 2), (777, 1, 2, 4), (513, 4, 4, 4), (100, 1, 1, 0)])
def test_checkpoint_buffers_hold_the_same_bytes(cube, n, xb, vb, idb):
    nf = 32
    pos, vel, ids = _random_particles(n, nf, 1712208)
    prm = cube.make_params(nf, n, x_bytes=xb, v_bytes=vb, id_bytes=idb, box=50.0)
    ctx = cube.cube_create(prm, torch.cuda.current_stream())
    try:
        cube.cube_encode(ctx, pos, vel, ids, 0.02, 0.5)
        size = cube.cube_checkpoint_size(prm)
        host = np.full(size, 7, dtype=np.uint8)
        cube.cube_checkpoint_save(ctx, host)
        bufs = [torch.full((size + 16,), 7, device="cuda", dtype=torch.uint8) for _ in range(2)]
        views = [bufs[0][:size], bufs[1][8:8 + size]]
        for v in views:
            cube.cube_checkpoint_save(ctx, v)
            assert np.array_equal(v.cpu().numpy(), host)
        assert bool((bufs[0][size:] == 7).all()) and bool((bufs[1][:8] == 7).all())
        out = [np.empty((3, n), np.float32) for _ in range(2)]
        cube.cube_decode(ctx, *out)
        for b in (host, *views):
            other = [np.empty((3, n), np.float32) for _ in range(2)]
            cube.cube_encode(ctx, pos[:, ::-1].copy(), vel, ids, 0.03, 0.7)
            cube.cube_checkpoint_load(ctx, b)
            cube.cube_decode(ctx, *other)
            assert all(np.array_equal(x, y) for x, y in zip(out, other))
            st = cube.cube_stats_get(ctx)
            assert st.error_flags == 0 and st.a == 0.02
    finally:
        cube.cube_destroy(ctx)


# 64 cells a CTA whatever the brick: bricks of one cell and of eight, a last
# CTA of 24 cells, 2-byte velocities past the re-sort's split with crowded
# bricks; whole numbers, exact
@pytest.mark.parametrize("nf,ratio,brick,n,xb,vb", [(24, 4, 1, 4001, 1, 1), (64, 4, 1, 20001, 2, 2), (128, 4, 2, 33000, 1, 2)])
def test_small_bricks_are_bit_exact(cube, nf, ratio, brick, n, xb, vb):
    pos, vel, ids = _mixed_particles(n, nf, 1712209)
    prm = cube.make_params(nf, n, ratio=ratio, x_bytes=xb, v_bytes=vb, brick=brick, box=50.0)
    ctx = cube.cube_create(prm, torch.cuda.current_stream())
    try:
        a = _EPOCHS
        cube.cube_encode(ctx, pos, vel, ids, a[0], 0.0)
        before = read_store(cube, ctx)
        assert_store_equal(before, pm.encode(oracle_params(pm, prm, brick), pos, vel, ids, a[0], before["sigma"],
                                             snap=False), "encode")
        cube.cube_keep_drifted(ctx, True)
        cube.cube_pm_step(ctx, a[0], a[1])
        cell, u, p = np.empty((3, n), np.int32), np.empty((3, n), np.float32), np.empty((3, n), np.float32)
        sig = cube.cube_debug_drifted(ctx, cell, u, p)
        g = read_store(cube, ctx)
        ref = pm.encode_drifted(oracle_params(pm, prm, brick), cell, u, p, before["ids"], sig, g["a"], g["a_p"])
        assert_store_equal(g, ref, "step")
    finally:
        cube.cube_destroy(ctx)
