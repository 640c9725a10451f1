"""Kernels at the sizes where their work split changes: edges of tiles,
remainders and the smallest and largest of their ranges, against the oracle."""
import numpy as np
import pytest

from oracle import pm

from gpu_util import oracle_params, read_store

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
