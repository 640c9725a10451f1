"""The power spectrum's binning beyond 300 shells, from several threads and
against sums of known modes."""
import math
import threading

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


def _particles(n, nf, seed):
    rng = np.random.default_rng(seed)
    pos = (rng.random((3, n)) * nf).astype(np.float32)
    pos[pos >= nf] = 0.0
    return pos, rng.normal(0.0, 0.3, (3, n)).astype(np.float32), np.arange(n, dtype=np.uint32)


def _spectrum(cube, ctx, n_bins):
    out = [np.empty(n_bins) for _ in range(3)]
    cube.cube_power_spectrum(ctx, n_bins, *out)
    return out


# 336 shells, more than 48 KB of the kernel's bins; empty bins beyond the
# corner.  Counts are exact, |k| 1e-12, P carries the FP32 transform (1e-4).
def test_bins_beyond_the_default_shared_memory(cube):
    nf, n, n_bins = 384, 7001, 2048
    pos, vel, ids = _particles(n, nf, 1712211)
    prm = cube.make_params(nf, n, x_bytes=2, v_bytes=1, box=50.0, omega_m=0.3, omega_l=0.7)
    ctx = cube.cube_create(prm, torch.cuda.current_stream())
    try:
        cube.cube_encode(ctx, pos, vel, ids, 0.02, 0.5)
        g = read_store(cube, ctx)
        ref = pm.encode(oracle_params(pm, prm, g["brick"]), pos, vel, ids, 0.02, g["sigma"], snap=False)
        k, p, m = _spectrum(cube, ctx, n_bins)
        rk, rp, rm = pm.power_spectrum(ref, n_bins)
        assert np.array_equal(m, rm)
        full = rm > 0
        assert np.all(np.isnan(k[~full])) and np.all(np.isnan(p[~full]))
        assert np.allclose(k[full], rk[full], rtol=1e-12, atol=0.0)
        assert np.allclose(p[full], rp[full], rtol=1e-4, atol=0.0)
    finally:
        cube.cube_destroy(ctx)


# independent contexts of eight threads, whose launches need different amounts
# of shared memory (300 and 336 shells) and start together each time: every
# call succeeds and gives what it gives alone
def test_spectra_from_several_threads(cube):
    nf, n, calls = 384, 5000, 200
    ctxs, alone, failed = [], [], []
    together = threading.Barrier(8)
    try:
        prm = cube.make_params(nf, n, box=50.0)
        for i in range(8):
            ctxs.append((cube.cube_create(prm, torch.cuda.Stream()), 300 if i % 2 else 336))
            cube.cube_encode(ctxs[-1][0], *_particles(n, nf, 1712212 + i), 0.02, 0.5)
            alone.append(_spectrum(cube, *ctxs[-1]))

        def work(i):
            try:
                torch.cuda.set_device(0)
                for _ in range(calls):
                    together.wait()
                    got = _spectrum(cube, *ctxs[i])
                    assert all(np.array_equal(a, b, equal_nan=True) for a, b in zip(got, alone[i]))
            except threading.BrokenBarrierError:
                pass                                         # another thread has failed and says so
            except BaseException as e:                       # noqa: B902 (reported by the main thread)
                failed.append(repr(e))
                together.abort()

        threads = [threading.Thread(target=work, args=(i,)) for i in range(8)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not failed, failed
    finally:
        for c, _ in ctxs:
            cube.cube_destroy(c)


# All particles on the node at the origin: every mode is that node's density,
# so the shells' sums are known to more bits than FP64 keeps.  Roundings on the
# way, of 2^-53 each and all sums of positive terms: one where a block's sums
# become FP64, ceil(blocks / 32) + 5 additions over the blocks, four in the
# final factors and quotient (blocks: of eight rows (|ky|, |kz|), 456 at most);
# the window weights are the host's, from the same expression.
@pytest.mark.parametrize("nf,n_bins", [(16, 13), (48, 24), (192, 150)])
def test_binning_keeps_every_bit_of_fp64(cube, nf, n_bins):
    n, box = 100003, 50.0
    prm = cube.make_params(nf, n, x_bytes=4, v_bytes=4, id_bytes=0, box=box)
    ctx = cube.cube_create(prm, torch.cuda.current_stream())
    try:
        cube.cube_encode(ctx, np.zeros((3, n), np.float32), np.zeros((3, n), np.float32), None, 0.02, 0.5)
        rho = np.empty((nf, nf, nf), np.float32)
        cube.cube_density(ctx, rho)
        assert np.count_nonzero(rho) == 1 and rho[0, 0, 0] > 0
        k, p, m = _spectrum(cube, ctx, n_bins)
    finally:
        cube.cube_destroy(ctx)
    real = np.longdouble
    h = nf // 2
    sinc = [1.0] + [math.sin(math.pi * i / nf) / (math.pi * i / nf) for i in range(1, h + 1)]
    w = np.array([math.pow(s, -4.0) for s in sinc]).astype(real)
    mult = np.where((np.arange(h + 1) == 0) | (np.arange(h + 1) == h), 1, 2)
    i2 = np.arange(h + 1, dtype=np.int64) ** 2
    n2 = (i2[:, None, None] + i2[:, None] + i2).ravel()
    count = (mult[:, None, None] * mult[:, None] * mult).ravel()
    root = np.sqrt(n2.astype(real))
    weight = (w[:, None, None] * w[:, None] * w).ravel()
    shell = np.floor(root.astype(np.float64) + 0.5).astype(np.int64)
    blocks = min(456, ((h + 1) ** 2 + 7) // 8)
    tol = (1 + -(-blocks // 32) + 5 + 4) * 2.0 ** -53
    for i in range(1, n_bins + 1):
        at = shell == i
        modes = int(count[at].sum())
        assert m[i - 1] == modes
        want_k = 2 * real(math.pi) / real(box) * (count[at] * root[at]).sum() / modes
        want_p = real(box) ** 3 / real(nf) ** 6 * real(rho[0, 0, 0]) ** 2 * (count[at] * weight[at]).sum() / modes
        assert abs(real(k[i - 1]) / want_k - 1) <= tol, (i, k[i - 1], want_k)
        assert abs(real(p[i - 1]) / want_p - 1) <= tol, (i, p[i - 1], want_p)
