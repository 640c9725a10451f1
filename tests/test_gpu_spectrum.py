"""The power spectrum's binning beyond 300 shells, from several threads and
against sums of known modes."""
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
