"""Steps of stores of so many bricks that the histograms' tile sums are
scanned on their own, against the oracle."""
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


# tiles of 16 bricks of 4^3 cells and of 128 bricks of one: 6912 tiles, each of
# which adds up the sums before its own, and more than 8192, whose sums are
# scanned.  The scan's launches show which way was taken; whole numbers, exact.
@pytest.mark.parametrize("nf,ratio,brick,tiles", [(192, 1, 4, 6912), (256, 1, 4, 16384), (768, 4, 1, 55296)])
def test_steps_of_many_tiles_are_bit_exact(cube, nf, ratio, brick, tiles):
    n = 60001
    assert (nf // ratio // brick) ** 3 == tiles * {4: 16, 1: 128}[brick]
    rng = np.random.default_rng(1712213)
    pos = (rng.random((3, n)) * nf).astype(np.float32)
    pos[:, :2000] = 9.0 + 0.5 * rng.random((3, 2000))
    pos[pos >= nf] = 0.0
    a = [0.5, 0.50005, 0.5001]                                # momenta cross 0.15 coarse cells (rms) in a step
    vel = (0.15 * ratio / (0.00005 / 0.5 ** 1.5) * rng.standard_normal((3, n))).astype(np.float32)
    ids = np.arange(n, dtype=np.uint32)
    prm = cube.make_params(nf, n, ratio=ratio, brick=brick, x_bytes=1, v_bytes=1, box=50.0)
    ctx = cube.cube_create(prm, torch.cuda.current_stream())
    try:
        cube.cube_encode(ctx, pos, vel, ids, a[0], 0.0)
        cube.cube_keep_drifted(ctx, True)
        for i in range(2):
            before = read_store(cube, ctx)
            launched = cube.cube_stats_get(ctx).kernel_launches
            cube.cube_pm_step(ctx, a[i], a[i + 1])
            cell, u, p = np.empty((3, n), np.int32), np.empty((3, n), np.float32), np.empty((3, n), np.float32)
            sig = cube.cube_debug_drifted(ctx, cell, u, p)
            g = read_store(cube, ctx)
            ref = pm.encode_drifted(oracle_params(pm, prm, brick), cell, u, p, before["ids"], sig, g["a"], g["a_p"])
            assert_store_equal(g, ref, f"step {i}")
            stats = cube.cube_stats_get(ctx)
            # (the second call of cube_stats_get counts the first one's own kernel)
            assert stats.kernel_launches - launched == 11 + (2 if tiles > 8192 else 0)
            assert stats.error_flags == 0
    finally:
        cube.cube_destroy(ctx)
