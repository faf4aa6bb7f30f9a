"""Volume preprocessing at the edges of its kernels' tiles, against the oracle bit for bit: x
lines around the 248-voxel chunk of the statistics and majorant pass and long enough that fewer
than 64 lines are staged at a time, row counts around a staged group, grids of one brick and of
ragged bricks, every pyramid level."""
import numpy as np
import pytest

from paper_1709_05418_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(3, 5, 247), (2, 9, 248), (9, 3, 249), (4, 17, 497), (1, 65, 300), (13, 5, 8),
                                   (70, 1, 1), (2, 2, 1100)])
def test_stats_bricks_and_levels_equal_the_oracle(shape):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import oracle
    from paper_1709_05418_gb300 import api
    rng = np.random.default_rng(sum(shape))
    dens = (rng.random(shape) * 40.0 * (rng.random(shape) < 0.6)).astype(np.float32)
    dens.flat[0] = 3.0
    ctx = api.Context()
    v = ctx.load_volume(torch.from_numpy(dens).cuda())
    ctx.build_mips(v)
    gi = ctx.get_volume_info(v)
    o = oracle.Volume(dens)
    oi = o.stats()
    for key in ("mean", "majorant", "nonzero", "levels", "mip_of_level"):
        assert gi[key] == oi[key], key
    assert np.array_equal(ctx.copy_brick_majorants(v).cpu().numpy(), o.brick_majorants())
    for lv in range(gi["levels"]):
        g, r = ctx.copy_mip_level(v, lv).cpu().numpy(), o.mip_level(lv, f32=True)
        assert np.array_equal(g.view(np.uint32), r.view(np.uint32)), lv
    o.close()
    ctx.close()


@pytest.mark.parametrize("shape", [(124, 124, 97), (80, 124, 97), (76, 129, 287), (51, 100, 288), (76, 128, 640), (76, 128, 681),
                                   (70, 139, 95), (16, 19, 1100), (17, 19, 2500)])
def test_levels_built_together_equal_the_oracle(shape):
    """Enough lines for the streaming x pass (5,016 up to 680 voxels, 15,200 below 144, any from 1,088) and just outside its range: the
    levels a descriptor reads are built together, so its values are the oracle's bit for bit."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import oracle
    from paper_1709_05418_gb300 import api
    rng = np.random.default_rng(sum(shape))
    dens = (rng.random(shape) * 40.0 * (rng.random(shape) < 0.6)).astype(np.float32)
    ctx = api.Context()
    v = ctx.load_volume(torch.from_numpy(dens).cuda())
    ctx.build_mips(v)
    x, d = W.random_queries(shape, 700, seed=3)
    x, d, wl = x.astype(np.float32), d.astype(np.float32), np.array([0.48, -0.6, 0.64], np.float32)
    got = ctx.extract_descriptors(v, *(torch.from_numpy(a).cuda() for a in (x, d, wl))).cpu().numpy()
    ctx.close()
    o = oracle.Volume(dens)
    ref = o.descriptor(x, d, wl, f32=True)
    o.close()
    assert np.array_equal(got[:, :, :225].view(np.uint32), ref[:, :, :225].view(np.uint32))


@pytest.mark.parametrize("shape", [(300, 270, 8), (290, 290, 9), (283, 290, 24), (298, 280, 25), (281, 290, 56), (290, 281, 57),
                                   (280, 281, 120), (281, 290, 121), (1200, 130, 1), (40, 129, 9)])
def test_bricks_of_short_lines_equal_the_oracle(shape):
    """Lines at the edges of the widths that 16 to 256 threads read, more rows of bricks than a wave (and
    fewer), rows that do not fill a block."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import oracle
    from paper_1709_05418_gb300 import api
    rng = np.random.default_rng(sum(shape))
    dens = (rng.random(shape) * 40.0 * (rng.random(shape) < 0.3)).astype(np.float32)
    dens.flat[-1] = 41.0
    ctx = api.Context()
    v = ctx.load_volume(torch.from_numpy(dens).cuda())
    ctx.build_mips(v)
    gi = ctx.get_volume_info(v)
    o = oracle.Volume(dens)
    oi = o.stats()
    for key in ("mean", "majorant", "nonzero"):
        assert gi[key] == oi[key], key
    assert np.array_equal(ctx.copy_brick_majorants(v).cpu().numpy(), o.brick_majorants())
    o.close()
    ctx.close()
