"""The persistent-lane traversal (trace modes 1 and 2) where one warp starts rays of objects with different grids:
every output bit equal to the voxel-by-voxel traversal (mode 0). The entry spreads lie within an eighth of some of the
grids and not of others, so that the lanes of one warp answer the question of neighbouring rays differently."""
import numpy as np
import pytest

from paper_2504_21627_gb300 import inputs as I

pytestmark = pytest.mark.gpu

GRIDS = (64, 128, 16, 256)


def _parallel_rays(n, lo, hi, axis, side, spread, seed):
    """Rays that enter through one face of the box, `spread` of its extent wide about a corner of the face."""
    g = I.rng(seed)
    lo, hi = np.asarray(lo, np.float64), np.asarray(hi, np.float64)
    ext = hi - lo
    o = lo + ext * spread * g.random((n, 3))
    o[:, axis] = lo[axis] - 0.1 * ext[axis] if side > 0 else hi[axis] + 0.1 * ext[axis]
    d = 0.6 * ext * g.random((n, 3))
    d[:, axis] = side * ext[axis]
    return I.pack_rays(o, d)


@pytest.fixture(scope="module")
def scene():
    from paper_2504_21627_gb300 import lsnif
    mesh = I.noise_torus_tris(4, 2000, n_mat=2)
    with lsnif.Context(0) as ctx:
        ids = []
        for i, V in enumerate(GRIDS):
            cfg = I.Config(V=V, H=18, L=4, F=2, log2_T=8, N_min=4, N_max=32, n_hidden=1, width=64, n_mat=2)
            p = I.random_params(cfg, seed=3 + i, table_range=0.5, bias_range=0.1)
            ids.append(ctx.load_object(mesh, cfg, tables=p.tables, mlp=p.packed_mlp()))
        info = ctx.object_info(ids[0])
        yield ctx, ids, np.array(info.bmin[:]), np.array(info.bmax[:])


# in voxels of the 128 grid; 12 is near there and not in the grid of 64
@pytest.mark.parametrize("voxels", [3, 12, 24, 100])
@pytest.mark.parametrize("axis,side", [(0, 1), (1, -1), (2, 1)])
def test_modes_agree_over_mixed_grids(scene, voxels, axis, side):
    import torch
    from paper_2504_21627_gb300 import lsnif
    ctx, ids, lo, hi = scene
    handles = torch.tensor(ids, dtype=torch.int32, device="cuda")
    for n in (2, 3, 31, 33, 4099):
        rays = torch.from_numpy(_parallel_rays(n, lo, hi, axis, side, voxels / 128, seed=n)).cuda()
        who = handles[torch.from_numpy(I.rng(n + 1).integers(0, len(ids), n)).cuda()].contiguous()
        got = []
        for mode in (0, 1, 2):
            ctx.set_trace_mode(mode)
            r = ctx.query_rays(rays, obj_per_ray=who, precision=lsnif.FP32_PLAIN)
            got.append([x.cpu().numpy().copy() for x in (r.hit, r.t, r.mat, r.normal, r.albedo)])
        ctx.check()
        for other in got[1:]:
            for a, b in zip(got[0], other):
                np.testing.assert_array_equal(a, b)
        if n > 1000 and voxels > 12:
            assert np.isfinite(got[0][1]).any()
