"""The persistent-lane traversal (trace modes 1 and 2) against the
voxel-by-voxel one (mode 0): every output bit equal, on the rays its position
test, its ray queue and its two kinds of rounds can get wrong."""
import numpy as np
import pytest

from paper_2504_21627_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _rays(kind, n, lo, hi, V, seed):
    g = I.rng(seed)
    lo, hi = np.asarray(lo, np.float64), np.asarray(hi, np.float64)
    c, ext = 0.5 * (lo + hi), hi - lo
    if kind == "sphere":
        return I.rays_sphere_to_box(n, 3.0, lo, hi, seed)
    if kind == "far":       # origins so far away that no position is clear of the planes
        return I.rays_sphere_to_box(n, 3e4, lo, hi, seed)
    if kind == "camera":    # neighbouring rays: long rounds
        side = int(np.ceil(np.sqrt(n)))
        return np.ascontiguousarray(I.rays_pinhole(I.seeded_camera(seed, radius=2.5, width=side, height=side))[:, :n])
    if kind == "inside":
        o = lo + ext * g.random((n, 3))
        r = I.pack_rays(o, g.normal(size=(n, 3)))
        r[6] = g.choice([0.0, 0.05, -0.5], n)
        return r
    # along the axes and the diagonals, origins exactly on voxel planes
    d = g.integers(-1, 2, (n, 3)).astype(np.float64)
    o = lo + ext * g.integers(0, V + 1, (n, 3)) / V
    o = np.where(d != 0, o - 2.0 * d * ext, o)
    r = I.pack_rays(o, d)
    r[0, ::97] = np.nan
    del c
    return r


@pytest.mark.parametrize("V", [2, 16, 128])
@pytest.mark.parametrize("kind", ["sphere", "far", "camera", "inside", "planes"])
def test_modes_agree_bit_for_bit(V, kind):
    import torch
    from paper_2504_21627_gb300 import lsnif
    cfg = I.Config(V=V, H=18, L=4, F=2, log2_T=8, N_min=4, N_max=32, n_hidden=1, width=64, n_mat=2)
    mesh = I.noise_torus_tris(4, 2000, n_mat=2)
    p = I.random_params(cfg, seed=3, table_range=0.5, bias_range=0.1)
    with lsnif.Context(0) as ctx:
        obj = ctx.load_object(mesh, cfg, tables=p.tables, mlp=p.packed_mlp())
        info = ctx.object_info(obj)
        for n in (1, 31, 33, 5003):
            rays = torch.from_numpy(_rays(kind, n, info.bmin[:], info.bmax[:], V, seed=n + V)).cuda()
            got = []
            for mode in (0, 1, 2):
                ctx.set_trace_mode(mode)
                r = ctx.query_rays(rays, obj=obj, precision=lsnif.FP32_PLAIN, logits=True)
                got.append([x.cpu().numpy().copy() for x in (r.hit, r.t, r.mat, r.logits)])
            ctx.check()
            for other in got[1:]:
                for a, b in zip(got[0], other):
                    np.testing.assert_array_equal(a, b)
            if kind != "planes" and n > 1000:
                assert np.isfinite(got[0][1]).any()


def test_histogram_beyond_the_default_shared_memory():
    """300 object slots: the histogram and the ray queue together pass 48 KiB."""
    import torch
    from paper_2504_21627_gb300 import lsnif
    cfg = I.Config(V=2, H=4, L=2, F=2, log2_T=4, N_min=2, N_max=4, n_hidden=1, width=64, n_mat=1)
    mesh = I.cube()
    p = I.random_params(cfg, seed=3, table_range=0.5, bias_range=0.1)
    with lsnif.Context(0) as ctx:
        objs = [ctx.load_object(mesh, cfg, tables=p.tables, mlp=p.packed_mlp()) for _ in range(300)]
        rays = torch.from_numpy(I.rays_sphere_to_box(3000, 3.0, [0, 0, 0], [1, 1, 1], 5)).cuda()
        who = torch.tensor(objs, dtype=torch.int32, device="cuda")[torch.arange(3000, device="cuda") % 300].contiguous()
        got = []
        for mode in (0, 1):
            ctx.set_trace_mode(mode)
            r = ctx.query_rays(rays, obj_per_ray=who, precision=lsnif.FP32_PLAIN)
            got.append([x.cpu().numpy().copy() for x in (r.hit, r.t)])
        ctx.check()
        for a, b in zip(*got):
            np.testing.assert_array_equal(a, b)
        assert np.isfinite(got[0][1]).mean() > 0.5
