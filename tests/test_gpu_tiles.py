"""The BF16 and FP16 fused kernels work on tiles of 128 rays in one, two or
four parts, by the number of live rays: each ray's outputs are the same bits
whatever the part it falls in, its row, and the rays beside it."""
import numpy as np
import pytest

from paper_2504_21627_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# L F a multiple of 16 (shared points read from the previous chunk's tile),
# 8 modulo 16 (gathered twice), F = 4 with width 128, 20 outputs
SHAPES = [(8, 2, 64, 3, 2, 0), (4, 2, 64, 2, 2, 1), (4, 4, 128, 2, 4, 0), (16, 2, 64, 4, 12, 0)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("precision", ["bf16", "fp16"])
def test_parts_of_tiles_give_the_same_bits(shape, precision):
    import torch
    from paper_2504_21627_gb300 import lsnif
    L, F, W, nh, n_mat, act = shape
    cfg = I.Config(V=32, H=18, L=L, F=F, log2_T=10, N_min=4, N_max=64, n_hidden=nh, width=W, n_mat=n_mat,
                   activation=act)
    mesh = I.noise_torus_tris(4, 2000, n_mat=1)
    p = I.random_params(cfg, seed=3, table_range=0.5, bias_range=0.1)
    prec = {"bf16": lsnif.BF16_FUSED, "fp16": lsnif.FP16_FUSED}[precision]
    rays = torch.from_numpy(I.rays_sphere_to_box(120000, 3.0, mesh.verts.min(0), mesh.verts.max(0), 5)).cuda()
    with lsnif.Context(0) as ctx:
        obj = ctx.load_object(mesh, cfg, tables=p.tables, mlp=p.packed_mlp())

        def query(r):
            out = ctx.query_rays(r.contiguous(), obj=obj, precision=prec, logits=True)
            ctx.check()
            return [x.cpu().numpy().copy() for x in (out.hit, out.t, out.mat, out.logits)]

        whole = query(rays)          # whole tiles
        assert np.isfinite(whole[1]).mean() > 0.5
        # about 1, 32, 33 rows; either side of one round of 32- and 64-row parts
        for n in (1, 40, 41, 127, 129, 6100, 6500, 12000, 13000, 24500, 26000):
            part = query(rays[:, 1000:1000 + n])
            for a, b in zip(whole, part):
                np.testing.assert_array_equal(a[1000:1000 + n], b)


@pytest.mark.parametrize("precision", ["bf16", "fp16"])
def test_parts_of_many_objects_tiles(precision):
    """Parts of tiles never straddle objects, and an object's weights are in place for its tiles."""
    import torch
    from paper_2504_21627_gb300 import lsnif
    cfg = I.Config(V=16, H=8, L=8, F=2, log2_T=8, N_min=4, N_max=32, n_hidden=2, width=64, n_mat=2)
    mesh = I.icosphere(2)
    prec = {"bf16": lsnif.BF16_FUSED, "fp16": lsnif.FP16_FUSED}[precision]
    n, k = 3000, 7
    rays = torch.from_numpy(I.rays_sphere_to_box(n, 3.0, mesh.verts.min(0), mesh.verts.max(0), 5)).cuda()
    with lsnif.Context(0) as ctx:
        objs = []
        for i in range(k):
            p = I.random_params(cfg, seed=i, table_range=0.5, bias_range=0.1)
            objs.append(ctx.load_object(mesh, cfg, tables=p.tables, mlp=p.packed_mlp()))
        who = torch.arange(n, device="cuda") ** 2 % k   # uneven shares
        handles = torch.tensor(objs, dtype=torch.int32, device="cuda")[who].contiguous()
        t = ctx.query_rays(rays, obj_per_ray=handles, precision=prec).t.cpu().numpy()
        ctx.check()
        for i, o in enumerate(objs):
            alone = ctx.query_rays(rays, obj=o, precision=prec).t.cpu().numpy()
            m = who.cpu().numpy() == i
            np.testing.assert_array_equal(t[m], alone[m])
