"""Networks at the line between the resident and the streamed FP16 kernel, which round a feature differently (F = 2:
interpolated in FP16 and in FP32): those just past it are streamed, and refused in BF16, which is never streamed."""
import numpy as np
import pytest

from paper_2504_21627_gb300 import inputs as I

pytestmark = pytest.mark.gpu

MESH = I.noise_torus_tris(4, 600, n_mat=2)


def _load(ctx, L, F, W, n_hidden, H=18, seed=3):
    cfg = I.Config(V=16, H=H, L=L, F=F, log2_T=9, N_min=4, N_max=48, n_hidden=n_hidden, width=W, n_mat=4)
    p = I.random_params(cfg, seed=seed, table_range=0.5, bias_range=0.1)
    return ctx.load_object(MESH, cfg, tables=p.tables, mlp=p.packed_mlp())


# within 1.7 KB past the line, by their hidden layers and by their segments
@pytest.mark.parametrize("shape", [(16, 2, 128, 2, 18), (4, 2, 128, 3, 48), (16, 2, 64, 2, 40)])
def test_a_network_past_the_line_is_streamed(shape):
    """Beside an object far past the line the whole batch is streamed: an object's results are the same bits alone."""
    import torch
    from paper_2504_21627_gb300 import lsnif
    L, F, W, n_hidden, H = shape
    n = 3000
    rays = torch.from_numpy(I.rays_sphere_to_box(n, 3.0, MESH.verts.min(0), MESH.verts.max(0), 5)).cuda()
    with lsnif.Context(0) as ctx:
        obj = _load(ctx, *shape)
        who = torch.full((n,), obj, dtype=torch.int32, device="cuda")

        def query(**kw):
            out = ctx.query_rays(rays, precision=lsnif.FP16_FUSED, **kw)
            ctx.check()
            return [x.cpu().numpy().copy() for x in (out.hit, out.t, out.mat, out.normal, out.albedo)]

        alone = query(obj=obj)
        big = _load(ctx, 16, F, W, 8 if W == 64 else 6, H=max(H, 30), seed=4)
        who[1::2] = big
        beside = query(obj_per_ray=who)
        assert np.isfinite(alone[1]).any()
        for a, b in zip(alone, beside):
            np.testing.assert_array_equal(a[..., ::2], b[..., ::2])


@pytest.mark.parametrize("shape", [(12, 2, 128, 2, 18), (16, 2, 64, 8, 16), (8, 4, 128, 2, 10)])
def test_a_network_past_the_line_is_refused_in_bf16(shape):
    import torch
    from paper_2504_21627_gb300 import lsnif
    rays = torch.from_numpy(I.rays_sphere_to_box(100, 3.0, MESH.verts.min(0), MESH.verts.max(0), 5)).cuda()
    with lsnif.Context(0) as ctx:
        obj = _load(ctx, *shape)
        for query in (lambda: ctx.query_rays(rays, obj=obj, precision=lsnif.BF16_FUSED),
                      lambda: ctx.query_rays_noalloc(rays, ctx._alloc_hits(100, 0, False), obj=obj)):
            with pytest.raises(lsnif.LsnifError) as e:
                query()
            assert e.value.code == -10
