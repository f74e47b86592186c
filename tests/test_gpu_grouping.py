"""Requests over at most 32 objects are grouped by one launch, over more by two: a ray's outputs are the same bits
either way, at the edges of blocks and of the rule."""
import numpy as np
import pytest

from paper_2504_21627_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# rays of one object, of a few, of the most that one launch takes
@pytest.mark.parametrize("objects", [1, 5, 32])
@pytest.mark.parametrize("mode", [0, 1])
def test_one_launch_groups_as_two_do(objects, mode):
    import torch
    from paper_2504_21627_gb300 import lsnif
    cfg = I.Config(V=16, H=8, L=8, F=2, log2_T=8, N_min=4, N_max=32, n_hidden=2, width=64, n_mat=2)
    mesh = I.icosphere(2)
    n = 330000
    rays = torch.from_numpy(I.rays_sphere_to_box(n, 3.0, mesh.verts.min(0), mesh.verts.max(0), 5)).cuda()
    with lsnif.Context(0) as ctx:
        ctx.set_group_mode(mode)
        ids = []

        def load(count):
            while len(ids) < count:
                p = I.random_params(cfg, seed=len(ids), table_range=0.5, bias_range=0.1)
                ids.append(ctx.load_object(mesh, cfg, tables=p.tables, mlp=p.packed_mlp()))

        load(objects)
        handles = torch.tensor(ids, device="cuda", dtype=torch.int32)[torch.arange(n, device="cuda") ** 2 % objects]

        def query(lo, hi):
            to = {"obj": ids[0]} if objects == 1 else {"obj_per_ray": handles[lo:hi].contiguous()}
            out = ctx.query_rays(rays[:, lo:hi].contiguous(), precision=lsnif.BF16_FUSED, **to)
            ctx.check()
            return [x.cpu().numpy().copy() for x in (out.hit, out.t, out.mat)]

        spans = ((0, 1), (7, 1030), (0, 1024), (5, 1030), (1000, 9193), (0, n))
        once = [query(*s) for s in spans]
        assert np.isfinite(once[-1][1]).mean() > 0.3
        load(33)
        for s, a in zip(spans, once):
            for x, y in zip(a, query(*s)):
                np.testing.assert_array_equal(x, y)
