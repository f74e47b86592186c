"""Graph replay after an object of the batch has been replaced: the replay returns what a direct call returns,
whatever the shape of the object that took the slot."""
import numpy as np
import pytest

from paper_2504_21627_gb300 import inputs as I

pytestmark = pytest.mark.gpu

N = 3000


def _load(ctx, L, F, W, seed):
    cfg = I.Config(V=16, H=18, L=L, F=F, log2_T=9, N_min=4, N_max=48, n_hidden=2, width=W, n_mat=2)
    p = I.random_params(cfg, seed=seed, table_range=0.5, bias_range=0.1)
    return ctx.load_object(I.noise_torus_tris(4, 600, n_mat=2), cfg, tables=p.tables, mlp=p.packed_mlp())


# the second object replaces the first: another F, more levels (a longer chunk than the captured shared memory),
# and shapes whose FP32 query takes the stage kernels
# -- and, with others = 1, beside an object that stays
@pytest.mark.parametrize("precision,first,second,others", [
    ("fp32", (16, 2, 64), (8, 4, 64), 0), ("bf16", (16, 2, 64), (8, 4, 64), 0), ("fp16", (16, 2, 64), (8, 4, 64), 0),
    ("fp8", (16, 2, 64), (8, 4, 64), 0), ("bf16", (4, 2, 64), (8, 2, 128), 0), ("fp32", (16, 2, 64), (32, 2, 64), 0),
    ("fp32", (16, 2, 64), (16, 2, 128), 0), ("fp32", (16, 2, 64), (16, 1, 64), 0), ("fp32", (8, 2, 64), (8, 2, 96), 0),
    ("fp32", (16, 2, 64), (32, 2, 64), 1), ("fp32", (16, 2, 64), (8, 4, 64), 1),
])
def test_replay_after_a_replaced_object(precision, first, second, others):
    import torch
    from paper_2504_21627_gb300 import lsnif
    prec = {"fp32": lsnif.FP32_PLAIN, "bf16": lsnif.BF16_FUSED, "fp16": lsnif.FP16_FUSED, "fp8": lsnif.FP8_FUSED}[precision]
    mesh = I.noise_torus_tris(4, 600, n_mat=2)
    rays = torch.from_numpy(I.rays_sphere_to_box(N, 3.0, mesh.verts.min(0), mesh.verts.max(0), 5)).cuda()
    side = torch.cuda.Stream()
    with lsnif.Context(0) as ctx:
        a = _load(ctx, *first, seed=3)
        rest = [_load(ctx, *first, seed=9) for _ in range(others)]
        who = torch.empty(N, dtype=torch.int32, device="cuda")
        out = ctx._alloc_hits(N, 0, False)

        def handles(h):
            who.fill_(h)
            for r in rest:
                who[::3] = r

        def query():  # the same buffers each time
            with torch.cuda.stream(side):
                ctx.query_rays(rays, obj_per_ray=who, precision=prec, out=out, stream=side)
            side.synchronize()
            ctx.check()
            return [x.cpu().numpy().copy() for x in (out.hit, out.t, out.mat, out.normal, out.albedo)]

        handles(a)
        torch.cuda.synchronize()
        ctx.set_graph_mode(True)
        before = [query() for _ in range(2)]
        for x, y in zip(*before):
            np.testing.assert_array_equal(x, y)
        ctx.unload_object(a)
        b = _load(ctx, *second, seed=4)
        assert (a & 0xFFFF) == (b & 0xFFFF), "the new object takes the slot"
        handles(b)
        torch.cuda.synchronize()
        replay = [query() for _ in range(2)]
        ctx.set_graph_mode(False)
        direct = query()
        for got in replay:
            for x, y in zip(got, direct):
                np.testing.assert_array_equal(x, y)
        assert not np.array_equal(before[0][1], direct[1]), "the objects differ"
        assert np.isfinite(direct[1]).any()
