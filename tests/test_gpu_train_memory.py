"""Training steps around allocations that fail: the object keeps its optimiser state, no step runs on buffers that are
gone, and the next step allocates them again."""
import numpy as np
import pytest

from paper_2504_21627_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CFG = I.Config(V=16, H=18, L=8, F=2, log2_T=10, N_min=4, N_max=24, n_hidden=2, width=64, n_mat=2)
MESH = I.noise_torus_tris(4, 600, n_mat=2)


def _batch(n):
    import torch
    rays = torch.from_numpy(I.rays_sphere_to_box(n, 2.0, MESH.verts.min(0), MESH.verts.max(0), 5)).cuda()
    g = torch.Generator("cuda").manual_seed(1)
    r = lambda *s: torch.rand(s, device="cuda", generator=g)  # noqa: E731
    return rays, {"occ": (r(n) < 0.7).float(), "t_local": r(n),
                  "normal": torch.nn.functional.normalize(r(n, 3) - 0.5, dim=1).contiguous(), "albedo": r(n, 3),
                  "mat": torch.randint(0, 2, (n,), device="cuda", generator=g, dtype=torch.int32)}


def _load(ctx):
    p = I.random_params(CFG, seed=3, table_range=0.5, bias_range=0.1)
    return ctx.load_object(MESH, CFG, tables=p.tables, mlp=p.packed_mlp())


def _step(ctx, obj, batch):
    """Loss and gradients of a step without update."""
    from paper_2504_21627_gb300 import lsnif
    st = ctx.train_step(*batch, obj, apply_update=False)
    ctx.check()
    return [np.array([st.total]), ctx.read_params(obj, lsnif.PARAM_GRAD_MLP), ctx.read_params(obj, lsnif.PARAM_GRAD_TABLES)]


def _same(a, b):
    # sums over the same rays in another order of the FP32 atomics: the bound of the batch sums in
    # test_gpu_train_shapes, 1e-4 of the largest
    for x, y in zip(a, b):
        assert np.abs(x - y).max() <= 1e-4 * np.abs(y).max()


def test_a_failed_allocation_leaves_a_usable_object():
    from paper_2504_21627_gb300 import lsnif
    small, large = _batch(300), _batch(3000)
    with lsnif.Context(0) as ctx:
        obj = _load(ctx)
        want = _step(ctx, obj, small)
        first = ctx.device_bytes()
        want_large = _step(ctx, obj, large)
        grown = ctx.device_bytes()
    failures = 0
    for k in range(64):
        with lsnif.Context(0) as ctx:
            obj = _load(ctx)
            # the first step fails at allocation k, or (all succeed) does not
            ctx.debug_fail_alloc_after(k)
            try:
                _step(ctx, obj, small)
                break
            except lsnif.LsnifError as e:
                assert e.code == -3
                failures += 1
            _same(_step(ctx, obj, small), want)
            assert ctx.device_bytes() == first
            # a growth that fails, then a step of the size that fitted before
            ctx.train_step(*small, obj, lr=1e-3)
            moments = ctx.train_step(*small, obj, lr=1e-12).step
            mlp = ctx.read_params(obj, lsnif.PARAM_MLP)
            ctx.debug_fail_alloc_after(min(k, 17))
            with pytest.raises(lsnif.LsnifError) as e:
                ctx.train_step(*large, obj, lr=1e-3)
            assert e.value.code == -3
            np.testing.assert_array_equal(ctx.read_params(obj, lsnif.PARAM_MLP), mlp)
            assert ctx.train_step(*small, obj, lr=1e-12).step == moments + 1
            ctx.check()
            # and the growth once there is memory again
            ctx.train_step(*large, obj, lr=1e-12)
            ctx.check()
            assert ctx.device_bytes() == grown
    assert failures > 20
    assert want_large[0] > 0
