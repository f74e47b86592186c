"""The training step's tensor-core kernels over the shapes and batch sizes that
choose between them: the fused layer chain, the fused input gradient and
scatter, and the split weight gradients."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import oracle as O  # noqa: E402
from paper_2504_21627_gb300 import inputs as I  # noqa: E402
from paper_2504_21627_gb300 import lsnif  # noqa: E402
from test_gpu_train import _batch, _cuda, _lab_cuda  # noqa: E402


def _object(L, F, W, nh, H, n_mat, act, N_max=24):
    cfg = I.Config(V=16, H=H, L=L, F=F, log2_T=12, N_min=4, N_max=N_max, n_hidden=nh, width=W, n_mat=n_mat,
                   activation=act)
    mesh = I.noise_torus_tris(4, 2000, n_mat=min(n_mat, 4))
    return cfg, mesh, I.random_params(cfg, seed=3, table_range=0.5, bias_range=0.1)


# one hidden layer; W 128 in the chain; the widest output layer; leaky; L F of
# 16, 32 and 64 (fused scatter) and 8 (separate one); a width outside the chain
@pytest.mark.parametrize("shape", [
    (8, 2, 64, 1, 18, 2, 0), (16, 2, 64, 3, 18, 4, 1), (4, 4, 128, 2, 18, 4, 0), (16, 4, 64, 2, 10, 56, 1),
    (2, 4, 128, 2, 18, 4, 1), (8, 2, 96, 2, 18, 2, 0),
])
def test_gradients_match_oracle_over_shapes(shape):
    """The bound of the step's gradients (1e-4 of the largest), kinks left out as in test_gpu_train."""
    cfg, mesh, p = _object(*shape)
    orc = O.build_object(mesh, cfg, p)
    rays, seg, lab = _batch({"orc": orc, "mesh": mesh}, 4000, seed=17)
    with lsnif.Context(0) as ctx:
        obj = ctx.load_object(mesh, cfg, tables=p.tables, mlp=p.packed_mlp())
        st = ctx.train_step(_cuda(rays), _lab_cuda(lab), obj, apply_update=False)
        ctx.check()
        g_mlp, g_tab = ctx.read_params(obj, lsnif.PARAM_GRAD_MLP), ctx.read_params(obj, lsnif.PARAM_GRAD_TABLES)
    terms, grads, gt = O.forward_backward(orc, rays, lab, seg)
    assert abs(st.total - terms["total"]) < 1e-4 * abs(terms["total"])
    ref = np.concatenate([np.concatenate([w.reshape(-1), b]) for w, b in grads])
    assert np.abs(g_mlp - ref).max() < 1e-4 * np.abs(ref).max()
    assert np.abs(g_tab - gt).max() < 1e-4 * np.abs(gt).max()


@pytest.mark.parametrize("shape", [(16, 2, 64, 2, 18, 4, 0), (8, 2, 64, 3, 18, 2, 1), (16, 4, 128, 2, 18, 4, 0)])
def test_a_batch_is_the_sum_of_its_parts(shape):
    """A batch large enough for the fused scatter against parts too small for it, ragged ones among them. The
    products of a ray are the same in both, only sums over rays take another order: FP32 sums of at most 18 x 5003
    terms per entry, whose rounding grows as sqrt(n) 2^-24 = 2e-5 of the terms' size; terms of both signs leave a
    sum a few times smaller than that, hence 1e-4 of the largest."""
    cfg, mesh, p = _object(*shape, N_max=40)
    n, ends = 5003, (0, 1, 130, 257, 700, 1400, 2100, 2800, 3500, 4200, 5003)
    torch_rays = torch.from_numpy(I.rays_sphere_to_box(n, 2.0, mesh.verts.min(0), mesh.verts.max(0), 5)).cuda()
    g = torch.Generator("cuda").manual_seed(1)
    r = lambda *s: torch.rand(s, device="cuda", generator=g)  # noqa: E731
    lab = {"occ": (r(n) < 0.7).float(), "t_local": r(n),
           "normal": torch.nn.functional.normalize(r(n, 3) - 0.5, dim=1).contiguous(), "albedo": r(n, 3),
           "mat": torch.randint(0, cfg.n_mat, (n,), device="cuda", generator=g, dtype=torch.int32)}

    def gradients(parts):
        with lsnif.Context(0) as ctx:
            obj = ctx.load_object(mesh, cfg, tables=p.tables, mlp=p.packed_mlp())
            k = ctx.trace(torch_rays, obj)[0]
            tab = mlp = loss = 0.0
            for lo, hi in parts:
                live = int((k[lo:hi] > 0).sum())
                st = ctx.train_step(torch_rays[:, lo:hi].contiguous(), {a: v[lo:hi].contiguous() for a, v in lab.items()},
                                    obj, apply_update=False)
                ctx.check()
                tab = tab + live * ctx.read_params(obj, lsnif.PARAM_GRAD_TABLES).astype(np.float64)
                mlp = mlp + live * ctx.read_params(obj, lsnif.PARAM_GRAD_MLP).astype(np.float64)
                loss = loss + live * st.total
            return loss, tab, mlp

    whole, parts = gradients([(0, n)]), gradients(list(zip(ends, ends[1:])))
    for a, b in zip(whole, parts):
        assert np.abs(b).max() > 0
        assert np.abs(a - b).max() <= 1e-4 * np.abs(b).max()


@pytest.mark.parametrize("shape", [(16, 2, 64, 2, 18, 4, 0), (8, 2, 64, 1, 18, 2, 1), (16, 4, 128, 2, 18, 4, 0),
                                   (4, 4, 128, 3, 10, 2, 0)])
@pytest.mark.parametrize("n,live", [(4999, 3000), (4608, 128), (4481, 1), (4480, 0)])
def test_rays_without_a_segment_change_nothing(shape, n, live):
    """The first layer's kernels take rays in order of their segment count and leave tiles without one out: a batch
    with rays that miss the box scattered through it against its other rays alone. Same products, sums in another
    order: the bound of the test above. No other ray at all: no loss, no gradient."""
    cfg, mesh, p = _object(*shape, N_max=12)
    rays = torch.from_numpy(I.rays_sphere_to_box(4 * n, 2.0, mesh.verts.min(0), mesh.verts.max(0), 7)).cuda()
    g = torch.Generator("cuda").manual_seed(2)
    r = lambda *s: torch.rand(s, device="cuda", generator=g)  # noqa: E731
    lab = {"occ": (r(n) < 0.7).float(), "t_local": r(n),
           "normal": torch.nn.functional.normalize(r(n, 3) - 0.5, dim=1).contiguous(), "albedo": r(n, 3),
           "mat": torch.randint(0, cfg.n_mat, (n,), device="cuda", generator=g, dtype=torch.int32)}
    with lsnif.Context(0) as ctx:
        obj = ctx.load_object(mesh, cfg, tables=p.tables, mlp=p.packed_mlp())
        rays = rays[:, ctx.trace(rays, obj)[0] > 0][:, :n].contiguous()
        assert rays.shape[1] == n
        keep = torch.zeros(n, dtype=torch.bool, device="cuda")
        keep[torch.randperm(n, device="cuda", generator=g)[:live]] = True
        rays[:3, ~keep] += 1000.0  # far outside, pointing past the box
        got = []
        for sel in (slice(None), keep):
            part = rays[:, sel].contiguous()
            if part.shape[1] == 0:
                continue
            st = ctx.train_step(part, {a: v[sel].contiguous() for a, v in lab.items()}, obj, apply_update=False)
            ctx.check()
            got.append((np.float64(st.total), ctx.read_params(obj, lsnif.PARAM_GRAD_TABLES),
                        ctx.read_params(obj, lsnif.PARAM_GRAD_MLP)))
    if live == 0:
        assert all(np.abs(x).max() == 0 for x in got[0])
        return
    for a, b in zip(*got):
        assert np.abs(b).max() > 0
        assert np.abs(a - b).max() <= 1e-4 * np.abs(b).max()
