"""The FP32 query's fused kernel (gather, network and decode in one launch)
against the FP64 oracle, at the edges of its tiles and shapes.

Tolerance: every output is a chain of at most n_in = 1152 FP32 fused
multiply-adds per layer over values of order 1, so its error is below
1152 x 2^-24 = 7e-5 of the largest logit per layer in the worst case and
around sqrt(1152) x 2^-24 = 2e-6 in practice; 1e-4 is the bound the FP32 path
is held to elsewhere."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2504_21627_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# (L, F, width, n_hidden, H, n_mat, activation): several segments per chunk,
# one, a chunk of two sub-chunks, the widest output layer, the largest L F
SHAPES = [
    (1, 2, 64, 1, 16, 1, 0),
    (2, 4, 128, 2, 18, 4, 0),
    (8, 2, 64, 3, 18, 2, 1),
    (16, 2, 64, 4, 18, 40, 0),
    (16, 4, 128, 4, 18, 56, 0),
    (16, 4, 64, 2, 10, 20, 1),
    (5, 2, 128, 1, 64, 8, 0),
    (8, 2, 64, 2, 2, 2, 0),
]


def _object(shape, seed=3):
    L, F, W, nh, H, n_mat, act = shape
    cfg = I.Config(V=16, H=H, L=L, F=F, log2_T=9, N_min=4, N_max=48, n_hidden=nh, width=W, n_mat=n_mat,
                   activation=act)
    return cfg, I.random_params(cfg, seed=seed, table_range=0.5, bias_range=0.1), I.noise_torus_tris(4, 600, n_mat=1)


def _query(cfg, params, mesh, rays):
    import torch
    from paper_2504_21627_gb300 import lsnif
    with lsnif.Context(0) as ctx:
        obj = ctx.load_object(mesh, cfg, tables=params.tables, mlp=params.packed_mlp())
        out = ctx.query_rays(torch.from_numpy(rays).cuda(), obj=obj, precision=lsnif.FP32_PLAIN, logits=True)
        ctx.check()
        return out.logits.cpu().numpy(), out.hit.cpu().numpy(), out.t.cpu().numpy()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("n", [1, 33, 1000])
def test_logits_match_the_oracle(shape, n):
    cfg, params, mesh = _object(shape)
    orc = O.build_object(mesh, cfg, params)
    rays = I.rays_sphere_to_box(n, 3.0, orc.bmin, orc.bmax, seed=7 + n)
    ref, seg = O.query(orc, rays)
    got, _, t = _query(cfg, params, mesh, rays)
    ok = ref.live & ~seg.near
    assert not np.isfinite(t[~ref.live & ~seg.near]).any()
    if ok.any():
        assert np.abs(got[ok] - ref.logits[ok]).max() <= 1e-4 * max(1.0, np.abs(ref.logits[ok]).max())


@pytest.mark.parametrize("shape", [SHAPES[2], SHAPES[4]])
def test_large_tiles_give_the_small_tiles_bits(shape):
    """More rays than 32-row tiles serve: each ray's outputs are those it has in a small call."""
    cfg, params, mesh = _object(shape)
    lo, hi = mesh.verts.min(0), mesh.verts.max(0)
    rays = I.rays_sphere_to_box(40001, 3.0, lo, hi, seed=5)
    big = _query(cfg, params, mesh, rays)
    small = _query(cfg, params, mesh, np.ascontiguousarray(rays[:, 20000:20333]))
    for b, s in zip(big, small):
        np.testing.assert_array_equal(b[20000:20333], s)


def test_a_non_finite_weight_of_an_empty_slot_reaches_the_outputs():
    """0 times a non-finite weight is not 0: segments no ray reaches are not skipped then."""
    cfg, params, mesh = _object(SHAPES[2])
    rays = I.rays_sphere_to_box(200, 3.0, mesh.verts.min(0), mesh.verts.max(0), seed=5)
    clean = _query(cfg, params, mesh, rays)[0]
    params.weights[0][0][:, -1] = np.inf
    got = _query(cfg, params, mesh, rays)[0]
    assert np.isnan(got[np.isfinite(clean).all(1)]).all()
