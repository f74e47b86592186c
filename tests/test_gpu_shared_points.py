"""Shared boundary points in the resident fused kernel (copied from the chunk before by the warp that multiplies) over
the rings it runs with: two, three and four slots, L F of 8 and of 0 modulo 16, both widths, against the oracle at the
16-bit paths' bounds."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import oracle as O  # noqa: E402
from paper_2504_21627_gb300 import inputs as I  # noqa: E402
from paper_2504_21627_gb300 import lsnif  # noqa: E402
from test_gpu_query import BF16_TOL, FP16_TOL, _query_compare, fp32_tol  # noqa: E402


# (L, F, width, hidden layers): the parameter study's shape and others of 8 modulo 16, then rings of 2, 3 and 4 slots
@pytest.mark.parametrize("shape", [(2, 4, 128, 2), (4, 2, 64, 2), (12, 2, 64, 4), (16, 4, 64, 1), (8, 2, 64, 3),
                                   (16, 2, 128, 1)])
@pytest.mark.parametrize("prec", [lsnif.BF16_FUSED, lsnif.FP16_FUSED])
def test_shared_points_over_the_rings(shape, prec):
    L, F, W, n_hidden = shape
    cfg = I.Config(V=32, H=18, L=L, F=F, log2_T=10, N_min=4, N_max=64, n_hidden=n_hidden, width=W, n_mat=2)
    mesh = I.noise_torus_tris(4, 2000, n_mat=2)
    p = I.random_params(cfg, seed=3, table_range=0.3, bias_range=0.1)
    orc = O.build_object(mesh, cfg, p)
    rays = I.rays_sphere_to_box(1500, 3.0, orc.bmin, orc.bmax, seed=11)
    with lsnif.Context(0) as ctx:
        o = {"h": ctx.load_object(mesh, cfg, tables=p.tables, mlp=p.packed_mlp()), "orc": orc}
        _, _, seg = _query_compare(ctx, o, rays, prec, (BF16_TOL if prec == lsnif.BF16_FUSED else FP16_TOL) + fp32_tol(cfg))
    s = np.arange(1, cfg.H // 2)
    shared = np.isclose(seg.pts[:, 2 * s], seg.pts[:, 2 * s - 1], rtol=0, atol=1e-9).all(-1) & (s[None] < seg.k[:, None])
    assert shared.mean() > 0.05, "the rays have shared points"
