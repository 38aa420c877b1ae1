"""The direction of a stage over the mesh does not show in its results (GPU).

Handles whose fields take more than 3/5 of L2 launch their stages from the first tetrahedron to the last and back in
turn; smaller ones always forward.  A batch of many copies of one small problem is over the line, two copies are
under it: every copy has to give the same bits, with a number of tetrahedra that leaves the last blocks
partly empty, in each of the kernels that take the direction (one and two warps per half tile, tensor cores, FP64).
"""
import math

import numpy as np
import pytest

from paper_2106_02858_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order,fp64,form", [(2, False, 1), (2, False, 4), (3, False, 7), (1, True, 1), (2, True, 3)])
def test_both_directions_give_the_same_bits(order, fp64, form):
    from paper_2106_02858_gb300 import build
    build.build()
    from paper_2106_02858_gb300 import cmcg
    p = I.cube_problem(5, order, 2 * math.pi, (0.5, 0.5, 0.5), (1, 0, 0), 0.3)
    np_ = (order + 1) * (order + 2) * (order + 3) // 6
    per_tet = 6 * np_ * (8 if fp64 else 4) * 3 + 16 + (53 * 8 if fp64 else 41 * 4)
    n = int(90e6 / (per_tet * p.nt)) + 1
    opt = cmcg.cmcg_default_options(order=order, precision=cmcg.CMCG_FP64 if fp64 else cmcg.CMCG_FP32,
                                    stage_variant=form)
    mesh = cmcg.make_mesh(p.mesh.verts, p.mesh.tets, p.mesh.tags)
    rng = np.random.default_rng(order)
    jr, ji = rng.standard_normal((2, p.nt, 3, np_))

    def run(count):
        h = cmcg.cmcg_create_batch([(mesh, p.eps, p.mu, p.omega)] * count, opt)
        try:
            return cmcg.cmcg_solve_batch(h, [jr] * count, [ji] * count, tol=1e-30, max_iter=2)
        finally:
            h.close()

    (e0, h0, _), (e1, h1, _) = run(2), run(n)
    assert np.isfinite(e0[0]).all() and np.abs(e0[0]).max() > 0
    for k in (0, 1, n // 2, n - 1):
        assert np.array_equal(e1[k], e0[0]) and np.array_equal(h1[k], h0[0]), k
