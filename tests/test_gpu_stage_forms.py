"""The stage-kernel form of a handle does not show in its results (GPU).

A handle takes the form that is fastest on its mesh by a timing at creation, so the forms it chooses
from (FP64: all three; FP32: 0 to 5 of orders 1 and 2, and the same code at order 3) have to give the
same bits in every kind of stage, on meshes with ragged half tiles.  A slot saved under one form and
restored under another then continues to the same bits too.
"""
import math

import numpy as np
import pytest

from paper_2106_02858_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_2106_02858_gb300 import build
    build.build()
    from paper_2106_02858_gb300 import cmcg
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return cmcg


@pytest.mark.parametrize("n", [2, 3])
@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_forms_give_the_same_bits(lib, prec, order, n):
    p = I.cube_problem(n, order, 4 * math.pi, (0.4, 0.5, 0.6), (0.2, 1.0, -0.3), 0.2)
    rng = np.random.default_rng(order)
    u = rng.standard_normal((p.nt, 6, p.np_))
    jr, ji = rng.standard_normal((2, p.nt, 3, p.np_))
    sigma = rng.uniform(0, 1, p.nt)
    gr, gi = rng.standard_normal((2, p.nt, 4, 3, (order + 1) * (order + 2) // 2))
    first = None
    for form in range(1, 7 if prec == "fp32" else 4):
        h, _ = lib.create_for_problem(p, precision=lib.CMCG_FP32 if prec == "fp32" else lib.CMCG_FP64,
                                      stage_variant=form)
        out = [lib.dgtd_period_forward(h, u), lib.dgtd_period_adjoint(h, u),
               *lib.dgtd_period_forward(h, u, jr, ji, filtered=True)]
        lib.cmcg_set_conductivity(h, sigma)
        lib.cmcg_set_boundary_data(h, gr, gi)
        out += [lib.dgtd_apply(h, 0.1, u, jr, ji), lib.dgtd_apply(h, 0.1, u, adjoint=True),
                *lib.dgtd_period_forward(h, u, jr, ji, filtered=True)]
        h.close()
        assert all(np.isfinite(x).all() for x in out)
        first = out if first is None else first
        assert [np.array_equal(x, y) for x, y in zip(out, first)] == [True] * len(first), form


@pytest.mark.parametrize("prec,forms", [("fp64", (1, 3, 2)), ("fp32", (2, 6, 5))])
def test_resume_under_another_form(lib, prec, forms):
    b = I.batched_rhs(nrhs=1, n=3, order=2, tol=1e-6)
    results = []
    for resumed in forms:
        hs = [lib.create_for_problem(
            I.Problem("one", b.mesh, b.eps, b.mu, b.omega, 2, b.j_re[0], b.j_im[0], 1e-6),
            precision=lib.CMCG_FP32 if prec == "fp32" else lib.CMCG_FP64, stage_variant=v)[0] for v in (forms[0], resumed)]
        lib.cmcg_slot_admit(hs[0], 0, b.j_re[0], b.j_im[0])
        for _ in range(5):
            lib.cmcg_slot_round(hs[0], 1e-6, 400)
        lib.cmcg_slot_restore(hs[1], 0, lib.cmcg_slot_save(hs[0], 0))
        while not lib.cmcg_slot_round(hs[1], 1e-6, 400):
            pass
        results.append(lib.cmcg_slot_take(hs[1], 0))
        for h in hs:
            h.close()
    for e, m, info in results:
        assert info.status == lib.CMCG_OK and info.iters == results[0][2].iters
        assert np.array_equal(e, results[0][0]) and np.array_equal(m, results[0][1])
