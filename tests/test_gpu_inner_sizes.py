"""The handle-free inner product at the edges of its launch (GPU).

Its kernel takes 128 components (21 1/3 tetrahedra) per block and pass, at most 2,432 blocks: below one block, across a
block's edge, past one pass of the grid (51,882 tetrahedra) with a ragged end, and at the largest size accepted; and
replayed from a captured graph.  Compared with the dense FP64 mass matrix.

Tolerance: the kernel's sums are at most 60 additions deep (21 passes, 5 + 4 within a block, 10 + 8 over the blocks,
the rest inside a component's form), the dense reference's at most 60 (20 + 20 in the products, pairwise sums), each
rounding 1.1e-16 of at most 0.3 |x||y| per component (the forms' coefficients over their denominators): 120 x 1.1e-16
x 0.3 = 4e-15, taken as 1e-14 sum w |x||y|.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _data(torch, order, nt):
    np_ = (order + 1) * (order + 2) * (order + 3) // 6
    rng = np.random.default_rng(nt + order)
    u, v = rng.standard_normal((2, nt, 6, np_))
    w = rng.uniform(0.5, 2.0, (nt, 2))
    from oracle.refelem import ref_element
    M = ref_element(order).M / 8  # bi-unit to unit tetrahedron
    wc = np.repeat(w, 3, axis=1)
    ref = float((wc * ((u @ M) * v).sum(2)).sum())
    tol = 1e-14 * float((wc * np.sqrt((u * u).sum(2) * (v * v).sum(2))).sum())
    dev = torch.device("cuda:0")
    t = [torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in (u, v, w)]
    return t, torch.full((1,), float("nan"), dtype=torch.float64, device=dev), ref, tol


@pytest.mark.parametrize("order,nt", [(q, nt) for q in (1, 2, 3) for nt in (1, 21, 22, 129)]
                         + [(2, 51_883), (3, 51_905), (1, 1_048_576)])
def test_inner_against_the_dense_matrix(order, nt):
    from paper_2106_02858_gb300 import build
    build.build()
    import torch
    from paper_2106_02858_gb300 import cmcg
    (u, v, w), out, ref, tol = _data(torch, order, nt)
    cmcg.cmcg_inner_noalloc(order, nt, u, v, w, out, torch.cuda.current_stream())
    assert abs(float(out.item()) - ref) <= tol, (out.item(), ref, tol)
    if nt != 129:
        return
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        cmcg.cmcg_inner_noalloc(order, nt, u, v, w, out, torch.cuda.current_stream())
    out.fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    assert abs(float(out.item()) - ref) <= tol, (out.item(), ref, tol)
