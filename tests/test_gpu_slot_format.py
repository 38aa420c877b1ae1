"""cmcg_slot_restore of a state in the first layout (GPU).

The first layout held nodal values as [tile of 32][component][node][lane] in the order of the shape
classes, with J_re and J_im apart.  A state saved now is rewritten into that layout here, restored,
and has to continue as the state itself does: to the same bits in FP32 (the values are only moved),
and in FP64 to 1e-9 of the converged solve with the same iteration count, the tolerance of converged
FP64 solves (the change of basis rounds, and CG amplifies rounding in its transient).

Meshes: one shape class per Kuhn tetrahedron (27 and 8 tetrahedra per class, ragged half tiles, the
half tiles of the classes interleaved) and a distorted mesh (a single class).
"""
import math
import struct

import numpy as np
import pytest

from paper_2106_02858_gb300 import inputs as I

pytestmark = pytest.mark.gpu

HEADER = 8 + 6 * 4 + 2 * 8 + 2 * 8 + 6 * 8 + 2 * 4  # magic, six int32, two int64, two doubles, the CG scalars


@pytest.fixture(scope="module")
def lib():
    from paper_2106_02858_gb300 import build
    build.build()
    from paper_2106_02858_gb300 import cmcg
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return cmcg


def _values_at_nodes(q):
    """Bernstein coefficients -> nodal values."""
    lat = I.node_lattice(q)
    full = np.concatenate([q - lat.sum(1, keepdims=True), lat], axis=1)
    f = math.factorial
    return np.array([[f(q) / math.prod(f(int(k)) for k in a) * math.prod((x / q) ** k for x, k in zip(p, a))
                      for a in full] for p in full])


def _first_layout(state, q, dtype, classes):
    np_ = I.n_nodes(q)
    body = np.frombuffer(state[HEADER:], dtype).reshape(4, -1, 3, np_, 16, 2)  # U0, R, D, J
    pos = np.concatenate([(np.arange(h) + 0.5) / h for h in classes])
    place = np.argsort(pos, kind="stable")
    old = np.empty_like(body)
    old[:, place] = body
    if dtype == np.float64:
        old = np.einsum("nm,vhcmlf->vhcnlf", _values_at_nodes(q), old)
    old = old.reshape(4, -1, 2, 3, np_, 16, 2).transpose(0, 1, 6, 3, 4, 2, 5)  # vector, tile, field, c, node, half, lane
    parts = [old[k].reshape(-1) for k in range(3)] + [old[3][:, f].reshape(-1) for f in range(2)]
    return b"CMCGSLT1" + state[8:HEADER] + np.concatenate(parts).astype(dtype).tobytes()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("q,kind", [(1, "cube3"), (2, "cube3"), (3, "cube2"), (2, "distorted")])
def test_state_of_the_first_layout_continues(lib, prec, q, kind):
    n = 2 if kind == "cube2" else 3
    p = I.cube_problem(n, q, 4 * math.pi, (0.4, 0.5, 0.6), (0.2, 1.0, -0.3), 0.2, tol=1e-6)
    classes = [2 * (-(-n**3 // 32))] * 6
    if kind == "distorted":
        v = p.mesh.verts
        inner = np.all((v > 1e-9) & (v < 1 - 1e-9), axis=1)
        v[inner] += np.random.default_rng(0).uniform(-0.04, 0.04, (int(inner.sum()), 3))
        classes = [2 * (-(-p.nt // 32))]
    dtype = np.float32 if prec == "fp32" else np.float64
    h, mesh = lib.create_for_problem(p, precision=lib.CMCG_FP32 if prec == "fp32" else lib.CMCG_FP64, stage_variant=1)
    lib.cmcg_slot_admit(h, 0, p.j_re, 0.5 * p.j_re)
    for _ in range(4):
        lib.cmcg_slot_round(h, 1e-6, 400)
    state = lib.cmcg_slot_save(h, 0)
    assert state[:8] == b"CMCGSLT2" and struct.unpack_from("<3i", state, 8)[1:] == (q, I.n_nodes(q))
    results = []
    for s in (state, _first_layout(state, q, dtype, classes)):
        lib.cmcg_slot_restore(h, 0, s)
        for _ in range(2000):
            if lib.cmcg_slot_round(h, 1e-6, 400):
                break
        results.append(lib.cmcg_slot_take(h, 0))
    h.close()
    (e, m, info), (e1, m1, info1) = results
    assert info.status == lib.CMCG_OK and info1.iters == info.iters
    if prec == "fp32":
        assert np.array_equal(e, e1) and np.array_equal(m, m1)
    else:
        scale = np.abs(np.concatenate([e, m], 1)).max()
        assert np.abs(e - e1).max() <= 1e-9 * scale and np.abs(m - m1).max() <= 1e-9 * scale
