"""GPU tests of the FP64 non-tensor operator with bases of the caller's own: no output of the integer slices has less
precision than a chain of FP64 FMAs over its own terms, whatever the element's other values are.

Each element has nodes of its own, so an output is one element's.  Bound, entry by entry: the chain's, P + Q + 8 rounding
errors of 2^-53 each against the sum of the magnitudes of the entry's terms, and 32 for the determinant.
"""
import numpy as np
import pytest

import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = np.array([1.0, 0.7, 1e-12, 3e-15, 1e-18, 2e-9])


def _mass(B, weights, x_of_element, n_elem=72):
    import paper_2109_05072_gb300 as ceed
    Q, P = B.shape
    m = synthetic.TetMesh(3, 2, 2, 1, seed=1)
    assert m.n_elem == n_elem
    dofs = np.arange(n_elem * P, dtype=np.int32).reshape(n_elem, P)
    qref = np.full((Q, 3), 0.25)
    h = ceed.ceed_nt_setup(n_elem, n_elem * P, B, np.zeros((3, Q, P)), weights, qref, torch.from_numpy(dofs).cuda(),
                           torch.from_numpy(m.vertices).cuda(), None)
    qd = ceed.alloc_nt_qdata(h, ceed.CEED_OP_MASS, ceed.CEED_F64)
    ceed.ceed_nt_build_qdata(h, ceed.CEED_OP_MASS, ceed.CEED_COEFF_ONE, None, ceed.CEED_F64, qd)
    x = np.stack([x_of_element(e) for e in range(n_elem)])
    xd = torch.from_numpy(np.ascontiguousarray(x.reshape(-1))).cuda()
    yd = torch.full_like(xd, float("nan"))
    ceed.ceed_nt_apply(h, ceed.CEED_OP_MASS, qd, ceed.CEED_F64, xd, yd)
    V = m.vertices
    det = np.abs(np.linalg.det(V[:, 1:] - V[:, :1]))
    h.close()
    return x, yd.cpu().numpy().reshape(n_elem, P), det


def _check(B, weights, x_of_element):
    x, y, det = _mass(B, weights, x_of_element)
    L = np.longdouble
    w = weights.astype(L)[None, :] * det.astype(L)[:, None]
    ref = np.einsum("qn,eq->en", B.astype(L), w * np.einsum("qn,en->eq", B.astype(L), x.astype(L)))
    mag = np.einsum("qn,eq->en", np.abs(B).astype(L), w * np.einsum("qn,en->eq", np.abs(B).astype(L), np.abs(x).astype(L)))
    assert np.all(np.abs(y - ref) <= (sum(B.shape) + 8 + 32) * L(2) ** -53 * mag), float(np.max(np.abs(y - ref) / np.where(mag > 0, mag, 1)))


@pytest.mark.parametrize("P,Q", [(4, 8), (12, 24), (35, 24)])
def test_blocks_of_nodes_keep_their_own_precision(P, Q):
    """Half of the nodes at half of the points, the others at the rest: sizes of one half say nothing about the other's."""
    rng = np.random.default_rng(P)
    B = np.zeros((Q, P))
    B[: Q // 2, : P // 2] = rng.uniform(0.5, 1.0, (Q // 2, P // 2))
    B[Q // 2:, P // 2:] = rng.uniform(-1.0, -0.5, (Q - Q // 2, P - P // 2))
    half = np.arange(P) < P // 2
    _check(B, np.ones(Q), lambda e: rng.uniform(-1, 1, P) * np.where(half, SIZES[e % 6], SIZES[(e // 6) % 6]))


@pytest.mark.parametrize("P", [4, 12])
def test_points_of_very_different_weight(P):
    """The last nodes see only the points of small weight, in the same group of eight and in another."""
    rng = np.random.default_rng(P)
    for small in (slice(4, 8), slice(8, 16)):
        B = rng.uniform(0.5, 1.0, (16, P))
        weights = np.ones(16)
        weights[small] = 1e-17
        big = np.ones(16, dtype=bool)
        big[small] = False
        B[np.ix_(big, [P - 2, P - 1])] = 0.0
        _check(B, weights, lambda e: rng.uniform(-1, 1, P))


@pytest.mark.parametrize("P", [4, 20])
def test_nodal_basis(P):
    rng = np.random.default_rng(P)
    _check(np.eye(P), rng.uniform(0.5, 1.0, P), lambda e: rng.uniform(-1, 1, P) * SIZES[rng.integers(0, 6, P)])


@pytest.mark.parametrize("P", [4, 35])
def test_spread_values_on_a_full_basis(P):
    rng = np.random.default_rng(P)
    _check(rng.uniform(-1, 1, (24, P)), rng.uniform(0.5, 1.0, 24), lambda e: rng.uniform(-1, 1, P) * SIZES[rng.integers(0, 6, P)])


def test_tables_of_any_scale():
    rng = np.random.default_rng(3)
    B, w = rng.uniform(0.5, 1.0, (8, 4)), np.ones(8)
    x0 = rng.uniform(-1, 1, (72, 4))
    _, y, _ = _mass(B, w, lambda e: x0[e])
    for k in (-450, 450):
        yk = _mass(np.ldexp(B, k), w, lambda e: x0[e])[1]
        assert np.max(np.abs(np.ldexp(yk, -2 * k) - y)) <= 1e-14 * np.max(np.abs(y))
    B[0, 0] = np.inf
    assert not np.isfinite(_mass(B, w, lambda e: x0[e])[1]).any()
    assert not _mass(np.zeros((8, 4)), w, lambda e: x0[e])[1].any()
