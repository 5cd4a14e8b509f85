"""GPU tests of the integer slices at the ends of FP64, for every operator they serve: zeros of both signs, subnormals,
powers of two, values past the integers' range and values that are not finite (Gauss quadrature included).

Tolerances: 1e-13 as in test_gpu_slices.py.  Subnormal inputs (2^-1043 and below) keep about 31 bits and the mass
operator's results down to 13 of them; each of the six contractions and the pointwise step may then be off by eight units of
2^-1074, together up to 1e-2 of the smallest results: 2e-2, where a line taken for zero gives 1.
"""
import numpy as np
import pytest

import synthetic
from _util import gpu_mesh, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [(5, "gll", "diffusion"), (6, "gll", "diffusion"), (7, "gll", "diffusion"), (5, "gauss", "mass"), (6, "gauss", "mass"),
         (5, "gauss", "diffusion"), (6, "gauss", "diffusion"), (1, "tet", "mass"), (2, "tet", "diffusion"), (4, "tet", "mass"),
         (4, "tet", "diffusion")]


def _case(p, kind, op, dims=(2, 2, 1)):
    import paper_2109_05072_gb300 as ceed
    cop = ceed.CEED_OP_DIFFUSION if op == "diffusion" else ceed.CEED_OP_MASS
    if kind == "tet":
        m = synthetic.TetMesh(*dims, p, seed=p)
        h = ceed.ceed_nt_setup(m.n_elem, m.n_ldof, *ceed.ceed_simplex_basis(p, p + 1), torch.from_numpy(m.elem_dofs).cuda(),
                               torch.from_numpy(m.vertices).cuda(), torch.from_numpy(m.boundary).cuda())
        qd = ceed.alloc_nt_qdata(h, cop, ceed.CEED_F64)
        ceed.ceed_nt_build_qdata(h, cop, ceed.CEED_COEFF_ONE, None, ceed.CEED_F64, qd)
    else:
        m = synthetic.HexMesh(*dims, p, seed=p)
        h = gpu_mesh(ceed, m, kind)
        qd = ceed.alloc_qdata(h, cop, ceed.CEED_F64)
        ceed.ceed_build_qdata(h, cop, ceed.CEED_COEFF_SINE, None, ceed.CEED_F64, qd)

    def apply(x):
        xd = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        yd = torch.full_like(xd, float("nan"))
        if kind == "tet":
            ceed.ceed_nt_apply(h, cop, qd, ceed.CEED_F64, xd, yd)
        else:
            (ceed.ceed_apply_diffusion if op == "diffusion" else ceed.ceed_apply_mass)(h, qd, ceed.CEED_F64, xd, yd)
        return yd.cpu().numpy()

    return m, h, apply


@pytest.mark.parametrize("p,kind,op", CASES)
def test_zeros_of_both_signs(p, kind, op):
    m, h, apply = _case(p, kind, op)
    z = np.zeros(m.n_ldof)
    assert not apply(z).any() and not apply(-z).any()
    z[::2] = -0.0
    assert not apply(z).any()
    h.close()


@pytest.mark.parametrize("p,kind,op", CASES)
def test_subnormal_values(p, kind, op):
    m, h, apply = _case(p, kind, op)
    x = synthetic.uniform(m.n_ldof, seed=11)
    y = apply(x)
    for k in (-1043, -1030):
        assert rel_err(np.ldexp(apply(np.ldexp(x, k)), 1000), np.ldexp(y, k + 1000)) <= 2e-2
    h.close()


@pytest.mark.parametrize("p,kind,op", [c for c in CASES if c[1] == "gauss"])
def test_gauss_powers_of_two_and_range(p, kind, op):
    m, h, apply = _case(p, kind, op)
    x = synthetic.uniform(m.n_ldof, seed=7)
    y = apply(x)
    for k in (-600, 600):
        assert np.array_equal(apply(np.ldexp(x, k)), np.ldexp(y, k))
    for k in (-950, 890):   # past either end of the integers' range
        assert rel_err(np.ldexp(apply(np.ldexp(x, k)), -k), y) <= 1e-13
    h.close()


@pytest.mark.parametrize("p,kind,op", [c for c in CASES if c[1] == "gauss"])
def test_gauss_nonfinite_values_stay_in_their_elements(p, kind, op):
    m, h, apply = _case(p, kind, op)
    x = synthetic.uniform(m.n_ldof, seed=9)
    y = apply(x)
    for bad in (np.nan, np.inf, -np.inf):
        z = x.copy()
        node = int(m.elem_dofs[0, 0])
        z[node] = bad
        out = apply(z)
        touched = np.zeros(m.n_ldof, dtype=bool)
        touched[m.elem_dofs[(m.elem_dofs == node).any(axis=1)]] = True
        assert not np.isfinite(out[node])
        assert np.array_equal(out[~touched], y[~touched])
    h.close()
