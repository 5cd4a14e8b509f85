"""GPU tests of the FP64 contractions by exact integer slices on the tensor cores: the collocated
diffusion operator with 6 to 8 points per direction, and the non-tensor operator with up to 35 basis
functions.

Tolerance against the oracle: every contraction is exact up to 2^-60 of its line's largest value and one
rounding; with six of them in a row, the pointwise step and the sums at shared nodes the norm-wise error
stays below 100 units of 2^-53, 1.1e-14; the oracle's own dense sums (512 terms a point) add up to
sqrt(512) units.  1e-13 covers both.  Everything is relative to a power of two, so scaling the input by one
scales the result exactly; inputs outside the integers' range take FP64 FMAs (1e-13 again).
"""
import numpy as np
import pytest

import synthetic
from oracle import fem
from oracle import simplex as sx
from _util import gpu_mesh, oracle_qdata, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-13


@pytest.fixture(scope="module")
def ceed():
    import paper_2109_05072_gb300 as c
    assert torch.cuda.is_available()
    return c


def _hex(ceed, p, dims, ncomp=1):
    m = synthetic.HexMesh(*dims, p, seed=p)
    mesh = gpu_mesh(ceed, m, "gll", ncomp=ncomp)
    qd = ceed.alloc_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_F64)
    ceed.ceed_build_qdata(mesh, ceed.CEED_OP_DIFFUSION, ceed.CEED_COEFF_SINE, None, ceed.CEED_F64, qd)

    def apply(x, nrhs=1, flags=0):
        xd = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        yd = torch.full_like(xd, float("nan"))
        ceed.ceed_apply_diffusion(mesh, qd, ceed.CEED_F64, xd, yd, nrhs, flags)
        return yd.cpu().numpy()

    return m, mesh, apply


def _tet(ceed, p, dims, op):
    m = synthetic.TetMesh(*dims, p, seed=p)
    nt = ceed.ceed_nt_setup(m.n_elem, m.n_ldof, *ceed.ceed_simplex_basis(p, p + 1), torch.from_numpy(m.elem_dofs).cuda(),
                            torch.from_numpy(m.vertices).cuda(), torch.from_numpy(m.boundary).cuda())
    cop = ceed.CEED_OP_DIFFUSION if op == "diffusion" else ceed.CEED_OP_MASS
    qd = ceed.alloc_nt_qdata(nt, cop, ceed.CEED_F64)
    ceed.ceed_nt_build_qdata(nt, cop,
                             ceed.CEED_COEFF_SINE if op == "diffusion" else ceed.CEED_COEFF_ONE, None, ceed.CEED_F64, qd)

    def apply(x, flags=0):
        xd = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        yd = torch.full_like(xd, float("nan"))
        ceed.ceed_nt_apply(nt, cop, qd, ceed.CEED_F64, xd, yd, flags=flags)
        return yd.cpu().numpy()

    return m, nt, apply


@pytest.mark.parametrize("p,dims,ncomp,nrhs", [(5, (3, 2, 2), 1, 1), (6, (2, 3, 2), 1, 1), (7, (3, 2, 2), 1, 1),
                                                (5, (1, 1, 1), 3, 2), (7, (1, 2, 1), 1, 3)])
def test_hex_against_oracle(ceed, p, dims, ncomp, nrhs):
    m, mesh, apply = _hex(ceed, p, dims, ncomp)
    cols = ncomp * nrhs
    x = synthetic.uniform(m.n_ldof * cols, seed=3).reshape(m.n_ldof, cols)
    sp_, qref = oracle_qdata(m, "gll", "diffusion", "sine")
    a = lambda v: fem.apply(sp_, m.elem_dofs, qref, v, fem.DIFFUSION)
    for flags, f in ((0, a), (ceed.CEED_APPLY_DIRICHLET, fem.masked(a, m.boundary))):
        y = apply(x, nrhs, flags)
        for c in range(cols):
            assert rel_err(y[:, c], f(np.ascontiguousarray(x[:, c]))) <= TOL
    mesh.close()


@pytest.mark.parametrize("p,op", [(1, "diffusion"), (2, "mass"), (3, "diffusion"), (4, "mass"), (4, "diffusion")])
def test_tet_against_oracle(ceed, p, op):
    m, nt, apply = _tet(ceed, p, (3, 2, 2), op)   # 72 elements: a full block of 64 and a rest
    x = synthetic.uniform(m.n_ldof, seed=5)
    sp_ = sx.SimplexSpace(p, p + 1)
    if op == "diffusion":
        qd, fop = sx.qdata_diffusion(sp_, m.vertices, "sine"), fem.DIFFUSION
    else:
        qd, fop = sx.qdata_mass(sp_, m.vertices), fem.MASS
    assert rel_err(apply(x), fem.apply(sp_, m.elem_dofs, qd, x, fop)) <= TOL
    nt.close()


def _cases(ceed):
    for p in (5, 6, 7):
        yield _hex(ceed, p, (2, 2, 1))
    for p in (1, 4):
        yield _tet(ceed, p, (2, 1, 1), "diffusion")


def test_powers_of_two_and_range(ceed):
    for m, h, apply in _cases(ceed):
        x = synthetic.uniform(m.n_ldof, seed=7)
        y = apply(x)
        for k in (-600, 600):
            assert np.array_equal(apply(np.ldexp(x, k)), np.ldexp(y, k))
        for k in (-950, 890):   # past either end of the integers' range
            assert rel_err(np.ldexp(apply(np.ldexp(x, k)), -k), y) <= TOL
        # values of very different size in one element
        z = np.ldexp(x, np.random.default_rng(1).integers(-40, 1, x.size))
        assert rel_err(apply(z) + apply(x - z), y) <= TOL
        assert not apply(np.zeros_like(x)).any()
        h.close()


def test_nonfinite_values_stay_in_their_elements(ceed):
    for m, h, apply in _cases(ceed):
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
