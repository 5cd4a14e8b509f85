"""GPU test of the fused PCG iteration where every block has several pieces of a colour (it waits at the first only and
counts itself once per colour): against the separate kernels, and the same bits on a second run.

The meshes hold more pieces a colour than blocks can be resident (152 SMs x 32 blocks of 9 threads at p = 2 with one
element a piece; 152 x 16 of 32 threads or more at p = 5), with a remainder.  The two ways differ in the grouping of
their sums only: about 1e-15 a step with FP64 and double-float operators, and where that moves the rounding of an entry to
FP32 by 2^-24 of the entry; 12 steps: 1e-11 and 1e-6.
"""
import pytest

import synthetic
from _util import gpu_mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,dims,prec,tol", [(2, (36, 34, 33), 0, 1e-11), (5, (28, 27, 27), 0, 1e-11),
                                              (2, (36, 34, 33), 1, 1e-6), (2, (36, 34, 33), 5, 1e-11)])
def test_several_pieces_per_block(p, dims, prec, tol):
    import paper_2109_05072_gb300 as ceed
    m = synthetic.HexMesh(*dims, p, seed=2)
    mesh = gpu_mesh(ceed, m, "gll")
    op = ceed.CEED_OP_DIFFUSION
    qd = ceed.alloc_qdata(mesh, op, ceed.CEED_F64)
    ceed.ceed_build_qdata(mesh, op, ceed.CEED_COEFF_SINE, None, ceed.CEED_F64, qd)
    kw = dict(mode=ceed.CEED_CG_FP64, fixed_iters=12, op=op)
    if prec != ceed.CEED_F64:
        lo = ceed.alloc_qdata(mesh, op, prec)
        ceed.ceed_build_qdata(mesh, op, ceed.CEED_COEFF_SINE, None, prec, lo)
        kw = dict(mode=ceed.CEED_CG_MIXED_RELIABLE, tol=1e-14, max_iter=12, qdata_lo=lo, prec_lo=prec, op=op)
    ceed.ceed_set_apply_variant(mesh, op, prec, 1, 0)
    b = torch.empty(m.n_ldof, dtype=torch.float64, device="cuda")
    ceed.ceed_manufactured_rhs(mesh, ceed.CEED_COEFF_SINE, b, flags=ceed.CEED_APPLY_DIRICHLET)
    xs = []
    for separate in (0, 0, 1):
        x = torch.zeros_like(b)
        st, rep = ceed.ceed_cg_solve(mesh, qd, ceed.CEED_F64, b, x, raise_on_error=False, separate_kernels=separate, **kw)
        assert st in (ceed.CEED_OK, ceed.CEED_ERR_NOT_CONVERGED) and rep["fused"] == 1 - separate
        assert rep["iterations"] == 12
        xs.append(x)
    assert torch.equal(xs[0], xs[1])
    assert float((xs[0] - xs[2]).norm() / xs[2].norm()) <= tol
    mesh.close()
