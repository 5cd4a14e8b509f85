"""GPU test of blocks that hold several of an element's columns: the same bits as one column at a time.

20^3 elements, one per block: 1,000 element blocks a colour.  Five columns then go to two groups, three columns and
two (2,432 / 1,000 groups at most); three columns to two groups, two and one; thirteen to two groups of
seven and six.
"""
import pytest

import synthetic
from _util import gpu_mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,qkind,op,prec", [(2, "gll", "diffusion", 0), (3, "gauss", "mass", 0), (5, "gll", "diffusion", 0),
                                             (5, "gauss", "mass", 0), (5, "gauss", "diffusion", 0), (2, "gll", "diffusion", 1),
                                             (2, "gll", "diffusion", 5), (3, "gauss", "diffusion", 5)])
@pytest.mark.parametrize("stage", [0, 1])
def test_column_groups(p, qkind, op, prec, stage):
    import paper_2109_05072_gb300 as ceed
    cop = ceed.CEED_OP_DIFFUSION if op == "diffusion" else ceed.CEED_OP_MASS
    f = ceed.ceed_apply_diffusion if op == "diffusion" else ceed.ceed_apply_mass
    m = synthetic.HexMesh(20, 20, 20, p, seed=p)
    mesh = gpu_mesh(ceed, m, qkind)
    qd = ceed.alloc_qdata(mesh, cop, prec)
    ceed.ceed_build_qdata(mesh, cop, ceed.CEED_COEFF_SINE, None, prec, qd)
    ceed.ceed_set_apply_variant(mesh, cop, prec, 1, stage)
    for ncol in (3, 5, 13):
        x = torch.from_numpy(synthetic.uniform(m.n_ldof * ncol, seed=ncol)).cuda()
        for flags in (0, ceed.CEED_APPLY_DIRICHLET):
            y = torch.full_like(x, float("nan"))
            f(mesh, qd, prec, x, y, ncol, flags)
            for c in range(ncol):
                x1 = x.reshape(-1, ncol)[:, c].contiguous()
                y1 = torch.full_like(x1, float("nan"))
                f(mesh, qd, prec, x1, y1, 1, flags)
                assert torch.equal(y1, y.reshape(-1, ncol)[:, c])
    ceed.ceed_mesh_status(mesh)
    mesh.close()
