"""GPU test of the one-cluster apply of small meshes (all colours in one launch): the same bits as the launches per colour.

Nine right-hand sides are more columns than a cluster holds, so they take the launches per colour; one takes the
cluster where the mesh fits it.  Meshes: one element, exactly full, one row of elements more than fit, ragged.
"""
import numpy as np
import pytest

import synthetic
from _util import gpu_mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,qkind,op,prec", [(1, "gll", "diffusion", 0), (2, "gauss", "mass", 0), (3, "gll", "diffusion", 1),
                                              (3, "gauss", "diffusion", 5), (5, "gll", "diffusion", 0), (7, "gll", "diffusion", 0),
                                              (6, "gauss", "mass", 0), (8, "gll", "diffusion", 0)])
@pytest.mark.parametrize("stage", [0, 1])
def test_cluster_gives_the_bits_of_the_colour_launches(p, qkind, op, prec, stage):
    import paper_2109_05072_gb300 as ceed
    cop = ceed.CEED_OP_DIFFUSION if op == "diffusion" else ceed.CEED_OP_MASS
    f = ceed.ceed_apply_diffusion if op == "diffusion" else ceed.ceed_apply_mass
    Q = p + 1 if qkind == "gll" else p + 2
    full = 8 * max(1, min(32, 256 // (Q * Q)))   # elements a cluster of 8 blocks of 256 threads holds
    for dims in ((1, 1, 1), (3, 2, 1), (full // 4, 2, 2), (full // 4 + 1, 2, 2)):
        m = synthetic.HexMesh(*[max(1, d) for d in dims], p, seed=p)
        mesh = gpu_mesh(ceed, m, qkind)
        qd = ceed.alloc_qdata(mesh, cop, prec)
        ceed.ceed_build_qdata(mesh, cop, ceed.CEED_COEFF_SINE, None, prec, qd)
        ceed.ceed_set_apply_variant(mesh, cop, prec, 1, stage)
        x = torch.from_numpy(synthetic.uniform(m.n_ldof * 9, seed=4)).cuda()
        for flags in (0, ceed.CEED_APPLY_DIRICHLET):
            y = torch.full_like(x, float("nan"))
            f(mesh, qd, prec, x, y, 9, flags)
            for col in (0, 8):
                x1 = x.reshape(-1, 9)[:, col].contiguous()
                y1 = torch.full_like(x1, float("nan"))
                f(mesh, qd, prec, x1, y1, 1, flags)
                assert torch.equal(y1, y.reshape(-1, 9)[:, col])
        ceed.ceed_mesh_status(mesh)
        mesh.close()
