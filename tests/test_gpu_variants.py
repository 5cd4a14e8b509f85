"""GPU test of the rule for the apply's launches: which variants a call runs, counted in a captured graph.

A variant that is set launches one kernel per colour; the default runs a mesh that fits one cluster in one launch; an
operator on the integer slices has no variants.  Boundaries of the cluster: 8 blocks of 128 threads in FP64, of 256 in
the other precisions, of one element in the slice kernels.
"""
import ctypes

import numpy as np
import pytest

import synthetic
from _util import gpu_mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _setup(ceed, p, qkind, op, prec, dims):
    cop = ceed.CEED_OP_DIFFUSION if op == "diffusion" else ceed.CEED_OP_MASS
    m = synthetic.HexMesh(*dims, p, seed=p)
    mesh = gpu_mesh(ceed, m, qkind)
    qd = ceed.alloc_qdata(mesh, cop, prec)
    ceed.ceed_build_qdata(mesh, cop, ceed.CEED_COEFF_SINE, None, prec, qd)
    f = ceed.ceed_apply_diffusion if op == "diffusion" else ceed.ceed_apply_mass
    return m, mesh, qd, cop, f


def _launches(call):
    """Nodes of the graph that a capture of the call gives."""
    call()                                # sets the kernels' attributes outside the capture
    torch.cuda.synchronize()
    path = next(line.split()[-1] for line in open("/proc/self/maps") if "libcudart" in line)
    rt = ctypes.CDLL(path)
    graph, n = ctypes.c_void_p(), ctypes.c_size_t()
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        h = ctypes.c_void_p(st.cuda_stream)
        assert rt.cudaStreamBeginCapture(h, 2) == 0      # relaxed
        call()
        assert rt.cudaStreamEndCapture(h, ctypes.byref(graph)) == 0
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    assert rt.cudaGraphDestroy(graph) == 0
    return n.value


@pytest.mark.parametrize("p,qkind,op,prec", [(2, "gauss", "mass", 0), (3, "gll", "diffusion", 1), (2, "gll", "diffusion", 5)])
def test_set_variants_launch_per_colour(p, qkind, op, prec):
    import paper_2109_05072_gb300 as ceed
    m, mesh, qd, cop, f = _setup(ceed, p, qkind, op, prec, (4, 4, 4))
    x = torch.from_numpy(synthetic.uniform(m.n_ldof, seed=1)).cuda()
    ys = []
    for ne, stage in ((0, 1), (1, 0), (1, 1), (2, 1)):
        ceed.ceed_set_apply_variant(mesh, cop, prec, ne, stage)
        y = torch.full_like(x, float("nan"))
        assert mesh.n_colors == 8 and _launches(lambda: f(mesh, qd, prec, x, y)) == (8 if ne else 1)
        ys.append(y)
    assert all(torch.equal(ys[0], y) for y in ys)
    mesh.close()


@pytest.mark.parametrize("p,qkind,op", [(7, "gll", "diffusion"), (5, "gauss", "mass")])
def test_slice_operators_have_one_kernel(p, qkind, op):
    import paper_2109_05072_gb300 as ceed
    m, mesh, qd, cop, f = _setup(ceed, p, qkind, op, 0, (6, 5, 4))
    x = torch.from_numpy(synthetic.uniform(m.n_ldof, seed=1)).cuda()
    y = torch.empty_like(x)
    for _ in range(8):
        ne, stage, ms = ceed.ceed_autotune_apply(mesh, cop, qd, 0, x, y)
        assert (ne, stage) == (1, 0) and ms > 0
    mesh.close()


@pytest.mark.parametrize("p,qkind,op,prec", [(5, "gll", "diffusion", 0), (6, "gll", "diffusion", 0), (7, "gll", "diffusion", 0),
                                             (5, "gauss", "mass", 0), (6, "gauss", "diffusion", 0), (2, "gll", "diffusion", 0),
                                             (3, "gauss", "mass", 0), (3, "gll", "diffusion", 1), (4, "gll", "diffusion", 5)])
def test_default_at_the_cluster_limit(p, qkind, op, prec):
    """One column (the cluster where the mesh fits) has the bits of nine (more than a cluster holds: per colour)."""
    import paper_2109_05072_gb300 as ceed
    Q = p + 1 if qkind == "gll" else p + 2
    slices = prec == 0 and Q >= 6
    full = 8 if slices else 8 * min(32, (128 if prec == 0 else 256) // (Q * Q))
    for dims in ((full - 1, 1, 1), (full // 2, 2, 1), (full + 1, 1, 1), (full // 4, 2, 2)):
        m, mesh, qd, cop, f = _setup(ceed, p, qkind, op, prec, dims)
        x = torch.from_numpy(synthetic.uniform(m.n_ldof * 9, seed=4)).cuda()
        x0 = x[: m.n_ldof].contiguous()
        y0 = torch.empty_like(x0)
        n = _launches(lambda: f(mesh, qd, prec, x0, y0))
        assert n == (1 if m.n_elem <= full else mesh.n_colors)
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


@pytest.mark.parametrize("prec", [0, 1, 5])
def test_copy_wait_expiry_of_the_colour_launches(prec):
    """Launches that overlap (each a dependent of the one before): copy waits that give up are reported, nothing of a given-up
    element is written, and the next apply is right.  100 elements: more than a cluster holds at p = 4."""
    import paper_2109_05072_gb300 as ceed
    m, mesh, qd, cop, f = _setup(ceed, 4, "gll", "diffusion", prec, (5, 5, 4))
    ceed.ceed_set_apply_variant(mesh, cop, prec, 1, 0)       # direct loads: no wait
    x = torch.from_numpy(synthetic.uniform(m.n_ldof, seed=2)).cuda()
    ref = torch.empty_like(x)
    f(mesh, qd, prec, x, ref)
    ceed.ceed_set_apply_variant(mesh, cop, prec, 2, 1)
    y = torch.zeros_like(x)
    ceed.ceed_set_wait_limits(0, -1)
    try:
        f(mesh, qd, prec, x, y)
        with pytest.raises(ceed.CeedError) as ei:
            ceed.ceed_mesh_status(mesh)
        assert ei.value.status == ceed.CEED_ERR_TIMEOUT
    finally:
        ceed.ceed_set_wait_limits(-1, -1)
    assert np.isfinite(y.cpu().numpy()).all()
    ceed.ceed_mesh_status(mesh)
    f(mesh, qd, prec, x, y)
    ceed.ceed_mesh_status(mesh)
    assert torch.equal(y, ref)
    mesh.close()


@pytest.mark.parametrize("p,qkind,op,prec,dims", [(2, "gauss", "mass", 0, (4, 4, 4)), (7, "gll", "diffusion", 0, (4, 4, 3)),
                                                  (3, "gll", "diffusion", 1, (8, 8, 6)), (3, "gll", "diffusion", 5, (8, 8, 6)),
                                                  (6, "gauss", "diffusion", 0, (2, 2, 2))])
def test_captured_applies_replay(p, qkind, op, prec, dims):
    """Cluster and overlapping launches in a captured graph: every replay gives the bits of the call."""
    import paper_2109_05072_gb300 as ceed
    m, mesh, qd, cop, f = _setup(ceed, p, qkind, op, prec, dims)
    x = torch.from_numpy(synthetic.uniform(m.n_ldof, seed=3)).cuda()
    ref, y, z = torch.empty_like(x), torch.empty_like(x), torch.empty_like(x)
    f(mesh, qd, prec, x, ref)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        f(mesh, qd, prec, x, y)
        f(mesh, qd, prec, y, z)
    for _ in range(3):
        y.fill_(float("nan"))
        z.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, ref)
        zz = torch.empty_like(x)
        f(mesh, qd, prec, y, zz)
        assert torch.equal(z, zz)
    mesh.close()
