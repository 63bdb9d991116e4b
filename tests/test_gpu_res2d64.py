"""FP64 residual and Jacobian-vector product of 2-D structured meshes against the
oracle at the sizes where the kernels' splits can go wrong: one and two elements
in a direction (own neighbours), fewer faces than SMs, three warps of roles with
few points, points beyond one warp (a thread per point), a last CTA with fewer
faces, more modes than threads, p = 0; and meshes just past the lines to the
thread-per-point kernels (the JVP's first).  Bar 1e-12 of the largest entry: sums
of some hundred FP64 terms in another order."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import dg as odg
from paper_1812_04789_gb300 import binding as B
from paper_1812_04789_gb300 import build
from paper_1812_04789_gb300 import workloads as wl
from tests.helpers import oracle_mesh, oracle_physics

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    B.load()


@pytest.mark.parametrize("n,p,space", [
    ((1, 3), 2, "P"), ((2, 2), 0, "P"), ((16, 16), 2, "P"), ((9, 7), 8, "P"), ((33, 17), 1, "P"), ((23, 29), 3, "P"),
    ((5, 6), 4, "Q"), ((70, 49), 2, "P"),
])
def test_res2d64(n, p, space):
    cfg = wl.make_config("vortex", 2, n, p, M=0.5, Re=200.0, space=space)
    om, oph = oracle_mesh(cfg), oracle_physics(cfg)
    W = wl.perturbed_state(cfg, amp=0.05)
    v = wl.random_vector(W.shape, 11)
    m = B.Mesh.from_workload(wl.mesh_desc(cfg), wl.physics(cfg))
    Wd, vd = torch.from_numpy(W).cuda(), torch.from_numpy(v).cuda()
    R, J = torch.empty_like(Wd), torch.empty_like(Wd)
    m.residual(Wd, R)
    m.jvp(Wd, vd, J, 0.7)
    assert m.status_sync() == B.DG_OK
    for got, ref in ((R, odg.residual(om, oph, W)), (J, odg.jvp(om, oph, W, v, 0.7))):
        err = float(np.abs(got.cpu().numpy() - ref).max() / np.abs(ref).max())
        print("%s p=%d %s: %.2e" % (n, p, space, err))
        assert err <= 1e-12
