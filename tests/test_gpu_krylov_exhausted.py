"""Krylov spaces that are used up (more iterations than unknowns), one-kernel
Arnoldi step and persistent smoother against the kernel per operation.

What is left of a new vector is then rounding, orthogonal to nothing, and its
norm must still be that of the vector: taken as the difference w.w - h.h of two
equal numbers it comes out as anything, or as zero, which a solve reports as a
residual of exactly zero.  The kernels per operation sum the norm over the
vector.  With tolerance zero neither solve converges (a remainder of 40 or more
entries does not round to zero in all of them), both use every iteration, and
the solution is the exact one to N eps times a condition number below 1e2:
1e-12.  The smoother's two paths agree to its usual bar (1e-4 in FP32, 1e-11 in
FP64)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1812_04789_gb300 import binding as B
from paper_1812_04789_gb300 import build
from paper_1812_04789_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    B.load()


def _mesh(case, n, p):
    cfg = wl.make_config(case, len(n), n, p, M=0.5 if len(n) == 2 else 0.1, Re=400.0, dt_conv=1.0)
    W = torch.from_numpy(wl.perturbed_state(cfg, amp=0.02)).cuda()
    return B.Mesh.from_workload(wl.mesh_desc(cfg), wl.physics(cfg)), W, 1.5 / wl.time_step(cfg)


@pytest.mark.parametrize("host", ["0", "1"])
@pytest.mark.parametrize("case,n,p,precision", [("vortex", (2, 2), 1, B.PREC_FP64),     # 48 unknowns, one CTA
                                                ("tgv", (2, 2, 2), 0, B.PREC_MIXED),    # 40
                                                ("vortex", (3, 5), 0, B.PREC_FP64)])    # 60
def test_arnoldi_of_an_exhausted_space(case, n, p, precision, host, monkeypatch):
    monkeypatch.setenv("DG_FGMRES_HOST", host)
    m, W, sigma = _mesh(case, n, p)
    b = torch.from_numpy(wl.random_vector(tuple(W.shape), 4)).cuda()
    out = []
    for off in ("1", "0"):
        monkeypatch.setenv("DG_PMG_NO_COOP", off)
        pmg = B.PMG(m, W, sigma, B.pmg_opts((p,), cycle=B.CYCLE_BJ, precision=precision, fgmres_restart=64))
        x, y = torch.empty_like(W), torch.empty_like(W)
        st = pmg.fgmres(W, b, x, restart=64, rtol=0.0, raise_on_error=False)
        m.jvp(W, x, y, sigma)
        assert m.status_sync() == B.DG_OK
        out.append((st["status"], st["iters"], float((y - b).norm() / b.norm())))
        pmg.close()
    print(case, n, p, out)
    assert out[0][:2] == (B.DG_ERR_NOT_CONVERGED, 64)
    assert out[1][:2] == out[0][:2]
    assert out[0][2] <= 1e-12 and out[1][2] <= 1e-12


@pytest.mark.parametrize("precision", [B.PREC_MIXED, B.PREC_FP64])
@pytest.mark.parametrize("case,n,p,levels,nuc", [("vortex", (2, 2), 2, (2, 1, 0), 64),    # 16 unknowns at p = 0
                                                 ("tgv", (2, 2, 2), 1, (1, 0), 64),       # 40
                                                 ("vortex", (3, 2), 2, (2, 0), 40)])      # 24
def test_smoother_of_an_exhausted_space(case, n, p, levels, nuc, precision, monkeypatch):
    m, W, sigma = _mesh(case, n, p)
    r = torch.from_numpy(wl.random_vector(tuple(W.shape), 7)).cuda()
    out = []
    for off in ("1", "0"):
        monkeypatch.setenv("DG_PMG_NO_COOP", off)
        pmg = B.PMG(m, W, sigma, B.pmg_opts(levels, 3, 3, nuc, precision=precision))
        z = torch.empty_like(r)
        pmg.apply(r, z)
        assert m.status_sync() == B.DG_OK
        out.append(z.cpu().numpy())
        pmg.close()
    err = float(np.abs(out[0] - out[1]).max() / np.abs(out[0]).max())
    print(case, n, p, precision, "%.2e" % err)
    assert err <= (1e-4 if precision == B.PREC_MIXED else 1e-11)
