"""The one-kernel Arnoldi step against the kernel per operation (DG_PMG_NO_COOP=1)
inside FGMRES with block Jacobi, at the sizes where it can go wrong: fewer
vectors' entries than threads of one CTA, few CTAs and more sums than CTAs or
warps (restart 60), groups of threads per row and four rows per thread, more
than 32 rotations, a restart in the middle, one iteration, FP64 and mixed.

The two solve the same least-squares problems over the same Krylov spaces in
FP64; the residual norms and the number of iterations agree (one iteration of
slack where the norm meets the tolerance), the solutions to the tolerance 1e-9 of
both, times ten for the condition of the preconditioned operator."""
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


@pytest.mark.parametrize("case,n,p,precision,kw,dt", [
    ("vortex", (2, 2), 1, B.PREC_FP64, dict(restart=10, max_restarts=4), 0.02),      # 48 unknowns: one CTA
    ("vortex", (5, 7), 2, B.PREC_FP64, dict(restart=60), 1.0),                      # 4 CTAs, 61 sums
    ("vortex", (5, 7), 2, B.PREC_MIXED, dict(restart=7, max_restarts=20), 0.02),
    ("tgv", (5, 4, 6), 3, B.PREC_FP64, dict(restart=40, max_restarts=4), 0.02),      # 79 entries per CTA
    ("tgv", (12, 12, 12), 3, B.PREC_FP64, dict(restart=30, max_restarts=4), 0.02),   # 1,137: four rows per thread
    ("tgv", (5, 4, 6), 2, B.PREC_FP64, dict(restart=1, max_restarts=30), 0.02),
])
def test_arnoldi_matches_kernel_per_operation(case, n, p, precision, kw, dt, monkeypatch):
    cfg = wl.make_config(case, len(n), n, p, M=0.5 if len(n) == 2 else 0.1, Re=400.0, dt_conv=dt)
    m = B.Mesh.from_workload(wl.mesh_desc(cfg), wl.physics(cfg))
    W = torch.from_numpy(wl.perturbed_state(cfg, amp=0.05)).cuda()
    b = torch.from_numpy(wl.random_vector(tuple(W.shape), 4)).cuda()
    out = []
    for off in ("1", "0"):
        monkeypatch.setenv("DG_PMG_NO_COOP", off)
        pmg = B.PMG(m, W, 1.5 / wl.time_step(cfg),
                    B.pmg_opts((p,), cycle=B.CYCLE_BJ, precision=precision, fgmres_restart=kw["restart"]))
        x = torch.empty_like(W)
        st = pmg.fgmres(W, b, x, rtol=1e-9, raise_on_error=False, **kw)
        out.append((st, x.cpu().numpy()))
        pmg.close()
    (s0, x0), (s1, x1) = out
    err = float(np.abs(x0 - x1).max() / np.abs(x0).max())
    print("%s %s p=%d %s: %d / %d iterations, %.2e" % (case, n, p, kw, s0["iters"], s1["iters"], err))
    assert s0["status"] == s1["status"]
    assert abs(s0["iters"] - s1["iters"]) <= 1
    assert err <= 1e-8
