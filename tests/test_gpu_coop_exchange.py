"""The persistent smoother's one-reduction Gram-Schmidt and its exchanges at the
sizes where they can go wrong, against the launch-per-operation smoother
(Gram-Schmidt twice, a kernel per operation): the last CTA with fewer elements
than the others, one element per CTA, a CTA count below the number of sums
(sums shared out over few CTAs), more than 32 iterations (more sums than lanes
of the collecting warp), one iteration, a periodic direction of one element
(an element that is its own neighbour), blocks in shared memory and streamed.

Both smoothers minimise the same residual over the same Krylov space in FP32;
they differ by rounding carried through at most 40 iterations of a
well-conditioned preconditioned operator: the bar of the smoother's other
comparison, 1e-4 relative max-norm."""
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


@pytest.mark.parametrize("case,dim,n,p,levels,nu,nuc", [
    ("vortex", 2, (23, 17), 3, (3, 2, 1, 0), 10, 30),   # 391 elements: chunks of 3, the last of 1
    ("vortex", 2, (5, 3), 2, (2, 1, 0), 6, 40),         # 15 CTAs, 41 sums per exchange
    ("vortex", 2, (64, 61), 2, (2, 0), 1, 1),           # one iteration, 26 elements per CTA
    ("tgv", 3, (1, 4, 5), 2, (2, 1, 0), 8, 12),         # an element that is its own neighbour
    ("tgv", 3, (7, 9, 8), 3, (3, 2, 1, 0), 10, 35),     # 504 elements: chunks of 4, streamed and resident blocks
    ("tri", 2, (2, 2), 1, (1, 0), 4, 8),                # 8 triangles, three faces each
    ("tri", 2, (13, 11), 4, (4, 2, 1, 0), 10, 30),      # 286 triangles: chunks of 2
])
def test_exchange_matches_launch_per_operation(case, dim, n, p, levels, nu, nuc, monkeypatch):
    if case == "tri":
        cfg = wl.tri_config(n, p, dt_conv=0.05)
        W = torch.from_numpy(wl.tri_perturbed_state(cfg, amp=0.02)).cuda()
        m = B.Mesh.from_tri_workload(wl.tri_mesh(cfg), wl.tri_physics(cfg), p)
    else:
        cfg = wl.make_config(case, dim, n, p, M=0.5 if dim == 2 else 0.1, Re=1000.0, dt_conv=0.05)
        W = torch.from_numpy(wl.perturbed_state(cfg, amp=0.02)).cuda()
        m = B.Mesh.from_workload(wl.mesh_desc(cfg), wl.physics(cfg))
    r = torch.from_numpy(wl.random_vector(W.shape, 7)).cuda()
    out = []
    for off in ("1", "0"):
        monkeypatch.setenv("DG_PMG_NO_COOP", off)
        pmg = B.PMG(m, W, 1.5 / wl.time_step(cfg), B.pmg_opts(levels, nu, nu, nuc, precision=B.PREC_MIXED))
        z = torch.empty_like(r)
        for _ in range(2):          # the second application reuses the exchange buffers
            pmg.apply(r, z)
        assert m.status_sync() == B.DG_OK
        out.append(z.cpu().numpy())
        pmg.close()
    err = float(np.abs(out[0] - out[1]).max() / np.abs(out[0]).max())
    print("%s %s p=%d: %.2e" % (case, n, p, err))
    assert err <= 1e-4
