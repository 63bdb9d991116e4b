"""The persistent smoother in FP64 (values as two words with an epoch each,
power-of-two scales, rotations behind the exchange) against the
launch-per-operation smoother at the sizes where it can go wrong: the last CTA
with fewer elements, few CTAs and more sums than lanes, one and two iterations
(no rotation behind an exchange), two elements in a direction, block columns
that are no multiple of a run, Q_p, triangles.

Bar 1e-11 relative max-norm: the FP32 comparison's 1e-4 times 2^-29 (the ratio of
the roundings) is 2e-13; the sums over the CTAs are plain FP64 here (152
roundings more at most)."""
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


@pytest.mark.parametrize("case,n,p,levels,nu,nuc,space", [
    ("vortex", (23, 17), 3, (3, 2, 1, 0), 10, 30, "P"),
    ("vortex", (5, 3), 2, (2, 1, 0), 6, 40, "P"),
    ("vortex", (64, 61), 2, (2, 0), 1, 1, "P"),
    ("vortex", (6, 7), 2, (2, 1), 2, 2, "Q"),
    ("tgv", (2, 4, 5), 2, (2, 1, 0), 8, 12, "P"),
    ("tgv", (7, 9, 8), 3, (3, 2, 1, 0), 10, 35, "P"),
    ("tri", (13, 11), 4, (4, 2, 1, 0), 10, 30, "P"),
])
def test_fp64_persistent_matches_launch_per_operation(case, n, p, levels, nu, nuc, space, monkeypatch):
    if case == "tri":
        cfg = wl.tri_config(n, p, dt_conv=0.05)
        W = torch.from_numpy(wl.tri_perturbed_state(cfg, amp=0.02)).cuda()
        m = B.Mesh.from_tri_workload(wl.tri_mesh(cfg), wl.tri_physics(cfg), p)
    else:
        cfg = wl.make_config(case, len(n), n, p, M=0.5 if len(n) == 2 else 0.1, Re=1000.0, dt_conv=0.05, space=space)
        W = torch.from_numpy(wl.perturbed_state(cfg, amp=0.02)).cuda()
        m = B.Mesh.from_workload(wl.mesh_desc(cfg), wl.physics(cfg))
    r = torch.from_numpy(wl.random_vector(W.shape, 7)).cuda()
    out = []
    for off in ("1", "0"):
        monkeypatch.setenv("DG_PMG_NO_COOP", off)
        pmg = B.PMG(m, W, 1.5 / wl.time_step(cfg), B.pmg_opts(levels, nu, nu, nuc, precision=B.PREC_FP64))
        z = torch.empty_like(r)
        for _ in range(2):
            pmg.apply(r, z)
        assert m.status_sync() == B.DG_OK
        out.append(z.cpu().numpy())
        pmg.close()
    err = float(np.abs(out[0] - out[1]).max() / np.abs(out[0]).max())
    print("%s %s p=%d %s: %.2e" % (case, n, p, space, err))
    assert err <= 1e-11
