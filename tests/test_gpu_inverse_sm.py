"""The inverse in shared memory by panels at the sizes where it can go wrong: the
smallest (40 rows: a last panel of 8 columns), two CTAs per SM and one, rows no
multiple of the 16-byte vector, a last panel that ends inside a vector (175 = 5 x
32 + 15), the first size of more than 128 rows, more blocks than CTAs, a small
shift.  Bars of the other inverse paths: |D^-1 D - I| <= 1e-10 in FP64, 2e-3 in FP32."""
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


@pytest.mark.parametrize("case,n,p,space,prec,sigma", [
    ("vortex", (18, 35), 3, "P", B.PREC_MIXED, 2.0),    # 40, 630 blocks
    ("vortex", (3, 4), 3, "P", B.PREC_FP64, 0.01),      # 40
    ("vortex", (5, 4), 5, "P", B.PREC_FP64, 2.0),       # 84 = 5 x 16 + 4
    ("tgv", (7, 6, 8), 3, "P", B.PREC_FP64, 0.5),       # 100, 336 blocks
    ("tgv", (7, 6, 8), 3, "P", B.PREC_MIXED, 0.5),
    ("tgv", (2, 3, 3), 2, "Q", B.PREC_FP64, 2.0),       # 135 = 8 x 16 + 7
    ("tgv", (2, 3, 3), 2, "Q", B.PREC_MIXED, 2.0),      # 135 = 4 x 32 + 7
    ("vortex", (3, 3), 5, "Q", B.PREC_FP64, 2.0),       # 144 = 9 x 16
    ("tgv", (6, 5, 6), 4, "P", B.PREC_MIXED, 0.5),      # 175
    ("vortex", (3, 2), 8, "P", B.PREC_MIXED, 0.01),     # 180 = 5 x 32 + 20
])
def test_inverse_times_block_is_identity(case, n, p, space, prec, sigma):
    cfg = wl.make_config(case, len(n), n, p, M=0.5 if len(n) == 2 else 0.2, Re=200.0, space=space)
    W = torch.from_numpy(wl.perturbed_state(cfg, amp=0.05)).cuda()
    m = B.Mesh.from_workload(wl.mesh_desc(cfg), wl.physics(cfg))
    pmg = B.PMG(m, W, sigma, B.pmg_opts((p,), cycle=B.CYCLE_BJ, precision=prec))
    nb = m.m * m.nm
    dt = torch.float64 if prec == B.PREC_FP64 else torch.float32
    D = torch.empty((m.E, nb, nb), dtype=dt, device="cuda")
    X = torch.empty_like(D)
    pmg.export_blocks(0, B.BLOCKS_DIAG, D)
    pmg.export_blocks(0, B.BLOCKS_DIAG_INV, X)
    assert m.status_sync() == B.DG_OK
    err = float((torch.bmm(X.double(), D.double()) - torch.eye(nb, dtype=torch.float64, device="cuda")).abs().max())
    print("%s %s p=%d %s: n_b %d, %.2e" % (case, n, p, space, nb, err))
    assert err <= (1e-10 if prec == B.PREC_FP64 else 2e-3)
