"""The panel inverse held in registers (blocks of up to 512 rows beyond registers
and shared memory) at the sizes where it can go wrong: a last panel of a few
columns, rows not a multiple of the tile, odd rows in FP64 (scalar accesses),
more blocks than CTAs, and a block whose pivots are far from the diagonal
(rows of the coefficients permuted through a strongly advective state).  Bars of
the other inverse paths: |D^-1 D - I| <= 1e-10 in FP64, 2e-3 in FP32."""
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
    ("vortex", (3, 3), 8, "Q", B.PREC_MIXED, 2.0),      # 324 = 10 x 32 + 4
    ("vortex", (2, 3), 8, "Q", B.PREC_FP64, 2.0),       # 324 = 20 x 16 + 4
    ("vortex", (3, 2), 8, "P", B.PREC_FP64, 0.01),      # 180 = 11 x 16 + 4, small shift
    ("tgv", (6, 5, 6), 4, "P", B.PREC_FP64, 2.0),       # 175, 180 blocks
    ("tgv", (6, 6, 5), 5, "P", B.PREC_MIXED, 0.5),      # 280, 180 blocks
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
