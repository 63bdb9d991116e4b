"""The FP64 block probe against the general probe kernel (DG_PROBE_SIMT=1) at the
sizes where it can go wrong: blocks of fewer entries than threads, blocks of one
pass and of several (the last pass shorter), neighbour blocks that do not fit
the registers (the general kernel then runs), both dimensions, P_p and Q_p,
unequal directions.  Both sum the same products in FP64 in another order: at
most 600 points x 4 products of rounding 2^-53 against the largest entry, bar
1e-12 of the largest entry."""
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


@pytest.mark.parametrize("case,n,p,levels,space", [
    ("vortex", (3, 4), 0, (0,), "P"),
    ("vortex", (4, 2), 1, (1, 0), "P"),
    ("vortex", (3, 5), 6, (6, 3, 0), "P"),      # 12,544 entries
    ("vortex", (2, 3), 3, (3, 2, 1), "Q"),
    ("tgv", (2, 3, 4), 1, (1, 0), "P"),
    ("tgv", (3, 2, 2), 3, (3, 2, 1, 0), "P"),   # 10,000 entries: one pass
    ("tgv", (2, 2, 3), 4, (4, 2, 1, 0), "P"),   # three passes
    ("tgv", (2, 2, 2), 4, (4, 3, 1), "P"),      # neighbour blocks of 100 rows
    ("tgv", (2, 2, 2), 5, (5, 4, 0), "P"),      # neighbour blocks of 175 rows: the general kernel
    ("tgv", (2, 3, 2), 2, (2, 1, 0), "Q"),
])
def test_probe64_matches_general_kernel(case, n, p, levels, space, monkeypatch):
    cfg = wl.make_config(case, len(n), n, p, M=0.5 if len(n) == 2 else 0.1, Re=200.0, space=space)
    W = torch.from_numpy(wl.perturbed_state(cfg, amp=0.02)).cuda()
    m = B.Mesh.from_workload(wl.mesh_desc(cfg), wl.physics(cfg))
    out = []
    for simt in ("0", "1"):
        monkeypatch.setenv("DG_PROBE_SIMT", simt)
        opts = B.pmg_opts(levels, cycle=B.CYCLE_FMG if len(levels) > 1 else B.CYCLE_BJ)
        pmg = B.PMG(m, W, 1.5 / wl.time_step(cfg), opts)
        nb = m.m * m.nm
        D = torch.empty((m.E, nb, nb), dtype=torch.float64, device="cuda")
        pmg.export_blocks(0, B.BLOCKS_DIAG, D)
        got = [D.cpu().numpy()]
        if len(levels) > 1:
            nbc = m.m * wl.n_modes(levels[1], len(n), space)
            O = torch.empty((m.E, 2 * len(n), nbc, nbc), dtype=torch.float64, device="cuda")
            pmg.export_blocks(1, B.BLOCKS_NEIGHBOUR, O)
            got.append(O.cpu().numpy())
        assert m.status_sync() == B.DG_OK
        out.append(got)
        pmg.close()
    for a, b in zip(*out):
        err = float(np.abs(a - b).max() / np.abs(b).max())
        print("%s %s p=%d: %.2e" % (case, n, p, err))
        assert err <= 1e-12
