"""A preconditioner built at a state that is not physical (its Jacobian blocks
hold NaN) reports it and leaves the handle and the context usable, with every
smoother of the coarsest level; refreshed at a good state it is as good as new."""
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


BILU = dict(coarse=B.COARSE_BILU, order=B.ORDER_MDF)
BJ = dict(cycle=B.CYCLE_BJ)


@pytest.mark.parametrize("precision", [B.PREC_MIXED, B.PREC_FP64])
@pytest.mark.parametrize("case,n,p,levels,kw", [
    ("vortex", (5, 4), 2, (2, 0), BILU),      # blocks of 24 and 4 rows: inverses in registers
    ("vortex", (5, 4), 2, (2, 0), {}),
    ("tgv", (2, 4, 5), 1, (1, 0), BILU),      # 20 and 5
    ("vortex", (3, 4), 3, (3,), BJ),          # 40: shared memory
    ("tgv", (2, 2, 3), 4, (4,), BJ),          # 175: shared memory, panels on memory in FP64
    ("tgv", (2, 2, 2), 6, (6,), BJ),          # 420: panels on memory
    ("tgv", (2, 2, 1), 7, (7,), BJ),          # 600: panels in shared memory
], ids=["bilu24", "bj24", "bilu20", "40", "175", "420", "600"])
def test_blocks_of_an_unphysical_state(case, n, p, levels, kw, precision):
    cfg = wl.make_config(case, len(n), n, p, M=0.5, Re=300.0, dt_conv=0.3)
    W = torch.from_numpy(wl.perturbed_state(cfg, amp=0.02)).cuda()
    bad = W.clone()
    bad[1, -1, 0] = -bad[1, -1, 0].abs()           # negative energy: p < 0
    nan = W.clone()
    nan[0, 1, 0] = float("nan")
    m = B.Mesh.from_workload(wl.mesh_desc(cfg), wl.physics(cfg))
    sigma = 1.5 / wl.time_step(cfg)
    opts = B.pmg_opts(levels, 3, 3, 8, precision=precision, **kw)
    for X in (bad, nan):
        with pytest.raises(B.DGError) as err:
            B.PMG(m, X, sigma, opts)
        print(case, n, p, precision, err.value)
        assert m.status_sync() in (B.DG_ERR_BREAKDOWN, B.DG_ERR_NONPHYSICAL)
    pmg = B.PMG(m, W, sigma, opts)
    r = torch.from_numpy(wl.random_vector(tuple(W.shape), 3)).cuda()
    z0, z1 = torch.empty_like(r), torch.empty_like(r)
    pmg.apply(r, z0)
    assert m.status_sync() == B.DG_OK
    for X in (bad, nan):
        pmg.refresh(X, sigma)
        pmg.apply(r, z1)
        assert m.status_sync() != B.DG_OK
    pmg.refresh(W, sigma)
    pmg.apply(r, z1)
    assert m.status_sync() == B.DG_OK
    assert torch.equal(z0, z1)
