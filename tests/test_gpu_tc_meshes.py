"""The tensor-core block probe and the shared-memory FP32 volume kernel on the
meshes that they serve, with more elements than CTAs (304 to 343 against 152 CTAs
of the probe; 512 against 3 x 152 slots of the volume kernel), so that TMEM
accumulators, mbarrier phases and slots are used again: 3-D P_p blocks of
a mesh with a direction of one element or another number of points, 3-D Q_p
(p + 2 points, P_p: the sum-factorised kernels, tests of their own).  Against the
FP64 oracle on elements around the CTA counts.

Bars relative to the largest entry, as reasoned in tests/test_gpu_probe_tc.py:
tensor-core diagonal blocks 1e-4 (three TF32 passes), neighbour blocks 1e-5, FP32
product 2e-5.  That the blocks come from another kernel than the general one
(DG_PROBE_SIMT=1) shows in their bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import blocks as oblocks
from oracle import dg as odg
from paper_1812_04789_gb300 import binding as B
from paper_1812_04789_gb300 import build
from paper_1812_04789_gb300 import workloads as wl
from tests.helpers import oracle_mesh, oracle_physics

pytestmark = pytest.mark.gpu
SIGMA = 2.5


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    B.load()


def _case(n, p, space, nq):
    cfg = wl.make_config("tgv", 3, n, p, M=0.1, Re=1600.0, space=space)
    om, oph = oracle_mesh(cfg, nq), oracle_physics(cfg)
    W = wl.perturbed_state(cfg, amp=0.05)
    return om, oph, W, B.Mesh.from_workload(wl.mesh_desc(cfg, nq), wl.physics(cfg))


def _rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


@pytest.mark.parametrize("n,p,space,nq,elems", [
    ((1, 18, 18), 4, "P", None, [0, 151, 152, 303, 304, 323]),
    ((1, 16, 19), 5, "P", None, [0, 152, 303]),
    ((1, 16, 19), 6, "P", None, [0, 303]),
    ((7, 7, 7), 2, "Q", None, [0, 151, 152, 304, 342]),
    ((6, 6, 9), 3, "Q", None, [0, 152, 323]),
    ((7, 7, 7), 4, "P", 7, [0, 151, 152, 304, 342]),
])
def test_tensor_core_diag_blocks(n, p, space, nq, elems, monkeypatch):
    om, oph, W, m = _case(n, p, space, nq)
    D = oblocks.diag_blocks(om, oph, W, SIGMA, elems=np.asarray(elems))
    out = []
    for simt in ("0", "1"):
        monkeypatch.setenv("DG_PROBE_SIMT", simt)
        pmg = B.PMG(m, torch.from_numpy(W).cuda(), SIGMA, B.pmg_opts((p,), cycle=B.CYCLE_BJ, precision=B.PREC_MIXED))
        Dg = torch.empty((om.E, om.nb, om.nb), dtype=torch.float32, device="cuda")
        pmg.export_blocks(0, B.BLOCKS_DIAG, Dg)
        assert m.status_sync() == B.DG_OK
        out.append(Dg[torch.as_tensor(elems, device="cuda")].cpu().numpy().astype(np.float64))
        pmg.close()
    err = _rel(out[0], D)
    print("%s %s%d nq %s: tensor-core blocks %.2e, general kernel %.2e" % (n, space, p, nq, err, _rel(out[1], D)))
    assert not np.array_equal(out[0], out[1])
    assert err <= 1e-4


def test_sum_factorised_blocks_across_elements(monkeypatch):
    """The mesh of tests/test_gpu_persistent_sizes.py whose blocks now come from the
    sum-factorised probe, at that kernel's FP32 bar (5e-6, tests/test_gpu_probe_sf.py)."""
    monkeypatch.delenv("DG_PROBE_SIMT", raising=False)
    elems = np.array([0, 151, 152, 303, 304, 455, 456, 511])
    om, oph, W, m = _case((8, 8, 8), 4, "P", None)
    D = oblocks.diag_blocks(om, oph, W, SIGMA, elems=elems)
    pmg = B.PMG(m, torch.from_numpy(W).cuda(), SIGMA, B.pmg_opts((4,), cycle=B.CYCLE_BJ, precision=B.PREC_MIXED))
    Dg = torch.empty((om.E, om.nb, om.nb), dtype=torch.float32, device="cuda")
    pmg.export_blocks(0, B.BLOCKS_DIAG, Dg)
    assert m.status_sync() == B.DG_OK
    err = _rel(Dg[torch.from_numpy(elems).cuda()].cpu().numpy().astype(np.float64), D)
    print("8^3 p = 4: sum-factorised blocks %.2e" % err)
    assert err <= 5e-6


@pytest.mark.parametrize("n,p,space,nq,pc,elems", [
    ((7, 7, 7), 2, "Q", None, 1, [0, 151, 152, 304, 342]),
    ((7, 7, 7), 4, "P", 7, 2, [0, 152, 342]),
])
def test_neighbour_blocks(n, p, space, nq, pc, elems, monkeypatch):
    monkeypatch.delenv("DG_PROBE_SIMT", raising=False)
    om, oph, W, m = _case(n, p, space, nq)
    nbc = om.m * wl.n_modes(pc, 3, space)
    O = oblocks.offdiag_blocks(om, oph, W, pc, elems=np.asarray(elems)).reshape(len(elems), 6, nbc, nbc)
    pmg = B.PMG(m, torch.from_numpy(W).cuda(), SIGMA,
                B.pmg_opts((p, pc), nu_pre=2, nu_post=2, nu_coarse=4, precision=B.PREC_MIXED))
    Og = torch.empty((om.E, 6, nbc, nbc), dtype=torch.float32, device="cuda")
    pmg.export_blocks(1, B.BLOCKS_NEIGHBOUR, Og)
    assert m.status_sync() == B.DG_OK
    err = _rel(Og[torch.as_tensor(elems, device="cuda")].cpu().numpy().astype(np.float64), O)
    print("%s %s%d nq %s: neighbour blocks %.2e" % (n, space, p, nq, err))
    assert err <= 1e-5


@pytest.mark.parametrize("cached", [True, False])
def test_fp32_product_of_another_number_of_points(cached, monkeypatch):
    monkeypatch.setenv("DG_PMG_NO_PRIMAL_CACHE", "0" if cached else "1")
    elems = np.array([0, 151, 152, 455, 456, 457, 511])
    om, oph, W, m = _case((8, 8, 8), 3, "P", 6)
    pmg = B.PMG(m, torch.from_numpy(W).cuda(), SIGMA,
                B.pmg_opts((3, 1), nu_pre=2, nu_post=2, nu_coarse=4, precision=B.PREC_MIXED))
    v = wl.random_vector(W.shape, 21)
    y = torch.empty_like(torch.from_numpy(v)).cuda()
    pmg.operator(0, torch.from_numpy(v).cuda(), y)
    assert m.status_sync() == B.DG_OK
    err = _rel(y.cpu().numpy()[elems], odg.jvp(om, oph, W, v, SIGMA, elems=elems))
    print("8^3 p = 3, 6 points, cached=%s: FP32 product %.2e" % (cached, err))
    assert err <= 2e-5
