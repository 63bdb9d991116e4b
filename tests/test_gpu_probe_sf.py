"""The sum-factorised block probe of 3-D P_p meshes and its neighbour blocks at
every coarse order, every order of both precisions, FP32 with the primal traces cached and interpolated, on meshes with
unequal directions (two elements in one, whose neighbours coincide), against
the general FP64 probe kernel (DG_PROBE_SIMT=1).

Bars, relative to the largest entry: FP64 1e-12 (600 points x a few products of
rounding 2^-53, summed in another order); FP32 5e-6 (state, tables and point
derivatives rounded at 2^-24 = 6e-8, sums of a few hundred terms in three
directions whose volume and face parts nearly cancel: tens of roundings)."""
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


def _blocks(m, cfg, W, precision, pc):
    pmg = B.PMG(m, W, 1.5 / wl.time_step(cfg), B.pmg_opts((cfg["p"], pc), precision=precision, cycle=B.CYCLE_FMG))
    nb, nbc = m.m * m.nm, m.m * wl.n_modes(pc, 3, "P")
    dt = torch.float64 if precision == B.PREC_FP64 else torch.float32
    D = torch.empty((m.E, nb, nb), dtype=dt, device="cuda")
    O = torch.empty((m.E, 6, nbc, nbc), dtype=dt, device="cuda")
    pmg.export_blocks(0, B.BLOCKS_DIAG, D)
    pmg.export_blocks(1, B.BLOCKS_NEIGHBOUR, O)
    assert m.status_sync() == B.DG_OK
    pmg.close()
    return [x.cpu().numpy().astype(np.float64) for x in (D, O)]


@pytest.mark.parametrize("n", [(2, 3, 5), (4, 3, 2)])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6])
def test_probe_sf_matches_general_kernel(p, n, monkeypatch):
    cfg = wl.make_config("tgv", 3, n, p, M=0.1, Re=200.0)
    W = torch.from_numpy(wl.perturbed_state(cfg, amp=0.02)).cuda()
    m = B.Mesh.from_workload(wl.mesh_desc(cfg), wl.physics(cfg))
    monkeypatch.setenv("DG_PROBE_SIMT", "1")
    ref = [_blocks(m, cfg, W, B.PREC_FP64, pc) for pc in range(p)]
    monkeypatch.setenv("DG_PROBE_SIMT", "0")
    for what, precision, no_cache, bar in (("fp64", B.PREC_FP64, "0", 1e-12), ("fp32 cached", B.PREC_MIXED, "0", 5e-6),
                                           ("fp32 interpolated", B.PREC_MIXED, "1", 5e-6)):
        monkeypatch.setenv("DG_PMG_NO_PRIMAL_CACHE", no_cache)
        for pc in range(p):
            got = _blocks(m, cfg, W, precision, pc)
            err = [float(np.abs(a - b).max() / np.abs(b).max()) for a, b in zip(got, ref[pc])]
            print("p=%d pc=%d %s %s: %.2e %.2e" % (p, pc, n, what, *err))
            assert max(err) <= bar
