"""A solve in which a bounded device wait runs out says so.  A test hook makes
the exchanges of the persistent smoother, or those of the one-kernel Arnoldi
step, wait for a CTA that does not exist; the wait ends after its bound and the
kernels return without their outputs.  The solve must then return
DG_ERR_TIMEOUT (not "not converged", which callers go on with) and add nothing:
dW = 0, and an ESDIRK step leaves Wout at the state it started from.  The status
word keeps the timeout until it is read, and a handle without the hook then
solves as usual."""
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


def _mesh(case):
    if case == "tri":
        cfg = wl.tri_config((4, 3), 2, dt_conv=0.05)
        W = torch.from_numpy(wl.tri_perturbed_state(cfg, amp=0.02)).cuda()
        return cfg, B.Mesh.from_tri_workload(wl.tri_mesh(cfg), wl.tri_physics(cfg), 2), W
    n = (5, 7) if case == "vortex" else (4, 3, 5)
    cfg = wl.make_config(case, len(n), n, 2, M=0.3, Re=400.0, dt_conv=0.05)
    W = torch.from_numpy(wl.perturbed_state(cfg, amp=0.02)).cuda()
    return cfg, B.Mesh.from_workload(wl.mesh_desc(cfg), wl.physics(cfg)), W


def _opts(hook, precision):
    if hook == "DG_TEST_ARNOLDI_EXTRA":     # no smoother: the outer solve's own waits
        return B.pmg_opts((2,), cycle=B.CYCLE_BJ, precision=precision)
    return B.pmg_opts((2, 1, 0), 3, 3, 5, precision=precision)


@pytest.mark.parametrize("hook", ["DG_TEST_COOP_BARRIER_EXTRA", "DG_TEST_ARNOLDI_EXTRA"])
@pytest.mark.parametrize("case,precision,host", [("tgv", B.PREC_MIXED, "0"), ("tgv", B.PREC_FP64, "0"),
                                                 ("vortex", B.PREC_FP64, "1"), ("tri", B.PREC_MIXED, "0")])
def test_run_out_wait_ends_the_solve(case, precision, host, hook, monkeypatch):
    monkeypatch.setenv("DG_FGMRES_HOST", host)
    cfg, m, W = _mesh(case)
    b = torch.from_numpy(wl.random_vector(tuple(W.shape), 4)).cuda()
    sigma = 1.5 / wl.time_step(cfg)
    monkeypatch.setenv(hook, "1")
    pmg = B.PMG(m, W, sigma, _opts(hook, precision))
    monkeypatch.delenv(hook)
    for again in range(2):      # the second call finds the status word set
        dW = torch.full_like(W, 3.0)
        st = pmg.fgmres(W, b, dW, rtol=1e-14, max_restarts=2, raise_on_error=False)
        print(case, precision, hook, {k: st[k] for k in ("iters", "status")})
        assert st["status"] == B.DG_ERR_TIMEOUT
        assert not dW.any()
        assert st["iters"] <= 1 - again or host == "1" or case == "tri"
    assert m.status_sync() == B.DG_ERR_TIMEOUT
    Wout = torch.empty_like(W)
    st = pmg.esdirk3_step(W, wl.time_step(cfg), Wout, raise_on_error=False)
    assert st["status"] == B.DG_ERR_TIMEOUT
    assert torch.equal(Wout, W)
    assert m.status_sync() == B.DG_ERR_TIMEOUT
    pmg.close()
    pmg = B.PMG(m, W, sigma, _opts(hook, precision))
    dW = torch.empty_like(W)
    assert pmg.fgmres(W, b, dW, rtol=1e-8, max_restarts=4)["status"] == B.DG_OK
    assert m.status_sync() == B.DG_OK


@pytest.mark.parametrize("host", ["0", "1"])
@pytest.mark.parametrize("case", ["tgv", "vortex"])
def test_timeout_of_another_handle_wins_over_not_converged(case, host, monkeypatch):
    """A handle that has solved before holds a residual and Hessenberg columns of
    that solve; with the mesh's status word showing a timeout its Arnoldi step
    writes nothing, and they must not be taken for this solve's."""
    monkeypatch.setenv("DG_FGMRES_HOST", host)
    cfg, m, W = _mesh(case)
    b = torch.from_numpy(wl.random_vector(tuple(W.shape), 4)).cuda()
    sigma = 0.05 / wl.time_step(cfg)
    good = B.PMG(m, W, sigma, B.pmg_opts((2,), cycle=B.CYCLE_BJ, precision=B.PREC_FP64, fgmres_restart=5))
    dW = torch.empty_like(W)
    st = good.fgmres(W, b, dW, restart=5, rtol=1e-14, raise_on_error=False)
    assert st["status"] == B.DG_ERR_NOT_CONVERGED
    monkeypatch.setenv("DG_TEST_COOP_BARRIER_EXTRA", "1")
    hooked = B.PMG(m, W, sigma, B.pmg_opts((2, 1, 0), 3, 3, 5, precision=B.PREC_MIXED))
    monkeypatch.delenv("DG_TEST_COOP_BARRIER_EXTRA")
    z = torch.empty_like(W)
    hooked.apply(b, z)
    st = good.fgmres(W, b, dW, restart=5, rtol=1e-14, raise_on_error=False)
    assert st["status"] == B.DG_ERR_TIMEOUT
    assert not dW.any()
    assert m.status_sync() == B.DG_ERR_TIMEOUT
    st = good.fgmres(W, b, dW, restart=5, rtol=1e-14, raise_on_error=False)
    assert st["status"] == B.DG_ERR_NOT_CONVERGED and dW.any()
