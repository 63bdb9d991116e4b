"""The FP32 product's kernels for 3-D P_p meshes (one instance per p, several
elements and faces per CTA) against the direct kernels (DG_NO_SUMFACT_FACE=1,
DG_NO_SUMFACT_P=1): every p they serve, element and face counts that leave the
last CTA partly empty, a direction of one element, with the state's traces
interpolated (the FP32 product mode) and cached (the preconditioner's fine-level
operator); p = 7 and p + 3 points stay with the direct kernels.  Both round in
FP32: bar 2e-5 relative max-norm, the FP32 mode's parity bar."""
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


@pytest.mark.parametrize("n,p,nq", [((3, 5, 1), 1, 0), ((2, 3, 3), 2, 0), ((4, 2, 3), 3, 0), ((3, 3, 2), 4, 0),
                                    ((1, 1, 1), 4, 0), ((2, 3, 1), 5, 0), ((3, 1, 1), 6, 0), ((2, 1, 2), 7, 0),
                                    ((2, 2, 3), 3, 6)])
def test_fp32_product_matches_direct_kernels(n, p, nq, monkeypatch):
    cfg = wl.make_config("tgv", 3, n, p, M=0.2, Re=200.0)
    W = torch.from_numpy(wl.perturbed_state(cfg, amp=0.05)).cuda()
    v = torch.from_numpy(wl.random_vector(W.shape, 12)).cuda()
    m = B.Mesh.from_workload(wl.mesh_desc(cfg, nq1d=nq or None), wl.physics(cfg))
    pmg = B.PMG(m, W, 3.0, B.pmg_opts((p, 0), 2, 2, 2, precision=B.PREC_MIXED))
    out = []
    for direct in (False, True):
        for name in ("DG_NO_SUMFACT_FACE", "DG_NO_SUMFACT_P"):
            monkeypatch.setenv(name, "1" if direct else "0")
        a, b = torch.empty_like(W), torch.empty_like(W)
        m.jvp(W, v, a, 3.0, mode=B.JVP_EXACT_FP32)
        pmg.operator(0, v, b)
        assert m.status_sync() == B.DG_OK
        out += [a.cpu().numpy(), b.cpu().numpy()]
    ref = np.abs(out[2]).max()
    for x, y in ((0, 2), (1, 3), (0, 1)):
        err = float(np.abs(out[x] - out[y]).max() / ref)
        print("%s p=%d: %.2e" % (n, p, err))
        assert err <= 2e-5
