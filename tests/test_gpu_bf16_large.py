"""The BF16 block-Jacobi product where the blocks exceed what the SMs should have in
flight at once (2,940 blocks of 420 rows, more elements than CTAs: each CTA takes
one or two): against the FP64 product of the exported BF16 values on the first,
last and the elements around the CTA count.  Bar 1e-5 of the largest entry: 420
FP32 products and sums of rounding 2^-24."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1812_04789_gb300 import binding as B
from paper_1812_04789_gb300 import build
from paper_1812_04789_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def test_bf16_apply_beyond_the_blocks_in_flight():
    build.build()
    B.load()
    cfg = wl.make_config("tgv", 3, (15, 14, 14), 6, M=0.1, Re=1600.0, dt_conv=0.05)
    m = B.Mesh.from_workload(wl.mesh_desc(cfg), wl.physics(cfg))
    W = torch.from_numpy(wl.perturbed_state(cfg, amp=0.02)).cuda()
    pmg = B.PMG(m, W, 1.5 / wl.time_step(cfg),
                B.pmg_opts((6,), cycle=B.CYCLE_BJ, precision=B.PREC_MIXED, storage=B.STORE_BF16))
    nb = m.m * m.nm
    X = torch.empty((m.E, nb, nb), dtype=torch.float32, device="cuda")
    pmg.export_blocks(0, B.BLOCKS_DIAG_INV, X)
    r = torch.from_numpy(wl.random_vector(tuple(W.shape), 3)).cuda()
    z = torch.empty_like(r)
    pmg.apply(r, z)
    assert m.status_sync() == B.DG_OK
    for e in (0, 151, 152, 2431, 2432, 2433, m.E - 1):
        ref = X[e].double() @ r.reshape(m.E, nb)[e].float().double()
        err = float((z.reshape(m.E, nb)[e] - ref).abs().max() / ref.abs().max())
        print("element %d: %.2e" % (e, err))
        assert err <= 1e-5
