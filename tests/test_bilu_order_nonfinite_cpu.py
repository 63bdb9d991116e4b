"""The MDF order of a block ILU(0) is a permutation whatever its weights hold: an
unphysical state, or one whose Jacobian leaves FP32, gives blocks and weights of
NaN and infinity, and the order indexes device memory afterwards.  Weights that
are not numbers count as infinite: such elements come last, in index order of
equal weights.  Run in a process of its own: an order that leaves elements out
reads and writes past its arrays."""
import os
import subprocess
import sys

from paper_1812_04789_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import sys
import numpy as np
sys.path.insert(0, %r)
from paper_1812_04789_gb300 import binding as B
from tests.test_bilu_order_cpu import face_nbr, pair_weights
B.load()
for n in ((5, 4), (4, 4, 2)):
    nbr = face_nbr(n)
    E = nbr.shape[0]
    cf, _ = pair_weights(nbr, np.random.default_rng(2))
    ref = B.bilu_order(nbr, B.ORDER_MDF, cf)[0]
    for what in ("nan", "inf", "one nan", "one inf", "nan and inf"):
        c = cf.copy()
        if what in ("nan", "inf"):
            c[c >= 0] = float(what)
        elif what == "nan and inf":
            c[: E // 2][c[: E // 2] >= 0] = np.nan
            c[E // 2:][c[E // 2:] >= 0] = np.inf
        else:
            c[E // 3][c[E // 3] >= 0] = float(what[4:])
        order, level, nl = B.bilu_order(nbr, B.ORDER_MDF, c)
        assert sorted(order) == list(range(E)), (n, what, order)
        assert level.min() == 0 and level.max() == nl - 1, (n, what, level)
        if what == "nan":
            assert list(order) == list(range(E)), (n, what, order)
    assert list(B.bilu_order(nbr, B.ORDER_MDF, cf)[0]) == list(ref)
print("ok")
"""


def test_mdf_order_of_nonfinite_weights_is_a_permutation():
    build.build()
    r = subprocess.run([sys.executable, "-c", SCRIPT % ROOT], capture_output=True, text=True, timeout=300, cwd=ROOT)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr[-2000:]
