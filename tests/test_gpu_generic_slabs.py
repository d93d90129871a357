"""Levels >= 2 of the block sizes 20 to 30 that no other test takes through Reg,
Interp and the interval products: slabs of planes and bundles of columns with a
remainder for every n_I, sibling groups with few children present.  Four
levels over scattered blocks, against the oracle; tolerances as in
test_gpu_parity.py (relative L-infinity 1e-12 in FP64, 1e-5 in FP32)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1402_6081_gb300 as lgfm
from oracle import fmm
from paper_1402_6081_gb300 import build as lgf_build

pytestmark = pytest.mark.gpu

BLOCKS = np.array([[0, 0, 0], [1, 0, 0], [1, 1, 1], [3, 0, 1], [4, 6, 1], [5, 7, 2], [10, 2, 0], [11, 3, 9]], dtype=np.int32)


@pytest.mark.parametrize("n_b", [20, 22, 26, 28, 30])
def test_levels_above_one(n_b):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lgf_build.build()
    f = np.random.default_rng(n_b).random((len(BLOCKS), n_b, n_b, n_b))
    ref = fmm.fmm_solve(BLOCKS, f, n_b, 4, 8)
    for dt, prec, tol in ((torch.float64, lgfm.LGF_FP64, 1e-12), (torch.float32, lgfm.LGF_FP32, 1e-5)):
        s = lgfm.Solver(BLOCKS, n_b, 4, 8, prec)
        assert s.stats()["top_product_level"] >= 2
        u = s(torch.from_numpy(f).to(dt).cuda())
        lgfm.lgf_plan_sync(s.plan)
        err = fmm.rel_linf(u.double().cpu().numpy(), ref)
        s.close()
        assert err <= tol, (n_b, dt, err)
