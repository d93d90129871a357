"""lgf_plan_kernel_launches counts kernels, where lgf_plan_timings counts the
phases of a solve: a phase of the grouped levels 0 and 1, or of the
run-time-size transforms, is several kernels.  Expected values by hand."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1402_6081_gb300 as lgfm
import workloads as W
from paper_1402_6081_gb300 import build as lgf_build

pytestmark = pytest.mark.gpu

BLOCK = np.zeros((1, 3), dtype=np.int32)
CASES = [
    # one block, one level: forward, products, inverse
    (BLOCK, 8, 1, lgfm.LGF_FP32, {}, 3, 4),                      # products: z lines to images, products
    (BLOCK, 8, 1, lgfm.LGF_FP64, {}, 3, 4),                      # forward: planes, z lines
    (BLOCK, 8, 1, lgfm.LGF_FP64, {"interval_kernel": 1}, 3, 3),
    (BLOCK, 24, 1, lgfm.LGF_FP64, {"interval_kernel": 1}, 3, 7),   # an axis per launch, both ways
    # 128^3, level 2 beside: Reg, forward, products, inverse, Interp; levels
    # 0 and 1 in two bands of columns
    (W.full_box_blocks(8), 16, 3, lgfm.LGF_FP32, {}, 8, 1 + 2 * 2 + 1 + 5),
]


@pytest.mark.parametrize("blocks,n_b,levels,prec,opts,phases,kernels", CASES)
def test_kernels_of_a_solve(blocks, n_b, levels, prec, opts, phases, kernels):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lgf_build.build()
    dt = torch.float64 if prec == lgfm.LGF_FP64 else torch.float32
    s = lgfm.Solver(blocks, n_b, levels, 6, prec, **opts)
    assert lgfm.lgf_plan_kernel_launches(s.plan) == 0
    f = torch.ones((len(blocks), n_b, n_b, n_b), dtype=dt, device="cuda")
    for _ in range(2):
        s(f)
        assert lgfm.lgf_plan_timings(s.plan)[1] == phases
        assert lgfm.lgf_plan_kernel_launches(s.plan) == kernels
    lgfm.lgf_plan_sync(s.plan)
    s.close()
