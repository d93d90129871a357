"""FP32 products of the grouped levels 0 and 1 in several bands of columns with a
shorter last one, for block sizes whose columns are taken 4, 2 and 1 at a time,
by one warp and by two, and whose second stage is odd; against the blocks' own
transforms (interval_kernel = 1), tolerance as in test_gpu_group.py.

A phase of b bands launches 2 b kernels and the planes 2, the blocks' own form 3
in all, so the launch counts of both plans tell b."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1402_6081_gb300 as lgfm
import workloads as W
from paper_1402_6081_gb300 import build as lgf_build

pytestmark = pytest.mark.gpu

# n_b, blocks per axis, values of a line's image (rows of n_b / 2 rounded up to
# pairs), columns of a band and of the last one
CASES = [
    (4, (28, 28, 28), 8 * 2, 96, 48),
    (6, (18, 18, 18), 8 * 4, 160, 152),
    (8, (16, 16, 16), 8 * 4, 288, 256),
    (10, (12, 12, 12), 8 * 6, 448, 392),
    (18, (8, 8, 6), 8 * 10, 1344, 1320),
    (22, (6, 6, 6), 8 * 12, 1984, 1976),
]


@pytest.mark.parametrize("n_b,nb,image,width,last", CASES)
def test_short_last_band(n_b, nb, image, width, last):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lgf_build.build()
    columns, groups = 4 * n_b * (2 * n_b + 1), int(np.prod([(k + 1) // 2 for k in nb]))
    assert columns == width + last and columns * (groups + 1) * image * 8 > 48 << 20
    blocks = W.full_box_blocks(*nb)
    f = torch.from_numpy(np.random.default_rng(n_b).uniform(0.0, 1.0, size=(len(blocks), n_b, n_b, n_b))).float().cuda()
    levels = max(2, int(np.ceil(np.log2(max(nb)))))
    u, kernels = [], []
    for opts in ({}, {"interval_kernel": 1}):
        s = lgfm.Solver(blocks, n_b, levels, min(n_b, 6), lgfm.LGF_FP32, **opts)
        u.append(s(f).double())
        lgfm.lgf_plan_sync(s.plan)
        kernels.append(lgfm.lgf_plan_kernel_launches(s.plan))
        s.close()
    assert float((u[0] - u[1]).abs().max()) <= 2e-5 * float(u[1].abs().max())
    if n_b < 18:   # (the run-time-size transforms launch more than one kernel each)
        assert kernels[0] - kernels[1] == 2 + 2 * 2 - 3
