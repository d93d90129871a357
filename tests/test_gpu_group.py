"""The grouped form of the merged levels 0 and 1 (the default): a sibling
group's 2 n_b cube transformed at once instead of its eight blocks, against the
blocks' own transforms (interval_kernel = 1) on the same plan arguments.

Both compute the same sums, so they differ by rounding only.  Bound: each is
within the precision's contract of the exact method (1e-12 / 1e-5 relative
L-infinity for non-negative sources, the bounds of test_gpu_parity.py), so the
two are within twice that of one another.  The domains are where the tables can
go wrong: a lone block, groups with absent children, absent neighbours inside a
row of four, isolated groups, negative and odd indices, one set of 2^3 groups
and several, and enough groups for more than one band of columns."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1402_6081_gb300 as lgfm
import workloads as W
from paper_1402_6081_gb300 import build as lgf_build

pytestmark = pytest.mark.gpu

SIZES = list(range(4, 33, 2))


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lgf_build.build()
    lgfm.library()


def solve(blocks, n_b, levels, prec, f, **opts):
    dt = torch.float64 if prec == lgfm.LGF_FP64 else torch.float32
    s = lgfm.Solver(blocks, n_b, levels, min(n_b, 6), prec, **opts)
    u = s(torch.from_numpy(f).to(dt).cuda())
    lgfm.lgf_plan_sync(s.plan)
    out = u.double().cpu().numpy()
    s.close()
    return out


def domains(n_b):
    rng = np.random.default_rng(n_b)
    box = W.full_box_blocks(7, 5, 6)
    yield np.array([[-3, 5, 2]]), 1
    yield np.array([[1, 1, 1], [2, 2, 2]]), 1                    # two groups, opposite children
    yield box[rng.uniform(size=len(box)) < 0.35] - [3, 4, 1], 4  # sparse, negative indices
    yield np.array([[0, 0, 0], [1, 0, 0], [9, 0, 3], [9, 9, 9], [4, 4, 4]]), 4


@pytest.mark.parametrize("prec,tol", [(lgfm.LGF_FP32, 2e-5), (lgfm.LGF_FP64, 2e-12)])
@pytest.mark.parametrize("n_b", SIZES)
def test_grouped_against_block_transforms(n_b, prec, tol):
    rng = np.random.default_rng(100 + n_b)
    for blocks, levels in domains(n_b):
        f = rng.uniform(0.0, 1.0, size=(len(blocks), n_b, n_b, n_b))
        u = solve(blocks, n_b, levels, prec, f)
        ref = solve(blocks, n_b, levels, prec, f, interval_kernel=1)
        assert np.abs(u - ref).max() <= tol * np.abs(ref).max(), len(blocks)


@pytest.mark.parametrize("prec,tol", [(lgfm.LGF_FP32, 2e-5), (lgfm.LGF_FP64, 2e-12)])
def test_grouped_several_bands(prec, tol):
    # 2197 blocks of 4^3 and 343 groups; 16^3: several bands of columns in FP32
    for n_b, nb in ((4, 13), (16, 9)):
        blocks = W.full_box_blocks(nb)
        f = np.random.default_rng(7).uniform(0.0, 1.0, size=(len(blocks), n_b, n_b, n_b))
        u = solve(blocks, n_b, 4, prec, f)
        ref = solve(blocks, n_b, 4, prec, f, interval_kernel=1)
        assert np.abs(u - ref).max() <= tol * np.abs(ref).max(), n_b
