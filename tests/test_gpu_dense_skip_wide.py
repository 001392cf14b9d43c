"""The skipped rounds of the dense FP64 products, at widths where M x has such rounds
(four strides of 256 pairs of entries and more), with warps whose last round is not
whole: infinities and NaN in the vector, entries that are subnormal (the upper word
of the smallest is zero), and sums whose value shows every skipped or added term."""
import os
import re

import pytest

from paper_2404_10928_gb300 import phantoms as ph

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2404_10928_gb300", "csrc")


def test_no_vote_depends_on_convergence():
    """CUDA does not promise that a warp has converged again at a vote, so no vote
    takes its lanes from __activemask."""
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, name), encoding="utf-8") as f:
                assert not re.search(r"__activemask", f.read()), name


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_10928_gb300 import build
    build.build()
    return torch


# columns: two whole rounds of M x; one round and a part; rounds of some warps only
# (2 n = 1538 + 20); odd (the scalar loop); fewer columns than a warp in the last block
@pytest.mark.gpu
@pytest.mark.parametrize("shape,K", [((64, 64), 33), ((52, 50), 40), ((41, 38), 17), ((47, 45), 24),
                                     ((97, 16), 130)])
def test_wide_products_with_zero_rounds(torch_cuda, shape, K):
    torch = torch_cuda
    from paper_2404_10928_gb300.api import Plan
    prob = ph.custom(2, shape, (1e-4, 1e-4), ph.ring_sensors(3, 1.2e-2), K, seed=96)
    gen = torch.Generator(device="cuda").manual_seed(K)
    rows, cols = prob.n_sensors * K, prob.n_pixels

    def rand(*size):
        return torch.rand(size, generator=gen, device="cuda")

    # small whole numbers: every sum is exact in FP64, in any order
    m = torch.randint(-8, 9, (rows, cols), generator=gen, device="cuda").double()
    m[m == 0] = 1.0
    # one entry in 512 (rounds of a warp with none, one and more), and none in most rows
    sparse = torch.where(rand(rows, cols) < 1 / 512, m, torch.zeros_like(m))
    sparse[rand(rows) < 0.5] = 0.0
    with Plan.from_problem(prob) as plan:
        for mat in (sparse, -sparse, m, torch.where(sparse == 0, -torch.zeros_like(m), m)):
            for tr in (False, True):
                a = mat.T if tr else mat
                v = torch.randint(-99, 100, (a.shape[1],), generator=gen, device="cuda").double()
                assert torch.equal(plan.dense_matvec(mat, v, transpose=tr), a @ v)
                for bad in (float("inf"), -float("inf"), float("nan")):
                    for at in (0, a.shape[1] // 2 + 1, a.shape[1] - 1):
                        w = v.clone()
                        w[at] = bad
                        got = plan.dense_matvec(mat, w, transpose=tr)
                        hit = a[:, at]
                        # 0 * inf and anything times NaN are NaN; x * inf keeps its sign
                        nan = (hit == 0) | (bad != bad)
                        assert torch.isnan(got[nan]).all()
                        assert torch.equal(got[~nan], torch.sign(hit[~nan]) * bad)
        # the only entries are subnormals times 2^1000: exact whole multiples of 2^-74
        tiny = sparse * 2.0 ** -1074
        for tr in (False, True):
            a = sparse.T if tr else sparse
            v = torch.randint(-99, 100, (a.shape[1],), generator=gen, device="cuda").double()
            out = plan.dense_matvec(tiny, v * 2.0 ** 1000, transpose=tr)
            assert torch.equal(out, (a @ v) * 2.0 ** -74)
        plan.sync_status()
