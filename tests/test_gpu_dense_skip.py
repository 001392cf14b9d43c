"""The dense FP64 products skip zero entries: bit for bit the products without the
skip (the same sums over a matrix without a zero entry are unaffected, so the
reference is FP64 torch), with infinities, NaN, negative zeros, odd sizes and
unaligned views, where a zero times a non-finite value is NaN."""
import numpy as np
import pytest

from paper_2404_10928_gb300 import phantoms as ph

pytestmark = pytest.mark.gpu

# rounding of sums of up to 2^12 FP64 products, relative to the sum of magnitudes
SUM_TOL = 4096 * 2.0 ** -53


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_10928_gb300 import build
    build.build()
    return torch


@pytest.mark.parametrize("shape,K", [((32, 16), 100), ((33, 31), 129), ((9, 5), 7)])
def test_products_with_zero_entries(torch_cuda, shape, K):
    torch = torch_cuda
    from paper_2404_10928_gb300.api import Plan
    prob = ph.custom(2, shape, (1e-4, 1e-4), ph.ring_sensors(3, 4e-3), K, seed=95)
    gen = torch.Generator(device="cuda").manual_seed(K)
    with Plan.from_problem(prob) as plan:
        rows, cols = prob.n_sensors * K, prob.n_pixels
        m = torch.randn((rows, cols), generator=gen, device="cuda", dtype=torch.float64)
        keep = torch.rand((rows, cols), generator=gen, device="cuda") < 0.02
        for mat in (plan.dense_assemble(), torch.where(keep, m, torch.zeros_like(m)),
                    torch.where(keep, m, -torch.zeros_like(m)), m):
            for tr in (False, True):
                a = mat.T if tr else mat
                v = torch.randn(a.shape[1], generator=gen, device="cuda", dtype=torch.float64)
                out = plan.dense_matvec(mat, v, transpose=tr)
                bound = SUM_TOL * (a.abs() @ v.abs())
                assert ((out - a @ v).abs() <= bound).all()
                assert not torch.signbit(plan.dense_matvec(torch.zeros_like(mat), v, transpose=tr)).any()
                for bad in (float("inf"), float("nan")):
                    w = v.clone()
                    w[a.shape[1] // 2] = bad
                    got = plan.dense_matvec(mat, w, transpose=tr)
                    hit = a[:, a.shape[1] // 2]
                    # 0 * inf and anything times NaN are NaN; x * inf keeps its sign
                    nan = (hit == 0) | (bad != bad)
                    assert torch.isnan(got[nan]).all()
                    assert torch.equal(got[~nan], torch.sign(hit[~nan]) * bad)
        plan.sync_status()
