"""The frequency-domain operators from one end of FP32's range to the other: the
tensor-core kernels scale their FP16 operands by powers of two, which must reach
every image and spectrum whose result is finite."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2404_10928_gb300 import phantoms as ph

from helpers import f32, rel_l2

pytestmark = pytest.mark.gpu

# the FP32 phase error bound of tests/test_gpu_freq.py (1.1e-5 rad at the same
# f |pixel - tile centre| / c as here), times ten; the scales are powers of two,
# and what becomes subnormal is below 2^-24 of the largest values
FREQ_TOL = 1e-4


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_10928_gb300 import build
    build.build()
    return torch


def _problem(unit):
    """70 x 33 pixels; unit = 1: 0.1 mm and 40 MHz, larger units stretch lengths and
    times alike (the same phases at frequencies divided by unit)."""
    sens = np.concatenate([ph.ring_sensors(8, 6e-3), [[0.213e-3, -0.547e-3]]]) * unit
    return ph.custom(2, (70, 33), (1e-4 * unit, 1e-4 * unit), sens, 64, seed=61, fs=40e6 / unit)


# unit, exponents of the image's and of the spectrum's scale.  Stretched by 2^21,
# frequencies reach 9.5 Hz and distances 20 km, so terms near the top of the range
# (an image of 2^125 over d, spectra of 2^119 times c k_n) still have finite sums.
CASES = [(1, -122, -122), (1, 60, 60), (2 ** 21, 0, 0), (2 ** 21, -105, -118), (2 ** 21, 125, 119)]


@pytest.mark.parametrize("unit,ex,ep", CASES)
def test_freq_over_the_range_of_fp32(torch_cuda, unit, ex, ep):
    torch = torch_cuda
    from paper_2404_10928_gb300.api import Plan
    prob = _problem(unit)
    geo = orc.Geometry.of(prob)
    q, df = 96, 20e6 / 96 / unit
    rng = np.random.default_rng(q)
    x = f32(prob.x_true)
    pq = rng.standard_normal((prob.n_sensors, q)) + 1j * rng.standard_normal((prob.n_sensors, q))
    pq = pq.astype(np.complex64).astype(np.complex128)
    with Plan.from_problem(prob) as plan:
        xt = torch.tensor(x * 2.0 ** ex, dtype=torch.float32, device="cuda")
        pt = torch.tensor(pq * 2.0 ** ep, dtype=torch.complex64, device="cuda")
        p = plan.freq_forward(xt, q, df, df).cpu().numpy().astype(np.complex128)
        g = plan.freq_adjoint(pt, q, df, df).cpu().numpy().astype(np.float64)
        plan.sync_status()
    assert rel_l2(p * 2.0 ** -ex, orc.freq_forward(geo, x, q, df, df)) <= FREQ_TOL
    assert rel_l2(g * 2.0 ** -ep, orc.freq_adjoint(geo, pq, q, df, df)) <= FREQ_TOL


def _coherent_problem():
    # a positive image: the terms of a sum at low frequencies all have one sign
    prob = ph.custom(2, (96, 75), (1e-4, 1e-4), ph.ring_sensors(8, 8e-3), 64, seed=63)
    prob.x_true = 1.0 + 0.1 * prob.x_true
    return prob


def _coherent_tol(f):
    """FP32 phases 2 pi s 2^-24 (s = cycles from a tile's centre to its corner, 1.46
    us of travel), plus in units of 2^-24: two sines within 1.5e-7 (5), operands as
    pairs of 22 bits (4), and the FP32 sums (3)."""
    return (2.0 * np.pi * 1.46e-6 * f + 12.0) * 2.0 ** -24


@pytest.mark.parametrize("q", [100, 200])
@pytest.mark.parametrize("fmax", [0.1e6, 0.7e6, 1.6e6, 1.8e6, 20e6])
def test_forward_of_like_terms_has_the_error_of_fp32(torch_cuda, q, fmax):
    torch = torch_cuda
    from paper_2404_10928_gb300.api import Plan
    prob = _coherent_problem()
    geo = orc.Geometry.of(prob)
    df = fmax / q
    x = f32(prob.x_true)
    with Plan.from_problem(prob) as plan:
        p = plan.freq_forward(torch.tensor(x, dtype=torch.float32, device="cuda"), q, df, df)
        p = p.cpu().numpy()
        plan.sync_status()
    ref = orc.freq_forward(geo, x, q, df, df)
    # the spectra up to 0.5 MHz (0.7 cycles, where a tile's sum does not cancel)
    low = [n for n in range(q) if (n + 1) * df <= 0.5e6]
    assert low
    for n in low[:3] + low[-3:]:
        err = rel_l2(p[:, n], ref[:, n])
        assert err <= _coherent_tol((n + 1) * df), (n, err)


@pytest.mark.parametrize("span", [2.0 ** 16, 2.0 ** 20, 2.0 ** 24, 2.0 ** 28])
def test_phases_of_many_cycles_keep_the_modulus(torch_cuda, span):
    """With more cycles across a tile than FP32 resolves, the phases carry no
    information, but every term keeps its modulus: |P| <= c k sum |x| / d."""
    torch = torch_cuda
    from paper_2404_10928_gb300.api import Plan
    prob = _problem(1)
    q = 200
    df = span / 1.5e-6 / q
    rng = np.random.default_rng(q)
    x = f32(prob.x_true)
    pq = (rng.standard_normal((9, q)) + 1j * rng.standard_normal((9, q))).astype(np.complex64)
    with Plan.from_problem(prob) as plan:
        p = plan.freq_forward(torch.tensor(x, dtype=torch.float32, device="cuda"), q, df, df)
        g = plan.freq_adjoint(torch.tensor(pq, device="cuda"), q, df, df)
        p, g = p.cpu().numpy(), g.cpu().numpy()
        plan.sync_status()
    o = np.asarray(prob.origin[:2])
    pix = np.stack(np.meshgrid(np.arange(70) * 1e-4 + o[0], np.arange(33) * 1e-4 + o[1]), -1)
    inv_d = 1.0 / np.linalg.norm(pix.reshape(-1, 1, 2) - prob.sensors[None], axis=2)  # [N][S]
    ck = 2.0 * np.pi * df * (1 + np.arange(q))
    # FP32 factors: moduli within 32 recurrence steps of 2^-22, rounded up
    assert (np.abs(p) <= 1.001 * (x @ inv_d)[:, None] * ck).all()
    assert (np.abs(g) <= 1.001 * (inv_d @ (np.abs(pq) @ ck))).all()
