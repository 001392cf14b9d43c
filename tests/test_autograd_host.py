"""Host side of the autograd functions, on the CPU with a small stand-in plan (a
dense matrix per speed of sound): what they accept as the speed of sound."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2404_10928_gb300 import autograd  # noqa: E402


class DensePlan:
    """The frame entry points of a plan that the autograd functions call."""

    n_pixels, n_sensors, n_samples = 6, 2, 5

    def __init__(self):
        gen = torch.Generator().manual_seed(3)
        self.base = torch.rand((self.n_sensors * self.n_samples, self.n_pixels), generator=gen)
        self.c = 1500.0

    def set_sound_speed(self, c):
        assert isinstance(c, float)
        self.c = c

    @property
    def a(self):
        return self.base * (1500.0 / self.c)

    def forward_frames(self, x):
        return (x @ self.a.T).reshape(-1, self.n_sensors, self.n_samples)

    def adjoint_frames(self, r):
        return r.reshape(-1, self.n_sensors * self.n_samples) @ self.a

    def landweber_step_frames(self, x, y, omega, nonneg):
        z = x + omega * self.adjoint_frames(y - self.forward_frames(x))
        return z.clamp_min(0.0) if nonneg else z


@pytest.mark.parametrize("c", [1520.0, np.float64(1520.0), np.float32(1520.0), 1520,
                               torch.tensor(1520.0), torch.tensor([1520.0])])
def test_speed_of_sound_as_a_number(c):
    plan = DensePlan()
    x = torch.rand((1, plan.n_pixels))
    y = torch.rand((1, plan.n_sensors, plan.n_samples))
    p = autograd.ForwardOp.apply(x, c, plan)
    assert plan.c == 1520.0
    assert torch.equal(p.reshape(1, -1), x @ plan.a.T)
    assert torch.equal(autograd.AdjointOp.apply(y, c, plan).reshape(1, -1), plan.adjoint_frames(y))
    step = autograd.LandweberStep.apply(x, y, c, plan, 0.1, True)
    assert torch.equal(step, plan.landweber_step_frames(x, y, 0.1, True))
    for checkpointing in (False, True):
        net = autograd.UnrolledLandweber(plan, 1, 0.1, checkpointing=checkpointing)
        assert torch.equal(net(x, y, c), step)


@pytest.mark.parametrize("checkpointing", [False, True])
@pytest.mark.parametrize("how", ["instance", "subclass"])
def test_replaced_step_takes_x_y_c_and_keeps_its_random_numbers(checkpointing, how):
    plan = DensePlan()
    c = torch.tensor(1500.0)
    y = torch.rand((1, plan.n_sensors, plan.n_samples))
    keep = []

    def step(x, y, c):
        # a step with random numbers: recomputing it in backward must draw the same
        mask = (torch.rand_like(x) < 0.5).to(x.dtype)
        keep.append(mask)
        return x * x * mask

    if how == "instance":
        net = autograd.UnrolledLandweber(plan, 2, 0.1, checkpointing=checkpointing)
        net.step = step
    else:
        class Net(autograd.UnrolledLandweber):
            def step(self, x, y, c):
                return step(x, y, c)
        net = Net(plan, 2, 0.1, checkpointing=checkpointing)
    x = torch.rand((1, plan.n_pixels), requires_grad=True)
    torch.manual_seed(5)
    out = net(x, y, c)
    m1, m2 = keep[:2]
    torch.manual_seed(6)  # backward runs with another state of the generator
    out.sum().backward()
    # out = m2 (m1 x^2)^2
    assert torch.allclose(x.grad, 4.0 * m2 * m1 * x.detach() ** 3)


def test_wrapped_bound_step_is_a_replacement():
    plan = DensePlan()
    net = autograd.UnrolledLandweber(plan, 3, 0.1)
    own, calls = net.step, []

    def traced(x, y, c):
        calls.append(float(c))
        return own(x, y, c)

    x, y = torch.rand((1, plan.n_pixels)), torch.rand((1, plan.n_sensors, plan.n_samples))
    expect = net(x, y, torch.tensor(1510.0))
    net.step = traced
    assert torch.equal(net(x, y, torch.tensor(1510.0)), expect)
    assert calls == [1510.0] * 3
