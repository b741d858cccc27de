"""GELU of the inference kernel, read out of p: a network whose only active unit is one of the
second layer with the bias a gives z = S gelu(a) + b3, with S a power of two and b3 cancelling all
but the last digits, so p holds gelu(a) to 1e-8 of its value.

Tolerances: a product, a polynomial of small value, one exp2 (2^-22.5) and a sum of FP32 add up to
3e-7 of the value where gelu does not cancel (a >= -1); below, the terms are at most |a| E(a) < 0.16
with the same relative errors, 7e-8; below -5.5 the value itself is under 2.1e-7 and a relative error
of a few percent (the fit's) leaves 1e-9."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

B2, W1, W2, W3, B3 = 4672, 0, 576, 4736, 4800


def _bf16(v):
    import torch
    return float(torch.tensor(v, dtype=torch.float64).bfloat16().double())


def _p(params, x):
    import torch
    import paper_1007_4895_gb300 as lb
    net = lb.MLP(params, np.concatenate([np.zeros(8), np.ones(8)]).astype(np.float32))
    out = torch.empty(x.shape[1], device="cuda", dtype=torch.float32)
    net.infer(torch.tensor(x, dtype=torch.float32, device="cuda"), out)
    net.close()
    return out.cpu().numpy().astype(np.float64)


def _gelu(a, unit=5):
    """gelu(a) as the kernel has it, and in FP64."""
    ref = 0.5 * a * math.erfc(-a / math.sqrt(2.0))
    th = np.zeros(4801, np.float32)
    s = 2.0 ** 24
    b3 = 0.0
    if a >= -5.5:
        s = 2.0 ** (9 - math.frexp(abs(ref))[1])   # S |gelu| in [256, 512)
        b3 = -_bf16(s * ref)
    th[B2 + unit], th[W3 + unit], th[B3] = a, s, b3
    p = _p(th, np.zeros((8, 1)))[0]
    return (math.log(p / (1.0 - p)) - b3) / s, ref


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("exponent", range(-10, 3))
def test_gelu_against_fp64(exponent, sign):
    for m in range(0, 128, 3):
        a = sign * 2.0 ** exponent * (1.0 + m / 128.0)   # a BF16 value
        got, ref = _gelu(a, unit=(7 * m) % 64)
        tol = 3e-7 * abs(ref) if a >= -1.0 else (7e-8 if a >= -5.5 else 1e-9)
        assert abs(got - ref) <= tol, (a, got, ref, abs(got - ref) / abs(ref))


def test_overflowing_pre_activations():
    """A finite feature that overflows a unit: the erf form's limits, NaN at -inf (no p: the map
    update falls back) and +inf at +inf (p = 1 through positive weights)."""
    x = np.zeros((8, 3))
    x[0] = (3e38, 0.0, 3e38)
    th = np.zeros(4801, np.float32)
    th[W3:W3 + 64] = 1.0
    th[W2:W2 + 4096] = 1.0
    th[W1 + 0] = -2.0
    p = _p(th, x)
    assert np.isnan(p[0]) and np.isnan(p[2]) and p[1] == 0.5
    th[W1 + 0] = 2.0
    p = _p(th, x)
    assert p[0] == 1.0 and p[2] == 1.0 and p[1] == 0.5
