"""Accuracy of N^-1 in its slowest modes, which a map-maker divides by the small values of the
noise spectrum there -- needs a GPU.

The input is one smooth pulse of 2^41 and integer samples, so that y = a + b holds exactly; what
N^-1 y - N^-1 a - N^-1 b leaves in the low frequencies is rounding alone (an error of the
kernel's spectrum cancels).  Its size against N^-1 y there: each transform rounds a value
about 60 times in quadrature (five passes, two of them forth and back, a dozen operations
each), 8 x 2^-53 = 9e-16 over three products in FP64; 2e-15.  Double-float rounds to 2^-48
and its sums to a few units of that: 32 times FP64's figure per operation and twice the
operations' error, 5e-14.  A product whose rounding is that of the largest spectrum value in
every bin leaves 1e-14 to 1e-13 in FP64 (h_low / h_max = 1e-3 to 3e-5 here).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1408_3048_gb300 import mm

pytestmark = pytest.mark.gpu

# (log2 block, lambda): one CTA small and largest, two and four CTAs
BLOCKS = [(12, 700), (14, 1000), (14, 4000), (15, 6000), (16, 8191)]


def _pulse(nt):
    x = (np.arange(nt) + 0.5) / nt
    return np.rint(2.0**40 * np.sin(np.pi * x)**8 * (1 + np.cos(6 * np.pi * x + 1)))


def _low(e, z):
    w = np.hanning(z.size)
    return np.linalg.norm(np.fft.rfft(e * w)[1:9]) / np.linalg.norm(np.fft.rfft(z * w)[1:9])


@pytest.mark.parametrize("log2B,lam", BLOCKS)
@pytest.mark.parametrize("fknee,alpha", [(1.0, 1.5), (2.0, 2.0)])
def test_rounding_in_the_low_modes(log2B, lam, fknee, alpha):
    nt = (1 << log2B) - 2 * lam
    plan = mm.Plan(np.arange(nt, dtype=np.int32), nt, None, [0, nt], [0], [(1.0, fknee, alpha)], lam, 100.0,
                   fft_log2=(log2B, 0))
    assert plan.fft_block_f64 == 1 << log2B
    y = _pulse(nt)
    a = np.rint(0.377 * y)
    zero = torch.zeros(nt, dtype=torch.float64, device="cuda")
    calls = [(2e-15, lambda v: plan.apply_ninv(v)), (2e-15, lambda v: plan.residual(v, zero, mm.MM_RESID_FP64)),
             (5e-14, lambda v: plan.residual(v, zero, mm.MM_RESID_DF32))]
    for tol, call in calls:
        z, za, zb = (call(torch.from_numpy(v).cuda()).cpu().numpy() for v in (y, a, y - a))
        err = _low(z - za - zb, z)
        assert err <= tol, err
    plan.close()
