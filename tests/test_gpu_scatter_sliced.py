"""The sliced scatter P^T z (csrc/scatter.cu) against the oracle where it can go wrong: pixel
counts around a slice of eight, hit counts around a step of four and a batch of eight steps,
one pixel much longer than its neighbours, few pixels with many samples (several warps per
slice), padding so large that the 32-lane form is kept -- needs a GPU.

Tolerances: FP64 sums of up to 2^17 values in short batches, 1e-13 relative; FP32 values and
weights (angle weights within 6e-7, values rounded to 2^-24, sums in exact pairs of batches
of eight): 2e-6.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.system import Problem
from paper_1408_3048_gb300 import mm

pytestmark = pytest.mark.gpu


def _hits(kind, rng):
    return {"one": [40], "seven": rng.integers(30, 40, 7), "nine": rng.integers(3, 9, 9),
            "fours": [4, 5, 8, 31, 32, 33, 36, 64, 65], "long_one": [20] * 11 + [400] + [20] * 30,
            "few_many": [40000, 39999, 38003], "many": rng.integers(40, 70, 3000),
            "ragged": [3, 3000] * 20}[kind]


@pytest.mark.parametrize("kind", ["one", "seven", "nine", "fours", "long_one", "few_many", "many", "ragged"])
@pytest.mark.parametrize("ncomp", [1, 3])
@pytest.mark.parametrize("eff", [1.0, 0.9])   # angle weights, stored pairs
def test_scatter(kind, ncomp, eff):
    if ncomp == 1 and eff != 1.0:
        pytest.skip("no weights")
    rng = np.random.default_rng(7)
    pix = np.repeat(np.arange(len(_hits(kind, rng))), _hits(kind, np.random.default_rng(7)))
    pix = rng.permutation(pix).astype(np.int32)
    nt, npix = pix.size, int(pix.max()) + 1
    phi = rng.uniform(0, np.pi, nt)
    w = eff * np.stack([np.cos(2 * phi), np.sin(2 * phi)], 1) if ncomp == 3 else None
    off = np.array([0, nt], dtype=np.int64)
    psd = [(1.0, 1.0, 1.0)]
    pr = Problem(pix, npix, w, off, [0], psd, 100.0, 2, ncomp)
    plan = mm.Plan(pix, npix, w, off, [0], psd, 2, 100.0)
    assert plan.n == pr.n
    z = rng.standard_normal((5, nt))
    ref = np.stack([pr.PT(v) for v in z])
    got = plan.scatter(torch.from_numpy(z[0]).cuda()).cpu().numpy()
    assert np.linalg.norm(got - ref[0]) <= 1e-13 * np.linalg.norm(ref[0])
    again = plan.scatter(torch.from_numpy(z[0]).cuda()).cpu().numpy()
    assert np.array_equal(got, again)
    got = plan.scatter(torch.from_numpy(z[0]).float().cuda(), mm.MM_FP32).double().cpu().numpy()
    assert np.linalg.norm(got - ref[0]) <= 2e-6 * np.linalg.norm(ref[0])
    # the batched form and the solver's fused dot product, through A
    X = rng.standard_normal((5, pr.n))
    Y = plan.apply_A_batch(torch.from_numpy(X).float().cuda()).double().cpu().numpy()
    for x, y in zip(X, Y):
        r = pr.A(x)
        assert np.linalg.norm(y - r) <= 2e-5 * np.linalg.norm(r)
    d = torch.from_numpy(z[1]).cuda()
    m, st, status = plan.solve(d, tol=1e-10, maxit=500)
    b = pr.rhs(z[1])
    assert status == mm.MM_OK and np.linalg.norm(b - pr.A(m.cpu().numpy())) <= 2e-10 * np.linalg.norm(b)
    plan.close()
