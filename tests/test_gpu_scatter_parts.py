"""The batched scatter with several warps per slice (csrc/scatter.cu), in FP32 and, by way of the
batched solve's residuals, in FP64, against the oracle: few pixels with many samples, uneven
hit counts, pixel counts around a slice, column counts around a group -- needs a GPU.

Tolerances: FP32 values and weights, sums in exact pairs of batches: 2e-5 for A x with its
transforms (test_gpu_scatter_sliced.py); a solve to 1e-10 in the oracle's arithmetic.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.system import Problem
from paper_1408_3048_gb300 import mm

pytestmark = pytest.mark.gpu

HITS = {"eight_long": [20000, 20003, 19998, 20001] * 2, "nine": [9000] * 9, "one": [30011],
        "uneven": [700, 690, 650, 705, 710, 698, 640, 702] * 40, "short": [70, 64, 66] * 500}


@pytest.mark.parametrize("hits", list(HITS))
@pytest.mark.parametrize("ncomp", [1, 3])
def test_batched_scatter(hits, ncomp):
    rng = np.random.default_rng(7)
    pix = rng.permutation(np.repeat(np.arange(len(HITS[hits])), HITS[hits])).astype(np.int32)
    nt, npix = pix.size, int(pix.max()) + 1
    phi = rng.uniform(0, np.pi, nt)
    w = np.stack([np.cos(2 * phi), np.sin(2 * phi)], 1) if ncomp == 3 else None
    off, psd = np.array([0, nt], dtype=np.int64), [(1.0, 1.0, 1.0)]
    pr = Problem(pix, npix, w, off, [0], psd, 100.0, 2, ncomp)
    plan = mm.Plan(pix, npix, w, off, [0], psd, 2, 100.0)
    for R in (1, 2, 5, 9):
        X = rng.standard_normal((R, pr.n)).astype(np.float32)
        Xc = torch.from_numpy(X).cuda()
        Y = plan.apply_A_batch(Xc)
        assert torch.equal(Y, plan.apply_A_batch(Xc))
        for x, y in zip(X, Y.cpu().numpy()):
            r = pr.A(x.astype(np.float64))
            assert np.linalg.norm(y - r) <= 2e-5 * np.linalg.norm(r)
    D = rng.standard_normal((5, nt))
    M, _, status = plan.solve_batch(torch.from_numpy(D).cuda(), tol=1e-10, maxit=500)
    assert status == mm.MM_OK
    for m, d in zip(M.cpu().numpy(), D):
        b = pr.rhs(d)
        assert np.linalg.norm(b - pr.A(m)) <= 2e-10 * np.linalg.norm(b)
    plan.close()
