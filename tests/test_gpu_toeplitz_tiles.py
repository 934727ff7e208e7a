"""The persistent FP32 Toeplitz kernel (csrc/toeplitz_ws.cu) on tiles whose positions and times
differ by no multiple of four and whose windows share nothing, as a plan lays them out where
the other layout would need more of them; and its load of FP64 data, with which a mixed solve
starts -- needs a GPU.

Tolerances: those of the kernel's transforms, 3e-6 (test_gpu_toeplitz_ws.py).  A solve stopped
after its first inner run has the FP32 right-hand side for its map: true residual against the
oracle's, inner tolerance 1e-6 and some hundred FP32 roundings of A's largest over smallest
eigenvalue (below 10 for white data): 1e-4.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1408_3048_gb300 import mm, synth
from problems import oracle_problem

pytestmark = pytest.mark.gpu

# (ncomp, lambda, interval lengths per detector, log2 block): intervals of exactly a tile's
# outputs; bands that leave two and six outputs; several tiles an interval
CASES = [(1, 1001, [14382] * 3, 14), (3, 1001, [14382, 14381], 14), (1, 8189, [9001], 14), (3, 8191, [8400], 14),
         (1, 2001, [28766, 28766], 15), (3, 16381, [16400, 16399], 15)]


def _problem(ncomp, lam, lengths, lb):
    nper, ndet = sum(lengths), 2
    scan = synth.raster_scan(12, 11, ndet, nper, ncomp, 1, lam, [(1.0, 1.0, 1.0), (0.8, 0.4, 1.5)], det_psd=[0, 1],
                             seed=11)
    scan.offsets = np.concatenate([[0], np.cumsum(lengths * ndet)]).astype(np.int64)
    scan.interval_psd = np.repeat(np.arange(ndet, dtype=np.int32), len(lengths))
    pr = oracle_problem(scan)
    plan = mm.Plan(scan.pix, scan.npix_sky, scan.weights, scan.offsets, scan.interval_psd, scan.psds, scan.lam,
                   scan.fsamp, fft_log2=(0, lb))
    assert plan.fft_block_f32 == 1 << lb
    return pr, plan


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"nc{c[0]}_lam{c[1]}_B{c[3]}")
def test_layout_without_shared_windows(case):
    pr, plan = _problem(*case)
    rng = np.random.default_rng(1)
    y = rng.standard_normal(pr.nt).astype(np.float32)
    ref = pr.Ninv(y.astype(np.float64), route="fft")
    z = plan.apply_ninv(torch.from_numpy(y).cuda(), mm.MM_FP32).cpu().numpy()
    assert np.linalg.norm(z - ref) <= 3e-6 * np.linalg.norm(ref)
    X = rng.standard_normal((3, pr.n)).astype(np.float32)
    Y = [plan.apply_A(torch.from_numpy(x).cuda(), mm.MM_FP32).cpu().numpy() for x in X]
    B = plan.apply_A_batch(torch.from_numpy(X).cuda()).cpu().numpy()
    for x, y1, y2 in zip(X, Y, B):
        ref = pr.A(x.astype(np.float64), route="fft")
        for v in (y1, y2):
            assert np.linalg.norm(v - ref) <= 2e-5 * np.linalg.norm(ref)
    plan.close()


@pytest.mark.parametrize("case", [(1, 63, [20000, 4001, 129], 14), (3, 511, [30001], 14), (3, 1001, [14382, 14381], 14),
                                  (1, 100, [3000, 2999, 5000, 7001], 15), (3, 4096, [40001, 9999], 15)],
                         ids=lambda c: f"nc{c[0]}_lam{c[1]}_B{c[3]}")
def test_rounded_data_of_a_mixed_solve(case):
    pr, plan = _problem(*case)
    D = np.random.default_rng(5).standard_normal((3, pr.nt))
    Dc = torch.from_numpy(D).cuda()
    o = mm.mm_solve_opts(tol=1e-12, maxit=2000, kind=mm.MM_PREC_BD, solver=mm.MM_SOLVE_MIXED, max_outer=1,
                         first_inner_tol=1e-6)
    plan.batch_config(3, mm.MM_BATCH_REAL)
    M = torch.empty(4, plan.n, dtype=torch.float64, device="cuda")
    mm.mm_solve_ex(plan.handle, Dc[0], o, M[3], raise_on_error=False)
    mm.mm_solve_batch(plan.handle, Dc, 3, o, M, raise_on_error=False)
    torch.cuda.synchronize()
    for m, d in zip(M.cpu().numpy(), np.concatenate([D, D[:1]])):
        b = pr.rhs(d, route="fft")
        assert np.linalg.norm(b - pr.A(m, route="fft")) <= 1e-4 * np.linalg.norm(b)
    plan.close()
