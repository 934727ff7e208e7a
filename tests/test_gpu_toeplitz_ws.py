"""The FP32 Toeplitz blocks of 2^14 and 2^15 reals (persistent kernel, csrc/toeplitz_ws.cu)
against the oracle where it can go wrong: one block and several per CTA, windows that share
positions and windows that do not (bands near half a block), blocks of one, two and three
intervals, odd bands and offsets, outputs that are not 16-byte aligned, several right-hand
sides -- needs a GPU.

Tolerance: an FFT pass of radix 16 rounds each value about seven times (two per twiddle, one
per level and constant), so two transforms of four passes and the product give about 60
roundings of 2^-24 / sqrt(3), in quadrature: 2.7e-7 of the block's input norm times the
largest |symbol|; the output's norm is at least that of the input times the smallest over the
largest symbol, here within a factor 10 for white data.  3e-6.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1408_3048_gb300 import mm, synth
from problems import oracle_problem

pytestmark = pytest.mark.gpu
TOL = 3e-6


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


# (ncomp, lambda, interval lengths per detector, log2 block)
CASES = [
    (1, 1, [300], 14),                        # one partly filled block
    (3, 63, [20000, 4001, 129], 14),
    (1, 511, [50001], 14),                    # many windows of one run, odd offsets
    (3, 2047, [30000, 30001, 2999], 14),
    (1, 8000, [40000, 16001], 14),            # the band fills the block: 384 outputs each
    (3, 100, [3000, 2999, 5000, 7001], 15),   # several intervals per block
    (1, 4096, [70000, 65537], 15),
    (3, 8191, [60000, 20001], 15),
    (1, 16000, [50000], 15),
]


@pytest.fixture(scope="module", params=CASES, ids=lambda c: f"nc{c[0]}_lam{c[1]}_B{c[3]}")
def case(request):
    ncomp, lam, lengths, lb = request.param
    nper, ndet = sum(lengths), 2
    scan = synth.raster_scan(12, 11, ndet, nper, ncomp, 1, lam, [(1.0, 1.0, 1.0), (0.8, 0.4, 1.5)], det_psd=[0, 1],
                             seed=11)
    scan.offsets = np.concatenate([[0], np.cumsum(lengths * ndet)]).astype(np.int64)
    scan.interval_psd = np.repeat(np.arange(ndet, dtype=np.int32), len(lengths))
    pr = oracle_problem(scan)
    plan = mm.Plan(scan.pix, scan.npix_sky, scan.weights, scan.offsets, scan.interval_psd, scan.psds, scan.lam,
                   scan.fsamp, fft_log2=(0, lb))
    assert plan.fft_block_f32 == 1 << lb
    yield scan, pr, plan
    plan.close()


def test_noise_weighting(case):
    _, pr, plan = case
    y = np.random.default_rng(1).standard_normal(pr.nt).astype(np.float32)
    ref = pr.Ninv(y.astype(np.float64), route="fft")
    yc = torch.from_numpy(y).cuda()
    z = plan.apply_ninv(yc, mm.MM_FP32).cpu().numpy()
    assert _rel(z, ref) <= TOL
    # input and output at addresses that are multiples of 4 bytes only: the same values
    buf = torch.empty(pr.nt + 1, dtype=torch.float32, device="cuda")
    src = torch.empty(pr.nt + 3, dtype=torch.float32, device="cuda")
    src[3:] = yc
    buf[0] = 7.0
    mm.mm_apply_ninv(plan.handle, mm.MM_FP32, src[3:], buf[1:])
    torch.cuda.synchronize()
    assert np.array_equal(buf[1:].cpu().numpy(), z) and float(buf[0]) == 7.0


def test_operator_and_right_hand_sides(case):
    _, pr, plan = case
    rng = np.random.default_rng(2)
    X = rng.standard_normal((3, pr.n)).astype(np.float32)
    ref = [pr.A(x.astype(np.float64), route="fft") for x in X]
    Xc = torch.from_numpy(X).cuda()
    assert _rel(plan.apply_A(Xc[0].clone(), mm.MM_FP32).cpu().numpy(), ref[0]) <= TOL
    plan.batch_config(3, mm.MM_BATCH_REAL)
    Y = plan.apply_A_batch(Xc).cpu().numpy()
    for r in range(3):
        assert _rel(Y[r], ref[r]) <= TOL
