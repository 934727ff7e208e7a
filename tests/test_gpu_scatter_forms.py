"""Every form of the one-column scatter that a plan can take by itself (mm_scatter_form), in FP32
and FP64, with weights formed from angles and stored ones, by itself and with the fused dot
product of the solvers, against the oracle -- needs a GPU.

Tolerances: FP64 sums in short batches, 1e-13; FP32 values and weights (angles within 6e-7,
values rounded to 2^-24, sums in exact pairs of batches of eight), 2e-6.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.system import Problem
from paper_1408_3048_gb300 import mm

pytestmark = pytest.mark.gpu


def _ragged(lo, hi, n):
    return np.random.default_rng(lo).integers(lo, hi, n)


# name: (components, hits per pixel, FP64 form, FP32 form); forms: (lanes, warps per slice)
FORMS = {"one_warp": (3, _ragged(17, 25, 30001), (4, 1), (4, 1)), "two_warps": (3, _ragged(96, 101, 12003), (4, 2), (4, 2)),
         "four_warps": (1, np.full(9001, 128), (4, 4), (4, 4)), "all_warps": (3, _ragged(4190, 4210, 601), (4, 32), (4, 32)),
         "all_warps_T": (1, _ragged(8200, 8210, 41), (4, 32), (4, 32)), "shortest": (3, _ragged(4, 9, 1003), (4, 1), (4, 1)),
         "shortest_T": (1, _ragged(1, 9, 9), (4, 1), (4, 1)), "lanes": (3, _ragged(310, 330, 2500), (32, 0), (32, 0)),
         "lanes_T": (1, _ragged(310, 330, 2500), (32, 0), (32, 0)), "lanes_f32": (3, _ragged(250, 262, 2500), (4, 8), (32, 0)),
         "long_lanes_T": (1, _ragged(4190, 4210, 1101), (32, 0), (32, 0)),
         "long": (3, _ragged(4190, 4210, 1101), (32, 0), (4, 32))}
# FP32 sums in exact pairs and weights of 2^-24: 3.4e-8 for the weights, 2.4e-8 sqrt(8) for the
# sums of eight, 3.4e-8 for the result, in quadrature 8e-8; plain sums and angles leave 2.6e-7
EXACT = {"one_warp", "two_warps", "four_warps", "all_warps", "all_warps_T", "lanes_T", "long_lanes_T", "long"}


@pytest.mark.parametrize("name,eff", [(k, e) for k in FORMS for e in ((1.0, 0.9) if FORMS[k][0] == 3 else (1.0,))])
def test_scatter_forms(name, eff):
    ncomp, hits, form64, form32 = FORMS[name]
    rng = np.random.default_rng(7)
    pix = rng.permutation(np.repeat(np.arange(len(hits)), hits)).astype(np.int32)
    nt, npix = pix.size, len(hits)
    phi = rng.uniform(0, np.pi, nt)
    w = eff * np.stack([np.cos(2 * phi), np.sin(2 * phi)], 1) if ncomp == 3 else None
    off, psd = np.array([0, nt], dtype=np.int64), [(1.0, 1.0, 1.0)]
    pr = Problem(pix, npix, w, off, [0], psd, 100.0, 2, ncomp)
    plan = mm.Plan(pix, npix, w, off, [0], psd, 2, 100.0)
    assert plan.n == pr.n
    assert (plan.scatter_form(mm.MM_FP64), plan.scatter_form(mm.MM_FP32)) == (form64, form32)
    z = rng.standard_normal(nt)
    zc = torch.from_numpy(z).cuda()
    ref = pr.PT(z)
    for prec, v, tol in ((mm.MM_FP64, zc, 1e-13), (mm.MM_FP32, zc.float(), 2e-7 if name in EXACT else 2e-6)):
        got = plan.scatter(v, prec)
        assert torch.equal(got, plan.scatter(v, prec))
        assert np.linalg.norm(got.double().cpu().numpy() - ref) <= tol * np.linalg.norm(ref)
    # p^T A p of the solvers' steps: as many of them as with the plain lanes
    lanes = mm.Plan(pix, npix, w, off, [0], psd, 2, 100.0, scatter_lanes=32)
    assert lanes.scatter_form(mm.MM_FP32) == (32, 0)
    for solver in (mm.MM_SOLVE_FP64, mm.MM_SOLVE_MIXED):
        m, st, status = plan.solve(zc, tol=1e-10, maxit=500, solver=solver)
        m2, st2, status2 = lanes.solve(zc, tol=1e-10, maxit=500, solver=solver)
        assert status == status2 == mm.MM_OK and abs(st["iters"] - st2["iters"]) <= 1
        b = pr.rhs(z)
        assert np.linalg.norm(b - pr.A(m.cpu().numpy())) <= 2e-10 * np.linalg.norm(b)
    plan.close()
    lanes.close()


def test_autotuned_plan_times_the_sliced_scatter():
    # 2500 pixels of 320: the rule says lanes; timed, either may win, and the form says which
    hits = FORMS["lanes_T"][1]
    pix = np.random.default_rng(7).permutation(np.repeat(np.arange(len(hits)), hits)).astype(np.int32)
    plan = mm.Plan(pix, len(hits), None, [0, pix.size], [0], [(1.0, 1.0, 1.0)], 2, 100.0, autotune=True)
    lanes, ms = plan.scatter_config()
    form = plan.scatter_form(mm.MM_FP32)
    assert form in ((lanes, 0), (4, 8)) and (np.asarray(ms) > 0).all()
    z = torch.randn(pix.size, dtype=torch.float64, device="cuda")
    ref = np.bincount(pix, weights=z.cpu().numpy())
    for prec, v, tol in ((mm.MM_FP64, z, 1e-13), (mm.MM_FP32, z.float(), 2e-6)):
        assert np.linalg.norm(plan.scatter(v, prec).double().cpu().numpy() - ref) <= tol * np.linalg.norm(ref)
    plan.close()
