"""Allocation failures in the library's host code, on the CPU: the library's objects linked with
a CUDA runtime of host memory and kernels that do nothing (fake_cuda.cpp).  Every allocation
of a call is made to fail in turn; the call reports MM_ERR_OOM (or does without), what it
held is given back, and the next calls launch with live tables only."""
import ctypes
import os
import shutil
import subprocess
import sys
from types import SimpleNamespace

import numpy as np
import pytest

from paper_1408_3048_gb300 import build, mm

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if shutil.which("g++") is None or not os.path.isdir(inc):
        pytest.skip("g++ or the CUDA headers not available")
    build.build()
    objs = [os.path.join(build.BUILD, f) for f in sorted(os.listdir(build.BUILD)) if f.endswith(".o")]
    so = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-Wl,-z,defs", "-I", inc, "-o", so,
                    os.path.join(HERE, "fake_cuda.cpp"), *objs, "-lpthread"], check=True)
    return load(so)


def load(so):
    L = ctypes.CDLL(so)
    for name, (res, args) in mm._SIGS.items():
        fn = getattr(L, name)
        fn.restype, fn.argtypes = res, args
    for name in ("fake_live_bytes", "fake_peak_bytes"):
        getattr(L, name).restype = ctypes.c_longlong
    L.fake_fail_after.argtypes = L.fake_room.argtypes = [ctypes.c_longlong]
    L.fake_launch_name.restype = ctypes.c_char_p
    return L


class Plan:
    """A plan of the fake device: two detectors of `lengths` each."""

    def __init__(self, L, lengths, lam, ncomp=3, side=16, npsd=2, psd_of=None, expect=mm.MM_OK, **opts):
        self.L = L
        lengths = list(lengths) * 2
        self.nt = sum(lengths)
        pix = (np.arange(self.nt) // 4 % (side * side)).astype(np.int32)
        phi = np.arange(self.nt) * 0.618
        w = np.stack([np.cos(2 * phi), np.sin(2 * phi)], 1) if ncomp == 3 else None
        off = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
        ipsd = (np.arange(len(lengths)) * npsd // len(lengths)).astype(np.int32)
        psd = (mm.mm_psd * npsd)(*[mm.mm_psd(1.0, 0.5, 1.0)] * npsd)
        o = mm.mm_opts(ncomp=ncomp, lambda_=lam, fsamp=100.0, **opts)
        self.h = ctypes.c_void_p()
        self.status = L.mm_plan(ctypes.byref(self.h), pix.ctypes.data, self.nt, side * side,
                                None if w is None else w.ctypes.data, off.ctypes.data, off.size - 1, ipsd.ctypes.data, psd,
                                npsd, ctypes.byref(o))
        assert self.status == expect
        if self.status == mm.MM_OK:
            n = ctypes.c_int64()
            b64, b32 = ctypes.c_int32(), ctypes.c_int32()
            L.mm_plan_info(self.h, None, ctypes.byref(n), None, ctypes.byref(b64), ctypes.byref(b32))
            self.n, self.block64, self.block32 = n.value, b64.value, b32.value
            self.X = np.zeros(64 * self.n, dtype=np.float32)

    def batch(self, R):
        """Status of Y = A X on R columns, and the launches of it."""
        self.L.fake_clear_launches()
        st = self.L.mm_apply_A_batch(self.h, R, self.X.ctypes.data, self.X.ctypes.data)
        return st, launches(self.L)

    def solve_batch(self, R):
        self.L.fake_clear_launches()
        D, M = np.zeros((R, self.nt)), np.zeros((R, self.n))
        o = mm.mm_solve_opts(tol=1e-6, maxit=10, kind=mm.MM_PREC_BD, solver=mm.MM_SOLVE_MIXED)
        st = self.L.mm_solve_batch(self.h, D.ctypes.data, R, ctypes.byref(o), M.ctypes.data, None)
        return st, launches(self.L)

    def config(self, R, kind=-1):
        """(form, log2 block) of the batched operator."""
        k, b = ctypes.c_int32(kind), ctypes.c_int32()
        st = self.L.mm_batch_config(self.h, R, ctypes.byref(k), ctypes.byref(b), None)
        assert st == mm.MM_OK
        return k.value, b.value

    def close(self):
        self.L.mm_destroy(self.h)


def launches(L):
    return [(L.fake_launch_name(i).decode(), L.fake_launch_grid(i), L.fake_launch_dead(i)) for i in range(L.fake_launches())]


def dead(ls):
    return [l for l in ls if l[2] != 0]


# (interval lengths, lambda, components): at 64 columns the pair form; the real form with the
# plan's kind of block, and with one of the persistent kernel's, neither of them the plan's
BATCHES = [([9000, 9000], 500, 3), ([40000, 40000], 500, 3), ([40000, 40000], 2000, 1)]


@pytest.mark.parametrize("lengths,lam,ncomp", BATCHES)
def test_batched_call_without_memory(lib, lengths, lam, ncomp):
    """A first batched call with each of its allocations failing in turn: it fails or does without,
    and later calls, on fewer columns too (which take other tables), launch with live ones."""
    base, failed = lib.fake_live_bytes(), 0
    for k in range(60):
        p = Plan(lib, lengths, lam, ncomp)
        lib.fake_fail_after(k)
        st, ls = p.batch(64)
        done = lib.fake_fail_after(-1) != 0
        assert st in (mm.MM_OK, mm.MM_ERR_OOM) and not dead(ls), k
        failed += st == mm.MM_ERR_OOM
        for call in (p.batch, p.solve_batch):
            for R in (1, 2, 64):
                st, ls = call(R)
                assert st == mm.MM_OK and not dead(ls), (k, R, dead(ls))
        p.close()
        assert lib.fake_live_bytes() == base, k
        if done:
            break
    assert failed >= 17 and done


@pytest.mark.parametrize("lengths,lam,ncomp", BATCHES + [([300000, 300000], 1024, 3), ([131072], 1024, 1)])
def test_batched_call_does_not_depend_on_the_calls_before(lib, lengths, lam, ncomp):
    """Form, block and launches of R columns are those of a fresh plan, whatever R came first."""
    def fresh(R):
        p = Plan(lib, lengths, lam, ncomp)
        out = p.batch(R), p.solve_batch(R)
        cfg = p.config(R)
        p.close()
        return out, cfg

    Rs = [1, 2, 7, 16, 64]
    want = {R: fresh(R) for R in Rs}
    for order in (Rs, Rs[::-1]):
        p = Plan(lib, lengths, lam, ncomp)
        for R in order:
            assert (p.batch(R), p.solve_batch(R)) == want[R][0], (order[0], R)
            assert p.config(R) == want[R][1]
        p.close()


def test_one_set_of_input_buffers_per_plan(lib):
    """The persistent kernel's input buffers (two of 2^15 floats per SM) are the plan's: a plan whose
    batch has a block of its own, both of that kernel, holds one set as a plan with one block."""
    buffers, held = 152 * 2 * (1 << 15) * 4, []
    for log2_f32, block in ((0, 1 << 14), (15, 1 << 15)):
        before = lib.fake_live_bytes()
        p = Plan(lib, [300000, 300000], 4000, 1, fft_log2_f32=log2_f32)
        assert p.block32 == block and p.config(8) == (1, 15)
        held.append(lib.fake_live_bytes() - before)
        p.close()
    assert buffers < held[0] < held[1] + buffers // 8


MANY_PSDS = r"""
import sys
sys.path[:0] = [{here!r}, {root!r}]
import test_host_alloc as t
L = t.load({so!r})
def rss():   # this process's peak (the resource module's figure includes its parent's)
    with open("/proc/self/status") as f:
        return 1024 * next(int(l.split()[1]) for l in f if l.startswith("VmHWM"))
small = t.Plan(L, [20000], 1000, 1, npsd=2, fft_log2_f64=14, fft_log2_f32=14)
small.close()
base, dev = rss(), L.fake_live_bytes()
p = t.Plan(L, [20000], 1000, 1, npsd=1500, fft_log2_f64=14, fft_log2_f32=14)
print(rss() - base - (L.fake_peak_bytes(0) - dev))
"""


def test_spectra_of_many_psds_one_at_a_time(lib):
    """Building a plan of many PSDs holds one arithmetic's table on the host beside the device's
    (147 MB of folded spectra here), not the spectra of all rows in several copies."""
    code = MANY_PSDS.format(here=HERE, root=os.path.dirname(HERE), so=lib._name)
    out = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, check=True).stdout
    table = 1500 * (8192 + 4096 + 2) * 8
    assert int(out) < 1.5 * table, (int(out), table)


# (lambda, log2 block of FP64 and FP32, interval length): as long as a tile's outputs, which are
# no multiple of four, or a band that leaves six outputs
@pytest.mark.parametrize("lam,logs,length,tiles", [(1001, (12, 12), 2094, 1), (512, (12, 12), 3071, 1), (1001, (14, 14), 14382, 1),
                                                   (2001, (15, 15), 28766, 1), (8189, (14, 14), 12000, 2000)])
def test_interval_of_a_tiles_outputs_takes_one_tile(lib, lam, logs, length, tiles):
    p = Plan(lib, [length] * 3, lam, 1, fft_log2_f64=logs[0], fft_log2_f32=logs[1])
    v = np.zeros(p.nt)
    want = tiles * 6
    for prec, cl in ((mm.MM_FP64, {15: 2}.get(logs[0], 1)), (mm.MM_FP32, 1)):
        lib.fake_clear_launches()
        assert lib.mm_apply_ninv(p.h, prec, v.ctypes.data, v.ctypes.data) == mm.MM_OK
        (name, grid, _), = launches(lib)
        if "toeplitz_ws" in name:   # CTAs of several tiles each
            assert grid == -(-want // -(-want // (152 << (15 - logs[1]))))
        else:
            assert grid == want * cl, name
    p.close()


def test_batched_scatter_of_few_pixels_fills_the_chip(lib):
    """64 pixels of 8192 samples are 8 slices: 32 warps take parts of each, for two columns and in
    each of the 16 groups of 64."""
    p = Plan(lib, [1 << 18], 100, 1, side=8)
    for R, grid, warps in ((2, 8, 32), (64, 8 * 16, 32)):
        name, blocks, _ = p.batch(R)[1][-1]
        assert "sliced_batch_parts_kernelIfLi1ELi4ELi%dE" % warps in name and blocks == grid, (R, name, blocks)
    p.close()
    p = Plan(lib, [1 << 17], 100, 3, side=64)   # 512 slices of 16 steps: two parts of eight
    name, blocks, _ = p.batch(4)[1][-1]
    assert "sliced_batch_parts_kernelIfLi3ELi4ELi8E" in name and blocks == 512 // 4
    p.close()


def scatters(L, p):
    """(FP64, FP32) forms of the plan, and the kernels that its scatters launch."""
    forms, names, v = [], [], np.zeros(max(p.nt, p.n))
    for prec in (mm.MM_FP64, mm.MM_FP32):
        lanes, warps = ctypes.c_int32(), ctypes.c_int32()
        assert L.mm_scatter_form(p.h, prec, ctypes.byref(lanes), ctypes.byref(warps)) == mm.MM_OK
        forms.append((lanes.value, warps.value))
        L.fake_clear_launches()
        assert L.mm_scatter(p.h, prec, v.ctypes.data, v.ctypes.data) == mm.MM_OK
        (name, _, _), = launches(L)
        names.append("sliced" if "sliced_scatter" in name else "lanes")
    return forms, names


def test_scatter_form_by_samples_and_memory(lib):
    for side, ncomp, want in ((32, 3, ["lanes", "lanes"]), (64, 3, ["sliced", "lanes"]), (128, 3, ["sliced", "sliced"]),
                              (32, 1, ["lanes", "lanes"]), (14, 1, ["lanes", "sliced"]), (8, 1, ["sliced", "sliced"])):
        p = Plan(lib, [1 << 19], 100, ncomp, side=side)   # 1024, 256, 64, 1024, 5349 and 16384 samples per pixel
        forms, names = scatters(lib, p)
        assert names == want and [f[0] for f in forms] == [4 if n == "sliced" else 32 for n in names], side
        for R in (2, 4):   # a small batch goes as one column does
            name = p.batch(R)[1][-1][0]
            assert ("sliced_batch" in name) == (R > 3 or names[1] == "sliced" or side <= 32), (side, R, name)
        p.close()
    # the layout takes a quarter of the free memory at most: 32 bytes for each of 2^20 samples
    for room, want in ((120 << 20, "lanes"), (140 << 20, "sliced")):
        lib.fake_room(room)
        p = Plan(lib, [1 << 19], 100, 3, side=128)
        assert scatters(lib, p)[1] == [want] * 2
        assert p.batch(4)[0] == mm.MM_OK
        p.close()
    lib.fake_room(270 << 30)


def test_batched_dot_products_use_the_chip(lib):
    """Two columns of 10^5 values: several blocks for each; many small columns: one each."""
    for side, R, want in ((180, 2, 2 * (3 * 180 * 180 // 16384)), (400, 2, 2 * (3 * 400 * 400 // 16384)), (16, 5, 5)):
        p = Plan(lib, [4 * side * side], 50, 3, side=side)
        dots = [grid for name, grid, _ in p.solve_batch(R)[1] if "dot_batch_kernel" in name]
        assert dots == [want], side
        p.close()


@pytest.mark.parametrize("lengths,lam,log2B", [([9001, 20003, 4999], 511, 14), ([14382, 14382], 1001, 14), ([3000, 2999, 5001], 101, 15),
                                              ([40001], 4095, 15), ([700] * 9, 64, 14), ([2094] * 5, 1001, 12),
                                              ([30000, 30001, 9999], 2047, 14)])
def test_bench_counts_the_plans_tiles(lib, lengths, lam, log2B):
    """bench.fft_tiles (its roofline's operations) against the launches' grids, in both layouts."""
    import bench
    p = Plan(lib, lengths, lam, 1, fft_log2_f64=log2B, fft_log2_f32=log2B)
    v = np.zeros(p.nt)
    scan = SimpleNamespace(lam=lam, offsets=np.concatenate([[0], np.cumsum(list(lengths) * 2)]),
                           interval_psd=np.repeat([0, 1], len(lengths)))
    for prec in (mm.MM_FP64, mm.MM_FP32):
        lib.fake_clear_launches()
        assert lib.mm_apply_ninv(p.h, prec, v.ctypes.data, v.ctypes.data) == mm.MM_OK
        (name, grid, _), = launches(lib)
        fours = "toeplitz_ws" in name
        assert fours == (prec == mm.MM_FP32 and log2B >= 14)
        ctas = 2 if "oscl" in name else 1   # per tile: two-CTA clusters; the persistent kernel: one tile each here
        assert grid == ctas * bench.fft_tiles(scan, 1 << log2B, fours=fours)
    p.close()
