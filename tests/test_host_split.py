"""Spectra of the FP64 and double-float block product (fold_split_spectrum in csrc/plan_host.cpp)
on the CPU: the product that the kernels form from a row, folded pairs of bins and chained
ones, equals the circular convolution with the row's spectrum; which bins are chained."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_1408_3048_gb300", "csrc")
CUDA_INC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")

DRIVER = r"""
#include <cstdio>
#include "mm_internal.h"
int main() {
    long long N;
    if (std::scanf("%lld", &N) != 1) return 2;
    std::vector<double> h((size_t)N + 1);
    for (auto& x : h) if (std::scanf("%lf", &x) != 1) return 2;
    std::vector<double> f((size_t)mm::split_size(N)), q = mm::quarter_wave(2 * N);
    mm::fold_split_spectrum(h, N, q, f.data());
    for (double x : f) std::printf("%.17g\n", x);
    for (double x : q) std::printf("%.17g\n", x);
    return 0;
}
"""


@pytest.fixture(scope="module")
def fold(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.isdir(CUDA_INC):
        pytest.skip("g++ or the CUDA headers not available")
    d = tmp_path_factory.mktemp("split")
    (d / "driver.cpp").write_text(DRIVER)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", SRC, "-I", os.path.join(ROOT, "include"), "-I", CUDA_INC, "-o",
                    str(d / "driver"), str(d / "driver.cpp"), os.path.join(SRC, "plan_host.cpp")], check=True)

    def run(h):
        text = f"{len(h) - 1}\n" + "\n".join(repr(float(v)) for v in h)
        out = subprocess.run([str(d / "driver")], input=text, capture_output=True, text=True, check=True).stdout
        f = np.array([float(v) for v in out.split()])
        N = len(h) - 1
        assert f.size == N + N // 2 + 2 + N // 2 + 1
        return f[:-(N // 2 + 1)], f[-(N // 2 + 1):]
    return run


def _product(f, quarter, U, N):
    """V from U as SplitRow::product forms it, bins k and N - k together."""
    al, be, kc = f[:N], f[N:N + N // 2 + 1], int(f[-1])
    V = np.empty(N, complex)
    for k in range(N // 2 + 1):
        u1, u2 = U[k], U[-k % N]
        if k < kc:
            h2 = be[0] if k == 0 else al[N - k]
            W = quarter[k] - 1j * quarter[N // 2 - k]
            E, O = u1 + np.conj(u2), -1j * (u1 - np.conj(u2))
            Z1, Z2 = al[k] * (E + W * O), h2 * (E - W * O)
            S, D = Z1 + Z2, np.conj(W) * (Z1 - Z2)
            V[-k % N], V[k] = np.conj(S - 1j * D), S + 1j * D
        else:
            V[-k % N] = al[-k % N] * u2 + 1j * be[k] * np.conj(u1)
            V[k] = al[k] * u1 + 1j * be[k] * np.conj(u2)
    return V, kc


def _spectra(N):
    f = np.arange(N + 1) / N
    rng = np.random.default_rng(3)
    return {"white": np.ones(N + 1), "knee": 1 / (1 + (0.04 / np.maximum(f, 1e-3))**2), "zero": np.zeros(N + 1),
            "falling": 1 / (1e-3 + f), "signs": np.cos(9 * f), "rough": rng.uniform(0.9, 1.0, N + 1) * (1 + 5 * (f > 0.7)),
            "steep": np.maximum(f, 1e-4)**2}


@pytest.mark.parametrize("N", [256, 1024])
@pytest.mark.parametrize("kind", ["white", "knee", "zero", "falling", "signs", "rough", "steep"])
def test_product(fold, kind, N):
    h = _spectra(N)[kind]
    f, quarter = fold(h)
    y = np.random.default_rng(1).standard_normal(2 * N)
    V, kc = _product(f, quarter, np.fft.fft(y[0::2] + 1j * y[1::2]), N)
    v = np.fft.ifft(V)
    z = np.stack([v.real, v.imag], 1).ravel()
    ref = np.fft.irfft(np.fft.rfft(y) * h, n=2 * N)
    assert np.linalg.norm(z - ref) <= 1e-14 * max(np.abs(h).max(), 1e-300) * np.linalg.norm(y)
    # chained: up to the last pair whose values differ by more than a factor 4, in whole warps
    k = np.arange(N // 2 + 1)
    a, b = np.abs(h[k]), np.abs(h[N - k])
    far = np.flatnonzero(np.minimum(a, b) < 0.25 * np.maximum(a, b))
    want = 0 if far.size == 0 else far[-1] + 1
    assert kc == min(-(-want // 32) * 32, N // 2 + 1)
    assert (kc > 0) == (kind not in ("white", "zero"))
