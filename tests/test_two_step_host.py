"""The two-step transforms on the CPU (tests/fft_host/two_step_host.cu): every codelet against numpy,
both steps of every x, y and z length that splits against numpy at the positions the tables name, the
phased twiddle tables, and what the kernels assume of the axis plans."""
from __future__ import annotations

import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "fft_host", "two_step_host.cu")
CSRC = os.path.join(os.path.dirname(HERE), "paper_2506_15411_gb300", "csrc")
P = ctypes.c_void_p
RADICES = [r for r in range(2, 37) if r <= 16 or r in (18, 20, 21, 22, 24, 25, 26, 27, 28, 30, 32, 35, 36)]
U = 2.0 ** -24   # half a unit in the last place of a value below 1


@pytest.fixture(scope="module")
def ts(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    out = str(tmp_path_factory.mktemp("two_step_host") / "libtwo_step_host.so")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-fPIC", "-shared", "--expt-relaxed-constexpr",
                    "-I", CSRC, "-o", out, SRC], check=True, capture_output=True)
    return ctypes.CDLL(out)


def _ptr(a):
    return a.ctypes.data_as(P)


def _lengths():
    def ok(m):
        for p in (2, 3, 5, 7, 11, 13):
            while m % p == 0:
                m //= p
        return m == 1
    return [n for n in range(4, 1025) if ok(n)]


def _plan(ts, n, which, rows=640 * 336):
    out = (ctypes.c_int * 8)()
    ts.ts_plan(n, which, ctypes.c_longlong(rows), out)
    return list(out)


@pytest.mark.parametrize("inv", [0, 1])
def test_codelets(ts, inv):
    """At most a dozen roundings of a value in sequence: 1e-6 of the norm is generous, a wrong index is 1."""
    rng = np.random.default_rng(5)
    for r in RADICES:
        x = (rng.standard_normal(r) + 1j * rng.standard_normal(r)).astype(np.complex64)
        v = x.copy()
        assert ts.ts_dft(r, inv, _ptr(v)) == 0
        want = np.fft.ifft(x.astype(complex)) * r if inv else np.fft.fft(x.astype(complex))
        assert np.linalg.norm(v - want) <= 1e-6 * np.linalg.norm(want), r


@pytest.mark.parametrize("which", [0, 1, 2])
def test_both_steps_of_every_length(ts, which):
    rng = np.random.default_rng(7 + which)
    done = 0
    for n in _lengths():
        if not _plan(ts, n, which)[0]:
            continue
        x = (rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(np.complex64)
        y, back, freq = np.zeros_like(x), np.zeros_like(x), np.zeros(n, np.int32)
        ph = n % 8
        assert ts.ts_transform(n, which, ph, 0, _ptr(x), _ptr(y), _ptr(freq)) == 0
        assert sorted(freq) == list(range(n))
        want = np.fft.fft(x.astype(complex))
        assert np.linalg.norm(y - want[freq]) <= 2e-6 * np.linalg.norm(want), n
        assert ts.ts_transform(n, which, (ph + 3) % 8, 1, _ptr(y), _ptr(back), _ptr(freq)) == 0
        assert np.linalg.norm(back - n * x) <= 4e-6 * n * np.linalg.norm(x), n
        done += 1
    assert done == (197, 194, 125)[which]


def test_phased_twiddles_average_to_the_twiddle(ts):
    """A phase is within a unit of the value; the carried error leaves the sum of the eight within half a
    unit of eight times the value."""
    for n, A in ((315, 35), (336, 28), (64, 4), (275, 11), (1024, 32), (12, 3)):
        B = n // A
        k1, j = np.divmod(np.arange(n), B)
        want = np.exp(-2j * np.pi * (k1 * j % n) / n)
        got = []
        for ph in range(8):
            t = np.zeros(n, np.complex64)
            ts.ts_twiddles(n, A, ph, _ptr(t))
            got.append(t.astype(complex))
            assert np.abs((got[-1] - want).real).max() <= 2 * U and np.abs((got[-1] - want).imag).max() <= 2 * U
        mean = np.mean(got, axis=0) - want
        assert max(np.abs(mean.real).max(), np.abs(mean.imag).max()) <= U / 8


def test_plans_hold_what_the_kernels_assume(ts):
    for n in _lengths():
        A, ldw, lde, rpb, sets, teams = _plan(ts, n, 0)[:6]
        if A:
            B = n // A
            pitch = B + (6 - B % 4) % 4
            assert pitch % 4 == 2 and ldw >= max(n + n % 2, A * pitch) and lde >= n + n % 2
            assert ldw % 2 == 0 and lde % 2 == 0                       # 16-byte rows
            assert 2 <= sets <= 8 and 1 <= teams <= 5 and teams <= sets - 1
            assert sets * rpb * (3 * ldw + 4 * lde) * 8 + (n + 1) // 2 * 16 + 8 * 17 + 16 <= 227 * 1024
        for which in (1, 2):
            A, tx, gt, groups, sets, held, box = _plan(ts, n, which)[:7]
            if not A:
                continue
            assert groups <= sets - 1 and groups <= 6 and groups * gt + 32 <= 736
            assert gt % 32 == 0 and gt % tx == 0
            assert held >= n and box <= (n if which == 1 else 256)
            if which == 2:
                assert box * tx * 8 % 128 == 0
            fixed = (n + 1) // 2 * 16 * which + 8 * 17 + 48
            assert sets * (2 * which - 1) * held * tx * 8 + fixed <= 227 * 1024
