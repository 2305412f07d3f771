"""The Arnoldi step's kernel by itself (tests/ortho_driver.cu): a wait that gives up sets the status word and the next
launch computes; a vector that holds the all-ones NaN (the word that stands for "not written yet" between the blocks)
gives NaN and no timeout; squared norms from subnormal to large are followed by a vector of unit length.

Tolerance: n fused multiply-adds per sum in FP64, 2^-53 n of the vectors' lengths, and as much again for the second
pass and the scaling: 4 n 2^-53 (9e-13 for 2,048 entries), relative to the new vector's length, and the rounding
of subnormal squares."""
import os
import shutil
import struct
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def step(tmp_path_factory):
    from paper_0809_4802_gb300 import build
    exe = str(tmp_path_factory.mktemp("ortho") / "driver")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, *build.ARCH, "-O3", "-std=c++17", "-I", build.CSRC, os.path.join(HERE, "ortho_driver.cu"), "-o", exe],
                   check=True)

    def run(V, blocks, limit):
        kk, n = V.shape[0] - 1, V.shape[1]
        p = subprocess.run([exe], input=struct.pack("4q", n, kk, blocks, limit) + V.tobytes(), capture_output=True,
                           timeout=60, check=True)
        size = 4 + 8 * (kk + 1 + n)
        assert len(p.stdout) == 2 * size
        got = []
        for raw in (p.stdout[:size], p.stdout[size:]):
            d = np.frombuffer(raw[4:], np.float64)
            got.append((struct.unpack("i", raw[:4])[0], d[:kk], d[kk], d[kk + 1:]))
        return got
    return run


def vectors(kk, n, length=1.0):
    rng = np.random.default_rng(n + kk)
    Q, _ = np.linalg.qr(rng.normal(size=(n, kk + 1)))
    V = np.ascontiguousarray(Q.T)
    V[kk] *= length
    return V


def check(got, V, norm2):
    status, h, nn, w = got
    assert status == 0
    n = V.shape[1]
    tol = 4 * n * 2.0 ** -53 + n * 2.0 ** -1074 / norm2   # each square rounded to a multiple of 2^-1074
    assert abs(nn / norm2 - 1) < 2 * tol
    ref = V[-1] / np.abs(V[-1]).max()
    assert np.abs(w - ref / np.linalg.norm(ref)).max() < tol


@pytest.mark.parametrize("kk,n,blocks", [(3, 1024, 2), (9, 2048, 4), (40, 8192, 16)])
def test_a_wait_that_gives_up_sets_the_status(step, kk, n, blocks):
    V = vectors(kk, n)
    first, second = step(V, blocks, 0)
    assert first[0] == 1
    check(second, V, 1.0)


@pytest.mark.parametrize("kk,n,blocks", [(1, 32, 1), (9, 2048, 4)])
def test_an_all_ones_nan_is_no_timeout(step, kk, n, blocks):
    V = vectors(kk, n)
    V[kk, 5] = np.array([-1], np.int64).view(np.float64)[0]
    for status, h, nn, w in step(V, blocks, 1 << 22):
        assert status == 0 and np.isnan(h).all() and np.isnan(nn)


@pytest.mark.parametrize("length", [1e-158, 3e-157, 1e-154, 1e-3, 1e150])
def test_unit_length_from_any_norm(step, length):
    V = vectors(2, 512, length)
    for got in step(V, 2, 1 << 22):
        check(got, V, length * length)
