"""The eigenvalue iteration of the stability scan (csrc/lbm_eig.cuh, the host
build of the same code) against LAPACK."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0706_0405_gb300", "csrc")

HARNESS = r"""
#include "lbm_eig.cuh"
extern "C" void radii(const double* a, int count, double* out) {
    for (int q = 0; q < count; ++q) {
        lbm::cplx H[81];
        for (int k = 0; k < 81; ++k) H[k] = lbm::cplx{a[2 * (81 * q + k)], a[2 * (81 * q + k) + 1]};
        out[q] = lbm::spectral_radius(H, 9);
    }
}
"""


@pytest.fixture(scope="module")
def radii(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("eig")
    src, lib = d / "harness.cpp", d / "libeig.so"
    src.write_text(HARNESS)
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True,
                   capture_output=True)
    fn = ctypes.CDLL(str(lib)).radii

    def run(A):
        A = np.ascontiguousarray(A, dtype=np.complex128)
        out = np.empty(len(A))
        fn(A.ctypes.data_as(ctypes.c_void_p), len(A), out.ctypes.data_as(ctypes.c_void_p))
        return out
    return run


@pytest.mark.parametrize("kind", ["dense", "tiny", "huge", "sparse", "block", "degenerate"])
def test_spectral_radius(radii, kind):
    """A backward error of 9 eps |A| (a few hundred rotations of 9 x 9
    entries) moves the eigenvalues of these matrices, whose condition numbers
    stay below a thousand, by less than 2e-12 of the radius."""
    rng = np.random.default_rng(5)
    A = rng.standard_normal((200, 9, 9)) + 1j * rng.standard_normal((200, 9, 9))
    scale = {"tiny": 1e-250, "huge": 1e250}.get(kind, 1.0)
    if kind == "sparse":
        A[np.abs(A) < 1.0] = 0.0
    elif kind == "block":
        A[:, 4:, :4] = 0.0
    elif kind == "degenerate":  # a normal matrix with eigenvalues of multiplicity three
        Q = np.linalg.qr(A)[0]
        A = Q @ (np.array([1, 1, 1, 0.5, 0.5, 0.5, -1j, -1j, 0])[None, :, None] * np.conj(Q.transpose(0, 2, 1)))
    want = np.abs(np.linalg.eigvals(A)).max(1)
    got = radii(A * scale)
    assert np.abs(got / scale / want - 1.0).max() <= 2e-12


def test_not_finite(radii):
    A = np.zeros((4, 9, 9), complex) + np.eye(9)
    A[1, 3, 4], A[2, 8, 0] = np.nan, -np.nan
    A[3] = 0.0
    got = radii(A)
    assert got[0] == 1.0 and np.isnan(got[1:3]).all() and got[3] == 0.0
