"""Host-side logic inside the CUDA sources, checked on the CPU by small
nvcc-built harnesses that run no kernel (tests/host/): the banded LU with an
arrow border of the moment coarse correction, the resampling matrices of
the mixed-N solver against the oracle's FFT-based resampling, and the
register-resident 32-point transform of the FP64 kernels against a direct
DFT."""
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

from oracle.resample import resample_axis

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HOST = os.path.join(ROOT, "tests", "host")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


def _build(name, tmp_path):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / name)
    subprocess.check_call([NVCC, "-std=c++17", "-O1", "-I" + os.path.join(ROOT, "include"),
                           "-I" + os.path.join(ROOT, "paper_2503_09580_gb300", "csrc"), "-o", exe,
                           os.path.join(HOST, name + ".cu")])
    return exe


def test_banded_lu_with_arrow_border(tmp_path):
    out = subprocess.run([_build("banded_lu", tmp_path)], check=True, capture_output=True, text=True).stdout
    rows = [line.split() for line in out.strip().splitlines()]
    assert len(rows) == 5
    for nb, nx, border, err in rows:
        assert err != "factor_failed", (nb, nx, border)
        assert float(err) < 1e-11, (nb, nx, border, err)


def test_resampling_matrices_match_the_oracle(tmp_path):
    pairs = [(16, 24), (24, 16), (32, 48), (48, 24), (24, 32), (64, 32)]
    L = 8.0
    inp = "".join("%d %d\n" % p for p in pairs)
    out = subprocess.run([_build("resample_matrix", tmp_path), str(L)], input=inp, check=True,
                         capture_output=True, text=True).stdout
    vals = np.array([float(x) for x in out.split()])
    o = 0
    for na, nb in pairs:
        R = vals[o:o + na * nb].reshape(nb, na)
        o += na * nb
        # the oracle resamples centred-order unit vectors (cyclic order inside)
        E = np.eye(na)
        cols = []
        for a in range(na):
            e = np.fft.ifftshift(E[a])
            cols.append(np.fft.fftshift(resample_axis(e, nb, 0)))
        ref = np.array(cols).T
        assert np.abs(R - ref).max() <= 1e-13, (na, nb, np.abs(R - ref).max())
    assert o == vals.size


def test_register_fft32_against_a_direct_dft(tmp_path):
    """The 32-point transform of the FP64 register kernels (scaled-twiddle
    radix-2, fft_reg.cuh) against a direct DFT in long double: a few units
    of the working precision's roundoff, forward and inverse, and the scaled
    twiddles reproduce W_32^m to about one unit of double roundoff."""
    out = subprocess.run([_build("fft_reg", tmp_path)], check=True, capture_output=True, text=True).stdout
    res = {" ".join(line.split()[:-1]): float(line.split()[-1]) for line in out.strip().splitlines()}
    assert res["double forward"] <= 8 * 2.0 ** -53 and res["double inverse"] <= 8 * 2.0 ** -53
    assert res["float forward"] <= 8 * 2.0 ** -24 and res["float inverse"] <= 8 * 2.0 ** -24
    assert res["twiddle"] <= 4 * 2.0 ** -53


def test_fixed_point_arithmetic_against_long_double(tmp_path):
    """The fixed-point products, pencil transforms and DCT-I (fx64.cuh) in units
    of the last place.  A product leaves out yl tl (below 1/4) and takes two
    floors balanced by 1: below 1.5; rounded once: below 1.  A transform's value
    passes at most 5 products and its output sums 4 of them: rms below 1.5
    sqrt(20); a DCT-I output sums at most H/2 doubled products.  The transforms
    have no mean error beyond the 1/4 of a halving (N = 24), and keep zeros."""
    out = subprocess.run([_build("fx64", tmp_path)], check=True, capture_output=True, text=True).stdout
    res = {r[0]: (float(r[1]), float(r[2])) for r in (line.split() for line in out.strip().splitlines())}
    assert res["mul"][0] < 1.5 and res["mul_signed"][0] < 1.5 and res["mul_signed_rounded"][0] < 1.0
    assert abs(res["mul_signed_rounded"][1]) < 0.01
    assert res["mul_pair"][0] < 2 * 1.5  # the sum of two products
    for n in (16, 24, 32):
        for d in "fi":
            err, bias = res["dft%d%s" % (n, d)]
            assert err < 1.5 * 20 ** 0.5 and abs(bias) < (0.25 if n == 24 else 0.02), (n, d, err, bias)
    for h in (8, 12, 16, 24, 32):
        assert res["dct%d" % h][0] < 2 * 1.5 * h / 2, h


def test_tables_are_uploaded_in_order_with_every_stream():
    """Outside the plan's build_tables, which ends with a device
    synchronisation, no source copies or clears a table on the legacy stream
    without waiting for it: kernels of a non-blocking stream would not be
    ordered behind it."""
    csrc = os.path.join(ROOT, "paper_2503_09580_gb300", "csrc")
    found = []
    for name in sorted(os.listdir(csrc)):
        if not name.endswith((".cu", ".cuh", ".h")) or name == "lbo.cu":
            continue
        with open(os.path.join(csrc, name)) as fh:
            text = fh.read()
        for call in re.finditer(r"cudaMemcpy\([^;]*cudaMemcpyHostToDevice\)|cudaMemcpyToSymbol\(|cudaMemset\(", text):
            if "cudaStreamSynchronize(cudaStreamLegacy)" not in text[call.start():call.start() + 1200]:
                found.append((name, call.group(0)))
    assert not found
    with open(os.path.join(csrc, "lbo.cu")) as fh:
        text = fh.read()
    assert not re.search(r"HostToDevice", text[text.index("build_phit(lbo_plan* p, const double* d_stab, T* d_phit) {"):])
    assert "cudaDeviceSynchronize()" in text[text.index("static lbo_status build_phit(lbo_plan* p, const double* d_stab, T* d_phit) {"):]


def test_fixed_point_workspaces_do_not_shrink_with_the_batch(tmp_path):
    """Q's fixed-point workspace, from the library itself: a smaller batch never
    needs a larger buffer, so a graph captured with one batch keeps its buffer
    when the plan is called with another."""
    lib = os.path.join(ROOT, "paper_2503_09580_gb300", "_lib")
    if not os.path.exists(os.path.join(lib, "liblbo.so")) or not os.path.exists(NVCC):
        pytest.skip("library or nvcc not available")
    exe = str(tmp_path / "fx_workspace")
    subprocess.check_call([NVCC, "-std=c++17", "-O1", "-o", exe, os.path.join(HOST, "fx_workspace.cu"), "-L" + lib,
                           "-llbo", "-Xlinker", "-rpath=" + lib])
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout
