"""The transforms on pairs of components, run on the CPU (no GPU needed).

`tests/native/fft_pair_host.cu` runs the kernels' own __host__ __device__ code with one cooperative fiber
per GPU lane, each lane as far as the next barrier lets it, in ascending and in descending order: a
shared-memory access that no barrier separates from another lane's write of the same place gives a wrong
result in one of the two. Covered: RegPlan::run on pairs (contiguous and strided lines),
run_regrouped at both exchanges with the rows of a row stage side by side, Fft16, and the inverse row transform of
FFT length 768 with the combination of its three residues.

Tolerance 1e-6 of the output's norm: FP32 rounding (6e-8) over at most four passes of at most four
roundings each, the bound of the plans' host test on single components."""
import os
import subprocess

import numpy as np
import pytest

from test_fft_reg_host import _nvcc

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "native", "fft_pair_host.cu")
RUN, STRIDED, FIRST, LAST, SIXTEEN, ROWS768 = range(6)


@pytest.fixture(scope="module")
def records(tmp_path_factory):
    cc = _nvcc()
    if cc is None:
        pytest.skip("nvcc not available")
    out = tmp_path_factory.mktemp("fft_pair_host")
    exe, path = str(out / "fft_pair_host"), str(out / "out.bin")
    cmd = [cc, "-std=c++20", "-O0", "--expt-relaxed-constexpr", "-diag-suppress", "20014",
           "-gencode", "arch=compute_103a,code=sm_103a", SRC, "-o", exe]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    res = subprocess.run([exe, path], capture_output=True, text=True, timeout=120)
    assert res.returncode == 0, res.stderr
    blob, off, recs = open(path, "rb").read(), 0, []
    while off < len(blob):
        head = tuple(int(v) for v in np.frombuffer(blob, np.int32, 8, off))
        n_in, n_out = head[6:]
        x = np.frombuffer(blob, np.complex128, n_in, off + 32)
        y = np.frombuffer(blob, np.complex128, n_out, off + 32 + 16 * n_in)
        off += 32 + 16 * (n_in + n_out)
        recs.append((*head[:6], x, y))
    return recs


@pytest.mark.parametrize("descending", [0, 1], ids=["ascending", "descending"])
@pytest.mark.parametrize("kind", [RUN, STRIDED, FIRST, LAST, SIXTEEN, ROWS768],
                         ids=["run", "strided", "regrouped_first", "regrouped_last", "sixteen", "rows_768"])
def test_pair_transforms_equal_the_dft(records, kind, descending):
    mine = [r for r in records if r[0] == kind and r[5] == descending]
    lengths = {RUN: {16, 32, 64, 128, 256, 512}, STRIDED: {16, 32, 64, 128}, FIRST: {16, 32, 64, 128, 256, 512},
               LAST: {16, 32, 64, 128, 256, 512}, SIXTEEN: {32, 64, 128, 256}, ROWS768: {768}}[kind]
    assert {r[1] for r in mine} == lengths
    for _, L, V, inv, _, _, x, y in mine:
        want = (L * np.fft.ifft(x) if inv else np.fft.fft(x))[:len(y)]
        err = np.linalg.norm(y - want) / np.linalg.norm(want)
        assert err <= 1e-6, (L, V, inv, err)
