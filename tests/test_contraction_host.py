"""The exact split-integer contraction of FC lines (fc_split.cuh, fc_mmtab.h) on the CPU:
every inner length's tables and arithmetic, with the digit products in plain loops, against
the circulant of the spectral derivative (eq. fc_der) and of the filter (eq. filtering) in
long double.

Tolerance, relative to the line's largest value (coefficients at most about 1): the dropped
digit products are sums of 5 H pairs of digits of standard deviation 2^8.2 in units 2^40, the
largest value is at least 2^56 times a coefficient of 2^59.5: 2^-53.5 for H = 512; truncated
data and rounded coefficients add less. Eight times that, for the largest of all rows and
both parts, and one FP64 rounding: 2^-50.5 + 2^-52 < 9e-16. Level sums must stay below 2^24,
where FP32 accumulation stops being exact."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.isdir(CUDA_INC):
        pytest.skip("g++ and the CUDA headers are needed to build the host harness")
    out = str(tmp_path_factory.mktemp("mm") / "contraction_host")
    r = subprocess.run([gxx, "-O2", "-std=c++17", "-w", f"-I{CUDA_INC}", "-o", out,
                        os.path.join(ROOT, "tests", "contraction_host.cpp")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return out


# edges of the padding to 16, both parities, the shortest and the longest inner lengths
LENGTHS = [16, 17, 30, 31, 32, 33, 34, 37, 64, 66, 155, 192, 224, 255, 256, 258, 288, 432, 510, 512, 514, 509, 800, 1024]


def test_contraction_matches_the_circulant(exe):
    r = subprocess.run([exe, *map(str, LENGTHS)], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    rows = [ln.split() for ln in r.stdout.splitlines()]
    assert len(rows) == 6 * len(LENGTHS)
    for L, op, kind, err, level in rows:
        assert float(err) < 9e-16, (L, op, kind, err)
        assert float(level) < 2 ** 24, (L, op, kind, level)


def test_level_sums_are_exact_for_aligned_data(exe):
    """Lines made so that one of the levels 1 to 3 is as large as it can be. The bound of the module's
    head; results are up to 14 times the largest value here (the derivative's coefficients sum
    to that), so their own FP64 rounding counts 8 times: 2^-50.5 + 2^-50 (levels 4 and 5, whose
    digits are random here, stay exact)."""
    r = subprocess.run([exe, "aligned", "17", "30", "64", "155", "256", "400", "509", "510", "512", "800", "1024"],
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr
    rows = [ln.split() for ln in r.stdout.splitlines()]
    assert len(rows) == 3 * 6 + 8 * 12
    for L, op, level, part, err, largest in rows:
        assert float(largest) < 2 ** 24, (L, op, level, part, largest)
        assert float(err) < 2.0 ** -50.5 + 2.0 ** -50, (L, op, level, part, err)


def test_every_length_has_exact_tables(exe):
    lengths = [L for L in range(16, 1025) if L % 2 == 0 or L <= 512]
    r = subprocess.run([exe, "tables", *map(str, lengths)], capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and [ln.split() for ln in r.stdout.splitlines()] == [[str(L), "1", "1"] for L in lengths]


# broad kernels (many coefficients of one size), an amplifying one, small ones throughout; p = 0
# scales all modes alike
@pytest.mark.parametrize("alpha,p", [(2000, 2), (1700, 2), (50, 1), (1e6, 4), (0, 2), (-5, 2), (10, 0), (10, -1)])
def test_filters_of_any_width(exe, alpha, p):
    r = subprocess.run([exe, "filter", str(alpha), str(p), "17", "64", "255", "511", "512", "1024"],
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    rows = [ln.split() for ln in r.stdout.splitlines()]
    assert len(rows) == 18
    for L, op, kind, err, level in rows:
        assert float(err) < 9e-16, (L, op, kind, err)


def test_filters_out_of_range_are_left_to_the_transforms(exe):
    # sigma up to e^2000 and down to e^-2000: neither is an FP64 number
    for alpha, p in (("-2000", "2"), ("2000", "0")):
        r = subprocess.run([exe, "filter", alpha, p, "64", "512"], capture_output=True, text=True)
        assert r.returncode == 0 and [ln.split()[1] for ln in r.stdout.splitlines()] == ["none"] * 2


def test_other_lengths_are_left_to_the_transforms(exe):
    r = subprocess.run([exe, "15", "513", "1026", "2048"], capture_output=True, text=True)
    assert r.returncode == 0 and [ln.split()[1] for ln in r.stdout.splitlines()] == ["none"] * 4


def test_quotients_round_as_the_division(exe):
    # the classifier's normalised values (bit for bit)
    r = subprocess.run([exe, "quotient"], capture_output=True, text=True, timeout=600)
    n, bad = map(int, r.stdout.split())
    assert r.returncode == 0 and n > 10 ** 7 and bad == 0, (n, bad)


@pytest.mark.parametrize("C,Q", [(27, 10), (32, 10), (71, 10), (33, 4), (128, 16)])
def test_continuation_products(exe, C, Q):
    # relative to the largest weighted end value: at most 16 values of 57 bits truncated (2^-57 each,
    # coefficients below 1), five levels of dropped products (2^-54.8 at eight deviations of 80 pairs):
    # below 2^-52.5 in all; and one FP64 rounding of a sum of up to Q such values, Q 2^-53
    r = subprocess.run([exe, "continuation", str(C), str(Q)], capture_output=True, text=True)
    assert r.returncode == 0 and float(r.stdout) < 2.0 ** -52.5 + Q * 2.0 ** -53, r.stdout
