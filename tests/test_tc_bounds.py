"""Ranges of the tensor-core transform stages at the smallest and largest moduli
that each limb configuration admits, with worst-case digits: limb sums exact in
fp32, values congruent to the exact sums, and E and O within what the stages
that follow need (no 64-bit wrap, below the bound the key's limbs are planned
for).  Host code only: the library's tables and recombination, compiled here."""
import os
import subprocess

import pytest

from paper_2310_12441_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
Q1, LAZY, TC1, TC2, WIDE = 1, 2, 4, 8, 16


def is_prime(n):
    d, s = n - 1, 0
    while d % 2 == 0:
        d, s = d // 2, s + 1
    for a in (2, 3, 5, 7, 11, 13, 17, 19, 23, 29, 31, 37):
        x = pow(a, d, n)
        if x in (1, n - 1):
            continue
        if not any((x := x * x % n) == n - 1 for _ in range(s - 1)):
            return False
    return True


def prime_at(limit, step):
    """The first prime c 2^32 + 1 from `limit` on (step 1) or below it (step -1)."""
    c = (limit - 1 >> 32) + (1 if step > 0 else 0)
    while not is_prime((c << 32) + 1):
        c += step
    return (c << 32) + 1


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("tc") / "tc_bounds")
    subprocess.run([B._nvcc(), *B.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-O1", "-I", B.CSRC, "-I", B.INCLUDE,
                    os.path.join(HERE, "native", "tc_bounds.cu"), "-o", exe], check=True)
    return exe


# (ring degree, digit bits, configuration, smallest and largest modulus): the
# lazy form from 2^58 / (1 + 4 log N) on, its limb sums below 15 2^56
KEYS = [(1024, 9, TC1, 2 ** 58 // 41, 2 ** 54), (2048, 9, TC1, 2 ** 58 // 45, 2 ** 54),
        (2048, 10, TC2, 2 ** 58 // 45, 15 * 2 ** 56 // 45), (2048, 10, TC2, 2 ** 58, 2 ** 60)]


@pytest.mark.parametrize("end", ["smallest", "largest", "middle"])
@pytest.mark.parametrize("N,bits,tc,low,high", KEYS)
def test_recombination_stays_in_range(prog, N, bits, tc, low, high, end):
    Q = {"smallest": prime_at(low, 1), "middle": prime_at((low + high) // 2, -1), "largest": prime_at(high, -1)}[end]
    out = subprocess.run([prog, str(N), str(Q), str(bits)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    variant, top, e0, e1, o0, o1 = map(int, out.stdout.split())
    assert variant & tc
    assert top <= 2 ** 24
    stages = N.bit_length() - 1 - 7
    if variant & LAZY:
        # X + T, X - T with T in [0, 4Q) in all stages but the last, X + 4Q - T there
        assert min(e0 + o0, e0 - o1) >= 4000 * (stages - 1)
        most = max(e1 + o1, e1 - o0) + 4000 * stages
        assert most <= 1000 * (1 + 4 * (stages + 7))
        assert most * Q < 1000 * 2 ** 60
        if N == 1024:        # whole rows of limb products in 64 bits
            assert most <= 26300
    else:
        # two stages, 8Q off values above 2^63, two stages
        assert min(e0 + o0, e0 - o1) >= 0
        first = (max(e1 + o1, e1 - o0) + 8000) * Q // 1000
        assert first < 2 ** 64
        assert max(2 ** 63, first - 8 * Q) + 8 * Q < 2 ** 64


@pytest.mark.parametrize("logN", range(8, 14))
def test_moduli_of_the_lazy_form_keep_it(prog, logN):
    """Every modulus c 2^32 + 1 with 2^58 < (1 + 4 log N) Q <= 2^60 has the lazy
    kernels of that form, with wider limbs from 15 2^56 on."""
    def variant(Q, bits):
        return int(subprocess.run([prog, str(1 << logN), str(Q), str(bits)], capture_output=True, text=True,
                                  check=True).stdout.split()[0])
    f = 1 + 4 * logN
    for Q, wide in ((prime_at(2 ** 58 // f + 1, 1), 0), (prime_at(15 * 2 ** 56 // f, -1), 0),
                    (prime_at(15 * 2 ** 56 // f + 1, 1), WIDE), (prime_at(2 ** 60 // f, -1), WIDE)):
        assert variant(Q, 15) == Q1 | LAZY | wide
