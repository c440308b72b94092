"""The key switch's launches for batches of several keys: the cheapest sequence of
tile and block launches by the measured costs, against every other one."""
import os
import subprocess

import numpy as np
import pytest

from paper_2310_12441_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
N1024 = (630, 1024, 4, 7)


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("ks") / "ks_plan")
    subprocess.run([B._nvcc(), *B.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-O1", "-I", B.CSRC, "-I", B.INCLUDE,
                    os.path.join(HERE, "native", "ks_plan.cu"), "-o", exe], check=True)
    return exe


def launches(prog, runs, sms=152):
    args = [str(v) for r in runs for v in r]
    out = subprocess.run([prog, str(sms), *args], capture_output=True, text=True)
    assert out.returncode == 0, (out.returncode, runs)
    return [tuple(map(int, line.split(":"))) for line in out.stdout.split()]


@pytest.mark.parametrize("keys,per", [(30, 80), (30, 77), (8, 150), (12, 100)])
def test_runs_of_less_than_a_gpu_stay_in_one_launch(prog, keys, per):
    assert launches(prog, [(*N1024, per)] * keys) == [(0, keys * per, 0)]


def test_long_runs_take_tiles(prog):
    got = launches(prog, [(*N1024, 1200)] * 2)
    assert [g[:2] for g in got] == [(0, 1200), (1200, 1200)] and all(g[2] for g in got)
    got = launches(prog, [(*N1024, 2), (*N1024, 515), (*N1024, 3), (*N1024, 5)])
    assert [g[:2] for g in got] == [(0, 2), (2, 515), (517, 8)] and [g[2] > 0 for g in got] == [False, True, False]


@pytest.mark.parametrize("seed", range(40))
def test_no_other_sequence_is_cheaper(prog, seed):
    rng = np.random.default_rng(seed)
    shapes = [N1024, (750, 2048, 4, 7), (64, 256, 4, 7), (512, 512, 5, 8), (830, 256, 7, 4), (17, 256, 8, 3)]
    runs = [(*shapes[rng.integers(len(shapes))], int(2 ** rng.uniform(0, 11))) for _ in range(rng.integers(1, 11))]
    launches(prog, runs, int(rng.choice([152, 148, 60])))
