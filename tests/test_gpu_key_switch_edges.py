"""The tiled key switch at the edges of its tiles, for every number of samples per
thread: counts one below, at and one above whole tiles that the launch rule
(compiled here) gives to that many, word for word against calls too small for
tiles."""
import os
import subprocess

import numpy as np
import pytest

from paper_2310_12441_gb300 import build as B
from paper_2310_12441_gb300 import params as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))
KEY = P.KeyParams(n=1000, N=256, Q=P.KEYS_N1024.Q, log2_B=9, l_B=6, log2_Bks=4, l_ks=7)


@pytest.fixture(scope="module")
def setup(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_12441_gb300 import api
    exe = str(tmp_path_factory.mktemp("ks") / "ks_plan")
    subprocess.run([B._nvcc(), *B.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-O1", "-I", B.CSRC, "-I", B.INCLUDE,
                    os.path.join(HERE, "native", "ks_plan.cu"), "-o", exe], check=True)
    sms = torch.cuda.get_device_properties(0).multi_processor_count

    def samples_per_thread(count):
        out = subprocess.run([exe, str(sms), *map(str, (KEY.n, KEY.N, KEY.log2_Bks, KEY.l_ks, count))],
                             capture_output=True, text=True, check=True).stdout
        return int(out.split(":")[2])

    return api, api.bm_keygen_seeded(KEY, 33)[1], sms, samples_per_thread


@pytest.mark.parametrize("edge", [-1, 0, 1])
@pytest.mark.parametrize("cpt", [4, 8, 12, 16, 20, 24])
def test_edges_of_tiles(setup, cpt, edge):
    api, ek, sms, samples_per_thread = setup
    count = next(c for k in range(1, 40) if (c := 8 * cpt * k + edge) > sms and samples_per_thread(c) == cpt)
    rng = np.random.default_rng(count)
    d = api.to_device_u64(rng.integers(0, KEY.Q, count * (KEY.N + 1), dtype=np.uint64))
    got = torch.full((count * (KEY.n + 1),), -1, dtype=torch.int64, device="cuda")
    want = torch.full_like(got, -2)
    api.bm_key_switch(ek, d, count, got)
    small = sms // 2
    assert samples_per_thread(small) == 0
    for a in range(0, count, small):
        c = min(small, count - a)
        api.bm_key_switch(ek, d[a * (KEY.N + 1):], c, want[a * (KEY.n + 1):])
    torch.cuda.synchronize()
    assert torch.equal(got, want)
