"""The key switch of many samples of one key (tiles of samples by columns)
against the kernel with one block per sample, word for word: the same samples
in one call and in calls too small for the tiles.  Counts around the tiles'
edges, columns that fill, exceed or miss a slice, digit widths with one or
several stages per coefficient and one too wide for the tiles; and the sample
extraction of bootstraps, with runs of several keys in one launch."""
import numpy as np
import pytest

from paper_2310_12441_gb300 import params as P
from paper_2310_12441_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

Q54 = P.KEYS_N1024.Q
SMALL = 60      # samples per call that never take the tiles


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_12441_gb300 import api as A
    A.load()
    return A


def kp(n, N, log2_Bks, l_ks):
    return P.KeyParams(n=n, N=N, Q=Q54, log2_B=9, l_B=6, log2_Bks=log2_Bks, l_ks=l_ks)


@pytest.mark.parametrize("count", [255, 256, 257, 511, 700, 2049])
@pytest.mark.parametrize("n,N,log2_Bks,l_ks", [(63, 256, 4, 7), (512, 512, 5, 8), (830, 256, 7, 4), (130, 1024, 1, 16),
                                               (17, 256, 8, 3), (1030, 256, 3, 9)])
def test_tiles_equal_single_samples(api, n, N, log2_Bks, l_ks, count):
    key = kp(n, N, log2_Bks, l_ks)
    _, ek = api.bm_keygen_seeded(key, 31)
    rng = np.random.default_rng(count)
    x = rng.integers(0, key.Q, (count, N + 1), dtype=np.uint64)
    x[0], x[1], x[-1] = 0, key.Q - 1, key.Q // 2
    d = api.to_device_u64(x.ravel())
    got = torch.full((count * (n + 1),), -1, dtype=torch.int64, device="cuda")
    want = torch.full_like(got, -2)
    api.bm_key_switch(ek, d, count, got)
    for a in range(0, count, SMALL):
        c = min(SMALL, count - a)
        api.bm_key_switch(ek, d[a * (N + 1):], c, want[a * (n + 1):])
    torch.cuda.synchronize()
    assert torch.equal(got, want)


@pytest.mark.parametrize("counts", [(300,), (290, 3), (2, 515), (280, 290, 40)])
def test_bootstraps_of_several_keys(api, counts):
    """Jobs in runs of one key: long runs take the tiles, short ones do not."""
    keys = [kp(5 + i, 1024, 4, 7) for i in range(len(counts))]
    eks = [api.bm_keygen_seeded(k, 40 + i)[1] for i, k in enumerate(keys)]
    count, m, t = sum(counts), 2, 64
    ki = np.repeat(np.arange(len(counts)), counts)
    W = max(k.n for k in keys) + 1
    rng = np.random.default_rng(count)
    ct = rng.integers(0, 2 * 1024 * m, (count, W), dtype=np.uint64)
    luts, _ = synth.luts(t, count, 9, mix="mixed")
    d_in, d_lut = api.to_device_u64(ct.ravel()), api.to_device_u32(luts.ravel())

    def run(lo, hi, out):
        i = np.arange(lo, hi)
        jobs = api.make_jobs(ki[i], m, t, i * W, i * t, i * W)
        ws = api.workspace(api.bm_workspace_bytes(eks, jobs))
        api.bm_bootstrap_batch(eks, jobs, d_in, d_lut, out, ws)
        torch.cuda.synchronize()

    got = torch.zeros(count * W, dtype=torch.int64, device="cuda")
    want = torch.zeros_like(got)
    run(0, count, got)
    for a in range(0, count, SMALL):
        run(a, min(a + SMALL, count), want)
    assert torch.equal(got, want)
