"""Moduli Q = c 2^32 + 1 whose lazy transform values pass 15 2^56 (a band below
2^60 / (1 + 4 log2 N)): the kernels of that form with 30-bit limbs, bit-exact
with the oracle in every launch form."""
import numpy as np
import pytest

from paper_2310_12441_gb300 import params as P
from paper_2310_12441_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# the first and last primes of the band
BAND = {256: (32753463548968961, 34936990562516993), 1024: (26362629521932289, 28119687757824001),
        2048: (24019419919286273, 25620429108412417), 4096: (22058479585853441, 23528994783625217),
        8192: (20393668657545217, 21753219080257537)}


@pytest.mark.parametrize("N", BAND)
@pytest.mark.parametrize("end", [0, 1], ids=["first", "last"])
@pytest.mark.parametrize("log2_B,l_B", [(10, 6), (15, 4)])
def test_band_matches_the_oracle(orc, N, end, log2_B, l_B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_12441_gb300 import api
    kp = P.KeyParams(n=2, N=N, Q=BAND[N][end], log2_B=log2_B, l_B=l_B, log2_Bks=2, l_ks=3)
    m, t, cnt, seed, W = (1, 32, 2, 5, 3) if N > 1024 else (3, 32, 3, 5, 3)
    qp = 2 * N * m
    sk, ek = api.bm_keygen_seeded(kp, seed)
    rnd = orc.seeded_key_randomness(kp, seed, bsk_keys=kp.n)
    bsk, ksk = orc.keygen_bsk(kp, rnd), orc.keygen_ksk(kp, rnd)
    ct = api.bm_encrypt_seeded(sk, qp, t, synth.messages(t, cnt, seed), seed + 1)
    luts, _ = synth.luts(t, cnt, seed + 2)
    want = orc.bootstrap(kp, m, t, bsk, ksk, ct, luts)
    jobs = api.make_jobs(0, m, t, np.arange(cnt) * W, np.arange(cnt) * t, np.arange(cnt) * W)
    d_in, d_lut = api.to_device_u64(ct.ravel()), api.to_device_u32(luts.ravel())
    for shape in api.kernel_shapes(N):
        api.set_kernel_shape(N, shape)
        for flags in (0, api.BATCH_ONE_BLOCK, api.BATCH_PERSISTENT):
            out = torch.zeros(cnt * W, dtype=torch.int64, device="cuda")
            ws = api.workspace(api.bm_workspace_bytes([ek], jobs))
            b = api.Batch([ek], jobs, d_in, d_lut, out, ws, flags)
            b.run()
            torch.cuda.synchronize()
            b.free()
            assert api.bm_workspace_status(ws) == 0
            assert np.array_equal(api.from_device_u64(out).reshape(cnt, W), want), (shape, flags)
    api.set_kernel_shape(N, api.SHAPE_DEFAULT)
