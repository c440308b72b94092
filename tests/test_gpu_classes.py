"""A persistent batch with a key of every (ring degree, arithmetic variant)
class, 19 in one launch sequence: accepted, and the same words as one block per
job."""
import numpy as np
import pytest

from paper_2310_12441_gb300 import params as P
from paper_2310_12441_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

Q54, Q60 = P.KEYS_N1024.Q, P.KEYS_N2048.Q          # c 2^32 + 1
G54, G59 = 18014398509309953, 576460752303415297    # 1 mod 8192, no such form

WIDE = {1024: 28119687757824001, 2048: 25620429108412417, 4096: 23528994783625217}    # lazy, 30-bit limbs

# per ring degree (modulus, digit bits, digits): lazy and corrected transforms
# with and without the form c 2^32 + 1, then the tensor-core configurations
COMMON = [(Q54, 15, 4), (Q60, 8, 8), (G54, 9, 6), (G59, 15, 4)]
CLASSES = [(1024, *k) for k in COMMON + [(Q54, 9, 6)]] + \
    [(2048, *k) for k in COMMON + [(Q54, 9, 6), (Q54, 10, 6), (Q60, 10, 6)]] + [(4096, *k) for k in COMMON] + \
    [(N, Q, 10, 6) for N, Q in WIDE.items()]


def test_one_key_of_every_class():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_12441_gb300 import api
    keys = [P.KeyParams(n=2, N=N, Q=Q, log2_B=b, l_B=l, log2_Bks=2, l_ks=2) for N, Q, b, l in CLASSES]
    eks = [api.bm_keygen_seeded(k, 20 + i)[1] for i, k in enumerate(keys)]
    count, t, W = len(keys), 64, 3
    rng = np.random.default_rng(1)
    ct = np.stack([rng.integers(0, 2 * k.N, W, dtype=np.uint64) for k in keys])
    luts, _ = synth.luts(t, count, 2, mix="mixed")
    jobs = api.make_jobs(np.arange(count), 1, t, np.arange(count) * W, np.arange(count) * t, np.arange(count) * W)
    d_in, d_lut = api.to_device_u64(ct.ravel()), api.to_device_u32(luts.ravel())
    outs = []
    for flags in (api.BATCH_ONE_BLOCK, api.BATCH_PERSISTENT):
        out = torch.zeros(count * W, dtype=torch.int64, device="cuda")
        ws = api.workspace(api.bm_workspace_bytes(eks, jobs))
        b = api.Batch(eks, jobs, d_in, d_lut, out, ws, flags)
        for _ in range(2):
            b.run()
        torch.cuda.synchronize()
        assert api.bm_workspace_status(ws) == 0
        b.free()
        outs.append(out)
    assert torch.equal(outs[0], outs[1])
