"""The tensor-core transform stages at the smallest moduli that their limb
configurations admit, against the CUDA-core kernel on the same inputs,
accumulators word for word."""
import numpy as np
import pytest

from paper_2310_12441_gb300 import params as P
from paper_2310_12441_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# the first primes c 2^32 + 1 with (1 + 4 log2 N) Q > 2^58, and at 2^58
Q_1024, Q_2048, Q_58 = 7030028239896577, 6405308066824193, 288230449166155777


@pytest.mark.parametrize("N,Q,log2_B", [(1024, Q_1024, 9), (2048, Q_2048, 9), (2048, Q_2048, 10), (2048, Q_58, 10)])
@pytest.mark.parametrize("m,count", [(3, 1), (2, 310)])
def test_smallest_moduli(N, Q, log2_B, m, count):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_12441_gb300 import api
    key = P.KeyParams(n=6, N=N, Q=Q, log2_B=log2_B, l_B=6, log2_Bks=4, l_ks=3)
    _, ek = api.bm_keygen_seeded(key, 8)
    W, t, vec = key.n + 1, 64, m * 2 * N
    rng = np.random.default_rng(count)
    ct = rng.integers(0, 2 * N * m, (count, W), dtype=np.uint64)
    luts, _ = synth.luts(t, count, 4, mix="mixed")
    jobs = api.make_jobs(0, m, t, np.arange(count) * W, np.arange(count) * t, np.arange(count) * vec)
    d_in, d_lut = api.to_device_u64(ct.ravel()), api.to_device_u32(luts.ravel())
    outs = []
    for shape in (0, 1):
        api.set_kernel_shape(N, shape)
        out = torch.zeros(count * vec, dtype=torch.int64, device="cuda")
        ws = api.workspace(api.bm_workspace_bytes([ek], jobs))
        api.bm_blind_rotate([ek], jobs, key.n, d_in, d_lut, out, ws)
        torch.cuda.synchronize()
        assert api.bm_workspace_status(ws) == 0
        outs.append(out)
    api.set_kernel_shape(N, api.SHAPE_DEFAULT)
    assert torch.equal(outs[0], outs[1])
