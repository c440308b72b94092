"""The blind rotation with its leading transform stages on the tensor cores
(kernel shape 1 at N = 1024 and 2048) against the CUDA-core kernel (shape 0) on
the same inputs, accumulators word for word: every limb configuration and
arithmetic, odd row counts, single clusters up to blocks that take several jobs
side by side and from the counter, step limits, several keys and a rejected
table in one launch, persistent launches."""
import numpy as np
import pytest

from paper_2310_12441_gb300 import params as P
from paper_2310_12441_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

Q54, Q60 = P.KEYS_N1024.Q, P.KEYS_N2048.Q


def kp(N, Q, log2_B, n=5):
    return P.KeyParams(n=n, N=N, Q=Q, log2_B=log2_B, l_B=6, log2_Bks=4, l_ks=7)


# (ring degree, modulus, digit bits): 9-bit digits at Q < 2^54, 10-bit digits at
# both moduli
KEYS = [kp(1024, Q54, 9), kp(2048, Q54, 9), kp(2048, Q54, 10), kp(2048, Q60, 10)]


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_12441_gb300 import api as A
    A.load()
    yield A
    for N in (1024, 2048):
        A.set_kernel_shape(N, A.SHAPE_DEFAULT)


def inputs(api, ks, m, t, count, seed, vec):
    """Jobs over the keys in turn, uniform ciphertexts, random and identity tables."""
    rng = np.random.default_rng(seed)
    W = max(k.n for k in ks) + 1
    ki = np.arange(count) % len(ks)
    ct = np.stack([rng.integers(0, 2 * ks[k].N * m, W, dtype=np.uint64) for k in ki])
    luts, _ = synth.luts(t, count, seed, mix="mixed")
    jobs = api.make_jobs(ki, m, t, np.arange(count) * W, np.arange(count) * t, np.arange(count) * vec)
    return jobs, api.to_device_u64(ct.ravel()), luts


def rotate(api, eks, jobs, steps, d_in, d_lut, words, shape, N):
    api.set_kernel_shape(N, shape)
    out = torch.zeros(words, dtype=torch.int64, device="cuda")
    ws = api.workspace(api.bm_workspace_bytes(eks, jobs))
    api.bm_blind_rotate(eks, jobs, steps, d_in, d_lut, out, ws)
    torch.cuda.synchronize()
    status = api.bm_workspace_status(ws)
    api.set_kernel_shape(N, api.SHAPE_DEFAULT)
    return out, status


@pytest.mark.parametrize("m,count,steps", [(1, 1, 5), (3, 1, 5), (4, 3, 2), (1, 153, 5), (3, 306, 3), (2, 470, 5),
                                           (33, 2, 1), (2, 4, 0)])
@pytest.mark.parametrize("key", KEYS, ids=["N1024_Q54_B9", "N2048_Q54_B9", "N2048_Q54_B10", "N2048_Q60_B10"])
def test_rotation_equals_the_cuda_core_kernel(api, key, m, count, steps):
    t = 2 * key.N * m if count < 4 else 64
    _, ek = api.bm_keygen_seeded(key, 77)
    vec = m * 2 * key.N
    jobs, d_in, luts = inputs(api, [key], m, t, count, 1000 + m, vec)
    d_lut = api.to_device_u32(luts.ravel())
    want, s0 = rotate(api, [ek], jobs, steps, d_in, d_lut, count * vec, 0, key.N)
    got, s1 = rotate(api, [ek], jobs, steps, d_in, d_lut, count * vec, 1, key.N)
    assert s0 == s1 == 0
    assert torch.equal(got, want)


@pytest.mark.parametrize("key", [KEYS[0], KEYS[3]], ids=["N1024", "N2048"])
def test_several_keys_and_a_rejected_table(api, key):
    m, t, count = 2, 64, 330
    longer = P.KeyParams(**{**key.__dict__, "n": 7})
    ks = [key, longer, key]
    eks = [api.bm_keygen_seeded(k, 80 + i)[1] for i, k in enumerate(ks)]
    vec = m * 2 * key.N
    jobs, d_in, luts = inputs(api, ks, m, t, count, 5, vec)
    luts[17, 3] = (luts[17, 3] + 1) % t          # no longer negacyclic
    d_lut = api.to_device_u32(luts.ravel())
    want, s0 = rotate(api, eks, jobs, 100, d_in, d_lut, count * vec, 0, key.N)
    got, s1 = rotate(api, eks, jobs, 100, d_in, d_lut, count * vec, 1, key.N)
    assert s0 == s1 == -4
    assert torch.equal(got, want)
    assert not want[17 * vec:18 * vec].any() and want.any()


def test_persistent_classes_equal_one_block_per_job(api):
    """Both ring degrees in one persistent launch, m = 1 .. 5, whole bootstraps."""
    ks = [KEYS[0], KEYS[3]]
    eks = [api.bm_keygen_seeded(k, 90 + i)[1] for i, k in enumerate(ks)]
    count, t, W = 400, 64, 6
    rng = np.random.default_rng(3)
    jobs, d_in, luts = inputs(api, ks, 5, t, count, 6, W)
    jobs["m"] = rng.integers(1, 6, count)
    ct = np.stack([rng.integers(0, 2 * ks[j["key"]].N * int(j["m"]), W, dtype=np.uint64) for j in jobs])
    d_in, d_lut = api.to_device_u64(ct.ravel()), api.to_device_u32(luts.ravel())
    outs = []
    for shape, flags in ((0, api.BATCH_ONE_BLOCK), (1, api.BATCH_PERSISTENT)):
        for k in ks:
            api.set_kernel_shape(k.N, shape)
        out = torch.zeros(count * W, dtype=torch.int64, device="cuda")
        ws = api.workspace(api.bm_workspace_bytes(eks, jobs))
        b = api.Batch(eks, jobs, d_in, d_lut, out, ws, flags)
        b.run()
        b.run()
        torch.cuda.synchronize()
        assert api.bm_workspace_status(ws) == 0
        b.free()
        outs.append(out)
    assert torch.equal(outs[0], outs[1])
