"""What an index with a forward table computes in the very bits of one without,
for single requests: the wide term of every type and whole scores of FP32 tables.
The results of batches agree to rounding."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2511_22460_gb300 import ebr  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
N, N_KEYS = 30_001, 900


def _both(dtype, d):
    rng = np.random.default_rng(d)
    pk = rng.integers(0, N_KEYS, 14 * N).astype(np.uint32)
    pa = np.repeat(np.arange(N), 14).astype(np.uint32)
    emb = rng.standard_normal((N, d)).astype(np.float32)
    return [ebr.build_index(N, N_KEYS, pk, pa, emb, dtype=dtype, debug_faults=f)
            for f in (0, ebr.FAULT_FORWARD_MEM)]


@pytest.mark.parametrize("dtype,d", [("f32", 4), ("f32", 8), ("f32", 16), ("f32", 32), ("f32", 64),
                                     ("f32", 128), ("bf16", 64), ("fp8e4m3", 64)])
def test_single_requests(dtype, d):
    w = torch.randn(N_KEYS, device=DEV)
    w[::7] *= 1e-6  # terms of every class
    q = ebr.Query(h_u=torch.randn(d, device=DEV), q_w=w, k=1)
    wide, score = [], []
    for ix in _both(dtype, d):
        wide.append(torch.empty(N, device=DEV))
        score.append(torch.empty(N, device=DEV))
        # the scan writes the wide term of a quantised table; of an FP32 one, the score of h_u = 0
        zero = ebr.Query(h_u=torch.zeros(d, device=DEV), q_w=w, k=1)
        ebr.score_all(ix, None, zero, wide[-1])
        ebr.score_all(ix, None, q, score[-1])
    assert torch.equal(*wide)
    if dtype == "f32":
        assert torch.equal(*score)


@pytest.mark.parametrize("dtype,d", [("bf16", 64), ("bf16", 128), ("fp8e4m3", 64)])
def test_batches(dtype, d):
    B, k = 70, 200
    rng = np.random.default_rng(1)
    cross = ebr.cross_create([50], [N_KEYS], [(0, 0)],
                             (rng.standard_normal(1 << 16) * 0.3).astype(np.float32),
                             hashed=True, hash_bits=16)
    h = torch.randn((B, d), device=DEV)
    u = torch.from_numpy(rng.integers(0, 50, (B, 1)).astype(np.int32)).to(DEV)
    got = []
    for ix in _both(dtype, d):
        ids = torch.empty((B, k), dtype=torch.int32, device=DEV)
        sc = torch.empty((B, k), device=DEV)
        ebr.score_topk(ix, cross, [ebr.Query(h_u=h[b], k=k, user_vals=u[b]) for b in range(B)],
                       ids, sc)
        assert ix.profile_read().batched == B
        got.append((ids, sc))
    # (a walk's list order among its threads is not fixed: FP32 sums may differ in the last bits)
    assert torch.allclose(got[0][1], got[1][1], rtol=0, atol=1e-4)
    same = (got[0][0] == got[1][0]).float().mean()
    assert float(same) > 0.99
