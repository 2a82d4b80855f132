"""Requests of different sizes from two threads at once, each on an index and a
stream of its own: every call succeeds and gives what it gave alone."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2511_22460_gb300 import ebr  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _side(n, k, B, dtype, seed):
    rng = np.random.default_rng(seed)
    n_keys, d = 600, 64
    pk = rng.integers(0, n_keys, 6 * n).astype(np.uint32)
    pa = np.repeat(np.arange(n), 6).astype(np.uint32)
    emb = rng.standard_normal((n, d)).astype(np.float32)
    ix = ebr.build_index(n, n_keys, pk, pa, emb, dtype=dtype)
    cross = ebr.cross_create([9], [n_keys], [(0, 0)],
                             (rng.standard_normal(1 << 12) * 0.3).astype(np.float32),
                             hashed=True, hash_bits=12)
    h = torch.from_numpy(rng.standard_normal((B, d)).astype(np.float32)).to(DEV)
    u = torch.from_numpy(rng.integers(0, 9, (B, 1)).astype(np.int32)).to(DEV)
    qs = [ebr.Query(h_u=h[b], k=k, user_vals=u[b]) for b in range(B)]
    st = torch.cuda.Stream()
    ids = torch.empty((B, k), dtype=torch.int32, device=DEV)
    sc = torch.empty((B, k), device=DEV)
    torch.cuda.synchronize()

    def call():
        ebr.score_topk(ix, cross, qs, ids, sc, stream=st)

    def result():
        st.synchronize()
        return ids.cpu(), sc.cpu()
    return call, result


@pytest.mark.parametrize("dtype,B,sizes", [
    ("f32", 1, ((20_000, 4000), (20_000, 1))),      # candidate buffers of different sizes
    ("bf16", 4, ((6_000, 2000), (6_000, 5))),       # merges of different depths
])
def test_calls_of_two_threads(dtype, B, sizes):
    sides = [_side(n, k, B, dtype, i) for i, (n, k) in enumerate(sizes)]
    want = []
    for call, result in sides:
        call()
        want.append(result())
    errors = []

    def work(call):
        try:
            for _ in range(4000):
                call()
        except Exception as e:  # reported below
            errors.append(e)

    threads = [threading.Thread(target=work, args=(call,)) for call, _ in sides]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
    for (call, result), (ids, sc) in zip(sides, want):
        got = result()
        assert torch.equal(got[0], ids) and torch.equal(got[1], sc)
