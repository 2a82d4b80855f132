"""The batched scan's three sources of an ad's keys (the walk over the window's
blocks, the forward table, the forward table with w^T in shared memory) at the
edges of their user groups, windows and key spaces: every user's top-K against
FP64 sums of the same weights (Eq. 1 + the HitMatch equation)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import oracle  # noqa: E402
from gpu_util import check_topk  # noqa: E402
from paper_2511_22460_gb300 import ebr  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _postings(n_ads, n_keys, most, even, rng):
    # uneven: one ad of each run has `most` keys, the others one (no forward table)
    cnt = np.full(n_ads, most) if even else np.where(np.arange(n_ads) % 32 == 5, most, 1)
    ad = np.repeat(np.arange(n_ads), cnt)
    nth = np.concatenate([np.arange(c) for c in cnt])
    key = (rng.integers(0, n_keys, n_ads)[ad] + nth * max(1, n_keys // (most + 1))) % n_keys
    return np.ascontiguousarray(np.unique(np.stack([key, ad]), axis=1).astype(np.uint32))


@pytest.mark.parametrize("n_ads,n_keys,most,even,d,dtype,B,k", [
    (127, 60, 3, True, 64, "bf16", 2, 10),         # w^T in shared memory, less than a window
    (20_000, 500, 32, True, 64, "fp8e4m3", 64, 300),
    (20_001, 500, 32, True, 64, "bf16", 65, 300),   # a second group of one user
    (9_000, 600, 17, True, 128, "bf16", 130, 200),  # w^T gathered from global memory
    (30_011, 70_000, 24, True, 64, "bf16", 256, 500),   # keys of 24 bits
    (12_345, 70_000, 9, True, 128, "fp8e4m3", 63, 700),
    (8_000, 900, 60, True, 64, "fp8e4m3", 33, 100),
    (9_999, 300, 40, False, 64, "bf16", 70, 400),   # the walk (no forward table)
    (5_000, 70_000, 40, False, 128, "fp8e4m3", 20, 300),
])
def test_every_user_of_a_batch(n_ads, n_keys, most, even, d, dtype, B, k):
    rng = np.random.default_rng(n_ads + B)
    pk, pa = _postings(n_ads, n_keys, most, even, rng)
    emb = (rng.standard_normal((n_ads, d)) / np.sqrt(d)).astype(np.float32)
    h = (rng.standard_normal((B, d)) / np.sqrt(d)).astype(np.float32)
    users = rng.integers(0, 50, (B, 1)).astype(np.uint32)
    ix = ebr.build_index(n_ads, n_keys, pk, pa, emb, dtype=dtype)
    cross = ebr.cross_create([50], [n_keys], [(0, 0)],
                             (rng.standard_normal(1 << 16) * 0.3).astype(np.float32),
                             hashed=True, hash_bits=16)
    w = torch.empty((B, n_keys), device=DEV)
    ebr.expand_query(cross, _dev(users.view(np.int32)), w)
    w = w.cpu().numpy().astype(np.float64)
    n_filt = B // 3
    masks = [rng.random(n_ads) < rng.uniform(0.05, 1.0) if b < n_filt else None for b in range(B)]

    def words(m):
        bits = np.zeros((n_ads + 63) // 64 * 64, bool)
        bits[:n_ads] = m
        return _dev(np.packbits(bits, bitorder="little").view(np.int64))

    qs = [ebr.Query(h_u=_dev(h[b]), k=k if b % 2 else max(1, k // 7),
                    user_vals=_dev(users[b].view(np.int32)),
                    filter=None if masks[b] is None else words(masks[b])) for b in range(B)]
    ids = torch.empty((B, k), dtype=torch.int32, device=DEV)
    sc = torch.empty((B, k), device=DEV)
    before = ix.profile_read()
    ebr.score_topk(ix, cross, qs, ids, sc)
    after = ix.profile_read()
    assert after.batched - before.batched == B and after.recomputed == before.recomputed
    ids, sc = ids.cpu().numpy().view(np.uint32), sc.cpu().numpy()
    e64 = emb.astype(np.float64)
    for b in range(B):
        wide, mag = np.zeros(n_ads), np.zeros(n_ads)
        np.add.at(wide, pa, w[b][pk])
        np.add.at(mag, pa, np.abs(w[b][pk]))
        ref = e64 @ h[b].astype(np.float64) + wide
        tol = oracle.tolerance(ref, np.abs(e64) @ np.abs(h[b]).astype(np.float64) + mag, 1e-5)
        kb = qs[b].k
        check_topk(ids[b, :kb], sc[b, :kb], ref, tol, kb, masks[b])
        assert np.all(ids[b, kb:] == 0xFFFFFFFF) and np.all(np.isneginf(sc[b, kb:]))


def test_waves_wider_than_two_groups():
    """A server whose user table is not a power of two of groups wide: 600
    requests at once, each with the result that a batched call gives it."""
    n_ads, n_keys, B, k = 1_000_000, 3000, 150, 50
    rng = np.random.default_rng(5)
    pk, pa = _postings(n_ads, n_keys, 4, True, rng)
    emb = (rng.standard_normal((n_ads, 64)) / 8).astype(np.float32)
    h = (rng.standard_normal((B, 64)) / 8).astype(np.float32)
    users = rng.integers(0, 50, (B, 1)).astype(np.uint32)
    ix = ebr.build_index(n_ads, n_keys, pk, pa, emb, dtype="bf16")
    cross = ebr.cross_create([50], [n_keys], [(0, 0)],
                             (rng.standard_normal(1 << 16) * 0.3).astype(np.float32),
                             hashed=True, hash_bits=16)
    hd, ud = _dev(h), _dev(users.view(np.int32))
    ids = torch.empty((B, k), dtype=torch.int32, device=DEV)
    sc = torch.empty((B, k), device=DEV)
    ebr.score_topk(ix, cross, [ebr.Query(h_u=hd[b], k=k, user_vals=ud[b]) for b in range(B)],
                   ids, sc)
    torch.cuda.synchronize()
    ids, sc = ids.cpu().numpy().view(np.uint32), sc.cpu().numpy()
    srv = ebr.Server(ix, cross, max_batch=B, max_slots=4 * B, k_max=k)
    try:
        tickets = [srv.submit(h[i % B], users[i % B], k) for i in range(4 * B)]
        for i, t in enumerate(tickets):
            gi, gs = srv.wait(t, k)
            b = i % B
            # the same FP32 rescoring; an FP32 sum of 68 terms below 2 orders ties
            assert np.max(np.abs(gs - sc[b])) <= 68 * 2.0 ** -22
            assert np.intersect1d(gi, ids[b]).size >= k - 1
        print("requests per wave: %.1f" % (4 * B / srv.stats().batches))
    finally:
        srv.close()
