"""The last selection of a request and the allocation-free scan, on scores that
are known exactly (h_u or the table zero but for one element): every id and
score must equal the sort's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2511_22460_gb300 import ebr  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
INF = float("inf")


def _scores(kind, n, rng):
    s = rng.standard_normal(n).astype(np.float32)
    if kind == "equal":
        s[:] = 0.5
    elif kind == "few":  # more equal scores at the cut than a bin may hold
        s = rng.integers(0, 4, n).astype(np.float32)
    elif kind == "inf":  # no finite range
        s[rng.integers(0, n, 1 + n // 50)] = INF
        s[rng.integers(0, n, 1 + n // 3)] = -INF
    elif kind == "outlier":  # one score far away: the others share a bin
        s[n // 2] = 3e38
        s[n // 3] = -3e38
    elif kind == "subnormal":
        s = (rng.integers(-5000, 5000, n) * 1e-44).astype(np.float32)
    elif kind == "rising":
        s = np.arange(n, dtype=np.float32) - n / 2
    return s


def _want(s, k, mask=None):
    ids = np.lexsort((np.arange(s.size), -s.astype(np.float64)))
    if mask is not None:
        ids = ids[mask[ids]]
    ids = ids[:k]
    pad = k - ids.size
    return (np.concatenate([ids, np.full(pad, 0xFFFFFFFF)]).astype(np.uint32),
            np.concatenate([s[ids], np.full(pad, -INF, np.float32)]))


def _noalloc(s, k, d, mask=None):
    n = s.size
    emb = torch.full((n, d), 2.0, device=DEV)
    h = torch.zeros(d, device=DEV)
    filt = None
    if mask is not None:
        bits = np.zeros((n + 63) // 64 * 64, bool)
        bits[:n] = mask
        filt = torch.from_numpy(np.packbits(bits, bitorder="little").view(np.int64)).to(DEV)
    ids = torch.full((k,), -7, dtype=torch.int32, device=DEV)
    sc = torch.full((k,), float("nan"), device=DEV)
    ebr.scan_topk_noalloc(emb, h, torch.from_numpy(s).to(DEV), filt, k, ids, sc)
    torch.cuda.synchronize()
    return ids.cpu().numpy().view(np.uint32), sc.cpu().numpy()


@pytest.mark.parametrize("kind", ["normal", "equal", "few", "inf", "outlier", "subnormal", "rising"])
@pytest.mark.parametrize("n,k,d", [(1, 1, 4), (1, 5, 128), (31, 64, 8), (700, 700, 16),
                                   (1025, 1024, 32), (12_288, 1000, 8), (12_289, 7, 8),
                                   (70_001, 1000, 4), (200_033, 1024, 64)])
def test_noalloc_selects_what_a_sort_does(kind, n, k, d):
    rng = np.random.default_rng(n + k)
    s = _scores(kind, n, rng)
    for mask in (None, rng.random(n) < 0.3):
        ids, sc = _noalloc(s, k, d, mask)
        want, want_sc = _want(s, k, mask)
        assert np.array_equal(ids, want) and np.array_equal(sc, want_sc)


@pytest.mark.parametrize("kind", ["normal", "equal", "few", "outlier", "rising"])
@pytest.mark.parametrize("n,k", [(9_000, 8192), (300, 8192), (12_288, 8192), (12_289, 50), (150_000, 8191), (150_000, 2049), (800_000, 20)])
def test_request_selects_what_a_sort_does(kind, n, k):
    rng = np.random.default_rng(n + k)
    s = _scores(kind, n, rng)
    emb = np.zeros((n, 4), np.float32)
    emb[:, 1] = s
    ix = ebr.build_index(n, 4, np.zeros(0, np.uint32), np.zeros(0, np.uint32), emb)
    h = torch.tensor([0.0, 1.0, 0.0, 0.0], device=DEV)
    ids = torch.full((k,), -7, dtype=torch.int32, device=DEV)
    sc = torch.full((k,), float("nan"), device=DEV)
    ebr.score_topk(ix, None, [ebr.Query(h_u=h, k=k, q_w=torch.zeros(4, device=DEV))], ids, sc)
    torch.cuda.synchronize()
    want, want_sc = _want(s, k)
    assert np.array_equal(ids.cpu().numpy().view(np.uint32), want)
    assert np.array_equal(sc.cpu().numpy(), want_sc)


@pytest.mark.parametrize("d", [4, 8, 16, 32, 64, 128])
@pytest.mark.parametrize("n", [1, 33, 5_003, 300_000])
def test_noalloc_inner_products(n, d):
    """Against FP64, within d roundings of the sum of the products' sizes."""
    rng = np.random.default_rng(n + d)
    emb = rng.standard_normal((n, d)).astype(np.float32)
    h = rng.standard_normal(d).astype(np.float32)
    wide = rng.standard_normal(n).astype(np.float32)
    k = min(n, 600)
    ids = torch.empty(k, dtype=torch.int32, device=DEV)
    sc = torch.empty(k, device=DEV)
    ebr.scan_topk_noalloc(torch.from_numpy(emb).to(DEV), torch.from_numpy(h).to(DEV),
                          torch.from_numpy(wide).to(DEV), None, k, ids, sc)
    torch.cuda.synchronize()
    ids, sc = ids.cpu().numpy(), sc.cpu().numpy().astype(np.float64)
    prod = emb.astype(np.float64) * h
    ref = prod.sum(1) + wide
    tol = (np.abs(prod).sum(1) + np.abs(wide)) * (d + 1) * 2.0 ** -24
    assert np.unique(ids).size == k
    assert np.all(np.abs(sc - ref[ids]) <= tol[ids])
    left = np.setdiff1d(np.arange(n), ids)
    if left.size:
        assert np.all(ref[left] - tol[left] <= sc[-1])
    assert np.all(np.diff(sc) <= 0)


@pytest.mark.parametrize("kind", ["normal", "equal", "few", "outlier", "rising"])
@pytest.mark.parametrize("n,k,B", [(5_000, 100, 3), (40, 64, 2), (9_000, 2000, 160), (200_000, 50, 64)])
def test_batch_selects_what_a_sort_does(kind, n, k, B):
    rng = np.random.default_rng(n + k)
    s = torch.from_numpy(_scores(kind, n, rng)).bfloat16().float().numpy()  # exact in the table
    emb = np.zeros((n, 64), np.float32)
    emb[:, 1] = s
    ix = ebr.build_index(n, 4, np.array([3], np.uint32), np.array([0], np.uint32), emb,
                         dtype="bf16")
    cross = ebr.cross_create([2], [4], [(0, 0)], np.zeros(16, np.float32), hashed=True, hash_bits=4)
    h = torch.zeros((B, 64), device=DEV)
    h[:, 1] = torch.tensor([1.0 if b % 2 else -1.0 for b in range(B)], device=DEV)
    users = torch.zeros((B, 1), dtype=torch.int32, device=DEV)
    ids = torch.full((B, k), -7, dtype=torch.int32, device=DEV)
    sc = torch.full((B, k), float("nan"), device=DEV)
    ebr.score_topk(ix, cross, [ebr.Query(h_u=h[b], k=k, user_vals=users[b]) for b in range(B)],
                   ids, sc)
    torch.cuda.synchronize()
    ids, sc = ids.cpu().numpy().view(np.uint32), sc.cpu().numpy()
    for b in range(B):
        want, want_sc = _want(s if b % 2 else -s, k)
        assert np.array_equal(sc[b], want_sc)
        assert np.array_equal(ids[b], want)
