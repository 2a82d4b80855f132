"""The forward scan's inner products (16-bit pieces of the user vector on the
tensor pipe) at the ends of the number ranges, against FP64 sums of the same
table."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_2511_22460_gb300 import ebr  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
INF = np.float32(np.inf)


def _index(emb, dtype):
    n = emb.shape[0]
    # one posting, so that the index has a forward table
    return ebr.build_index(n, 3, np.zeros(1, np.uint32), np.zeros(1, np.uint32), emb, dtype=dtype)


def _table(ix, dtype):
    codes, scale = ix.export_emb()
    if dtype == "bf16":
        return (codes.astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    vals = np.array([oracle.fp8_e4m3_value(c) for c in range(256)], np.float64)
    return vals[codes] * scale.astype(np.float64)[:, None]


def _query(h, **kw):
    return ebr.Query(h_u=torch.from_numpy(h).to(DEV), q_w=torch.zeros(3, device=DEV), **kw)


def _scores(ix, h):
    out = torch.empty(int(ix.info().n_ads), device=DEV)
    ebr.score_all(ix, None, _query(h, k=1), out)
    return out.cpu().numpy()


@pytest.mark.parametrize("d", [8, 16, 64, 128])
@pytest.mark.parametrize("huge", [INF, np.float32(3.4e38)])  # (rounds to infinity in BF16)
def test_infinite_elements_of_bf16_tables(d, huge):
    n = 5_000
    rng = np.random.default_rng(d)
    emb = rng.standard_normal((n, d)).astype(np.float32)
    emb[7::50, 3] = huge
    emb[9::50, d - 1] = -huge
    emb[11::50, [0, 5]] = [huge, -huge]  # both signs: NaN
    ix = _index(emb, "bf16")
    table = _table(ix, "bf16")
    for h in (rng.standard_normal(d).astype(np.float32),
              np.full(d, 0.5, np.float32)):  # one piece, the others zero
        with np.errstate(invalid="ignore"):
            ref = (table * h.astype(np.float64)).sum(1)
        got = _scores(ix, h)
        fin = np.isfinite(ref)
        assert np.array_equal(np.isnan(got), np.isnan(ref))
        assert np.array_equal(got[np.isinf(ref)].astype(np.float64), ref[np.isinf(ref)])
        tol = 1e-5 * (np.abs(table[fin]) @ np.abs(h).astype(np.float64))
        assert np.all(np.abs(got[fin] - ref[fin]) <= tol)


@pytest.mark.parametrize("n", [5_000, 20_000])  # keys of all ads, and running bounds
@pytest.mark.parametrize("sign", [-1, 1])
def test_infinite_ads_in_the_top_k(n, sign):
    # at least 500 infinite ads, more than (R - 1) K: last, or first by their ids
    d, k = 64, 20
    rng = np.random.default_rng(0)
    emb = rng.standard_normal((n, d)).astype(np.float32)
    emb[::10, 3] = sign * INF
    h = np.abs(rng.standard_normal(d)).astype(np.float32)
    ix = _index(emb, "bf16")
    ids = torch.empty(k, dtype=torch.int32, device=DEV)
    sc = torch.empty(k, device=DEV)
    ebr.score_topk(ix, None, [_query(h, k=k)], ids, sc)
    got, sc = ids.cpu().numpy(), sc.cpu().numpy()
    if sign > 0:
        assert np.array_equal(got, 10 * np.arange(k)) and np.all(sc == INF)
        return
    ref = (emb.astype(np.float64) * h).sum(1)
    tol = 1e-5 * (np.abs(emb).astype(np.float64) * h).sum(1)
    assert np.unique(got).size == k and np.all(np.isfinite(ref[got]))
    assert np.all(np.abs(sc - ref[got]) <= tol[got])
    kth = np.sort(ref)[::-1][k - 1]
    assert np.all(ref[got] >= kth - 2 * tol[np.isfinite(ref)].max())


@pytest.mark.parametrize("d", [16, 64, 128])
@pytest.mark.parametrize("top", [1e30, 9e34, 1.8e35])
def test_huge_user_vectors_on_fp8_tables(d, top):
    # four elements a row: the sum of h x codes (at most 448) stays finite too
    n = 3_000
    rng = np.random.default_rng(d)
    emb = np.zeros((n, d), np.float32)
    for i in range(4):
        emb[np.arange(n), rng.integers(0, d, n)] = rng.standard_normal(n) / d
    ix = _index(emb, "fp8e4m3")
    table = _table(ix, "fp8e4m3")
    h = rng.uniform(-1, 1, d).astype(np.float32)
    h = h / np.abs(h).max() * np.float32(top)
    ref = (table * h.astype(np.float64)).sum(1)
    tol = 1e-5 * (np.abs(table) @ np.abs(h).astype(np.float64))
    assert np.all(np.abs(_scores(ix, h) - ref) <= tol)


def test_an_infinite_user_element_on_an_fp8_table():
    n, d = 3_000, 64
    rng = np.random.default_rng(1)
    ix = _index(rng.standard_normal((n, d)).astype(np.float32), "fp8e4m3")
    table = _table(ix, "fp8e4m3")
    h = (rng.standard_normal(d) * 1e6).astype(np.float32)  # beyond FP16 unless scaled
    h[5] = INF
    with np.errstate(invalid="ignore"):
        ref = (table * h.astype(np.float64)).sum(1)  # infinite, or NaN where the element is 0
    got = _scores(ix, h)
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    assert np.array_equal(got[~np.isnan(ref)].astype(np.float64), ref[~np.isnan(ref)])


@pytest.mark.parametrize("d", [16, 64, 128])
@pytest.mark.parametrize("dtype", ["bf16", "fp8e4m3"])
def test_ads_that_only_see_small_user_elements(dtype, d):
    # each ad is nonzero only where h_u has one of these magnitudes
    n, ratio = 4_000, [0, -25, -32, -40, -60, -75, -40, -32]
    rng = np.random.default_rng(d)
    part = np.arange(n) % len(ratio)
    own = np.arange(d) % len(ratio)
    emb = rng.standard_normal((n, d)).astype(np.float32) * (part[:, None] == own[None, :])
    ix = _index(emb.astype(np.float32), dtype)
    table = _table(ix, dtype)
    h = np.ldexp(rng.uniform(1, 2, d), np.array(ratio)[own]).astype(np.float32)
    for scale in (-30, 0, 50):
        hs = np.ldexp(h, scale).astype(np.float32)
        ref = (table * hs.astype(np.float64)).sum(1)
        tol = 1e-5 * (np.abs(table) @ np.abs(hs).astype(np.float64))
        assert np.all(np.abs(_scores(ix, hs) - ref) <= tol)
