"""The index build at the edges of its sort tiles and window walks, bit for bit
against Algorithm 1's oracle (Sec. 3.4)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_2511_22460_gb300 import ebr  # noqa: E402

pytestmark = pytest.mark.gpu


def _check(n_ads, n_keys, pk, pa):
    emb = np.zeros((n_ads, 4), np.float32)
    ix = ebr.build_index(n_ads, n_keys, pk, pa, emb)
    ref = oracle.build_index(n_keys, n_ads, pk, pa)
    for g in range(9):
        for got, want in zip(ix.export(g), (ref["keys"][g], ref["header"][g], ref["values"][g])):
            np.testing.assert_array_equal(got, want, err_msg="g=%d" % g)
    assert ix.info().nnz_unique == len(set(zip(pk.tolist(), pa.tolist())))


# pairs around one and two sort tiles (4096), key spaces of 0, 9 and 17 bits
@pytest.mark.parametrize("nnz", [0, 1, 31, 4095, 4096, 4097, 8193])
@pytest.mark.parametrize("n_keys,n_ads", [(1, 1), (1, 70_000), (300, 257), (70_000, 65_536)])
def test_sizes_around_the_sort_tiles(nnz, n_keys, n_ads):
    rng = np.random.default_rng(nnz + n_keys)
    _check(n_ads, n_keys, rng.integers(0, n_keys, nnz).astype(np.uint32),
           rng.integers(0, n_ads, nnz).astype(np.uint32))


@pytest.mark.parametrize("n_full,n_ads", [(16, 256), (17, 256), (40, 700), (40, 512)])
def test_windows_of_full_blocks_across_the_walks_chunks(n_full, n_ads):
    # n_full keys hold every ad: blocks of 256 that end at, before and past
    # the 4096-word chunks, after one-ad blocks that shift them off the grid
    rng = np.random.default_rng(n_full)
    pk = np.concatenate([np.repeat(np.arange(100, 100 + n_full), n_ads),
                         rng.integers(0, 100, 77)]).astype(np.uint32)
    pa = np.concatenate([np.tile(np.arange(n_ads), n_full),
                         rng.integers(0, n_ads, 77)]).astype(np.uint32)
    p = rng.permutation(pk.size)
    _check(n_ads, 100 + n_full, pk[p], pa[p])


def test_long_runs_of_one_repeated_pair():
    # 9000 copies of one pair (longer than a chunk and its lookahead) among others
    rng = np.random.default_rng(5)
    pk = np.concatenate([np.full(9000, 3), rng.integers(0, 9, 3000)]).astype(np.uint32)
    pa = np.concatenate([np.full(9000, 300), rng.integers(0, 600, 3000)]).astype(np.uint32)
    p = rng.permutation(pk.size)
    _check(600, 9, pk[p], pa[p])


def test_key_space_beyond_28_bits_sorts_64_bit_records():
    n_keys, n_ads = (1 << 28) + 5, 1000
    pk = np.array([0, n_keys - 1, n_keys - 1, 7, 1 << 28, 7], np.uint32)
    pa = np.array([5, 999, 3, 300, 301, 301], np.uint32)
    ix = ebr.build_index(n_ads, n_keys, pk, pa, np.zeros((n_ads, 4), np.float32))
    dev = torch.device("cuda:0")
    q_key = torch.tensor([7, n_keys - 1, 0], dtype=torch.int32, device=dev)
    q_w = torch.tensor([1.0, 2.0, 4.0], device=dev)
    out = torch.empty(n_ads, device=dev)
    q = ebr.Query(h_u=torch.zeros(4, device=dev), k=1, q_key=q_key, q_w=q_w)
    ebr.wide_scores(ix, None, q, out)
    want = np.zeros(n_ads, np.float32)
    want[[300, 301]] = 1.0
    want[[999, 3]] = 2.0
    want[5] = 4.0
    np.testing.assert_array_equal(out.cpu().numpy(), want)
