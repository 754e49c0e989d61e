"""The table build's partition and placement at the sizes where it can go wrong: vocabularies below and just past a
tile, codes one bit wider than a radix digit, parts far too crowded for shared memory, bins whose values tie."""
import numpy as np
import pytest

from paper_2201_12667_b200 import binding as ds
from paper_2201_12667_b200.workloads import DWTA, SIMHASH
from tests.gpu_harness import Pair

pytestmark = pytest.mark.gpu


def same_tables(pr):
    for name in ("bucket_off", "bucket_ids"):
        assert np.array_equal(ds.dslide_get_tensor(pr.ctx, name), pr.o.view(name)), name


@pytest.mark.parametrize("family,K,L,N,H,cap", [
    (SIMHASH, 10, 3, 2000, 32, 16), (SIMHASH, 12, 5, 6143, 64, 16), (SIMHASH, 17, 2, 6145, 32, 4), (SIMHASH, 20, 2, 5000, 64, 16),
    (DWTA, 4, 7, 12289, 64, 20), (DWTA, 6, 11, 20011, 136, 32), (DWTA, 6, 5, 3001, 1024, 16), (DWTA, 3, 9, 7001, 72, 16), (DWTA, 1, 17, 129, 8, 64),
    (SIMHASH, 9, 3, 9001, 36, 16), (SIMHASH, 1, 2, 77, 4, 16),
])
def test_tables(family, K, L, N, H, cap):
    pr = Pair(D=40, H=H, N=N, family=family, K=K, L=L, bucket_cap=cap, max_batch=4, seed=K + N)
    try:
        same_tables(pr)
        ds.dslide_rebuild_tables(pr.ctx)
        ds.dslide_sync(pr.ctx)
        pr.o.rebuild_tables()
        same_tables(pr)
    finally:
        pr.close()


@pytest.mark.parametrize("K,L,N,H,nnz", [
    (7, 70, 20011, 128, 0),     # four rows per lane, all tables at a time
    (12, 60, 1601, 400, 0),     # four rows per lane, the functions of some tables beside them
    (6, 33, 129, 440, 0),       # two rows per lane, a last tile of one row
    (9, 40, 801, 856, 0),       # one or two rows per lane, few tables at a time
    (5, 30, 333, 1024, 0),      # one row per lane
    (8, 1, 31, 100, 0),         # one table, less than a tile
    (17, 5, 1601, 256, 0),      # few tables at a time: a table's functions shared out between warps
    (5, 7, 4001, 400, 0),       # the same, every function by a warp of its own
    (18, 3, 333, 1024, 0),      # the same with one row per lane
    (13, 4, 700, 600, 600),     # dense projections
])
def test_simhash_tables_at_every_width(K, L, N, H, nnz):
    pr = Pair(D=40, H=H, N=N, family=SIMHASH, K=K, L=L, srp_nnz=nnz, bucket_cap=16, max_batch=4, seed=K + N)
    try:
        same_tables(pr)
        ds.dslide_rebuild_tables(pr.ctx)
        ds.dslide_sync(pr.ctx)
        pr.o.rebuild_tables()
        same_tables(pr)
    finally:
        pr.close()


@pytest.mark.parametrize("K,N", [(4, 9001), (6, 30011)])
def test_crowded_parts_and_bins_that_tie(K, N):
    """Rows with few distinct values, zeros of both signs, infinities, values beyond 2^87 and smaller than any normal
    number: winners are decided by position, most ids share a few codes, and some rows take the chain of comparisons."""
    pr = Pair(D=40, H=64, N=N, family=DWTA, K=K, L=6, bucket_cap=16, max_batch=4, seed=1)
    try:
        r = np.random.default_rng(5)
        W = np.zeros((N, 64), dtype=np.float32)
        W[N // 2:] = r.choice(np.array([0.0, -0.0, 1.0, 1e-45, 3e-45, -1e-45], dtype=np.float32), (N - N // 2, 64))
        W[5] = np.inf
        W[6] = -np.inf
        W[7, ::3] = np.inf
        W[8] = r.standard_normal(64).astype(np.float32) * np.float32(1e30)
        W[9] = r.choice(np.array([1.0, 1.0 + 2.0 ** -23], dtype=np.float32), 64)
        pr.o.set("W2", W.ravel())
        pr.push_state()
        pr.o.build_tables()
        same_tables(pr)
    finally:
        pr.close()


@pytest.mark.parametrize("K,N", [(1, 301), (3, 301), (4, 3001), (6, 7001)])
def test_bins_of_large_values_of_one_sign(K, N):
    """Rows whose bins hold distinct finite values all far below -2^88, or far above 2^87: the differences of the quick
    way to a bin's winner overflow, and the chain of comparisons has to decide."""
    pr = Pair(D=40, H=64, N=N, family=DWTA, K=K, L=6, bucket_cap=16, max_batch=4, seed=2)
    try:
        r = np.random.default_rng(6)
        W = r.standard_normal((N, 64)).astype(np.float32)
        for rows, scale in ((slice(3, 40), -1e30), (slice(50, 70), 1e30), (slice(80, 100), -3.3e38), (slice(110, 130), -2.0 ** 88), (slice(140, 160), -2.0 ** 86)):
            W[rows] = (r.uniform(0.5, 1.0, W[rows].shape) * scale).astype(np.float32)
        pr.o.set("W2", W.ravel())
        pr.push_state()
        pr.o.build_tables()
        same_tables(pr)
    finally:
        pr.close()
