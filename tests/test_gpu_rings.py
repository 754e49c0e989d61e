"""The pass over the active rows by the warps' rings (hidden layers wider than 128 units, sets of more than a chunk; always beyond 256
units) and the selection of the k best scores, against the oracle: widths at the edges of a lane's pieces, sets of a few rows and of
thousands, groups of rows that end in the middle, fewer rings than warps, equal scores and zeros of both signs."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2201_12667_b200 import workloads
    from tests.gpu_harness import Pair
    from tests.test_gpu_parity import check_predict
    from tests.test_gpu_shapes import dense_features_batch, one_and_two_steps

SIMHASH, DWTA = 0, 1


@pytest.mark.parametrize("H,N,K,L,cap,B", [
    (132, 3001, 4, 12, 64, 5), (196, 3001, 4, 12, 64, 3), (252, 3001, 5, 9, 41, 6), (256, 9001, 3, 12, 400, 4),      # 2 pieces per lane
    (260, 3001, 4, 12, 64, 5), (512, 2003, 4, 8, 37, 4), (516, 2003, 4, 8, 37, 4), (1020, 1501, 4, 6, 50, 3),
    (260, 3001, 10, 2, 1, 7), (1024, 1501, 9, 2, 2, 5),                                                              # a row or two per sample, or labels alone
])
def test_steps_and_predictions_by_rings(H, N, K, L, cap, B):
    pr = Pair(D=501, H=H, N=N, family=SIMHASH, K=K, L=L, bucket_cap=cap, max_batch=B, max_labels=3, lr=1e-3, seed=H + N)
    try:
        wl = workloads.Workload(dict(workloads.config("tiny"), D=501, N=N, batch=B), seed=5)
        for k in (1, 7, 64):
            check_predict(pr, wl.batch(0), 0, k)
        one_and_two_steps(pr, [wl.batch(0), wl.batch(1)])
    finally:
        pr.close()


@pytest.mark.parametrize("H,k", [(64, 1), (64, 64), (260, 5), (260, 64)])
def test_equal_scores_go_by_id(H, k):
    """Thousands of retrieved neurons score the same: the cut leaves more of them than are counted against one another."""
    pr = Pair(D=501, H=H, N=4001, family=SIMHASH, K=2, L=4, bucket_cap=700, max_batch=4, max_labels=3, seed=3)
    try:
        pr.o.set("W2", np.zeros(4001 * H, dtype=np.float32))
        pr.o.build_tables()
        wl = workloads.Workload(dict(workloads.config("tiny"), D=501, N=4001, batch=4), seed=5)
        check_predict(pr, wl.batch(0), 0, k, b2=np.where(np.arange(4001) % 701 == 5, 0.5, 0.25).astype(np.float32), same_ids=True)
    finally:
        pr.close()


@pytest.mark.parametrize("H,K,L", [(64, 4, 8), (200, 9, 50), (260, 5, 51), (512, 14, 50), (1024, 13, 40), (1020, 21, 50)])
def test_simhash_bits_of_queries(H, K, L):
    """The packed table of the hash functions mirrored whole, partly after the hidden layer, in two pieces and more (an odd number of
    functions: pieces that end inside a 16-byte word), and read from global memory (more than 1,024 functions)."""
    pr = Pair(D=501, H=H, N=1501, family=SIMHASH, K=K, L=L, bucket_cap=8, max_batch=6, max_labels=3, lr=1e-3, seed=H + K)
    try:
        wl = workloads.Workload(dict(workloads.config("tiny"), D=501, N=1501, batch=6), seed=5)
        one_and_two_steps(pr, [wl.batch(0), wl.batch(1)])
    finally:
        pr.close()


@pytest.mark.parametrize("H,K,max_labels,nlab,budget,least", [
    (512, 16, 4096, 190, 0, 160),      # five rings: a warp's first 32 rows are the set's first 160
    (1024, 10, 16, 3, 250, 224),       # seven rings, one group deep
    (1020, 10, 16, 3, 231, 224),
])
def test_fewer_rings_than_warps(H, K, max_labels, nlab, budget, least):
    """1,024 tables and many labels leave staging space for fewer rings than the block has warps.  Sets between the rows that the
    rings' warps count first and 256: all of them are handed to the update kernel, in steps after one another."""
    N = 1500
    pr = Pair(D=501, H=H, N=N, family=SIMHASH, K=K, L=1024, srp_nnz=8, bucket_cap=1, max_batch=6, max_labels=max_labels, budget=budget, lr=1e-3, seed=H)
    try:
        r = np.random.default_rng(H)
        one_and_two_steps(pr, [dense_features_batch(r, 6, 501, N, 20, nlab) for _ in range(2)])
        cnt = pr.gpu_active_sets(6)[1]
        assert cnt.min() > least and cnt.max() <= 256, cnt
    finally:
        pr.close()


@pytest.mark.parametrize("H,k", [(64, 1), (64, 20), (260, 20)])
def test_zeros_of_both_signs_are_equal(H, k):
    """Scores of minus zero (a bias of minus zero, products too small for a number) and of zero go by id, too."""
    N = 901
    pr = Pair(D=501, H=H, N=N, family=SIMHASH, K=1, L=8, bucket_cap=N, max_batch=4, max_labels=3, seed=3)
    try:
        W2 = np.zeros((N, H), dtype=np.float32)
        W2[::2] = -1e-30
        pr.o.set("W2", W2.ravel())
        pr.o.set("W1", np.zeros(501 * H, dtype=np.float32))
        pr.o.set("b1", np.full(H, 1e-30, dtype=np.float32))
        pr.o.build_tables()
        wl = workloads.Workload(dict(workloads.config("tiny"), D=501, N=N, batch=4), seed=5)
        check_predict(pr, wl.batch(0), 0, k, b2=np.full(N, -0.0, dtype=np.float32), same_ids=True)
    finally:
        pr.close()
