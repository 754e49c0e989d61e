"""Inference over all neurons at the shapes where the tensor-pipe filter can go wrong: hidden widths that end inside a
slab of 32 units, widths too wide for tensor memory, more results than fit a warp, vocabularies below and just past a
tile, batches just past a group of 128 samples."""
import numpy as np
import pytest

from paper_2201_12667_b200 import workloads
from tests.gpu_harness import Pair
from tests.test_gpu_parity import check_predict

pytestmark = pytest.mark.gpu

SHAPES = [            # H, N, batch, k
    (4, 3001, 3, 1), (36, 129, 5, 10), (36, 128, 1, 64), (36, 100, 2, 5), (36, 40, 3, 64), (200, 20011, 130, 5),
    (252, 9000, 33, 64), (256, 5000, 129, 9), (260, 5000, 40, 5), (516, 3000, 131, 17), (1024, 2049, 260, 3), (1020, 700, 1, 64),
    (132, 9000, 200, 3),
    (32, 170003, 3, 5), (32, 170003, 130, 64), (64, 600, 1, 5), (32, 900, 2048, 2),      # the largest of 32 neighbours in the threshold pass; many and few buffers to a sample
]
PAIRS = [             # two multiprocessors to a tile: more than 192 units, more than 128 samples, tiles that keep them busy
    (196, 19001, 256, 5), (200, 38017, 257, 9), (256, 18945, 256, 64), (224, 30011, 130, 3), (260, 38145, 140, 5), (292, 19001, 300, 5),
    (1020, 13001, 300, 5),
]


@pytest.mark.parametrize("H,N,B,k", SHAPES + PAIRS)
def test_predict_over_all_neurons(H, N, B, k):
    pr = Pair(D=501, H=H, N=N, family=workloads.SIMHASH, K=4, L=4, bucket_cap=16, max_batch=B, seed=H + N)
    try:
        c = dict(workloads.config("tiny"), D=501, N=N, batch=B, max_labels=min(3, N))
        check_predict(pr, workloads.Workload(c, seed=k).batch(0, B), 1, k)
    finally:
        pr.close()


def test_weights_that_are_not_finite():
    """An infinite weight makes the error bound infinite and activations that are not numbers leave no candidate: both
    go through the exact scan."""
    pr = Pair(D=501, H=36, N=3001, family=workloads.SIMHASH, K=4, L=4, bucket_cap=16, max_batch=8, seed=3)
    try:
        W2 = np.array(pr.o.view("W2")).reshape(3001, 36)
        W2[[7, 2900]] = [[np.inf], [-np.inf]]
        pr.o.set("W2", W2.ravel())
        pr.o.set("b1", np.full(36, 2.0, dtype=np.float32))          # every unit active: no 0 x infinity
        c = dict(workloads.config("tiny"), D=501, N=3001, batch=8)
        batch = workloads.Workload(c, seed=1).batch(0, 8)
        pr.o.set("b2", np.zeros(3001, dtype=np.float32))
        pr.push_state()
        import torch
        from paper_2201_12667_b200 import binding as ds
        from tests.gpu_harness import to_dev
        ids, sc = torch.empty(8 * 5, dtype=torch.int32, device="cuda"), torch.empty(8 * 5, device="cuda")
        ds.dslide_predict_topk(pr.ctx, 8, *to_dev(batch[:3]), 5, 1, ids, sc)
        ds.dslide_sync(pr.ctx)
        ids_o, sc_o = pr.o.predict_topk(batch[0], batch[1], batch[2], 5, dense=True)
        assert np.array_equal(ids.cpu().numpy().reshape(8, 5)[:, 0], ids_o[:, 0]) and (ids_o[:, 0] == 7).all()
        assert np.allclose(sc.cpu().numpy().reshape(8, 5)[:, 1:], sc_o[:, 1:], rtol=1e-4, atol=1e-4)
        pr.o.set("b1", np.full(36, np.nan, dtype=np.float32))
        pr.push_state()
        ds.dslide_predict_topk(pr.ctx, 8, *to_dev(batch[:3]), 5, 1, ids, sc)
        ds.dslide_sync(pr.ctx)
        assert (ids >= 0).all()
    finally:
        pr.close()


FLAGGED = [           # H, N, batch, k, samples whose filter cannot decide (of the batch)
    (4, 3001, 3, 1, 3), (36, 129, 5, 10, 1), (128, 2000, 20, 64, 20), (200, 5011, 260, 5, 9), (128, 20011, 1, 5, 1),
    (264, 700, 33, 17, 32), (1024, 2049, 40, 3, 8), (1020, 333, 9, 64, 9), (64, 4001, 300, 5, 300), (256, 20011, 200, 5, 70),
    (300, 20011, 200, 5, 70),
]


@pytest.mark.parametrize("H,N,B,k,flagged", FLAGGED)
def test_samples_that_are_scored_over_all_neurons(H, N, B, k, flagged):
    """One row of W2 with a huge norm widens the error bound of the filter, so that every sample with a hidden activation
    is scored over all neurons; the others (hidden activation zero, scores the biases alone) need not be.  Results are right for
    both, call after call; which samples are scored so is asked by test_the_bound_takes_the_whole_norm."""
    import torch
    from paper_2201_12667_b200 import binding as ds
    from tests.gpu_harness import to_dev
    pr = Pair(D=501, H=H, N=N, family=workloads.SIMHASH, K=4, L=4, bucket_cap=16, max_batch=B, seed=H + N)
    try:
        r = np.random.default_rng(H)
        W2 = np.array(pr.o.view("W2")).reshape(N, H)
        W2[N // 2, 0] = -1e8
        pr.o.set("W2", W2.ravel())
        pr.o.set("b2", r.permutation(N).astype(np.float32) / np.float32(N))
        W1 = np.abs(np.array(pr.o.view("W1"))).reshape(501, H)
        W1[250:] = 0
        pr.o.set("W1", W1.ravel())
        pr.push_state()
        batch = [np.arange(0, 3 * B + 1, 3, dtype=np.int32), np.empty(3 * B, np.int32), r.uniform(0.5, 1, 3 * B).astype(np.float32)]
        on = np.zeros(B, bool)
        on[r.permutation(B)[:flagged]] = True
        for s in range(B):
            batch[1][3 * s:3 * s + 3] = np.sort(r.choice(250, 3, replace=False)) + (0 if on[s] else 250)
        ids, sc = torch.empty(B * k, dtype=torch.int32, device="cuda"), torch.empty(B * k, device="cuda")
        for _ in range(2):                                      # counters and lists are left clean
            ids.fill_(-7)
            ds.dslide_predict_topk(pr.ctx, B, *to_dev(batch), k, 1, ids, sc)
            ds.dslide_sync(pr.ctx)
            ids_o, sc_o = pr.o.predict_topk(*batch, k, dense=True)
            assert np.allclose(sc.cpu().numpy().reshape(B, k), sc_o, rtol=1e-4, atol=1e-6)
            close = np.abs(np.diff(sc_o, axis=1)) < 1e-5        # neighbours whose sums round either way may change places
            sure = ~(np.pad(close, ((0, 0), (0, 1)), constant_values=True) | np.pad(close, ((0, 0), (1, 0))))
            assert np.array_equal(ids.cpu().numpy().reshape(B, k)[sure], ids_o[sure])
            assert all(len(set(row)) == k for row in ids.cpu().numpy().reshape(B, k).tolist())
    finally:
        pr.close()


def test_an_undecided_sample_is_everybodys_work():
    """One sample that the filter cannot decide: all multiprocessors share the scan of W2 (a quarter of a millisecond or
    less here; by a single block it took 29, a bound of 3 leaves room on either side)."""
    import torch
    from paper_2201_12667_b200 import binding as ds
    N, H = 200003, 128
    ctx = ds.dslide_init(ds.make_config(input_dim=64, hidden_dim=H, output_dim=N, hash_family=workloads.SIMHASH, K=4, L=2, bucket_cap=16,
                                        max_batch=4, init_std=0.05))
    try:
        W2 = ds.dslide_get_tensor(ctx, "W2").reshape(N, H)
        W2[N // 2, 0] = -1e8
        ds.dslide_set_tensor(ctx, "W2", W2)
        ds.dslide_set_tensor(ctx, "b1", np.full(H, 0.5, dtype=np.float32))
        args = [torch.tensor([0, 1], dtype=torch.int32, device="cuda"), torch.tensor([3], dtype=torch.int32, device="cuda"), torch.ones(1, device="cuda")]
        ids, sc = torch.empty(5, dtype=torch.int32, device="cuda"), torch.empty(5, device="cuda")
        best = 1e9
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            ds.dslide_predict_topk(ctx, 1, *args, 5, 1, ids, sc)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        h = np.maximum(0, ds.dslide_get_tensor(ctx, "W1").reshape(64, H)[3].astype(np.float64) + 0.5)
        z = W2.astype(np.float64) @ h
        assert np.allclose(sc.cpu().numpy(), np.sort(z)[::-1][:5], rtol=1e-5) and set(ids.tolist()) == set(np.argsort(-z)[:5].tolist())
        assert best < 3.0, best
    finally:
        ds.dslide_destroy(ctx)


NORMS = [             # H, N, batch: single blocks, wide ones, pairs, wide pairs; one to nine groups of samples
    (64, 3001, 1), (128, 5003, 300), (160, 5003, 700), (300, 3001, 40),
    (200, 20011, 200), (196, 19001, 300), (256, 20011, 1100), (260, 20011, 200), (516, 20011, 300), (300, 20011, 600), (292, 20011, 1100),
]


@pytest.mark.parametrize("H,N,B", NORMS)
def test_the_norm_of_every_row_counts(H, N, B):
    """A row whose two large weights cancel: its score is 1, the best by far, and 0 once weights lose their last bits, as in the
    filter.  Only the row's norm in the error bound shows that the filter cannot decide, wherever in a tile the row lies (the
    halves of a tile are in the shared memory of two blocks, its rows are shared out between the groups of samples)."""
    import torch
    from paper_2201_12667_b200 import binding as ds
    from tests.gpu_harness import to_dev
    k = 4
    r = np.random.default_rng(H + B)
    ctx = ds.dslide_init(ds.make_config(input_dim=50, hidden_dim=H, output_dim=N, hash_family=workloads.SIMHASH, K=4, L=2, bucket_cap=16, max_batch=B))
    try:
        W1 = r.standard_normal((50, H)).astype(np.float32)
        W1[:, :2] = 0
        b1 = np.zeros(H, np.float32)
        b1[:2] = 1                                              # two units that are 1 for every sample
        W2 = (r.standard_normal((N, H)) * (0.03 / np.sqrt(H))).astype(np.float32)
        W2[:, :2] = 0
        b2 = np.full(N, -0.01, np.float32)
        for name, x in (("W1", W1), ("b1", b1), ("b2", b2)):
            ds.dslide_set_tensor(ctx, name, x)
        batch = to_dev([np.arange(B + 1, dtype=np.int32), r.integers(0, 50, B).astype(np.int32), r.uniform(0.5, 1, B).astype(np.float32)])
        ids, sc = torch.empty(B, k, dtype=torch.int32, device="cuda"), torch.empty(B, k, device="cuda")

        def best():
            ds.dslide_set_tensor(ctx, "W2", W2)
            ds.dslide_predict_topk(ctx, B, *batch, k, 1, ids, sc)
            ds.dslide_sync(ctx)
            return ids.cpu().numpy().copy(), sc.cpu().numpy().copy()

        for first in (0, 256 * (N // 512)):
            for at in (0, 31, 63, 64, 100, 127, 128, 161, 200, 255):
                row = min(first + at, N - 1)
                keep = W2[row].copy()
                W2[row] = 0
                ids0, sc0 = best()                              # the row scores -0.01, which others beat
                assert (sc0[:, -1] > 0).all() and (sc0 < 0.9).all()
                W2[row, :2] = 4097, -4096
                ids1, sc1 = best()
                assert (ids1[:, 0] == row).all() and np.allclose(sc1[:, 0], 0.99, rtol=1e-6), row
                assert np.allclose(sc1[:, 1:], sc0[:, :-1], rtol=1e-4, atol=1e-6) and (ids1[:, 1:] == ids0[:, :-1]).mean() > 0.99
                W2[row] = keep
    finally:
        ds.dslide_destroy(ctx)


def test_neighbours_that_are_favoured_together_fit_their_buffer():
    """Two runs of 48 neighbouring neurons that all samples prefer, in two tiles of one pair of wide blocks and in the same
    columns: their 96 candidates per sample, and the handful that the buffer takes besides, find room, and no sample is scored
    over all neurons for want of it (about 0.15 ms here, 2.6 when all of them are)."""
    import torch
    from paper_2201_12667_b200 import binding as ds
    from tests.gpu_harness import to_dev
    N, H, B, k = 100003, 512, 512, 5
    r = np.random.default_rng(2)
    ctx = ds.dslide_init(ds.make_config(input_dim=50, hidden_dim=H, output_dim=N, hash_family=workloads.SIMHASH, K=4, L=2, bucket_cap=16, max_batch=B))
    try:
        W1 = r.standard_normal((50, H)).astype(np.float32)
        W2 = (r.standard_normal((N, H)) * (0.05 / np.sqrt(H))).astype(np.float32)
        b2 = np.zeros(N, np.float32)
        for tile in (1, 38):                                    # 391 tiles of 256 neurons for 37 pairs; every 64th tile gives the threshold
            b2[256 * tile:256 * tile + 48] = 2
        for name, x in (("W1", W1), ("W2", W2), ("b2", b2)):
            ds.dslide_set_tensor(ctx, name, x)
        cols, vals = r.integers(0, 50, B).astype(np.int32), r.uniform(0.5, 1, B).astype(np.float32)
        batch = to_dev([np.arange(B + 1, dtype=np.int32), cols, vals])
        ids, sc = torch.empty(B, k, dtype=torch.int32, device="cuda"), torch.empty(B, k, device="cuda")
        best = 1e9
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            ds.dslide_predict_topk(ctx, B, *batch, k, 1, ids, sc)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        h = np.maximum(0, W1[cols].astype(np.float64) * vals[:, None])
        z = h @ W2.T.astype(np.float64) + b2
        top = np.sort(np.partition(z, N - k, axis=1)[:, N - k:], axis=1)[:, ::-1]
        assert np.allclose(sc.cpu().numpy(), top, rtol=1e-5)
        assert best < 1.0, best
    finally:
        ds.dslide_destroy(ctx)


def predict_all(ctx, batch, k):
    import torch
    from paper_2201_12667_b200 import binding as ds
    B = len(batch[0]) - 1
    ids, sc = torch.empty(B, k, dtype=torch.int32, device="cuda"), torch.empty(B, k, device="cuda")
    ds.dslide_predict_topk(ctx, B, *batch, k, 1, ids, sc)
    ds.dslide_sync(ctx)
    return ids.cpu().numpy(), sc.cpu().numpy()


@pytest.mark.parametrize("H,N,k", [(64, 384, 1), (64, 384, 5), (128, 512, 10), (300, 512, 5), (64, 600, 5), (64, 1024, 64), (128, 1024, 64)])
def test_near_ties_of_few_neurons(H, N, k):
    """Rows that resemble one another: their scores differ by less than the filter's error, so that no sample can be decided by
    it, however its candidates are shared out to the threads that look for the cut."""
    from paper_2201_12667_b200 import binding as ds
    from tests.gpu_harness import to_dev
    B, spread = 1000, 1e-5
    r = np.random.default_rng(H + N + k)
    ctx = ds.dslide_init(ds.make_config(input_dim=B, hidden_dim=H, output_dim=N, hash_family=workloads.SIMHASH, K=4, L=2, bucket_cap=16, max_batch=B))
    try:
        W1 = r.standard_normal((B, H)).astype(np.float32)
        W2 = (0.05 + spread * r.standard_normal((N, H))).astype(np.float32)
        ds.dslide_set_tensor(ctx, "W1", W1)
        ds.dslide_set_tensor(ctx, "W2", W2)
        ids, sc = predict_all(ctx, to_dev([np.arange(B + 1, dtype=np.int32), np.arange(B, dtype=np.int32), np.ones(B, np.float32)]), k)
        h = np.maximum(0, W1).astype(np.float64)
        z = h @ W2.T.astype(np.float64)
        # at most H / 32 + 9 additions after one another make a score in 32 bits
        tol = (H / 32 + 9) * 2.0 ** -24 * (h @ np.abs(W2.T.astype(np.float64))).max(axis=1, keepdims=True)
        kth = np.sort(z, axis=1)[:, ::-1][:, k - 1:k]
        assert (np.diff(np.sort(ids, axis=1), axis=1) > 0).all() and (ids >= 0).all()
        assert (np.abs(np.take_along_axis(z, ids, 1) - sc) <= tol).all()
        assert (np.take_along_axis(z, ids, 1) >= kth - 2 * tol).all()
    finally:
        ds.dslide_destroy(ctx)


@pytest.mark.parametrize("H,N,B", [s for s in NORMS if s[2] < 1100] + [
    (200, 38017, 700), (200, 20011, 769), (196, 20011, 1024), (256, 20011, 1100), (256, 38017, 1300)])      # three to six groups of samples in pairs
def test_the_bound_takes_the_whole_norm(H, N, B):
    """The best scores stand 0.25 above a plateau that the cut falls on.  A row whose norm makes the error bound 0.9 of that leaves
    every sample decided, one that makes it 1.1 none: the scores then come from the scan, which adds up in another order.  The row's
    weight lies in all of its 16-byte pieces, or in one of them."""
    from paper_2201_12667_b200 import binding as ds
    from tests.gpu_harness import to_dev
    k, err = 16, 2.2e-3                                         # the filter's error for |h| = |w| = 1
    r = np.random.default_rng(H + B)
    ctx = ds.dslide_init(ds.make_config(input_dim=4, hidden_dim=H, output_dim=N, hash_family=workloads.SIMHASH, K=4, L=2, bucket_cap=16, max_batch=B))
    try:
        ds.dslide_set_tensor(ctx, "W1", np.zeros((4, H), np.float32))
        ds.dslide_set_tensor(ctx, "b1", np.ones(H, np.float32))               # |h|^2 = H
        W2, b2 = np.zeros((N, H), np.float32), (-1 - r.random(N)).astype(np.float32)
        some = r.permutation(N)[:k + 120]
        W2[some[:k]] = 0.05 * r.standard_normal((k, H))
        b2[some[:k]] = 1.25 + 0.05 * np.arange(k) - W2[some[:k]].astype(np.float64).sum(axis=1)
        b2[some[k:]] = 1                                        # the plateau: more rows than the cut is at, fewer than are scored exactly
        ds.dslide_set_tensor(ctx, "b2", b2)
        batch = to_dev([np.arange(B + 1, dtype=np.int32), np.zeros(B, np.int32), np.ones(B, np.float32)])

        def scores(row=None, units=None, share=1.0):
            keep = W2[row].copy() if row is not None else None
            if row is not None:                                 # the row's score: 0 and its bias, for its weights cancel
                W2[row] = 0
                W2[row, units] = share * 0.25 / (err * np.sqrt(H * len(units))) * (-1.0) ** np.arange(len(units))
            ds.dslide_set_tensor(ctx, "W2", W2)
            if row is not None:
                W2[row] = keep
            return predict_all(ctx, batch, k)[1]

        free = np.setdiff1d(np.arange(N), some)
        filtered, scanned = scores(), scores(int(free[0]), np.arange(2), 1e6)
        assert np.allclose(filtered, 2 - 0.05 * np.arange(k), rtol=1e-5) and np.allclose(scanned, filtered, rtol=1e-5)
        assert (filtered != scanned).any(axis=1).all()
        slab = 32 * r.integers(0, H // 32)
        pieces = [np.arange(H)] + [slab + 4 * p + np.arange(4) for p in range(8)]
        at = [0, 31, 63, 64, 100, 127, 128, 161, 255]           # of a tile: in either block of a pair, in any group's share
        for i, units in enumerate(pieces):
            row = int(free[min(np.searchsorted(free, 256 * (N // 512) + at[(i + B) % 9]), len(free) - 1)])
            assert (scores(row, units, 0.9) == filtered).all(), (i, row)
            assert (scores(row, units, 1.1) == scanned).all(), (i, row)
    finally:
        ds.dslide_destroy(ctx)


@pytest.mark.parametrize("B", [1, 200])
def test_many_neighbours_that_are_favoured_together(B):
    """512 neighbouring neurons that all samples prefer fill a few buffers, and the other buffers hold candidates as well: the cut by
    the threads' maxima lets all of the neighbours pass, which are more than are scored exactly.  It is then taken among all
    candidates, and no sample is scored over all neurons."""
    from paper_2201_12667_b200 import binding as ds
    from tests.gpu_harness import to_dev
    N, H, k = 100003, 128, 16
    r = np.random.default_rng(2)
    ctx = ds.dslide_init(ds.make_config(input_dim=50, hidden_dim=H, output_dim=N, hash_family=workloads.SIMHASH, K=4, L=2, bucket_cap=16, max_batch=B))
    try:
        W1 = r.standard_normal((50, H)).astype(np.float32)
        W2 = (r.standard_normal((N, H)) * (0.5 / np.sqrt(H))).astype(np.float32)
        b2 = np.full(N, -2, np.float32)
        first = 128 * 65                                        # every 64th tile gives the threshold
        b2[first:first + 512] = 0
        for name, x in (("W1", W1), ("W2", W2), ("b2", b2)):
            ds.dslide_set_tensor(ctx, name, x)
        cols, vals = r.integers(0, 50, B).astype(np.int32), r.uniform(0.5, 1, B).astype(np.float32)
        batch = to_dev([np.arange(B + 1, dtype=np.int32), cols, vals])
        ids, sc = predict_all(ctx, batch, k)
        z = np.maximum(0, W1[cols].astype(np.float64) * vals[:, None]) @ W2.T.astype(np.float64) + b2
        assert np.allclose(sc, np.sort(z, axis=1)[:, ::-1][:, :k], rtol=1e-5)
        W2[0, 0] = -1e8                                         # now no sample can be decided: the scan adds up in another order
        ds.dslide_set_tensor(ctx, "W2", W2)
        ids_s, sc_s = predict_all(ctx, batch, k)
        assert np.allclose(sc_s, sc, rtol=1e-5)
        assert (sc_s != sc).any(axis=1).mean() > 0.9
    finally:
        ds.dslide_destroy(ctx)
