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
]


@pytest.mark.parametrize("H,N,B,k", SHAPES)
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
