"""The work a user of libdslide has it do, as cases that can be measured through the binding's public entry points.

A case is a dict: `kind` says which call is made, the rest is the model's shape, its hashing, and the batch.

  train         dslide_train_step on batches that live in device memory
  train_host    dslide_train_step_host_async on batches that live in host memory
  rebuild       dslide_rebuild_tables (new hash functions, every output neuron hashed and grouped again)
  predict       dslide_predict_topk over the retrieved neurons
  predict_all   dslide_predict_topk over all output neurons

A training step works on a model that goes on training, so a state holds several batches and every pass takes the
next one.  The scheduled rebuild is off in the training cases and measured by itself.
"""
import math

import numpy as np
import torch

from paper_2201_12667_b200 import binding as ds

SIMHASH, DWTA = ds.SIMHASH, ds.DWTA
BATCHES = 8            # distinct batches of a training state
ZIPF_S = 1.1
BIN = 8                # entries of a DWTA bin
LR, BETA1, BETA2, EPS = (float(np.float32(v)) for v in (1e-4, 0.9, 0.999, 1e-8))      # as the 32-bit configuration holds them

# shapes of the package's workloads (paper_2201_12667_b200/workloads.py)
_TINY = dict(D=1000, H=32, N=2000, family=SIMHASH, K=4, L=8, cap=64, batch=32, nnz=20, labels=2)
_670K = dict(D=135909, H=128, N=670091, family=DWTA, K=6, L=50, cap=128, batch=256, nnz=76, labels=5)
_325K = dict(D=1617899, H=128, N=325056, family=SIMHASH, K=9, L=50, cap=128, batch=256, nnz=42, labels=3)
_TEXT8 = dict(D=253855, H=200, N=253855, family=SIMHASH, K=9, L=50, cap=128, batch=1024, nnz=1, labels=4)
_1B = dict(D=200000, H=256, N=4000000, family=DWTA, K=7, L=64, cap=256, batch=512, nnz=100, labels=4)
# the large hidden layer and batch of the paper's Table 3 over a vocabulary that keeps a state small
_WIDE = dict(D=20011, H=1024, N=50021, family=DWTA, K=5, L=50, cap=128, batch=1024, nnz=76, labels=5)


def _case(kind, shape, **more):
    c = dict(kind=kind, k=0, budget=0, densify=0)
    c.update(shape)
    c.update(more)
    return c


def listed():
    return [
        # the smallest model of the configurations: launches and latency count, not bytes
        dict(_case("train", _TINY), name="train-tiny"),
        # the headline: extreme classification with 670,091 labels (Amazon-670K's shape), batches resident on the device
        dict(_case("train", _670K), name="train-670k"),
        # the same step for a program whose loader hands out host arrays
        dict(_case("train_host", _670K), name="train-670k-host"),
        # SimHash tables with full buckets: about 6,100 active neurons per sample (WikiLSHTC-325K's shape)
        dict(_case("train", _325K), name="train-325k"),
        # the word model: one-hot inputs, a hidden width that is no power of two, a large batch
        dict(_case("train", _TEXT8), name="train-text8"),
        # the widest hidden layer that is supported
        dict(_case("train", _WIDE), name="train-wide"),
        # the scheduled rebuild of the headline model
        dict(_case("rebuild", _670K), name="rebuild-670k"),
        # serving: one request, best answer
        dict(_case("predict", _670K, batch=1, k=1), name="predict-one"),
        # evaluation of a batch through the tables, precision at 5
        dict(_case("predict", _670K, k=5), name="predict-670k"),
        # evaluation over all classes, precision at 5
        dict(_case("predict_all", _670K, k=5), name="predict-all-670k"),
        # the same for the word model: all words scored for every context
        dict(_case("predict_all", _TEXT8, k=5), name="predict-all-text8"),
        # the largest model: a billion weights in the output layer
        dict(_case("predict_all", _1B, k=5), name="predict-all-1b"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _retrieved(c):
    """(neurons a sample retrieves, neurons the tables hand out at all): what the tables' shape makes likely."""
    bits = c["K"] * (1 if c["family"] == SIMHASH else 3)
    mean = c["N"] / 2.0 ** bits
    per = min(c["cap"], mean + (1 if c["family"] == DWTA else 0))
    pool = min(c["N"], 1.6 * c["cap"] * 2.0 ** bits) if mean > c["cap"] else c["N"]
    got = pool * -math.expm1(-c["L"] * per / pool)
    return (min(got, c["budget"]) if c["budget"] else got), pool


def draw(rng):
    """One more case of the same ranges: the sizes between those listed, odd ones among them."""
    while True:
        kind = rng.choice(["train", "train", "train", "train_host", "rebuild", "predict", "predict_all", "predict_all"])
        family = rng.choice([SIMHASH, DWTA])
        H = _log_int(rng, 32, 1024)
        H -= H % (4 if family == SIMHASH else 8)
        D, N = _log_int(rng, 1000, 1600000), _log_int(rng, 2000, 670000)
        if family == DWTA:
            K = max(2, min(7, int(round(math.log(N / rng.uniform(1, 30), 8)))))
        else:
            K = rng.randint(4, 12)
        c = dict(kind=kind, D=D, H=H, N=N, family=family, K=K, L=rng.randint(8, 64), cap=_log_int(rng, 16, 256),
                 batch=_log_int(rng, 1, 2048), nnz=_log_int(rng, 1, 120), labels=rng.randint(1, 6),
                 k=0, budget=0, densify=0)
        c["nnz"] = min(c["nnz"], D // 8)
        if kind.startswith("predict"):
            c["k"] = rng.choice([1, 3, 5, 10])
        elif kind.startswith("train"):
            if family == DWTA and rng.random() < 0.25:
                c["densify"] = 1
            if rng.random() < 0.2:
                c["budget"] = rng.choice([256, 1024])
        # no more than the largest listed ones: weights, gathered rows, scores of all neurons
        if H * N > 86000000 or H * D > 208000000 or c["budget"] > N:
            continue
        if c["budget"] and 5 * c["L"] * c["cap"] + 8 * c["budget"] > 60000:      # what a sampling budget has room for
            continue
        if kind.startswith("train") and c["batch"] * max(_retrieved(c)[0], c["labels"]) * H > 1.2e9:
            continue
        if kind == "predict" and c["batch"] * _retrieved(c)[0] * H > 1.2e9:
            continue
        if kind == "predict_all" and c["batch"] * N * H > 5.2e10:
            continue
        return c


# ---- inputs -----------------------------------------------------------------------------------------
def _zipf_rows(rng, M, mean, most, B):
    """B rows of distinct ids in [0, M), as (row_ptr, ids by row, unsorted): ids follow a Zipf law through a permutation."""
    n = np.ones(B, np.int64) if mean <= 1 else np.clip(rng.poisson(mean - 1, B) + 1, 1, most)
    cdf = np.cumsum(np.arange(1, M + 1, dtype=np.float64) ** -ZIPF_S)
    ranks = np.minimum(np.searchsorted(cdf, rng.random((B, 3 * int(n.max()) + 8)) * cdf[-1], side="right"), M - 1)
    order = np.argsort(ranks, axis=1, kind="stable")
    srt = np.take_along_axis(ranks, order, 1)
    again = np.zeros(ranks.shape, bool)
    np.put_along_axis(again, order[:, 1:], srt[:, 1:] == srt[:, :-1], 1)
    keep = ~again & (np.cumsum(~again, 1) <= n[:, None])
    ptr = np.zeros(B + 1, np.int32)
    ptr[1:] = np.cumsum(keep.sum(1))
    return ptr, ranks[keep]


def _batches(c, seed, count):
    """CSR rows with lognormal values of unit length, and label lists."""
    rng = np.random.Generator(np.random.PCG64([seed, 17]))
    feat, lab = rng.permutation(c["D"]).astype(np.int32), rng.permutation(c["N"]).astype(np.int32)
    got = []
    for _ in range(count):
        ptr, ranks = _zipf_rows(rng, c["D"], c["nnz"], min(4 * c["nnz"], c["D"]), c["batch"])
        row = np.repeat(np.arange(c["batch"]), np.diff(ptr))
        ids = feat[ranks]
        ids = ids[np.lexsort((ids, row))]
        v = np.exp(rng.standard_normal(ids.size))
        v = (v / np.sqrt(np.bincount(row, v * v, c["batch"]))[row]).astype(np.float32)
        lptr, lranks = _zipf_rows(rng, c["N"], c["labels"], 16, c["batch"])
        got.append((ptr, ids, v, lptr, lab[lranks]))
    return got


def _hash_functions(c, seed):
    """Coordinates (and signs) of the hash functions, in the layout of the tensors hash_idx and hash_sign."""
    rng = np.random.Generator(np.random.PCG64([seed, 23]))
    KL, H = c["K"] * c["L"], c["H"]
    if c["family"] == DWTA:
        perms = -(-KL * BIN // H)
        return np.argsort(rng.random((perms, H)), 1).reshape(-1)[:KL * BIN].astype(np.int32).reshape(KL, BIN), None
    m = (H + 2) // 3
    idx = np.sort(np.argsort(rng.random((KL, H)), 1)[:, :m], 1).astype(np.int32)
    return idx, rng.choice(np.array([-1, 1], np.int32), (KL, m))


def _own_weights(c):
    """Whether the state's weights are made here; the largest model keeps the library's initial draw."""
    return c["H"] * c["N"] <= 200000000


def _weights(c, seed, device):
    """Weights as a trained model has them: rows of the output layer of different lengths, biases that are not zero."""
    g = torch.Generator(device).manual_seed(seed * 1000003 + 5)
    r = lambda *n: torch.randn(*n, generator=g, device=device)  # noqa: E731
    W1 = r(c["D"], c["H"]) * 0.05
    W2 = r(c["N"], c["H"]) * 0.05 * torch.exp(0.3 * r(c["N"], 1))
    return dict(W1=W1, b1=r(c["H"]) * 0.02, W2=W2, b2=r(c["N"]) * 0.05)


class _Model:
    """A context and what a program keeps beside it; the context goes with the object."""

    ctx = None

    def __init__(self, c, seed):
        self.c, self.turn = c, 0
        self.ctx = ds.dslide_init(ds.make_config(
            input_dim=c["D"], hidden_dim=c["H"], output_dim=c["N"], hash_family=c["family"], K=c["K"], L=c["L"],
            bucket_cap=c["cap"], rebuild_period0=0, max_batch=c["batch"], max_labels=16, lr=1e-4, init_std=0.05,
            seed=seed, dwta_densify=c["densify"], sample_budget=c["budget"], inputs_ready=1))
        if _own_weights(c):
            for name, w in _weights(c, seed, "cuda").items():
                ds.dslide_set_tensor(self.ctx, name, w.cpu())
            idx, sign = _hash_functions(c, seed)
            ds.dslide_set_tensor(self.ctx, "hash_idx", idx)
            if sign is not None:
                ds.dslide_set_tensor(self.ctx, "hash_sign", sign)
            ds.dslide_build_tables(self.ctx)
        ds.dslide_sync(self.ctx)

    def __del__(self):
        if self.ctx is not None:
            ds.dslide_destroy(self.ctx)


class _Tensors(dict):
    """The context's own tensors by name, as dslide_get_tensor gives them to whoever looks one up."""

    def __init__(self, model, names):
        super().__init__((n, None) for n in names)
        self.model = model

    def __getitem__(self, name):
        return ds.dslide_get_tensor(self.model.ctx, name)


MODEL_TENSORS = ["W1", "b1", "W2", "b2", "mW1", "vW1", "mb1", "vb1", "mW2", "vW2", "mb2", "vb2"]


def prepare(case, seed):
    m = _Model(case, seed)
    B, kind = case["batch"], case["kind"]
    if kind == "rebuild":
        m.tables = _Tensors(m, ["hash_idx", "bucket_off", "bucket_ids"] + (["hash_sign"] if case["family"] == SIMHASH else []))
        return m
    m.tensors = _Tensors(m, MODEL_TENSORS)
    m.batches = _batches(case, seed, BATCHES if kind.startswith("train") else 1)
    if kind != "train_host":
        m.batches = [[torch.from_numpy(a).cuda() for a in b] for b in m.batches]
    m.loss = torch.zeros(1, device="cuda")
    m.ids = torch.empty(B * case["k"], dtype=torch.int32, device="cuda")
    m.scores = torch.empty(B * case["k"], device="cuda")
    torch.cuda.synchronize()
    return m


def run(m):
    c, B = m.c, m.c["batch"]
    if c["kind"] == "rebuild":
        ds.dslide_rebuild_tables(m.ctx)
        return m.tables
    b = m.batches[m.turn % len(m.batches)]
    m.turn += 1
    if c["kind"] == "train":
        ds.dslide_train_step(m.ctx, B, *b, m.loss)
        return {"loss": m.loss, "model": m.tensors}
    if c["kind"] == "train_host":
        return {"loss": ds.dslide_train_step_host_async(m.ctx, B, *b), "model": m.tensors}      # the step before's loss
    ds.dslide_predict_topk(m.ctx, B, b[0], b[1], b[2], c["k"], c["kind"] == "predict_all", m.ids, m.scores)
    return {"ids": m.ids, "scores": m.scores}


# ---- what a pass cannot do without --------------------------------------------------------------------
def _distinct(M, draws):
    """Distinct ids among so many Zipf draws from [0, M)."""
    p = np.arange(1, M + 1, dtype=np.float64) ** -ZIPF_S
    return float(-np.expm1(draws * np.log1p(-np.minimum(p / p.sum(), 0.999999))).sum())


def work(case):
    c = case
    B, H, N, L = c["batch"], c["H"], c["N"], c["L"]
    bits = c["K"] * (1 if c["family"] == SIMHASH else 3)
    nz = B * c["nnz"]
    if c["kind"] == "rebuild":
        fn = c["K"] * L * (BIN if c["family"] == DWTA else (H + 2) // 3)
        return {"bytes": 4.0 * H * N + 4.0 * N * L + 4.0 * L * (2 ** bits + 1), "flops": float(N) * fn}
    u1 = min(nz, _distinct(c["D"], nz))
    read = 8.0 * nz + 4 * (B + 1) + 4.0 * H * u1
    if c["kind"] == "predict_all":
        return {"bytes": read + 4.0 * (H + 1) * N + 8.0 * B * c["k"], "flops": 2.0 * H * (nz + float(B) * N)}
    got, pool = _retrieved(c)
    rows = pool * -math.expm1(-B * got / pool)
    if c["kind"] == "predict":
        return {"bytes": read + 8.0 * B * L + 4.0 * B * got + 4.0 * (H + 1) * rows + 8.0 * B * c["k"], "flops": 2.0 * H * (nz + B * got)}
    act = B * (got + c["labels"])
    u2 = rows + min(B * c["labels"], _distinct(N, B * c["labels"]))
    return {"bytes": 8.0 * nz + 4.0 * B * c["labels"] + 8.0 * (B + 1) + 24.0 * H * u1 + 24.0 * (H + 1) * u2 + 24.0 * H + 8.0 * B * L + 4.0 * act,
            "flops": 4.0 * H * nz + 6.0 * H * act + 12.0 * H * (u1 + u2)}


def tolerance(case):
    if case["kind"] == "rebuild":
        return "exact"
    # 32-bit sums: the scores are within 2e-7 of exact(), the gradients' moments within 7e-7.  Ids differ where two scores
    # tie.  A weight whose gradient cancels to rounding moves by up to the learning rate either way: 2e-4 over weights of 0.05.
    if case["kind"].startswith("predict"):
        return {"rel": 1e-6, "max": 1e-5, "differ": 0.002}
    return {"rel": 5e-6, "max": 1e-2}


# ---- the same results in 64 bits, from the definitions --------------------------------------------------
def _codes(c, X, idx, sign):
    """Bucket codes [rows, L] of the rows of X (32 bits: the codes are defined on 32-bit sums and comparisons)."""
    K, L = c["K"], c["L"]
    if c["family"] == DWTA:
        best, at = X[:, idx[:, 0]], torch.zeros(X.shape[0], idx.shape[0], dtype=torch.int32, device=X.device)
        for i in range(1, BIN):
            v = X[:, idx[:, i]]
            at = torch.where(v > best, i, at)
            best = torch.maximum(best, v)
        shift = 3
    else:
        s = torch.zeros(X.shape[0], idx.shape[0], device=X.device)
        for i in range(idx.shape[1]):
            s += X[:, idx[:, i]] * sign[:, i]
        at, shift = (s >= 0).int(), 1
    w = (1 << (shift * torch.arange(K, device=X.device))).int()
    return (at.view(-1, L, K) * w).sum(2, dtype=torch.int32)


def _hidden(c, W, ptr, cols, vals):
    """Hidden activations in 64 bits, and as the chain of 32-bit multiply-adds in stored order that the codes are taken of."""
    B, dev = c["batch"], "cuda"
    ptr, cols, vals = (torch.from_numpy(a).to(dev) for a in (ptr, cols, vals))
    n = (ptr[1:] - ptr[:-1]).long()
    h64 = W["b1"].double().repeat(B, 1)
    h32 = W["b1"].repeat(B, 1)
    for i in range(int(n.max())):
        s = (n > i).nonzero()[:, 0]
        e = ptr[s].long() + i
        t = vals[e].double()[:, None] * W["W1"][cols[e].long()].double()
        h64[s] += t
        h32[s] = (h32[s].double() + t).float()
    return h64.clamp_min(0), h32.clamp_min(0)


def _active(c, W, h32, seed):
    """[B, N] truth values: the neurons that the samples' buckets hold, the lowest ids of each up to the cap."""
    idx, sign = _hash_functions(c, seed)
    idx = torch.from_numpy(idx).cuda().long()
    sign = torch.from_numpy(sign).cuda().float() if sign is not None else None
    N = c["N"]
    step = max(1, 250000000 // (c["K"] * c["L"]))
    codes = torch.cat([_codes(c, W["W2"][a:a + step], idx, sign) for a in range(0, N, step)])
    query = _codes(c, h32, idx, sign)
    act = torch.zeros(c["batch"], N, dtype=torch.bool, device="cuda")
    row = torch.arange(c["batch"], device="cuda")[:, None]
    for t in range(c["L"]):
        srt, order = torch.sort(codes[:, t], stable=True)
        q = query[:, t].contiguous()
        beg, end = torch.searchsorted(srt, q), torch.searchsorted(srt, q, right=True)
        at = beg[:, None] + torch.arange(c["cap"], device="cuda")
        ok = at < end[:, None]
        act[row.expand_as(at)[ok], order[at[ok]]] = True
    return act


def _adam(w, g, on):
    """One first step of Adam from zero moments where `on`: (weights, first moments, second moments)."""
    m, v = (1 - BETA1) * g, (1 - BETA2) * g * g
    new = w - LR * (m / (1 - BETA1)) / (torch.sqrt(v / (1 - BETA2)) + EPS)
    return torch.where(on, new, w), m, v


def exact(case, seed):
    c = case
    if c["kind"] == "rebuild" or not _own_weights(c) or c["budget"] or c["densify"]:
        return None
    B, N, k = c["batch"], c["N"], c["k"]
    W = _weights(c, seed, "cuda")
    ptr, cols, vals, lptr, labs = _batches(c, seed, 1)[0]
    h, h32 = _hidden(c, W, ptr, cols, vals)
    act = _active(c, W, h32, seed) if c["kind"] != "predict_all" else None
    b2 = W["b2"].double()
    if c["kind"].startswith("predict"):
        ids, scores = [], []
        for a in range(0, B, 64):
            if act is None:
                z = torch.cat([h[a:a + 64] @ W["W2"][j:j + 100000].double().T for j in range(0, N, 100000)], 1) + b2
            else:
                z = torch.full((h[a:a + 64].shape[0], N), -math.inf, dtype=torch.float64, device="cuda")
                for s in range(z.shape[0]):
                    j = act[a + s].nonzero()[:, 0]
                    z[s, j] = W["W2"][j].double() @ h[a + s] + b2[j]
            v, i = torch.topk(z, k, 1)
            scores.append(v)
            ids.append(torch.where(torch.isinf(v), -1, i))
        return {"ids": torch.cat(ids).int().reshape(-1), "scores": torch.cat(scores).reshape(-1)}
    lrow = torch.from_numpy(np.repeat(np.arange(B), np.diff(lptr))).cuda()
    labs = torch.from_numpy(labs).cuda().long()
    act[lrow, labs] = True
    ny = torch.bincount(lrow, minlength=B).double()
    gW2 = torch.zeros(N, c["H"], dtype=torch.float64, device="cuda")
    gb2 = torch.zeros(N, dtype=torch.float64, device="cuda")
    dh = torch.zeros_like(h)
    loss = torch.zeros(B, dtype=torch.float64, device="cuda")
    for s in range(B):
        j = act[s].nonzero()[:, 0]
        w = W["W2"][j].double()
        logp = torch.log_softmax(w @ h[s] + b2[j], 0)
        y = torch.searchsorted(j, labs[lptr[s]:lptr[s + 1]])
        loss[s] = -logp[y].mean()
        g = logp.exp()
        g[y] -= 1 / ny[s]
        g /= B
        dh[s] = g @ w
        gW2[j] += g[:, None] * h[s]
        gb2[j] += g
    dh = torch.where(h > 0, dh, 0.0)
    gW1 = torch.zeros(c["D"], c["H"], dtype=torch.float64, device="cuda")
    row = torch.from_numpy(np.repeat(np.arange(B), np.diff(ptr))).cuda()
    cols = torch.from_numpy(cols).cuda().long()
    gW1.index_add_(0, cols, torch.from_numpy(vals).cuda().double()[:, None] * dh[row])
    on1 = torch.zeros(c["D"], 1, dtype=torch.bool, device="cuda")
    on1[cols] = True
    on2 = act.any(0)
    out = {}
    for name, g, on in (("W1", gW1, on1), ("b1", dh.sum(0), torch.ones_like(dh[0], dtype=torch.bool)), ("W2", gW2, on2[:, None]), ("b2", gb2, on2)):
        w, m, v = _adam(W[name].double(), g, on)
        out.update({name: w.reshape(-1), "m" + name: m.reshape(-1), "v" + name: v.reshape(-1)})
    return {"loss": loss.mean().reshape(1) if c["kind"] == "train" else None, "model": out}
