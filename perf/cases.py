"""Performance cases of the turn-aware OPD loss: what a training program has this library do, through its public
entry points.

A case is a plain dict.  Common keys:

``path``    "logits" (the loss step on stored logits), "topk" (the teacher top-K loss), "fused" (both LM heads inside
            the loss) or "shard" (one rank of the vocabulary-parallel split)
``batch``   the turn structure of the packed batch: "even" (alternating spans of 16), "packed" (long dense turns),
            "household" (short actions between observations, a masked tail) or "multihop" (ragged, heavy-tailed)
``traj``, ``len``  trajectories, and tokens of each (multihop: the longest)
``vocab``, ``ld``  vocabulary, and the row stride of the logits in elements

The number of tokens and of supervised tokens follows from the case alone; the seed draws every value and the order of
the trajectories.  A pass is what a training step runs on one batch: blend weights, loss and gradient, turn statistics.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2607_05804_gb300 as lib
from paper_2607_05804_gb300.step import LossStep

V_MAIN = 151_936
TYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
BYTES = {"bf16": 2, "f32": 4, "none": 0}
MAX_TURNS = {"even": 4, "packed": 30, "household": 50, "multihop": 12}


def listed():
    """Twelve cases: the smallest call, ordinary ones of each path, data type and option, and the largest."""
    return [
        # a unit-test or debugging batch: two short trajectories, fp32 rows, one row per token; launches are all it costs
        dict(name="tiny_f32_dense", path="logits", batch="even", traj=2, len=128, vocab=1024, ld=1024, logits="f32",
             grad="f32", mode="full", layout="dense", zero_masked=False, alpha=0.5, floor=False),
        # KL of a short probe trajectory for the depth controller: losses and turn statistics, no gradient
        dict(name="probe_forward", path="logits", batch="packed", traj=1, len=1024, vocab=V_MAIN, ld=V_MAIN,
             logits="bf16", grad="none", mode="full", layout="compact", zero_masked=False, alpha=0.5, floor=False),
        # the ordinary training step: 8 trajectories of 4096 tokens, bf16 logits and gradient
        dict(name="packed_bf16", path="logits", batch="packed", traj=8, len=4096, vocab=V_MAIN, ld=V_MAIN,
             logits="bf16", grad="bf16", mode="full", layout="compact", zero_masked=False, alpha=0.5, floor=False),
        # household tasks with the turn-reliability floor; the gradient kept in fp32 for an fp32 head
        dict(name="household_f32_grad", path="logits", batch="household", traj=16, len=8192, vocab=V_MAIN, ld=V_MAIN,
             logits="bf16", grad="f32", mode="full", layout="compact", zero_masked=False, alpha=0.5, floor=True),
        # long ragged search rollouts with the one-sample estimator: most tokens are observations
        dict(name="multihop_sampled", path="logits", batch="multihop", traj=64, len=16384, vocab=V_MAIN, ld=V_MAIN,
             logits="bf16", grad="bf16", mode="sampled", layout="compact", zero_masked=False, alpha=0.5, floor=False),
        # fp32 logits and gradient, as a program without mixed precision has them
        dict(name="packed_f32", path="logits", batch="packed", traj=4, len=4096, vocab=V_MAIN, ld=V_MAIN,
             logits="f32", grad="f32", mode="full", layout="compact", zero_masked=False, alpha=0.5, floor=False),
        # a vocabulary that nobody padded: an odd row stride; one row per token, masked rows zeroed, as autograd wants it
        dict(name="odd_vocab_dense", path="logits", batch="packed", traj=4, len=1024, vocab=50_001, ld=50_001,
             logits="bf16", grad="bf16", mode="full", layout="dense", zero_masked=True, alpha=0.5, floor=False),
        # the practical loss of the method, K = 50, on the ragged batch: sparse ids and gradient
        dict(name="multihop_topk50", path="topk", batch="multihop", traj=64, len=16384, vocab=V_MAIN, ld=V_MAIN,
             logits="bf16", grad="none", k=50, alpha=0.5),
        # a wider support with a dense gradient for autograd
        dict(name="packed_topk256_dense", path="topk", batch="packed", traj=4, len=4096, vocab=V_MAIN, ld=V_MAIN,
             logits="bf16", grad="bf16", k=256, alpha=0.5),
        # one micro-batch of a memory-bound program: hidden states and heads in, both gradients out
        dict(name="fused_micro_dw", path="fused", batch="packed", traj=1, len=512, vocab=V_MAIN, d_s=4096, d_t=5120,
             dw=True, alpha=1.0),
        # the same path at full size with a frozen head
        dict(name="fused_8x2048", path="fused", batch="packed", traj=8, len=2048, vocab=V_MAIN, d_s=4096, d_t=5120,
             dw=False, alpha=1.0),
        # one rank of a 4-way vocabulary-parallel head: statistics, merge, its own gradient columns
        dict(name="shard_4way", path="shard", batch="packed", traj=4, len=4096, vocab=V_MAIN, shards=4, rank=1,
             logits="bf16", grad="bf16", alpha=0.5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _vocab(rng, lo, hi):
    """A vocabulary over the logarithm of its range: half padded to 64, a quarter a multiple of 8, a quarter as it comes."""
    v, kind = _log(rng, lo, hi), rng.random()
    return max(64, v // 64 * 64) if kind < 0.5 else v // 8 * 8 if kind < 0.75 else v


def draw(rng):
    """One more case of the same ranges."""
    path = rng.choices(("logits", "topk", "fused", "shard"), (50, 20, 12, 18))[0]
    while True:
        batch = rng.choices(("even", "packed", "household", "multihop"), (1, 5, 2, 2))[0]
        c = dict(path=path, batch=batch, traj=_log(rng, 1, 64), alpha=round(rng.random(), 3))
        if batch == "multihop":
            c["len"] = _log(rng, 1024, 16384)
        else:
            c["len"] = _log(rng, 128, 8192) if batch != "even" else 32 * rng.randint(1, 4)
        if path == "fused":
            c.update(vocab=_vocab(rng, 8192, V_MAIN), d_s=256 * rng.randint(4, 16), d_t=64 * rng.randint(16, 80),
                     dw=rng.random() < 0.5)
        elif path == "shard":
            c.update(vocab=_vocab(rng, 16_384, V_MAIN), shards=rng.choice((2, 4, 8)), logits=rng.choice(("bf16", "bf16", "f32")))
            c.update(rank=rng.randrange(c["shards"]), grad=c["logits"])
        else:
            c.update(vocab=_vocab(rng, 1024, V_MAIN), logits=rng.choice(("bf16", "bf16", "f32")))
            c["ld"] = c["vocab"] if rng.random() < 0.5 else (c["vocab"] + 63) // 64 * 64
            if path == "topk":
                c.update(k=_log(rng, 8, 256), grad=rng.choice(("none", "none", c["logits"])))
            else:
                c.update(grad=rng.choice((c["logits"], c["logits"], "f32", "none")), mode=rng.choice(("full", "full", "sampled")),
                         layout=rng.choice(("compact", "compact", "dense")), floor=rng.random() < 0.3)
                c["zero_masked"] = c["layout"] == "dense" and c["grad"] != "none" and rng.random() < 0.5
        rows, T = _layout(c)["supervised"], _layout(c)["tokens"]
        stored = T if c.get("layout") == "dense" else rows
        if rows < 16 or stored * c["vocab"] > 3_000_000_000 or (path == "fused" and T > 16_384):
            continue
        return c


# ---------------------------------------------------------------- batches

def _fit(lengths, total):
    cum = np.cumsum(np.asarray(lengths, np.int64))
    cum = np.round(cum * (total / cum[-1])).astype(np.int64)
    cum[-1] = total
    return np.diff(np.concatenate([[0], cum]))


def _spans(batch, n, length, rng):
    """Span lengths of one trajectory, observation and action in turn."""
    if batch == "even":
        return [16] * (length // 16)
    if batch == "packed":
        turns = int(min(rng.integers(10, 31), max(1, length // 8)))
        total = rng.geometric(1.0 / 150.0, size=turns) + 2
        obs = np.round(0.4 * total).astype(np.int64)
        inter = np.empty(2 * turns, np.int64)
        inter[0::2], inter[1::2] = obs, total - obs
        return list(_fit(inter, length))
    if batch == "household":
        out = []
        for _ in range(int(rng.integers(10, 51))):
            out += [int(rng.integers(100, 301)), int(rng.integers(10, 41))]
        return out
    turns = int(rng.integers(2, 13))
    obs = rng.integers(200, 1501, size=turns).astype(np.int64)
    act = np.minimum(np.floor(8.0 * (1.0 + rng.pareto(1.5, size=turns))), 2000).astype(np.int64)
    if obs.sum() + act.sum() < length:
        obs = _fit(obs, max(turns, length - int(act.sum())))
    out = np.empty(2 * turns, np.int64)
    out[0::2], out[1::2] = obs, act
    return list(out)


@functools.lru_cache(maxsize=64)
def _trajectories(batch, n, length):
    """The trajectories of a batch: (turn_id, loss_mask) of each."""
    rng = np.random.default_rng([n, length])
    out = []
    for b in range(n):
        want = length if batch != "multihop" else int(rng.integers(512, length + 1))
        tid, msk = np.full(want, -1, np.int32), np.zeros(want, np.uint8)
        at = turn = 0
        for k, span in enumerate(_spans(batch, n, want, rng)):
            end = min(want, at + int(span))
            if k % 2 and end > at:
                tid[at:end], msk[at:end] = turn, 1
                turn += 1
            at = end
        out.append((tid, msk))
    return out


def _layout(case):
    t = _trajectories(case["batch"], case["traj"], case["len"])
    return dict(tokens=sum(x.size for x, _ in t), supervised=int(sum(int(m.sum()) for _, m in t)))


def _batch(case, seed):
    """The batch on the GPU, its trajectories in an order drawn from the seed."""
    t = _trajectories(case["batch"], case["traj"], case["len"])
    order = np.random.default_rng(seed).permutation(len(t))
    tid, msk = (np.concatenate([t[b][k] for b in order]) for k in (0, 1))
    off = np.concatenate([[0], np.cumsum([t[b][0].size for b in order])]).astype(np.int64)
    rows = np.full(tid.size, -1, np.int32)
    at = np.nonzero(msk)[0]
    rows[at] = np.arange(at.size, dtype=np.int32)
    put = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    return dict(turn_id=put(tid), loss_mask=put(msk), offsets=put(off), rows=put(rows), at=put(at.astype(np.int64)))


def _logits(rows, vocab, ld, dtype, seed):
    """Student and teacher logits of one vocabulary: correlated normals, five ids in common that stand out."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    zs = torch.zeros((rows, ld), dtype=dtype, device="cuda")
    zt = torch.zeros((rows, ld), dtype=dtype, device="cuda")
    step = max(1, 200_000_000 // vocab)
    for r in range(0, rows, step):
        n = min(step, rows - r)
        a = torch.randn((n, vocab), generator=gen, device="cuda").mul_(3.0)
        b = torch.randn((n, vocab), generator=gen, device="cuda").mul_(1.8).add_(a, alpha=0.8)
        ids = torch.randint(vocab, (n, 5), generator=gen, device="cuda")
        a.scatter_(1, ids, a.gather(1, ids) + 8.0)
        b.scatter_(1, ids, b.gather(1, ids) + 8.0)
        zs[r:r + n, :vocab] = a
        zt[r:r + n, :vocab] = b
    return zs, zt


def _sample(zs, vocab, seed):
    """One token of each row, drawn from the student's softmax."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 77)
    out = torch.empty(zs.shape[0], dtype=torch.int32, device="cuda")
    step = max(1, 200_000_000 // vocab)
    for r in range(0, zs.shape[0], step):
        z = zs[r:r + step, :vocab].float()
        e = torch.empty_like(z).exponential_(generator=gen).clamp_(min=1e-30)
        out[r:r + step] = torch.argmax(z - e.log_(), dim=1).to(torch.int32)
    return out


def _heads(tokens, case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def one(n, d, std):
        out = torch.empty((n, d), dtype=torch.bfloat16, device="cuda")
        step = max(1, 200_000_000 // d)
        for r in range(0, n, step):
            m = min(step, n - r)
            out[r:r + m] = torch.randn((m, d), generator=gen, device="cuda").mul_(std)
        return out

    V, ds, dt = case["vocab"], case["d_s"], case["d_t"]
    return one(tokens, ds, 1.0), one(V, ds, 0.02), one(tokens, dt, 1.0), one(V, dt, 0.02)


def _cuts(case):
    n, r = case["shards"], case["rank"]
    return case["vocab"] * r // n, case["vocab"] * (r + 1) // n


def _shard_statistics(zs, zt):
    """(m_s, S_s, A, d, m_t, S_t) of each row of a shard, in the dtype of the arguments."""
    ms, at = zs.max(dim=1, keepdim=True)
    mt = zt.max(dim=1, keepdim=True).values
    e, x = torch.exp(zs - ms), zs - zt
    d = x.gather(1, at)
    return torch.cat([ms, e.sum(1, keepdim=True), (e * (x - d)).sum(1, keepdim=True), d, mt,
                      torch.exp(zt - mt).sum(1, keepdim=True)], dim=1)


# ---------------------------------------------------------------- a pass

def _inputs(case, seed):
    b = _batch(case, seed)
    T, R = b["turn_id"].numel(), b["at"].numel()
    if case["path"] == "fused":
        b["h_s"], b["W_s"], b["h_t"], b["W_t"] = _heads(T, case, seed)
        return b
    dense = case.get("layout") == "dense"
    ld = case["vocab"] if case["path"] == "shard" else case["ld"]
    b["zs"], b["zt"] = _logits(T if dense else R, case["vocab"], ld, TYPES[case["logits"]], seed)
    if dense:
        b["rows"] = None
    if case.get("mode") == "sampled":
        y = _sample(b["zs"], case["vocab"], seed)
        if not dense:
            full = torch.zeros(T, dtype=torch.int32, device="cuda")
            full[b["at"]] = y
            y = full
        b["y"] = y
    return b


def prepare(case, seed):
    """The batch and the step object with its buffers, as a training program holds them before the call."""
    s = _inputs(case, seed)
    path, T = case["path"], s["turn_id"].numel()
    mode = lib.TURNOPD_SAMPLED_TOKEN if case.get("mode") == "sampled" else lib.TURNOPD_FULL_VOCAB
    s["step"] = LossStep(s["turn_id"], s["loss_mask"], s["offsets"], MAX_TURNS[case["batch"]], case["vocab"],
                         row_of_token=s["rows"], sampled_ids=s.get("y"), mode=mode, alpha=case["alpha"],
                         n_min=lib.turnopd_turn_floor(case["traj"]) if case.get("floor") else 0,
                         flags=lib.TURNOPD_ZERO_MASKED_GRAD if case.get("zero_masked") else 0, k_top=case.get("k", 0))
    s["path"] = path
    if path == "fused":
        s["ws"] = torch.empty(lib.turnopd_fused_workspace_bytes(T, case["vocab"], case["d_s"], case["d_t"]),
                              dtype=torch.uint8, device="cuda")
        s["dh"] = torch.zeros((T, case["d_s"]), dtype=torch.float32, device="cuda")
        s["dW"] = torch.zeros((case["vocab"], case["d_s"]), dtype=torch.float32, device="cuda") if case["dw"] else None
        return s
    if path == "shard":
        # the other ranks' partial statistics, as the all-gather delivers them (this rank's own are written into their
        # slot by the pass; they are no output, since the reference difference of a tied maximum is either one's)
        s["parts"] = torch.zeros((case["shards"], T, 6), dtype=torch.float32, device="cuda")
        s["merged"] = torch.zeros((T, 6), dtype=torch.float32, device="cuda")
        V, n = case["vocab"], case["shards"]
        for k in range(n):
            if k != case["rank"]:
                lo, hi = V * k // n, V * (k + 1) // n
                s["parts"][k, s["at"]] = _chunked(lambda a, b: _shard_statistics(a[:, lo:hi].float(), b[:, lo:hi].float()),
                                                  s["zs"], s["zt"])
        lo, hi = _cuts(case)
        s["zs"], s["zt"] = s["zs"][:, lo:hi].contiguous(), s["zt"][:, lo:hi].contiguous()
        s["own"] = s["parts"][case["rank"]]
    grad = case["grad"]
    s["grad"] = None if grad == "none" else torch.zeros(s["zs"].shape, dtype=TYPES[grad], device="cuda")
    return s


def run(s):
    """One step: blend weights, loss and gradient, turn statistics."""
    step = s["step"]
    out = {}
    if s["path"] == "fused":
        step.weights()
        lib.turnopd_fused_lmhead_fwd_bwd(s["h_s"], s["W_s"], s["h_t"], s["W_t"], step.loss_mask, step.w[:step.T],
                                         lib.TURNOPD_FULL_VOCAB, s["dh"], step.token_loss[:step.T], step.loss, s["ws"],
                                         step.dev_status, dW_s_out=s["dW"])
        step.turn_stats()
        out["dh"] = s["dh"]
        if s["dW"] is not None:
            out["dW"] = s["dW"]
    elif s["path"] == "shard":
        step.weights()
        lib.turnopd_vocab_shard_stats(s["zs"], s["zt"], step.row_of_token, step.loss_mask, s["own"], step.ws_l,
                                      step.dev_status)
        lib.turnopd_vocab_stats_merge(s["parts"], step.loss_mask, s["merged"])
        lib.turnopd_vocab_shard_loss_grad(s["zs"], s["zt"], step.row_of_token, step.loss_mask, step.w[:step.T],
                                          s["merged"], s["grad"], 0, step.token_loss[:step.T], step.loss, step.ws_l,
                                          step.dev_status)
        step.turn_stats()
    else:
        step.run(s["zs"], s["zt"], s["grad"])
    if s.get("grad") is not None:
        out["grad"] = s["grad"]
    if step.k_top:
        out["topk_ids"], out["topk_grad"] = step.topk_ids, step.topk_grad
    out.update(loss=step.loss, token_loss=step.token_loss, weights=step.w, turn_sum=step.turn_sum,
               turn_cnt=step.turn_cnt, turn_surv=step.turn_surv, traj_turn_sum=step.traj_turn_sum,
               traj_turn_cnt=step.traj_turn_cnt, status=step.dev_status)
    return out


# ---------------------------------------------------------------- what a pass needs

def work(case):
    n = _layout(case)
    T, R, V = n["tokens"], n["supervised"], case["vocab"]
    # turn id, mask, row index in; weight and loss out (and read again by the loss and the statistics)
    tokens = 17.0 * T
    if case["path"] == "fused":
        ds, dt = case["d_s"], case["d_t"]
        flops = 2.0 * R * V * (ds + dt) + 2.0 * R * V * ds * (2 if case["dw"] else 1)
        return {"bytes": tokens + 2.0 * V * (ds + dt) + 2.0 * R * (ds + dt) + 4.0 * T * ds + (4.0 * V * ds if case["dw"] else 0.0),
                "flops": flops}
    esz, gsz = BYTES[case["logits"]], BYTES[case["grad"]]
    if case["path"] == "shard":
        # the statistics and the gradient are two calls with the exchange between them: each reads the shard
        lo, hi = _cuts(case)
        return {"bytes": tokens + float(R) * (hi - lo) * (4 * esz + gsz), "flops": 20.0 * R * (hi - lo)}
    if case["path"] == "topk":
        k = case["k"]
        return {"bytes": tokens + float(R) * (V * (esz + gsz) + k * (esz + 8)), "flops": float(R) * V}
    zeros = float(T - R) * V * gsz if case["zero_masked"] else 0.0
    return {"bytes": tokens + float(R) * V * (2 * esz + gsz) + zeros, "flops": 20.0 * R * V}


def tolerance(case):
    """About four times the error against 64 bits, over all outputs.  fp32 results are 1e-6 off: the rounding of sums over
    the vocabulary and of the exponents' arguments.  bf16 gradients are 1.5e-3 to 2.8e-3 off, each value rounded once to 8
    bits; the fused path rounds dL/dz to bf16 before its second product."""
    if case["path"] == "fused" or case["grad"] == "bf16":
        return {"rel": 1e-2, "max": 0.05}
    return {"rel": 5e-6, "max": 2e-4}


# ---------------------------------------------------------------- 64 bits

def _chunked(f, *rows):
    step = max(1, 60_000_000 // rows[0].shape[1])
    return torch.cat([f(*(x[r:r + step] for x in rows)) for r in range(0, rows[0].shape[0], step)])


def _weights64(case, b):
    """w = [(1 - alpha) / N_b + alpha share] / B' per supervised token, in 64 bits."""
    B, Tm, a = case["traj"], MAX_TURNS[case["batch"]], case["alpha"]
    at = b["at"]
    traj = torch.bucketize(at, b["offsets"][1:], right=True)
    key = traj * Tm + b["turn_id"][at].long()
    n_bt = torch.bincount(key, minlength=B * Tm).reshape(B, Tm)
    N, S = n_bt.sum(1), (n_bt > 0).sum(0)
    n_min = max(8, math.ceil(0.15 * B - 1e-9)) if case.get("floor") else 0
    rel = (S >= n_min)[None, :] & (n_bt > 0) if n_min > 0 else n_bt > 0
    unrel = torch.where(rel, 0, n_bt).sum(1)
    Nd, R = N.double().clamp(min=1), rel.sum(1)
    w_traj = (1.0 / Nd)[:, None].expand(B, Tm)
    w_turn = ((1.0 - unrel.double() / Nd) / R.double().clamp(min=1))[:, None] / n_bt.double().clamp(min=1)
    w_turn = torch.where(rel & (R > 0)[:, None], w_turn, w_traj)
    w = ((1.0 - a) * w_traj + a * w_turn) / max(1, int((N > 0).sum()))
    return w.reshape(-1)[key], key, n_bt, S


def exact(case, seed):
    """What run() returns, from plain torch in float64."""
    if case["path"] == "fused" and work(case)["flops"] > 1.2e13:
        return None
    b = _inputs(case, seed)
    w, key, n_bt, S = _weights64(case, b)
    at, T, V, Tm, B = b["at"], b["turn_id"].numel(), case["vocab"], MAX_TURNS[case["batch"]], case["traj"]
    full = lambda v: torch.zeros(T, dtype=torch.float64, device="cuda").index_copy_(0, at, v)  # noqa: E731
    out = {}
    if case["path"] == "fused":
        h = b["h_s"][at].double()
        zs, zt = h @ b["W_s"].double().T, b["h_t"][at].double() @ b["W_t"].double().T
    else:
        r = at if b["rows"] is None else b["rows"][at].long()
        zs, zt = b["zs"][:, :V], b["zt"][:, :V]
        if not torch.equal(r, torch.arange(zs.shape[0], device="cuda")):
            zs, zt = zs[r], zt[r]

    def row(i):
        """l, the gradient over the vocabulary, and (top-K) the support, of rows i."""
        x, t = zs[i].double(), zt[i].double()
        if case["path"] == "topk":
            # the lower id first among equal logits
            ids = torch.sort(t, dim=1, descending=True, stable=True).indices[:, :case["k"]]
            x, t = x.gather(1, ids), t.gather(1, ids)
        ls = torch.log_softmax(x, 1)
        lt = torch.log_softmax(t, 1)
        p, wi = ls.exp(), w[i, None]
        if case.get("mode") == "sampled":
            y = b["y"][at[i]].long()[:, None]
            ell = (ls - lt).gather(1, y)
            g = -wi * ell * p
            rest = p.scatter(1, y, 0.0).sum(1, keepdim=True)
            return ell, g.scatter(1, y, wi * ell * rest)
        d = ls.sub_(lt)
        ell = (p * d).sum(1, keepdim=True)
        g = wi * p * (d - ell)
        return (ell, g, ids) if case["path"] == "topk" else (ell, g)

    n, K = at.numel(), case.get("k", 0)
    ell = torch.empty(n, dtype=torch.float64, device="cuda")
    keep = case["path"] == "fused" or case["grad"] != "none"
    lo, hi = _cuts(case) if case["path"] == "shard" else (0, V)
    ld = hi - lo if case["path"] == "shard" else case.get("ld", V)
    G = None
    if keep:
        dense = case.get("layout") == "dense"
        G = torch.zeros((T if dense else n, ld), dtype=torch.float64, device="cuda")
    if K:
        out["topk_ids"] = torch.full((T, K), -1, dtype=torch.int32, device="cuda")
        out["topk_grad"] = torch.zeros((T, K), dtype=torch.float64, device="cuda")
    step = max(1, 60_000_000 // V)
    for r0 in range(0, n, step):
        i = torch.arange(r0, min(n, r0 + step), device="cuda")
        got = row(i)
        ell[i] = got[0][:, 0]
        rows = at[i] if case.get("layout") == "dense" else i
        if K:
            out["topk_ids"][at[i]], out["topk_grad"][at[i]] = got[2].int(), got[1]
            if keep:
                G[rows[:, None], got[2]] = got[1]
        elif keep:
            G[rows, :hi - lo] = got[1][:, lo:hi]
    if case["path"] == "fused":
        out["dh"] = torch.zeros((T, case["d_s"]), dtype=torch.float64, device="cuda")
        out["dh"][at] = G @ b["W_s"].double()
        if case["dw"]:
            out["dW"] = G.T @ h
    elif case["path"] == "shard":
        out["grad"] = G
    elif keep:
        out["grad"] = G
    sums = torch.zeros(B * Tm, dtype=torch.float64, device="cuda").index_add_(0, key, ell)
    out.update(loss=(w * ell).sum().reshape(1), token_loss=full(ell), weights=full(w), turn_sum=sums.reshape(B, Tm).sum(0),
               turn_cnt=n_bt.sum(0), turn_surv=S.int(), traj_turn_sum=sums, traj_turn_cnt=n_bt.reshape(-1).int(),
               status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    return out
