"""GPU parity of the teacher top-K reverse KL (turnopd_topk_loss_fwd_bwd)
against the fp64 oracle.

The selected ids are compared bit for bit (the selection is a decision on the
bf16/fp32 teacher logits, taken exactly on both sides).  Per-token loss and
total loss use the loss path's bounds; the gradient at the selected ids is
within 1e-4 of the row's largest |g| (fp32 output), and a dense gradient row
holds exactly those fp32 values (rounded to nearest even when it is bf16) at
the selected ids and zeros elsewhere.
"""
import numpy as np
import pytest

import workloads as W
from parity import assert_loss, assert_token_loss

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2607_05804_gb300 as P

    P.load()
    return P


def host(t):
    if t.dtype == torch.bfloat16:
        return t.view(torch.int16).cpu().numpy().view(np.uint16)
    return t.cpu().numpy()


def run_topk(P, zs, zt, V, mask, w, K, rot=None, dense=None, flags=0, ids_fill=-7, g_fill=9.0):
    T = mask.numel()
    dev = zs.device
    ids = torch.full((T, K), ids_fill, dtype=torch.int32, device=dev)
    gk = torch.full((T, K), g_fill, dtype=torch.float32, device=dev)
    tl = torch.full((T,), 5.0, dtype=torch.float32, device=dev)
    loss = torch.zeros(1, dtype=torch.float64, device=dev)
    st = torch.zeros(1, dtype=torch.int32, device=dev)
    ws = torch.empty(max(P.turnopd_loss_workspace_bytes(T), 256), dtype=torch.uint8, device=dev)
    P.turnopd_topk_loss_fwd_bwd(zs, zt, V, rot, mask, w, K, ids, gk, dense, flags, tl, loss, ws, st)
    torch.cuda.synchronize()
    return ids.cpu().numpy(), gk.cpu().numpy(), tl.cpu().numpy(), loss.item(), st.item()


def check_against_oracle(oracle, zs, zt, V, mask, w, K, ids, gk, tl, loss, rot=None, subset=None):
    m = mask.cpu().numpy()
    rids, rg, _, rtl, rloss = oracle.topk_loss(host(zs), host(zt), V, m, w.cpu().numpy(), K,
                                               row_of_token=None if rot is None else rot.cpu().numpy(),
                                               subset=subset)
    toks = np.nonzero(m)[0] if subset is None else np.asarray([t for t in subset if m[t]])
    np.testing.assert_array_equal(ids[toks], rids[toks])
    assert_token_loss(tl[toks], rtl[toks])
    rowmax = np.abs(rg[toks]).max(axis=1, keepdims=True)
    err = np.abs(gk[toks] - rg[toks])
    assert (err <= 1e-4 * rowmax + 1e-30).all(), float((err / np.maximum(rowmax, 1e-30)).max())
    if subset is None:
        assert_loss(loss, rloss)
    return rids, rg


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("K", [1, 5, 50])
def test_tiny_all_rows(P, oracle, dtype, K):
    b = W.tiny(seed=1)
    V = 1024
    zs, zt = W.make_logits(b.num_tokens, V, "tiny", dtype, seed=11, device="cuda")
    mask = torch.from_numpy(b.loss_mask).cuda()
    w = torch.rand(b.num_tokens, generator=torch.Generator().manual_seed(2)).cuda()
    ids, gk, tl, loss, st = run_topk(P, zs, zt, V, mask, w, K)
    assert st == 0
    check_against_oracle(oracle, zs, zt, V, mask, w, K, ids, gk, tl, loss)
    m = b.loss_mask == 0
    assert (tl[m] == 0).all()
    assert (ids[m] == -7).all() and (gk[m] == 9.0).all()  # masked rows untouched without the flag


def test_ties_and_signed_zero(P, oracle):
    """Rows built from few distinct dyadic bf16 values: many equal teacher
    logits around the K-th, and rows mixing +0 and -0."""
    g = torch.Generator().manual_seed(3)
    T, V, K = 64, 5000, 50
    levels = torch.tensor([-2.0, -1.0, -0.0, 0.0, 0.5, 1.0, 1.5], dtype=torch.float32)
    pick = torch.randint(0, len(levels), (T, V), generator=g)
    zt = levels[pick].to(torch.bfloat16)
    zs = (torch.randn(T, V, generator=g) * 2).to(torch.bfloat16)
    # a few rows with a unique top and otherwise all equal logits
    zt[5] = 0.0
    zt[5, 4321] = 1.0
    zt[6] = -0.0
    zt[6, 7] = 0.0
    zs, zt = zs.cuda(), zt.cuda()
    mask = torch.ones(T, dtype=torch.uint8, device="cuda")
    w = torch.full((T,), 0.5, dtype=torch.float32, device="cuda")
    ids, gk, tl, loss, st = run_topk(P, zs, zt, V, mask, w, K)
    assert st == 0
    check_against_oracle(oracle, zs, zt, V, mask, w, K, ids, gk, tl, loss)
    assert ids[5, 0] == 4321 and ids[5, 1:].tolist() == list(range(K - 1))
    assert ids[6].tolist() == list(range(K))


def test_all_equal_row_takes_the_lowest_ids(P, oracle):
    """Every teacher logit equal: the candidate buffer overflows and the
    selection settles by the id bytes."""
    T, V, K = 4, 151936, 50
    zt = torch.full((T, V), 0.75, dtype=torch.bfloat16, device="cuda")
    zs = torch.randn(T, V, generator=torch.Generator(device="cuda").manual_seed(4), device="cuda").to(torch.bfloat16)
    mask = torch.ones(T, dtype=torch.uint8, device="cuda")
    w = torch.ones(T, dtype=torch.float32, device="cuda")
    ids, gk, tl, loss, st = run_topk(P, zs, zt, V, mask, w, K)
    assert st == 0
    for i in range(T):
        assert ids[i].tolist() == list(range(K))
    check_against_oracle(oracle, zs, zt, V, mask, w, K, ids, gk, tl, loss, subset=[0, 3])


def test_k_equals_v_is_the_full_kl(P, oracle):
    T, V = 16, 256
    zs, zt = W.make_logits(T, V, "tiny", torch.float32, seed=5, device="cuda")
    mask = torch.ones(T, dtype=torch.uint8, device="cuda")
    w = torch.ones(T, dtype=torch.float32, device="cuda")
    ids, gk, tl, loss, st = run_topk(P, zs, zt, V, mask, w, V)
    assert st == 0
    _, tl_full, _ = oracle.loss_fwd_bwd(host(zs), host(zt), V, mask.cpu().numpy(), w.cpu().numpy(),
                                        grad=False)
    assert_token_loss(tl, tl_full)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_dense_gradient_misaligned_stride_and_zero_flag(P, oracle, dtype):
    """Row stride not a multiple of 16 bytes (the scalar path), dense gradient
    rows, compact rows through row_of_token, and TURNOPD_ZERO_MASKED_GRAD."""
    b = W.packed(seed=7, num_traj=2, traj_len=300)
    T, V, K = b.num_tokens, 3001, 50
    ld = 3003
    rows = b.num_valid
    zs, zt = W.make_logits(rows, V, "agent", dtype, seed=13, device="cuda", ld=ld)
    rot_np = np.full(T, -1, np.int32)
    rot_np[b.loss_mask == 1] = np.arange(rows, dtype=np.int32)
    rot = torch.from_numpy(rot_np).cuda()
    mask = torch.from_numpy(b.loss_mask).cuda()
    w = torch.rand(T, generator=torch.Generator().manual_seed(8)).cuda()
    dense = torch.full_like(zs, 3.0)
    ids, gk, tl, loss, st = run_topk(P, zs, zt, V, mask, w, K, rot=rot, dense=dense,
                                     flags=P.TURNOPD_ZERO_MASKED_GRAD)
    assert st == 0
    rids, rg = check_against_oracle(oracle, zs[:, :V], zt[:, :V], V, mask, w, K, ids, gk, tl, loss,
                                    rot=rot)
    m = b.loss_mask == 0
    assert (ids[m] == -1).all() and (gk[m] == 0).all()
    dn = dense.float().cpu().numpy()
    assert (dn[:, V:] == 3.0).all()  # padding columns untouched
    # the dense row holds the sparse fp32 values (checked against the oracle above),
    # rounded to nearest even in bf16, at the support ids and zeros elsewhere
    gk_dense = torch.from_numpy(gk).to(dtype).float().numpy()
    for t in np.nonzero(b.loss_mask)[0]:
        want = np.zeros(V, np.float32)
        want[ids[t]] = gk_dense[t]
        assert np.array_equal(dn[rot_np[t], :V], want)


@pytest.mark.parametrize("workload", ["packed", "household", "multihop"])
def test_full_vocab_sampled_rows_and_properties(P, oracle, workload):
    """The bench workloads at full size (packed 8 x 4096: 19,669 rows; household
    16 x 8192: 10,918; multihop, 64 ragged trajectories: 8,020; V = 151,936 bf16,
    compact rows): the oracle recomputes a few rows; every row is checked by the
    selection's defining properties."""
    b = W.CONFIGS[workload](seed=0)
    V, K = W.V_QWEN, 50
    R = b.num_valid
    zs, zt = W.make_logits(R, V, "agent", torch.bfloat16, seed=1000, device="cuda")
    T = b.num_tokens
    rot_np = np.full(T, -1, np.int32)
    rot_np[b.loss_mask == 1] = np.arange(R, dtype=np.int32)
    rot = torch.from_numpy(rot_np).cuda()
    mask = torch.from_numpy(b.loss_mask).cuda()
    w = torch.rand(T, generator=torch.Generator().manual_seed(9)).cuda()
    ids, gk, tl, loss, st = run_topk(P, zs, zt, V, mask, w, K, rot=rot)
    assert st == 0
    toks = np.nonzero(b.loss_mask)[0]
    pick = list(toks[:2]) + list(toks[-2:]) + list(np.random.default_rng(0).choice(toks, 6, replace=False))
    check_against_oracle(oracle, zs, zt, V, mask, w, K, ids, gk, tl, loss, rot=rot, subset=pick)
    # properties on every row: the selected teacher logits are the K largest, in order
    ar = torch.arange(V, device="cuda").unsqueeze(0)
    for c0 in range(0, toks.size, 2048):
        tk = toks[c0:c0 + 2048]
        sel = torch.from_numpy(ids[tk].astype(np.int64)).cuda()
        ztf = zt[torch.from_numpy(rot_np[tk].astype(np.int64)).cuda()].float()
        vals = torch.gather(ztf, 1, sel)
        assert bool((vals[:, :-1] >= vals[:, 1:]).all())
        eq = vals[:, :-1] == vals[:, 1:]
        assert bool((~eq | (sel[:, :-1] < sel[:, 1:])).all())
        ztf.scatter_(1, sel, -float("inf"))
        kth = vals[:, -1:]
        assert bool((ztf.max(dim=1, keepdim=True).values <= kth).all())
        # an unselected id equal to the K-th logit must come after every selected id of that logit
        last_eq_id = torch.where(vals == kth, sel, torch.full_like(sel, -1)).max(dim=1, keepdim=True).values
        assert not bool(((ztf == kth) & (ar < last_eq_id)).any())
    assert (tl[toks] >= -1e-6).all()
    assert abs(loss - float(np.dot(w.cpu().numpy().astype(np.float64)[toks], tl[toks].astype(np.float64)))) \
        <= 1e-6 * abs(loss)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("K", [65, 200, 256, 257, 513, 1024])
def test_large_k_full_vocab(P, oracle, dtype, K):
    """K above 64: the bound is the K-th largest group bucket; above 256
    candidates the buffer is sorted, and above K = 512 it holds 2,048."""
    V, T = W.V_QWEN, 6
    zs, zt = W.make_logits(T, V, "agent", dtype, seed=17 + K, device="cuda")
    mask = torch.ones(T, dtype=torch.uint8, device="cuda")
    w = torch.linspace(0.1, 1.0, T, dtype=torch.float32, device="cuda")
    ids, gk, tl, loss, st = run_topk(P, zs, zt, V, mask, w, K)
    assert st == 0
    check_against_oracle(oracle, zs, zt, V, mask, w, K, ids, gk, tl, loss)


@pytest.mark.parametrize("K", [50, 256, 1024])
def test_sorted_rows(P, oracle, K):
    """Teacher rows in ascending and descending id order, and a row with the
    top ids spread by a stride: orders that defeat sampling-based bounds."""
    V, T = W.V_QWEN, 3
    base = torch.linspace(-8.0, 8.0, V, dtype=torch.float32)
    zt = torch.stack([base, base.flip(0), base[torch.randperm(V, generator=torch.Generator().manual_seed(9))]])
    zt = zt.to(torch.bfloat16).cuda()
    zs = (torch.randn(T, V, generator=torch.Generator().manual_seed(10)) * 2).to(torch.bfloat16).cuda()
    mask = torch.ones(T, dtype=torch.uint8, device="cuda")
    w = torch.ones(T, dtype=torch.float32, device="cuda")
    ids, gk, tl, loss, st = run_topk(P, zs, zt, V, mask, w, K)
    assert st == 0
    check_against_oracle(oracle, zs, zt, V, mask, w, K, ids, gk, tl, loss)


def test_largest_vocabulary_and_largest_k(P, oracle):
    """V = TURNOPD_TOPK_MAX_VOCAB with K = TURNOPD_TOPK_MAX: the shared-memory layout at its
    largest (two rows of buckets, the K-sized arrays)."""
    V, K = P.TURNOPD_TOPK_MAX_VOCAB, P.TURNOPD_TOPK_MAX
    T = 3
    zs, zt = W.make_logits(T, V, "agent", torch.bfloat16, seed=31, device="cuda")
    mask = torch.ones(T, dtype=torch.uint8, device="cuda")
    w = torch.full((T,), 0.25, dtype=torch.float32, device="cuda")
    ids, gk, tl, loss, st = run_topk(P, zs, zt, V, mask, w, K)
    assert st == 0
    check_against_oracle(oracle, zs, zt, V, mask, w, K, ids, gk, tl, loss)


def test_empty_and_all_masked(P):
    V, K = 512, 8
    zs = torch.zeros((4, V), dtype=torch.bfloat16, device="cuda")
    mask = torch.zeros(4, dtype=torch.uint8, device="cuda")
    w = torch.ones(4, dtype=torch.float32, device="cuda")
    ids, gk, tl, loss, st = run_topk(P, zs, zs, V, mask, w, K)
    assert st == 0 and loss == 0.0 and (tl == 0).all()
    e = torch.zeros((0, V), dtype=torch.bfloat16, device="cuda")
    ids, gk, tl, loss, st = run_topk(P, e, e, V, torch.zeros(0, dtype=torch.uint8, device="cuda"),
                                     torch.zeros(0, dtype=torch.float32, device="cuda"), K)
    assert st == 0 and loss == 0.0


# Longest rows of the register-held selection, 64 elements a thread less 7 for the alignment,
# for CTAs of 32, 128, 256 and 512 threads, and one more (the last: the streaming kernel).
SHORT_EDGES = [64 * nt - 7 for nt in (32, 128, 256, 512)]


@pytest.mark.parametrize("V", [3, 9, 100] + [e + d for e in SHORT_EDGES for d in (0, 1)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_short_rows_at_the_edges(P, oracle, V, dtype):
    """Odd strides (rows start anywhere in a vector; the logits end with the last row's last
    column, NaN behind it), K = 1, 50 and 256, every row against the oracle; some rows hold
    many equal largest logits (more ties than the candidate buffer), signed zeros, and the
    type's lowest value outside their first ids; the dense gradient holds the sparse one and zeros."""
    T, ld = 24, V + 2
    gen = torch.Generator(device="cuda")
    gen.manual_seed(V)
    base = torch.randn((T, V), generator=gen, device="cuda") * 3
    zs0 = (base + torch.randn((T, V), generator=gen, device="cuda")).to(dtype)
    zt0 = base.to(dtype)
    zt0[1] = 1.5                               # all equal
    zt0[2, V // 3:] = 4.25                     # two thirds tied
    zt0[3, ::2], zt0[3, 1::2] = 0.0, -0.0      # signed zeros are one logit
    if V >= 600:
        zt0[4, 600:] = torch.finfo(dtype).min  # a masked vocabulary
    z = []
    for src in (zs0, zt0):
        buf = torch.full((T * ld + 64,), float("nan"), dtype=dtype, device="cuda")
        v = buf[3:3 + T * ld].view(T, ld)      # a base that is not 16-byte aligned
        v[:, :V] = src
        z.append(v)
    mask = torch.ones(T, dtype=torch.uint8, device="cuda")
    mask[7] = 0
    w = torch.rand(T, generator=gen, device="cuda")
    for K in sorted({1, min(50, V), min(256, V)}):
        if V >= 600 and K > 600:
            continue
        dense = torch.full((T, ld), 6.0, dtype=torch.float32, device="cuda")
        ids, gk, tl, loss, st = run_topk(P, z[0], z[1], V, mask, w, K, dense=dense)
        assert st == 0
        check_against_oracle(oracle, z[0].contiguous()[:, :V].contiguous(), z[1].contiguous()[:, :V].contiguous(), V,
                             mask, w, K, ids, gk, tl, loss)
        d = dense.cpu().numpy()
        assert (d[:, V:] == 6.0).all() and (d[7] == 6.0).all()
        for t in range(T):
            if t != 7:
                want = np.zeros(V, np.float32)
                want[ids[t]] = gk[t]
                np.testing.assert_array_equal(d[t, :V], want)


@pytest.mark.parametrize("V", [e // 8 * 8 + d for e in SHORT_EDGES[1:] for d in (0, 8)])
@pytest.mark.parametrize("K", [1, 63, 64, 239, 240, 289])
def test_aligned_rows_at_the_selection_lines(P, oracle, V, K):
    """Aligned rows on both sides of the lengths and the K from which they are streamed."""
    T = 12
    gen = torch.Generator(device="cuda")
    gen.manual_seed(V + K)
    zt = torch.randn((T, V), generator=gen, device="cuda") * 3
    zs = (zt + torch.randn((T, V), generator=gen, device="cuda")).to(torch.bfloat16)
    zt = zt.to(torch.bfloat16)
    mask = torch.ones(T, dtype=torch.uint8, device="cuda")
    mask[5] = 0
    w = torch.rand(T, generator=gen, device="cuda")
    ids, gk, tl, loss, st = run_topk(P, zs, zt, V, mask, w, K)
    assert st == 0
    check_against_oracle(oracle, zs, zt, V, mask, w, K, ids, gk, tl, loss)


@pytest.mark.parametrize("V,K,dense", [(131072, 320, False), (131088, 288, False), (131088, 289, False),
                                       (131088, 448, False), (131088, 449, False), (131088, 320, True),
                                       (14336, 50, True), (14352, 50, True), (14352, 128, True), (65536, 128, True),
                                       (65552, 50, True), (65552, 128, True)])
def test_fp32_rows_at_the_streaming_lines(P, oracle, V, K, dense):
    """fp32 rows on both sides of the lines between two and four selector warps, and between a dense
    row's zeros by the selector and by the streaming warps; more rows than CTAs at the short ones, so
    that a CTA's buffers come round."""
    T = 700 if V < 20000 else 12
    gen = torch.Generator(device="cuda")
    gen.manual_seed(V + K)
    zt = torch.randn((T, V), generator=gen, device="cuda") * 3
    zs = zt + torch.randn((T, V), generator=gen, device="cuda")
    zt[1] = 1.5
    mask = torch.ones(T, dtype=torch.uint8, device="cuda")
    mask[5] = 0
    w = torch.rand(T, generator=gen, device="cuda")
    d = torch.full((T, V), 6.0, dtype=torch.float32, device="cuda") if dense else None
    ids, gk, tl, loss, st = run_topk(P, zs, zt, V, mask, w, K, dense=d)
    assert st == 0
    sub = np.arange(0, T, 7) if T > 12 else None
    check_against_oracle(oracle, zs, zt, V, mask, w, K, ids, gk, tl, loss, subset=sub)
    if dense:
        want = torch.zeros((T, V), dtype=torch.float32, device="cuda")
        want.scatter_(1, torch.from_numpy(ids).cuda().long().clamp(min=0), torch.from_numpy(gk).cuda())
        want[5] = 6.0
        assert torch.equal(d, want)


@pytest.mark.parametrize("V,ld,K,threads", [(64, 64, 8, 32), (1040, 1041, 1024, 32), (2042, 2042, 8, 128),
                                            (2042, 2042, 320, 128), (8186, 8187, 64, 256), (16378, 16379, 20, 512)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_short_rows_many_to_a_cta(P, oracle, V, ld, K, threads, dtype):
    """Three rounds and more of the CTAs that an SM holds (32 of 32 threads, 1,024 threads' worth of
    the larger ones), so that a CTA takes several rows, their kinds in a varying order: ordinary,
    all equal, two thirds equal, more ties than the candidates or the list hold, masked by the
    lowest value, and rows without loss.  What a row leaves behind must not enter the next."""
    T = 152 * (32 if threads == 32 else 1024 // threads) * 3 + 77
    gen = torch.Generator(device="cuda")
    gen.manual_seed(V)
    zs = torch.empty((T, ld), dtype=dtype, device="cuda")
    zt = torch.empty((T, ld), dtype=dtype, device="cuda")
    kind = torch.randint(7, (T,), generator=gen, device="cuda")
    for r in range(0, T, 512):
        n = min(512, T - r)
        t = torch.randn((n, ld), generator=gen, device="cuda") * 3
        k = kind[r:r + n, None]
        s = 0.2 * t + 0.3 * torch.randn((n, ld), generator=gen, device="cuda")  # no token near p = 1, where g cancels
        zs[r:r + n] = torch.where(k == 4, s + 1000.0, s).to(dtype)
        col = torch.arange(ld, device="cuda")[None]
        t = torch.where(k == 1, 1.5, t)
        t = torch.where((k == 2) & (col >= V // 3), 4.25, t)
        t = torch.where((k == 3) & (col % 8 == 5), 9.0, t)          # an eighth of the ids tied at the top
        t = torch.where(k == 4, t + 1000.0, t)                      # few distinct leading bits
        t = torch.where((k == 5) & (col >= K + 9), torch.finfo(dtype).min, t)
        zt[r:r + n] = t.to(dtype)
    mask = (torch.rand(T, generator=gen, device="cuda") < 0.9).to(torch.uint8)
    w = torch.rand(T, generator=gen, device="cuda")
    dense = torch.full((T, ld), 6.0, dtype=torch.float32, device="cuda")
    ids, gk, tl, loss, st = run_topk(P, zs, zt, V, mask, w, K, dense=dense)
    assert st == 0
    check_against_oracle(oracle, zs, zt, V, mask, w, K, ids, gk, tl, loss)
    m = mask.bool()
    want = torch.zeros((T, ld), dtype=torch.float32, device="cuda")
    want.scatter_(1, torch.from_numpy(ids).cuda().long().clamp(min=0), torch.from_numpy(gk).cuda())
    assert torch.equal(dense[m][:, :V], want[m][:, :V])
    assert (dense[~m] == 6.0).all() and (dense[:, V:] == 6.0).all()
