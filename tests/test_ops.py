"""Single-kernel entry points against the oracle's per-operation functions."""
import numpy as np
import pytest

from oracle import mslt_oracle as O

pytestmark = pytest.mark.gpu


def run_cross_entropy(fn, dtype, logits, labels, V, want_grad=True, **kw):
    import torch
    R = logits.shape[0]
    ldl = (V + 7) // 8 * 8
    buf = torch.zeros((R, ldl), dtype=torch.float32, device="cuda")
    buf[:, :V] = torch.from_numpy(logits).cuda()
    d_lab = torch.from_numpy(labels.astype(np.int32)).cuda()
    dl = torch.full((R, ldl), 3.0, device="cuda", dtype=torch.float32 if dtype == 0 else torch.bfloat16) \
        if want_grad else None
    loss = torch.zeros(1, device="cuda")
    fn(dtype, buf, d_lab, V, dl, loss, stream=torch.cuda.current_stream().cuda_stream, **kw)
    return float(loss.item()), None if dl is None else dl.float().cpu().numpy()


@pytest.mark.parametrize("dtype", [0, 1], ids=["fp32", "bf16"])
@pytest.mark.parametrize("R,V", [(7, 11), (64, 1037), (300, 30522)])
def test_cross_entropy_matches_oracle(dtype, R, V):
    import torch
    from paper_2011_13635_b200 import binding as Bd
    rng = np.random.default_rng(R + V)
    logits = (rng.standard_normal((R, V)) * 3).astype(np.float32)
    labels = rng.integers(0, V, size=R)
    labels[::5] = -1
    n_valid = int((labels >= 0).sum())
    scratch = torch.empty(Bd.lib.mslt_op_cross_entropy_scratch_bytes(R), dtype=torch.uint8, device="cuda")
    loss, dl = run_cross_entropy(Bd.mslt_op_cross_entropy, dtype, logits, labels, V, scratch=scratch)
    want_loss, want_dl = O.cross_entropy(logits.astype(np.float64), labels, n_valid)
    assert abs(loss - want_loss) / want_loss < 1e-5
    tol = 1e-5 if dtype == 0 else 6e-3
    assert np.abs(dl[:, :V] - want_dl).max() / np.abs(want_dl).max() < tol
    assert np.all(dl[:, V:] == 0)                  # padding columns are cleared
    assert np.all(dl[labels < 0] == 0)             # ignored rows carry no gradient
    # no valid row at all: loss 0, zero gradient
    loss, dl = run_cross_entropy(Bd.mslt_op_cross_entropy, dtype, logits, np.full(R, -1), V, scratch=scratch)
    assert loss == 0.0 and not dl.any()
    # loss only
    loss, _ = run_cross_entropy(Bd.mslt_op_cross_entropy, dtype, logits, labels, V, want_grad=False,
                                scratch=scratch)
    assert abs(loss - want_loss) / want_loss < 1e-5


def _t(x, dtype):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda().to(
        torch.bfloat16 if dtype == 1 else torch.float32)


def _stream():
    import torch
    return torch.cuda.current_stream().cuda_stream


@pytest.mark.parametrize("dtype", [0, 1], ids=["fp32", "bf16"])
@pytest.mark.parametrize("rows,H", [(5, 128), (37, 192), (130, 768), (64, 1024), (9, 320)])
def test_layernorm_forward_and_backward_match_oracle(dtype, rows, H):
    import torch
    from paper_2011_13635_b200 import binding as Bd
    rng = np.random.default_rng(rows * H)
    z = _t(rng.standard_normal((rows, H)) * 2 + 0.5, dtype)
    gamma = (1 + 0.1 * rng.standard_normal(H)).astype(np.float32)
    beta = (0.1 * rng.standard_normal(H)).astype(np.float32)
    dy = _t(rng.standard_normal((rows, H)), dtype)
    d_g, d_b = torch.from_numpy(gamma).cuda(), torch.from_numpy(beta).cuda()
    y = torch.empty_like(z)
    stats = torch.empty((rows, 2), device="cuda")
    Bd.mslt_op_layernorm(z, d_g, d_b, y, stats, 1e-12, _stream())
    z64, dy64 = z.double().cpu().numpy(), dy.double().cpu().numpy()
    y_ref, xhat, rstd = O.layer_norm(z64, gamma.astype(np.float64), beta.astype(np.float64), 1e-12)
    tol = 2e-5 if dtype == 0 else 6e-3
    assert np.abs(y.double().cpu().numpy() - y_ref).max() / np.abs(y_ref).max() < tol
    st = stats.cpu().numpy()
    np.testing.assert_allclose(st[:, 0], z64.mean(-1), atol=1e-5)
    np.testing.assert_allclose(st[:, 1], rstd[:, 0], rtol=1e-5)
    # without statistics (frozen layers)
    y2 = torch.empty_like(z)
    Bd.mslt_op_layernorm(z, d_g, d_b, y2, None, 1e-12, _stream())
    assert torch.equal(y, y2)
    # backward
    dz = torch.empty_like(z)
    dgam = torch.zeros(H, device="cuda"); dbet = torch.zeros(H, device="cuda")
    dbias = torch.zeros(H, device="cuda")
    Bd.mslt_op_layernorm_bwd(dy, z, stats, d_g, dz, dgam, dbet, _stream(), dbias=dbias)
    dz_ref, dg_ref, db_ref = O.layer_norm_backward(dy64, xhat, rstd, gamma.astype(np.float64))
    assert np.abs(dz.double().cpu().numpy() - dz_ref).max() / np.abs(dz_ref).max() < tol
    # the fused bias gradient: column sums of dz (they nearly cancel within a row, so compare
    # against the size of dz rather than of the sums)
    assert np.abs(dbias.cpu().numpy() - dz_ref.sum(axis=0)).max() < (1e-4 if dtype == 0 else 2e-2) * np.abs(dz_ref).max() * np.sqrt(dz_ref.shape[0])
    assert np.abs(dgam.cpu().numpy() - dg_ref).max() / np.abs(dg_ref).max() < 1e-4
    assert np.abs(dbet.cpu().numpy() - db_ref).max() / np.abs(db_ref).max() < 1e-4
    # the column sums are accumulated: a second call doubles them
    Bd.mslt_op_layernorm_bwd(dy, z, stats, d_g, dz, dgam, dbet, _stream())
    assert np.abs(dbet.cpu().numpy() - 2 * db_ref).max() / np.abs(db_ref).max() < 2e-4


@pytest.mark.parametrize("dtype", [0, 1], ids=["fp32", "bf16"])
@pytest.mark.parametrize("S", [8, 64, 72, 128, 512])
def test_softmax_forward_and_backward_match_oracle(dtype, S):
    import torch
    from paper_2011_13635_b200 import binding as Bd
    B, A = 3, 2
    rng = np.random.default_rng(S)
    sc = _t(rng.standard_normal((B * A * S, S)) * 3, dtype)
    lens = np.array([S, max(1, S // 3), 1], dtype=np.int32)
    d_lens = torch.from_numpy(lens).cuda()
    p = torch.empty_like(sc)
    Bd.mslt_op_softmax(sc, p, d_lens, A * S, 0.125, _stream())
    sc64 = sc.double().cpu().numpy().reshape(B, A, S, S)
    p_ref = O.masked_softmax(sc64 * 0.125, lens).reshape(B * A * S, S)
    got = p.double().cpu().numpy()
    tol = 2e-6 if dtype == 0 else 4e-3
    assert np.abs(got - p_ref).max() < tol
    assert np.all(got[p_ref == 0] == 0)
    # in place
    sc2 = sc.clone()
    Bd.mslt_op_softmax(sc2, sc2, d_lens, A * S, 0.125, _stream())
    assert torch.equal(sc2, p)
    # backward
    dp = _t(rng.standard_normal((B * A * S, S)), dtype)
    dp64 = dp.double().cpu().numpy()
    ref = O.softmax_backward(dp64, got) * 0.125
    Bd.mslt_op_softmax_bwd(dp, p, 0.125, _stream())
    assert np.abs(dp.double().cpu().numpy() - ref).max() / np.abs(ref).max() < (2e-5 if dtype == 0 else 6e-3)


@pytest.mark.parametrize("dtype", [0, 1], ids=["fp32", "bf16"])
@pytest.mark.parametrize("rows,N,ld", [(7, 8, 8), (300, 768, 768), (1000, 1040, 1048), (64, 30528, 30528)])
def test_colsum_matches_numpy(dtype, rows, N, ld):
    import torch
    from paper_2011_13635_b200 import binding as Bd
    rng = np.random.default_rng(rows + N)
    x = _t(rng.standard_normal((rows, ld)), dtype)
    out = torch.full((ld,), 0.5, device="cuda")
    Bd.mslt_op_colsum(x, N, out, _stream())
    ref = 0.5 + x.double().cpu().numpy()[:, :N].sum(0)
    got = out.cpu().numpy()
    assert np.abs(got[:N] - ref).max() < 1e-4 * max(1.0, np.abs(ref).max())
    assert np.all(got[N:] == 0.5)                   # nothing past N is touched


def test_op_argument_checks():
    import torch
    from paper_2011_13635_b200 import binding as Bd
    z = torch.zeros((4, 100), device="cuda")        # row length not a multiple of 8
    g = torch.zeros(100, device="cuda")
    with pytest.raises(Bd.MsltError) as ei:
        Bd.mslt_op_layernorm(z, g, g, z, None, 1e-12, _stream())
    assert ei.value.code == -1
    s = torch.zeros((4, 1024), device="cuda")       # row longer than the softmax kernels hold
    with pytest.raises(Bd.MsltError) as ei:
        Bd.mslt_op_softmax(s, s, None, 4, 1.0, _stream())
    assert ei.value.code == -1


@pytest.mark.parametrize("B,S,A,masked", [(2, 128, 2, False), (3, 128, 12, True), (2, 100, 3, True),
                                          (5, 64, 2, True), (1, 24, 1, False), (37, 128, 12, True),
                                          (2, 256, 2, False), (3, 512, 4, True), (2, 384, 3, True),
                                          (3, 200, 2, True), (40, 512, 16, True), (1, 136, 1, False)])
@pytest.mark.parametrize("want_probs", [True, False], ids=["probs", "noprobs"])
def test_fused_attention_matches_oracle(B, S, A, masked, want_probs):
    """Scores, masked softmax and context in one kernel against the oracle's definition
    (einsum, masked_softmax, einsum) on the same bf16-rounded inputs."""
    import math
    import torch
    from paper_2011_13635_b200 import binding as Bd
    d, H = 64, A * 64
    rng = np.random.default_rng(B * 1000 + S + A)
    qkv = torch.from_numpy((rng.standard_normal((B * S, 3 * H)) * 1.5).astype(np.float32)).cuda().bfloat16()
    lens = rng.integers(1, S + 1, size=B).astype(np.int32) if masked else np.full(B, S, np.int32)
    if masked:
        lens[0] = S
        lens[-1] = 1 if B > 1 else S
    d_lens = torch.from_numpy(lens).cuda() if masked else None
    probs = torch.full((B, A, S, S), 7.0, device="cuda", dtype=torch.bfloat16) if want_probs else None
    ctx = torch.full((B * S, H), 7.0, device="cuda", dtype=torch.bfloat16)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    scale = 1.0 / math.sqrt(d)
    for _ in range(2):   # twice: the second call must not depend on what the first left behind
        Bd.mslt_op_attention(qkv, probs, ctx, d_lens, B, S, A, scale, status, _stream())
    assert int(status.item()) == 0
    x = qkv.float().cpu().numpy().astype(np.float64).reshape(B, S, 3, A, d)
    q, k, v = (x[:, :, i].transpose(0, 2, 1, 3) for i in range(3))          # [B, A, S, d]
    p_ref = O.masked_softmax(np.einsum("bhid,bhjd->bhij", q, k) * scale, lens)
    c_ref = np.einsum("bhij,bhjd->bhid", p_ref, v).transpose(0, 2, 1, 3).reshape(B * S, H)
    if want_probs:
        got = probs.float().cpu().numpy()
        for b in range(B):
            # rows at padded query positions are unspecified (a long-row kernel skips tiles of them)
            assert np.abs(got[b, :, :lens[b]] - p_ref[b, :, :lens[b]]).max() < 6e-3   # bf16 resolution at p <= 1
            assert not got[b, :, :, lens[b]:].any()                          # masked keys exactly 0
            assert np.isfinite(got[b]).all()
    # rows at padded query positions are unspecified: compare valid rows only
    got = ctx.float().cpu().numpy().reshape(B, S, H)
    assert np.isfinite(got).all()                                            # padded rows too: later layers read them
    ref = c_ref.reshape(B, S, H)
    for b in range(B):
        err = np.abs(got[b, :lens[b]] - ref[b, :lens[b]]).max()
        assert err / np.abs(ref[b, :lens[b]]).max() < 1.5e-2, (b, err)


def test_fused_attention_of_more_items_than_a_block_keeps_a_list_of():
    """Rows of more than 128 keys: a block describes its first 256 (sequence, head, query tile) items in shared
    memory and reads the words of any further ones from global memory; with one block per SM those are the second
    query tiles of the last sequences here."""
    import math
    import torch
    from paper_2011_13635_b200 import binding as Bd
    S, A, d = 136, 10, 64
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    B = (sms * 256 + 1500) // (2 * A)
    H = A * d
    gen = torch.Generator(device="cuda").manual_seed(3)
    qkv = torch.empty((B * S, 3 * H), device="cuda", dtype=torch.bfloat16).normal_(generator=gen)
    lens = torch.full((B,), S, device="cuda", dtype=torch.int32)
    lens[-3:] = torch.tensor([129, 90, 133], dtype=torch.int32)
    ctx = torch.full((B * S, H), 7.0, device="cuda", dtype=torch.bfloat16)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Bd.mslt_op_attention(qkv, None, ctx, lens, B, S, A, 1.0 / math.sqrt(d), status, _stream())
    assert int(status.item()) == 0
    for first in (0, B - 8):
        x = qkv.view(B, S, 3, A, d)[first:first + 8].double()
        q, k, v = (x[:, :, i].transpose(1, 2) for i in range(3))
        mask = torch.arange(S, device="cuda")[None] < lens[first:first + 8, None]
        p = torch.softmax((q @ k.transpose(-1, -2) / math.sqrt(d)).masked_fill(~mask[:, None, None], float("-inf")), -1)
        ref = (p @ v).transpose(1, 2).reshape(8, S, H)
        err = (ctx.view(B, S, H)[first:first + 8].double() - ref)[mask].abs().max() / ref.abs().max()
        assert err < 1.5e-2


def test_fused_attention_rejects_other_shapes():
    import torch
    from paper_2011_13635_b200 import binding as Bd
    qkv = torch.zeros((256, 192), device="cuda", dtype=torch.bfloat16)
    ctx = torch.zeros((256, 64), device="cuda", dtype=torch.bfloat16)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    with pytest.raises(Bd.MsltError):
        Bd.mslt_op_attention(qkv, None, ctx, None, 1, 1024, 1, 0.125, status, _stream())
    with pytest.raises(Bd.MsltError):
        Bd.mslt_op_attention(qkv, None, ctx, None, 0, 128, 1, 0.125, status, _stream())


@pytest.mark.parametrize("B,S,A,masked", [(2, 128, 2, False), (3, 128, 12, True), (2, 104, 3, True),
                                          (5, 64, 2, True), (1, 24, 1, False), (37, 128, 12, True)])
def test_fused_attention_backward_matches_oracle(B, S, A, masked):
    """dQ, dK, dV of one kernel against the reverse-mode formulas written with the oracle's
    softmax_backward, on the same bf16-rounded inputs (probabilities from the oracle's softmax)."""
    import math
    import torch
    from paper_2011_13635_b200 import binding as Bd
    d, H = 64, A * 64
    rng = np.random.default_rng(B * 977 + S + A)
    bf = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda().bfloat16()
    qkv = bf(rng.standard_normal((B * S, 3 * H)) * 1.5)
    dctx = bf(rng.standard_normal((B * S, H)))
    lens = rng.integers(1, S + 1, size=B).astype(np.int32) if masked else np.full(B, S, np.int32)
    scale = 1.0 / math.sqrt(d)
    x = qkv.float().cpu().numpy().astype(np.float64).reshape(B, S, 3, A, d)
    q, k, v = (x[:, :, i].transpose(0, 2, 1, 3) for i in range(3))            # [B, A, S, d]
    probs = bf(O.masked_softmax(np.einsum("bhid,bhjd->bhij", q, k) * scale, lens))
    p = probs.float().cpu().numpy().astype(np.float64)
    dc = dctx.float().cpu().numpy().astype(np.float64).reshape(B, S, A, d).transpose(0, 2, 1, 3)
    dv = np.einsum("bhij,bhid->bhjd", p, dc)
    ds = O.softmax_backward(np.einsum("bhid,bhjd->bhij", dc, v), p) * scale
    dq = np.einsum("bhij,bhjd->bhid", ds, k)
    dk = np.einsum("bhij,bhid->bhjd", ds, q)
    want = np.stack([dq, dk, dv], axis=0).transpose(1, 3, 0, 2, 4).reshape(B * S, 3 * H)   # [B,S,3,A,d]
    dqkv = torch.full((B * S, 3 * H), 7.0, device="cuda", dtype=torch.bfloat16)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for _ in range(2):
        Bd.mslt_op_attention_bwd(qkv, probs, dctx, dqkv, B, S, A, scale, status, _stream())
    assert int(status.item()) == 0
    got = dqkv.float().cpu().numpy().reshape(B, S, 3, H)
    want = want.reshape(B, S, 3, H)
    for which, name in enumerate(("dq", "dk", "dv")):
        err = np.abs(got[:, :, which] - want[:, :, which]).max() / np.abs(want[:, :, which]).max()
        assert err < 1.5e-2, (name, err)


@pytest.mark.parametrize("k_mean,v_mean", [(0.0, 0.0), (4.0, 16.0)])
@pytest.mark.parametrize("B,S,A", [(2, 136, 2), (1, 200, 3), (2, 256, 2), (3, 384, 1), (2, 512, 2), (13, 264, 12)])
def test_long_row_attention_backward_matches_oracle(B, S, A, k_mean, v_mean):
    """Rows of more than 128 keys, whose probabilities are formed again in the backward, at the tolerance of
    the shorter rows.  With a common part in the keys and values, whatever the rows of dS lack to a sum of
    zero shows in dQ (times the keys' part) and dK: with the row term from the bf16 context alone dQ is off by
    0.10 to 0.23 of its range here (formed in float64 with the same roundings), corrected by 0.004 to 0.006."""
    import math
    import torch
    from paper_2011_13635_b200 import binding as Bd
    d, H = 64, A * 64
    rng = np.random.default_rng(B * 977 + S + A)
    bf = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda().bfloat16()
    x = rng.standard_normal((B, S, 3, A, d)) * 1.5
    x[:, :, 1] += k_mean * rng.standard_normal((1, 1, A, d))
    x[:, :, 2] += v_mean * rng.standard_normal((1, 1, A, d))
    qkv = bf(x.reshape(B * S, 3 * H))
    dctx = bf(rng.standard_normal((B * S, H)))
    scale = 1.0 / math.sqrt(d)
    x = qkv.float().cpu().numpy().astype(np.float64).reshape(B, S, 3, A, d)
    q, k, v = (x[:, :, i].transpose(0, 2, 1, 3) for i in range(3))            # [B, A, S, d]
    s = np.einsum("bhid,bhjd->bhij", q, k) * scale
    p = O.masked_softmax(s, np.full(B, S))
    dc = dctx.float().cpu().numpy().astype(np.float64).reshape(B, S, A, d).transpose(0, 2, 1, 3)
    ds = O.softmax_backward(np.einsum("bhid,bhjd->bhij", dc, v), p) * scale
    want = [np.einsum("bhij,bhjd->bhid", ds, k), np.einsum("bhij,bhid->bhjd", ds, q), np.einsum("bhij,bhid->bhjd", p, dc)]
    ctx = torch.full((B * S, H), 7.0, device="cuda", dtype=torch.bfloat16)
    lse = torch.full((A, B * S), 7.0, device="cuda")
    scratch = torch.full((3, A, B * S), float("nan"), device="cuda")
    dqkv = torch.full((B * S, 3 * H), 7.0, device="cuda", dtype=torch.bfloat16)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for _ in range(2):
        Bd.mslt_op_attention_lse(qkv, ctx, lse, B, S, A, scale, status, _stream())
        Bd.mslt_op_attention_lse_bwd(qkv, ctx, lse, dctx, dqkv, scratch, B, S, A, scale, status, _stream())
    assert int(status.item()) == 0
    lse_ref = np.log2(np.exp(s - s.max(-1, keepdims=True)).sum(-1)) + s.max(-1) * math.log2(math.e)
    got = lse.cpu().numpy().reshape(A, B, S).transpose(1, 0, 2)
    # a score is four steps of 16 products, each truncated by less than 2^-22 of the sum of magnitudes; the
    # exponentials (2^-22 each) and the logarithm of their sum add less than 2^-19
    size = np.einsum("bhid,bhjd->bhij", np.abs(q), np.abs(k)).max() * scale * math.log2(math.e)
    assert np.abs(got - lse_ref).max() < 2.0 ** -20 * size + 2.0 ** -19
    got = dqkv.float().cpu().numpy().reshape(B, S, 3, A, d)
    for which, name in enumerate(("dq", "dk", "dv")):
        ref = want[which].transpose(0, 2, 1, 3)
        err = np.abs(got[:, :, which] - ref).max() / np.abs(ref).max()
        assert err < 1.5e-2, (name, err)


@pytest.mark.parametrize("which", ["forward", "backward"])
def test_long_row_attention_wait_that_runs_out_is_reported(which):
    """As for the other attention kernels below: an idle producer and a 20 ms limit leave the status bit set, and
    the next call works again."""
    import torch
    from paper_2011_13635_b200 import binding as Bd
    B, S, A = 2, 200, 2
    rng = np.random.default_rng(5)
    bf = lambda *s: torch.from_numpy(rng.standard_normal(s).astype(np.float32)).cuda().bfloat16()
    qkv, dctx = bf(B * S, 3 * 64 * A), bf(B * S, 64 * A)
    ctx, dqkv = torch.zeros_like(dctx), torch.zeros_like(qkv)
    lse, scratch = torch.zeros((A, B * S), device="cuda"), torch.zeros((3, A, B * S), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    calls = dict(forward=lambda: Bd.mslt_op_attention_lse(qkv, ctx, lse, B, S, A, 0.125, status, _stream()),
                 backward=lambda: Bd.mslt_op_attention_lse_bwd(qkv, ctx, lse, dctx, dqkv, scratch, B, S, A, 0.125, status,
                                                               _stream()))
    calls["forward"]()
    calls["backward"]()
    want = dqkv.clone()
    Bd.lib.mslt_debug_starve_next_attention(1)
    with pytest.raises(Bd.MsltError) as ei:
        calls[which]()
    assert ei.value.code == -5 and int(status.item()) & 1
    status.zero_()
    calls["forward"]()
    calls["backward"]()
    assert int(status.item()) == 0 and torch.equal(dqkv, want)


@pytest.mark.parametrize("S", [136, 200, 264, 512])
def test_long_row_attention_with_scores_far_above_the_first(S):
    """The exponentials are formed relative to the row's largest score, which the warps of a row's parts find together.
    Here it lies 2^64 and more above the first ones, in the first block or in a later one, in another place from row
    to row.  Probabilities are rounded to bf16 as in the other attention tests; the sums' logarithms reach a few
    thousand and are held to 2^-17 of that."""
    import torch
    from paper_2011_13635_b200 import binding as Bd
    B, A, d = 2, 2, 64
    rng = np.random.default_rng(S)
    x = rng.standard_normal((B, S, 3, A, d))
    for at, much in ((20, 3.0), (40, 40.0), (100, 100.0), (130, 300.0), (260, 600.0), (S - 1, 900.0)):
        if at < S:
            x[:, at, 1] *= much
    qkv = torch.from_numpy(x.reshape(B * S, 3 * A * d).astype(np.float32)).cuda().bfloat16()
    x = qkv.float().cpu().numpy().astype(np.float64).reshape(B, S, 3, A, d)
    q, k, v = (x[:, :, i].transpose(0, 2, 1, 3) for i in range(3))
    s = np.einsum("bhid,bhjd->bhij", q, k) * 0.125
    top = s.max(-1, keepdims=True)
    e = np.exp(s - top)
    want = np.einsum("bhij,bhjd->bhid", e / e.sum(-1, keepdims=True), v).transpose(0, 2, 1, 3).reshape(B * S, A * d)
    want_lse = ((top + np.log(e.sum(-1, keepdims=True)))[..., 0] / np.log(2)).transpose(1, 0, 2).reshape(A, B * S)
    ctx = torch.full((B * S, A * d), 7.0, device="cuda", dtype=torch.bfloat16)
    lse = torch.full((A, B * S), 7.0, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Bd.mslt_op_attention_lse(qkv, ctx, lse, B, S, A, 0.125, status, _stream())
    assert int(status.item()) == 0
    assert np.abs(ctx.double().cpu().numpy() - want).max() / np.abs(want).max() < 1.5e-2
    assert np.abs(lse.double().cpu().numpy() - want_lse).max() / np.abs(want_lse).max() < 2.0 ** -17


@pytest.mark.parametrize("S", [136, 200, 512])
@pytest.mark.parametrize("where", ["spread", "first", "middle", "last"])
def test_long_row_attention_loses_nothing_to_rounding_probabilities(S, where):
    """Probabilities are rounded to bf16 relative to the row's largest, which so is exactly 1: a key that takes 0.3 of
    a row's weight, wherever it lies, leaves no rounding of its own.  Held against the same definition in float64
    with these two roundings (probabilities, context); sums in fp32 change an error of 2^-9 by 2^-14 of it, and the
    roundings that they flip move its norm over 32768 values and more by less than 1 %.  With another reference the
    error was 1.19 to 1.27 times as large for a key in the middle or at the end, and 1.03 to 1.06 times for spread
    scores of rms 1 to 2."""
    import torch
    from paper_2011_13635_b200 import binding as Bd
    B, A, d = 2, 4, 64
    rng = np.random.default_rng(S)
    x = rng.standard_normal((B, S, 3, A, d))
    if where == "spread":
        x[:, :, :2] *= 1.4                                 # scores of rms 2
    else:
        x[:, :, :2] *= 0.3
        x[:, :, 0, :, 0], x[:, :, 1, :, 0] = 4.0, 0.0
        x[:, {"first": 5, "middle": 100, "last": S - 3}[where], 1, :, 0] = 2.0 * np.log(0.3 / 0.7 * S)
    qkv = torch.from_numpy(x.reshape(B * S, 3 * A * d).astype(np.float32)).cuda().bfloat16()
    y = qkv.double().view(B, S, 3, A, d)
    q, k, v = (y[:, :, i].transpose(1, 2) for i in range(3))
    s = q @ k.transpose(-1, -2) * 0.125
    e = torch.exp(s - s.amax(-1, keepdim=True))
    total = e.sum(-1, keepdim=True)
    rounded = lambda t: t.float().bfloat16().double()  # noqa: E731
    want, model = (e / total) @ v, rounded((rounded(e) @ v) / total)
    ctx = torch.full((B * S, A * d), 7.0, device="cuda", dtype=torch.bfloat16)
    lse = torch.empty((A, B * S), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Bd.mslt_op_attention_lse(qkv, ctx, lse, B, S, A, 0.125, status, _stream())
    got = ctx.double().view(B, S, A, d).transpose(1, 2)
    assert int(status.item()) == 0
    assert (got - want).norm().item() < 1.01 * (model - want).norm().item()


def test_long_row_attention_of_large_values_stays_finite():
    """No probability exceeds 1, so no context exceeds the largest value, also where a late key is far above the rest."""
    import torch
    from paper_2011_13635_b200 import binding as Bd
    B, S, A, d = 2, 256, 2, 64
    x = torch.randn((B, S, 3, A, d), generator=torch.Generator().manual_seed(1))
    x[:, 200, 1] *= 12.0
    x[:, :, 2] *= 1e30
    qkv = x.reshape(B * S, 3 * A * d).cuda().bfloat16()
    ctx = torch.full((B * S, A * d), 7.0, device="cuda", dtype=torch.bfloat16)
    lse = torch.empty((A, B * S), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Bd.mslt_op_attention_lse(qkv, ctx, lse, B, S, A, 0.125, status, _stream())
    y = qkv.double().view(B, S, 3, A, d)
    q, k, v = (y[:, :, i].transpose(1, 2) for i in range(3))
    want = (torch.softmax(q @ k.transpose(-1, -2) * 0.125, -1) @ v).transpose(1, 2).reshape(B * S, A * d)
    assert bool(torch.isfinite(ctx.float()).all()) and bool(torch.isfinite(lse).all())
    assert ((ctx.double() - want).abs().max() / want.abs().max()).item() < 1.5e-2


def test_long_row_attention_with_more_items_than_a_block_lists():
    """A block describes up to 256 of its items in shared memory and reads any beyond from memory.  An item's result
    does not depend on the others, so the last sequences of a batch of 257 items a block and more are those of a
    call on them alone."""
    import torch
    from paper_2011_13635_b200 import binding as Bd
    S, A, d = 136, 32, 64
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    B = sms * 256 // (2 * A) + 3                           # two query tiles a head and sequence
    gen = torch.Generator(device="cuda").manual_seed(1)
    qkv = torch.randn((B * S, 3 * A * d), device="cuda", dtype=torch.bfloat16, generator=gen)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")

    def run(x, n):
        ctx = torch.full((n * S, A * d), 7.0, device="cuda", dtype=torch.bfloat16)
        lse = torch.full((A, n * S), 7.0, device="cuda")
        Bd.mslt_op_attention_lse(x, ctx, lse, n, S, A, 0.125, status, _stream())
        return ctx, lse
    ctx, lse = run(qkv, B)
    for first in (0, B - 6):
        rows = slice(first * S, (first + 6) * S)
        c, l = run(qkv[rows], 6)
        assert torch.equal(ctx[rows], c) and torch.equal(lse[:, rows], l)
    assert int(status.item()) == 0


@pytest.mark.parametrize("B,S,A", [(1, 128, 2), (1, 520, 1), (0, 256, 1)])
def test_long_row_attention_backward_rejects_other_shapes(B, S, A):
    import torch
    from paper_2011_13635_b200 import binding as Bd
    x = torch.zeros((520, 3 * 128), device="cuda", dtype=torch.bfloat16)
    f = torch.zeros((3, 2, 520), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    with pytest.raises(Bd.MsltError):
        Bd.mslt_op_attention_lse(x, x, f, B, S, A, 0.125, status, _stream())
    with pytest.raises(Bd.MsltError):
        Bd.mslt_op_attention_lse_bwd(x, x, f, x, x, f, B, S, A, 0.125, status, _stream())


@pytest.mark.parametrize("which", ["forward", "forward_long_rows", "backward"])
def test_attention_wait_that_runs_out_is_reported_and_leaves_the_device_usable(which):
    """Every wait in the attention kernels is bounded.  With the test hook armed the next launch has
    an idle producer and a 20 ms limit: the kernel must come back with the status bit set (no
    fault, no hang), and the very next call must work and be correct again."""
    import math
    import torch
    from paper_2011_13635_b200 import binding as Bd
    B, A = 2, 2
    S = 256 if which == "forward_long_rows" else 128
    H = A * 64
    rng = np.random.default_rng(5)
    qkv = torch.from_numpy(rng.standard_normal((B * S, 3 * H)).astype(np.float32)).cuda().bfloat16()
    ctx = torch.zeros((B * S, H), device="cuda", dtype=torch.bfloat16)
    probs = torch.zeros((B, A, S, S), device="cuda", dtype=torch.bfloat16)
    dqkv = torch.zeros((B * S, 3 * H), device="cuda", dtype=torch.bfloat16)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    scale = 1.0 / math.sqrt(64)

    def call():
        if which == "backward":
            Bd.mslt_op_attention_bwd(qkv, probs, ctx, dqkv, B, S, A, scale, status, _stream())
        else:
            Bd.mslt_op_attention(qkv, probs, ctx, None, B, S, A, scale, status, _stream())

    Bd.lib.mslt_debug_starve_next_attention(1)
    with pytest.raises(Bd.MsltError) as ei:
        call()
    assert ei.value.code == -5
    assert int(status.item()) & 1
    status.zero_()
    Bd.mslt_op_attention(qkv, probs, ctx, None, B, S, A, scale, status, _stream())   # disarmed: works again
    assert int(status.item()) == 0
    x = qkv.float().cpu().numpy().astype(np.float64).reshape(B, S, 3, A, 64)
    q, k, v = (x[:, :, i].transpose(0, 2, 1, 3) for i in range(3))
    p_ref = O.masked_softmax(np.einsum("bhid,bhjd->bhij", q, k) * scale, np.full(B, S))
    c_ref = np.einsum("bhij,bhjd->bhid", p_ref, v).transpose(0, 2, 1, 3).reshape(B * S, H)
    assert np.abs(ctx.float().cpu().numpy() - c_ref).max() / np.abs(c_ref).max() < 1.5e-2
    if which == "backward":
        call()
        assert int(status.item()) == 0
