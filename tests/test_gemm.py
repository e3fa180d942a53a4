"""The dense contraction kernel alone (mslt_op_gemm) against numpy float64, for every operand
layout the step uses (forward: k contiguous; input gradient and weight gradient: row index
contiguous), batched attention addressing, ragged edges and each fused epilogue."""
import math

import numpy as np
import pytest
from scipy.special import erf

from tests import parity as PT

pytestmark = pytest.mark.gpu


def _gelu(u):
    return 0.5 * u * (1 + erf(u / math.sqrt(2)))


def _dgelu(u):
    return 0.5 * (1 + erf(u / math.sqrt(2))) + u * np.exp(-0.5 * u * u) / math.sqrt(2 * math.pi)


def _run(dtype, M, N, K, a_major, b_major, *, bias=False, act=0, residual=False, aux_out=False,
         d_fp32=False, accumulate=False, alpha=1.0, split_k=0, seed=0, planes=False, spoil=None, tol=None,
         form=None):
    """planes: the fp32 form on split operands; spoil(A, B) changes the operands before they are stored; form: what
    mslt_debug_last_gemm_form has to report."""
    import torch
    from paper_2011_13635_b200 import binding as Bd
    tdt = torch.float32 if dtype == 0 else torch.bfloat16
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((M, K)).astype(np.float32)
    B = rng.standard_normal((N, K)).astype(np.float32)
    if spoil:
        spoil(A, B)
    tA = torch.from_numpy(A).cuda().to(tdt)
    tB = torch.from_numpy(B).cuda().to(tdt)
    A64, B64 = tA.double().cpu().numpy(), tB.double().cpu().numpy()
    # K-major: stored [rows, K]; MN-major: stored [K, rows] (leading dimension padded to 8)
    def store(t, major):
        if major == "k":
            return t.contiguous(), t.shape[1], 1
        ld = (t.shape[0] + 7) // 8 * 8
        buf = torch.zeros((t.shape[1], ld), dtype=t.dtype, device="cuda")
        buf[:, : t.shape[0]] = t.t()
        return buf, 1, ld
    sA, a_rs, a_ks = store(tA, a_major)
    sB, b_rs, b_ks = store(tB, b_major)
    ldd = (N + 7) // 8 * 8
    D0 = rng.standard_normal((M, ldd)).astype(np.float32)
    tD = torch.from_numpy(D0).cuda().to(torch.float32 if d_fp32 else tdt)
    with np.errstate(invalid="ignore"):
        ref = alpha * (A64 @ B64.T)
    d = Bd.GemmDesc()
    d.dtype, d.M, d.N, d.K, d.batch, d.hdiv = dtype, M, N, K, 1, 1
    d.A, d.a_rs, d.a_ks = sA.data_ptr(), a_rs, a_ks
    d.B, d.b_rs, d.b_ks = sB.data_ptr(), b_rs, b_ks
    d.D, d.ldd = tD.data_ptr(), ldd
    d.d_fp32, d.accumulate, d.alpha, d.act, d.split_k = int(d_fp32), int(accumulate), alpha, act, split_k
    keep = [sA, sB, tD]
    if bias:
        bv = rng.standard_normal(N).astype(np.float32)
        tb = torch.from_numpy(bv).cuda()
        d.bias = tb.data_ptr()
        ref = ref + bv.astype(np.float64)
        keep.append(tb)
    taux = None
    if act == 1:
        if aux_out:
            taux = torch.zeros((M, ldd), dtype=tdt, device="cuda")
            d.aux = taux.data_ptr()
        pre = ref
        ref = _gelu(ref)
    elif act == 2:
        U = rng.standard_normal((M, ldd)).astype(np.float32)
        taux = torch.from_numpy(U).cuda().to(tdt)
        d.aux = taux.data_ptr()
        ref = ref * _dgelu(taux.double().cpu().numpy()[:, :N])
    if residual:
        Rm = rng.standard_normal((M, ldd)).astype(np.float32)
        tr = torch.from_numpy(Rm).cuda().to(tdt)
        d.residual = tr.data_ptr()
        ref = ref + tr.double().cpu().numpy()[:, :N]
        keep.append(tr)
    if accumulate:
        ref = ref + D0[:, :N].astype(np.float64)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    if planes:
        scratch = torch.full((Bd.mslt_op_gemm_f32_split_scratch_bytes(d),), 255, dtype=torch.uint8, device="cuda")
        Bd.mslt_op_gemm_f32_split(d, scratch, torch.cuda.current_stream().cuda_stream, status)
    else:
        Bd.mslt_op_gemm(d, torch.cuda.current_stream().cuda_stream, status)
    if form:
        assert Bd.mslt_debug_last_gemm_form() == form
    out = tD.double().cpu().numpy()
    if spoil:
        return out[:, :N], ref
    tol = tol or (2e-5 if dtype == 0 else (1e-5 if d_fp32 else 6e-3))
    scale = np.abs(ref).max()
    assert np.abs(out[:, :N] - ref).max() / scale < tol, (M, N, K, a_major, b_major)
    # columns past N (padding of the leading dimension) are never written
    if ldd > N:
        init = torch.from_numpy(D0).cuda().to(tD.dtype).double().cpu().numpy()
        assert np.array_equal(out[:, N:], init[:, N:])
    if act == 1 and aux_out:
        assert np.abs(taux.double().cpu().numpy()[:, :N] - pre).max() / np.abs(pre).max() < (2e-5 if dtype == 0 else 6e-3)


SHAPES = [(128, 128, 64), (256, 256, 128), (200, 136, 72), (130, 1037, 192), (517, 64, 520),
          (64, 72, 8), (1, 8, 16)]


@pytest.mark.parametrize("dtype", [0, 1], ids=["fp32", "bf16"])
@pytest.mark.parametrize("majors", [("k", "k"), ("k", "mn"), ("mn", "mn"), ("mn", "k")])
@pytest.mark.parametrize("shape", SHAPES)
def test_layouts_and_ragged_edges(dtype, majors, shape):
    _run(dtype, *shape, majors[0], majors[1], seed=hash(shape) % 1000)


@pytest.mark.parametrize("dtype", [0, 1], ids=["fp32", "bf16"])
def test_epilogues(dtype):
    _run(dtype, 200, 136, 72, "k", "k", bias=True)
    _run(dtype, 200, 136, 72, "k", "k", bias=True, act=1, aux_out=True)
    _run(dtype, 200, 136, 72, "k", "k", bias=True, act=1)
    _run(dtype, 200, 136, 72, "k", "mn", act=2)
    _run(dtype, 200, 136, 72, "k", "mn", residual=True, alpha=0.125)
    _run(dtype, 200, 136, 72, "k", "k", bias=True, residual=True)
    _run(dtype, 200, 136, 72, "k", "k", bias=True, d_fp32=True)
    _run(dtype, 136, 200, 1000, "mn", "mn", d_fp32=True, accumulate=True)


@pytest.mark.parametrize("variant", [0, 1, 2, 4, 6], ids=["auto", "single", "pair", "auto-rowstores", "pair-rowstores"])
def test_bf16_epilogues_over_several_wide_tiles(variant):
    """Every bf16 epilogue flavour on outputs of several 256-wide tiles with ragged last tiles, in
    each tiling form and with both ways of storing the output (through shared memory and the copy
    engine, or row segments from registers)."""
    from paper_2011_13635_b200 import binding as Bd
    assert Bd.lib.mslt_debug_set_gemm_variant(variant) == 0
    try:
        _run(1, 700, 840, 200, "k", "k", bias=True)
        _run(1, 700, 840, 200, "k", "k", bias=True, act=1, aux_out=True)
        _run(1, 700, 832, 136, "k", "k", bias=True, act=1)
        _run(1, 520, 800, 72, "k", "mn", act=2)
        _run(1, 520, 800, 72, "k", "mn", bias=True, residual=True, alpha=0.125)
        _run(1, 300, 1037, 192, "k", "k", bias=True)           # row pitch 1040: columns end inside a chunk
        _run(1, 33, 168, 64, "mn", "k", bias=True, act=1)      # one 128-wide tile and a ragged second one
    finally:
        Bd.lib.mslt_debug_set_gemm_variant(0)


@pytest.mark.parametrize("variant", [0, 1, 2, 4], ids=["auto", "single", "pair", "auto-rowstores"])
@pytest.mark.parametrize("shape", [(33, 36, 64), (1, 32, 72), (257, 60, 136), (300, 1037, 192), (130, 1022, 200), (520, 768, 392)])
def test_bf16_operands_with_fp32_output(shape, variant):
    """fp32 outputs, stored and added to what is there, at row and column counts where the 32 x 32 tiles that leave
    through the copy engine end inside the output, or inside a 16-byte piece of it."""
    from paper_2011_13635_b200 import binding as Bd
    assert Bd.lib.mslt_debug_set_gemm_variant(variant) == 0
    try:
        _run(1, *shape, "k", "k", bias=True, d_fp32=True)
        _run(1, *shape, "mn", "mn", d_fp32=True, accumulate=True)
        _run(1, *shape, "k", "mn", d_fp32=True, accumulate=True, split_k=2, alpha=0.5)
    finally:
        Bd.lib.mslt_debug_set_gemm_variant(0)


def test_bf16_long_contraction_split_k():
    """Weight-gradient shape: small output, long contraction, partial sums added in fp32."""
    _run(1, 768, 256, 4096, "mn", "mn", d_fp32=True, accumulate=True)
    _run(1, 768, 256, 4096, "mn", "mn", d_fp32=True, accumulate=True, split_k=7)
    _run(1, 300, 264, 2500, "mn", "mn", d_fp32=True, accumulate=True, split_k=3)


@pytest.mark.parametrize("dtype", [0, 1], ids=["fp32", "bf16"])
def test_batched_attention_addressing(dtype):
    """Scores and context of multi-head attention read straight from the fused [T, 3H] buffer."""
    import torch
    from paper_2011_13635_b200 import binding as Bd
    Bn, A, S, dh = 3, 2, 72, 64
    H = A * dh
    tdt = torch.float32 if dtype == 0 else torch.bfloat16
    rng = np.random.default_rng(3)
    qkv = torch.from_numpy(rng.standard_normal((Bn * S, 3 * H)).astype(np.float32)).cuda().to(tdt)
    q64 = qkv.double().cpu().numpy().reshape(Bn, S, 3, A, dh)
    sc = torch.zeros((Bn * A, S, S), dtype=tdt, device="cuda")
    d = Bd.GemmDesc()
    d.dtype, d.M, d.N, d.K, d.batch, d.hdiv, d.alpha = dtype, S, S, dh, Bn * A, A, 0.125
    d.A, d.a_rs, d.a_ks, d.a_bo, d.a_bi = qkv.data_ptr(), 3 * H, 1, S * 3 * H, dh
    d.B, d.b_rs, d.b_ks, d.b_bo, d.b_bi = qkv.data_ptr() + H * qkv.element_size(), 3 * H, 1, S * 3 * H, dh
    d.D, d.ldd, d.d_bo, d.d_bi = sc.data_ptr(), S, A * S * S, S * S
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Bd.mslt_op_gemm(d, torch.cuda.current_stream().cuda_stream, status)
    ref = 0.125 * np.einsum("bihd,bjhd->bhij", q64[:, :, 0], q64[:, :, 1]).reshape(Bn * A, S, S)
    tol = 2e-5 if dtype == 0 else 6e-3
    assert np.abs(sc.double().cpu().numpy() - ref).max() / np.abs(ref).max() < tol
    # context = P V with V read row-contiguous (its k index strided)
    p = torch.from_numpy(rng.random((Bn * A, S, S)).astype(np.float32)).cuda().to(tdt)
    ctx = torch.zeros((Bn * S, H), dtype=tdt, device="cuda")
    d = Bd.GemmDesc()
    d.dtype, d.M, d.N, d.K, d.batch, d.hdiv, d.alpha = dtype, S, dh, S, Bn * A, A, 1.0
    d.A, d.a_rs, d.a_ks, d.a_bo, d.a_bi = p.data_ptr(), S, 1, A * S * S, S * S
    d.B, d.b_rs, d.b_ks, d.b_bo, d.b_bi = qkv.data_ptr() + 2 * H * qkv.element_size(), 1, 3 * H, S * 3 * H, dh
    d.D, d.ldd, d.d_bo, d.d_bi = ctx.data_ptr(), H, S * H, dh
    Bd.mslt_op_gemm(d, torch.cuda.current_stream().cuda_stream, status)
    p64 = p.double().cpu().numpy().reshape(Bn, A, S, S)
    ref = np.einsum("bhij,bjhd->bihd", p64, q64[:, :, 2]).reshape(Bn * S, H)
    assert np.abs(ctx.double().cpu().numpy() - ref).max() / np.abs(ref).max() < tol


@pytest.mark.parametrize("S", [128, 72, 64, 8])
def test_bf16_softmax_epilogue(S):
    """Attention scores with the scaled masked softmax applied in the kernel's epilogue."""
    import torch
    from paper_2011_13635_b200 import binding as Bd
    Bn, A, dh = 3, 2, 64
    H = A * dh
    rng = np.random.default_rng(S)
    qkv = torch.from_numpy(rng.standard_normal((Bn * S, 3 * H)).astype(np.float32) * 2).cuda().to(torch.bfloat16)
    lens = np.array([S, max(1, S // 3), 1], dtype=np.int32)
    d_lens = torch.from_numpy(lens).cuda()
    prob = torch.full((Bn * A, S, S), 7.0, dtype=torch.bfloat16, device="cuda")
    d = Bd.GemmDesc()
    d.dtype, d.M, d.N, d.K, d.batch, d.hdiv, d.alpha = 1, S, S, dh, Bn * A, A, 0.125
    d.A, d.a_rs, d.a_ks, d.a_bo, d.a_bi = qkv.data_ptr(), 3 * H, 1, S * 3 * H, dh
    d.B, d.b_rs, d.b_ks, d.b_bo, d.b_bi = qkv.data_ptr() + H * 2, 3 * H, 1, S * 3 * H, dh
    d.D, d.ldd, d.d_bo, d.d_bi = prob.data_ptr(), S, A * S * S, S * S
    d.act, d.seq_lens = 3, d_lens.data_ptr()
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Bd.mslt_op_gemm(d, torch.cuda.current_stream().cuda_stream, status)
    q64 = qkv.double().cpu().numpy().reshape(Bn, S, 3, A, dh)
    sc = 0.125 * np.einsum("bihd,bjhd->bhij", q64[:, :, 0], q64[:, :, 1])
    valid = (np.arange(S)[None, :] < lens[:, None])[:, None, None, :]
    sc = np.where(valid, sc, -np.inf)
    e = np.exp(sc - sc.max(-1, keepdims=True))
    ref = (e / e.sum(-1, keepdims=True)).reshape(Bn * A, S, S)
    got = prob.double().cpu().numpy()
    assert np.abs(got - ref).max() < 6e-3
    assert np.all(got[ref == 0] == 0)                  # masked keys are exactly zero
    np.testing.assert_allclose(got.sum(-1), 1.0, atol=2e-2)


def test_wait_that_runs_out_is_reported_and_leaves_the_device_usable():
    """Failure path without a fault: the producer of one launch issues no copies, the first wait
    runs out after ~20 ms, the kernel drains and returns, and the call reports MSLT_ERR_DEVICE."""
    import torch
    from paper_2011_13635_b200 import binding as Bd
    M = N = 128
    K = 64
    a = torch.randn((M, K), device="cuda").to(torch.bfloat16)
    b = torch.randn((N, K), device="cuda").to(torch.bfloat16)
    out = torch.zeros((M, N), device="cuda", dtype=torch.bfloat16)
    d = Bd.GemmDesc()
    d.dtype, d.M, d.N, d.K, d.batch, d.hdiv, d.alpha = 1, M, N, K, 1, 1, 1.0
    d.A, d.a_rs, d.a_ks = a.data_ptr(), K, 1
    d.B, d.b_rs, d.b_ks = b.data_ptr(), K, 1
    d.D, d.ldd = out.data_ptr(), N
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    Bd.lib.mslt_debug_starve_next_gemm(1)
    with pytest.raises(Bd.MsltError) as ei:
        Bd.mslt_op_gemm(d, stream, status)
    assert ei.value.code == -5
    assert int(status.item()) & 1
    # the hook disarms itself: the same call now succeeds and is correct
    status.zero_()
    Bd.mslt_op_gemm(d, stream, status)
    ref = a.double() @ b.double().t()
    assert (out.double() - ref).abs().max() / ref.abs().max() < 6e-3
    assert int(status.item()) == 0


@pytest.mark.parametrize("shape,majors,form", [
    ((1024, 768, 768), ("k", "k"), (32, 1, 1)),
    ((1024, 2304, 96), ("k", "k"), (128, 1, 1)),
    ((160, 768, 2500), ("k", "mn"), (64, 1, 8)),         # last slice ragged
    ((2304, 760, 1000), ("mn", "mn"), (64, 1, 1)),       # ragged columns
    ((1024, 760, 1000), ("mn", "mn"), (64, 1, 2)),
    ((600, 600, 2000), ("k", "mn"), (64, 1, 4)),
    ((3000, 760, 200), ("mn", "mn"), (128, 1, 1)),       # ragged both ways
    ((1000, 1000, 500), ("k", "mn"), (128, 1, 2)),
    ((512, 128, 512), ("k", "k"), (32, 4, 2)),           # warps of a block share k, and a cluster does
    ((33, 31, 260), ("mn", "k"), (32, 4, 4)), ((1, 1, 1), ("k", "k"), (32, 4, 1))])
def test_fp32_tiles_and_cluster_splits(shape, majors, form):
    """Every tile size and k split that the fp32 kernel's rule chooses, with remainders.  Sums of K
    products of unit normals: the error of a running fp32 sum grows as sqrt(K) * 2^-24 of its range."""
    wgrad = majors == ("mn", "mn")
    tile, groups, splits = form
    _run(0, *shape, *majors, bias=not wgrad, d_fp32=True, accumulate=wgrad, form=(3, tile, tile, groups, splits))


@pytest.mark.parametrize("shape,planes", [
    ((1, 1, 2100), False), ((3, 41, 4000), False), ((33, 2, 1500), False), ((65, 66, 3000), False), ((130, 250, 2500), False),
    ((129, 136, 4104), True), ((2, 304, 2064), True)])
def test_fp32_clusters_with_little_output(shape, planes):
    """Blocks of a cluster each finish a share of the tile's rows.  Here most shares, or their last columns, lie beyond
    the output: such blocks read nothing from the others and leave at once, while theirs is still read."""
    from paper_2011_13635_b200 import binding as Bd
    for majors, kw in ((("k", "k"), dict(bias=True)), (("mn", "mn"), dict(accumulate=True)), (("k", "mn"), dict(residual=True))):
        _run(0, *shape, *majors, d_fp32=True, planes=planes, **kw)
        assert Bd.mslt_debug_last_gemm_form()[4] > 1


@pytest.mark.parametrize("shape,majors,kw,form", [
    ((664, 1040, 16), ("k", "k"), dict(bias=True, act=1, aux_out=True), (32, 4, 1)),
    ((976, 744, 24), ("k", "k"), dict(residual=True), (32, 1, 1)),
    ((440, 3000, 48), ("k", "mn"), dict(act=2), (32, 1, 1)),
    ((592, 1385, 25), ("mn", "mn"), dict(accumulate=True), (32, 4, 1)),
    ((538, 1422, 17), ("k", "mn"), dict(bias=True, act=1), (32, 4, 1))])
def test_fp32_short_k_takes_tiles_of_few_outputs_per_thread(shape, majors, kw, form):
    """Where k is short the epilogue is the time, and a thread of a 64 x 64 tile has 64 outputs of it: two to
    three times slower than these."""
    tile, groups, splits = form
    _run(0, *shape, *majors, d_fp32=True, form=(3, tile, tile, groups, splits), **kw)


def test_fp32_unaligned_operands_take_the_element_wise_copies():
    import torch
    from paper_2011_13635_b200 import binding as Bd
    M, N, K, ld = 70, 41, 67, 71                    # odd pitch and odd base: no 16-byte access anywhere
    g = torch.Generator(device="cuda").manual_seed(3)
    A, B = torch.randn(M * ld + 1, generator=g, device="cuda"), torch.randn(N * ld + 1, generator=g, device="cuda")
    D = torch.zeros(M, N, device="cuda")
    d = Bd.GemmDesc()
    d.dtype, d.M, d.N, d.K, d.batch, d.hdiv, d.alpha = 0, M, N, K, 1, 1, 1.0
    d.A, d.a_rs, d.a_ks = A.data_ptr() + 4, ld, 1
    d.B, d.b_rs, d.b_ks = B.data_ptr() + 4, ld, 1
    d.D, d.ldd, d.d_fp32 = D.data_ptr(), N, 1
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Bd.mslt_op_gemm(d, torch.cuda.current_stream().cuda_stream, status)
    a, b = A[1:].view(M, ld)[:, :K].double(), B[1:].view(N, ld)[:, :K].double()
    ref = a @ b.t()
    assert ((D.double() - ref).abs().max() / ref.abs().max()).item() < 2e-5


@pytest.mark.parametrize("shape,majors,kw,form", [
    # one CTA: rows, columns, k blocks per round, k splits
    ((33, 72, 64), ("k", "k"), dict(bias=True), (128, 64, 1, 1)),
    ((64, 768, 200), ("k", "k"), dict(bias=True, residual=True), (128, 64, 2, 1)),
    ((130, 72, 136), ("k", "mn"), dict(act=2), (128, 64, 2, 1)),
    ((160, 96, 136), ("k", "mn"), dict(act=2), (128, 64, 2, 1)),
    ((24, 768, 4000), ("k", "mn"), dict(d_fp32=True, accumulate=True), (128, 64, 2, 11)),
    ((2056, 544, 136), ("k", "k"), dict(bias=True, residual=True), (128, 128, 2, 1)),
    ((2056, 544, 136), ("k", "mn"), dict(act=2), (128, 128, 2, 1)),
    ((2100, 520, 136), ("k", "k"), dict(bias=True, act=1, aux_out=True), (128, 128, 2, 1)),
    ((130, 3072, 1160), ("mn", "mn"), dict(d_fp32=True, accumulate=True), (128, 128, 2, 3)),
    ((1100, 2304, 136), ("k", "k"), dict(bias=True), (128, 192, 1, 1)),
    ((4096, 760, 264), ("k", "k"), dict(bias=True, residual=True), (128, 192, 1, 1)),     # general epilogue
    ((4096, 768, 320), ("k", "mn"), dict(residual=True), (128, 192, 1, 1)),
    ((4096, 736, 264), ("k", "k"), dict(residual=True), (128, 192, 1, 1)),                # ragged last tile
    ((520, 4104, 136), ("k", "k"), dict(bias=True, act=1, aux_out=True), (128, 192, 1, 1)),
    ((4000, 520, 136), ("k", "k"), dict(bias=True, act=1), (128, 192, 1, 1)),
    ((4000, 768, 1160), ("k", "k"), dict(bias=True, act=1, aux_out=True), (128, 192, 1, 1)),
    ((2304, 768, 2408), ("mn", "mn"), dict(d_fp32=True, accumulate=True), (128, 192, 1, 2)),
    ((3000, 1160, 136), ("k", "k"), dict(bias=True, act=1), (128, 256, 1, 1)),
    ((3000, 1184, 136), ("k", "k"), dict(residual=True), (128, 256, 1, 1)),
    ((3000, 1184, 136), ("k", "k"), dict(act=2), (128, 256, 1, 1)),
    ((3000, 1160, 136), ("k", "k"), dict(d_fp32=True, bias=True), (128, 256, 1, 1)),
    ((1100, 1040, 2408), ("mn", "mn"), dict(d_fp32=True, accumulate=True), (128, 256, 1, 3)),
    # a pair of CTAs
    ((2056, 520, 2408), ("k", "k"), dict(bias=True, act=1, aux_out=True), (256, 128, 2, 1)),
    ((2056, 544, 2408), ("k", "mn"), dict(residual=True), (256, 128, 2, 1)),
    ((2056, 544, 2408), ("k", "k"), dict(act=2), (256, 128, 2, 1)),
    ((4000, 520, 2408), ("k", "k"), dict(bias=True, act=1), (256, 192, 2, 1)),
    ((520, 4104, 2408), ("k", "k"), dict(bias=True, act=1, aux_out=True), (256, 192, 2, 1)),
    ((520, 4128, 2408), ("k", "k"), dict(bias=True, residual=True), (256, 192, 2, 1)),
    ((520, 4128, 2408), ("k", "k"), dict(act=2), (256, 192, 2, 1)),
    ((8200, 520, 2408), ("k", "k"), dict(d_fp32=True, accumulate=True), (256, 192, 2, 2)),
    ((6000, 1160, 2408), ("k", "k"), dict(bias=True, act=1), (256, 256, 2, 1)),
    ((6000, 1184, 2408), ("k", "mn"), dict(act=2), (256, 256, 2, 1)),
    ((8200, 1160, 2408), ("mn", "mn"), dict(d_fp32=True, accumulate=True), (256, 256, 2, 2))])
def test_bf16_tile_forms_the_estimate_picks(shape, majors, kw, form):
    """Every form of the persistent kernel and epilogues on each; small shapes with the few-tile kernel off."""
    from paper_2011_13635_b200 import binding as Bd
    few = form[1] == 64 and not kw.get("d_fp32")
    if few:
        Bd._check(Bd.lib.mslt_debug_set_gemm_variant(1))
    try:
        _run(1, *shape, *majors, form=(1,) + form, **kw)
    finally:
        if few:
            Bd._check(Bd.lib.mslt_debug_set_gemm_variant(0))


@pytest.mark.parametrize("shape,majors,kw,splits", [
    ((1, 8, 64), ("k", "k"), dict(bias=True), 1),                              # one row, one round
    ((64, 768, 3072), ("k", "k"), dict(bias=True, residual=True), 8),          # k over a cluster of eight
    ((130, 776, 3080), ("k", "mn"), dict(residual=True, alpha=0.5), 4),        # second row tile of two rows, ragged k and columns
    ((200, 768, 1160), ("mn", "k"), dict(bias=True, act=1, aux_out=True), 4),  # ring reused inside a block
    ((300, 776, 776), ("k", "k"), dict(bias=True, act=1), 2),
    ((33, 136, 72), ("mn", "mn"), dict(act=2), 1), ((129, 64, 640), ("k", "k"), dict(bias=True, act=1), 4)])
def test_bf16_few_tile_kernel(shape, majors, kw, splits):
    """Outputs of few tiles: partial sums added inside a cluster, every epilogue."""
    _run(1, *shape, *majors, form=(2, 128, 64, 1, splits), **kw)


@pytest.mark.parametrize("N,kw", [(129, dict(act=3)), (200, dict(act=3)), (64, dict(act=3, d_fp32=1)), (64, dict(split_k=2)),
                                  (64, dict(split_k=2, d_fp32=1)), (64, dict(hdiv=2))])
def test_bf16_descriptors_without_a_kernel_are_refused(N, kw):
    """A softmax over rows that no tile holds, a k split without an output to add into, a batch that its inner
    index does not divide: refused before a tile form is looked for."""
    import torch
    from paper_2011_13635_b200 import binding as Bd
    A = torch.zeros((64, 256), device="cuda", dtype=torch.bfloat16)
    B = torch.zeros((N, 256), device="cuda", dtype=torch.bfloat16)
    D = torch.zeros((64, 256), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    d = Bd.GemmDesc()
    d.dtype, d.M, d.N, d.K, d.batch, d.hdiv, d.alpha = 1, 64, N, 256, 1, 1, 1.0
    d.A, d.a_rs, d.a_ks = A.data_ptr(), 256, 1
    d.B, d.b_rs, d.b_ks = B.data_ptr(), 256, 1
    d.D, d.ldd = D.data_ptr(), 256
    for k, v in kw.items():
        setattr(d, k, v)
    for call in (Bd.mslt_op_gemm, Bd.mslt_op_gemm_enqueue):
        with pytest.raises(Bd.MsltError) as ei:
            call(d, torch.cuda.current_stream().cuda_stream, status)
        assert ei.value.code == -1


def _in_step_operands(M, N, K, batch=1, majors="kk", d_fp32=True):
    import torch
    from paper_2011_13635_b200 import binding as Bd
    gen = torch.Generator(device="cuda").manual_seed(M + N + K)
    make = lambda rows, major: torch.randn((batch, rows, K) if major == "k" else (batch, K, rows), device="cuda",  # noqa: E731
                                           generator=gen).bfloat16()
    A, B = make(M, majors[0]), make(N, majors[1])
    d = Bd.GemmDesc()
    d.dtype, d.M, d.N, d.K, d.batch, d.hdiv, d.alpha = 1, M, N, K, batch, 1, 1.0
    d.A, d.a_bo = A.data_ptr(), M * K
    d.a_rs, d.a_ks = (K, 1) if majors[0] == "k" else (1, M)
    d.B, d.b_bo = B.data_ptr(), N * K
    d.b_rs, d.b_ks = (K, 1) if majors[1] == "k" else (1, N)
    d.d_fp32, d.ldd = int(d_fp32), (N + 7) // 8 * 8
    d.d_bo = M * d.ldd
    return d, A, B


@pytest.mark.parametrize("M,N,K,split_k,room", [
    (2560, 768, 30520, 7, 8), (300, 1032, 4104, 8, 39), (33, 192, 1040, 0, 5), (33, 192, 1040, 0, 2), (33, 192, 4104, 0, 1),
    (520, 100, 2048, 3, 3), (40, 64, 64, 0, 8)])
def test_bf16_results_by_split(M, N, K, split_k, room):
    """Each split's sum over its own k, in its own result: added in their order they give the product, and nothing
    beyond the number that is reported is written.  k is cut at multiples of 128, the last split takes the rest."""
    import torch
    from paper_2011_13635_b200 import binding as Bd
    d, A, B = _in_step_operands(M, N, K)
    D = torch.full((9, M, d.ldd), 7.0, device="cuda")
    d.D, d.split_k = D.data_ptr(), split_k
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    parts = Bd.mslt_debug_gemm_in_step(d, torch.cuda.current_stream().cuda_stream, status, parts=room)
    assert parts == Bd.mslt_debug_last_gemm_form()[4] and parts <= min(room, 8) and parts <= max(split_k, 1 if K < 512 else 8)
    per = (-(-K // 128) + parts - 1) // parts * 128 if split_k else None
    a, b = A[0].double(), B[0].double()
    top = (a @ b.t()).abs().max().item()
    if per:
        for i in range(parts):
            want = a[:, i * per:(i + 1) * per] @ b[:, i * per:(i + 1) * per].t()
            assert (D[i, :, :N].double() - want).abs().max().item() < 2e-5 * top
    assert (D[:parts, :, :N].double().sum(0) - a @ b.t()).abs().max().item() < 2e-5 * top
    assert bool((D[parts:] == 7.0).all()) and bool((D[:, :, N:] == 7.0).all())


@pytest.mark.parametrize("kw", [dict(bias=True), dict(act=1), dict(act=2), dict(residual=True), dict(accumulate=1), dict(d_fp32=0),
                                dict(split_k=9), dict(split_k=4, room=3), dict(room=-1), dict(rows=True), dict(batch=2)], ids=str)
def test_bf16_results_by_split_without_a_kernel_are_refused(kw):
    import torch
    from paper_2011_13635_b200 import binding as Bd
    kw = dict(kw)
    room = kw.pop("room", 8)
    rows = torch.full((1,), 64, dtype=torch.int32, device="cuda") if kw.pop("rows", False) else None
    d, A, B = _in_step_operands(64, 64, 1024, batch=kw.pop("batch", 1))
    D = torch.zeros((9, 2, 64, 64), device="cuda")
    extra = torch.zeros((2, 64, 64), device="cuda")
    d.D = D.data_ptr()
    if kw.pop("bias", False):
        d.bias = extra.data_ptr()
    if kw.pop("residual", False):
        d.residual = extra.data_ptr()
    d.aux = extra.data_ptr()
    for k, v in kw.items():
        setattr(d, k, v)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    with pytest.raises(Bd.MsltError) as ei:
        Bd.mslt_debug_gemm_in_step(d, torch.cuda.current_stream().cuda_stream, status, rows=rows, parts=room)
    assert ei.value.code == -1


@pytest.mark.parametrize("M,N,K,batch,count,rows_are_k,d_fp32", [
    (520, 768, 768, 1, 300, False, False), (520, 768, 768, 1, 1, False, False), (4096, 768, 200, 1, 130, False, False),
    (520, 136, 192, 3, 130, False, False), (1040, 264, 72, 2, 1040, False, True),
    (768, 264, 4096, 1, 1000, True, True), (3072, 768, 8192, 1, 128, True, True), (136, 72, 2048, 1, 2048, True, True)])
def test_bf16_weights_read_early_beside_a_device_row_count(M, N, K, batch, count, rows_are_k, d_fp32):
    """b_static with a row count that only the device knows: the tiles of B that are asked for early are the ones that
    are multiplied, whatever the count does to the split of k and to the place of a batch in the list of tiles."""
    import torch
    from paper_2011_13635_b200 import binding as Bd
    d, A, B = _in_step_operands(M, N, K, batch, ("mn", "mn") if rows_are_k else ("k", "k"), d_fp32)
    if rows_are_k:
        A[:, count:] = 0
        B[:, count:] = 0
        d.accumulate = 1
        want = (A[0].double().t() @ B[0].double())[None]
    else:
        want = A.double() @ B.double().transpose(1, 2)
    D = torch.full((batch, M, d.ldd), 0.0 if rows_are_k else 7.0, device="cuda", dtype=torch.float32 if d_fp32 else torch.bfloat16)
    d.D = D.data_ptr()
    rows = torch.full((1,), count, dtype=torch.int32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Bd.mslt_debug_gemm_in_step(d, torch.cuda.current_stream().cuda_stream, status, rows=rows, rows_are_k=rows_are_k, b_static=True)
    have = M if rows_are_k else count
    err = (D[:, :have, :N].double() - want[:, :have]).abs().max().item() / want.abs().max().item()
    assert err < (2e-5 if d_fp32 else 6e-3)
    assert rows_are_k or bool((D[:, -(-count // 256) * 256:] == 7.0).all())


@pytest.mark.parametrize("M,form", [(256, (2, 128, 64, 1, 4)), (768, (2, 128, 64, 1, 2)), (1024, (1, 128, 64, 2, 1)), (2048, (1, 128, 64, 2, 1))])
def test_bf16_form_of_a_product_whose_rows_only_the_device_knows(M, form):
    """The few-tile kernel is made for one wave of blocks.  1024 rows in clusters of two are 192 of them: fewer than the SMs
    at a fill of 0.7, but an evaluation of 8 full sequences took 687 us with it and 555 without."""
    import torch
    from paper_2011_13635_b200 import binding as Bd
    d, A, B = _in_step_operands(M, 768, 3072, d_fp32=False)
    D = torch.full((M, d.ldd), 7.0, device="cuda", dtype=torch.bfloat16)
    d.D = D.data_ptr()
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for count in (M, M // 3):
        rows = torch.full((1,), count, dtype=torch.int32, device="cuda")
        Bd.mslt_debug_gemm_in_step(d, torch.cuda.current_stream().cuda_stream, status, rows=rows, b_static=True)
        assert Bd.mslt_debug_last_gemm_form() == form
        want = A[0, :count].double() @ B[0].double().t()
        assert (D[:count].double() - want).abs().max().item() < 6e-3 * want.abs().max().item()


def test_fp32_more_rows_than_narrow_tiles_can_index():
    """Over 65535 x 32 rows only the tiles of more rows fit the launch grid."""
    _run(0, 65535 * 32 + 70, 8, 8, "k", "k", bias=True, d_fp32=True, form=(3, 64, 64, 1, 1))


# with the tile width and the k split
PLANE_SHAPES = [((64, 72, 200), ("k", "k"), (64, 1)), ((130, 328, 136), ("mn", "k"), (64, 1)),
                ((704, 760, 520), ("k", "mn"), (64, 2)), ((256, 768, 768), ("mn", "mn"), (64, 4)),
                ((72, 136, 3072), ("k", "k"), (64, 8)), ((1000, 3072, 520), ("k", "k"), (128, 1)),
                ((600, 1160, 1160), ("k", "mn"), (128, 2)), ((520, 760, 1160), ("mn", "k"), (128, 4)),
                ((160, 768, 30520), ("k", "mn"), (128, 8)), ((1, 8, 8), ("k", "k"), (64, 1))]


@pytest.mark.parametrize("shape,majors,form", PLANE_SHAPES)
def test_fp32_product_on_split_operands(shape, majors, form):
    """A sum of 64 products leaves tensor memory within 2^-21 of its size, and K / 64 of them are added in fp32:
    far below the 2e-5 of the plain kernel's chain."""
    wgrad = majors == ("mn", "mn")
    _run(0, *shape, *majors, bias=not wgrad, residual=not wgrad, d_fp32=True, accumulate=wgrad, planes=True, tol=1e-6,
         form=(4, 128, form[0], 1, form[1]))


@pytest.mark.parametrize("kw", [dict(act=1, aux_out=True, bias=True), dict(act=2), dict(alpha=0.125, residual=True)])
def test_fp32_split_operands_epilogues(kw):
    _run(0, 200, 136, 264, "k", "mn", d_fp32=True, planes=True, tol=2e-6, **kw)


@pytest.mark.parametrize("ea,eb", [(-100, 58), (58, -100), (-58, -40), (58, 57)])
def test_fp32_split_operands_over_the_exponent_range(ea, eb):
    def scale(A, B):
        A *= np.float32(2.0 ** ea)
        B *= np.float32(2.0 ** eb)
    out, ref = _run(0, 130, 136, 520, "k", "k", d_fp32=True, planes=True, spoil=scale)
    assert np.abs(out - ref).max() / np.abs(ref).max() < 1e-6


@pytest.mark.parametrize("shape,majors", [((130, 136, 520), ("k", "k")), ((72, 136, 3072), ("mn", "k")), ((600, 1160, 1160), ("k", "mn"))])
def test_fp32_split_operands_with_infinities_and_the_largest_values(shape, majors):
    """What has no sum of three bf16 values: the product is what fp32 multiply-adds give, infinite or NaN in
    exactly the same places, and as precise as ever everywhere else."""
    M, N, K = shape
    def spoil(A, B):
        B[:, 3] = np.exp2(np.floor(np.log2(np.abs(B[:, 3]) + 0.1)))   # powers of two: their lower planes are zero
        A[5, 3], A[6, 3] = np.inf, -np.inf
        A[7, 3], B[:, 4], A[7, 4] = np.inf, 2.0, -np.inf              # inf - inf
        A[8, :] = 0.0
        A[8, 5], B[:, 5] = 3.4028235e38, 0.25                         # would round to infinity in bf16
        A[9, 6], B[:, 6] = np.nan, 1.0
        B[2, 7], A[:, 7] = np.inf, np.where(np.arange(M) % 2, 1.0, 0.0)
    out, ref = _run(0, M, N, K, *majors, d_fp32=True, planes=True, spoil=spoil)
    assert np.isinf(ref[5]).any() and np.isnan(ref[7]).all() and np.isnan(ref[9]).all() and np.isfinite(ref[8]).sum() >= N - 1
    assert np.array_equal(np.isnan(out), np.isnan(ref))
    assert np.array_equal(np.isinf(out), np.isinf(ref)) and np.array_equal(np.sign(out[np.isinf(ref)]), np.sign(ref[np.isinf(ref)]))
    fin = np.isfinite(ref)
    small = fin & (np.arange(M) != 8)[:, None]
    assert np.abs(out - ref)[small].max() / np.abs(ref[small]).max() < 2e-5
    assert (np.abs(out[8] - ref[8]) / np.abs(ref[8]))[fin[8]].max() < 1e-6
