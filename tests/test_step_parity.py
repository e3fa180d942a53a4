"""GPU parity of the whole stage step against the CPU oracle, element by element, through the
C ABI.  Sizes are chosen so that the oracle finishes in seconds while the contractions still
span several tiles and ragged tails."""
import math

import numpy as np
import pytest

from paper_2011_13635_b200 import inputs as I
from tests import parity as PT

pytestmark = pytest.mark.gpu

TINY = I.CONFIGS["tiny"]


def _run(cfg, steps, lr, batch_seed=None, **opt):
    m, oracle = PT.build_pair(cfg, lr=lr, **opt)
    tol = PT.TOL[cfg.dtype]
    rep = []
    for s in range(steps):
        batch = I.make_batch(cfg, seed=(batch_seed or I.config_seed(cfg)) + s)
        PT.compare_step(m, oracle, cfg, batch, tol, rep)
    m.close()
    return rep


# -- fp32 path -------------------------------------------------------------------------------

def test_tiny_fp32_staged_step():
    """The small configuration as given: 1 frozen + 1 trainable layer, fp32."""
    rep = _run(TINY, steps=3, lr=1e-3)
    assert abs(rep[0]["loss_gpu"] - math.log(TINY.vocab)) < 0.2


@pytest.mark.parametrize("top_k", [0, 2])
def test_fp32_head_only_and_all_trainable(top_k):
    _run(I.scaled(TINY, trainable=top_k), steps=2, lr=1e-3)


def test_fp32_ragged_shapes_with_padding():
    cfg = I.StageConfig("ragged32", hidden=192, heads=3, ffn=320, vocab=1037, max_pos=80, layers=3,
                        trainable=2, batch=3, seq=72, pred=7, dtype="fp32", varlen=(20, 72),
                        seed_index=11)
    _run(cfg, steps=2, lr=1e-3)
    _run(I.scaled(cfg, trainable=3), steps=2, lr=1e-3)


def test_fp32_lamb_staged_and_all_trainable():
    """LAMB at the learning rate of the paper's experiments (Section 4.1): per-tensor trust ratios."""
    _run(TINY, steps=3, lr=0.00088, lamb=1)
    _run(I.scaled(TINY, trainable=2), steps=2, lr=0.00088, lamb=1, weight_decay=0.0)


def _run_nsp(cfg, steps, lr, drop_labels=False):
    """Both objectives (Section 4.1): segment embeddings, pooler and two-way classifier."""
    m, oracle = PT.build_pair(cfg, lr=lr)
    assert oracle.nsp and "emb.type" in m.tensors() and "head.nsp.weight" in m.tensors()
    rep = []
    for s in range(steps):
        seed = I.config_seed(cfg) + s
        tok, lens, pos, lab = I.make_batch(cfg, seed=seed)
        seg, nlab = I.make_nsp(cfg, lens, seed=seed)
        if s == 1:
            nlab[0] = -1                               # an ignored sequence
        PT.compare_step(m, oracle, cfg, (tok, lens, pos, lab, seg, None if drop_labels else nlab),
                        PT.TOL[cfg.dtype], rep)
    m.close()
    return rep


def test_fp32_nsp_objective_staged_and_all_trainable():
    cfg = I.scaled(TINY, nsp=True, varlen=(20, 64))
    rep = _run_nsp(cfg, steps=2, lr=1e-3)
    assert abs(rep[0]["loss_gpu"] - (math.log(cfg.vocab) + math.log(2))) < 0.3      # MLM + NSP at the start
    _run_nsp(I.scaled(cfg, trainable=2), steps=2, lr=1e-3)
    rep = _run_nsp(cfg, steps=1, lr=1e-3, drop_labels=True)                         # segments only
    assert abs(rep[0]["loss_gpu"] - math.log(cfg.vocab)) < 0.2


# -- bf16 path ---------------------------------------------------------------------------------

BASE_SMALL = I.scaled(I.CONFIGS["base_stage"], layers=3, trainable=2, batch=4)


def test_bf16_base_shapes_staged():
    """BERT-Base widths and vocabulary, 1 frozen + 2 trainable layers, 4 sequences of 128."""
    rep = _run(BASE_SMALL, steps=2, lr=1e-4)
    assert abs(rep[0]["loss_gpu"] - math.log(30522)) < 0.3


def test_bf16_base_shapes_all_trainable():
    _run(I.scaled(BASE_SMALL, layers=2, trainable=2, batch=3), steps=2, lr=1e-4)


def test_bf16_lamb_base_shapes():
    _run(BASE_SMALL, steps=2, lr=0.00088, lamb=1)
    _run(I.scaled(BASE_SMALL, layers=2, trainable=2, batch=2), steps=1, lr=0.00088, lamb=1)


def test_bf16_nsp_objective_base_shapes():
    cfg = I.scaled(BASE_SMALL, nsp=True)
    _run_nsp(cfg, steps=2, lr=1e-4)
    _run_nsp(I.scaled(cfg, layers=2, trainable=2, batch=3), steps=1, lr=1e-4)


def test_bf16_head_only():
    _run(I.scaled(BASE_SMALL, layers=1, trainable=0, batch=2), steps=1, lr=1e-4)


def test_bf16_ragged_shapes_with_padding():
    cfg = I.StageConfig("ragged16", hidden=192, heads=3, ffn=320, vocab=1037, max_pos=80, layers=2,
                        trainable=1, batch=3, seq=72, pred=7, dtype="bf16", varlen=(20, 72),
                        seed_index=12)
    _run(cfg, steps=2, lr=1e-4)
    _run(I.scaled(cfg, trainable=2), steps=1, lr=1e-4)


def test_bf16_large_long_shapes():
    """BERT-Large widths at sequence length 512 with per-sequence padding."""
    cfg = I.scaled(I.CONFIGS["large_long"], layers=2, trainable=1, batch=2)
    _run(cfg, steps=1, lr=1e-4)


# -- forward-only entry point ----------------------------------------------------------------------

@pytest.mark.parametrize("cfg", [TINY, I.scaled(BASE_SMALL, batch=2),
                                 I.scaled(I.CONFIGS["large_long"], layers=2, trainable=1, batch=2)],
                         ids=["tiny", "base", "large_long"])
def test_forward_matches_oracle(cfg):
    import torch
    m, oracle = PT.build_pair(cfg, lr=1e-3)
    tok, lens, pos, lab = I.make_batch(cfg)
    d_tok, d_lens, d_pos = PT.to_cuda(torch, tok, lens if cfg.varlen else None, pos)
    hidden, logits = m.mslt_forward(d_tok, d_lens, d_pos)
    h_ref, l_ref = oracle.forward(tok, lens, pos)
    hidden = hidden.float().cpu().numpy()
    tol = PT.TOL[cfg.dtype]["hidden"]
    for b in range(cfg.batch):       # rows at padded positions are unspecified
        n = int(lens[b])
        assert PT.max_rel(hidden[b, :n], h_ref[b, :n]) < tol
    ok = (pos >= 0).reshape(-1)
    lg = logits.cpu().numpy()
    assert PT.max_rel(lg[ok], l_ref[ok]) < tol
    # the loss recomputed from these logits equals the loss the training step reports
    labels = np.where(ok, lab.reshape(-1), -1)
    lg64 = lg.astype(np.float64)
    lse = np.log(np.exp(lg64 - lg64.max(1, keepdims=True)).sum(1)) + lg64.max(1)
    nll = (lse - lg64[np.arange(len(labels)), np.maximum(labels, 0)])[ok]
    d_lab = PT.to_cuda(torch, lab)[0]
    m.mslt_set_optimizer(lr=0.0)
    loss = m.mslt_step(d_tok, d_lens, d_pos, d_lab)
    assert abs(loss - nll.mean()) / nll.mean() < 1e-5
    assert m.mslt_debug_check_guards() == 0
    m.close()


def test_bf16_step_with_unfused_attention_in_a_child_process():
    """The batched-product attention path (what longer rows and odd lengths fall back to) is selected
    by an environment switch the library reads once, so it runs in a child process: same parity
    check as above on BERT-Base widths with a padding mask."""
    import os
    import subprocess
    import sys
    code = (
        "import math\n"
        "from paper_2011_13635_b200 import inputs as I\n"
        "from tests import parity as PT\n"
        "cfg = I.scaled(I.CONFIGS['base_stage'], layers=2, trainable=1, batch=3)\n"
        "cfg = I.StageConfig('unfused', hidden=cfg.hidden, heads=cfg.heads, ffn=cfg.ffn, vocab=cfg.vocab,\n"
        "                    max_pos=cfg.max_pos, layers=2, trainable=1, batch=3, seq=128, pred=cfg.pred,\n"
        "                    dtype='bf16', varlen=(40, 128), seed_index=23)\n"
        "m, oracle = PT.build_pair(cfg, lr=1e-4)\n"
        "before = m.launch_count\n"
        "PT.compare_step(m, oracle, cfg, I.make_batch(cfg), PT.TOL[cfg.dtype])\n"
        "print('launches', m.launch_count - before)\n"
        "m.close()\n")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    counts = {}
    for unfused in ("0", "1"):
        env = dict(os.environ, MSLT_UNFUSED_ATTENTION=unfused, PYTHONPATH=root)
        r = subprocess.run([sys.executable, "-c", code], cwd=root, env=env, capture_output=True, text=True,
                           timeout=600)
        assert r.returncode == 0, r.stdout + r.stderr
        counts[unfused] = int(r.stdout.strip().split()[-1])
    # two launches per layer forward become three, one per trainable layer backward becomes five
    assert counts["1"] > counts["0"]


@pytest.mark.parametrize("seq,varlen,nsp", [(128, (1, 128), False), (136, (1, 136), True), (256, (120, 256), False),
                                            (512, (60, 512), False), (136, None, False), (384, None, False)])
def test_bf16_packed_batches_and_long_row_backward(seq, varlen, nsp):
    """Batches with lengths run without their padding, rows of more than 128 keys recompute their
    probabilities in the backward pass: lengths of 1, ragged last tiles, every layer and the
    embeddings trained, and the same without lengths."""
    cfg = I.StageConfig("packed", hidden=192, heads=3, ffn=320, vocab=1037, max_pos=512, layers=2, trainable=2,
                        batch=5, seq=seq, pred=9, dtype="bf16", varlen=varlen, seed_index=31, nsp=nsp)
    if nsp:
        _run_nsp(cfg, steps=2, lr=1e-4)
    else:
        _run(cfg, steps=2, lr=1e-4)


def test_bf16_forward_zeroes_the_padding_of_a_packed_batch():
    import torch
    cfg = I.scaled(I.CONFIGS["base_stage"], layers=1, trainable=1, batch=3, varlen=(20, 128))
    m, oracle = PT.build_pair(cfg, lr=1e-3)
    tok, lens, pos, lab = I.make_batch(cfg)
    d_tok, d_lens = PT.to_cuda(torch, tok, lens)
    hidden, _ = m.mslt_forward(d_tok, d_lens)
    hidden = hidden.float().cpu().numpy()
    h_ref, _ = oracle.forward(tok, lens, pos)
    for b in range(cfg.batch):
        n = int(lens[b])
        assert PT.max_rel(hidden[b, :n], h_ref[b, :n]) < PT.TOL["bf16"]["hidden"]
        assert not hidden[b, n:].any()
    m.close()


@pytest.mark.parametrize("layers,trainable,batch,seq", [(2, 1, 3, 72), (1, 1, 9, 128)])
def test_fp32_base_shapes_on_split_operands(layers, trainable, batch, seq):
    """BERT-Base widths in fp32: the linear products are large enough for the tensor-core form on
    operands split into bf16 planes (ragged rows, k split over clusters, the vocabulary-long
    contractions), held to the fp32 tolerances."""
    cfg = I.scaled(I.CONFIGS["base_stage"], layers=layers, trainable=trainable, batch=batch, seq=seq, pred=11,
                   dtype="fp32", varlen=(seq // 3, seq))
    _run(cfg, steps=2, lr=1e-3)


@pytest.mark.parametrize("seq,varlen", [(8, (1, 8)), (40, None), (64, (1, 64)), (72, (5, 72)), (128, (30, 128)), (136, (1, 136))])
def test_fp32_attention_row_lengths(seq, varlen):
    """The fused fp32 attention at the edges of its 32-row blocks and 64-row buffers (and the batched
    products just beyond its range), lengths that leave whole blocks without keys."""
    cfg = I.StageConfig("attn32", hidden=128, heads=2, ffn=128, vocab=131, max_pos=136, layers=1, trainable=1, batch=4,
                        seq=seq, pred=5, dtype="fp32", varlen=varlen, seed_index=37)
    _run(cfg, steps=2, lr=1e-3)


@pytest.mark.parametrize("batch,rest", [(32, 1), (32, 9), (4, 8)])
def test_packed_batch_of_few_rows(batch, rest):
    """Sequences far shorter than the batch is wide: most blocks of a launch find no rows left for them, after they
    have asked for their first weights."""
    cfg = I.scaled(I.CONFIGS["base_stage"], layers=2, trainable=1, batch=batch, varlen=(1, 128))
    m, oracle = PT.build_pair(cfg, lr=1e-4)
    PT.compare_step(m, oracle, cfg, _batch_of_lengths(cfg, (40,) + (rest,) * (batch - 1)), PT.TOL["bf16"])
    m.close()


@pytest.mark.parametrize("vocab,trainable", [(500, 1), (768, 2), (1700, 1)])
def test_vocabulary_not_much_wider_than_the_hidden_state(vocab, trainable):
    """The sums of the head's input gradient lie in the logits' memory: none fit beside a row of 500 logits, one in 768,
    two in 1704."""
    _run(I.scaled(I.CONFIGS["base_stage"], layers=2, trainable=trainable, batch=2, vocab=vocab), steps=2, lr=1e-4)


@pytest.mark.parametrize("dtype,seq,varlen,pred", [("fp32", 40, None, 5), ("fp32", 72, (20, 72), 33), ("bf16", 136, (40, 136), 9),
                                                   ("bf16", 64, None, 40)])
def test_slots_that_name_a_position_twice(dtype, seq, varlen, pred):
    """The slots' gradients are gathered by row: rows with no slot, one, several (some in another group
    of 32 slots), empty slots, and the rows that pad a packed batch."""
    cfg = I.StageConfig("twice", hidden=128, heads=2, ffn=128, vocab=131, max_pos=136, layers=1, trainable=1, batch=3,
                        seq=seq, pred=pred, dtype=dtype, varlen=varlen, seed_index=41)
    m, oracle = PT.build_pair(cfg, lr=1e-4)
    tok, lens, pos, lab = I.make_batch(cfg)
    pos, lab = pos.copy(), lab.copy()
    pos[:, -1] = pos[:, 0]
    pos[:, 2] = pos[:, 1]
    lab[:, -1], lab[:, 2] = lab[:, 0], lab[:, 1]
    lab[0, 3] = -1
    PT.compare_step(m, oracle, cfg, (tok, lens, pos, lab), PT.TOL[dtype], [])
    m.close()


def _batch_of_lengths(cfg, lens):
    """tokens, lengths, positions and labels of a batch with the given lengths."""
    rng = np.random.default_rng(5)
    tok = rng.integers(1, cfg.vocab, size=(cfg.batch, cfg.seq)).astype(np.int32)
    pos = np.full((cfg.batch, cfg.pred), -1, dtype=np.int32)
    lab = np.full((cfg.batch, cfg.pred), -1, dtype=np.int32)
    for b, n in enumerate(lens):
        tok[b, n:] = 0
        k = min(cfg.pred, n)
        pos[b, :k] = np.sort(rng.choice(n, size=k, replace=False))
        lab[b, :k] = rng.integers(0, cfg.vocab, size=k)
    return tok, np.array(lens, dtype=np.int32), pos, lab


PACKED_EDGES = [(128, (30, 28, 20, 20, 30)), (256, (130, 20, 70, 6, 30)), (512, (3, 300, 1, 129, 79))]


@pytest.mark.parametrize("seq,lens", PACKED_EDGES)
def test_packed_batch_does_not_see_the_rows_of_an_earlier_call(seq, lens):
    """A full batch with a NaN weight fills every activation buffer with NaN; the weights are restored
    and a short packed batch follows whose last sequence ends a tile of 128 rows exactly, so that its
    own tile reaches into rows that only the first call wrote."""
    import torch
    cfg = I.StageConfig("stale", hidden=192, heads=3, ffn=320, vocab=1037, max_pos=512, layers=2, trainable=1,
                        batch=5, seq=seq, pred=9, dtype="bf16", varlen=(1, seq), seed_index=43)
    assert sum(lens) % 128 == 0
    m, oracle = PT.build_pair(cfg, lr=1e-4)
    weights = {n: m.mslt_get_param(n) for n in oracle.p}
    bad = weights["emb.word"].copy()
    bad[:] = np.nan
    m.mslt_set_param("emb.word", bad)
    tok, _, pos, lab = _batch_of_lengths(cfg, (seq,) * cfg.batch)
    assert math.isnan(m.mslt_step(*PT.to_cuda(torch, tok, None, pos, lab)))
    m.set_params(weights)
    m.mslt_set_trainable(cfg.trainable)      # moments and step count start again
    PT.compare_step(m, oracle, cfg, _batch_of_lengths(cfg, lens), PT.TOL["bf16"])
    m.close()


@pytest.mark.parametrize("seq,lens", PACKED_EDGES)
def test_packed_sequence_does_not_see_its_neighbour(seq, lens):
    """A token whose word vector is infinite makes its own sequence NaN and no other."""
    import torch
    cfg = I.StageConfig("neighbour", hidden=192, heads=3, ffn=320, vocab=1037, max_pos=512, layers=2, trainable=1,
                        batch=5, seq=seq, pred=9, dtype="bf16", varlen=(1, seq), seed_index=43)
    m, oracle = PT.build_pair(cfg, lr=1e-4)
    tok, length, pos, _ = _batch_of_lengths(cfg, lens)
    tok[tok == 7] = 8
    h_ref, _ = oracle.forward(tok, length, pos)
    word = m.mslt_get_param("emb.word")
    word[7] = np.inf
    m.mslt_set_param("emb.word", word)
    tok[1, 0] = tok[3, 0] = 7
    hidden = m.mslt_forward(*PT.to_cuda(torch, tok, length))[0].float().cpu().numpy()
    for b, n in enumerate(lens):
        if b in (1, 3):
            assert np.isnan(hidden[b, :n]).all()
        else:
            assert PT.max_rel(hidden[b, :n], h_ref[b, :n]) < PT.TOL["bf16"]["hidden"]
    m.close()


@pytest.mark.parametrize("lens", [(1, 15, 16, 17, 79), (31, 32, 33, 16, 16), (96, 97, 127, 128, 64)])
def test_packed_sequences_around_the_ends_of_contraction_steps(lens):
    """The context of rows of up to 128 keys is contracted 16 keys at a time, up to the last one of the sequence."""
    test_packed_batch_does_not_see_the_rows_of_an_earlier_call(128, lens)
    test_packed_sequence_does_not_see_its_neighbour(128, lens)


@pytest.mark.parametrize("hidden,ffn", [(384, 1088), (448, 1280)])
def test_fp32_one_head_of_one_sequence(hidden, ffn):
    """The attention products of a single (sequence, head) have no batch and are as large as the linear ones,
    but read views of the fused projection; compare_step checks that no kernel wrote outside its buffer."""
    cfg = I.StageConfig("onehead", hidden=hidden, heads=1, ffn=ffn, vocab=131, max_pos=512, layers=1, trainable=1, batch=1,
                        seq=512, pred=5, dtype="fp32", varlen=None, seed_index=47)
    _run(cfg, steps=2, lr=1e-3)


@pytest.mark.parametrize("varlen", [None, (20, 72)])
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
def test_forward_outputs_need_no_alignment(dtype, varlen):
    """The hidden states and logits of the C call go to any address of their element type."""
    import ctypes as C
    import torch
    from paper_2011_13635_b200 import binding as Bd
    cfg = I.StageConfig("align", hidden=128, heads=2, ffn=128, vocab=130, max_pos=72, layers=2, trainable=1, batch=3, seq=72,
                        pred=5, dtype=dtype, varlen=varlen, seed_index=51)
    m, _ = PT.build_pair(cfg, lr=1e-4)
    tok, lens, pos, _ = I.make_batch(cfg)
    d_tok, d_lens, d_pos = PT.to_cuda(torch, tok, lens if varlen else None, pos)
    h_ref, l_ref = m.mslt_forward(d_tok, d_lens, d_pos)
    buf = torch.zeros(h_ref.numel() + 2, dtype=h_ref.dtype, device="cuda")
    lbuf = torch.zeros(l_ref.numel() + 2, device="cuda")
    Bd._check(Bd.lib.mslt_forward(m.h, d_tok.data_ptr(), Bd._ptr(d_lens), cfg.batch, cfg.seq,
                                  C.c_void_p(buf[1:].data_ptr()), d_pos.data_ptr(), cfg.pred,
                                  C.c_void_p(lbuf[1:].data_ptr())))
    assert torch.equal(buf[1:-1].view_as(h_ref), h_ref) and torch.equal(lbuf[1:-1].view_as(l_ref), l_ref)
    assert not buf[0] and not buf[-1] and not lbuf[0] and not lbuf[-1]
    m.close()
