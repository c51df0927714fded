"""mtp_heads_topk (Sec. III-B heads, log-softmax and top-k in one pass) where its candidate
exchange can go wrong: more candidates in one half of a vocabulary slice than are sent, rows
with too few above the threshold beside ordinary ones, ties at the k-th place; and where the
rows are read: in place (aligned fp32 and bf16) or after a conversion (rows at odd addresses)."""
import numpy as np
import pytest

import synth
from oracle import select as S

from gpu_util import lib_module, logp32

pytestmark = pytest.mark.gpu

MODEL = synth.TINY_BF16


def _run(mtp, dec, hidden, dtype, n, k):
    import torch
    b, v = hidden.shape[0], MODEL.codec_vocab
    ids = torch.full((b, n, k), -5, dtype=torch.int32, device="cuda")
    lp = torch.zeros((b, n, k), device="cuda")
    lg, lse = torch.zeros((b, n, v), device="cuda"), torch.zeros((b, n), device="cuda")
    mtp.mtp_heads_topk(dec.ctx, b, hidden, dtype, n, k, ids, lp, lg, lse)
    torch.cuda.synchronize()
    return [t.cpu().numpy() for t in (ids, lp, lg, lse)]


def _decoder(mtp, bias):
    w = dict(synth.make_weights(MODEL))
    w["b_heads"] = np.broadcast_to(bias, (MODEL.n_heads_max, MODEL.codec_vocab)).astype(np.float32).copy()
    return mtp.MTPDecoder(MODEL, w, synth.weight_names(MODEL), synth.is_matrix, 16, 64)


def _biases():
    v = MODEL.codec_vocab
    i = np.arange(v)
    return {
        "plain": np.zeros(v),
        "clustered": np.where(i < 64, 6.0, 0.0),                    # 64 candidates in one half
        "edge": np.where((i >= 960) & (i < 992), 6.0, 0.0),         # exactly as many as are sent
        "few": np.where(i == 700, 60.0, np.where(i == 20, 40.0, 0.0)),  # two outliers set the threshold
        "steps": 0.25 * (i % 5),                                    # many near-ties
    }


@pytest.mark.parametrize("bias", ["plain", "clustered", "edge", "few", "steps"])
@pytest.mark.parametrize("rows,n,k", [(9, 8, 1), (33, 2, 4), (128, 3, 16), (129, 8, 32), (300, 1, 7)])
def test_candidates(bias, rows, n, k):
    torch = pytest.importorskip("torch")
    mtp = lib_module()
    dec = _decoder(mtp, _biases()[bias])
    try:
        h = torch.from_numpy(synth.make_hidden(rows, MODEL.d_model, seed=rows + k)).cuda()
        ids, lp, lg, lse = _run(mtp, dec, h, 0, n, k)
        for b in range(rows):  # exact on the call's own scores
            r_ids, r_vals = S.top_k_rows(logp32(lg[b], lse[b]), k)
            assert np.array_equal(ids[b], r_ids), f"row {b}"
            assert np.array_equal(lp[b].view(np.uint32), r_vals.view(np.uint32)), f"row {b}"
    finally:
        dec.close()


@pytest.mark.parametrize("rows", [1, 5, 8, 9, 200])
@pytest.mark.parametrize("offset", [0, 1, 2, 4])
def test_rows_in_place_or_converted(rows, offset):
    """The same rows at every alignment, fp32 and bf16 (their values are bf16): one result."""
    torch = pytest.importorskip("torch")
    mtp = lib_module()
    dec = _decoder(mtp, np.zeros(MODEL.codec_vocab))
    try:
        h = torch.from_numpy(synth.make_hidden(rows, MODEL.d_model, seed=rows)).cuda()
        want = _run(mtp, dec, h, 0, 4, 8)
        for dtype, t in ((0, h), (1, h.bfloat16())):
            room = torch.zeros(t.numel() + offset, dtype=t.dtype, device="cuda")
            shifted = room[offset:].view_as(t)
            shifted.copy_(t)
            for got, ref in zip(_run(mtp, dec, shifted, dtype, 4, 8), want):
                assert np.array_equal(got, ref)
    finally:
        dec.close()
