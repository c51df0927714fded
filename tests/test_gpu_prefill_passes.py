"""Prefill passes (Sec. III-A: the prompt runs through the blocks as one sequence)
against the oracle at the sizes where a pass can go wrong: fewer rows than an
attention group, the edges of the 128-row tiles, and prompts or batches of
prompts just below, at and past the rows one pass holds (96 per SM)."""
import copy

import numpy as np
import pytest

import synth
from oracle.mtp import MTPOracle

from gpu_util import assert_logits_close, decoder, lib_module

pytestmark = pytest.mark.gpu

MODEL = synth.TINY_BF16


@pytest.mark.parametrize("length", [1, 7, 9, 127, 129, 257, 304, 305, 385, 1025, 4095, 4097])
def test_one_prompt(length):
    ph, ac = synth.make_prompt(300 + length, length // 3, length - length // 3, MODEL.phone_vocab)
    dec, w = decoder(MODEL, max_batch=1, max_ctx=length + 32)
    try:
        dec.prefill(0, ph, ac, 8)
        dec.decode_step(4, 4)
        o = MTPOracle(MODEL, w)
        o.prefill(ph, ac, 8)
        assert_logits_close(dec.logits(4)[0][0], o.step(4, 4).logits, f"prompt of {length}")
        assert dec.state(0)["len"] == length
    finally:
        dec.close()


def _lengths(kind, rows):
    """Prompt lengths around the `rows` rows of a pass (a multiple of 8; prompts take whole groups of 8)."""
    if kind in ("one pass", "a row more"):   # full, and one prompt row left for the second pass
        rest = rows % 1024 or 1024
        return [1024] * ((rows - rest) // 1024) + [rest - 8, 8 if kind == "one pass" else 9]
    if kind == "cut":                        # a prompt cut by the end of the pass
        return [900, 333] * (rows // (904 + 336) + 3)
    return kind


@pytest.mark.parametrize("kind,passes", [
    ([5, 130, 61], 1), ([700, 1300, 900, 1100, 500, 33], 1), ("one pass", 1), ("a row more", 2), ("cut", 2),
])
def test_admitted_prompts(kind, passes):
    torch = pytest.importorskip("torch")
    mtp = lib_module()
    lengths = _lengths(kind, 96 * torch.cuda.get_device_properties(0).multi_processor_count)
    prompts = [synth.make_prompt(320 + b, t // 4, t - t // 4, MODEL.phone_vocab) for b, t in enumerate(lengths)]
    dec, w = decoder(MODEL, max_batch=len(lengths), max_ctx=max(lengths) + 32)
    try:
        for b, (ph, ac) in enumerate(prompts):
            dec.admit(b, ph, ac, 8)
        assert mtp.mtp_prefill_pending(dec.ctx) == passes
        dec.decode_step(4, 4)
        lg = dec.logits(4)[0]
        first = MTPOracle(MODEL, w)
        for b, (ph, ac) in enumerate(prompts):
            o = copy.copy(first)
            o.prefill(ph, ac, 8)
            assert_logits_close(lg[b], o.step(4, 4).logits, f"slot {b}")
            assert dec.state(b)["len"] == lengths[b]
    finally:
        dec.close()
    assert np.isfinite(lg).all()
