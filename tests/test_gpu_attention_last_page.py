"""Decode attention copies of a context's last page only the 16-key tiles that hold
a key.  Contexts that end just below, at and past the edges of those tiles, of
the pages and of the 64-key batches give the same logits for every page size
(only the order of the sums differs), and the oracle's."""
import copy

import numpy as np
import pytest

import synth
from oracle.mtp import MTPOracle

from gpu_util import assert_logits_close, decoder

pytestmark = pytest.mark.gpu

MODEL = synth.TINY_BF16
N = 4
# keys of the step that feeds N rows: lengths + N
KEYS = [5, 15, 16, 17, 31, 32, 33, 63, 64, 65, 79, 80, 81, 127, 128, 129, 130, 144, 145]
# A key or value fed this step may round to the other bf16 neighbour (2^-9 relative, one of its keys); a key
# too few or too many moves an attention output by about 1 / KEYS of a value.
ATOL = 2e-3


def run(page_size):
    prompts = [synth.make_prompt(700 + k, (k - N) // 3, k - N - (k - N) // 3, MODEL.phone_vocab) for k in KEYS]
    dec, w = decoder(MODEL, max_batch=len(KEYS), max_ctx=256, page_size=page_size)
    try:
        for b, (ph, ac) in enumerate(prompts):
            dec.prefill(b, ph, ac, 4 * N)
        dec.decode_step(N, 2)
        first = dec.logits(N)[0].copy()
        dec.decode_step(N, 2)
        states = [dec.state(b) for b in range(len(KEYS))]
        return first, dec.logits(N)[0].copy(), [s["len"] for s in states], prompts, w
    finally:
        dec.close()


@pytest.fixture(scope="module")
def by_128():
    return run(128)


@pytest.mark.parametrize("page_size", [16, 32, 64])
def test_same_logits_for_every_page_size(page_size, by_128):
    first, second, lens, _, _ = run(page_size)
    assert lens == by_128[2]
    assert np.abs(first - by_128[0]).max() <= ATOL
    assert np.abs(second - by_128[1]).max() <= ATOL


def test_oracle(by_128):
    _, second, lens, prompts, w = by_128
    first = MTPOracle(MODEL, w)
    for b, (ph, ac) in enumerate(prompts):
        o = copy.copy(first)
        o.prefill(ph, ac, 4 * N)
        o.step(N, 2)
        assert_logits_close(second[b], o.step(N, 2).logits, f"{KEYS[b]} keys")
