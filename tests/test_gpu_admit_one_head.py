"""A prompt admitted mid-generation while one token is decoded at a time: the lane's attention groups
are single rows, taken by a CTA each where there are few heads."""
import pytest

import synth

from test_gpu_admit import _admit_mid_generation

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,admit_len", [(3, 300), (10, 700)])
def test_one_row_groups(batch, admit_len):
    _admit_mid_generation(synth.TINY_BF16, batch, 1, 4, admit_len, 2, 9, 900)
