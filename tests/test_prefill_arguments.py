"""What Koala.prefill hands to the library (host logic; the library is a stand-in)."""
import types

import numpy as np
import pytest
import torch

from paper_2408_08146_b200 import Koala


class Recorder:
    def koala_ingest(self, ctx, tok, stride, lens, n_parts):
        self.stride, self.lens, self.n_parts = stride, list(lens), n_parts
        return 0


def _engine(B, N=15):
    eng = object.__new__(Koala)
    eng.cfg, eng.dev, eng.lib, eng._ctx = types.SimpleNamespace(B=B, N=N), torch.device("cpu"), Recorder(), None
    eng.buffers = lambda: {"tree_n": None}
    eng.koala_accept = lambda forced: None
    return eng


def test_fewer_prompts_than_sequences_are_refused():
    """The library reads B lengths."""
    eng = _engine(3)
    with pytest.raises(IndexError):
        eng.prefill([[1, 2, 3], [4, 5]], 2)
    assert not hasattr(eng.lib, "lens")


def test_prompts_beyond_the_batch_are_left_out():
    eng = _engine(2)
    eng.prefill([np.arange(20), list(range(9)), np.arange(16)], 10)
    assert (eng.lib.stride, eng.lib.lens, eng.lib.n_parts) == (20, [20, 9], 2)
