"""Which workspace the binding lends to NVFP4 decode calls of 5 to 16 columns: the questions to the library, with a stand-in for it."""
import types

import torch

import paper_2609_26333_b200.binding as binding


class _Library:
    """Answers dq_decode_nvfp4_workspace_bytes with the statuses given, one after the other, and 4096 bytes where the status is 0."""

    def __init__(self, *statuses):
        self.statuses, self.asked = list(statuses), 0

    def dq_decode_nvfp4_workspace_bytes(self, handle, B, any_, out):
        self.asked += 1
        st = self.statuses.pop(0)
        if st == 0:
            out._obj.value = 4096
        return st


def _handle():
    return types.SimpleNamespace(handle=1, packed=torch.empty(0), N=512, K=2048, formats=binding.FMT_NVFP4, nvfp4_ws={})


def test_a_question_without_an_answer_is_asked_again(monkeypatch):
    """A first call that fails (another device current, a CUDA error) does without a workspace and leaves nothing behind: later calls of the
    same handle and batch get theirs.  Answers are kept, for other handles of the same shape too."""
    L = _Library(1, 6, 0)
    monkeypatch.setattr(binding, "lib", lambda: L)
    monkeypatch.setattr(binding, "_nvfp4_ws_known", {})
    monkeypatch.setattr(binding, "_capturing", lambda: False)
    w, other, X = _handle(), _handle(), torch.empty(8, 2048)
    lent = [binding._lent_workspace(w, X, 8, None) for _ in range(4)]
    assert [None if t is None else t.numel() for t in lent] == [None, None, 4096, 4096]
    assert binding._lent_workspace(other, X, 8, None).numel() == 4096
    assert L.asked == 3
