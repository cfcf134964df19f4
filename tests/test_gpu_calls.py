"""The native host path of the Python calls: what it holds while a call is being made."""
import weakref

import pytest
import torch

from paper_2602_16994_b200 import binding
from paper_2602_16994_b200.synth import Workload, make_batch

pytestmark = pytest.mark.gpu


def test_outputs_are_held_until_the_call_is_enqueued():
    """An outputs object whose attributes are computed: nobody but the call holds the tensors it gives out."""
    w = Workload("held", 2, 2000, "f32", 2, 0, 2, 0.8)
    b = make_batch(w, seed=1, device="cuda")
    seen = []

    class Computed:
        def __getattr__(self, name):
            if name not in ("accepted_node", "accept_len", "out_tokens", "bonus_token", "status"):
                return None
            t = torch.empty((w.B, w.N) if name == "out_tokens" else w.B, dtype=torch.int32, device="cuda")
            seen.append(weakref.ref(t))
            return t

    class Stream:
        """Asked for after the outputs have been read, before the launches."""

        @property
        def cuda_stream(self):
            alive.append([r() is not None for r in seen])
            return torch.cuda.current_stream().cuda_stream

    alive = []
    binding.verify_specinfer(b.target_logits, b.draft_logits, b.parent, b.token, b.u_accept, b.u_bonus,
                             outputs=Computed(), stream=Stream())
    torch.cuda.synchronize()
    assert alive == [[True] * 5]
