"""The node kernels at the sizes where they can go wrong: chains (every node has one child), rows at odd offsets from a 16-byte
boundary, trees of more than 32 nodes, peaked rows (normalisers and weights retaken in fp64), vocabularies of one chunk."""
import numpy as np
import pytest
import torch

from paper_2602_16994_b200 import binding
from paper_2602_16994_b200.synth import Workload, make_batch
from tests.parity import check_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("algo", ["specinfer", "traversal"])
@pytest.mark.parametrize("w", [
    Workload("chain", 5, 4099, "bf16", 1, 0, 7, 0.8),
    Workload("chain_peaked", 6, 8193, "bf16", 1, 2, 4, 0.6, temperature=0.25),
    Workload("one_chunk", 9, 7, "f32", 2, 1, 2, 0.8),
    Workload("chunk_edge", 4, 2049, "f32", 3, 1, 2, 0.8),
    Workload("peaked", 6, 16385, "bf16", 3, 2, 3, 0.5, temperature=0.3),
    Workload("forty_nodes", 3, 5003, "bf16", 6, 3, 6, 0.8),
    Workload("many", 400, 2000, "bf16", 2, 1, 2, 0.8),
], ids=lambda w: w.name)
def test_nodes(w, algo):
    check_batch(make_batch(w, seed=3, device="cuda"), algo, full=False)


@pytest.mark.parametrize("shift", [(1, 1), (1, 2), (0, 3)])
def test_rows_at_any_alignment(shift):
    """Target and draft tensors that start at their own odd offsets: the same results as aligned ones."""
    b = make_batch(Workload("shifted", 4, 6001, "bf16", 3, 1, 3, 0.7), seed=5, device="cuda")
    rest = (b.parent, b.token, b.u_accept, b.u_bonus)

    def moved(t, by):
        buf = torch.empty(t.numel() + 8, dtype=t.dtype, device=t.device)
        v = buf[by:by + t.numel()].view(t.shape)
        v.copy_(t)
        return v
    for call in (binding.verify_specinfer, binding.verify_traversal):
        want = call(b.target_logits, b.draft_logits, *rest)
        got = call(moved(b.target_logits, shift[0]), moved(b.draft_logits, shift[1]), *rest)
        for f in ("accepted_node", "accept_len", "out_tokens", "bonus_token", "status"):
            assert np.array_equal(getattr(want, f).cpu().numpy(), getattr(got, f).cpu().numpy()), f


@pytest.mark.parametrize("per_seq", [False, True])
def test_host_call_leaves_childless_rows_behind(per_seq):
    """Rows long enough that the host-buffer call skips the draft rows of childless nodes; the same decisions."""
    w = Workload("host", 3, 40000, "bf16", 3, 1, 2, 0.7)
    d = make_batch(w, seed=2, device="cuda")
    several = lambda t: t.reshape(1, -1).repeat(w.B, 1).contiguous() if per_seq else t
    for algo, call in (("specinfer", binding.verify_specinfer), ("traversal", binding.verify_traversal)):
        want = call(d.target_logits, d.draft_logits, several(d.parent), d.token, d.u_accept, d.u_bonus)
        hv = binding.HostVerifier(w.B, w.N, w.V, torch.bfloat16, algorithm=algo, per_sequence_topology=per_seq)
        host = [t.cpu().pin_memory() for t in (d.target_logits, d.draft_logits, several(d.parent), d.token, d.u_accept, d.u_bonus)]
        got = hv.run(*host)
        for f in ("accepted_node", "accept_len", "out_tokens", "bonus_token", "status"):
            assert np.array_equal(getattr(want, f).cpu().numpy(), got[f].numpy()), (algo, f)
        assert hv.h2d_bytes(host[2]) < hv.h2d_bytes()
