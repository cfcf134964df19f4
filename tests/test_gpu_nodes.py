"""The node kernels at the sizes where they can go wrong: chains (every node has one child), rows at odd offsets from a 16-byte
boundary, trees of more than 32 nodes, peaked rows (normalisers and weights retaken in fp64), vocabularies of one chunk."""
import os
import subprocess
import sys

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


@pytest.mark.parametrize("algo", ["specinfer", "traversal"])
@pytest.mark.parametrize("w", [
    Workload("v420001", 2, 420001, "bf16", 3, 1, 2, 0.7),                          # registers in the recursion, none in the draw
    Workload("v450001", 2, 450001, "bf16", 3, 2, 2, 0.6, temperature=0.5),
    Workload("v620003", 1, 620003, "f32", 3, 1, 2, 0.7),                           # close to the largest V
], ids=lambda w: w.name)
def test_vocabularies_beyond_shared_memory(w, algo):
    """Above about 400000 tokens a node's e no longer fit in the shared memory of 16 CTAs: eight chunks per thread stay in
    registers, in every cluster kernel (the plain SpecInfer call is the walk, the others go node by node)."""
    check_batch(make_batch(w, seed=4, device="cuda"), algo)


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


@pytest.mark.parametrize("busy", [False, True])
@pytest.mark.parametrize("per_seq", [False, True])
def test_host_call_leaves_childless_rows_behind(per_seq, busy):
    """Rows long enough that the host-buffer call skips the draft rows of childless nodes, also on a stream that still has
    work to do; the same decisions."""
    w = Workload("host", 3, 40000, "bf16", 3, 1, 2, 0.7)
    d = make_batch(w, seed=2, device="cuda")
    several = lambda t: t.reshape(1, -1).repeat(w.B, 1).contiguous() if per_seq else t
    for algo, call in (("specinfer", binding.verify_specinfer), ("traversal", binding.verify_traversal)):
        want = call(d.target_logits, d.draft_logits, several(d.parent), d.token, d.u_accept, d.u_bonus)
        hv = binding.HostVerifier(w.B, w.N, w.V, torch.bfloat16, algorithm=algo, per_sequence_topology=per_seq)
        host = [t.cpu().pin_memory() for t in (d.target_logits, d.draft_logits, several(d.parent), d.token, d.u_accept, d.u_bonus)]
        hv.staging.fill_(0xA5)
        torch.cuda.synchronize()
        if busy:
            with torch.cuda.stream(hv.stream):
                torch.cuda._sleep(20_000_000)                  # about 10 ms
        got = hv.run(*host)
        off = -hv.staging.data_ptr() % 256 + (w.B * w.N * w.V * 2 + 255) // 256 * 256        # the staged draft rows
        rows = hv.staging[off:off + w.B * w.N * w.V * 2].view(w.B, w.N, w.V * 2)
        left = int((rows == 0xA5).all(-1).sum())
        assert left * w.V * 2 == hv.h2d_bytes() - hv.h2d_bytes(host[2])
        for f in ("accepted_node", "accept_len", "out_tokens", "bonus_token", "status"):
            assert np.array_equal(getattr(want, f).cpu().numpy(), got[f].numpy()), (algo, f)
        assert hv.h2d_bytes(host[2]) < hv.h2d_bytes()


# branching nodes below one-child nodes whose rows are peaked; the third batch has so many of them that each is left to one warp,
# the last rows so long that the node kernels find no room for each other on an SM
ORDER = [Workload("trunk", 3, 8193, "bf16", 3, 3, 2, 0.5, temperature=0.25),
         Workload("trunk_cut", 2, 32000, "bf16", 2, 2, 2, 0.6, temperature=0.6, top_p=0.95),
         Workload("many_peaked", 400, 2003, "f32", 3, 2, 2, 0.6, temperature=0.25),
         Workload("no_room", 1, 151936, "f32", 2, 2, 2, 0.6, temperature=0.3)]


def in_order():
    """Every workload of ORDER against the oracle, plain and with diagnostics, and a batch with faults."""
    for w in ORDER:
        check_batch(make_batch(w, seed=8, device="cuda"), "traversal")
    b = make_batch(ORDER[0], seed=8, device="cuda")
    args = lambda parent, token: (b.target_logits, b.draft_logits, parent, token, b.u_accept, b.u_bonus)
    want = binding.verify_traversal(*args(b.parent, b.token), temperature=0.25)
    parent = b.parent.reshape(1, -1).repeat(3, 1).contiguous()
    token = b.token.clone()
    parent[0, 2] = 7                     # a trunk node without a parent, branching node below it
    token[1, 1] = -1                     # a trunk node with a token outside the vocabulary
    got = binding.verify_traversal(*args(parent, token), temperature=0.25, node_thr=True, node_w_in=True)
    status = got.status.cpu().numpy()
    assert status[0] == 1 and status[1] == 2 and status[2] == 0, status
    for f in ("accepted_node", "accept_len", "out_tokens", "bonus_token"):
        assert np.array_equal(getattr(want, f)[2].cpu().numpy(), getattr(got, f)[2].cpu().numpy()), f


@pytest.mark.parametrize("blocking", ["0", "1"])
def test_no_kernel_waits_for_a_later_one(blocking):
    """The same results when every kernel has ended before the next one starts."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", "from tests.test_gpu_nodes import in_order; in_order()"], cwd=root,
                       env=dict(os.environ, CUDA_LAUNCH_BLOCKING=blocking), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


def test_two_streams():
    """Calls of two streams at once, a workspace each, share the chip: the results of calls one after the other."""
    batches = [make_batch(Workload("stream", 4, 128256, "bf16", 4, 2, 3, 0.8, temperature=t), seed=i, device="cuda")
               for i, t in enumerate((1.0, 0.4))]
    args = [(b.target_logits, b.draft_logits, b.parent, b.token, b.u_accept, b.u_bonus, b.workload.temperature) for b in batches]
    fields = ("accepted_node", "accept_len", "out_tokens", "bonus_token", "status")
    want = [binding.verify_traversal(*a) for a in args]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in batches]
    ws = [binding.Workspace(a[0].device) for a in args]
    got = [[], []]
    for _ in range(20):
        for i, s in enumerate(streams):
            with torch.cuda.stream(s):
                got[i].append(binding.verify_traversal(*args[i], workspace=ws[i]))
    torch.cuda.synchronize()
    for i in range(2):
        for o in got[i]:
            for f in fields:
                assert np.array_equal(getattr(want[i], f).cpu().numpy(), getattr(o, f).cpu().numpy()), (i, f)
