"""Host threads that issue calls of different sizes at the same time, each on its own stream
and workspace. A kernel's limit of dynamic shared memory belongs to the function: no call may
lower it between another thread's setting and its launch, which would then be refused. Every
call must be accepted and give what it gave alone."""

import threading

import numpy as np
import pytest
import torch

from paper_2609_04010_gb300 import binding
from paper_2609_04010_gb300 import workloads as W

from helpers import attn_tensors, dev, logits_dev

pytestmark = pytest.mark.gpu

CALLS = 3000


def draw_call(vocab, max_top_k, seed):
    """One drafter row of an odd vocabulary (unaligned rows), filtered where max_top_k > 0."""
    inp = W.make_accept_inputs(1, 1, vocab, "f32", 3.0, 1.0, [1.0], seed=seed)
    dl, T, u = logits_dev(inp.drafter_logits), dev(inp.temperature), dev(inp.uniforms)
    tok = torch.empty(1, 1, dtype=torch.int32, device="cuda")
    q = torch.empty(1, 1, dtype=torch.float32, device="cuda")
    d = binding.draft_args(dl, T, u, tok, q)
    keep = [dl, T, u]
    f = None
    if max_top_k:
        k, p = dev(np.full(1, max_top_k, np.int32)), dev(np.full(1, 0.9, np.float32))
        f = binding.filter_args(k, p, 1, max_top_k)
        keep += [k, p]
    ws = binding.new_workspace(binding.draft_workspace_size(d, f))
    return (lambda s: binding.sample_block_args(d, f, ws, s)), [tok, q], keep


def attention_call(batch, path, seed):
    inp = W.make_attn_inputs(batch, 1, 8, 2, 128, 16, (20, 60), True, seed=seed)
    q, k, v, pt, kl = attn_tensors(inp)
    out = torch.empty_like(q)
    a = binding.attn_args(q, k, v, pt, kl, out, None, path=path)
    ws = binding.new_workspace(binding.workspace_size(a, None))
    return (lambda s: binding.verify_attention_args(a, ws, s)), [out], [q, k, v, pt, kl]


CASES = {
    "draft": lambda: (draw_call(151937, 0, 1), draw_call(300001, 0, 2)),
    "filtered": lambda: (draw_call(50001, 1, 3), draw_call(50001, 1024, 4)),
    "attention_small_groups": lambda: (attention_call(1, binding.ATTN_AUTO, 5),
                                       attention_call(1024, binding.ATTN_AUTO, 6)),
    "attention_row_tiles": lambda: (attention_call(1, binding.ATTN_TENSOR_CORES, 7),
                                    attention_call(1024, binding.ATTN_TENSOR_CORES, 8)),
    "attention_keys_on_lanes": lambda: (attention_call(1, binding.ATTN_TENSOR_CORES_KEYS_ON_LANES, 9),
                                        attention_call(200, binding.ATTN_TENSOR_CORES_KEYS_ON_LANES, 10)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_calls_of_two_sizes_at_once(name):
    calls = CASES[name]()
    alone = []
    for call, outs, _ in calls:
        call(None)
        torch.cuda.synchronize()
        alone.append([o.clone() for o in outs])
    errors = []
    gate = threading.Barrier(len(calls))

    def work(call):
        s = torch.cuda.Stream()
        try:
            gate.wait()
            for i in range(CALLS):
                call(s)
                if i % 256 == 255:
                    s.synchronize()
            s.synchronize()
        except Exception as e:  # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(c[0],)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for (_, outs, _), want in zip(calls, alone):
        for o, w in zip(outs, want):
            assert torch.equal(o, w)
