"""GPU parity of the fused LM head + row statistics (spec_lm_head_stats) with the oracle.

Tolerances: the kernel accumulates in fp32 (tensor cores) and the oracle in fp64, so a
logit may differ by up to ERR = 2^-20 * sum_i |h_i w_vi| (the oracle's abs_bound). row_max
and token_logit within ERR; row_sum within 1e-4 relative plus 2 ERR / T (its
exponents shift by at most ERR / T); row_argmax exact unless the oracle's two largest
logits lie within 2 ERR; bf16 logits within one bf16 rounding of the oracle's plus ERR."""

import numpy as np
import pytest
import torch

from paper_2609_04010_gb300 import binding
from paper_2609_04010_gb300 import workloads as W

from helpers import bf16_dev, dev

pytestmark = pytest.mark.gpu


def gpu_lm(h, w, T, rps, tok=None, want_logits=False):
    r = binding.lm_head_stats(bf16_dev(h), bf16_dev(w), dev(T), rps,
                              tokens=None if tok is None else dev(tok), want_logits=want_logits)
    torch.cuda.synchronize()
    out = {}
    for k, v in r.items():
        out[k] = v.float().cpu().numpy() if k == "logits" else v.cpu().numpy()
    return out


def check(oracle_mod, h, w, T, rps, tok, rows=None):
    g = gpu_lm(h, w, T, rps, tok)
    o = oracle_mod.lm_head_stats(h, w, T, rps, tokens=tok, rows=rows)
    sel = np.arange(h.shape[0]) if rows is None else np.asarray(rows)
    err = 2.0 ** -20 * o["abs_bound"]
    Te = np.array([float(T[r // rps]) if T[r // rps] > 0 else 1.0 for r in sel])
    np.testing.assert_array_less(np.abs(g["row_max"][sel] - o["row_max"]), err + 1e-30)
    np.testing.assert_array_less(np.abs(g["row_sum"][sel] - o["row_sum"]),
                                 o["row_sum"] * (1e-4 + 2 * err / Te))
    srt = np.sort(o["logits"], axis=1)
    gap = srt[:, -1] - srt[:, -2] if o["logits"].shape[1] > 1 else np.full(len(sel), np.inf)
    clear = gap > 2 * err
    np.testing.assert_array_equal(g["row_argmax"][sel][clear], o["row_argmax"][clear])
    if tok is not None:
        ok = ~np.isnan(o["token_logit"])
        np.testing.assert_array_equal(np.isnan(g["token_logit"][sel]), ~ok)
        np.testing.assert_array_less(np.abs(g["token_logit"][sel][ok] - o["token_logit"][ok]), err[ok] + 1e-30)
    return g, o


@pytest.mark.parametrize("R,H,V,rps", [(7, 64, 300, 7), (200, 512, 5000, 16), (130, 1000, 777, 13),
                                       (64, 2048, 32000, 8), (1, 8, 1, 1)])
def test_lm_head_shapes(oracle_mod, R, H, V, rps):
    h, w, T, tok = W.make_lm_inputs(R, H, V, rps, temperature=[1.0, 0.0, 0.7], seed=R + V)
    check(oracle_mod, h, w, T, rps, tok)


def test_lm_head_llama8b_shape_all_rows(oracle_mod):
    # the verify step's rows at the Llama-3-8B head: 8 sequences x 8 positions, 4096 -> 128,256
    h, w, T, tok = W.make_lm_inputs(64, 4096, 128256, 8, seed=5)
    check(oracle_mod, h, w, T, 8, tok)


def test_lm_head_logits_output(oracle_mod):
    h, w, T, tok = W.make_lm_inputs(40, 256, 3000, 8, seed=6)
    g = gpu_lm(h, w, T, 8, tok, want_logits=True)
    o = oracle_mod.lm_head_stats(h, w, T, 8, tokens=tok)
    ref = o["logits"]
    err = 2.0 ** -20 * o["abs_bound"][:, None]
    # within one bf16 rounding (relative 2^-8) of the oracle's logit, plus ERR
    assert np.all(np.abs(g["logits"] - ref) <= np.abs(ref) * 2.0 ** -8 + err + 1e-30)
    srt = np.sort(ref, axis=1)
    clear = srt[:, -1] - srt[:, -2] > 2 * err[:, 0]
    np.testing.assert_array_equal(g["row_argmax"][clear], np.argmax(ref, axis=1)[clear])


def test_lm_head_token_edges_and_bad_rows(oracle_mod):
    h, w, T, tok = W.make_lm_inputs(12, 128, 1000, 4, seed=7)
    tok = tok.copy()
    tok[1] = -1
    tok[2] = 1000
    tok[3] = 999
    h = h.copy()
    h[5, 17] = np.uint16(0x7FC0)  # NaN
    ws = binding.new_workspace(1 << 20)
    r = binding.lm_head_stats(bf16_dev(h), bf16_dev(w), dev(T), 4, tokens=dev(tok), ws=ws)
    torch.cuda.synchronize()
    assert binding.read_device_status(ws)[1] == binding.FLAG_BAD_LOGITS
    g = {k: v.cpu().numpy() for k, v in r.items()}
    assert g["row_argmax"][5] == -1
    assert np.isnan(g["token_logit"][1]) and np.isnan(g["token_logit"][2])
    good = [i for i in range(12) if i != 5]
    o = oracle_mod.lm_head_stats(h, w, T, 4, tokens=tok, rows=good)
    np.testing.assert_array_equal(g["row_argmax"][good], o["row_argmax"])
    assert abs(g["token_logit"][3] - o["token_logit"][good.index(3)]) < 1e-3


# One block per row tile up to 128 rows, two above; vocabularies that leave a tile of one
# 16-row unit, a ragged last unit, tiles of two sizes, and fewer tiles than SMs.
@pytest.mark.parametrize("R,H,V,rps", [(128, 72, 16 * 152 + 1, 16), (129, 72, 31, 16), (256, 136, 40001, 16),
                                       (257, 64, 8192, 1), (700, 200, 77777, 7), (5, 4096, 39000, 1)])
def test_lm_head_tile_plan_edges(oracle_mod, R, H, V, rps):
    h, w, T, tok = W.make_lm_inputs(R, H, V, rps, temperature=[1.0, 0.7], seed=R + V)
    rows = sorted({0, 1, R // 2, min(R, 128) - 1, R - 1, min(R - 1, 255), min(R - 1, 256)})
    check(oracle_mod, h, w, T, rps, tok, rows=rows)


@pytest.mark.parametrize("R,V", [(260, 3000), (130, 2999)])
def test_lm_head_pair_logits_output(oracle_mod, R, V):
    h, w, T, tok = W.make_lm_inputs(R, 256, V, 8, seed=8)
    g = gpu_lm(h, w, T, 8, tok, want_logits=True)
    o = oracle_mod.lm_head_stats(h, w, T, 8, tokens=tok)
    err = 2.0 ** -20 * o["abs_bound"][:, None]
    assert np.all(np.abs(g["logits"] - o["logits"]) <= np.abs(o["logits"]) * 2.0 ** -8 + err + 1e-30)


def test_lm_head_pair_bad_row_and_repeated_maximum():
    # a NaN marks its own row only; equal maxima far apart keep the lowest index
    R, H, V = 200, 64, 50000
    h, w, T, tok = W.make_lm_inputs(R, H, V, 8, seed=9)
    h, w = h.copy(), w.copy()
    h[150, 3] = np.uint16(0x7FC0)
    at = [17, 9000, 49999]
    w[at] = h[20]  # the row itself: its largest logit, three times
    ws = binding.new_workspace(1 << 24)
    r = binding.lm_head_stats(bf16_dev(h), bf16_dev(w), dev(T), 8, tokens=dev(tok), ws=ws)
    torch.cuda.synchronize()
    assert binding.read_device_status(ws)[1] == binding.FLAG_BAD_LOGITS
    arg = r["row_argmax"].cpu().numpy()
    assert arg[150] == -1 and np.all(arg[np.arange(R) != 150] >= 0)
    assert arg[20] == 17


def test_lm_head_pair_wait_runs_out():
    R, H, V = 300, 256, 9000
    h, w, T, tok = W.make_lm_inputs(R, H, V, 8, seed=94)
    out = dict(row_max=torch.empty(R, device="cuda"), row_sum=torch.empty(R, device="cuda"),
               row_argmax=torch.empty(R, dtype=torch.int32, device="cuda"), token_logit=None)
    keep = (bf16_dev(h), bf16_dev(w), dev(T))
    a = binding.lm_head_args(*keep, 8, out)
    ws = binding.new_workspace(binding.lm_head_workspace_size(a))
    binding.test_lm_head_wait_timeout_args(a, ws)
    torch.cuda.synchronize()
    code, flags = binding.read_device_status(ws)
    assert code == 6 and flags & binding.FLAG_TIMEOUT
    binding.lm_head_stats_args(a, ws)
    torch.cuda.synchronize()
    assert binding.read_device_status(ws) == (0, 0)
    ref = keep[0].double() @ keep[1].double().T
    assert torch.equal(out["row_argmax"].long().cpu(), ref.argmax(-1).cpu())


@pytest.mark.parametrize("R", [40, 300])
@pytest.mark.parametrize("T", [1.0, 0.1, 1e-2, 1e-3, 1e-6, 1e-8])
def test_lm_head_sums_at_low_temperatures(R, T):
    # Hidden states and weights are small integers, so every logit is exact and the sums are
    # those of the row's differences: |max| / T reaches 3e10 where the weights' exponents are
    # small. The exponents carry two roundings of at most 104 log2(e) 2^-23 for a weight above
    # 2^-150: 1.8e-5 of it, and less than 1e-5 of a sum that holds the maximum's weight of 1.
    rng = np.random.default_rng(R)
    H, V = 64, 5003
    h = rng.integers(-2, 3, (R, H)).astype(np.float32)
    w = rng.integers(-8, 9, (V, H)).astype(np.float32)
    w[rng.choice(V, 200, replace=False)] = w[0]  # ties
    bits = lambda x: (x.view(np.uint32) >> 16).astype(np.uint16)  # exact in bf16
    temp = np.full((R + 7) // 8, T, np.float32)
    g = gpu_lm(bits(h), bits(w), temp, 8)
    logits = h.astype(np.float64) @ w.T.astype(np.float64)
    top = logits.max(1)
    want = np.exp((logits - top[:, None]) / float(np.float32(T))).sum(1)
    np.testing.assert_array_equal(g["row_max"], top)
    np.testing.assert_array_equal(g["row_argmax"], logits.argmax(1))
    np.testing.assert_allclose(g["row_sum"], want, rtol=1e-5)
