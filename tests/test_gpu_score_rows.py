"""Tensor-core scoring over its range of window rows (G * w from 1 to 256, padded
inside the kernel to 32, 64, 128 or 256 rows) and head dims (64, 128): votes and
selection against the oracle at row counts on, below and above each padding
step, prompts that end on, before and after a key tile, and units of one and
several work items; the multi-layer call against the per-layer calls."""
import numpy as np
import pytest
import torch

from oracle import ripple_oracle as O
from paper_2608_08684_gb300 import synth
from tests import gpu_common as C

pytestmark = pytest.mark.gpu
DEV = "cuda"

# (query heads per KV head, window, head dim, prompt length)
SHAPES = [
    (1, 1, 64, 130), (1, 31, 64, 257), (1, 32, 128, 1153), (3, 11, 128, 300), (2, 32, 64, 1300),
    (4, 16, 128, 2500), (5, 13, 64, 512), (3, 32, 128, 640), (7, 18, 64, 385), (4, 32, 64, 1281),
    (43, 3, 128, 200), (5, 32, 64, 389), (3, 64, 128, 700), (8, 32, 64, 9000), (6, 42, 128, 131),
]


# few units of more than 1024 tiles: items of 64 tiles, more than 16 a unit
LONG = [(8, 32, 64, 140900)]


@pytest.mark.parametrize("G,w,d,T", SHAPES + LONG)
def test_votes_and_selection_match_oracle(lib, G, w, d, T):
    wl = synth.WORKLOADS["tiny"].replace(
        batch=1, n_q_heads=2 * G, n_kv_heads=2, head_dim=d, seq_len=T, window=w, dtype="bf16",
        kv_dist="scaled_sinks", seed=500 + G + w + T)
    budget = max(w + 1, T // 5)
    q, k, v = (t.to(DEV) for t in C.layer_inputs(wl, 0, "cpu"))
    out = C.run_compress(lib, wl, budget, q, k, v, cap_extra=2)
    assert int(out["status"].item()) == 0
    agree = total = 0
    for h in range(2):
        a, t = C.check_compress_unit(wl, out, q, k, v, 0, h, budget)
        agree, total = agree + a, total + t
    assert agree >= 0.999 * total


@pytest.mark.parametrize("G,w,d,T", [SHAPES[4], SHAPES[7], SHAPES[11], SHAPES[13]])
def test_layers_call_equals_per_layer_calls(lib, G, w, d, T):
    # a layer that keeps every token is not scored; the others keep their slots
    wl = synth.WORKLOADS["tiny"].replace(
        n_layers=3, batch=1, n_q_heads=2 * G, n_kv_heads=2, head_dim=d, seq_len=T, window=w,
        dtype="bf16", kv_dist="scaled_sinks", seed=600 + G + w + T)
    budgets = [T // 4, T, T // 9]
    ins = [tuple(t.to(DEV) for t in C.layer_inputs(wl, l, "cpu")) for l in range(3)]
    refs = [C.run_compress(lib, wl, budgets[l], *ins[l]) for l in range(3)]
    desc = lib.layer_desc(1, 2 * G, 2, d, T, w, wl.pool_kernel, "max", torch.bfloat16)
    k_out = [torch.zeros_like(r["k_out"]) for r in refs]
    v_out = [torch.zeros_like(r["v_out"]) for r in refs]
    idx = [torch.full((2 * r["n"],), -1, dtype=torch.int32, device=DEV) for r in refs]
    tables = lib.CompressTables([x[0] for x in ins], [x[1] for x in ins], [x[2] for x in ins],
                                k_out, v_out, idx)
    ws = torch.empty(lib.ripple_compress_layers_workspace_bytes(desc, 3), dtype=torch.uint8,
                     device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    lib.ripple_compress_layers(desc, budgets, tables, ws, dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    for l, r in enumerate(refs):
        assert torch.equal(idx[l], r["idx"].reshape(-1)), l
        assert torch.equal(k_out[l], r["k_out"]) and torch.equal(v_out[l], r["v_out"]), l


# Votes against 64 bits. A logit is a sum of d exact products in fp32, off by at
# most d 2^-24 sum |q_c k_c| (1e-4 in log2 units for these inputs, a few 1e-6 in
# fact, as the terms' errors average out); an exponential adds 2^-22, a normaliser
# the errors of its largest terms, and a vote's rows average again. So no vote is
# off by more than 1e-5 of it (3e-6 seen) and all of them by more than 2e-6 in the
# 2-norm (3e-7 seen, as with fp32 multiply-adds and exp2f in place of the tensor
# cores and ex2).
@pytest.mark.parametrize("G,w,d,T", [SHAPES[i] for i in (1, 2, 4, 5, 7, 9, 11, 12, 13)] + LONG)
def test_votes_to_fp32_precision(lib, G, w, d, T):
    wl = synth.WORKLOADS["tiny"].replace(
        batch=1, n_q_heads=2 * G, n_kv_heads=2, head_dim=d, seq_len=T, window=w, dtype="bf16",
        kv_dist="scaled_sinks", seed=520 + G + w + T)
    q, k, v = (t.to(DEV) for t in C.layer_inputs(wl, 0, "cpu"))
    out = C.run_compress(lib, wl, max(w + 1, T // 5), q, k, v)
    for h in range(2):
        q64, k64, _ = C.unit_f64(wl, q, k, v, 0, h)
        ref = O.window_votes(q64, k64, 1.0 / np.sqrt(d))[0][:T - w]
        err = np.abs(out["scores"][0, h].cpu().numpy().astype(np.float64) - ref)
        assert np.linalg.norm(err) <= 2e-6 * np.linalg.norm(ref)
        assert (err <= 1e-5 * ref).all(), (err / ref).max()
