"""fp32 scoring: votes and selection against the oracle at window-row counts around
the 64-row register block, prompts around the 128-key chunk, units of up to and
more than the 16 chunks that pass 2 merges by itself; the multi-layer call against
the per-layer calls bit for bit."""
import pytest
import torch

from paper_2608_08684_gb300 import synth
from tests import gpu_common as C

pytestmark = pytest.mark.gpu
DEV = "cuda"

# (query heads per KV head, window, head dim, prompt length)
SHAPES = [(1, 1, 64, 2), (1, 63, 64, 128), (2, 32, 128, 129), (5, 13, 64, 255), (4, 32, 64, 2048),
          (3, 43, 128, 2049), (8, 32, 64, 513), (7, 9, 128, 3000)]


def _layer(wl, l):
    return tuple(t.to(DEV) for t in C.layer_inputs(wl, l, "cpu"))


@pytest.mark.parametrize("G,w,d,T", SHAPES)
def test_votes_and_selection(lib, G, w, d, T):
    wl = synth.WORKLOADS["tiny"].replace(n_layers=2, batch=1, n_q_heads=2 * G, n_kv_heads=2,
                                         head_dim=d, seq_len=T, window=w,
                                         kv_dist="scaled_sinks", seed=800 + T)
    budgets = [max(w + 1, T // 5), T // 3]
    ins = [_layer(wl, l) for l in range(2)]
    refs = [C.run_compress(lib, wl, budgets[l], *ins[l]) for l in range(2)]
    agree = total = 0
    for h in range(2):
        a, t = C.check_compress_unit(wl, refs[0], *ins[0], 0, h, budgets[0])
        agree, total = agree + a, total + t
    assert agree >= 0.999 * total
    desc = lib.layer_desc(1, 2 * G, 2, d, T, w, wl.pool_kernel, "max", torch.float32)
    k_out = [torch.zeros_like(r["k_out"]) for r in refs]
    v_out = [torch.zeros_like(r["v_out"]) for r in refs]
    idx = [torch.full((2 * r["n"],), -1, dtype=torch.int32, device=DEV) for r in refs]
    tables = lib.CompressTables([x[0] for x in ins], [x[1] for x in ins], [x[2] for x in ins],
                                k_out, v_out, idx)
    ws = torch.empty(lib.ripple_compress_layers_workspace_bytes(desc, 2), dtype=torch.uint8,
                     device=DEV)
    lib.ripple_compress_layers(desc, budgets, tables, ws)
    torch.cuda.synchronize()
    for l, r in enumerate(refs):
        assert torch.equal(idx[l], r["idx"].reshape(-1))
        assert torch.equal(k_out[l], r["k_out"]) and torch.equal(v_out[l], r["v_out"])
