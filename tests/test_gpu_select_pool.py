"""Selection with the gather over prefixes of up to 131072 tokens (and just
beyond, where another kernel takes over): bit-exact against the oracle on shared
votes, at prefix lengths around the edges of a warp's rows, of a CTA and of a
cluster, few and many units, every pooling; ties, equal votes (the radix bucket
does not fit the candidate list), zeros at the threshold (the search starts over
on all bits), and every budget edge."""
import numpy as np
import pytest
import torch

from oracle import ripple_oracle as O
from paper_2608_08684_gb300 import synth
from tests import gpu_common as C

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _run(lib, votes, budget, w, pool, kernel, check):
    units, P = votes.shape
    g = torch.Generator(device=DEV).manual_seed(P + units)
    k = torch.randn(1, units, P + w, 64, dtype=torch.bfloat16, device=DEV, generator=g)
    v = torch.randn(1, units, P + w, 64, dtype=torch.bfloat16, device=DEV, generator=g)
    desc = lib.layer_desc(1, units, units, 64, P + w, w, kernel, pool, torch.bfloat16)
    n = lib.ripple_keep_count(budget, P + w, w)
    k_out = torch.zeros(1, units, n + 1, 64, dtype=torch.bfloat16, device=DEV)
    v_out = torch.zeros_like(k_out)
    idx = torch.full((units * n,), -1, dtype=torch.int32, device=DEV)
    ws = torch.empty(lib.ripple_compress_workspace_bytes(desc), dtype=torch.uint8, device=DEV)
    assert lib.ripple_select_layer(desc, budget, votes.to(DEV), k, v, k_out, v_out, idx, ws) == n
    torch.cuda.synchronize()
    got = idx.view(units, n).cpu().numpy()
    for u in check:
        want = O.select_tokens(O.pool_scores(votes[u].numpy(), kernel, pool), n, P + w, w)
        np.testing.assert_array_equal(got[u], want)
        at = torch.from_numpy(want).long().to(DEV)
        assert torch.equal(k_out[0, u, :n], k[0, u][at])
        assert torch.equal(v_out[0, u, :n], v[0, u][at])
    assert not k_out[0, :, n].any()  # rows past the kept ones are left alone


@pytest.mark.parametrize("P", [1, 31, 33, 255, 257, 4095, 4096, 4097, 8191, 8193, 16385, 32768,
                               32769, 65537, 131071, 131072, 131073, 212992, 212993])
def test_prefix_lengths(lib, P):
    votes = synth.synthetic_votes(900 + P, 2, P, 0)
    _run(lib, votes, 8 + max(1, P // 7), 8, "max", 7, range(2))


@pytest.mark.parametrize("units,P", [(600, 700), (1300, 300), (160, 9000), (620, 8200)])
def test_many_units(lib, units, P):
    votes = synth.synthetic_votes(950 + P, units, P, 200)
    _run(lib, votes, 8 + P // 5, 8, "max", 7, [0, units // 2, units - 1])


@pytest.mark.parametrize("pool,kernel", [("max", 1), ("max", 3), ("max", 5), ("max", 13),
                                         ("max", 31), ("avg", 3), ("avg", 5), ("avg", 31),
                                         ("none", 7)])
@pytest.mark.parametrize("P", [20, 1000, 9001])
def test_pooling(lib, pool, kernel, P):
    votes = synth.synthetic_votes(970 + P, 2, P, 50 if kernel == 5 else 0)
    _run(lib, votes, 8 + P // 3, 8, pool, kernel, range(2))


@pytest.mark.parametrize("P", [500, 9001, 40000])
@pytest.mark.parametrize("kind", ["equal", "zeros", "mostly_zero", "two_values", "spread"])
def test_vote_distributions(lib, kind, P):
    r = np.random.default_rng(P)
    x = {"equal": np.full((2, P), 0.25), "zeros": np.zeros((2, P)),
         "mostly_zero": np.where(r.random((2, P)) < 0.01, r.random((2, P)), 0.0),
         "two_values": np.where(r.random((2, P)) < 0.5, 1.0, 1.0 + 2.0 ** -20),
         "spread": np.exp(30 * (r.random((2, P)) - 0.9))}[kind]
    votes = torch.from_numpy(x.astype(np.float32))
    _run(lib, votes, 8 + P // 3, 8, "max", 3, range(2))


@pytest.mark.parametrize("budget", [0, 8, 9, 8999, 9007, 9008, 9009, 10**7])
def test_budget_edges(lib, budget):
    votes = synth.synthetic_votes(990, 2, 9000, 0)
    _run(lib, votes, budget, 8, "max", 7, range(2))


@pytest.mark.parametrize("n", [1, 2, 191, 192, 193, 2048, 2049])
@pytest.mark.parametrize("base,step", [(1.0, 2.0 ** -18), (1.0, 2.0 ** -22), (2.0 ** -55, 2.0 ** -70),
                                       (511.0, 2.0 ** -12), (600.0, 2.0 ** -10), (1e30, 1e25),
                                       (2.0 ** -60, 2.0 ** -75), (-3.0, 2.0 ** -16)])
def test_threshold_bucket(lib, n, base, step):
    """n keys, half of them in pairs of equal ones, hold the threshold; the others
    lie well above or below: bins of the first round of one key up to more than are
    copied, inside the round's range and on either side of it."""
    P = 9000
    r = np.random.default_rng(n)
    x = np.where(r.random((2, P)) < 0.3, base + abs(base), base - abs(base) / 2).astype(np.float32)
    keep = []
    for u in range(2):
        at = r.choice(P, n, replace=False)
        i = np.arange(n)
        x[u, at] = base + step * np.where(i < n // 2, i // 2, i)
        keep.append(int((x[u] > base + step * n).sum()))
    for u in range(2):  # the threshold at the first, a middle and the last of them
        for k in {keep[u] + 1, keep[u] + (n + 1) // 2, keep[u] + n}:
            _run(lib, torch.from_numpy(x), 8 + k, 8, "none", 1, range(2))


# one 1024-thread CTA a unit; three, five, six and seven CTAs a unit, the last of
# them nearly empty or full; one wave of CTAs and more
@pytest.mark.parametrize("units,P,keep", [
    (160, 16385, 40), (160, 24576, 700), (200, 24577, 30), (153, 32768, 90), (100, 32767, 5000),
    (3, 24576, 100), (40, 40000, 50), (3, 50000, 77), (20, 61440, 3000), (3, 70000, 100),
    (2, 98304, 100), (2, 98305, 100), (3, 114688, 2000), (320, 9000, 300), (320, 9000, 4000),
    (260, 20000, 5000), (300, 32768, 600)])
def test_cta_shapes(lib, units, P, keep):
    votes = synth.synthetic_votes(1000 + P, units, P, 100)
    _run(lib, votes, 8 + keep, 8, "max", 7, [0, units // 2, units - 1])


# many rows a CTA: copied by the gather kernel; around the line between the two
@pytest.mark.parametrize("units,P,keep", [
    (1, 3000, 1031), (1, 3000, 1032), (1, 3000, 2999), (2, 9000, 8000), (1, 131072, 131071),
    (8, 20000, 12000), (3, 70000, 60000), (1, 50000, 50000), (2, 9000, 9000), (8, 700, 700)])
def test_rows_copied_apart(lib, units, P, keep):
    votes = synth.synthetic_votes(1100 + P, units, P, 100)
    _run(lib, votes, 8 + keep, 8, "max", 7, range(units))


def test_layers_of_different_size_copied_apart(lib):
    wl = synth.WORKLOADS["tiny"].replace(n_layers=4, batch=1, n_q_heads=4, n_kv_heads=2,
                                         head_dim=64, seq_len=6000, dtype="bf16", seed=88)
    budgets = [6000, 32, 5000, 700]  # every token, the window only, most, some
    ins = [tuple(t.to(DEV) for t in C.layer_inputs(wl, l, "cpu")) for l in range(4)]
    refs = [C.run_compress(lib, wl, budgets[l], *ins[l], cap_extra=1) for l in range(4)]
    desc = lib.layer_desc(1, 4, 2, 64, 6000, wl.window, wl.pool_kernel, "max", torch.bfloat16)
    k_out = [torch.zeros_like(r["k_out"]) for r in refs]
    v_out = [torch.zeros_like(r["v_out"]) for r in refs]
    idx = [torch.full((2 * r["n"],), -1, dtype=torch.int32, device=DEV) for r in refs]
    tables = lib.CompressTables([x[0] for x in ins], [x[1] for x in ins], [x[2] for x in ins],
                                k_out, v_out, idx)
    ws = torch.empty(lib.ripple_compress_layers_workspace_bytes(desc, 4), dtype=torch.uint8,
                     device=DEV)
    lib.ripple_compress_layers(desc, budgets, tables, ws)
    torch.cuda.synchronize()
    for l, r in enumerate(refs):
        assert torch.equal(idx[l], r["idx"].reshape(-1)), l
        assert torch.equal(k_out[l], r["k_out"]) and torch.equal(v_out[l], r["v_out"]), l
        C.check_compress_unit(wl, r, *ins[l], 0, 1, budgets[l])
