"""bf16 decode on mma.sync: cache lengths around the edges of a 16-row warp step,
of a 4 KB chunk, of a sub-chunk and of a work item, for every group size and
head dim, against the oracle to the decode precision bound; rows past the
cached ones never count, whatever shared memory holds there. Scores and values
that are not finite, on fp32 caches as well."""
import numpy as np
import pytest
import torch

from oracle import ripple_oracle as O
from paper_2608_08684_gb300 import synth
from tests import gpu_common as C
from tests.test_gpu_decode import Session

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _step(lib, wl, lens0, kc, vc):
    s = Session(lib, wl, range(wl.n_layers), [t.shape[2] for t in kc], lens0, kc, vc)
    q, kn, vn = synth.decode_inputs(wl, 0)
    return s, q, kn, vn, s.step(q, kn, vn)


def _check(wl, lens0, kc, vc, q, kn, vn, got, layers, units):
    G = wl.group
    for i in layers:
        for b, h in units:
            n = lens0[i]
            rk = np.vstack([synth.to_f64(kc[i][b, h, :n]), synth.to_f64(kn[i, b, h])[None]])
            rv = np.vstack([synth.to_f64(vc[i][b, h, :n]), synth.to_f64(vn[i, b, h])[None]])
            ref = O.decode_attention(synth.to_f64(q[i, b, h * G:(h + 1) * G]), rk, rv,
                                     1.0 / np.sqrt(wl.head_dim))
            C.assert_decode_close(got[i, b, h * G:(h + 1) * G], ref)


# with the new token: n + 1 rows
LENS = [0, 1, 14, 15, 16, 30, 31, 32, 126, 127, 128, 159, 254, 255, 256, 257, 511, 4097]


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("G", [1, 2, 4, 8])
def test_lengths_around_every_edge(lib, G, d):
    wl = synth.WORKLOADS["tiny"].replace(n_layers=len(LENS), batch=1, n_q_heads=G, n_kv_heads=1,
                                         head_dim=d, dtype="bf16", kv_dist="scaled_sinks",
                                         seed=700 + G + d)
    kc, vc = zip(*[synth.decode_caches(wl, i, n + 3) for i, n in enumerate(LENS)])
    s, q, kn, vn, got = _step(lib, wl, LENS, kc, vc)
    assert int(s.status.item()) == 0
    _check(wl, LENS, kc, vc, q, kn, vn, got, range(len(LENS)), [(0, 0)])
    for i, n in enumerate(LENS):
        assert torch.equal(s.k[i][:, :, n].cpu(), kn[i]) and torch.equal(s.v[i][:, :, n].cpu(), vn[i])
        assert torch.equal(s.k[i][:, :, n + 1:].cpu(), kc[i][:, :, n + 1:])


@pytest.mark.parametrize("G,d", [(4, 128), (8, 64)])
def test_rows_past_the_cache_never_count(lib, G, d):
    # more groups than CTAs, so that every CTA stages groups of the long layer,
    # whose values are infinite, before groups of the short ones
    wl = synth.WORKLOADS["tiny"].replace(n_layers=3, batch=80, n_q_heads=4 * G, n_kv_heads=4,
                                         head_dim=d, dtype="bf16", seed=750 + G)
    lens0 = [300, 5, 17]
    kc, vc = zip(*[synth.decode_caches(wl, i, n + 2) for i, n in enumerate(lens0)])
    vc[0].fill_(float("inf"))
    kc[0][:, :, 1:] = float("nan")
    s, q, kn, vn, got = _step(lib, wl, lens0, kc, vc)
    assert int(s.status.item()) == 0
    assert np.isfinite(got[1:]).all()
    _check(wl, lens0, kc, vc, q, kn, vn, got, [1, 2], [(0, 0), (41, 2), (79, 3)])


@pytest.mark.parametrize("G,d,dtype", [(1, 64, "bf16"), (2, 128, "bf16"), (4, 128, "bf16"),
                                       (8, 64, "bf16"), (8, 128, "bf16"), (1, 64, "f32"),
                                       (4, 128, "f32"), (8, 64, "f32")])
def test_infinite_values_stay_infinite(lib, G, d, dtype):
    # A probability is positive, so a column that holds an infinite value has an
    # infinite output, whatever parts the probability is split into (1, of one
    # bf16 part, and the largest of a row included); the other columns stay as
    # they are.
    wl = synth.WORKLOADS["tiny"].replace(n_layers=4, batch=1, n_q_heads=2 * G, n_kv_heads=2,
                                         head_dim=d, dtype=dtype, seed=760 + G + d)
    lens0 = [1, 40, 300, 5000]
    kc, vc = zip(*[synth.decode_caches(wl, i, n + 2) for i, n in enumerate(lens0)])
    for i, n in enumerate(lens0):
        vc[i][0, 0, 0, 3] = float("inf")
        vc[i][0, 0, n // 2, d - 1] = -float("inf")
        vc[i][0, 1, n - 1, d // 2] = float("inf")
        vc[i][0, 1, : n // 2 + 1, 7] = -float("inf")
    s, q, kn, vn, got = _step(lib, wl, lens0, kc, vc)
    assert int(s.status.item()) == 0
    bad = np.zeros((2, d), np.float64)
    bad[0, 3], bad[0, d - 1], bad[1, d // 2], bad[1, 7] = np.inf, -np.inf, np.inf, -np.inf
    for i in range(len(lens0)):
        for h in range(2):
            at = np.isinf(bad[h])
            o = got[i, 0, h * G:(h + 1) * G]
            assert (o[:, at] == bad[h][at]).all(), (i, h, o[:, at])
            vc[i][0, h][:, at] = 0.0
    _check(wl, lens0, kc, vc, q, kn, _zeroed(vn, bad), _zero_cols(got, bad, G),
           range(len(lens0)), [(0, 0), (0, 1)])


def _zeroed(vn, bad):
    vn = vn.clone()
    for h in range(2):
        vn[:, 0, h, np.isinf(bad[h])] = 0.0
    return vn


def _zero_cols(got, bad, G):
    got = got.copy()
    for h in range(2):
        got[:, 0, h * G:(h + 1) * G, np.isinf(bad[h])] = 0.0
    return got


@pytest.mark.parametrize("G,d,dtype", [(1, 64, "bf16"), (4, 128, "bf16"), (8, 64, "bf16"),
                                       (8, 128, "bf16"), (2, 64, "f32"), (8, 128, "f32")])
def test_scores_that_are_not_finite_or_huge(lib, G, d, dtype):
    # Three groups, in caches of which most end inside a sub-chunk: a NaN in a key
    # makes the group's outputs NaN (a row counts for nothing by its place past the
    # cached ones, not by its score); keys whose score is -infinity, a first row and
    # a whole run of them, count for nothing; a score so large that its rounding
    # alone is many powers of two takes all the weight.
    wl = synth.WORKLOADS["tiny"].replace(n_layers=5, batch=1, n_q_heads=3 * G, n_kv_heads=3,
                                         head_dim=d, dtype=dtype, seed=790 + G + d)
    lens0 = [2, 40, 256, 700, 5000]
    kc, vc = zip(*[synth.decode_caches(wl, i, n + 2) for i, n in enumerate(lens0)])
    s0 = Session(lib, wl, range(5), [t.shape[2] for t in kc], lens0, kc, vc)
    q, kn, vn = synth.decode_inputs(wl, 0)
    q[:, :, G:2 * G, 5] = q[:, :, G:2 * G, 5].abs() + 1
    q[:, :, 2 * G:, 9] = 2.0
    kept = [list(range(n)) for n in lens0]
    for i, n in enumerate(lens0):
        kc[i][0, 0, n - 1, 3] = float("nan")
        gone = range(0, 1) if n == 2 else range(0, n // 2)
        kc[i][0, 1, list(gone), 5] = -float("inf")
        kept[i] = [r for r in range(n) if r not in gone]
        kc[i][0, 2, n // 2, 9] = 1e30
    s0.k = [t.to(DEV) for t in kc]
    s0.tables = lib.DecodeTables(s0.k, s0.v)
    got = s0.step(q, kn, vn)
    assert int(s0.status.item()) == 0
    for i, n in enumerate(lens0):
        assert np.isnan(got[i, 0, :G]).all(), i
        rows = kept[i]
        rk = np.vstack([synth.to_f64(kc[i][0, 1, rows]), synth.to_f64(kn[i, 0, 1])[None]])
        rv = np.vstack([synth.to_f64(vc[i][0, 1, rows]), synth.to_f64(vn[i, 0, 1])[None]])
        ref = O.decode_attention(synth.to_f64(q[i, 0, G:2 * G]), rk, rv, 1.0 / np.sqrt(d))
        C.assert_decode_close(got[i, 0, G:2 * G], ref)
        np.testing.assert_array_equal(
            got[i, 0, 2 * G:], np.tile(vc[i][0, 2, n // 2].float().numpy(), (G, 1)))
