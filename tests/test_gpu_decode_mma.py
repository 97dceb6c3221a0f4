"""bf16 decode on mma.sync: cache lengths around the edges of a 16-row warp step,
of a 4 KB chunk, of a sub-chunk and of a work item, for every group size and
head dim, against the oracle to the decode precision bound; rows past the
cached ones never count, whatever shared memory holds there."""
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
