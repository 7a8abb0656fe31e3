"""Sizes where a kernel's split can go wrong, against the oracle: the head's two CTA
sizes, and the seed's foot points on strongly curved tracks."""
import dataclasses

import numpy as np
import pytest

from oracle import seed_oracle as S
from oracle import trackfit_oracle as O
from paper_2609_32479_gb300 import workloads as W
from tests.helpers import FP16_TOL, track_errors

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def T():
    import os
    from paper_2609_32479_gb300 import trackfit
    if not os.path.exists(trackfit.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    trackfit.load()
    return trackfit


def forward(T, model, blob, hits, n_hits):
    dev = torch.device("cuda:0")
    h, n = torch.from_numpy(np.ascontiguousarray(hits)).to(dev), torch.from_numpy(n_hits).to(dev)
    out = torch.full((n.shape[0], 5), -7.0, device=dev)
    with T.Trackfit(model, blob) as tf:
        tf.forward(h, n, out)
        torch.cuda.synchronize()
        return out.cpu().numpy(), tf.device_errors()


@pytest.mark.parametrize("n", [1, 16, 17, 4865])
def test_head_cta_sizes(T, n):
    """16 tracks a CTA up to 32 an SM, 32 above: the paper's 384-wide readout against
    the oracle on the last rows, and each row the same as in a small batch."""
    w = W.workload("paper", n_tracks=n)
    tb = W.gen_tracks(w)
    hits, blob = W.paper_hits(tb, w), W.gen_weights(w.model, 2)
    got, _ = forward(T, w.model, blob, hits, tb.n_hits)
    last = slice(max(0, n - 40), n)
    ref = O.forward(dataclasses.asdict(w.model), blob, hits[last], tb.n_hits[last])
    few, _ = forward(T, w.model, blob, hits[last], tb.n_hits[last])
    np.testing.assert_array_equal(got[last], few)
    if n > 1:   # the bar is relative to a column's RMS over the batch
        assert track_errors(got[last], ref).max() <= FP16_TOL


@pytest.mark.parametrize("n,pt", [(1, (1.0, 2.0)), (33, (0.2, 0.5)), (500, (0.16, 0.4)), (500, (20.0, 500.0))])
def test_seed_foot_points(T, n, pt):
    """Turning angles past the series of the angle (0.64) and very stiff tracks, in
    batches that do not fill a CTA; bars as for the other seed tests."""
    w = W.Workload("t", n, W.workload("small").model, layout="barrel", pt_range=pt, min_hits=5)
    tb = W.gen_tracks(w, seed=5)
    dev = torch.device("cuda:0")
    h, nh = torch.from_numpy(tb.hits).to(dev), torch.from_numpy(tb.n_hits).to(dev)
    sd = torch.empty((n, 5), dtype=torch.float64, device=dev)
    ft = torch.full((n, 12, 3), -9.0, device=dev)
    T.seed(h, nh, 2.0, sd, ft)
    got, feats = sd.cpu().numpy(), ft.cpu().numpy()
    ref = S.seed_from_hits(tb.hits, tb.n_hits, 2.0)
    fref = S.seed_features(ref, tb.hits, tb.n_hits, 2.0)
    np.testing.assert_array_equal(np.isnan(got), np.isnan(ref))
    valid = (np.arange(12)[None, :] < tb.n_hits[:, None]) & ~np.isnan(ref[:, :1])
    assert np.all(feats[~valid] == 0.0)
    fv, rv = feats[valid].astype(np.float64), fref[valid]
    near = (np.abs(np.sinh(rv[:, 0])) < 50.0) & (np.abs(np.sinh(rv[:, 1])) < 50.0)
    assert near.mean() > 0.8
    d = np.abs(fv - rv)[near]
    assert np.max(d[:, :2]) < 2e-6 and np.max(d[:, 2] / np.maximum(np.abs(rv[near, 2]), 1.0)) < 1e-6
