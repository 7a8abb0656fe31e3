"""The tile kernels of the paper's model and the Transformer beyond small fp16 batches: bf16
operands, packed input, many tiles a CTA (the metadata buffers in turn) and the second chunk
of the Fourier workspace, with tracks of an invalid hit count among the compared ones."""
import dataclasses

import numpy as np
import pytest

from oracle import trackfit_oracle as O
from paper_2609_32479_gb300 import workloads as W
from tests.helpers import FP16_TOL, track_errors
from tests.test_gpu_kernels import T, TILE_SHAPES, forward, tile_case   # noqa: F401 (T: a fixture)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# bf16 keeps 8 bits of an operand, fp16 11: eight times the rounding error at the same places
BF16_TOL = 8 * FP16_TOL
PAPER = (W.TOPOLOGY_CONCAT, 15, 2, 0, 192, 24)
TRANSFORMER = (W.TOPOLOGY_ATTENTION, 15, 3, 4, 288, 24)


@pytest.mark.parametrize("shape", TILE_SHAPES)
def test_tile_kernel_shapes_bf16(T, shape):
    m, h, nh = tile_case(*shape)
    m = m.with_(precision=W.PRECISION_BF16)
    blob = W.gen_weights(m, 2)
    few = np.r_[0:min(len(nh), 150), max(150, len(nh) - 50):len(nh)]
    bad = [5, len(nh) - 3] if len(nh) > 8 else []
    nh[bad] = [0, m.max_hits + 1][:len(bad)]
    got, (status, n_bad) = forward(T, m, blob, h, nh)
    ref = O.forward(dataclasses.asdict(m), blob, h[few], nh[few])
    assert n_bad == len(bad) and status == (T.ERR_BAD_HITS if bad else T.OK)
    np.testing.assert_array_equal(np.isnan(got[few]), np.isnan(ref))
    ok = ~np.isnan(ref[:, 0])
    if len(nh) > 1:
        assert track_errors(got[few][ok], ref[ok]).max() <= BF16_TOL
    else:   # one track has no column RMS to measure by: relative to its largest parameter
        assert np.abs(got - ref).max() <= BF16_TOL * np.abs(ref).max()


@pytest.mark.parametrize("prec", [W.PRECISION_FP16, W.PRECISION_BF16])
@pytest.mark.parametrize("model", [PAPER, TRANSFORMER], ids=["paper", "transformer"])
def test_many_tiles_and_a_second_chunk(T, model, prec):
    """140,000 tracks: 90 tiles a CTA, past the workspace's chunk (132,096 and 136,192 tracks):
    the same bits as the 4,000 tracks that they repeat, which are held to the oracle."""
    n, unique = 140000, 4000
    m, h, nh = tile_case(*model, unique)
    m = m.with_(precision=prec)
    blob = W.gen_weights(m, 2)
    nh[[7, 3990]] = [0, m.max_hits + 1]
    want, (_, n_bad) = forward(T, m, blob, h, nh)
    assert n_bad == 2
    few = np.r_[0:100, 3950:4000]
    ref = O.forward(dataclasses.asdict(m), blob, h[few], nh[few])
    np.testing.assert_array_equal(np.isnan(want[few]), np.isnan(ref))
    ok = ~np.isnan(ref[:, 0])
    assert track_errors(want[few][ok], ref[ok]).max() <= (FP16_TOL if prec == W.PRECISION_FP16 else BF16_TOL)
    got, (status, n_bad) = forward(T, m, blob, np.resize(h, (n, *h.shape[1:])), np.resize(nh, n))
    assert status == T.ERR_BAD_HITS and n_bad == 2 * n // unique
    np.testing.assert_array_equal(got, np.resize(want, (n, 5)))


@pytest.mark.parametrize("prec", [W.PRECISION_FP16, W.PRECISION_BF16])
@pytest.mark.parametrize("model", [PAPER, TRANSFORMER], ids=["paper", "transformer"])
def test_packed_input_is_the_padded_one(T, model, prec):
    m, h, nh = tile_case(*model, 9000)
    m = m.with_(precision=prec)
    blob = W.gen_weights(m, 2)
    want, _ = forward(T, m, blob, h, nh)
    dev = torch.device("cuda:0")
    rows = h[np.arange(h.shape[1])[None, :] < nh[:, None]]
    offs = np.concatenate([[0], np.cumsum(nh)]).astype(np.int64)
    out = torch.full((9000, 5), -7.0, device=dev)
    with T.Trackfit(m, blob) as tf:
        tf.forward_packed(torch.from_numpy(np.ascontiguousarray(rows)).to(dev), torch.from_numpy(offs).to(dev), out)
        torch.cuda.synchronize()
        assert tf.device_errors() == (T.OK, 0)
    np.testing.assert_array_equal(out.cpu().numpy(), want)
