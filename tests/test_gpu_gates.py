"""Gates of the fused kernels at the ends of their arguments: a gate that is shut lets
nothing through however large the value beside it, and a gate whose argument is not a
number shows in every result.  Each expectation is exact: sigma of an argument below -150
is below 1e-64, which no product with a finite fp32 value brings back."""
import numpy as np
import pytest

from paper_2609_32479_gb300 import workloads as W
from tests.test_gpu_kernels import T, forward, ragged, tile_case   # noqa: F401 (T: a fixture)

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")

MERGE128, MERGE256, CONCAT, ATTN = "merge128", "merge256", "concat", "attention"


def case(kind, n=300):
    if kind in (MERGE128, MERGE256):
        D = 128 if kind == MERGE128 else 256
        m = W.ModelConfig(max_hits=12, d_model=D, d_hidden=3 * D // 2, n_layers=2, precision=W.PRECISION_FP16)
        h, nh = ragged(m, n)
    else:
        topo, width = (W.TOPOLOGY_CONCAT, 192) if kind == CONCAT else (W.TOPOLOGY_ATTENTION, 288)
        m, h, nh = tile_case(topo, 5, 2, 4, width, 12, n)
    return m, W.split_weights(m, W.gen_weights(m, 2)), h, nh


def run(T, m, w, h, nh):
    out, (status, _) = forward(T, m, W.join_weights(m, w), h, nh)
    assert status == T.OK
    return out


@pytest.mark.parametrize("kind", [MERGE128, MERGE256])
def test_a_shut_output_gate_adds_nothing(T, kind):
    m, w, h, nh = case(kind)
    ch = [3, m.d_model - 1]
    w["layer0.b_in"][4 * m.d_hidden + np.array(ch)] = -200.0
    w["layer0.b_m"][ch] = 0.0
    want = run(T, m, w, h, nh)
    w["layer0.b_m"][ch] = 1e20
    np.testing.assert_array_equal(run(T, m, w, h, nh), want)


@pytest.mark.parametrize("kind", [MERGE128, MERGE256, CONCAT])
@pytest.mark.parametrize("z", [-60.0, -87.6, -95.0, -200.0])
def test_a_shut_update_gate_keeps_the_state(T, kind, z):
    """z towards 0 on both sides of where e^-z overflows: the state stays what it was (the
    candidate's bias 1e15 times 8.8e-27 is below the smallest fp16), never a NaN."""
    m, w, h, nh = case(kind)
    H = m.d_hidden
    for g in (0, 2 * H):   # forward, reverse
        w["layer0.w_in"][g + 5] = 0.0
        w["layer0.b_in"][g + 5] = z
        w["layer0.b_in"][g + H + 5] = 0.0
    want = run(T, m, w, h, nh)
    assert np.isfinite(want).all()
    for g in (0, 2 * H):
        w["layer0.b_in"][g + H + 5] = 1e15
    np.testing.assert_array_equal(run(T, m, w, h, nh), want)


def test_silu_of_a_large_negative_value_is_zero(T):
    m, w, h, nh = case(ATTN)
    w["layer1.b1"][7] = -1e4
    want = run(T, m, w, h, nh)
    w["layer1.b1"][7] = -1e30
    np.testing.assert_array_equal(run(T, m, w, h, nh), want)


@pytest.mark.parametrize("kind,row", [(MERGE128, "z"), (MERGE128, "gate"), (MERGE256, "z"), (MERGE256, "gate"),
                                      (CONCAT, "z")])
def test_a_gate_argument_that_is_not_a_number_shows(T, kind, row):
    m, w, h, nh = case(kind)
    w["layer0.b_in"][5 if row == "z" else 4 * m.d_hidden + 5] = np.nan
    assert not np.isfinite(run(T, m, w, h, nh)).any()


@pytest.mark.parametrize("kind,n", [(MERGE128, 300), (MERGE128, 3000), (MERGE256, 300), (MERGE256, 3000)])
def test_a_track_with_infinite_hits_leaves_the_others_alone(T, kind, n):
    """One-slab tiles and pairs of tiles at d_model 128, one tile at 256: a track whose valid
    hits hold infinities or NaN spoils its own row only, bit for bit."""
    m, w, h, nh = case(kind, n)
    want = run(T, m, w, h, nh)
    h[17, : nh[17]] = np.inf
    h[140, 0, 2] = np.nan
    got = run(T, m, w, h, nh)
    assert not np.isfinite(got[[17, 140]]).any()
    others = np.setdiff1d(np.arange(n), [17, 140])
    np.testing.assert_array_equal(got[others], want[others])
