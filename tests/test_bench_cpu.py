"""bench.py's reference arm (the CPU oracle timed on bounded samples) runs without
a GPU and prints one JSON line in the contract's shape."""
import json
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reference_arm_prints_one_contract_line():
    cmd = [sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--steps", "1", "--warmup", "0",
           "--workload", "medium", "--n-tracks", "4096"]
    r = subprocess.run(cmd, cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [l for l in r.stdout.splitlines() if l.strip().startswith("{")]
    assert len(lines) == 1
    d = json.loads(lines[0])
    assert d["impl"] == "reference"
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better",
              "scaling", "vs_baseline", "dtype", "data", "config", "cpu_baseline", "e2e"):
        assert k in d, k
    assert d["value"] > 0 and d["unit"] == "tracks/s" and d["higher_is_better"] is True
    assert d["config"]["workload"] == "medium"
    cb = d["cpu_baseline"]
    assert cb["kind"] == "oracle" and cb["cores"] >= 1 and cb["value"] == d["value"]
    assert d["e2e"] == {"value": d["value"], "unit": "tracks/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}


def test_oracle_pool_matches_one_process():
    """The CPU baseline's process pool (the oracle on every core, tracks in chunks)
    returns what one call of the oracle returns on the same tracks, in order: equal
    up to the fp64 rounding that a matrix product's blocking over a different batch
    size changes (1e-13 relative measured; 1e-11 allowed)."""
    import dataclasses
    import numpy as np
    sys.path.insert(0, ROOT)
    import bench
    from oracle import trackfit_oracle as O
    from paper_2609_32479_gb300 import workloads as W
    w = W.workload("small", n_tracks=150)
    tb = W.gen_tracks(w)
    blob = W.gen_weights(w.model, w.weight_seed)
    ref = O.forward(dataclasses.asdict(w.model), blob, tb.hits, tb.n_hits)
    pool = bench.OraclePool(w)
    try:
        got = pool.forward(tb.hits, tb.n_hits, chunk=32)
    finally:
        pool.close()
    assert pool.workers >= 1
    assert got.shape == ref.shape
    np.testing.assert_allclose(got, ref, rtol=1e-11, atol=1e-13)


def test_kernel_names():
    """What the bench line calls the timed kernel: the fused fp32 encoder only for the models
    that it takes, and the profile's digest covers every source of the wide kernel."""
    sys.path.insert(0, ROOT)
    import bench
    from paper_2609_32479_gb300 import workloads as W
    tiny, large = W.workload("tiny").model, W.workload("large").model
    assert bench.kernel_name("simt-fp32", tiny) == "encoder_fp32_kernel"
    for m, path in ((tiny.with_(precision=W.PRECISION_BF16), "simt-bf16"), (large.with_(precision=W.PRECISION_FP32), "simt-fp32"),
                    (W.workload("paper").model.with_(precision=W.PRECISION_FP32), "simt-fp32")):
        assert bench.kernel_name(path, m) == "CUDA-core encoder, a launch a step"
    assert bench.kernel_name("tcgen05-bf16", W.workload("medium").model) == "tc_pair_kernel"
    assert bench.kernel_name("tcgen05-bf16", large) == "tc_forward_kernel"
    assert bench.kernel_name("tcgen05-rows-fp16", W.workload("paper").model) == "concat_kernel"
    assert {os.path.basename(f) for f in bench.KERNEL_SRC} == {"tc_forward.cu", "tc_epilogue.cuh", "sm100_ptx.cuh"}
