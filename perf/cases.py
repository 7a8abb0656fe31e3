"""What the framework is timed on: the track fits that its users run.

A case is one call pattern of a reconstruction program: a loaded encoder, a batch
of tracks, and one pass through the public entry points.  The encoders are the
ones that this repository configures (workloads.py): the fp32 shapes `tiny` and
`small`, the 16-bit gated-merge shapes `medium`, `large` and the length sweep, the
paper's concatenation model and its Transformer, and the analytic seed.  Batches
go from one collision event (tens to hundreds of tracks, where the latency of the
call counts) to a million tracks of an offline pass.

Keys of a case
  kind    "merge" | "concat" | "attention" (an encoder) or "seed" (the seed alone)
  layout  the synthetic detector: "barrel", "sweep" (as many layers as hits) or
          "endcap" (barrel and disks, 8-20 hits on a track)
  call    "forward"   padded hits on the device, the median parameters
          "export"    the same with the quantiles and the pooled vector
          "packed"    unpadded hits with offsets
          "host"      pinned host buffers in and out (copies included)
          "noalloc"   the entry point that allocates nothing
          "chain"     seed, features written into the hits, encoder, decode
          "seed"      seed and residual features
  hits, d_model, layers, precision, heads, drop, tracks   sizes
"""
import math

import numpy as np
import torch

from paper_2609_32479_gb300 import trackfit
from paper_2609_32479_gb300 import workloads as W

FP32, BF16, FP16 = W.PRECISION_FP32, W.PRECISION_BF16, W.PRECISION_FP16
POOL = 4096            # generated tracks; a batch is drawn from them with random rotations and reflections
MOST_FLOPS = 1.6e14    # the largest listed case's work


def _case(name, kind, call, tracks, hits, d_model, layers, precision, layout="endcap", drop=0, heads=4):
    c = dict(kind=kind, call=call, tracks=tracks, hits=hits, d_model=d_model, layers=layers, precision=precision,
             layout=layout, drop=drop, heads=heads)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest call: a unit's worth of tracks on the fp32 encoder, all latency
        _case("tiny_fp32", "merge", "forward", 256, 10, 32, 2, FP32, "barrel"),
        # an ordinary fp32 batch with dropped hits
        _case("small_fp32", "merge", "forward", 16384, 12, 64, 4, FP32, "barrel", drop=3),
        # one collision event through the 16-bit encoder, quantiles exported: latency
        _case("event_bf16", "merge", "export", 101, 24, 128, 6, BF16),
        # an ordinary batch of the 16-bit encoder, padded to 24 hits
        _case("medium_bf16", "merge", "forward", 262144, 24, 128, 6, BF16),
        # full-length long tracks with the quantiles and pooled vectors exported
        _case("long_tracks_bf16", "merge", "export", 4096, 64, 128, 6, BF16, "sweep"),
        # the wide encoder on packed input in fp16, an odd batch
        _case("wide_packed_fp16", "merge", "packed", 20011, 24, 256, 8, FP16),
        # the wide encoder from and to pinned host memory, as an offline job calls it
        _case("wide_host_bf16", "merge", "host", 300001, 24, 256, 8, BF16),
        # the paper's model at the paper's batch: seed, encoder, decode
        _case("paper_chain_fp16", "concat", "chain", 131072, 24, 128, 2, FP16),
        # the paper's model on one event's tracks, packed
        _case("paper_event_fp16", "concat", "packed", 997, 24, 128, 2, FP16),
        # the Transformer at the paper's batch
        _case("transformer_fp16", "attention", "forward", 131072, 24, 128, 3, FP16),
        # the seed with its residual features over an offline batch
        _case("seed_features", "seed", "seed", 524288, 24, 128, 1, FP32),
        # the largest: a million tracks through the wide encoder, device resident
        _case("large_bf16", "merge", "forward", 1048576, 24, 256, 8, BF16),
    ]


def draw(rng):
    """One more case of the ranges above: sizes over their logarithm, odd ones among them."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    family = rng.choice(["fp32", "merge", "merge", "concat", "attention", "seed"])
    layout = rng.choice(["endcap", "sweep"])
    hits = 24 if layout == "endcap" else log_int(8, 64)
    drop = 0 if layout == "endcap" else rng.randint(0, hits // 2)
    heads, layers, d = 4, 1, 128
    if family == "fp32":
        kind, prec, d, layers = "merge", FP32, rng.choice([32, 64, 128]), rng.randint(2, 4)
        call, top = rng.choice(["forward", "export", "packed", "noalloc"]), 65536
    elif family == "merge":
        kind, prec, d, layers = "merge", rng.choice([BF16, FP16]), rng.choice([128, 256]), rng.randint(2, 8)
        call, top = rng.choice(["forward", "export", "packed", "host"]), 1048576
    elif family == "concat":
        kind, prec, layers = "concat", FP16, rng.randint(1, 3)
        call, top = rng.choice(["forward", "export", "packed", "chain"]), 262144
    elif family == "attention":
        kind, prec, layers, heads = "attention", FP16, rng.randint(1, 4), rng.choice([2, 4, 8])
        call, top = rng.choice(["forward", "export", "packed", "chain"]), 262144
    else:
        kind, call, prec, top = "seed", "seed", FP32, 1048576
    c = _case(None, kind, call, log_int(32, top), hits, d, layers, prec, layout, drop, heads)
    budget = 2e12 if family == "fp32" else MOST_FLOPS / 2
    while work(c)["flops"] > budget or c["tracks"] * hits > 25165824:
        c["tracks"] = max(32, c["tracks"] * 2 // 3)
    return c


def _workload(case):
    layout = {"endcap": "barrel_endcap"}.get(case["layout"], case["layout"])
    T, D = case["hits"], case["d_model"]
    if case["kind"] in ("concat", "attention"):
        base = W.WORKLOADS["paper" if case["kind"] == "concat" else "transformer"].model
        m = base.with_(max_hits=T, n_layers=case["layers"], precision=case["precision"], n_heads=case["heads"])
    else:
        m = W.ModelConfig(max_hits=T, d_model=D, d_hidden=3 * D // 2, n_layers=case["layers"],
                          precision=case["precision"])
    return W.Workload("case", POOL, m, layout=layout, pt_range=(1.0, 100.0), drop_max=case["drop"],
                      n_barrel=T if layout == "sweep" else 10,
                      min_hits=8 if layout == "barrel_endcap" else min(T, 10) if layout == "barrel" else T)


def _inputs(case, seed):
    """hits [B, T, F] and n_hits [B] on the GPU, and the weight blob (numpy)."""
    w = _workload(case)
    B = case["tracks"]
    tb = W.gen_tracks(w, n_tracks=min(B, POOL), seed=seed)
    rows = W.paper_hits(tb, w) if w.model.n_features == 15 else tb.hits
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    pick = torch.randint(tb.n_hits.size, (B,), generator=g, device=dev)
    a = (torch.rand(B, generator=g, device=dev) * 2 - 1) * math.pi
    flip = torch.where(torch.rand(B, generator=g, device=dev) < 0.5, -1.0, 1.0)
    n = torch.from_numpy(tb.n_hits).to(dev)[pick]
    h = torch.from_numpy(rows).to(dev)[pick]
    # each track turned about the beam line and, for half of them, mirrored in z
    ca, sa = torch.cos(a)[:, None], torch.sin(a)[:, None]
    x, y = h[..., 0].clone(), h[..., 1].clone()
    h[..., 0] = x * ca - y * sa
    h[..., 1] = x * sa + y * ca
    h[..., 2] *= flip[:, None]
    h[..., 4] = torch.atan2(h[..., 1], h[..., 0])
    if w.model.n_features == 15:
        h[..., 5] = torch.where(flip[:, None] < 0, math.pi - h[..., 5], h[..., 5])
        h[..., 6] *= flip[:, None]
        h[..., 8], h[..., 9] = torch.cos(h[..., 4]), torch.sin(h[..., 4])
    t = torch.arange(case["hits"], device=dev)[None, :]
    h = torch.where((t < n[:, None])[..., None], h, torch.zeros((), device=dev)).contiguous()
    return w, h, n, W.gen_weights(w.model, seed + 1)


def prepare(case, seed):
    w, h, n, blob = _inputs(case, seed)
    m, B, call = w.model, case["tracks"], case["call"]
    dev = h.device
    st = dict(call=call, model=m, b_field=w.b_field, n=n)
    if case["kind"] == "seed":
        st.update(hits=h, seed=torch.empty((B, 5), dtype=torch.float64, device=dev),
                  features=torch.empty((B, m.max_hits, 3), dtype=torch.float32, device=dev))
        return st
    if call == "noalloc":
        st["weights"] = torch.from_numpy(blob).to(dev)
    else:
        st["fit"] = trackfit.Trackfit(m, blob)
    if call == "host":
        st["hits"] = torch.empty(h.shape, pin_memory=True).copy_(h).numpy()
        st["n"] = torch.empty(B, dtype=torch.int32, pin_memory=True).copy_(n).numpy()
        st["out"] = torch.empty((B, 5), pin_memory=True).numpy()
        return st
    st["out"] = torch.empty((B, 5), device=dev)
    if call == "packed":
        valid = torch.arange(m.max_hits, device=dev)[None, :] < n[:, None]
        st["hits"] = h[valid].contiguous()
        st["offsets"] = torch.cat([torch.zeros(1, dtype=torch.int64, device=dev), n.to(torch.int64).cumsum(0)])
        return st
    st["hits"] = h
    if call == "export":
        st["quantiles"] = torch.empty((B, 5, m.n_quantiles), device=dev)
        st["pooled"] = torch.empty((B, m.pooled_dim), device=dev)
    if call == "chain":
        st["seed"] = torch.empty((B, 5), dtype=torch.float64, device=dev)
        st["params"] = torch.empty((B, 5), device=dev)
    return st


def run(st):
    call = st["call"]
    if call == "seed":
        trackfit.seed(st["hits"], st["n"], st["b_field"], st["seed"], st["features"])
        return {"seed": st["seed"], "features": st["features"]}
    out = st["out"]
    if call == "noalloc":
        trackfit.forward_noalloc(st["model"], st["weights"], st["hits"], st["n"], out)
        return {"out": out}
    fit = st["fit"]
    if call == "host":
        fit.forward_host(st["hits"], st["n"], out)
        return {"out": out}
    if call == "packed":
        fit.forward_packed(st["hits"], st["offsets"], out)
        return {"out": out}
    if call == "export":
        fit.forward(st["hits"], st["n"], out, quantiles=st["quantiles"], pooled=st["pooled"])
        return {"out": out, "quantiles": st["quantiles"], "pooled": st["pooled"]}
    if call == "chain":
        trackfit.seed(st["hits"], st["n"], st["b_field"], st["seed"], in_place_at=12)
        fit.forward(st["hits"], st["n"], out)
        trackfit.decode(st["seed"], out, st["params"])
        return {"seed": st["seed"], "features": st["hits"][..., 12:15], "corrections": out, "params": st["params"]}
    fit.forward(st["hits"], st["n"], out)
    return {"out": out}


def _mean_hits(case):
    if case["layout"] == "endcap":
        return 12.5
    return (10 if case["layout"] == "barrel" else case["hits"]) - 0.5 * case["drop"]


def work(case):
    """Valid hits only; a multiply-add is two operations, the seed about 300 a hit
    (a foot point with one refinement, two asinh) and 400 a track in fp64."""
    B, hits = case["tracks"], case["tracks"] * _mean_hits(case)
    if case["kind"] == "seed":
        return {"bytes": hits * 12 + B * (4 + 40) + B * case["hits"] * 12, "flops": 300 * hits + 400 * B}
    m = _workload(case).model
    D, H, E, L, P = m.d_model, m.d_hidden, m.embed_dim, m.n_layers, m.pooled_dim
    mac = E * D + D * D
    if case["kind"] == "concat":
        mac += 4 * H * (D + (L - 1) * 2 * H)
    elif case["kind"] == "attention":
        mac += L * (4 * D * D + 2 * D * H + 2 * D * _mean_hits(case))
    else:
        mac += L * ((4 * H + D) * D + 2 * H * D + 2 * D * D)
    flops = 2 * hits * mac + 2 * B * m.head_hidden * (P + m.n_out)
    weights = W.weight_count(m)
    nbytes = hits * 4 * m.n_features + B * (4 + 20) + weights * (4 if case["precision"] == FP32 else 2)
    if case["call"] == "export":
        nbytes += B * 4 * (m.n_out + P)
    if case["call"] == "packed":
        nbytes += B * 4
    if case["call"] == "chain":
        nbytes += hits * 12 + B * (40 + 20)
        flops += 300 * hits + 400 * B
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times the spread measured between two correct evaluations (the
    tensor-core and the CUDA-core kernels on the same tracks: relative 5e-4 and at
    most 4e-3 with bf16 operands, 1.7e-4 and 9e-4 with fp16; fp32 4e-7 off the 64-bit
    result).  A 16-bit operand that rounds to its neighbour moves the whole network.
    The decode wraps phi: a value at the end of its range may land on the other one."""
    if case["kind"] == "seed":
        return {"rel": 2e-7, "max": 2e-5}
    if case["call"] == "chain":
        return {"rel": 2e-3, "max": 0.6}
    return {FP32: {"rel": 4e-6, "max": 4e-5}, BF16: {"rel": 3e-3, "max": 2e-2}, FP16: {"rel": 8e-4, "max": 5e-3}}[
        case["precision"]]


# ---------------------------------------------------------------------------
# the same in 64 bits, plain torch
# ---------------------------------------------------------------------------

def _rms(x, g, eps):
    return x / torch.sqrt((x * x).mean(-1, keepdim=True) + eps) * g


def _silu(x):
    return x * torch.sigmoid(x)


def _scan(z, c):
    """h_t = h_{t-1} + z_t (c_t - h_{t-1}) along axis 1 from 0."""
    h, out = torch.zeros_like(c[:, 0]), torch.empty_like(c)
    for t in range(c.shape[1]):
        h = h + z[:, t] * (c[:, t] - h)
        out[:, t] = h
    return out


def _encoder(m, w, hits, n):
    """(out, quantiles, pooled) of hits [B, T, F] fp64; per-hit products on the valid rows only."""
    B, T, _ = hits.shape
    dev = hits.device
    t = torch.arange(T, device=dev)[None, :]
    valid = t < n[:, None]
    back = torch.where(valid, n[:, None] - 1 - t, t.expand(B, T))   # each track's hits in reverse

    def pad(v):
        o = torch.zeros((B, T, v.shape[-1]), dtype=v.dtype, device=dev)
        o[valid] = v
        return o

    def lin(v, p, q):
        return v @ w[p].T + w[q]

    def scans(pr):
        H = m.d_hidden
        f = _scan(torch.sigmoid(pad(pr[:, :H])), pad(pr[:, H:2 * H]))
        at = back[..., None].expand(B, T, H)
        r = _scan(torch.sigmoid(pad(pr[:, 2 * H:3 * H])).gather(1, at), pad(pr[:, 3 * H:4 * H]).gather(1, at))
        return torch.cat([f, r.gather(1, at)], -1)

    lo = torch.tensor(m.feat_min, dtype=torch.float64, device=dev)
    hi = torch.tensor(m.feat_max, dtype=torch.float64, device=dev)
    s = torch.tensor(m.fourier_scale, dtype=torch.float64, device=dev)
    arg = math.pi * ((hits[valid] - lo) / (hi - lo))[..., None] * s
    e = torch.cat([torch.sin(arg), torch.cos(arg)], -1).reshape(arg.shape[0], -1)
    x = lin(_silu(lin(e, "emb.w1", "emb.b1")), "emb.w2", "emb.b2")
    for l in range(m.n_layers):
        p = f"layer{l}."
        if m.topology == W.TOPOLOGY_CONCAT:
            y = scans(lin(x, p + "w_in", p + "b_in"))
            x = y[valid]
        elif m.topology == W.TOPOLOGY_ATTENTION:
            D, dh = m.d_model, m.d_model // m.n_heads
            qkv = pad(lin(_rms(x, w[p + "g1"], m.rms_eps), p + "w_qkv", p + "b_qkv"))
            q, k, v = (a.reshape(B, T, m.n_heads, dh).transpose(1, 2) for a in qkv.split(D, -1))
            sc = (q @ k.transpose(-1, -2) / math.sqrt(dh)).masked_fill(~valid[:, None, None, :], -math.inf)
            o = (torch.softmax(sc, -1) @ v).transpose(1, 2).reshape(B, T, D)[valid]
            x1 = x + lin(o, p + "w_o", p + "b_o")
            x = x1 + lin(_silu(lin(_rms(x1, w[p + "g2"], m.rms_eps), p + "w1", p + "b1")), p + "w2", p + "b2")
        else:
            pr = lin(_rms(x, w[p + "g"], m.rms_eps), p + "w_in", p + "b_in")
            x1 = x + lin(scans(pr)[valid], p + "w_m", p + "b_m") * torch.sigmoid(pr[:, 4 * m.d_hidden:])
            x = x1 + lin(_silu(lin(x1, p + "w1", p + "b1")), p + "w2", p + "b2")
    if m.pool == W.POOL_ENDPOINTS:
        H = m.d_hidden
        pv = torch.cat([y[torch.arange(B, device=dev), (n - 1).long(), :H], y[:, 0, H:]], -1)
    else:
        pv = pad(x).sum(1) / n[:, None]
    q = lin(_silu(lin(_rms(pv, w["head.g"], m.rms_eps), "head.w1", "head.b1")), "head.w2", "head.b2")
    q = q.reshape(B, 5, m.n_quantiles)
    return q[:, :, m.n_quantiles // 2], q, pv


def _mod2pi(x):
    return torch.remainder(x, 2 * math.pi)


def _seed(hits, n, b_field):
    """Perigee [B, 5] and residual features [B, T, 3] (0 on padding) in fp64."""
    B, T = hits.shape[:2]
    dev = hits.device
    p = hits[..., :3].double()
    t = torch.arange(T, device=dev)[None, :]
    valid = t < n[:, None]
    rows = torch.arange(B, device=dev)
    tri, last = [p[:, 0]], torch.zeros(B, dtype=torch.int64, device=dev)
    for _ in range(2):   # the first later hit more than 10 mm from the previous one
        far = ((p - tri[-1][:, None]).square().sum(-1).sqrt() > 10.0) & (t > last[:, None]) & valid
        last = far.double().argmax(1)
        tri.append(p[rows, last])
    a, b, c = tri
    ax, ay, bx, by = b[:, 0] - a[:, 0], b[:, 1] - a[:, 1], c[:, 0] - a[:, 0], c[:, 1] - a[:, 1]
    na, nb = ax * ax + ay * ay, bx * bx + by * by
    u1, v1, u2, v2 = ax / na, ay / na, bx / nb, by / nb
    det = u1 * v2 - u2 * v1
    ccx, ccy = (v2 - v1) / (2 * det), (u1 - u2) / (2 * det)
    Cx, Cy, R = a[:, 0] + ccx, a[:, 1] + ccy, torch.hypot(ccx, ccy)
    q = -torch.sign(ax * by - ay * bx)
    dc = torch.hypot(Cx, Cy)
    px, py = Cx - R * Cx / dc, Cy - R * Cy / dc
    phi0 = torch.atan2(q * Cx / dc, -q * Cy / dc)
    d0 = -px * torch.sin(phi0) + py * torch.cos(phi0)
    gp = torch.atan2(py - Cy, px - Cx)
    s0 = R * _mod2pi(-q * (torch.atan2(a[:, 1] - Cy, a[:, 0] - Cx) - gp))
    s2 = R * _mod2pi(-q * (torch.atan2(c[:, 1] - Cy, c[:, 0] - Cx) - gp))
    cot = (c[:, 2] - a[:, 2]) / (s2 - s0)
    z0, theta = a[:, 2] - s0 * cot, torch.atan2(torch.ones_like(cot), cot)
    qop = q * torch.sin(theta) / (0.299792458 * b_field * R / 1000.0)
    seed = torch.stack([d0, z0, phi0, theta, qop], -1)
    # features: the foot point by Newton's method on (hit - p(al)) . t(al)
    st, ct = torch.sin(theta)[:, None], torch.cos(theta)[:, None]
    q, R, phi0, z0 = q[:, None], R[:, None], phi0[:, None], z0[:, None]
    cx = -d0[:, None] * torch.sin(phi0) + q * R * torch.sin(phi0)
    cy = d0[:, None] * torch.cos(phi0) - q * R * torch.cos(phi0)
    g0 = torch.atan2(-(-q * R * torch.cos(phi0)), -(q * R * torch.sin(phi0)))
    x, y, z = p.unbind(-1)
    al = _mod2pi(-q * (torch.atan2(y - cy, x - cx) - g0) + math.pi) - math.pi
    rcot = R * ct / st
    turn = 2 * math.pi * torch.floor(((z - z0) / rcot - al) / (2 * math.pi) + 0.5)
    al = torch.where(2 * math.pi * rcot.abs() > 1.0, al + turn, al)

    def at(al):
        sp, cp = torch.sin(phi0 - q * al), torch.cos(phi0 - q * al)
        return sp, cp, x - (cx - q * R * sp), y - (cy + q * R * cp), z - (z0 + rcot * al)
    for _ in range(12):
        sp, cp, rx, ry, rz = at(al)
        al = al - (st * (rx * cp + ry * sp) + ct * rz) / (-R / st + q * st * (rx * sp - ry * cp))
    sp, cp, rx, ry, rz = at(al)
    du = -sp * rx + cp * ry
    dv = -ct * (cp * rx + sp * ry) + st * rz
    f = torch.stack([torch.asinh(du), torch.asinh(dv), R * al / st], -1)
    return seed, torch.where(valid[..., None], f, torch.zeros((), dtype=f.dtype, device=dev))


def exact(case, seed):
    if work(case)["flops"] > 9e12:
        return None   # more than about 20 seconds in 64 bits
    w, h, n, blob = _inputs(case, seed)
    m, call = w.model, case["call"]
    tens = {k: torch.from_numpy(v.astype(np.float64)).to(h.device) for k, v in W.split_weights(m, blob).items()}
    parts = []
    step = max(1, (1 << 27) // (case["hits"] * max(m.embed_dim, 6 * m.d_hidden)))
    for b in range(0, case["tracks"], step):
        hb, nb = h[b:b + step].double(), n[b:b + step]
        if call in ("seed", "chain"):
            sd, f = _seed(hb, nb, w.b_field)
            if call == "seed":
                parts.append((sd, f))
                continue
            hb[..., 12:15] = f
        out, q, pv = _encoder(m, tens, hb, nb)
        parts.append((sd, f, out) if call == "chain" else (out, q, pv))
    cat = [torch.cat(v) for v in zip(*parts)]
    if call == "seed":
        return {"seed": cat[0], "features": cat[1]}
    if call == "chain":
        sd, f, c = cat
        params = sd + c
        params[:, 2] = math.pi - _mod2pi(math.pi - params[:, 2])
        params[:, 4] = sd[:, 4] + c[:, 4] * (sd[:, 4].abs() + 0.02)
        return {"seed": sd, "features": f, "corrections": c, "params": params}
    if call == "export":
        return {"out": cat[0], "quantiles": cat[1], "pooled": cat[2]}
    return {"out": cat[0]}
