"""What is timed: the calls a user of this library makes, over the sizes they make them at.

A case is a dict of plain values; ``op`` names the call:

* ``search``    tnn_knn over every point of an index (the contexts of a whole data set);
* ``nowcast``   tnn_nowcast: wind at positions that are not in the index (IDW or the MLP);
* ``batch``     one Batch.run over many windows of uneven size;
* ``build``     tnn_build_segments and the export of its segment table;
* ``host``      tnn_knn_host: host points in, host neighbour lists out;
* ``features``  tnn_context_features: MLP inputs and the IDW average of given contexts;
* ``mlp_grad``  MLP.gradients: forward and backward of the learned aggregator;
* ``gka_grad``  GKAMLP.gradients: forward and backward of the learned-scale kernel average.

Searches use the library's default knobs, as a first call does.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2112_10408_gb300 import tnn

SIGMA = (1.0, 1.0, 10.0, 0.01)  # weights of x, y, z (km) and t (s) in the metric
BOX_KM = 2000.0
SPAN_S = 21600.0
STEP_S = 4.0  # radar period
DEV = "cuda"


def listed():
    return [
        # smallest data set of the test strategy: 200 flights of 50 samples, one call, latency
        dict(name="search_tiny_10k", op="search", layout="flights", traj=200, samples=50, ragged=False,
             seg_len=10, k=8, lag=0.0),
        # the headline workload: six hours over a 2000 x 2000 km airspace
        dict(name="search_medium_400k", op="search", layout="flights", traj=2000, samples=200, ragged=False,
             seg_len=20, k=32, lag=0.0),
        # smoothed random walks of uneven length (no shared routes), about a million points
        dict(name="search_walks_1m", op="search", layout="walks", traj=5001, samples=200, ragged=True,
             seg_len=20, k=32, lag=0.0),
        # a dense day: four million points
        dict(name="search_dense_4m", op="search", layout="flights", traj=20000, samples=200, ragged=False,
             seg_len=20, k=32, lag=0.0),
        # serving: wind for the aircraft now in the air, one position each, half-hour lag
        dict(name="nowcast_serve_1037", op="nowcast", traj=5000, samples=200, m=1037, k=32, lag=1800.0,
             flightwise=False, mlp=True, hidden=256),
        # evaluation over held-out flights of the learned form
        dict(name="nowcast_heldout_185k", op="nowcast", traj=4000, samples=200, m=185376, k=32, lag=1800.0,
             flightwise=True, mlp=True, hidden=256),
        # independent airspace/time windows answered by one graph launch
        dict(name="batch_24_windows", op="batch", windows=24, lo=10000, hi=300000),
        # index of a new window (rebuilt as the window moves)
        dict(name="build_medium_400k", op="build", layout="flights", traj=2000, samples=200, ragged=False,
             seg_len=20),
        # host to host: points in, lists out in page-locked memory
        dict(name="host_medium_400k", op="host", layout="flights", traj=2000, samples=200, ragged=False,
             seg_len=20, k=32, lag=0.0, pinned=True),
        # training inputs of the learned form: a million contexts
        dict(name="features_1m", op="features", traj=5000, samples=200, k=32),
        # one training batch of the learned form (192 -> 256 -> 2)
        dict(name="mlp_grad_4096", op="mlp_grad", batch=4096, k=32, hidden=256),
        # one training batch of the kernel average with scales from the location
        dict(name="gka_grad_4096", op="gka_grad", traj=1000, samples=200, batch=4096, k=32, hidden=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["search", "search", "search", "nowcast", "nowcast", "batch", "build", "host", "features",
                     "mlp_grad", "gka_grad"])
    samples = rng.randint(50, 280)
    if op in ("search", "build", "host"):
        layout = rng.choice(["flights", "flights", "walks"])
        n = _log_int(rng, 3000, 2000000 if op != "host" and layout == "flights" else 800000)
        c = dict(op=op, layout=layout, traj=max(2, n // samples), samples=samples, ragged=rng.random() < 0.5,
                 seg_len=rng.randint(8, 40))
        if op != "build":
            c.update(k=rng.choice([rng.randint(4, 64), 8, 16, 32]), lag=1800.0 if rng.random() < 0.15 else 0.0)
        if op == "host":
            c.update(pinned=rng.random() < 0.7)
        return c
    if op == "nowcast":
        return dict(op=op, traj=max(100, _log_int(rng, 100000, 1000000) // samples), samples=samples,
                    m=_log_int(rng, 200, 180000), k=rng.choice([8, 16, 32]), lag=rng.choice([600.0, 1800.0]),
                    flightwise=rng.random() < 0.5, mlp=rng.random() < 0.5, hidden=rng.choice([64, 128, 256]))
    if op == "batch":
        return dict(op=op, windows=rng.randint(3, 24), lo=_log_int(rng, 5000, 20000),
                    hi=_log_int(rng, 50000, 300000))
    if op == "features":
        return dict(op=op, traj=max(8, _log_int(rng, 5000, 900000) // samples), samples=samples,
                    k=rng.randint(4, 64))
    if op == "mlp_grad":
        return dict(op=op, batch=_log_int(rng, 256, 40000), k=rng.choice([8, 16, 32, 64]),
                    hidden=rng.choice([64, 128, 256, 512]))
    return dict(op=op, traj=1000, samples=samples, batch=_log_int(rng, 256, 40000), k=rng.randint(8, 64),
                hidden=rng.randint(8, 32))


# ------------------------------------------------------------------- inputs

class _Rand:
    """Seeded device draws."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV).manual_seed(int(seed) * 1000003 + 17)

    def uniform(self, lo, hi, shape):
        return torch.rand(shape, generator=self.g, device=DEV, dtype=torch.float64) * (hi - lo) + lo

    def normal(self, sd, shape):
        return torch.randn(shape, generator=self.g, device=DEV, dtype=torch.float64) * sd

    def integers(self, lo, hi, shape):
        return torch.randint(lo, hi, shape, generator=self.g, device=DEV)


def _lengths(traj, samples, ragged):
    """Samples per trajectory: the same for every seed of a case, so that its outputs keep their shape."""
    if not ragged:
        return torch.full((traj,), samples, device=DEV, dtype=torch.int64)
    rng = np.random.default_rng(traj)
    return torch.from_numpy(rng.integers(max(3, samples // 4), 2 * samples - samples // 4, traj)).to(DEV)


def _points(seed, layout, traj, samples, ragged, n_routes=64):
    """(xyzt float32 [n, 4] on the device, wind float32 [n, 2], traj_off int64 on the host)."""
    r = _Rand(seed)
    lens = _lengths(traj, samples, ragged)
    S = int(lens.max())
    step = torch.arange(S, device=DEV, dtype=torch.float64)
    if layout == "flights":
        # polylines of 3 to 5 waypoints; a flight follows one with a lateral offset and a cruise level per leg
        nw = r.integers(3, 6, (n_routes,))
        wp = r.uniform(0.0, BOX_KM, (n_routes, 5, 2))
        leg = wp[:, 1:] - wp[:, :-1]
        ll = leg.norm(dim=2)
        ll = torch.where(torch.arange(4, device=DEV)[None] < (nw - 1)[:, None], ll, torch.zeros_like(ll))
        cum = torch.cat([torch.zeros(n_routes, 1, device=DEV, dtype=torch.float64), ll.cumsum(1)], 1)
        route = r.integers(0, n_routes, (traj,))
        speed = r.uniform(0.20, 0.26, (traj,))
        flen = speed * STEP_S * (lens - 1).double()
        s0 = r.uniform(0.0, 1.0, (traj,)) * (cum[route, 4] - flen).clamp_min(0.0)
        s = s0[:, None] + speed[:, None] * STEP_S * step[None]
        last = (nw - 2)[route][:, None]
        li = torch.minimum((s[:, :, None] >= cum[route][:, None, 1:4]).sum(2), last)
        dirs = leg / ll.clamp_min(1e-6)[:, :, None]
        d = dirs[route[:, None], li]
        along = s - cum[route[:, None], li]
        lat = r.normal(5.0, (traj, 1, 1))
        nrm = torch.stack([-d[..., 1], d[..., 0]], 2)
        p = wp[route[:, None], li] + d * along[..., None] + nrm * lat
        z0 = r.uniform(8.5, 12.0, (traj, 1))
        steps = (r.integers(0, 2, (traj, 4)).double() * 1.2 - 0.6)
        steps[:, 0] = 0.0
        z = (z0 + steps.cumsum(1)).clamp(8.5, 12.0).gather(1, li)
        p = p + r.normal(0.05, p.shape)
        z = z + r.normal(0.05, z.shape)
    else:
        head = r.uniform(0.0, 2 * math.pi, (traj, 1)) + r.normal(0.002, (traj, S)).cumsum(1).cumsum(1)
        x = r.uniform(0.0, BOX_KM, (traj, 1)) + (0.23 * STEP_S * head.cos()).cumsum(1)
        y = r.uniform(0.0, BOX_KM, (traj, 1)) + (0.23 * STEP_S * head.sin()).cumsum(1)
        p = torch.stack([x, y], 2)
        z = (r.uniform(8.5, 12.0, (traj, 1)) + r.normal(0.005, (traj, S)).cumsum(1)).clamp(0.0, 12.0)
    t0 = r.uniform(0.0, 1.0, (traj,)) * (SPAN_S - STEP_S * (lens - 1).double()).clamp_min(0.0)
    t = t0[:, None] + STEP_S * step[None]
    keep = step[None] < lens[:, None]
    xyzt = torch.stack([p[..., 0], p[..., 1], z, t], 2)[keep]
    # wind: a mean flow and plane waves, with measurement noise
    wind = torch.tensor([[20.0, 5.0]], device=DEV, dtype=torch.float64).repeat(xyzt.shape[0], 1)
    for _ in range(6):
        k = r.normal(2 * math.pi / 900.0, (2,))
        w = r.normal(2 * math.pi / 30000.0, (1,))
        amp, ph = r.normal(4.0, (2,)), r.uniform(0.0, 2 * math.pi, (2,))
        th = xyzt[:, 0] * k[0] + xyzt[:, 1] * k[1] + xyzt[:, 2] * 0.5 + xyzt[:, 3] * w
        wind += amp[None] * torch.cos(th[:, None] + ph[None])
    wind += r.normal(1.0, wind.shape)
    off = np.zeros(traj + 1, np.int64)
    off[1:] = np.cumsum(lens.cpu().numpy())
    return xyzt.float().contiguous(), wind.float().contiguous(), off


def _contexts(seed, xyzt, off, k):
    """Neighbour lists (idx int32, d2 float32, by distance) with the locality of real ones: the samples before
    the point on its own flight and runs of two other flights; -1 / inf where a flight has too few samples."""
    r = _Rand(seed + 7)
    n, T = xyzt.shape[0], off.shape[0] - 1
    offd = torch.from_numpy(off).to(DEV)
    row = torch.arange(n, device=DEV)
    tr = torch.bucketize(row, offd[1:], right=True)
    own = k - k // 3
    base = r.integers(0, T, (T, 2))
    other = torch.where((row % 2 == 0)[:, None], base[tr, :1], base[tr, 1:])
    lo, ln = offd[other[:, 0]], (offd[1:] - offd[:-1])[other[:, 0]]
    j = torch.arange(k, device=DEV)
    idx = row[:, None] - 1 - j[None]
    idx = torch.where(idx >= offd[tr][:, None], idx, torch.full_like(idx, -1))
    run = lo[:, None] + ((row - offd[tr])[:, None] + j[None]) % ln[:, None]
    idx = torch.where(j[None] < own, idx, run)
    d = xyzt[idx.clamp_min(0)] - xyzt[:, None]
    d2 = (d * d * torch.tensor(SIGMA, device=DEV)).sum(2)
    d2 = torch.where(idx >= 0, d2, torch.full_like(d2, math.inf))
    d2, o = d2.sort(dim=1)
    return idx.gather(1, o).int().contiguous(), d2.contiguous()


def _nowcast_inputs(case, seed):
    """An index's points and winds, and positions on other flights of the same routes, late enough that their
    contexts are full: whole flights, or one sample of each of many flights in no order."""
    m, T, S = case["m"], case["traj"], case["samples"]
    more = int(m / S * 1.8) + 20 if case["flightwise"] else int(1.8 * m) + 50
    xyzt, wind, off = _points(seed, "flights", T + more, S, False)
    n = int(off[T])
    q = xyzt[n:]
    if not case["flightwise"]:
        q = q.view(more, S, 4)[torch.arange(more, device=DEV), _Rand(seed + 3).integers(0, S, (more,))]
    q = q[q[:, 3] > 6000.0]
    return xyzt[:n].contiguous(), wind[:n].contiguous(), off[: T + 1], q[:m].contiguous()


def _mlp_weights(seed, d_in, dh):
    r = _Rand(seed + 31)
    a, b = 1.0 / math.sqrt(d_in), 1.0 / math.sqrt(dh)
    w = torch.cat([r.uniform(-a, a, (d_in * dh + dh,)), r.uniform(-b, b, (2 * dh + 2,))])
    return w.float().cpu().numpy()


def _norm():
    """Channel means and deviations of the features a user standardises with."""
    return np.array([0, 0, 0, -180.0, 20, 5], np.float32), np.array([20, 20, 1, 60.0, 9, 9], np.float32)


def _window_cases(case, seed):
    rng = np.random.default_rng(case["windows"])  # sizes and k belong to the case
    out = []
    for w in range(case["windows"]):
        n = math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"])))
        out.append((max(1, int(round(n / 200.0))), int(rng.choice([16, 32, 64])), seed * 1000 + w))
    return out


def prepare(case, seed):
    op = case["op"]
    s = {"op": op, "case": case}
    if op in ("search", "build", "host"):
        xyzt, _, off = _points(seed, case["layout"], case["traj"], case["samples"], case["ragged"])
        if op == "search":
            s["ix"] = tnn.tnn_build_segments(xyzt, off, SIGMA, case["seg_len"])
        elif op == "build":
            s.update(xyzt=xyzt, off=off)
        else:
            n = xyzt.shape[0]
            out = (torch.empty((n, case["k"]), dtype=torch.int32), torch.empty((n, case["k"])))
            h = xyzt.cpu()
            if case["pinned"]:
                h, out = h.pin_memory(), tuple(o.pin_memory() for o in out)
            s.update(xyzt=h, off=off, out=out)
    elif op == "nowcast":
        xyzt, wind, off, q = _nowcast_inputs(case, seed)
        s.update(ix=tnn.tnn_build_segments(xyzt, off, SIGMA, 20), wind=wind, q=q, mlp=None)
        if case["mlp"]:
            s["mlp"] = tnn.MLP(6 * case["k"], case["hidden"])
            s["mlp"].set_params(_mlp_weights(seed, 6 * case["k"], case["hidden"]))
            s["mean"], s["std"] = _norm()
        else:
            s["mean"] = s["std"] = None
    elif op == "batch":
        ixs, ks = [], []
        for nf, k, sd in _window_cases(case, seed):
            xyzt, _, off = _points(sd, "flights", nf, 200, False)
            ixs.append(tnn.tnn_build_segments(xyzt, off, SIGMA, 20))
            ks.append(k)
        s["batch"] = tnn.Batch(ixs, ks)
    elif op == "features":
        xyzt, wind, off = _points(seed, "flights", case["traj"], case["samples"], False)
        idx, d2 = _contexts(seed, xyzt, off, case["k"])
        s.update(ix=tnn.tnn_build_segments(xyzt, off, SIGMA, 20), wind=wind, idx=idx, d2=d2)
        s["mean"], s["std"] = _norm()
    elif op == "mlp_grad":
        x, y = _mlp_batch(case, seed)
        s["mlp"] = tnn.MLP(6 * case["k"], case["hidden"])
        s["mlp"].set_params(_mlp_weights(seed, 6 * case["k"], case["hidden"]))
        s.update(x=x, y=y)
    else:
        xyzt, wind, off, idx, rows, w = _gka_inputs(case, seed)
        s.update(ix=tnn.tnn_build_segments(xyzt, off, SIGMA, 20), wind=wind, idx=idx, rows=rows)
        s["gka"] = tnn.GKAMLP((1.0, 10.0, 0.01), case["hidden"])
        s["gka"].set_params(w)
    return s


def run(s):
    op, c = s["op"], s["case"]
    if op == "search":
        return tnn.tnn_knn(s["ix"], c["k"], c["lag"])
    if op == "nowcast":
        return tnn.tnn_nowcast(s["ix"], s["wind"], c["k"], c["lag"], q=s["q"], mlp=s["mlp"], mean=s["mean"],
                               std=s["std"])
    if op == "batch":
        s["batch"].run()
        return s["batch"].idx, s["batch"].d2
    if op == "build":
        return tnn.tnn_index_export(tnn.tnn_build_segments(s["xyzt"], s["off"], SIGMA, c["seg_len"]))
    if op == "host":
        return tnn.tnn_knn_host(s["xyzt"], s["off"], SIGMA, c["seg_len"], c["k"], c["lag"], out=s["out"])
    if op == "features":
        return tnn.tnn_context_features(s["ix"], s["wind"], s["idx"], s["d2"], mean=s["mean"], std=s["std"])
    if op == "mlp_grad":
        return s["mlp"].gradients(s["x"], s["y"])
    return s["gka"].gradients(s["ix"], s["wind"], s["rows"], s["idx"])


def _mlp_batch(case, seed):
    r = _Rand(seed)
    x = r.normal(1.0, (case["batch"], 6 * case["k"])).to(torch.bfloat16)
    y = torch.tensor([20.0, 5.0], device=DEV) + r.normal(9.0, (case["batch"], 2)).float()
    return x.contiguous(), y.contiguous()


def _gka_inputs(case, seed):
    xyzt, wind, off = _points(seed, "flights", case["traj"], case["samples"], False)
    idx, _ = _contexts(seed, xyzt, off, case["k"])
    r = _Rand(seed + 13)
    full = (idx >= 0).all(1).nonzero()[:, 0]
    rows = full[r.integers(0, full.shape[0], (case["batch"],))].int().contiguous()
    H = case["hidden"]
    a = 1.0 / math.sqrt(3.0)
    w = torch.cat([r.uniform(-a, a, (4 * H,)), r.normal(0.05, (3 * H,)),
                   torch.tensor([0.004, 0.1, 0.0002], device=DEV, dtype=torch.float64).log()])
    return xyzt, wind, off, idx, rows, w.float().cpu().numpy()


# -------------------------------------------------------- necessary work

def work(case):
    """Bytes: inputs once, outputs once.  Operations: the distances of the k results (11 each), or the products."""
    op = case["op"]
    n = case.get("traj", 0) * case.get("samples", 0)
    k = case.get("k", 0)
    if op in ("search", "host"):
        return {"bytes": 16 * n + 8 * n * k, "flops": 11 * n * k}
    if op == "build":
        S = case["traj"] * -(-case["samples"] // case["seg_len"])
        return {"bytes": 16 * n + 68 * S, "flops": 25 * n}
    if op == "nowcast":
        m = case["m"]
        mac = m * (6 * k * case["hidden"] + 2 * case["hidden"]) if case["mlp"] else 0
        return {"bytes": min(24 * n, 24 * k * m) + 24 * m, "flops": 11 * m * k + 2 * mac}
    if op == "batch":
        n, k = case["windows"] * math.sqrt(case["lo"] * case["hi"]) * 1.3, 37
        return {"bytes": 16 * n + 8 * n * k, "flops": 11 * n * k}
    if op == "features":
        return {"bytes": n * (24 + 8 * k + 12 * k + 8), "flops": 30 * n * k}
    if op == "mlp_grad":
        d, h, B = 6 * k, case["hidden"], case["batch"]
        P = d * h + 3 * h + 2
        return {"bytes": 2 * B * d + 8 * B + 6 * P, "flops": 4 * B * d * h + 8 * B * h}
    B = case["batch"]
    return {"bytes": B * (28 + 28 * k), "flops": B * (40 * k + 14 * case["hidden"])}


# ---------------------------------------------------------------- in 64 bits

def _knn64(xyzt, q, k, lag):
    """(idx int64, d2 float64) of the k nearest points with t < t_q - lag, by (d2, index)."""
    p = xyzt.double()
    sg = torch.tensor(SIGMA, device=DEV, dtype=torch.float64)
    oi, od = [], []
    step = max(1, (1 << 27) // p.shape[0])  # rows of the distance matrix held at once
    for a in range(0, q.shape[0], step):
        qq = q[a:a + step].double()
        d = torch.zeros((qq.shape[0], p.shape[0]), device=DEV, dtype=torch.float64)
        for c in range(4):
            e = p[None, :, c] - qq[:, None, c]
            d += sg[c] * (e * e)
        d[p[None, :, 3] >= qq[:, None, 3] - lag] = math.inf
        v, i = d.topk(k, dim=1, largest=False, sorted=True)
        oi.append(torch.where(v < math.inf, i, torch.full_like(i, -1)))
        od.append(v)
    return torch.cat(oi), torch.cat(od)


def _gelu(z):
    return z * 0.5 * (1.0 + torch.erf(z / math.sqrt(2.0)))


def _split(w, d, h):
    w = torch.from_numpy(w).to(DEV).double()
    return w[: d * h].view(d, h), w[d * h: d * h + h], w[d * h + h: d * h + 3 * h].view(h, 2), w[d * h + 3 * h:]


def _features64(xyzt, wind, q, idx, mean, std):
    p, w = xyzt.double(), wind.double()
    sg = torch.tensor(SIGMA, device=DEV, dtype=torch.float64).sqrt()
    j = idx.long().clamp_min(0)
    f = torch.cat([(p[j] - q.double()[:, None]) * sg, w[j]], 2)
    f = (f - torch.from_numpy(mean).to(DEV).double()) / torch.from_numpy(std).to(DEV).double()
    return torch.where((idx >= 0)[..., None], f, torch.zeros_like(f))


def _idw64(wind, idx, d2, eps=1e-6):
    wt = torch.where(idx >= 0, 1.0 / (d2.double() + eps), torch.zeros_like(d2, dtype=torch.float64))
    return (wt[..., None] * wind.double()[idx.long().clamp_min(0)]).sum(1) / wt.sum(1, keepdim=True)


def exact(case, seed):
    op = case["op"]
    if op == "search":
        xyzt, _, _ = _points(seed, case["layout"], case["traj"], case["samples"], case["ragged"])
        if xyzt.shape[0] > 60000:
            return None
        _, d2 = _knn64(xyzt, xyzt, case["k"], case["lag"])
        return None, d2
    if op == "nowcast":
        if case["m"] * case["traj"] * case["samples"] > 2e10:
            return None
        xyzt, wind, _, q = _nowcast_inputs(case, seed)
        idx, d2 = _knn64(xyzt, q, case["k"], case["lag"])
        if not case["mlp"]:
            return _idw64(wind, idx, d2)
        W1, b1, W2, b2 = _split(_mlp_weights(seed, 6 * case["k"], case["hidden"]), 6 * case["k"], case["hidden"])
        f = _features64(xyzt, wind, q, idx, *_norm())
        return _gelu(f.flatten(1) @ W1 + b1) @ W2 + b2
    if op == "build":
        xyzt, _, off = _points(seed, case["layout"], case["traj"], case["samples"], case["ragged"])
        return _segments64(xyzt, off, case["seg_len"])
    if op == "features":
        xyzt, wind, off = _points(seed, "flights", case["traj"], case["samples"], False)
        idx, d2 = _contexts(seed, xyzt, off, case["k"])
        f = [_features64(xyzt, wind, xyzt[a:a + 65536], idx[a:a + 65536], *_norm()).flatten(1).float()
             for a in range(0, idx.shape[0], 65536)]
        v = [_idw64(wind, idx[a:a + 65536], d2[a:a + 65536]) for a in range(0, idx.shape[0], 65536)]
        return torch.cat(f), torch.cat(v)
    if op == "mlp_grad":
        x, y = _mlp_batch(case, seed)
        d, h = 6 * case["k"], case["hidden"]
        W = [w.clone().requires_grad_() for w in _split(_mlp_weights(seed, d, h), d, h)]
        out = _gelu(x.double() @ W[0] + W[1]) @ W[2] + W[3]
        loss = ((out - y.double()) ** 2).mean()
        g = torch.autograd.grad(loss, W)
        return loss.detach().view(1), torch.cat([v.reshape(-1) for v in g])
    if op == "gka_grad":
        xyzt, wind, off, idx, rows, w = _gka_inputs(case, seed)
        H = case["hidden"]
        w = torch.from_numpy(w).to(DEV).double().requires_grad_()
        p, r = xyzt.double(), rows.long()
        lo, hi = p.min(0).values, p.max(0).values
        u = ((p[r] - lo) / (hi - lo))[:, :3]
        th = torch.tanh(u @ w[: 3 * H].view(3, H) + w[3 * H: 4 * H]) @ w[4 * H: 7 * H].view(H, 3) + w[7 * H:]
        sc = th.exp()
        j = idx[r].long()
        e = (p[j] - p[r][:, None]) ** 2
        ex = sc[:, :1] * (e[..., 0] + e[..., 1]) + sc[:, 1:2] * e[..., 2] + sc[:, 2:] * e[..., 3]
        a = torch.softmax(-ex, dim=1)
        out = (a[..., None] * wind.double()[j]).sum(1)
        loss = ((out - wind.double()[r]) ** 2).mean()
        g, = torch.autograd.grad(loss, w)
        return loss.detach().view(1), g
    return None


def _segments64(xyzt, off, K):
    """Segment records ordered by start time, as the library lays them out, and the running largest end time."""
    first, count, traj = [], [], []
    for t in range(off.shape[0] - 1):
        f = np.arange(off[t], off[t + 1], K)
        first.append(f)
        count.append(np.minimum(K, off[t + 1] - f))
        traj.append(np.full(f.shape, t))
    first, count, traj = (torch.from_numpy(np.concatenate(v)).to(DEV) for v in (first, count, traj))
    S = first.shape[0]
    q = torch.tensor(SIGMA[:3], device=DEV, dtype=torch.float64).sqrt()
    p = xyzt.double()
    a = p[first, :3] * q
    ab = (p[first + count - 1, :3] * q) - a
    n2 = (ab * ab).sum(1)
    u = torch.where(n2[:, None] > 1e-30, ab / n2.clamp_min(1e-300)[:, None], torch.zeros_like(ab))
    rad = torch.zeros(S, device=DEV, dtype=torch.float64)
    for j in range(K):
        d = p[torch.minimum(first + j, first + count - 1), :3] * q - a
        lam = (d * u).sum(1).clamp(0.0, 1.0)
        rad = torch.maximum(rad, (d - lam[:, None] * ab).norm(dim=1))
    tA, tB = p[first, 3], p[first + count - 1, 3]
    ids = torch.stack([first, count, traj, torch.arange(S, device=DEV)], 1).int().view(torch.float32).double()
    rec = torch.cat([a, tA[:, None], u, tB[:, None], ab, rad[:, None], ids], 1)
    o = torch.sort(tA, stable=True).indices
    return rec[o], torch.cummax(tB[o], 0).values
