"""Measured cases of the library: what a user's program has it do, through its public calls.

A case is one pass of a user's program over one synthetic dataset (the workloads of
``paper_1903_12294_gb300.synth``, cropped to the case's grid). Kinds:

  field    label a small field-only window without any allocation (a real-time loop)
  step     new point samples in a resident dataset: bin, label, feature statistics
  query    one interactive query over a resident, binned dataset
  index    bin the points and read the per-voxel index back
  batch    many queries with their own thresholds and windows in one call
  serve    a burst of queries through the query server, labels taken by the client
  cluster  the 4D clustering of field and point samples
  summary  what follows a clustering: merge, relabel, per-cluster summaries, trajectory pieces
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1903_12294_gb300 import msf, synth

DEV = "cuda"
FEATURE_CAP = 1 << 20  # most feature records a case keeps room for (the benchmark's table)


def listed():
    return [
        # the smallest call: a real-time loop labels a small window, ragged in every dimension
        {"name": "field_small", "kind": "field", "data": "tiny", "nx": 45, "ny": 37, "nz": 21,
         "T": 6, "edges": 3},
        # the tiny workload end to end: launches and host work dominate
        {"name": "step_tiny", "kind": "step", "data": "tiny", "nx": 32, "ny": 32, "nz": 32, "T": 8,
         "P": 20000, "edges": 7},
        # points saved more often than the field, on a ragged grid that some of them leave
        {"name": "step_multirate", "kind": "step", "data": "multirate", "nx": 61, "ny": 53,
         "nz": 47, "T": 9, "r": 4, "P": 30001, "edges": 7},
        # the mid-size dataset (128^3 x 32, 1M tracers): one query
        {"name": "query_mid", "kind": "query", "data": "mid", "nx": 128, "ny": 128, "nz": 128,
         "T": 32, "P": 1 << 20, "t0": 0, "t1": 32, "edges": 7},
        # its preprocessing index, read back by the program
        {"name": "index_mid", "kind": "index", "data": "mid", "nx": 128, "ny": 128, "nz": 128,
         "T": 32, "P": 1 << 20, "sumq": False},
        # the benchmark's dataset (256^3 x 24, 8M particles, 4 attributes): the query alone
        {"name": "query_combustion", "kind": "query", "data": "combustion", "nx": 256, "ny": 256,
         "nz": 256, "T": 24, "P": 8 << 20, "t0": 0, "t1": 24, "edges": 7},
        # and the whole hot path on it, the largest case
        {"name": "step_combustion", "kind": "step", "data": "combustion", "nx": 256, "ny": 256,
         "nz": 256, "T": 24, "P": 8 << 20, "edges": 7},
        # 2D + time traffic: one interactive query over 64 of the 96 steps
        {"name": "query_city", "kind": "query", "data": "city", "nx": 1024, "ny": 1024, "nz": 1,
         "T": 96, "P": 208334, "t0": 16, "t1": 80, "edges": 7},
        # sixteen queries of uneven windows on the batched dataset (192^3 x 32, 4M particles)
        {"name": "batch_blobs", "kind": "batch", "data": "blobs", "nx": 192, "ny": 192, "nz": 192,
         "T": 32, "P": 4 << 20, "nq": 16},
        # a burst of sixteen queries at the query server over the traffic dataset
        {"name": "serve_city", "kind": "serve", "data": "city", "nx": 1024, "ny": 1024, "nz": 1,
         "T": 96, "P": 208334, "nq": 16},
        # the paper's own clustering of the mid dataset: 16,384 centres, ten updates
        {"name": "cluster_mid", "kind": "cluster", "data": "mid", "nx": 128, "ny": 128, "nz": 128,
         "T": 32, "P": 1 << 20, "k0": 16, "k1": 16, "k2": 16, "k3": 4, "iters": 10},
        # what a user does with such a clustering
        {"name": "summary_mid", "kind": "summary", "data": "mid", "nx": 128, "ny": 128, "nz": 128,
         "T": 32, "P": 1 << 20, "k0": 16, "k1": 16, "k2": 16, "k3": 4},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _grid(rng, lo, hi):
    """Either a cube of whole 32-voxel rows or a ragged box."""
    n = _log_int(rng, lo, hi)
    if n >= 32 and rng.random() < 0.4:
        n = n // 32 * 32
        return n, n, n
    return tuple(max(lo // 2, int(n * rng.uniform(0.6, 1.0))) for _ in range(3))


def draw(rng):
    kind = rng.choice(["field", "step", "query", "index", "batch", "serve", "cluster", "summary"])
    if kind == "field":
        nx, ny, nz = _grid(rng, 16, 96)
        T = _log_int(rng, 1, 24)
        # windows of up to about four million voxel-timesteps fit the call's fixed scratch
        while T > 1 and -(-nx // 32) * -(-ny // 16) * -(-nz // 16) * 4 * -(-T // 4) > 560:
            T -= 1
        return {"kind": kind, "data": "tiny", "nx": nx, "ny": ny, "nz": nz, "T": T,
                "edges": rng.choice([3, 3, 1])}
    if kind == "serve" or (kind == "query" and rng.random() < 0.4):
        nx, ny = _log_int(rng, 200, 1024), _log_int(rng, 200, 1024)
        T = _log_int(rng, 16, 96)
        c = {"kind": kind, "data": "city", "nx": nx, "ny": ny, "nz": 1, "T": T,
             "P": _log_int(rng, 5000, 208334)}
        if kind == "serve":
            return dict(c, nq=rng.randint(2, 16))
    else:
        data = {"step": ["tiny", "multirate", "mid", "combustion"],
                "query": ["tiny", "multirate", "mid", "combustion"],
                "index": ["tiny", "mid", "blobs", "combustion"], "batch": ["blobs"],
                "cluster": ["mid", "multirate"], "summary": ["mid"]}[kind]
        data = rng.choice(data)
        hi = {"tiny": 64, "multirate": 64, "mid": 128, "blobs": 192, "combustion": 224}[data]
        if kind in ("index", "cluster", "summary"):
            hi = min(hi, 128)
        nx, ny, nz = _grid(rng, 24, hi)
        T = _log_int(rng, 3, 24)
        c = {"kind": kind, "data": data, "nx": nx, "ny": ny, "nz": nz, "T": T,
             "P": _log_int(rng, 2000, min(8 << 20, max(4000, nx * ny * nz)))}
        if data == "multirate":
            c["r"] = rng.randint(2, 4)
    if kind in ("step", "query"):
        c["edges"] = rng.choice([7, 7, 7, 3, 5])
    if kind == "query":
        c["t0"] = rng.randint(0, T // 3)
        c["t1"] = rng.randint(c["t0"] + 2, T)
    if kind == "index":
        c["sumq"] = rng.random() < 0.3
    if kind == "batch":
        c["nq"] = rng.randint(3, 16)
    if kind in ("cluster", "summary"):
        for i, e in enumerate((nx, ny, nz)):
            c["k%d" % i] = max(1, e // rng.randint(7, 12))
        c["k3"] = max(1, T // rng.randint(3, 8))
    if kind == "cluster":
        c["iters"] = rng.randint(2, 10)
    return c


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------

def _workload(case, seed):
    """The case's dataset on the GPU, from the seed alone: a synthetic workload, cropped to the
    grid (points beyond it have left the domain)."""
    nx, ny, nz, T, data = case["nx"], case["ny"], case["nz"], case["T"], case["data"]
    n = max(nx, ny, nz)
    seed = synth.SEED_BASE + 1000 + int(seed)
    P = case.get("P", 64)
    if data == "tiny":
        wl = synth.tiny(DEV, n, T, P, seed)
    elif data == "multirate":
        wl = synth.multirate(DEV, n, T, case["r"], P, seed)
    elif data == "mid":
        wl = synth.mid(DEV, n, T, P, seed)
    elif data == "combustion":
        wl = synth.combustion(DEV, n, T, P, seed)
    elif data == "blobs":
        wl = synth.batched(DEV, n, T, P, seed, nq=case.get("nq", 1))
    else:
        wl = synth.serving(DEV, n, T, P, seed, nq=max(1, case.get("nq", 1)))
    if case["kind"] in ("batch", "serve"):  # the seed's criteria over the case's windows
        wl.queries = [(a, b, p, e) for (a, b), (_, _, p, e) in zip(_windows(case), wl.queries)]
    if (nz, ny, nx) != tuple(wl.field.shape[1:]):
        wl.field = wl.field[:, :nz, :ny, :nx].contiguous()
    wl.t0, wl.t1 = case.get("t0", 0), case.get("t1", T)
    wl.edges = case.get("edges", 7)
    return wl


def _windows(case):
    """Windows of a case's queries: lengths spread evenly over 2..32 steps of the dataset (batch)
    or 4..64 (serve), in mixed order, starting anywhere."""
    T, nq = case["T"], case["nq"]
    lo, hi = (2, min(32, T)) if case["kind"] == "batch" else (4, min(64, T))
    out = []
    for i in range(nq):
        tw = lo + (hi - lo) * (i * 7 % nq if nq % 7 else i) // max(nq - 1, 1)
        t0 = i * 7919 % (T - tw + 1)
        out.append((t0, t0 + tw))
    return out


def _attrs(case):
    return {"tiny": 1, "multirate": 2, "mid": 2, "combustion": 4, "blobs": 3, "city": 2}[case["data"]]


def _point_steps(case, tw=None):
    return (case["T"] if tw is None else tw) * case.get("r", 1)


def _resident(wl, sumq=False):
    ctx = msf.Context(0)
    ctx.load(wl.field, wl.pos, wl.attr, wl.field_step)
    ctx.bin(sumq)
    return ctx


def _cells(case):
    return case["k0"] * case["k1"] * case["k2"] * case["k3"]


def _clustering(case, wl, seed):
    """Labels and centres as a clustering leaves them: every sample in or near the seed-grid cell
    that holds it, boundaries shifted by the sample's value, centre values the samples' means."""
    T, nz, ny, nx = wl.field.shape
    k = [case["k0"], case["k1"], case["k2"], case["k3"]]
    C = [nx / k[0], ny / k[1], nz / k[2], T / k[3]]

    def cell(u, i, shift):
        return torch.clamp(((u / C[i]) + shift).floor(), 0, k[i] - 1).to(torch.int32)

    def label(x, y, z, t, v):
        s = 0.35 * torch.sin(9.0 * v)  # a smooth value moves the boundary by up to 0.35 cells
        return ((cell(t, 3, 0.0 * s) * k[2] + cell(z, 2, s)) * k[1] + cell(y, 1, -s)) * k[0] \
            + cell(x, 0, s)

    def ax(n):
        return torch.arange(n, device=DEV, dtype=torch.float32) + 0.5

    K = _cells(case)
    fl = torch.empty((T, nz, ny, nx), dtype=torch.int32, device=DEV)
    pl = torch.empty((T, wl.pos.shape[2]), dtype=torch.int32, device=DEV)
    sums = torch.zeros((2, K), dtype=torch.int64, device=DEV)
    cnt = torch.zeros((2, K), dtype=torch.int64, device=DEV)
    for t in range(T):
        tt = torch.full((1,), t + 0.5, device=DEV)
        fl[t] = label(ax(nx)[None, None, :], ax(ny)[None, :, None], ax(nz)[:, None, None], tt,
                      wl.field[t])
        x, y, z = wl.pos[t]
        pv = wl.attr[t, 0]
        inside = (x >= 0) & (x < nx) & (y >= 0) & (y < ny) & (z >= 0) & (z < nz)
        pl[t] = torch.where(inside, label(x, y, z, tt, pv), -1)
        for i, (l, v) in enumerate(((pl[t][inside], pv[inside]),
                                    (fl[t].reshape(-1), wl.field[t].reshape(-1)))):
            l = l.long()
            sums[i].index_add_(0, l, torch.round(v.double() * (1 << 20)).long())
            cnt[i].index_add_(0, l, torch.ones_like(l))
    cen = torch.empty((K, 6), device=DEV)
    i = torch.arange(K, device=DEV)
    cen[:, 0] = (i % k[0] + 0.5) * C[0]
    cen[:, 1] = (i // k[0] % k[1] + 0.5) * C[1]
    cen[:, 2] = (i // (k[0] * k[1]) % k[2] + 0.5) * C[2]
    cen[:, 3] = (i // (k[0] * k[1] * k[2]) + 0.5) * C[3]
    cen[:, 4:] = (sums.double() / (1 << 20) / cnt.clamp_min(1)).t().float()
    return fl, pl, cen.contiguous(), K


def prepare(case, seed):
    kind = case["kind"]
    wl = _workload(case, seed)
    T, nz, ny, nx = wl.field.shape
    if kind == "field":
        return {"kind": kind, "field": wl.field, "labels": torch.empty(wl.field.shape, dtype=torch.int32, device=DEV),
                "pred": wl.preds[0], "edges": wl.edges}
    s = {"kind": kind, "ctx": _resident(wl, case.get("sumq", False))}
    if kind in ("step", "query"):
        s["crit"] = msf.make_criteria(wl.t0, wl.t1, _preds(case, wl), wl.edges)
        s["labels"] = torch.empty((wl.t1 - wl.t0, nz, ny, nx), dtype=torch.int32, device=DEV)
    if kind == "step":
        words = msf.FEATURE_DTYPE.itemsize // 8
        s["table"] = torch.zeros((_cap(case), words), dtype=torch.int64, device=DEV)
        s["A"] = wl.attr.shape[1]
    elif kind == "index":
        s["sumq"] = case["sumq"]
    elif kind == "batch":
        s["queries"] = wl.queries
        s["labels"] = [torch.empty((t1 - t0, nz, ny, nx), dtype=torch.int32, device=DEV)
                       for t0, t1, _, _ in wl.queries]
    elif kind == "serve":
        s["queries"] = wl.queries
        s["server"] = msf.Server(s["ctx"], pool_bytes=8 << 30)
    elif kind == "cluster":
        s["args"] = (0, T, 0, (case["k0"], case["k1"], case["k2"], case["k3"]))
        s["iters"] = case["iters"]
    elif kind == "summary":
        s["fl"], s["pl"], s["centers"], s["K"] = _clustering(case, wl, seed)
        s["map"] = torch.empty(s["K"], dtype=torch.int32, device=DEV)
        s["pieces"] = torch.zeros((T * wl.pos.shape[2] // 2 + 1, 4), dtype=torch.int32, device=DEV)
        s["T"] = T
    return s


def _cap(case):
    """Feature records the program keeps room for."""
    return min(FEATURE_CAP, max(1024, case["nx"] * case["ny"] * case["nz"] * case["T"] // 16))


def _preds(case, wl):
    # the traffic workload's criteria come with its queries, the others have one of their own
    return wl.queries[0][2] if case["data"] == "city" else wl.preds


# ---------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------

def run(s):
    kind = s["kind"]
    if kind == "field":
        n = msf.msf_segment_field_noalloc(s["field"], s["labels"], s["pred"], s["edges"])
        return {"labels": s["labels"], "n": n}
    ctx = s["ctx"]
    if kind == "query":
        return {"labels": s["labels"], "n": msf.msf_segment(ctx.h, s["crit"], s["labels"])}
    if kind == "step":
        ctx.bin()
        n = msf.msf_segment(ctx.h, s["crit"], s["labels"])
        return {"labels": s["labels"], "n": n, "features": _features(s)}
    if kind == "index":
        st = ctx.bin(s["sumq"])
        key, count, mean, sumq = ctx.bins(DEV, s["sumq"])
        return {"key": key, "count": count, "mean": mean, "sumq": sumq,
                "in_domain": int(st.in_domain)}
    if kind == "batch":
        labels, n = ctx.segment_batch(s["queries"], s["labels"])
        return {"labels": labels, "n": n}
    if kind == "serve":
        srv, nq = s["server"], len(s["queries"])
        for i, (t0, t1, preds, edges) in enumerate(s["queries"]):
            srv.submit(i, t0, t1, preds, edges)
        labels, n, got = [None] * nq, [0] * nq, 0
        while got < nq:
            for r in srv.poll(nq, timeout_ms=10000):
                if r.status != msf.MSF_OK:
                    raise msf.MsfError(r.status, "query server")
                n[r.tag] = int(r.n_features)
                labels[r.tag] = srv.take_labels(r)
                got += 1
        return {"labels": labels, "n": n}
    if kind == "cluster":
        t0, t1, attr, k = s["args"]
        fl, pl, centers, counts, it = ctx.cluster(t0, t1, attr, k, w_p=1.0, w_f=1.0, w_d=0.05,
                                                  c_f=1.0, eps_c=1e-3, max_iter=s["iters"])
        return {"field_labels": fl, "point_labels": pl, "centers": centers, "counts": counts,
                "updates": it}
    # summary: merge the centres, relabel the samples through the map (a fixed point after the
    # first pass: every pass reads and writes all of them), summarise and cut the trajectories
    m, groups = ctx.merge_clusters(s["centers"], 0.02, out=s["map"])
    ctx.relabel(s["fl"], m)
    ctx.relabel(s["pl"], m)
    st = ctx.cluster_stats(0, s["T"], 0, s["fl"], s["pl"], s["K"])
    pieces, n = ctx.split_trajectories(0, s["T"], s["pl"], msf.MSF_SPACE_POINTS, 2, s["pieces"])
    return {"map": m, "groups": groups, "field_labels": s["fl"], "point_labels": s["pl"],
            "stats": {f: st[f] for f in st.dtype.names}, "pieces": pieces, "n_pieces": n}


def _features(s):
    """The features of the labelling into the program's device table (the C call): its columns,
    zero past the last feature."""
    ct, ctx, tab = msf.ctypes, s["ctx"], s["table"]
    n = ct.c_int64(0)
    st = msf.load_library().msf_extract_features(
        ctx.h, ct.byref(s["crit"]), s["labels"].data_ptr(), msf.MSF_DEVICE, tab.data_ptr(),
        msf.MSF_DEVICE, tab.shape[0], ct.byref(n))
    if st != msf.MSF_OK:
        raise msf.MsfError(st, "msf_extract_features")
    A = s["A"]

    def col(name, dtype, count=0):
        o = getattr(msf.msf_feature, name).offset // dtype.itemsize
        v = tab.view(dtype)
        return v[:, o:o + count] if count else v[:, o]

    i32, i64, f32, f64 = torch.int32, torch.int64, torch.float32, torch.float64
    return {"n": n.value, "label": col("label", i32), "bbox_min": col("bbox_min", i32, 4),
            "bbox_max": col("bbox_max", i32, 4), "n_vox": col("n_vox", i64),
            "n_pts": col("n_pts", i64), "sum_field": col("sum_field", f64),
            "mean_field": col("mean_field", f64), "std_field": col("std_field", f64),
            "min_field": col("min_field", f32), "max_field": col("max_field", f32),
            "centroid": col("centroid", f64, 4), "sumq": col("sumq", i64, A),
            "mean_attr": col("mean_attr", f64, A), "std_attr": col("std_attr", f64, A)}


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------

def _query_bytes(case, tw, n_arrays, edges):
    V = case["nx"] * case["ny"] * case["nz"]
    traj = 4 * case.get("P", 0) * _point_steps(case, tw) if edges & 4 else 0  # the window's keys
    return V * tw * (4 * n_arrays + 4) + traj


def work(case):
    kind = case["kind"]
    V, T = case["nx"] * case["ny"] * case["nz"], case["T"]
    N = V * T
    if kind == "field":
        return {"bytes": 8 * N, "flops": 0}
    A, P = _attrs(case), case["P"]
    NP = P * _point_steps(case)
    n_arrays = 3 if case["data"] == "combustion" else 2
    index = NP * (12 + 4 * A) + N * (4 + 4 * A)  # samples in, counts and means out
    if kind == "query":
        return {"bytes": _query_bytes(case, case["t1"] - case["t0"], n_arrays, case["edges"]),
                "flops": 0}
    if kind == "step":  # samples and field in, index and labels out
        return {"bytes": index + 8 * N, "flops": 0}
    if kind == "index":  # the index kept and the copies handed out (keys included)
        return {"bytes": index + 4 * NP + (8 * A * N if case["sumq"] else 0), "flops": 0}
    if kind in ("batch", "serve"):
        return {"bytes": sum(_query_bytes(case, b - a, 2, 7) for a, b in _windows(case)),
                "flops": 0}
    if kind == "cluster":
        # per assignment: sample in, label out; the sixteen centres a 2C region holds on average,
        # about 20 operations each
        it = case["iters"]
        return {"bytes": it * (8 * N + 20 * NP), "flops": it * 16 * 20 * (N + NP)}
    # labels read and written by the relabelling, labels and values read by the summaries, point
    # labels read for the pieces
    return {"bytes": 8 * (N + NP) + 8 * N + 20 * NP + 4 * NP, "flops": _cells(case) ** 2 * 6}


# ---------------------------------------------------------------------------------------------
# the computed numbers in 64 bits, with plain torch
# ---------------------------------------------------------------------------------------------

def exact(case, seed):
    if case["kind"] == "index":
        return _exact_index(case, seed)
    if case["kind"] == "step":
        return _exact_step(case, seed)
    if case["kind"] == "summary":
        return _exact_summary(case, seed)
    # labels and counts only, or (the clustering) centres that follow from fp32 decisions
    return None


def _keys(wl):
    """Voxel of every point sample of point step j, -1 outside the grid."""
    T, nz, ny, nx = wl.field.shape

    def key(j):
        x, y, z = (wl.pos[j, i].floor() for i in range(3))
        ok = (x >= 0) & (x < nx) & (y >= 0) & (y < ny) & (z >= 0) & (z < nz)
        k = (z.long() * ny + y.long()) * nx + x.long()
        return torch.where(ok, k, -1)

    return key


def _fstep(wl):
    return list(wl.field_step) if wl.field_step is not None else list(range(wl.field.shape[0]))


def _exact_index(case, seed):
    wl = _workload(case, seed)
    T, nz, ny, nx = wl.field.shape
    V, A, key = nz * ny * nx, wl.attr.shape[1], _keys(wl)
    mean = torch.empty((A, T, nz, ny, nx), dtype=torch.float64, device=DEV)
    for j, t in enumerate(_fstep(wl)):  # one point step per field step in these cases
        k = key(j)
        m = k >= 0
        c = torch.zeros(V, dtype=torch.int64, device=DEV).index_add_(0, k[m], torch.ones_like(k[m]))
        for a in range(A):
            s = torch.zeros(V, dtype=torch.float64, device=DEV)
            s.index_add_(0, k[m], wl.attr[j, a][m].double())
            mean[a, t] = (s / c).view(nz, ny, nx)  # 0 / 0: NaN, an empty voxel
    return {"key": None, "count": None, "mean": mean, "sumq": None, "in_domain": None}


def _components(n, u, v):
    """Smallest member of each member's component over the edges (u, v)."""
    f = torch.arange(n, device=DEV)
    while True:
        fu, fv = f[u], f[v]
        live = fu != fv
        if not bool(live.any()):
            return f
        u, v, fu, fv = u[live], v[live], fu[live], fv[live]
        m = torch.minimum(fu, fv)
        f.scatter_reduce_(0, fu, m, "amin")
        f.scatter_reduce_(0, fv, m, "amin")
        while True:
            g = f[f]
            if torch.equal(g, f):
                break
            f = g


def _compare(x, op, lo, hi):
    lo, hi = np.float32(lo).item(), np.float32(hi).item()
    return {0: lambda: x > lo, 1: lambda: x >= lo, 2: lambda: x < lo, 3: lambda: x <= lo,
            4: lambda: (x >= lo) & (x <= hi)}[op]()


def _exact_step(case, seed):
    wl = _workload(case, seed)
    T, nz, ny, nx = wl.field.shape
    V, A, key, fs = nz * ny * nx, wl.attr.shape[1], _keys(wl), _fstep(wl)
    Tp, P = wl.pos.shape[0], wl.pos.shape[2]
    # membership, with the per-voxel mean as the header defines it: exact fixed-point sums at
    # the scale of the whole dataset, then fp32
    b = (P * Tp).bit_length()
    ks = [62 - math.frexp(float(wl.attr[:, a].abs().max()))[1] - b for a in range(A)]
    mask = torch.empty((T, V), dtype=torch.bool, device=DEV)
    for t in range(T):
        js = [j for j in range(Tp) if fs[j] == t]
        k = torch.cat([key(j) for j in js])
        m = k >= 0
        c = torch.zeros(V, dtype=torch.int64, device=DEV).index_add_(0, k[m], torch.ones_like(k[m]))
        act = torch.ones(V, dtype=torch.bool, device=DEV)
        for src, a, op, lo, hi in wl.preds:
            if src == synth.SRC_FIELD:
                x = wl.field[t].reshape(-1)
            elif src == synth.SRC_COUNT:
                x, lo, hi = c, int(lo), int(hi)
            else:
                v = torch.cat([wl.attr[j, a] for j in js])[m].double()
                s = torch.zeros(V, dtype=torch.int64, device=DEV)
                s.index_add_(0, k[m], torch.round(v * 2.0 ** ks[a]).long())
                h = ks[a] // 2
                x = (s.float() / c.float()) * 2.0 ** -h * 2.0 ** -(ks[a] - h)
            act &= _compare(x, op, lo, hi)
        mask[t] = act
    ids = mask.reshape(-1).nonzero().reshape(-1)
    n = ids.numel()
    idm = torch.full((T * V,), -1, dtype=torch.int32, device=DEV)
    idm[ids] = torch.arange(n, device=DEV, dtype=torch.int32)
    g = idm.view(T, nz, ny, nx)
    us, vs = [], []

    def edges(p, q):
        e = (p >= 0) & (q >= 0)
        us.append(p[e].long())
        vs.append(q[e].long())

    if wl.edges & 1:
        for t in range(T):
            for dz in (0, 1):
                for dy in (-1, 0, 1):
                    for dx in (-1, 0, 1):
                        if (dz, dy, dx) > (0, 0, 0):
                            def cut(d, n, first):
                                lo, hi = max(0, -d), min(n, n - d)
                                return slice(lo, hi) if first else slice(lo + d, hi + d)
                            edges(g[t, cut(dz, nz, 1), cut(dy, ny, 1), cut(dx, nx, 1)],
                                  g[t, cut(dz, nz, 0), cut(dy, ny, 0), cut(dx, nx, 0)])
    if wl.edges & 2:
        for t in range(T - 1):
            edges(g[t], g[t + 1])
    if wl.edges & 4:
        for j in range(Tp - 1):
            k, q = key(j), key(j + 1)
            ok = (k >= 0) & (q >= 0)
            edges(idm[fs[j] * V + k[ok]], idm[fs[j + 1] * V + q[ok]])
    roots, fid = torch.unique(_components(n, torch.cat(us), torch.cat(vs)), return_inverse=True)
    del us, vs
    F = roots.numel()

    def total(i, v):
        return torch.zeros(F, dtype=torch.float64, device=DEV).index_add_(0, i, v)

    def spread(i, v, cnt):  # mean and population deviation
        mean = total(i, v) / cnt
        return mean, (total(i, (v - mean[i]).square()) / cnt).sqrt()

    nv = total(fid, torch.ones(n, dtype=torch.float64, device=DEV))
    f = wl.field.reshape(-1)[ids]
    mf, sf = spread(fid, f.double(), nv)
    inf = math.inf
    fmin = torch.full((F,), inf, device=DEV).scatter_reduce_(0, fid, f, "amin")
    fmax = torch.full((F,), -inf, device=DEV).scatter_reduce_(0, fid, f, "amax")
    cen = torch.stack([total(fid, c.double()) / nv for c in
                       (ids // V, ids // (ny * nx) % nz, ids // nx % ny, ids % nx)], 1)
    pf, pa = [], [[] for _ in range(A)]
    for j in range(Tp):
        k = key(j)
        i = idm[fs[j] * V + k.clamp_min(0)]
        ok = (k >= 0) & (i >= 0)
        pf.append(fid[i[ok].long()])
        for a in range(A):
            pa[a].append(wl.attr[j, a][ok].double())
    pf = torch.cat(pf)
    npt = total(pf, torch.ones(pf.numel(), dtype=torch.float64, device=DEV))
    at = [spread(pf, torch.cat(pa[a]), npt) for a in range(A)]
    def table(v):  # as the program's table has it: zero past the last feature
        return torch.cat([v.double(), v.new_zeros((_cap(case) - F, *v.shape[1:])).double()])

    return {"labels": None, "n": None, "features": {
        "n": None, "label": None, "bbox_min": None, "bbox_max": None, "n_vox": None,
        "n_pts": None, "sum_field": table(mf * nv), "mean_field": table(mf),
        "std_field": table(sf), "min_field": table(fmin), "max_field": table(fmax),
        "centroid": table(cen), "sumq": None,
        "mean_attr": table(torch.stack([m for m, _ in at], 1)),
        "std_attr": table(torch.stack([s for _, s in at], 1))}}


def _exact_summary(case, seed):
    wl = _workload(case, seed)
    fl, pl, cen, K = _clustering(case, wl, seed)
    T, nz, ny, nx = wl.field.shape
    # merge: the match graph over all pairs (fp32 as defined), its components
    us, vs = [], []
    for lo in range(0, K, 2048):
        hi = min(K, lo + 2048)
        ok = torch.ones((hi - lo, K), dtype=torch.bool, device=DEV)
        for c in (4, 5):
            p, q = cen[lo:hi, c, None], cen[None, :, c]
            ok &= (p == q) | (2.0 * (p - q).abs() < np.float32(0.02).item() * (p.abs() + q.abs()))
        u, v = ok.nonzero(as_tuple=True)
        keep = v > u + lo
        us.append(u[keep] + lo)
        vs.append(v[keep])
    m = _components(K, torch.cat(us), torch.cat(vs))

    def stats(l, v):
        cnt = torch.zeros(K, dtype=torch.float64, device=DEV)
        cnt.index_add_(0, l, torch.ones_like(v))
        mean = torch.zeros_like(cnt).index_add_(0, l, v) / cnt
        dev = torch.zeros_like(cnt).index_add_(0, l, (v - mean[l]).square())
        return mean.cpu(), (dev / cnt).sqrt().cpu()

    mf, sf = stats(m[fl.reshape(-1).long()], wl.field.reshape(-1).double())
    ok = pl >= 0
    mp, sp = stats(m[pl[ok].long()], wl.attr[:, 0][ok].double())
    return {"map": None, "groups": None, "field_labels": None, "point_labels": None,
            "stats": {"n_field": None, "n_point": None, "lo": None, "hi": None, "mean_field": mf,
                      "std_field": sf, "mean_point": mp, "std_point": sp},
            "pieces": None, "n_pieces": None}
