"""The work that users of the tracker have it do, as measurable cases.

A case names one use of the library and its sizes:

* ``sector``   one sector's frame through ``Tracker.track`` (host arrays, results as numpy copies);
* ``frame``    a 1 ms full-TPC frame in the float format, host or device resident;
* ``refined``  the same with the two seeding and fit options and drift times instead of z;
* ``tf``       a fixed-format Time Frame of some orbits on a context with the captured path;
* ``chunks``   sub-Time-Frame chunks submitted together, one captured batch;
* ``stream``   several uneven Time Frames in flight from pinned host memory;
* ``compress`` a Time Frame with its compressed form;
* ``decode``   the host decoder on such a compressed form;
* ``digits``   the clusterizer on raw ADC digits;
* ``sort``     the allocation-free binning and sort.

All inputs are the seeded synthetic workloads of ``synth`` at the densities
of the benchmark (50 collisions of 2900 primaries per ms, 50 kHz Pb-Pb).
"""
import ctypes
import math
import weakref

import numpy as np
import torch

from paper_2106_03636_gb300 import o2tpc, synth

DEV = "cuda:0"
CLUSTERS_PER_PRIMARY = 146.0  # of the 1 ms frames, noise included
CLUSTERS_PER_ORBIT = 1.89e6   # of the 50 kHz Pb-Pb Time Frame


def listed():
    return [
        # the smallest call: one sector's collision, as in the single-sector workload (latency, launches)
        {"name": "sector_80", "kind": "sector", "ntracks": 80},
        # a pp-like 400 us chunk alone on a captured context (latency of one graph launch)
        {"name": "chunk_pp", "kind": "chunks", "chunks": 1, "coll": 20, "pp": True},
        # three collisions in pageable host arrays: an ordinary small frame, upload included
        {"name": "frame_3", "kind": "frame", "coll": 3, "ntracks": 2900, "host": True},
        # the 1 ms full-TPC frame of the benchmark, device resident, regular path
        {"name": "frame_50", "kind": "frame", "coll": 50, "ntracks": 2900, "host": False},
        # row step 2 and angle-dependent errors on frames that lost clusters, drift times given
        {"name": "refined_10", "kind": "refined", "coll": 10, "ntracks": 2900, "drop": 0.05},
        # uneven chunks in one captured batch
        {"name": "chunks_8", "kind": "chunks", "chunks": 8, "coll": 20, "pp": False},
        # a quarter of the 128-orbit Time Frame on the captured path: the headline workload
        {"name": "tf_32", "kind": "tf", "orbits": 32},
        # three Time Frames in flight, uploads and downloads overlapped
        {"name": "stream_3x4", "kind": "stream", "tfs": 3, "orbits": 4},
        # a Time Frame stored as its compressed form
        {"name": "compress_4", "kind": "compress", "orbits": 4},
        # reading a compressed Time Frame back
        {"name": "decode_1", "kind": "decode", "orbits": 1},
        # raw ADC digits of 20 collisions (the benchmark's raw workload)
        {"name": "digits_20", "kind": "digits", "coll": 20, "ntracks": 2900},
        # the static sort near its largest size
        {"name": "sort_240k", "kind": "sort", "clusters": 240001},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sector", "frame", "frame", "refined", "tf", "chunks", "stream", "compress", "decode", "digits",
                       "sort"])
    if kind == "sector":
        return {"kind": kind, "ntracks": _log_int(rng, 20, 2000)}
    if kind == "frame":
        return {"kind": kind, "coll": _log_int(rng, 1, 50), "ntracks": _log_int(rng, 150, 2900),
                "host": rng.random() < 0.5}
    if kind == "refined":
        return {"kind": kind, "coll": _log_int(rng, 1, 20), "ntracks": _log_int(rng, 300, 2900),
                "drop": round(rng.uniform(0.0, 0.2), 3)}
    if kind == "tf":
        return {"kind": kind, "orbits": _log_int(rng, 1, 30)}
    if kind == "chunks":
        return {"kind": kind, "chunks": rng.randint(1, 8), "coll": _log_int(rng, 4, 24), "pp": rng.random() < 0.3}
    if kind == "stream":
        return {"kind": kind, "tfs": rng.randint(2, 3), "orbits": _log_int(rng, 1, 6)}
    if kind == "compress":
        return {"kind": kind, "orbits": _log_int(rng, 1, 6)}
    if kind == "decode":
        return {"kind": kind, "orbits": 1, "rate_khz": round(rng.uniform(10.0, 49.0), 1)}
    if kind == "digits":
        return {"kind": kind, "coll": _log_int(rng, 1, 19), "ntracks": _log_int(rng, 150, 2900)}
    return {"kind": kind, "clusters": _log_int(rng, 500, 262144)}


# ---------------------------------------------------------------- contexts
_contexts = weakref.WeakValueDictionary()


def _context(**cfg):
    """The long-lived context a program keeps for its configuration."""
    key = tuple(sorted(cfg.items()))
    trk = _contexts.get(key)
    if trk is None:
        trk = o2tpc.Tracker(**cfg)
        _contexts[key] = trk
    return trk


class _State:
    """What the program has in hand: inputs and context."""

    def __init__(self, kind, **kw):
        self.kind = kind
        self.__dict__.update(kw)


_FIELDS = {  # field: (type, values per track)
    "x": (np.float32, 1), "alpha": (np.float32, 1), "par": (np.float32, 5), "cov": (np.float32, 15),
    "chi2": (np.float32, 1), "ndf": (np.int32, 1), "sector": (np.uint8, 1), "flags": (np.uint8, 1),
    "zeta_ref": (np.int32, 1), "t0": (np.float32, 1), "t0_err": (np.float32, 1), "t0_lo": (np.float32, 1),
    "t0_hi": (np.float32, 1), "mate": (np.int32, 1), "collision": (np.int32, 1),
}
_CHUNK_FIELDS = ("par", "cov", "chi2", "t0", "collision")  # what the chunk user takes (7 arrays a chunk)


def _buffers(clusters, fields=tuple(_FIELDS), ctf=False):
    """The program's own arrays for one frame's results, with room for `clusters` (a track holds at least ten, and
    over thirty on average); zero behind the results."""
    tracks = clusters // 30 + 64
    out = {"offsets": np.zeros(tracks + 1, np.int64), "cluster_idx": np.zeros(clusters, np.int32)}
    for f in fields:
        dt, per = _FIELDS[f]
        out[f] = np.zeros(per * tracks, dt)
    if ctf:
        out["ctf"] = np.zeros(3 * clusters + 100000, np.uint8)
    return {k: torch.from_numpy(v) for k, v in out.items()}


def _put(dst, ptr, n):
    """Copies n values of a result into the program's array (on all host cores, as torch copies)."""
    if n:
        size = n * dst.element_size()
        mem = (ctypes.c_char * size).from_address(ctypes.cast(ptr, ctypes.c_void_p).value)
        dst[:n].copy_(torch.frombuffer(mem, dtype=dst.dtype))


def _take(trk, res, out):
    """A polled result into the program's arrays; then it goes back to the library."""
    r = res.contents
    status, n = int(r.status), int(r.n_tracks)
    if status == o2tpc.O2TPC_OK:
        ncl = int(r.offsets[n])
        for f, dst in out.items():
            if f == "offsets":
                _put(dst, r.offsets, n + 1)
            elif f == "cluster_idx":
                _put(dst, r.cluster_idx, ncl)
            elif f == "ctf":
                _put(dst, r.ctf, int(r.ctf_bytes))
            else:
                _put(dst, getattr(r, f), _FIELDS[f][1] * n)
    o2tpc.o2tpc_result_release(trk.ctx, res)
    if status != o2tpc.O2TPC_OK:
        raise o2tpc.O2TPCError(status, "tracking")
    return n


def _on_device(tf):
    names = ("packed",) if tf.fmt == synth.FMT_FIXED else ("sector", "row", "y", "z" if tf.z is not None else "time")
    return {k: torch.from_numpy(getattr(tf, k)).to(DEV) for k in names}


# ------------------------------------------------------------------ inputs
def _frame(case, seed, fmt, **kw):
    return synth.full_tpc_1ms(seed=seed, n_coll=case["coll"], ntracks=case["ntracks"], fmt=fmt, with_truth=False, **kw)


def _digits(tf, seed):
    """Raw digits of a fixed-format frame, by the recipe of ``synth.digits_from``
    (5 x 5 cells around each cluster, Gaussian spread, noise, zero
    suppression), deposited on the GPU: (sector, row, pad, time, adc)."""
    rec = torch.from_numpy(tf.packed).to(DEV)
    w = rec.view(torch.int32)
    t64 = w[:, 0].double()
    p64 = (w[:, 1] & 0xFFFF).double()
    q = 20.0 + ((w[:, 1] >> 16) & 0xFFFF).double() / 6.0
    sr = rec[:, 9].long() * 152 + rec[:, 8].long()
    pc, tc = (p64 / 64.0), (t64 / 64.0)
    p0, t0 = pc.floor().long() - 2, tc.floor().long() - 2

    def shares(centre, first, sigma):
        edges = first.double()[:, None] + torch.arange(6, device=DEV)[None, :]
        return torch.special.ndtr((edges - centre[:, None]) / sigma).diff(dim=1).float()

    sp, st = shares(pc, p0, 0.7), shares(tc, t0, 0.8)
    keys, vals = [], []
    for i in range(5):
        for j in range(5):
            p, t = p0 + i, t0 + j
            ok = (p >= 0) & (p < 256) & (t >= 0)
            keys.append(((sr << 40) | (t << 8) | p)[ok])
            vals.append((q.float() * sp[:, i] * st[:, j])[ok])
    cells, where = torch.unique(torch.cat(keys), return_inverse=True)
    charge = torch.zeros(len(cells), dtype=torch.float64, device=DEV).index_add_(0, where, torch.cat(vals).double())
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    adc = (charge.float() + 0.6 * torch.randn(len(cells), generator=g, device=DEV)).round().clamp_(max=1023.0)
    keep = adc >= 2
    cells, adc = cells[keep], adc[keep]
    sr = cells >> 40
    return {"sector": (sr // 152).to(torch.uint8), "row": (sr % 152).to(torch.uint8),
            "pad": (cells & 0xFF).to(torch.uint8), "time": ((cells >> 8) & 0xFFFFFFFF).to(torch.int32),
            "adc": adc.to(torch.int16)}


def _room(case):
    """Clusters that contexts and result arrays have room for: three spreads of the falling multiplicity above the
    expected number, in whole quarters of a million; where the multiplicities are fixed, a margin."""
    n = _clusters(case)
    if case["kind"] in ("sector", "frame", "refined") or case.get("pp"):
        return int((2.0 if n < 1e6 else 1.15) * n) + 2000
    return int(math.ceil((n + 3.0 * math.sqrt(n * 9.0e5)) / 250000.0) + 1) * 250000


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sector":
        tf = synth.single_sector(seed=seed, ntracks=case["ntracks"], with_truth=False)
        return _State(kind, trk=_context(), tf=tf, out=_buffers(_room(case)))
    if kind == "frame":
        tf = _frame(case, seed, synth.FMT_FLOAT)
        arrays = None if case["host"] else _on_device(tf)
        return _State(kind, trk=_context(), tfs=[tf], arrays=[arrays], host=case["host"], out=[_buffers(_room(case))])
    if kind == "refined":
        tf = synth.float_time_from_fixed(_frame(case, seed, synth.FMT_FIXED, row_drop=case["drop"],
                                                angular_errors=True))
        trk = _context(flags=o2tpc.O2TPC_FLAG_ROW_STEP2 | o2tpc.O2TPC_FLAG_ANGULAR_ERRORS)
        return _State(kind, trk=trk, tfs=[tf], arrays=[_on_device(tf)], host=False, out=[_buffers(_room(case))])
    if kind == "tf":
        tf = synth.full_tf(seed=seed, orbits=case["orbits"], with_truth=False)
        trk = _context(graph_max_clusters=_room(case), graph_max_tfs=1)
        return _State(kind, trk=trk, tfs=[tf], arrays=[_on_device(tf)], host=False, out=[_buffers(_room(case))])
    if kind == "chunks":
        rng = np.random.default_rng(seed)
        tfs = []
        for c in range(case["chunks"]):
            k = max(1, int(rng.poisson(case["coll"])))
            t0 = np.sort(rng.uniform(0.0, 400.0, k))
            ntr = (np.full(k, 11, np.int32) if case["pp"] or c % 4 == 3
                   else np.rint(1.8 * synth.falling_multiplicity(rng, k)).astype(np.int32))
            tfs.append(synth.generate(seed=seed * 1000 + c, t0=t0, ntracks=ntr, zvtx_sigma=5.0, t_window=400.0,
                                      fmt=synth.FMT_FIXED, with_truth=False))
        trk = _context(graph_max_clusters=_room(case), graph_max_tfs=case["chunks"])
        one = _room(dict(case, chunks=1))
        return _State(kind, trk=trk, tfs=tfs, arrays=[_on_device(t) for t in tfs], host=False,
                      out=[_buffers(one, _CHUNK_FIELDS) for _ in tfs])
    if kind == "stream":
        tfs = [synth.full_tf(seed=seed * 10 + i, orbits=max(1, case["orbits"] - i), with_truth=False)
               for i in range(case["tfs"])]
        arrays = [{"packed": torch.from_numpy(t.packed).pin_memory()} for t in tfs]
        room = _room({"kind": "tf", "orbits": case["orbits"]})
        trk = _context(flags=o2tpc.O2TPC_FLAG_NO_BATCHING, graph_max_clusters=room, graph_max_tfs=1)
        return _State(kind, trk=trk, tfs=tfs, arrays=arrays, host=True, out=[_buffers(room) for _ in tfs])
    if kind in ("compress", "decode"):
        tf = synth.full_tf(seed=seed, orbits=case["orbits"], rate_khz=case.get("rate_khz", synth.PBPB_RATE_KHZ),
                           with_truth=False)
        trk = _context(flags=o2tpc.O2TPC_FLAG_COMPRESS)
        if kind == "compress":
            return _State(kind, trk=trk, tfs=[tf], arrays=[_on_device(tf)], host=False,
                          out=[_buffers(_room(case), ctf=True)])
        n = _room(case)
        out = {k: torch.zeros(n, dtype=torch.int32) for k in ("sector", "row", "y", "zeta")}
        out["track_len"] = torch.zeros(n // 30 + 64, dtype=torch.int32)
        out["records"] = torch.zeros((n, 12), dtype=torch.uint8)
        return _State(kind, blob=trk.track(tf)["ctf"], out=out)
    if kind == "digits":
        room = int(1.3 * _clusters(case)) + 20000
        return _State(kind, digits=_digits(_frame(case, seed, synth.FMT_FIXED), seed),
                      out=torch.zeros((room, 12), dtype=torch.uint8, device=DEV))
    tf = synth.single_sector(seed=seed, ntracks=5400, with_truth=False)
    n = case["clusters"]
    pick = np.random.default_rng(seed).permutation(tf.n)[:n]
    sector = (np.random.default_rng(seed + 1).integers(0, 36, n)).astype(np.uint8)
    arrays = {"sector": sector, "row": tf.row[pick], "y": tf.y[pick],
              "z": np.where(sector < 18, tf.z[pick], -tf.z[pick]).astype(np.float32)}
    host = {k: np.ascontiguousarray(v) for k, v in arrays.items()}
    dev = {k: torch.from_numpy(v).to(DEV) for k, v in host.items()}
    t = synth.TimeFrame(n=n, fmt=synth.FMT_FLOAT, sector=host["sector"], row=host["row"], y=host["y"], z=host["z"])
    cap = n // 4 + 46 * 5472 + 2
    out = {"sorted_orig": torch.zeros(n, dtype=torch.int32, device=DEV),
           "sorted_yz": torch.zeros((n, 2), dtype=torch.int32, device=DEV),
           "row_grid": torch.zeros((5472, 8), dtype=torch.int32, device=DEV),
           "cell_start": torch.zeros(cap, dtype=torch.int32, device=DEV)}
    return _State(kind, tf=o2tpc.make_tf(t, o2tpc.O2TPC_LOC_DEVICE, dev), arrays=dev, out=out, cap=cap)


# -------------------------------------------------------------------- pass
def run(state):
    kind, out = state.kind, state.out
    if kind == "sector":
        r = state.trk.track(state.tf)
        for f, dst in out.items():
            v = r[f].reshape(-1)
            dst.numpy()[: len(v)] = v
        return {"n": r["n_tracks"], **out}
    if kind == "decode":
        r = o2tpc.ctf_decode(state.blob)
        for f, dst in out.items():
            dst[: len(r[f])].copy_(torch.from_numpy(r[f].view(np.uint8 if f == "records" else np.int32)))
        return {"n": len(r["records"]), **out}
    if kind == "digits":
        rc, records, n = o2tpc.clusterize(state.digits)
        if rc != o2tpc.O2TPC_OK:
            raise o2tpc.O2TPCError(rc, "o2tpc_clusterize")
        out[:n].copy_(records)
        return {"n": n, "records": out}
    if kind == "sort":
        rc = o2tpc.o2tpc_sort_tf_static(state.tf, synth.VDRIFT, out["sorted_orig"].data_ptr(),
                                        out["sorted_yz"].data_ptr(), out["row_grid"].data_ptr(),
                                        out["cell_start"].data_ptr(), state.cap,
                                        torch.cuda.current_stream().cuda_stream)
        if rc != o2tpc.O2TPC_OK:
            raise o2tpc.O2TPCError(rc, "o2tpc_sort_tf_static")
        return out
    # the C-ABI cycle: submit, wait, take the results, give them back
    loc = o2tpc.O2TPC_LOC_HOST if state.host else o2tpc.O2TPC_LOC_DEVICE
    ts = [o2tpc.make_tf(tf, loc, a) for tf, a in zip(state.tfs, state.arrays)]
    rc, tickets = o2tpc.o2tpc_submit_many(state.trk.ctx, ts)
    if rc != o2tpc.O2TPC_OK:
        raise o2tpc.O2TPCError(rc, "o2tpc_submit_many")
    got = []
    for ticket, dst in zip(tickets, out):
        rc, res = o2tpc.o2tpc_poll(state.trk.ctx, ticket, -1)
        if rc != o2tpc.O2TPC_OK:
            raise o2tpc.O2TPCError(rc, "o2tpc_poll")
        got.append(dict(dst, n=_take(state.trk, res, dst)))
    return got


# -------------------------------------------------------------------- work
def _clusters(case):
    """Expected clusters of a case."""
    kind = case["kind"]
    if kind == "sector":
        return 62.0 * case["ntracks"]
    if kind in ("frame", "refined", "digits"):
        return CLUSTERS_PER_PRIMARY * case["coll"] * case["ntracks"] * (1.0 - case.get("drop", 0.0))
    if kind == "chunks":
        c = case["chunks"]
        pp = c if case["pp"] else c // 4
        return case["coll"] * (110000.0 * (c - pp) + 1500.0 * pp)
    if kind == "tf":
        return CLUSTERS_PER_ORBIT * case["orbits"]
    if kind == "stream":
        return CLUSTERS_PER_ORBIT * sum(max(1, case["orbits"] - i) for i in range(case["tfs"]))
    if kind in ("compress", "decode"):
        return CLUSTERS_PER_ORBIT * case["orbits"] * case.get("rate_khz", synth.PBPB_RATE_KHZ) / synth.PBPB_RATE_KHZ
    return float(case["clusters"])


def work(case):
    n = _clusters(case)
    kind = case["kind"]
    if kind == "decode":  # 2.34 bytes read a cluster; four integers and a 12-byte record written
        return {"bytes": (2.34 + 28.0) * n, "flops": 0.0}
    if kind == "digits":  # 9-byte digits, about ten a cluster; 12-byte records, about one a cluster
        return {"bytes": (9.0 * 10.0 + 12.0) * n, "flops": 0.0}
    if kind == "sort":  # 10 bytes read; index and coordinates written
        return {"bytes": (10.0 + 12.0) * n, "flops": 0.0}
    # the clusters read; an index a track cluster and about 150 bytes a track (0.7 % of the clusters) written;
    # every track cluster fitted once (transport and update of five parameters and their covariance)
    read = 10.0 if kind in ("sector", "frame", "refined") else 12.0
    written = 4.0 + 1.0 + (2.34 if kind == "compress" else 0.0)
    return {"bytes": (read + written) * n, "flops": 300.0 * n}


# ------------------------------------------------------------------- exact
def exact(case, seed):
    """In 64 bits with numpy: the sort and the clusterizer (whole numbers).
    The tracker's floating outputs follow from its whole pattern recognition,
    which takes minutes in plain numpy: none."""
    if case["kind"] == "sort":
        s = prepare(case, seed)
        a = {k: v.cpu().numpy() for k, v in s.arrays.items()}
        row = a["sector"].astype(np.int64) * 152 + a["row"]
        y = np.rint(a["y"] * np.float32(160)).astype(np.int64)
        d = np.where(a["sector"] < 18, np.float32(250) - a["z"], np.float32(250) + a["z"]).astype(np.float32)
        z = np.rint(d * np.float32(1.0 / (0.003125 * synth.VDRIFT))).astype(np.int64)
        pads = np.floor(2.0 * (85.0 + np.arange(152) * 160.0 / 151.0) * math.tan(math.radians(10.0)) / 0.4)
        half = 32 * np.tile(pads.astype(np.int64), 36)
        ny = np.maximum(1, (2 * half + 319) // 320)
        cnt = np.bincount(row, minlength=5472)
        nz = np.clip((cnt + 4 * ny - 1) // (4 * ny), 1, 1 << 20)
        zmin, zmax = np.full(5472, 1 << 40), np.full(5472, -(1 << 40))
        np.minimum.at(zmin, row, z)
        np.maximum.at(zmax, row, z)
        some = cnt > 0
        cz = np.where(some, (zmax - zmin + 1 + nz - 1) // nz, 1)
        zmin = np.where(some, zmin, 0)
        iy = np.clip((y + half[row]) // 320, 0, ny[row] - 1)
        iz = (z - zmin[row]) // cz[row]
        base = np.concatenate([[0], np.cumsum(ny * nz)])
        cell = base[row] + iz * ny[row] + iy
        order = np.argsort(cell, kind="stable")
        start = np.concatenate([[0], np.cumsum(cnt)])[:-1]
        grid = np.stack([start, cnt, base[:-1], ny, nz, cz, zmin, np.zeros(5472, np.int64)], axis=1)
        cs = np.concatenate([[0], np.cumsum(np.bincount(cell, minlength=base[-1]))])
        out = np.zeros(s.cap, np.int32)
        out[: len(cs)] = cs
        return {"sorted_orig": order.astype(np.int32), "sorted_yz": np.stack([y[order], z[order]], 1).astype(np.int32),
                "row_grid": grid.astype(np.int32), "cell_start": out}
    if case["kind"] == "digits":
        d = {k: v.cpu().numpy().astype(np.int64) for k, v in _digits(_frame(case, seed, synth.FMT_FIXED), seed).items()}
        if len(d["adc"]) > 20_000_000:
            return None
        key = ((d["sector"] * 152 + d["row"]) << 40) | (d["time"] << 8) | d["pad"]
        adc, pad, tim = d["adc"], d["pad"], d["time"]
        peak = adc >= 3
        q, sp, st = adc.copy(), adc * (64 * pad + 32), adc * (64 * tim + 32)
        for dt in (-1, 0, 1):
            for dp in (-1, 0, 1):
                if dt == 0 and dp == 0:
                    continue
                ok = (pad + dp >= 0) & (pad + dp <= 255) & (tim + dt >= 0)
                want = key + 256 * dt + dp
                j = np.minimum(np.searchsorted(key, want), len(key) - 1)
                b = np.where(ok & (key[j] == want), adc[j], 0)
                there = b > 0
                before = dt < 0 or (dt == 0 and dp < 0)
                peak &= ~there | ((adc > b) if before else (adc >= b))
                q += b
                sp += b * (64 * (pad + dp) + 32)
                st += b * (64 * (tim + dt) + 32)
        i = np.flatnonzero(peak)
        rec = np.zeros((len(i), 3), np.uint32)
        rec[:, 0] = (2 * st[i] + q[i]) // (2 * q[i])
        rec[:, 1] = (((2 * sp[i] + q[i]) // (2 * q[i])) & 0xFFFF) | (np.minimum(q[i], 65535) << 16)
        rec[:, 2] = d["row"][i] | (d["sector"][i] << 8)
        room = np.zeros((int(1.3 * _clusters(case)) + 20000, 12), np.uint8)
        room[: len(i)] = rec.view(np.uint8).reshape(-1, 12)
        return {"n": len(i), "records": room}
    return None
