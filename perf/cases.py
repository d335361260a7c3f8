"""The calls whose speed this repository keeps: whole passes of the conformal Hough hit filter
through its public entry points, on synthetic events of the generator's workloads.

A case is one call as a user's program makes it again and again: a batch of events resident on
the GPU (``run``), a batch in pinned host memory (``HostRunner``), or requests given to the
continuous-batching loop (``Server``). ``prepare`` makes the batch from the seed and allocates the
outputs that such a program keeps; ``run`` is one pass over it.
"""
import dataclasses
import math

import numpy as np
import torch

import gen
import paper_2607_04067_gb300 as hough

# mean hits an event of each workload (measured over its first events)
HITS = {"plain_small": 616, "plain_paper": 1290, "batched": 2022, "served": 2022, "stress": 4720, "paper_1000": 1290}


def _case(name, workload, events, entry="run", peaks=0, **kw):
    """A case with its workload's own parameters, but for those given; peaks: mean stored records an event."""
    cfg = gen.CONFIGS[workload]
    c = {"name": name, "entry": entry, "workload": workload, "events": events, "n_theta": cfg.n_theta,
         "n_rho": cfg.n_rho, "threshold": cfg.threshold, "keep_halfwidth": cfg.keep_halfwidth,
         "max_peaks": cfg.max_peaks, "peak_mode": 0, "rel_num": 0, "rel_den": 1, "nms_radius": 1, "batched": True,
         "checksum": False, "circles": False, "peaks": peaks}
    c.update(kw)
    return c


ITER = {"peak_mode": 1, "rel_num": 1, "rel_den": 2, "nms_radius": 3}


def listed():
    return [
        # one triggered event, filtered as it arrives: the latency of a call
        _case("event_256", "batched", 1, peaks=1620),
        # a hundred small events on a coarse accumulator: a quick-look filter, bound by launch and tail
        _case("small_64", "plain_small", 100, peaks=126),
        # a thousand events of the paper's occupancy: an ordinary batch of an offline job
        _case("paper_256", "plain_paper", 1000, peaks=780),
        # a large batch of mixed occupancies: bulk reprocessing, the headline path
        _case("batched_256", "batched", 20000, peaks=1620),
        # the same with the paper's own peak finder
        _case("batched_256_iter", "batched", 5000, peaks=246, **ITER),
        # high-occupancy events on a finer accumulator, which takes several theta tiles an event
        _case("stress_512", "stress", 1000, peaks=7530),
        _case("stress_512_iter", "stress", 400, peaks=1437, **ITER),
        # the paper's discretisation, 1000 x 1000 (sixteen theta tiles)
        _case("paper_1000", "paper_1000", 1000, peaks=105),
        # the same with the paper's finder and the circles of its peaks: track finding
        _case("paper_1000_iter_circles", "paper_1000", 500, peaks=51, circles=True, **ITER),
        # odd column and row counts (no mirror pairs), one CTA an event, accumulator fingerprints for validation
        _case("odd_101x63", "plain_paper", 500, peaks=289, n_theta=101, n_rho=63, threshold=8, max_peaks=1024,
              batched=False, checksum=True),
        # host buffers in and out: a job whose events come from files
        _case("host_256", "batched", 10000, entry="host", peaks=1620),
        # a burst of requests to the serving loop, results to the callers' buffers: the online filter
        _case("served_256", "served", 4000, entry="served", peaks=1620),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "iter", "iter", "host", "served"])
    if kind in ("host", "served"):
        n = _log_int(rng, 50, 10000 if kind == "host" else 4000)
        c = _case("", rng.choice(["batched", "plain_paper"]) if kind == "host" else "served", n, entry=kind,
                  peaks=1200, keep_halfwidth=rng.choice([0, 1, 1, 2]))
        del c["name"]
        return c
    workload = rng.choice(["plain_small", "plain_paper", "batched", "stress"])
    if rng.random() < 0.5:
        nt = nr = rng.choice([64, 128, 256, 512])
    else:
        nt, nr = _log_int(rng, 48, 1024), _log_int(rng, 48, 1024)
    thr = max(4, gen.CONFIGS[workload].threshold * min(nt, nr) // gen.CONFIGS[workload].n_theta)
    # votes of a batch stay below those of the largest listed batch; the iterative finder and tiles cost more a vote
    votes = 4e9 / (3.0 if kind == "iter" else 1.0) / (1.0 + nt * nr / 131072.0)
    n = _log_int(rng, 1, max(2, min(20000, int(votes / (HITS[workload] * nt)))))
    kw = dict(n_theta=nt, n_rho=nr, threshold=thr, keep_halfwidth=rng.choice([0, 1, 1, 2]),
              max_peaks=4096 if nt * nr <= 65536 else 16384, batched=rng.random() < 0.75,
              checksum=rng.random() < 0.25, peaks=int(0.025 * nt * nr))
    if kind == "iter":
        num, den = rng.choice([(1, 2), (1, 2), (2, 3), (2, 5)])
        kw.update(peak_mode=1, rel_num=num, rel_den=den, nms_radius=rng.choice([1, 2, 3, 3, 4, 6]),
                  peaks=int(0.004 * nt * nr))
    c = _case("", workload, n, **kw)
    del c["name"]
    return c


def _events(case, seed):
    cfg = gen.CONFIGS[case["workload"]]
    cfg = dataclasses.replace(cfg, seed=(cfg.seed + 0x9E3779B97F4A7C15 * (seed + 1)) % (1 << 64))
    return gen.generate(cfg, case["events"], with_truth=False)


def _params(case):
    return hough.params(*(case[k] for k in ("n_theta", "n_rho", "threshold", "keep_halfwidth", "max_peaks")),
                        **{k: case[k] for k in ("peak_mode", "rel_num", "rel_den", "nms_radius")})


def _room(case):
    """Hits that the buffers of such a program have room for: batches differ in their hits."""
    return int(1.1 * HITS[case["workload"]] * case["events"] + 4096 * math.sqrt(case["events"]))


_streams = {}


def _stream():
    """The program's one stream for its filter calls, made on first use."""
    d = torch.cuda.current_device()
    if d not in _streams:
        _streams[d] = torch.cuda.Stream()
    return _streams[d]


class _Loop:
    """A serving loop that closes with the state that holds it."""

    def __init__(self, p):
        self.server = hough.Server(p)

    def __del__(self):
        self.server.close()


def prepare(case, seed):
    ev, p = _events(case, seed), _params(case)
    s = {"case": case, "p": p}
    assert ev.n_hits <= _room(case)
    if case["entry"] == "host":
        n = ev.n_events
        s["xy"], s["off"] = torch.from_numpy(ev.xy).pin_memory(), torch.from_numpy(ev.off).pin_memory()
        s["runner"] = hough.HostRunner(ev.n_hits, n, p, peaks_cap=n * (p.max_peaks if n <= 500 else 2400))
        s["runner"].mask = torch.zeros(_room(case), dtype=torch.uint8).pin_memory()
        s["stream"] = _stream()
    elif case["entry"] == "served":
        n = ev.n_events
        s["xy"], s["off"], s["arrival"] = ev.xy, ev.off, np.zeros(n, np.int64)
        s["mask"] = np.zeros(_room(case), np.uint8)
        s["peaks"] = np.zeros((n, p.max_peaks, 4), np.int16)
        s["results"] = hough.Server.result_array(n)
        s["loop"] = _Loop(p)
    else:
        s["xy"], s["off"] = torch.from_numpy(ev.xy).cuda(), torch.from_numpy(ev.off).cuda()
        s["out"] = hough.alloc_outputs(_room(case), ev.n_events, p, checksum=case["checksum"])
        if case["circles"]:
            s["circles"] = torch.zeros((ev.n_events, p.max_peaks, 4), dtype=torch.float32, device="cuda")
        s["stream"] = _stream()
        s["stream"].wait_stream(torch.cuda.current_stream())
    return s


def run(s):
    case, p = s["case"], s["p"]
    if case["entry"] == "host":
        r = s["runner"]
        flags = r(s["xy"], s["off"], stream=s["stream"])
        return {"npeaks": r.npeaks, "peak_off": r.peak_off, "peaks": r.peaks, "mask": r.mask, "nkept": r.nkept,
                "flags": flags}
    if case["entry"] == "served":
        srv, res = s["loop"].server, s["results"]
        srv.replay(s["xy"], s["off"], s["arrival"], mask_out=s["mask"], peaks_out=s["peaks"], results_out=res)
        srv.drain()
        return {"npeaks": res["npeaks"], "nkept": res["nkept"], "flags": res["status"], "mask": s["mask"],
                "peaks": s["peaks"]}
    out = hough.run(s["xy"], s["off"], p, out=s["out"], batched=case["batched"], stream=s["stream"])
    got = {"npeaks": out.npeaks, "peaks": out.peaks, "mask": out.mask, "nkept": out.nkept, "flags": out.status[:1]}
    if case["checksum"]:
        got["checksum"] = out.checksum
    if case["circles"]:
        got["circles"] = hough.circles(out.npeaks, out.peaks, p, out=s["circles"], stream=s["stream"])
    return got


def work(case):
    """Hits read (8 B) and flags written (1 B), offsets, counts and stored records (and circles) of
    every event; u c + v s and its bin for every hit and theta column."""
    n, hits = case["events"], HITS[case["workload"]] * case["events"]
    stored = min(case["peaks"], case["max_peaks"]) * n
    nbytes = hits * 9 + n * (16 + 8 * case["checksum"]) + stored * (8 + 16 * case["circles"])
    return {"bytes": nbytes, "flops": 4 * hits * case["n_theta"]}


# ---- the circles in 64 bits, from the hits alone, in plain torch ----

_H = 703687442  # rho range of the accumulator in units of 2^-46 per um


def _accumulate(xy, nt, nr):
    """Votes of one event: int64 [nt * nr]."""
    x, y = xy[:, 0].long(), xy[:, 1].long()
    r2 = x * x + y * y
    u = torch.div(x * (1 << 33), r2, rounding_mode="floor")
    v = torch.div(y * (1 << 33), r2, rounding_mode="floor")
    th = (np.arange(nt) + 0.5) * np.pi / nt
    c = torch.from_numpy(np.copysign(np.floor(np.abs(16384 * np.cos(th)) + 0.5), np.cos(th)).astype(np.int64)).to(xy.device)
    s = torch.from_numpy(np.floor(16384 * np.sin(th) + 0.5).astype(np.int64)).to(xy.device)
    t = u[:, None] * c[None, :] + v[:, None] * s[None, :] + _H
    k = torch.div(t * nr, 2 * _H, rounding_mode="floor").clamp_(0, nr - 1)
    cell = (torch.arange(nt, device=xy.device)[None, :] * nr + k).reshape(-1)
    return torch.bincount(cell, minlength=nt * nr)


def _greedy(key, case):
    """Peaks of a batch by extraction: key [events, nt * nr] = votes * cells + (cells - 1 - cell), zeroed where
    suppressed. Returns int64 [events, max_peaks] cells, -1 past each event's peaks."""
    nt, nr, rad, mx = case["n_theta"], case["n_rho"], case["nms_radius"], case["max_peaks"]
    cells, n, dev = nt * nr, key.shape[0], key.device
    need = None
    found = torch.full((n, mx), -1, dtype=torch.int64, device=dev)
    d = torch.arange(-rad, rad + 1, device=dev)
    for q in range(mx):
        top = key.max(dim=1).values
        votes, cell = top // cells, cells - 1 - top % cells
        if need is None:
            need = torch.clamp(-(-(case["rel_num"] * votes) // case["rel_den"]), min=case["threshold"])
        ok = votes >= need
        if not bool(ok.any()):
            break
        found[:, q] = torch.where(ok, cell, torch.full_like(cell, -1))
        j = (cell // nr)[:, None, None] + d[None, :, None]
        k = (cell % nr)[:, None, None] + d[None, None, :]
        inside = (k >= 0) & (k < nr) & ok[:, None, None]
        wrap = (j < 0) | (j >= nt)
        k = torch.where(wrap, nr - 1 - k, k)
        j = j % nt
        e = torch.arange(n, device=dev)[:, None, None].expand_as(k)
        inside = inside.expand_as(k)
        key[e[inside], (j.expand_as(k) * nr + k)[inside]] = 0
    return found


def exact(case, seed):
    if not case.get("circles") or not case["peak_mode"]:
        return None
    ev = _events(case, seed)
    nt, nr, mx, n = case["n_theta"], case["n_rho"], case["max_peaks"], case["events"]
    cells = nt * nr
    out = np.zeros((n, mx, 4))
    xy = torch.from_numpy(ev.xy).cuda()
    rank = cells - 1 - torch.arange(cells, device="cuda")
    for a in range(0, n, 50):
        b = min(n, a + 50)
        key = torch.stack([_accumulate(xy[ev.off[e]:ev.off[e + 1]], nt, nr) * cells + rank for e in range(a, b)])
        cell = _greedy(key, case).cpu().numpy()
        th, k = (cell // nr + 0.5) * np.pi / nt, cell % nr
        rho = (-1.0 + (2.0 * k + 1.0) / nr) * 0.01
        with np.errstate(divide="ignore"):
            rc = 1.0 / np.abs(rho)
            got = np.stack([np.cos(th) / rho, np.sin(th) / rho, rc, 0.3 * rc], axis=-1)
        out[a:b] = np.where((cell >= 0)[..., None], got, 0.0)
    return {"npeaks": None, "peaks": None, "mask": None, "nkept": None, "flags": None, "circles": out}
