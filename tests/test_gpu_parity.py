"""GPU parity: the CUDA path through the C ABI against the CPU oracle, element by element.

Integer path, so the bar is bit-exact equality of accumulators, peak lists, masks,
kept counts and accumulator checksums.
"""
import os

import numpy as np
import pytest

import gen
import oracle
from parity_util import assert_event_outputs_equal, peaks_np, sub_batch, to_np

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

THREADS = max(1, os.cpu_count() or 1)


@pytest.fixture(scope="module")
def h():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2607_04067_gb300 as hough
    hough.load()
    return hough


def cfg_params(h, cfg, **kw):
    return h.params(cfg.n_theta, cfg.n_rho, cfg.threshold, cfg.keep_halfwidth, cfg.max_peaks, **kw)


def dev(ev):
    return torch.from_numpy(ev.xy).cuda(), torch.from_numpy(ev.off).cuda()


def oracle_of(cfg, ev, with_acc=False, max_peaks=None, **kw):
    p = oracle.params(kw.get("n_theta", cfg.n_theta), kw.get("n_rho", cfg.n_rho), kw.get("threshold", cfg.threshold),
                      kw.get("keep_halfwidth", cfg.keep_halfwidth), max_peaks or cfg.max_peaks)
    return oracle.run(ev.xy, ev.off, p, with_acc=with_acc, threads=THREADS)


# ---------------------------------------------------------------- stepwise path

def test_stepwise_matches_oracle(h):
    cfg = gen.CONFIGS["plain_small"]
    ev = gen.generate(cfg)
    ref = oracle_of(cfg, ev, with_acc=True)
    xy, off = dev(ev)
    p = cfg_params(h, cfg)
    st = h.new_status()
    uq, vq = h.map_hits(xy, off, st)
    exp_u = np.array([oracle.map_hit(x, y)[1] for x, y in ev.xy[:2000]])
    exp_v = np.array([oracle.map_hit(x, y)[2] for x, y in ev.xy[:2000]])
    assert np.array_equal(to_np(uq)[:2000], exp_u) and np.array_equal(to_np(vq)[:2000], exp_v)
    acc = h.vote(uq, vq, off, p, st)
    assert np.array_equal(to_np(acc), ref.acc)
    npk, pk = h.peaks(acc, p, st)
    mask, nkept = h.select(uq, vq, off, p, npk, pk, st)
    assert h.status(st) == 0
    assert_event_outputs_equal(ref, npk, pk, mask, nkept, ev.off)


def test_stepwise_vote_tiled_large_accumulator(h):
    cfg = gen.CONFIGS["stress"]
    ev = gen.generate(cfg, 6)
    ref = oracle_of(cfg, ev, with_acc=True)
    xy, off = dev(ev)
    p = cfg_params(h, cfg)
    st = h.new_status()
    uq, vq = h.map_hits(xy, off, st)
    acc = h.vote(uq, vq, off, p, st)
    assert np.array_equal(to_np(acc), ref.acc)
    npk, pk = h.peaks(acc, p, st)
    mask, nkept = h.select(uq, vq, off, p, npk, pk, st)
    assert h.status(st) == 0
    assert_event_outputs_equal(ref, npk, pk, mask, nkept, ev.off)


# ---------------------------------------------------------------- fused path

@pytest.mark.parametrize("name,n", [("plain_small", None), ("plain_paper", None), ("batched", 400), ("stress", 24),
                                    ("paper_1000", 200)])
@pytest.mark.parametrize("batched", [False, True])
def test_fused_matches_oracle(h, name, n, batched):
    cfg = gen.CONFIGS[name]
    ev = gen.generate(cfg, n)
    ref = oracle_of(cfg, ev)
    xy, off = dev(ev)
    out = h.run(xy, off, cfg_params(h, cfg), checksum=True, batched=batched)
    assert h.status(out.status) == 0
    assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off, checksum=out.checksum)


@pytest.mark.parametrize("n_theta,n_rho,tiles,block", [
    (256, 256, 2, 0), (256, 256, 4, 0), (256, 256, 8, 0), (256, 256, 1, 256), (256, 256, 1, 1024),
    (256, 256, 3, 0), (64, 64, 2, 0), (64, 64, 1, 64), (100, 63, 1, 0), (100, 63, 3, 0), (4, 4, 1, 0),
    (1024, 1024, 0, 0), (1000, 1000, 0, 0), (37, 257, 2, 0),
    (512, 512, 4, 0), (512, 512, 8, 0), (128, 64, 2, 0), (128, 63, 2, 0)])
def test_shapes_and_tiles(h, n_theta, n_rho, tiles, block):
    cfg = gen.CONFIGS["plain_paper"]
    ev = gen.generate(cfg, 40)
    thr = max(2, cfg.threshold * min(n_theta, n_rho) // 256)
    ref = oracle.run(ev.xy, ev.off, oracle.params(n_theta, n_rho, thr, 1, 4096), threads=THREADS)
    xy, off = dev(ev)
    for batched in (False, True):
        out = h.run(xy, off, h.params(n_theta, n_rho, thr, 1, 4096, theta_tiles=tiles, block=block), checksum=True,
                    batched=batched)
        assert h.status(out.status) == 0
        assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off, checksum=out.checksum)


def test_checksum_off_gives_same_results(h):
    cfg = gen.CONFIGS["plain_paper"]
    ev = gen.generate(cfg, 50)
    xy, off = dev(ev)
    a = h.run(xy, off, cfg_params(h, cfg), checksum=True, batched=True)
    b = h.run(xy, off, cfg_params(h, cfg), checksum=False, batched=True)
    assert torch.equal(a.mask, b.mask) and torch.equal(a.npeaks, b.npeaks) and torch.equal(a.nkept, b.nkept)
    assert np.array_equal(peaks_np(a.peaks), peaks_np(b.peaks))


# ---------------------------------------------------------------- full-size workloads, sampled

@pytest.mark.parametrize("name,sample", [("batched", 300), ("stress", 60), ("paper_1000", 100)])
def test_full_size_sampled(h, name, sample):
    """Whole workload in the launch configuration the benchmark times (batched, no checksum),
    then the oracle recomputes a random sample of events one by one."""
    cfg = gen.CONFIGS[name]
    ev = gen.generate(cfg, with_truth=False)
    xy, off = dev(ev)
    p = cfg_params(h, cfg)
    out = h.run(xy, off, p, checksum=False, batched=True)
    assert h.status(out.status) == 0
    rng = np.random.default_rng(1)
    events = np.sort(rng.choice(ev.n_events, size=sample, replace=False))
    events[0] = 0
    events[-1] = ev.n_events - 1
    sxy, soff = sub_batch(ev.xy, ev.off, events)
    ref = oracle.run(sxy, soff, oracle.params(cfg.n_theta, cfg.n_rho, cfg.threshold, cfg.keep_halfwidth,
                                              cfg.max_peaks), threads=THREADS)
    assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off, events=events)
    # properties over every event
    nk = to_np(out.nkept)
    m = to_np(out.mask)
    csum = np.concatenate([[0], np.cumsum(m.astype(np.int64))])
    assert np.array_equal(csum[ev.off[1:]] - csum[ev.off[:-1]], nk)
    assert np.all(to_np(out.npeaks) <= cfg.max_peaks)
    assert set(np.unique(m)) <= {0, 1}
    # the shape the benchmark times: tuned on the first 10,000 events, whole batch again
    ns = min(ev.n_events, 10000)
    pt, _ = h.autotune(xy[: int(ev.off[ns])], off[: ns + 1], p)
    out2 = h.run(xy, off, pt, checksum=False, batched=True)
    assert h.status(out2.status) == 0
    assert torch.equal(out2.npeaks, out.npeaks) and torch.equal(out2.nkept, out.nkept)
    assert torch.equal(out2.mask, out.mask) and torch.equal(out2.peaks, out.peaks)


def test_full_size_sampled_iterative(h):
    """The batched workload (100,000 events) with the paper's iterative finder in the
    benchmark's configuration (half the maximum, radius 3, autotuned shape); the oracle
    recomputes a random sample of events one by one."""
    cfg = gen.CONFIGS["batched"]
    ev = gen.generate(cfg, with_truth=False)
    xy, off = dev(ev)
    kw = dict(peak_mode=1, rel_num=1, rel_den=2, nms_radius=3)
    p = cfg_params(h, cfg, **kw)
    p, _ = h.autotune(xy[: int(ev.off[10000])], off[:10001], p)
    out = h.run(xy, off, p, checksum=False, batched=True)
    assert h.status(out.status) == 0
    rng = np.random.default_rng(2)
    events = np.sort(rng.choice(ev.n_events, size=120, replace=False))
    events[0] = 0
    events[-1] = ev.n_events - 1
    sxy, soff = sub_batch(ev.xy, ev.off, events)
    ref = oracle.run(sxy, soff, oracle.params(cfg.n_theta, cfg.n_rho, cfg.threshold, cfg.keep_halfwidth,
                                              cfg.max_peaks, **kw), threads=THREADS)
    assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off, events=events)


# ---------------------------------------------------------------- edge cases

def test_empty_batch_and_empty_events(h):
    p = h.params(64, 64, 2)
    xy = torch.zeros((0, 2), dtype=torch.int32, device="cuda")
    off = torch.zeros(1, dtype=torch.int64, device="cuda")
    for batched in (False, True):
        out = h.run(xy, off, p, batched=batched)
        assert h.status(out.status) == 0
    ev = gen.generate("plain_small", 5)
    parts = [gen.Events(np.zeros((0, 2), np.int32), np.zeros(1, np.int64), None), ev,
             gen.Events(np.zeros((0, 2), np.int32), np.zeros(2, np.int64), None)]
    cat = gen.concat(parts)
    ref = oracle.run(cat.xy, cat.off, oracle.params(64, 64, 12), threads=THREADS)
    xy, off = dev(cat)
    for batched in (False, True):
        out = h.run(xy, off, h.params(64, 64, 12), checksum=True, batched=batched)
        assert h.status(out.status) == 0
        assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, cat.off, checksum=out.checksum)


def test_bad_hits_and_small_radii(h):
    """r = 0 and out-of-range hits are skipped and flagged; hits inside r ~ 195 mm take the
    int64 path (rho clamped to the edge bins)."""
    rng = np.random.default_rng(9)
    ev = gen.generate("plain_paper", 30)
    xy = ev.xy.copy()
    idx = rng.choice(len(xy), 60, replace=False)
    xy[idx[:10]] = 0
    xy[idx[10:15], 0] = 2 ** 24 + 5
    small = rng.integers(-150000, 150000, size=(45, 2)).astype(np.int32)
    xy[idx[15:]] = small
    ref = oracle.run(xy, ev.off, oracle.params(256, 256, 16, 1, 4096), threads=THREADS)
    assert ref.status == oracle.F_BAD_HIT
    t_xy, off = torch.from_numpy(xy).cuda(), torch.from_numpy(ev.off).cuda()
    for batched in (False, True):
        for tiles in (1, 2):
            out = h.run(t_xy, off, h.params(256, 256, 16, 1, 4096, theta_tiles=tiles), checksum=True, batched=batched)
            assert h.status(out.status) == h.F_BAD_HIT
            assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off,
                                       checksum=out.checksum)
    st = h.new_status()
    uq, vq = h.map_hits(t_xy, off, st)
    assert h.status(st) == h.F_BAD_HIT
    u = to_np(uq)
    assert np.all(u[idx[:15]] == np.iinfo(np.int64).min)


def test_coordinates_of_any_int32(h):
    """Coordinates up to the ends of int32 are bad hits like any other beyond 2^24, and the last good ones are good."""
    ev = gen.generate("plain_small", 3)
    ends = [-2 ** 31, -2 ** 31 + 1, -2 ** 31 + 2 ** 24, -2 ** 24 - 1, 2 ** 24 + 1, 2 ** 31 - 2 ** 24, 2 ** 31 - 1]
    bad = [(c, 5) for c in ends] + [(-5, c) for c in ends] + [(c, d) for c in ends for d in ends]
    xy = np.concatenate([ev.xy, np.array(bad + [(2 ** 24, -2 ** 24), (-2 ** 24, 2 ** 24)], np.int64).astype(np.int32)])
    off = np.append(ev.off, len(xy))
    ref = oracle.run(xy, off, oracle.params(64, 64, 12, 1, 256), threads=THREADS)
    t_xy, t_off = torch.from_numpy(xy).cuda(), torch.from_numpy(off).cuda()
    out = h.run(t_xy, t_off, h.params(64, 64, 12, 1, 256), checksum=True)
    assert h.status(out.status) == ref.status == h.F_BAD_HIT
    assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, off, checksum=out.checksum)
    uq, _ = h.map_hits(t_xy, t_off, h.new_status())
    assert np.array_equal(to_np(uq)[len(ev.xy):] == np.iinfo(np.int64).min, [True] * len(bad) + [False] * 2)


def test_map_edges(h):
    """The map's quotients at radii up to 400 mm (the float estimate gives way to plain division at 2^20, 8 mm), on the axes, at the largest coordinates and at the smallest radii, against Python integers."""
    rng = np.random.default_rng(12)
    r = np.concatenate([np.full(3000, 131072), rng.uniform(1, 400000, 3000), rng.uniform(4e5, 2 ** 24, 2000)])
    a = rng.uniform(0, 2 * np.pi, len(r))
    xy = np.stack([np.rint(r * np.cos(a)), np.rint(r * np.sin(a))], axis=1).astype(np.int32)
    xy[:3000] += rng.integers(-3, 4, size=(3000, 2)).astype(np.int32)
    xy = np.concatenate([xy, [[1, 0], [0, -1], [2 ** 24, 2 ** 24], [-2 ** 24, 1], [131072, 0], [0, 131073], [7, -7],
                              [3 * 5 * 7 * 11, 4 * 5 * 7 * 11]]]).astype(np.int32)
    xy = np.ascontiguousarray(xy[np.any(xy != 0, axis=1)])
    off = torch.tensor([0, len(xy)], dtype=torch.int64, device="cuda")
    st = h.new_status()
    uq, vq = h.map_hits(torch.from_numpy(xy).cuda(), off, st)
    assert h.status(st) == 0
    exp = [((int(x) << 33) // (int(x) ** 2 + int(y) ** 2), (int(y) << 33) // (int(x) ** 2 + int(y) ** 2)) for x, y in xy]
    assert to_np(uq).tolist() == [e[0] for e in exp] and to_np(vq).tolist() == [e[1] for e in exp]


@pytest.mark.parametrize("name,n,tiles,grab", [("paper_1000", 200, 16, 0), ("paper_1000", 40, 16, 5), ("stress", 310, 4, 0),
                                               ("batched", 700, 1, 3), ("plain_paper", 5, 2, 0)])
def test_queue_runs(h, name, n, tiles, grab):
    """Runs of tiles from the queue with their hits staged once, single items at the end, runs across events."""
    cfg = gen.CONFIGS[name]
    ev = gen.generate(cfg, n)
    ref = oracle_of(cfg, ev)
    xy, off = dev(ev)
    out = h.run(xy, off, cfg_params(h, cfg, theta_tiles=tiles, events_per_cta=grab), checksum=True, batched=True)
    assert h.status(out.status) == 0
    assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off, checksum=out.checksum)


def test_all_hits_small_radius_event(h):
    """Every hit on the int64 path, across several staging chunks."""
    rng = np.random.default_rng(4)
    xy = rng.integers(-190000, 190000, size=(9000, 2)).astype(np.int32)
    xy[np.all(xy == 0, axis=1)] = 1
    off = np.array([0, 3000, 9000], np.int64)
    ref = oracle.run(xy, off, oracle.params(128, 128, 40, 1, 8192), threads=THREADS)
    t_xy, t_off = torch.from_numpy(xy).cuda(), torch.from_numpy(off).cuda()
    for tiles in (1, 2):
        out = h.run(t_xy, t_off, h.params(128, 128, 40, 1, 8192, theta_tiles=tiles), checksum=True, batched=True)
        assert h.status(out.status) == 0
        assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, off, checksum=out.checksum)


def test_large_event_chunks_and_too_large(h):
    """An event bigger than one staging chunk, and one above 32767 hits (skipped, flagged)."""
    ev = gen.generate("stress", 8)
    big = np.tile(ev.xy, (1, 1))[:32767]
    huge = np.concatenate([ev.xy] * 2)[:32768]
    xy = np.concatenate([big, huge, ev.xy[:500]])
    off = np.array([0, len(big), len(big) + len(huge), len(xy)], np.int64)
    ref = oracle.run(xy, off, oracle.params(256, 256, 200, 1, 4096), threads=THREADS)
    assert ref.status == oracle.F_EVENT_TOO_LARGE
    t_xy, t_off = torch.from_numpy(xy).cuda(), torch.from_numpy(off).cuda()
    for tiles in (1, 4):
        out = h.run(t_xy, t_off, h.params(256, 256, 200, 1, 4096, theta_tiles=tiles), checksum=True, batched=True)
        assert h.status(out.status) == h.F_EVENT_TOO_LARGE
        assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, off, checksum=out.checksum)


def test_bad_offsets_write_nothing(h):
    ev = gen.generate("plain_small", 10)
    bad = ev.off.copy()
    bad[3], bad[4] = bad[4], bad[3]
    xy, off = torch.from_numpy(ev.xy).cuda(), torch.from_numpy(bad).cuda()
    for batched in (False, True):
        out = h.run(xy, off, h.params(64, 64, 12), batched=batched)
        out.npeaks.fill_(-7)
        out.status.zero_()
        h.run(xy, off, h.params(64, 64, 12), out=out, batched=batched)
        assert h.status(out.status) == h.F_BAD_OFFSETS
        assert torch.all(out.npeaks == -7)
    st = h.new_status()
    h.map_hits(xy, off, st)
    assert h.status(st) == h.F_BAD_OFFSETS


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("n", [1, 2, 152, 153, 256, 257])
def test_offsets_checked_by_either_kernel(h, n, batched):
    """Few events: the fused kernel checks the offsets itself; more than the CTAs or a CTA's threads: a kernel before."""
    ev = gen.generate("plain_small", n)
    ref = oracle.run(ev.xy, ev.off, oracle.params(64, 64, 12, 1, 256), threads=THREADS)
    xy, off = dev(ev)
    p = h.params(64, 64, 12, 1, 256, block=256)
    out = h.run(xy, off, p, batched=batched)
    assert h.status(out.status) == ref.status
    assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off)
    for at, value in ((0, 1), (n, int(ev.off[-1]) + 1), (n // 2, -1), (n - 1, int(ev.off[-1]) + 1)):
        bad = off.clone()
        bad[at] = value
        out.npeaks.fill_(-7)
        out.status.zero_()
        h.run(xy, bad, p, out=out, batched=batched)
        assert h.status(out.status) == h.F_BAD_OFFSETS
        assert torch.all(out.npeaks == -7)
    out.status.zero_()
    h.run(xy, off, p, out=out, batched=batched)  # a refused call leaves nothing behind
    assert h.status(out.status) == ref.status
    assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off)


def best_us(f, stream, reps=10, rounds=7):
    """Time of one of `reps` calls back to back, the best of `rounds`."""
    for _ in range(3):
        f()
    stream.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for _ in range(rounds):
        a.record(stream)
        for _ in range(reps):
            f()
        b.record(stream)
        b.synchronize()
        best = min(best, a.elapsed_time(b) / reps * 1e3)
    return best


def time_run(h, xy, off, p, stream, batched=True):
    t_xy, t_off = torch.from_numpy(np.ascontiguousarray(xy)).cuda(), torch.from_numpy(off).cuda()
    out = h.alloc_outputs(len(xy), len(off) - 1, p)
    torch.cuda.synchronize()
    return best_us(lambda: h.run(t_xy, t_off, p, out=out, batched=batched, stream=stream), stream)


def test_uneven_events_in_two_turns(h):
    """A CTA an event, half of them large, and eight small events more. Two small ones one after the other (1,500 hits) end
    before a large one (6,000), so the eight should cost next to nothing beside eight empty ones; behind large ones they
    cost a small event's time, which a call of small ones bounds from above."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ev = gen.generate("stress", 200)
    p = h.params(256, 256, 40, 1, 4096, theta_tiles=1)
    s = torch.cuda.Stream()

    def call(large, small, extra):
        sizes = np.array([large] * (sms // 2) + [small] * (sms - sms // 2) + [extra] * 8)
        off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        return time_run(h, np.resize(ev.xy, (int(off[-1]), 2)), off, p, s)

    assert call(6000, 1500, 1500) - call(6000, 1500, 0) < 0.5 * call(1500, 1500, 0)


@pytest.mark.parametrize("n", [152, 153, 305, 609])
@pytest.mark.parametrize("nt,nr", [(64, 64), (101, 63), (100, 100), (130, 64), (128, 160), (63, 131)])
@pytest.mark.parametrize("iterative", [False, True])
def test_several_ctas_an_sm(h, nt, nr, n, iterative):
    """Small accumulators: four, three or two CTAs an SM where there are events for them."""
    ev = gen.generate("plain_small", n)
    kw = dict(peak_mode=1, rel_num=1, rel_den=2, nms_radius=2) if iterative else {}
    ref = oracle.run(ev.xy, ev.off, oracle.params(nt, nr, 9, 1, 512, **kw), threads=THREADS)
    xy, off = dev(ev)
    for batched in (False, True):
        out = h.run(xy, off, h.params(nt, nr, 9, 1, 512, **kw), checksum=True, batched=batched)
        assert h.status(out.status) == ref.status
        assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off, checksum=out.checksum)


def uneven_batch(n, small, large, n_large, seed=6):
    """n events, n_large of them of `large` hits, the others of about `small`."""
    rng = np.random.default_rng(seed)
    sizes = rng.integers(small - small // 8, small + small // 8 + 1, n)
    sizes[rng.choice(n, n_large, replace=False)] = large
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    return np.resize(gen.generate("stress", 300).xy, (int(off[-1]), 2)), off


def test_tiles_of_a_second_turn_go_to_ctas_without_a_merge(h):
    """Equal events in four tiles, as many that each CTA has one and a half of them. The CTA of an event's last tile merges and
    selects; with half the CTAs free for a second tile nobody needs to take one after that, while in two full turns a
    quarter must. So the call takes a turn and a half and not two: nine tenths of the two at most."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ev, s = gen.generate("stress", 80), torch.cuda.Stream()
    p = h.params(512, 512, 20, 1, 16384)
    assert h.resolve(p).theta_tiles == 4

    def call(n):
        off = np.arange(n + 1, dtype=np.int64) * 4720
        return time_run(h, np.resize(ev.xy, (int(off[-1]), 2)), off, p, s)

    assert call(3 * sms // 8) < 0.9 * call(sms // 2)


@pytest.mark.parametrize("n,small,large,n_large", [(153, 1600, 5000, 1), (160, 1600, 8000, 5), (200, 1600, 1700, 5), (228, 1600, 5000, 30),
                                                   (228, 0, 20000, 100), (229, 1600, 5000, 30), (608, 40, 3000, 10), (1000, 40, 3000, 10)])
@pytest.mark.parametrize("nt,nr", [(64, 64), (101, 63), (128, 128)])
@pytest.mark.parametrize("iterative", [False, True])
def test_uneven_events_on_small_accumulators(h, nt, nr, n, small, large, n_large, iterative):
    """Few more events than SMs with many hits each on small accumulators, where two launches look whether the events are even:
    even, uneven, mostly empty ones, one event more than that, bad offsets; and uneven events of larger calls."""
    kw = dict(peak_mode=1, rel_num=1, rel_den=2, nms_radius=2) if iterative else {}
    xy, off = uneven_batch(n, small, large, n_large)
    off[1] = 0  # the first event is empty, the second has its hits too
    ref = oracle.run(xy, off, oracle.params(nt, nr, 9, 1, 512, **kw), threads=THREADS)
    t_xy, t_off = torch.from_numpy(np.ascontiguousarray(xy)).cuda(), torch.from_numpy(off).cuda()
    p = h.params(nt, nr, 9, 1, 512, **kw)
    for batched in (False, True):
        out = h.run(t_xy, t_off, p, checksum=True, batched=batched)
        assert h.status(out.status) == ref.status
        assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, off, checksum=out.checksum)
        bad = t_off.clone()
        bad[n // 2] = -1
        out.npeaks.fill_(-7)
        out.status.zero_()
        h.run(t_xy, bad, p, out=out, batched=batched)
        assert h.status(out.status) == h.F_BAD_OFFSETS
        assert torch.all(out.npeaks == -7)
    out = h.alloc_outputs(len(xy), n, p, checksum=True)
    h.run_static(t_xy, t_off, p, out)
    assert h.status(out.status) == ref.status
    assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, off, checksum=out.checksum)


@pytest.mark.parametrize("nt", [100, 128])
def test_uneven_events_take_one_cta_an_sm(h, nt):
    """160 events of 500 to 3,650 hits: the few beyond an event an SM are small and end behind small ones, while two CTAs
    an SM, of half the threads, would take a fifth longer for the large ones (iterative finder)."""
    ev = gen.generate("batched", 160)
    kw, s = dict(theta_tiles=1, peak_mode=1, rel_num=1, rel_den=2, nms_radius=3), torch.cuda.Stream()
    one = time_run(h, ev.xy, ev.off, h.params(nt, nt, 8, 1, 4096, block=1024, **kw), s)
    assert time_run(h, ev.xy, ev.off, h.params(nt, nt, 8, 1, 4096, **kw), s) < 1.1 * one


def test_uneven_events_in_one_turn_are_staged_whole(h):
    """400 events of 500 to 3,650 hits at 128 x 128: a third CTA an SM would have room only with 3,072 staged hits, so the events
    that end the call would take two chunks and a fifth longer than with two CTAs of 512 threads."""
    ev, s = gen.generate("batched", 400), torch.cuda.Stream()
    two = time_run(h, ev.xy, ev.off, h.params(128, 128, 8, 1, 4096, theta_tiles=1, block=512), s)
    assert time_run(h, ev.xy, ev.off, h.params(128, 128, 8, 1, 4096), s) < 1.1 * two


@pytest.mark.parametrize("n", [1, 12, 13, 32, 33, 72, 73])
@pytest.mark.parametrize("nt,nr", [(66, 310), (130, 160), (131, 161), (256, 256), (258, 100), (512, 300), (640, 33)])
def test_few_events_in_clusters(h, nt, nr, n):
    """Calls of few events: their tiles as the CTAs of a cluster, at the last and first counts of 8, 4, 2 tiles and none."""
    ev = gen.generate("plain_small", n)
    k = int(ev.off[n // 2])
    xy, off = ev.xy.copy(), ev.off.copy()
    xy[k:k + 3] = ((2, 1), (0, 1), (0, 0))  # one event with 64-bit votes and a bad hit
    off[-1:] = len(xy)
    t_xy, t_off = torch.from_numpy(xy).cuda(), torch.from_numpy(off).cuda()
    for thr, maxp, hw in ((4, 4096, 1), (6, 50, 0)):
        ref = oracle.run(xy, off, oracle.params(nt, nr, thr, hw, maxp), threads=THREADS)
        for batched in (False, True):
            out = h.run(t_xy, t_off, h.params(nt, nr, thr, hw, maxp), checksum=True, batched=batched)
            assert h.status(out.status) == ref.status
            assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, off, checksum=out.checksum)
            out = h.run(t_xy, t_off, h.params(nt, nr, thr, hw, maxp), batched=batched)
            assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, off)


@pytest.mark.parametrize("nt,nr,tiles", [(64, 64, 1), (64, 64, 2), (63, 65, 1), (256, 256, 0), (512, 257, 4), (1000, 1000, 0), (1001, 900, 0)])
def test_records_by_keys(h, nt, nr, tiles):
    """Tiles of few records, ranked one by one: thresholds from a record an event to more than are ranked."""
    ev = gen.generate("plain_paper", 5)
    xy, off = dev(ev)
    for iterative in (False, True):
        kw = dict(peak_mode=1, rel_num=1, rel_den=3, nms_radius=2) if iterative else {}
        for thr, maxp in ((40, 512), (16, 512), (8, 7), (4, 8192)):
            ref = oracle.run(ev.xy, ev.off, oracle.params(nt, nr, thr, 1, maxp, **kw), threads=THREADS)
            for batched in (False, True):
                out = h.run(xy, off, h.params(nt, nr, thr, 1, maxp, theta_tiles=tiles, **kw), checksum=True, batched=batched)
                assert h.status(out.status) == ref.status
                assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off, checksum=out.checksum)


@pytest.mark.parametrize("nt", [65, 101, 513])
def test_autotune_odd_theta(h, nt):
    """A shape for an odd column count, in mirror pairs or columns, that the run then accepts."""
    ev = gen.generate("plain_small", 40)
    xy, off = dev(ev)
    tuned, _ = h.autotune(xy, off, h.params(nt, 200, 9, 1, 512))
    ref = oracle.run(ev.xy, ev.off, oracle.params(nt, 200, 9, 1, 512), threads=THREADS)
    out = h.run(xy, off, tuned, checksum=True, batched=True)
    assert h.status(out.status) == ref.status
    assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off, checksum=out.checksum)


@pytest.mark.parametrize("copies", [1, 12])
def test_large_events_in_clusters(h, copies):
    """Events in several staging chunks, one too large (skipped, flagged) and an empty one, in clusters of 4 and 2."""
    ev = gen.generate("stress", 8)
    sizes = [32767, 32768, 500, 0, 9000] * copies
    xy = np.concatenate([np.concatenate([ev.xy] * 2)[:s] for s in sizes])
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    ref = oracle.run(xy, off, oracle.params(256, 256, 100, 1, 4096), threads=THREADS)
    assert ref.status == oracle.F_EVENT_TOO_LARGE
    t_xy, t_off = torch.from_numpy(xy).cuda(), torch.from_numpy(off).cuda()
    out = h.run(t_xy, t_off, h.params(256, 256, 100, 1, 4096), checksum=True, batched=True)
    assert h.status(out.status) == h.F_EVENT_TOO_LARGE
    assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, off, checksum=out.checksum)


@pytest.mark.parametrize("nt,nr,tiles", [(5, 40, 1), (5, 40, 2), (9, 33, 3), (63, 64, 1), (65, 30, 1), (65, 30, 2), (127, 96, 1),
                                         (129, 61, 1), (129, 61, 4), (131, 64, 11), (199, 200, 0), (255, 256, 0), (257, 100, 3),
                                         (511, 513, 0), (1023, 255, 0)])
def test_odd_theta_edges(h, nt, nr, tiles):
    """An odd column count in mirror pairs: the middle column alone, in a word group or a tile of its own, beside a halo."""
    ev = gen.generate("plain_small", 12)
    mid = [p for p in ((0, 3000), (0, -3000), (3000, 0), (1, 2500), (-1, 2500), (30000, 7)) for _ in range(40)]
    wide = mid + [(2, 1), (-1, 2), (0, 1)] * 20  # 64-bit votes
    xy = np.concatenate([ev.xy[: ev.off[-1]], np.array(mid + wide)]).astype(np.int32)
    off = np.concatenate([ev.off, ev.off[-1] + np.array([240, 540])]).astype(np.int64)
    t_xy, t_off = torch.from_numpy(xy).cuda(), torch.from_numpy(off).cuda()
    it = dict(peak_mode=1, rel_num=1, rel_den=3)
    for thr, maxp, hw, kw in ((3, 4096, 1, {}), (12, 60, 0, {}), (30, 4096, 40, {}), (3, 4096, 1, dict(it, nms_radius=1)),
                              (2, 4096, 0, dict(it, nms_radius=min(5, (nt - 1) // 2)))):
        ref = oracle.run(xy, off, oracle.params(nt, nr, thr, hw, maxp, **kw), threads=THREADS)
        for batched in (False, True):
            out = h.run(t_xy, t_off, h.params(nt, nr, thr, hw, maxp, theta_tiles=tiles, **kw), checksum=True, batched=batched)
            assert h.status(out.status) == ref.status
            assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, off, checksum=out.checksum)


def test_peak_overflow_keeps_first_in_raster_order(h):
    cfg = gen.CONFIGS["plain_paper"]
    ev = gen.generate(cfg, 20)
    ref = oracle.run(ev.xy, ev.off, oracle.params(256, 256, 16, 1, 100), threads=THREADS)
    assert ref.status == oracle.F_PEAK_OVERFLOW
    xy, off = dev(ev)
    for tiles in (1, 2, 3, 4):  # 2 and 4: mirror-pair tiles (low and high segments), 3: plain tiles
        out = h.run(xy, off, h.params(256, 256, 16, 1, 100, theta_tiles=tiles), batched=True)
        assert h.status(out.status) == h.F_PEAK_OVERFLOW
        assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off)


@pytest.mark.parametrize("hw", [0, 3])
def test_keep_halfwidth(h, hw):
    cfg = gen.CONFIGS["plain_paper"]
    ev = gen.generate(cfg, 30)
    ref = oracle.run(ev.xy, ev.off, oracle.params(256, 256, 16, hw, 4096), threads=THREADS)
    xy, off = dev(ev)
    out = h.run(xy, off, h.params(256, 256, 16, hw, 4096), batched=True)
    assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off)


def test_permutation_invariance_on_gpu(h):
    cfg = gen.CONFIGS["plain_paper"]
    ev = gen.generate(cfg, 20)
    rng = np.random.default_rng(2)
    perm = np.concatenate([ev.off[e] + rng.permutation(ev.off[e + 1] - ev.off[e]) for e in range(20)])
    xy, off = dev(ev)
    a = h.run(xy, off, cfg_params(h, cfg), checksum=True, batched=True)
    b = h.run(torch.from_numpy(ev.xy[perm]).cuda(), off, cfg_params(h, cfg), checksum=True, batched=True)
    assert torch.equal(a.npeaks, b.npeaks) and torch.equal(a.checksum, b.checksum)
    assert np.array_equal(peaks_np(a.peaks), peaks_np(b.peaks))
    assert np.array_equal(to_np(a.mask)[perm], to_np(b.mask))


def test_non_default_stream_and_graph_replay(h):
    cfg = gen.CONFIGS["plain_paper"]
    ev = gen.generate(cfg, 64)
    ref = oracle_of(cfg, ev)
    xy, off = dev(ev)
    s = torch.cuda.Stream()
    out = h.alloc_outputs(ev.n_hits, ev.n_events, cfg_params(h, cfg), checksum=True)
    torch.cuda.synchronize()
    for _ in range(3):  # the second and third calls replay the cached graph
        out.mask.fill_(7)
        with torch.cuda.stream(s):
            h.run(xy, off, cfg_params(h, cfg), out=out, batched=True, stream=s)
        s.synchronize()
        assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off, checksum=out.checksum)


# ---------------------------------------------------------------- the mirror-pair vote at its edges

def near_boundary_hits(ev, n_theta, n_rho, n_hits):
    """The hits of ev with the most theta columns whose exact bin position lies within 5e-5 of a boundary."""
    x, y = ev.xy[:, 0].astype(np.int64), ev.xy[:, 1].astype(np.int64)
    r2 = x * x + y * y
    u, v = (x << 33) // r2, (y << 33) // r2
    th = (np.arange(n_theta) + 0.5) * np.pi / n_theta
    c, s = np.rint(16384 * np.cos(th)), np.rint(16384 * np.sin(th))
    k = (u[:, None] * c + v[:, None] * s + 703687442) * n_rho / (2.0 * 703687442)
    near = (np.abs(k - np.rint(k)) < 5e-5).sum(axis=1)
    return ev.xy[np.argsort(-near, kind="stable")[:n_hits]]


@pytest.mark.parametrize("n_theta,n_rho,tiles", [(64, 64, 1), (128, 100, 1), (130, 64, 1), (256, 256, 1), (256, 256, 2),
                                                 (512, 512, 4), (1000, 500, 8), (258, 256, 3)])
def test_vote_edges(h, n_theta, n_rho, tiles):
    """One and two words a lane; events of 0, 1, 2, 3, ... hits (fewer pairs than warps, odd counts, one
    staging chunk and one hit more); hits repeated so that their near-boundary columns overflow the
    list of ambiguous steps. Accumulators by checksum, and every output."""
    ev = gen.generate("batched", 12)
    near = near_boundary_hits(ev, n_theta, n_rho, 3)
    parts = [ev.xy[i:i + n] for i, n in enumerate([0, 1, 2, 3, 7, 31, 64, 65, 127, 130, 257, 4096, 4097])]
    parts += [np.repeat(near[i:i + 1], 3001 + i, axis=0) for i in range(3)]
    off = np.concatenate([[0], np.cumsum([len(p) for p in parts])]).astype(np.int64)
    xy = np.ascontiguousarray(np.concatenate(parts))
    ref = oracle.run(xy, off, oracle.params(n_theta, n_rho, 3, 1, 16384), threads=THREADS)
    d_xy, d_off = torch.from_numpy(xy).cuda(), torch.from_numpy(off).cuda()
    for batched in (False, True):
        out = h.run(d_xy, d_off, h.params(n_theta, n_rho, 3, 1, 16384, theta_tiles=tiles), checksum=True, batched=batched)
        assert h.status(out.status) == ref.status
        assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, off, checksum=out.checksum)


@pytest.mark.parametrize("r0", [8192, 131072, 1024, 200000])
def test_map_where_the_estimate_ends(h, r0):
    """Quotients around 2^20 (where the float estimate ends), 2^16, far above and in the ordinary range, against integers."""
    rng = np.random.default_rng(r0)
    r, a = rng.uniform(0.97 * r0, 1.03 * r0, 100_000), rng.uniform(0, 2 * np.pi, 100_000)
    xy = np.stack([r * np.cos(a), r * np.sin(a)], 1).astype(np.int32)
    xy[:8] = [(r0, 0), (-r0, 0), (0, r0), (0, -r0), (r0 - 1, 1), (r0 + 1, -1), (-r0 + 1, 0), (0, -r0 - 1)]
    x, y = xy[:, 0].astype(np.int64), xy[:, 1].astype(np.int64)
    uq, vq = h.map_hits(torch.from_numpy(xy).cuda(), torch.tensor([0, len(xy)], dtype=torch.int64, device="cuda"), h.new_status())
    assert np.array_equal(to_np(uq), (x << 33) // (x * x + y * y)) and np.array_equal(to_np(vq), (y << 33) // (x * x + y * y))


def test_near_hits_map_as_fast_as_far_ones(h):
    """The quotients of hits at 9 to 100 mm are settled by the same few operations as those at 200 to 800 mm, so the same
    number of them takes the same time (1.5 leaves room for the clock; the 64-bit divisions take twice as long)."""
    rng = np.random.default_rng(5)
    n, s, us = 1 << 22, torch.cuda.current_stream(), []
    for lo, hi in ((9e3, 100e3), (200e3, 800e3)):
        r, a = rng.uniform(lo, hi, n), rng.uniform(0, 2 * np.pi, n)
        xy = torch.from_numpy(np.stack([r * np.cos(a), r * np.sin(a)], 1).astype(np.int32)).cuda()
        off, st = torch.tensor([0, n], dtype=torch.int64, device="cuda"), h.new_status()
        uq, vq = h.map_hits(xy, off, st)
        us.append(best_us(lambda: h.map_hits(xy, off, st, uq, vq), s))
    assert us[0] < 1.5 * us[1]


# ---------------------------------------------------------------- exhaustive bin function

@pytest.mark.parametrize("n_rho", [4, 63, 64, 256, 512, 1000, 1024])
def test_bin_function_exhaustive(h, n_rho):
    """Every rho in [-H - 10^6, H + 10^6]: the device's multiply-high binning equals plain
    64-bit floor division with clamping."""
    H = 703687442
    m = h.selftest_bin(n_rho, -H - 10 ** 6, H + 10 ** 6)
    assert int(m.item()) == 0


@pytest.mark.parametrize("n_theta,n_rho", [(64, 64), (256, 256), (512, 512), (1000, 1000), (1024, 1024), (37, 63)])
def test_float_bin_path_random_tuples(h, n_theta, n_rho):
    """The vote bins through a float estimate and falls back to integer arithmetic when an
    integer lies within the estimate's error bound of it; 2e8 random tuples must all agree
    with exact division, for the general estimate and for the mirror-pair layout's row read
    off the float's bit pattern (whose window is a power of two of 2^-F units, F = 23 - b)."""
    bad, amb, bad_mp, amb_mp, n_mp = h.selftest_fpbin(n_theta, n_rho, 12345 + n_rho, 200_000_000)
    assert bad == 0
    assert 0 < amb < 200_000_000 * 4e-3  # the fallback is exercised, and rare
    assert bad_mp == 0
    assert n_mp > 100_000_000
    b = (n_rho + 1).bit_length()  # 2^b >= n_rho + 2
    assert 0 < amb_mp < n_mp * 2 * 4 * 2.0 ** -(23 - b)  # window of 4 units, twice for slack


def test_autotuned_shape_gives_identical_results(h):
    cfg = gen.CONFIGS["plain_paper"]
    ev = gen.generate(cfg, 200)
    xy, off = dev(ev)
    p = cfg_params(h, cfg)
    tuned, ms = h.autotune(xy, off, p)
    assert ms > 0 and tuned.theta_tiles >= 1 and tuned.block % 32 == 0 and tuned.events_per_cta >= 1
    again, ms2 = h.autotune(xy, off, p)  # cached
    assert ms2 == -1.0 and [getattr(again, f) for f, _ in again._fields_] == [getattr(tuned, f) for f, _ in tuned._fields_]
    ref = oracle_of(cfg, ev)
    out = h.run(xy, off, tuned, checksum=True, batched=True)
    assert h.status(out.status) == 0
    assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off, checksum=out.checksum)


@pytest.mark.parametrize("n", [1, 16])
def test_autotuned_few_events_are_no_slower_than_untuned(h, n):
    """A call of few events takes the CTAs of clusters when its launch fields are zero, a quarter faster than any shape with
    them: the autotuner finds it, also after a large batch of the same parameters has been tuned."""
    ev = gen.generate("batched", 1000)
    p = h.params(256, 256, 18, 1, 4096)
    xy, off = dev(ev)
    _, ms = h.autotune(xy, off, p)
    few, few_off = xy[: int(ev.off[n])].contiguous(), off[: n + 1].contiguous()
    tuned, ms_few = h.autotune(few, few_off, p)
    assert ms_few > 0  # not the large batch's
    ref = oracle.run(ev.xy[: ev.off[n]], ev.off[: n + 1], oracle.params(256, 256, 18, 1, 4096), threads=THREADS)
    out = h.run(few, few_off, tuned, checksum=True, batched=True)
    assert h.status(out.status) == ref.status
    assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off[: n + 1], checksum=out.checksum)
    s = torch.cuda.Stream()
    us = [time_run(h, ev.xy[: ev.off[n]], ev.off[: n + 1], q, s) for q in (tuned, p)]
    assert us[0] < 1.1 * us[1]


def test_autotune_cache_keys_the_peak_finder(h):
    """The autotuner writes only the launch shape, and its cache tells the peak finders apart:
    tuning the 3x3 finder first must not hand the iterative finder's tuning the 3x3 parameters.
    (Threshold 17 is used by no other test, so both keys are new to this process.)"""
    cfg = gen.CONFIGS["plain_paper"]
    ev = gen.generate(cfg, 300)
    xy, off = dev(ev)
    algo = ("n_theta", "n_rho", "threshold", "keep_halfwidth", "max_peaks", "peak_mode", "rel_num", "rel_den",
            "nms_radius")
    p0 = h.params(cfg.n_theta, cfg.n_rho, 17, cfg.keep_halfwidth, 512)
    t0, ms0 = h.autotune(xy, off, p0)
    assert ms0 > 0 and [getattr(t0, f) for f in algo] == [getattr(p0, f) for f in algo]
    p1 = h.params(cfg.n_theta, cfg.n_rho, 17, cfg.keep_halfwidth, 512, peak_mode=1, rel_num=1, rel_den=2,
                  nms_radius=3)
    t1, ms1 = h.autotune(xy, off, p1)
    assert ms1 > 0, "the iterative finder's tuning came from the 3x3 finder's cache entry"
    assert [getattr(t1, f) for f in algo] == [getattr(p1, f) for f in algo]
    t1b, ms1b = h.autotune(xy, off, p1)
    assert ms1b == -1.0 and [getattr(t1b, f) for f, _ in t1b._fields_] == [getattr(t1, f) for f, _ in t1._fields_]
    op = oracle.params(cfg.n_theta, cfg.n_rho, 17, cfg.keep_halfwidth, 512, peak_mode=1, rel_num=1, rel_den=2,
                       nms_radius=3)
    ref = oracle.run(ev.xy, ev.off, op, threads=THREADS)
    out = h.run(xy, off, t1, batched=True)
    assert h.status(out.status) == ref.status
    assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off)


def test_host_errors(h):
    xy = torch.zeros((4, 2), dtype=torch.int32, device="cuda")
    off = torch.tensor([0, 4], dtype=torch.int64, device="cuda")
    for bad in (h.params(3, 64, 2), h.params(64, 1025, 2), h.params(64, 64, 0), h.params(64, 64, 2, max_peaks=0),
                h.params(64, 64, 2, block=48), h.params(64, 64, 2, theta_tiles=65)):
        with pytest.raises(h.HoughError) as ei:
            h.run(xy, off, bad, out=h.alloc_outputs(4, 1, h.params(64, 64, 2)))
        assert ei.value.code == h.EPARAM
    p = h.params(64, 64, 2)
    out = h.alloc_outputs(4, 1, p)
    out.ws = out.ws[:16]
    with pytest.raises(h.HoughError) as ei:
        h.run(xy, off, p, out=out)
    assert ei.value.code == h.EWORKSPACE
    # peak records are written as 8-byte stores: a buffer 2 bytes off is refused before launch
    out = h.alloc_outputs(4, 1, p)
    out.peaks = torch.zeros(4 * p.max_peaks + 4, dtype=torch.int16, device="cuda")[1:]
    for batched in (False, True):
        with pytest.raises(h.HoughError) as ei:
            h.run(xy, off, p, out=out, batched=batched)
        assert ei.value.code == h.EINVAL
    with pytest.raises(h.HoughError) as ei:
        h.run_static(xy, off, p, out)
    assert ei.value.code == h.EINVAL
    # output tensors too small or of the wrong type are refused before anything is enqueued
    out = h.alloc_outputs(4, 1, p)
    out.peaks = out.peaks[:, :10]
    with pytest.raises(ValueError):
        h.run(xy, off, p, out=out)
    out = h.alloc_outputs(4, 1, p)
    out.mask = torch.zeros(4, dtype=torch.int32, device="cuda")
    with pytest.raises(TypeError):
        h.run(xy, off, p, out=out, batched=True)


# ---------------------------------------------------------------- Eq. (2) circle recovery

@pytest.mark.parametrize("name,n", [("plain_paper", 200), ("stress", 20), ("paper_1000", 50)])
def test_circles_match_oracle(h, name, n):
    """Circle of every stored peak (float32 on the GPU from double arithmetic) against the
    oracle's float64, to float rounding; records past each event's stored peaks untouched."""
    cfg = gen.CONFIGS[name]
    ev = gen.generate(cfg, n)
    xy, off = dev(ev)
    p = cfg_params(h, cfg)
    out = h.run(xy, off, p, batched=True)
    circ = torch.full((n, p.max_peaks, 4), -7.0, dtype=torch.float32, device="cuda")
    h.circles(out.npeaks, out.peaks, p, 1.0, out=circ)
    got = to_np(circ)
    npk = np.minimum(to_np(out.npeaks), p.max_peaks)
    pk = to_np(out.peaks)
    for e in range(n):
        recs = pk[e, : npk[e]].astype(np.int16).view(oracle.PEAK_DTYPE).reshape(-1)
        ref = oracle.circles(recs, cfg.n_theta, cfg.n_rho, 1.0)
        np.testing.assert_allclose(got[e, : npk[e]], ref.astype(np.float32), rtol=1e-6, atol=0)
        assert np.all(got[e, npk[e]:] == -7.0)


def test_circles_odd_rho_and_field(h):
    """Odd N_rho has a bin centre at rho = 0 (infinite radius); pT scales with the field."""
    p = h.params(4, 5, 1, 1, 8)
    pk = torch.zeros((1, 8, 4), dtype=torch.int16, device="cuda")
    pk[0, :3, 0] = torch.tensor([0, 1, 3], dtype=torch.int16)
    pk[0, :3, 1] = torch.tensor([0, 2, 4], dtype=torch.int16)
    npk = torch.tensor([3], dtype=torch.int32, device="cuda")
    got = to_np(h.circles(npk, pk, p, 1.5))[0, :3]
    recs = to_np(pk)[0, :3].view(oracle.PEAK_DTYPE).reshape(-1)
    ref = oracle.circles(recs, 4, 5, 1.5).astype(np.float32)
    assert np.isinf(got[1, 2]) and np.isinf(got[1, 3]) and np.isinf(ref[1, 2])
    fin = np.isfinite(ref)
    np.testing.assert_allclose(got[fin], ref[fin], rtol=1e-6)
    assert np.array_equal(np.sign(got[~fin]), np.sign(ref[~fin]))


# ---------------------------------------------------------------- iterative peak finder (Sec. 2)

ITER = [  # (workload, events, n_theta, n_rho, threshold, rel_num, rel_den, nms_radius, max_peaks)
    ("plain_paper", 60, 256, 256, 16, 1, 2, 3, 64),
    ("plain_paper", 40, 64, 64, 8, 1, 3, 1, 256),
    ("batched", 60, 256, 256, 16, 2, 5, 2, 128),
    ("plain_small", 30, 64, 64, 6, 0, 1, 0, 300),    # no relative cut, no neighbourhood: every cell >= T
    ("plain_paper", 30, 100, 63, 8, 1, 4, 2, 512),   # N_theta not a multiple of 64, odd N_rho
    ("plain_paper", 20, 256, 256, 16, 1, 10, 1, 8),  # overflow: more peaks than stored
    # 20k-40k candidates an event, above the sorted form's 8,192 keys: one pass per peak
    ("batched", 12, 256, 256, 4, 0, 1, 6, 512),
    # 1k-10k candidates: events of both forms in one launch, sorts of up to 8,192 keys
    ("batched", 40, 256, 256, 16, 1, 3, 3, 1024),
]


@pytest.mark.parametrize("name,n,nt,nr,thr,num,den,R,mx", ITER)
def test_iterative_fused_and_stepwise_match_oracle(h, name, n, nt, nr, thr, num, den, R, mx):
    cfg = gen.CONFIGS[name]
    ev = gen.generate(cfg, n)
    op = oracle.params(nt, nr, thr, 1, mx, peak_mode=1, rel_num=num, rel_den=den, nms_radius=R)
    ref = oracle.run(ev.xy, ev.off, op, with_acc=True, threads=THREADS)
    xy, off = dev(ev)
    p = h.params(nt, nr, thr, 1, mx, peak_mode=1, rel_num=num, rel_den=den, nms_radius=R)
    for batched in (False, True):
        out = h.run(xy, off, p, checksum=True, batched=batched)
        assert h.status(out.status) == ref.status
        assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off, checksum=out.checksum)
    # stepwise: the iterative finder on the oracle's accumulator in HBM
    st = h.new_status()
    acc = torch.from_numpy(ref.acc).cuda()
    npk, pk = h.peaks(acc, p, st)
    assert np.array_equal(to_np(npk), ref.npeaks)
    assert np.array_equal(peaks_np(pk), peaks_np(torch.from_numpy(ref.peaks.view(np.int16).reshape(n, mx, 4))))


def test_iterative_cell_above_4095_votes(h):
    """4,200 copies of one hit put 4,200 votes into a cell of every column: beyond the 12-bit vote
    field of the sorted form's keys, so that event takes one pass per peak; its neighbours in the
    batch take the sorted form. Fused, batched and stepwise results as the oracle's."""
    ev = gen.generate(gen.CONFIGS["plain_paper"], 3)
    a, b = int(ev.off[1]), int(ev.off[2])
    xy = np.concatenate([ev.xy[:b], np.repeat(ev.xy[a:a + 1], 4200, axis=0), ev.xy[b:]])
    off = ev.off.copy()
    off[2:] += 4200
    n_t, n_r = 128, 128
    op = oracle.params(n_t, n_r, 10, 1, 512, peak_mode=1, rel_num=1, rel_den=2, nms_radius=2)
    ref = oracle.run(xy, off, op, with_acc=True, threads=THREADS)
    assert ref.acc.reshape(3, n_t, n_r)[1].max() >= 4200
    p = h.params(n_t, n_r, 10, 1, 512, peak_mode=1, rel_num=1, rel_den=2, nms_radius=2)
    d_xy, d_off = torch.from_numpy(xy).cuda(), torch.from_numpy(off).cuda()
    for batched in (False, True):
        out = h.run(d_xy, d_off, p, checksum=True, batched=batched)
        assert h.status(out.status) == ref.status
        assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, off, checksum=out.checksum)
    npk, pk = h.peaks(torch.from_numpy(ref.acc).cuda(), p, h.new_status())
    assert np.array_equal(to_np(npk), ref.npeaks)
    assert np.array_equal(peaks_np(pk), peaks_np(torch.from_numpy(ref.peaks.view(np.int16).reshape(3, 512, 4))))


def test_iterative_stepwise_large_accumulator(h):
    """1000 x 1000 (2 MB accumulator, no single-CTA fused plan): the stepwise finder keeps its
    suppression bitmap in shared memory."""
    cfg = gen.CONFIGS["paper_1000"]
    ev = gen.generate(cfg, 6)
    op = oracle.params(1000, 1000, 12, 1, 256, peak_mode=1, rel_num=1, rel_den=2, nms_radius=4)
    ref = oracle.run(ev.xy, ev.off, op, with_acc=True, threads=THREADS)
    p = h.params(1000, 1000, 12, 1, 256, peak_mode=1, rel_num=1, rel_den=2, nms_radius=4)
    st = h.new_status()
    npk, pk = h.peaks(torch.from_numpy(ref.acc).cuda(), p, st)
    assert h.status(st) == 0
    assert np.array_equal(to_np(npk), ref.npeaks)
    n = ref.npeaks
    got = peaks_np(pk)
    exp = peaks_np(torch.from_numpy(ref.peaks.view(np.int16).reshape(len(n), 256, 4)))
    for e in range(len(n)):
        assert np.array_equal(got[e][: min(n[e], 256)], exp[e][: min(n[e], 256)])


@pytest.mark.parametrize("nt,nr,thr,num,den,R,tiles", [
    (256, 256, 1, 0, 1, 1, 1),    # more undecided candidates than are listed, more peaks than are ranked at once
    (256, 256, 2, 0, 1, 8, 1),    # a window of more than 16 columns; candidates by bitmap words
    (130, 90, 4, 1, 3, 20, 1),    # more columns than lanes, taller than a bitmap word
    (256, 256, 60, 1, 1, 3, 1),   # the maximum's own votes: few candidates, or none
    (256, 256, 2, 0, 1, 2, 4),    # candidate lists that leave no room beside the staged hits
    (256, 200, 4, 1, 4, 8, 64),   # 128 segments to merge
    (250, 64, 3, 1, 3, 1, 8),     # tiles of uneven width
    (255, 64, 3, 1, 3, 4, 5),     # column tiles: no local maxima marked
    (459, 206, 12, 1, 2, 3, 1),   # whole columns that leave no room for lists: one pass a peak
    (467, 204, 12, 1, 3, 2, 1),   # whole columns with the shortest list: events past it
    (467, 204, 40, 3, 4, 1, 1),   # and within it
])
def test_iterative_edges(h, nt, nr, thr, num, den, R, tiles):
    """Whole and tiled finders where their lists, windows and merges have their edges; two events of one and
    no hits among the others."""
    ev = gen.generate(gen.CONFIGS["plain_paper"], 3)
    a = int(ev.off[1])
    xy, off = ev.xy, np.array([0, a, a, a + 1, int(ev.off[2]), int(ev.off[3])], np.int64)
    run_iterative_tiled(h, xy, off, nt, nr, thr, num, den, R, 20000, tiles)


# ---------------------------------------------------------------- iterative finder on theta tiles

ITER_TILED = [  # (workload, events, n_theta, n_rho, threshold, rel_num, rel_den, nms_radius, max_peaks, tiles)
    ("plain_paper", 40, 256, 256, 16, 1, 2, 3, 2048, 2),
    ("plain_paper", 30, 256, 256, 16, 1, 2, 3, 2048, 4),   # windows across three tile edges
    ("stress", 8, 512, 512, 20, 1, 2, 3, 16384, 4),        # the stress shape (13k candidates an event)
    ("plain_paper", 20, 101, 63, 8, 1, 4, 2, 512, 3),      # odd N_theta: column tiles, no mirror pairs
    ("plain_paper", 12, 1000, 1000, 12, 1, 2, 4, 1024, 16),  # the paper's discretisation
    ("plain_small", 20, 64, 64, 6, 0, 1, 0, 300, 2),       # every cell >= T, no neighbourhood
    ("batched", 16, 256, 256, 16, 1, 2, 64, 256, 8),       # windows wider than a tile (R = 64)
]


def run_iterative_tiled(h, xy_np, off_np, nt, nr, thr, num, den, R, mx, tiles):
    op = oracle.params(nt, nr, thr, 1, mx, peak_mode=1, rel_num=num, rel_den=den, nms_radius=R)
    ref = oracle.run(xy_np, off_np, op, threads=THREADS)
    xy, off = torch.from_numpy(xy_np).cuda(), torch.from_numpy(off_np).cuda()
    p = h.params(nt, nr, thr, 1, mx, theta_tiles=tiles, peak_mode=1, rel_num=num, rel_den=den, nms_radius=R)
    assert h.resolve(p).theta_tiles == tiles
    deferred = []
    for batched in (False, True):
        out = h.run(xy, off, p, checksum=True, batched=batched)
        assert h.status(out.status) == ref.status
        assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, off_np, checksum=out.checksum)
        deferred.append(int(out.ws[8:12].view(torch.int32).item()))  # events the fallback kernel took
    return ref, deferred


@pytest.mark.parametrize("name,n,nt,nr,thr,num,den,R,mx,tiles", ITER_TILED)
def test_iterative_tiled_matches_oracle(h, name, n, nt, nr, thr, num, den, R, mx, tiles):
    """The paper's iterative finder with the accumulator split over theta tiles: each tile
    publishes its candidates, the last tile of the event settles them; fused and batched
    launches, outputs and accumulator checksums equal the oracle's."""
    ev = gen.generate(gen.CONFIGS[name], n)
    run_iterative_tiled(h, ev.xy, ev.off, nt, nr, thr, num, den, R, mx, tiles)


def test_iterative_tiled_deferred_events(h):
    """Events whose candidates do not fit the tiles' record slots (max_peaks 32 here) go to the
    fallback kernel (HBM accumulator, the stepwise finder): results still equal the oracle's,
    peak-list overflow included, and the fallback really ran."""
    ev = gen.generate(gen.CONFIGS["plain_paper"], 24)
    ref, deferred = run_iterative_tiled(h, ev.xy, ev.off, 256, 256, 16, 1, 2, 3, 32, 4)
    assert min(deferred) > 0 and ref.status & 4  # some events deferred; some peak lists overflowed


def test_iterative_tiled_cell_above_4095_votes(h):
    """A cell above 4,095 votes (beyond the candidate keys' vote field) defers its event; its
    neighbours in the batch take the tiles' candidate lists."""
    ev = gen.generate(gen.CONFIGS["plain_paper"], 3)
    a, b = int(ev.off[1]), int(ev.off[2])
    xy = np.concatenate([ev.xy[:b], np.repeat(ev.xy[a:a + 1], 4200, axis=0), ev.xy[b:]])
    off = ev.off.copy()
    off[2:] += 4200
    _, deferred = run_iterative_tiled(h, xy, off, 256, 256, 10, 1, 2, 2, 4096, 2)
    assert deferred == [1, 1]  # the event with the 4,200-vote cells, in both launches


@pytest.mark.parametrize("name,sample", [("stress", 40), ("paper_1000", 80)])
def test_full_size_sampled_iterative_tiled(h, name, sample):
    """The stress (512 x 512) and 1000 x 1000 workloads, whole, with the iterative finder (half the
    maximum, radius 3) in the autotuned launch shape; the oracle recomputes a random sample."""
    cfg = gen.CONFIGS[name]
    ev = gen.generate(cfg, with_truth=False)
    xy, off = dev(ev)
    kw = dict(peak_mode=1, rel_num=1, rel_den=2, nms_radius=3)
    p = cfg_params(h, cfg, **kw)
    ns = min(ev.n_events, 2000)
    p, _ = h.autotune(xy[: int(ev.off[ns])], off[: ns + 1], p)
    assert h.resolve(p).theta_tiles > 1
    out = h.run(xy, off, p, checksum=False, batched=True)
    assert h.status(out.status) == 0
    rng = np.random.default_rng(3)
    events = np.sort(rng.choice(ev.n_events, size=sample, replace=False))
    events[0] = 0
    events[-1] = ev.n_events - 1
    sxy, soff = sub_batch(ev.xy, ev.off, events)
    ref = oracle.run(sxy, soff, oracle.params(cfg.n_theta, cfg.n_rho, cfg.threshold, cfg.keep_halfwidth,
                                              cfg.max_peaks, **kw), threads=THREADS)
    assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, ev.off, events=events)


# ---------------------------------------------------------------- host-buffer path (pipelined chunks)

@pytest.mark.parametrize("name,n,iterative", [("plain_paper", 300, False), ("batched", 9000, False),
                                               ("stress", 4100, False), ("batched", 5000, True)])
def test_host_path_matches_oracle(h, name, n, iterative):
    """hough_run_host: pinned host inputs in, host results out. 9,000, 5,000 and 4,100 events run
    as several pipelined chunks (rebased offsets, peaks packed per chunk and re-based on the
    host); also with the iterative finder (half the maximum, radius 3)."""
    cfg = gen.CONFIGS[name]
    ev = gen.generate(cfg, n)
    kw = dict(peak_mode=1, rel_num=1, rel_den=2, nms_radius=3) if iterative else {}
    ref = oracle.run(ev.xy, ev.off, oracle.params(cfg.n_theta, cfg.n_rho, cfg.threshold, cfg.keep_halfwidth,
                                                  cfg.max_peaks, **kw), threads=THREADS)
    p = cfg_params(h, cfg, **kw)
    r = h.HostRunner(ev.n_hits, ev.n_events, p)
    xy = torch.from_numpy(ev.xy).pin_memory()
    off = torch.from_numpy(ev.off).pin_memory()
    for _ in range(2):  # a second call reuses the cached graphs and streams
        assert r(xy, off) == 0
        assert np.array_equal(r.npeaks.numpy(), ref.npeaks)
        assert np.array_equal(r.nkept.numpy(), ref.nkept)
        assert np.array_equal(r.mask.numpy()[: ev.n_hits], ref.mask)
        po = r.peak_off.numpy()
        stored = np.minimum(ref.npeaks, cfg.max_peaks)
        assert po[0] == 0 and np.array_equal(np.diff(po), stored)
        dense = r.peaks.numpy()[: po[-1]].astype(np.int16).view(oracle.PEAK_DTYPE).reshape(-1)
        for e in range(n):
            assert np.array_equal(dense[po[e]: po[e + 1]], ref.peaks[e, : stored[e]]), e


def test_host_path_errors(h):
    cfg = gen.CONFIGS["plain_paper"]
    ev = gen.generate(cfg, 50)
    p = cfg_params(h, cfg)
    xy = torch.from_numpy(ev.xy).pin_memory()
    off = torch.from_numpy(ev.off).pin_memory()
    small = h.HostRunner(ev.n_hits, ev.n_events, p, peaks_cap=10)
    with pytest.raises(h.HoughError) as ei:
        small(xy, off)
    assert ei.value.code == h.EWORKSPACE
    ref = oracle_of(cfg, ev)
    assert np.array_equal(small.npeaks.numpy(), ref.npeaks)  # counts and offsets still valid
    assert small.peak_off.numpy()[-1] == np.minimum(ref.npeaks, cfg.max_peaks).sum()
    bad = off.clone()
    bad[10] = bad[11] + 1  # offsets must not decrease: refused on the host, nothing enqueued
    r = h.HostRunner(ev.n_hits, ev.n_events, p)
    with pytest.raises(h.HoughError) as ei:
        r(xy, bad)
    assert ei.value.code == h.EINVAL


@pytest.mark.parametrize("nt,nr,thr,hw,tiles", [(256, 256, 60, 1, 1), (256, 94, 40, 31, 1), (128, 63, 60, 2, 1), (4, 4, 900, 1, 1),
                                                (1000, 1000, 14, 0, 16), (64, 30, 120, 1, 1), (256, 256, 3000, 1, 1)])
def test_selection_edges(h, nt, nr, thr, hw, tiles):
    """Few peak columns (fewer than four, than twelve, none), many hits that meet every column, guard bits at
    the ends of bitmap words, wide windows; events above the staged size and one of a single hit."""
    ev = gen.generate("batched", 14)
    k = int(ev.off[3])
    xy = np.concatenate([ev.xy, ev.xy[:7500]])
    off = np.concatenate([ev.off, [ev.off[-1] + 7500]]).astype(np.int64)
    off[4] = k + 1  # the fourth event keeps one hit, the fifth gets the rest
    ref = oracle.run(xy, off, oracle.params(nt, nr, thr, hw, 4096), threads=THREADS)
    d_xy, d_off = torch.from_numpy(xy).cuda(), torch.from_numpy(off).cuda()
    for batched in (False, True):
        out = h.run(d_xy, d_off, h.params(nt, nr, thr, hw, 4096, theta_tiles=tiles), batched=batched)
        assert h.status(out.status) == ref.status
        assert_event_outputs_equal(ref, out.npeaks, out.peaks, out.mask, out.nkept, off)
