"""Kernels at the sizes where their tiling can go wrong, against the oracle: the search and the
clipped statistics at the edges of a warp's passes and segments, the corner turn of spectra that
start at any byte, the staged direct kernel with and without a split of the channels, and the
128-trial tile. Series, moments and statistics are whole numbers and are compared exactly."""
import threading

import numpy as np
import pytest

import oracle
from synth import configs
from _parity import clipped_trial_snr, compare_candidates

torch = pytest.importorskip("torch")
import paper_2101_00941_gb300 as dd  # noqa: E402
from _gpu_check import _arrivals, check, staged_takes  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    dd.build()
    dd.lib()


def _series(trials, n, seed):
    rng = np.random.default_rng(seed)
    y = np.rint(rng.normal(60000.0, 300.0, (trials, n))).astype(np.int32)
    for t in range(trials):  # pulses at the window's ends and inside
        for j in (0, n // 2, n - 1):
            y[t, max(0, j - 2):j + 3] += 900
    return y


# a warp's pass is 512 samples, a segment 2 to 16 passes; rows that start off a 16-byte boundary
@pytest.mark.parametrize("n", [1, 31, 512, 513, 1023, 4097, 20001, 65541])
@pytest.mark.parametrize("widths,block,shift", [((1, 2, 4, 8, 16, 32, 64, 128, 256), 32, 0),
                                                ((1, 3, 5, 600, 1024), 8, 1), ((1,), 1, 3)])
def test_search_window_edges(n, widths, block, shift):
    trials, d = 3, 1
    y = _series(trials, n, 70 + n)
    stride = n + shift + 4
    buf = torch.zeros(trials * stride, dtype=torch.int32, device="cuda")
    view = buf.as_strided((trials, n), (stride, 1), shift)
    view.copy_(torch.from_numpy(y))
    cap = trials * n
    cands = torch.zeros(cap * dd.CAND_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    thr = 4.0
    torch.cuda.synchronize()
    dd.dd_sps_static(view.data_ptr(), trials, n, stride, 0, d, 17, widths, thr, block,
                     cands.data_ptr(), cap, count.data_ptr())
    torch.cuda.synchronize()
    got = cands.cpu().numpy().view(dd.CAND_DTYPE)[:int(count.item())]
    w = [k for k in widths if k <= n]
    want = oracle.sps(y, np.arange(trials), 0, d, 17, w, block, thr) if w else got[:0]
    order = lambda c: c[np.lexsort((c["width"], c["t_start"], c["trial"]))]
    got, want = order(got), order(want)
    assert got.size == want.size
    for f in ("trial", "t_start", "width", "snr"):
        np.testing.assert_array_equal(got[f], want[f], err_msg=f)


def _coarse(ranges, nchans, nsamp, index, bw=300.0):
    w = configs.mid(nsamp=nsamp, chunk_len=4096, n_streams=2, npulses=3, nchans=4096,
                    ranges=ranges, index=index)
    w.nchans, w.foff = nchans, -bw / nchans
    w.pulses = tuple(configs.PulseSpec(p.dm * 0.05, min(p.t_ref, nsamp // 2), p.width,
                                       p.amp * 8.0) for p in w.pulses)
    return w


@pytest.mark.parametrize("widths,sizes", [
    ((1, 2, 4, 7, 12, 24, 48, 96, 100, 128, 200, 256, 500, 512, 1000, 1024), [4000, 4096, 3000]),
    ((2,), [130, 4096])])
def test_clipped_statistics_edges(widths, sizes):
    """16 widths (three groups a sweep) with a 1024-sample history, and one width; windows that
    end inside a pass."""
    w = _coarse((configs.DMRange(0.0, 1.0, 5, 1), configs.DMRange(5.0, 2.0, 3, 2)), 64, 1 << 14, 71)
    w.widths, w.threshold = widths, 4.0
    x = w.generate(_arrivals(w))
    ranges = w.ranges_array()
    ref = oracle.run(x[:sum(sizes)], w.freqs(), w.tsamp, ranges, widths, w.threshold, 32, sizes)
    plan = dd.Plan(w.freqs(), w.tsamp, ranges, 4096, n_streams=1, max_width=max(widths))
    try:
        xs, T = torch.from_numpy(x).cuda(), 0
        for n, per in zip(sizes, ref["chunks"]):
            seq = plan.run(xs[T:T + n], n)
            T += n
            plan.search(widths, w.threshold, estimator=dd.DD_EST_CLIPPED)
            got, want = plan.candidates(seq), []
            for r in range(len(ranges)):
                y, d = per[r]["series"], int(ranges[r][3])
                wd = [k for k in oracle.widths_for_range(widths, d) if k <= y.shape[1]]
                if y.shape[1] and wd:
                    want.append(oracle.sps_clipped(y, per[r]["trials"], r, d, per[r]["J0"], wd, 32,
                                                   w.threshold))
            want = np.concatenate(want) if want else got[:0]
            compare_candidates(got, want, w.threshold, 32,
                               lambda r, t, per=per: per[r]["series"][t],
                               lambda r, per=per: per[r]["J0"], lambda r: int(ranges[r][3]),
                               trial_snr=clipped_trial_snr(3.0, 3))
    finally:
        plan.close()


@pytest.mark.parametrize("nchans", [17, 63, 80, 129])
@pytest.mark.parametrize("offset", [0, 1, 6])
def test_corner_turn_any_start(nchans, offset):
    """Spectra of any length from a chunk at any byte address (chunks of 4-sample and ragged
    lengths): one trial of DM 0 is the sum over channels."""
    n = 1024
    x = np.random.default_rng(72).integers(0, 256, (n, nchans), dtype=np.uint8)
    f = 1500.0 - np.arange(nchans) * 1.0
    plan = dd.Plan(f, 64e-6, [(0.0, 1.0, 1, 1)], n, n_streams=1, max_width=4)
    try:
        buf = torch.zeros(offset + n * nchans, dtype=torch.uint8, device="cuda")
        buf[offset:] = torch.from_numpy(x.reshape(-1)).cuda()
        at = 0
        for m in (1, 258, 63, 702):
            plan.run(buf[offset + at * nchans:offset + (at + m) * nchans].view(m, nchans), m)
            np.testing.assert_array_equal(plan.series(0)[0].cpu().numpy()[0],
                                          x[at:at + m].sum(1, dtype=np.int64))
            at += m
    finally:
        plan.close()


@pytest.mark.parametrize("nchans,trials,sizes", [
    (200, 70, [4096, 4096]),    # few tiles: the channels split among CTAs
    (200, 70, [4096, 1280, 256]),
    (41, 2500, [2048, 2048]),   # 40 trial tiles: whole channel sums, seven padding channels
])
def test_staged_direct_kernel(nchans, trials, sizes):
    """Coarse channels at x1, x2, x32 (last decimation whose eight-channel sums are packed), x64
    and x256: every series and moment."""
    ranges = (configs.DMRange(0.0, 0.5, trials, 1), configs.DMRange(10.0, 1.0, 65, 2),
              configs.DMRange(20.0, 4.0, 20, 32), configs.DMRange(30.0, 8.0, 9, 64),
              configs.DMRange(40.0, 20.0, 3, 256))
    if trials > 1000:
        ranges = (configs.DMRange(0.0, 0.02, trials, 1), configs.DMRange(10.0, 1.0, 65, 64))
    w = _coarse(ranges, nchans, 1 << 13, 73)
    w.widths = (1, 4, 64, 256)
    x = w.generate(_arrivals(w))
    plan = dd.Plan(w.freqs(), w.tsamp, w.ranges_array(), 4096, n_streams=1, max_width=256)
    try:
        assert plan.kernel(0)[0] == plan.kernel(len(ranges) - 1)[0] == dd.DD_KERNEL_DIRECT
    finally:
        plan.close()
    check(w, x[:sum(sizes)], sizes, 1)


@pytest.mark.parametrize("ranges,sizes", [
    (((0.0, 1.4, 65, 1),), [8448, 8448, 300]),
    (((0.0, 2.4, 65, 2), (0.0, 1.2, 65, 1)), [8448, 8446, 258])])
def test_staged_kernel_widest_rows(ranges, sizes):
    """Trial tiles whose rows fill shared memory, and a last tile of one trial at the largest
    delay: its rows end where the ring ends."""
    w = _coarse(tuple(configs.DMRange(*r) for r in ranges), 64, 1 << 15, 77, bw=400.0)
    w.fch1, w.widths = 1500.0, (2, 4, 64, 256)
    x = w.generate(_arrivals(w))
    assert staged_takes(w, 8448) == [1] * len(ranges)
    plan = dd.Plan(w.freqs(), w.tsamp, w.ranges_array(), 8448, n_streams=1, max_width=256)
    try:
        for r in range(len(ranges)):
            assert plan.kernel(r)[0] == dd.DD_KERNEL_DIRECT
    finally:
        plan.close()
    check(w, x[:sum(sizes)], sizes, 1)


@pytest.mark.parametrize("trials,sizes", [(1024, [10240, 10240]), (1000, [10240, 10238, 9000])])
def test_wide_trial_tile(trials, sizes):
    """Plans that take the 128-trial tile, for uint8 and uint16 data: full and ragged last tiles,
    odd last windows, fifteen groups of channels (the last stage holds one)."""
    ranges = (configs.DMRange(0.0, 0.05, trials, 1), configs.DMRange(50.0, 0.1, trials, 2))
    w = configs.mid(nsamp=1 << 15, chunk_len=4096, n_streams=2, npulses=4, nchans=4096,
                    ranges=ranges, index=74)
    w.nchans, w.foff = 120, -300.0 / 4096
    w.pulses = tuple(configs.PulseSpec(p.dm * 0.05, min(p.t_ref, 25000), p.width, p.amp * 6.0)
                     for p in w.pulses)
    x = w.generate(_arrivals(w))
    plan = dd.Plan(w.freqs(), w.tsamp, w.ranges_array(), 10240, n_streams=1, max_width=256)
    try:
        for r in range(2):
            assert plan.model(r, 512)["tile_trials"] == 128
            assert plan.kernel(r) == (dd.DD_KERNEL_TILED, 256)
    finally:
        plan.close()
    check(w, x[:sum(sizes)], sizes, 2)


@pytest.mark.parametrize("block", [2, 16, 32])
@pytest.mark.parametrize("widths", [(1, 2, 3, 17, 100, 301, 512), (2, 6)])
def test_fused_blocks_equal_plain(block, widths):
    """The fused search's two block loops (16 and 32 samples; smaller) over widths of every
    residue mod 4, segment starts and ragged windows: the plain path's candidates, SNRs included,
    one for every block (threshold far below any SNR)."""
    ranges = (configs.DMRange(0.0, 0.0625, 70, 1), configs.DMRange(4.375, 0.125, 20, 2))
    w = configs.mid(nsamp=1 << 14, chunk_len=4096, n_streams=1, npulses=3, nchans=4096,
                    ranges=ranges, index=76)
    w.nchans, w.foff = 128, -300.0 / 1024
    x = torch.from_numpy(w.generate(_arrivals(w))).cuda()
    got = []
    for fuse in (True, False):
        plan = dd.Plan(w.freqs(), w.tsamp, w.ranges_array(), 6144, n_streams=1,
                       max_width=max(widths), peak_block=block)
        try:
            if fuse:
                assert plan.fuse_search(widths) == 2
            out, T = [], 0
            for n in (6144, 5000, 1030, 4210 - 1):
                n -= n % 2
                seq = plan.run(x[T:T + n], n)
                T += n
                plan.search(widths, -1e30)
                out.append(plan.candidates(seq))
        finally:
            plan.close()
        got.append(np.concatenate(out))
    assert got[0].size == got[1].size > 1000
    for f in ("range", "trial", "t_start", "width", "snr"):
        np.testing.assert_array_equal(got[0][f], got[1][f], err_msg=f)


def _both(*calls):
    """Run the calls on host threads at once; the first exception of any is raised here."""
    errors = []

    def guarded(f):
        try:
            f()
        except Exception as e:  # noqa: BLE001 - handed to the test's thread
            errors.append(e)

    threads = [threading.Thread(target=guarded, args=(f,)) for f in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        raise errors[0]


def test_clipped_searches_on_two_threads():
    """Two plans on two host threads, whose clipped statistics need 147 KB and 67 KB of shared
    memory: neither thread's launches fail for the other's, and every pass gives the same
    candidates."""
    x = torch.randint(96, 160, (256, 8), dtype=torch.uint8, device="cuda",
                      generator=torch.Generator("cuda").manual_seed(78))
    x[100:104] = 255
    torch.cuda.synchronize()
    f = 1500.0 - np.arange(8.0)

    def loop(widths):
        plan = dd.Plan(f, 64e-6, [(0.0, 1.0, 1, 1)] * 8, 256, n_streams=1, max_width=1024)
        try:  # eight launches a pass
            first = None
            for _ in range(800):
                seq = plan.run(x, 256)
                plan.search(widths, 4.0, estimator=dd.DD_EST_CLIPPED)
                got = plan.candidates(seq)
                got["t_start"] -= 256 * seq
                first = got if first is None else first
                np.testing.assert_array_equal(got, first)
            assert first.size > 0
        finally:
            plan.close()

    _both(lambda: loop((1, 2, 4, 7, 12, 24, 48, 96, 100, 128, 200, 256, 500, 512, 1000, 1024)),
          lambda: loop((1, 2, 4, 8, 16, 32, 64)))


def test_persistent_batches_on_two_threads():
    """Two persistent batches on two host threads whose tiles need different amounts of shared
    memory: neither thread's launches fail for the other's."""
    f = 1550.0 - np.arange(256) * 300.0 / 4096
    x = torch.randint(96, 160, (1 << 15, 256), dtype=torch.uint8, device="cuda",
                      generator=torch.Generator("cuda").manual_seed(79))
    torch.cuda.synchronize()

    def loop(step):
        b = dd.Batch([(f, 64e-6, x)], [(0.0, step, 64, 1)], 2048, (1, 2, 4), 9.0, persistent=True)
        try:
            assert b.info(0)[2] == 512  # the tiled kernel, one instance for both
            for _ in range(2000):  # sixteen rounds, a launch each
                b.run()
                b.wait()
        finally:
            b.close()

    _both(lambda: loop(0.02), lambda: loop(0.6))
