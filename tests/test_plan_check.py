"""Host logic of the tiled kernel's plan (no GPU): the plan-time delay-class tables, staging
windows and build work lists, checked against the delay tables they come from.

The delay tables are the oracle's (the GPU builds the same table bit for bit; see the parity
tests), padded to a multiple of 8 channels by repeating the last channel as the library does.
"""
import numpy as np
import pytest

import oracle
from synth import configs
import paper_2101_00941_gb300 as dd


@pytest.fixture(scope="module", autouse=True)
def _built():
    dd.build()
    dd.lib()


def _tables(w):
    tabs = oracle.shift_tables(w.freqs(), w.tsamp, w.ranges_array())
    out = []
    for t in tabs:
        cp = -(-t.shape[1] // 8) * 8
        out.append(np.pad(t, ((0, 0), (0, cp - t.shape[1])), mode="edge").astype(np.int32))
    return out


SHAPES = [(512, 64), (256, 64), (256, 32)]


@pytest.mark.parametrize("tt,trials", SHAPES)
def test_4096_channel_plan(tt, trials):
    w = configs.mid(nsamp=1 << 17)
    for tab, r in zip(_tables(w), w.ranges):
        ok, bad = dd.dd_tiled_plan_check(tab, r.decimation, tt, trials)
        assert (ok, bad) == (1, 0), r


@pytest.mark.parametrize("tt,trials", SHAPES)
def test_8192_channel_plan_edges(tt, trials):
    w = configs.out_of_core(nsamp=1 << 20)
    tabs = _tables(w)
    for k in (0, len(w.ranges) - 1):  # x1 and the widest, x16
        ok, bad = dd.dd_tiled_plan_check(tabs[k], w.ranges[k].decimation, tt, trials)
        assert bad == 0, w.ranges[k]
        # a two-CTA shape must fit half an SM's shared memory: the 64 x 256 tile of this plan's
        # x1 range does not (117 KB), the 32 x 256 tile does
        if k == 0:
            assert ok == (0 if (tt, trials) == (256, 64) else 1)


def test_ragged_channels_and_trial_tiles():
    """1001 channels (padded to 1008) and ranges of 150, 75, 130, 70, 40, 30, 20, 10 trials;
    above x16 the sum of two groups' eight channels does not fit a pair word's 16-bit lanes."""
    ranges = (configs.DMRange(0.0, 0.0625, 150, 1), configs.DMRange(9.375, 0.125, 75, 2),
              configs.DMRange(18.75, 0.15625, 130, 4), configs.DMRange(39.0625, 0.3125, 70, 8),
              configs.DMRange(60.9375, 0.625, 40, 16), configs.DMRange(85.9375, 1.25, 30, 32),
              configs.DMRange(123.4375, 2.5, 20, 64), configs.DMRange(173.4375, 5.0, 10, 128))
    w = configs.mid(nsamp=1 << 15, nchans=4096, ranges=ranges)
    w.nchans, w.foff = 1001, -300.0 / 1024
    for tab, r in zip(_tables(w), w.ranges):
        for tt, trials in SHAPES:
            ok, bad = dd.dd_tiled_plan_check(tab, r.decimation, tt, trials)
            assert bad == 0
            assert ok == (1 if r.decimation <= 16 else 0), (r, tt, trials)


def test_odd_group_count():
    """993 channels: padded to 1000, 125 eight-channel groups, so the last stage holds one."""
    ranges = (configs.DMRange(0.0, 0.0625, 100, 1), configs.DMRange(6.25, 0.125, 50, 2))
    w = configs.mid(nsamp=1 << 15, nchans=4096, ranges=ranges)
    w.nchans, w.foff = 993, -300.0 / 1024
    for tab, r in zip(_tables(w), w.ranges):
        assert tab.shape[1] == 1000
        assert dd.dd_tiled_plan_check(tab, r.decimation, 512) == (1, 0), r


def test_coarse_channels_and_bad_tables_are_refused():
    w = configs.tiny()  # 64 coarse channels: up to 63 delay classes per group
    (tab,) = _tables(w)
    assert dd.dd_tiled_plan_check(tab, 1, 512) == (0, 0)
    mid = _tables(configs.mid(nsamp=1 << 17))[0].copy()
    mid[10, 5] = mid[11, 5] + 1  # a delay that decreases with DM
    assert dd.dd_tiled_plan_check(mid, 1, 512) == (0, 0)
    with pytest.raises(dd.DDError):
        dd.dd_tiled_plan_check(np.zeros((4, 12), np.int32), 1, 512)  # 12 channels: not padded


@pytest.mark.parametrize("tt,trials", SHAPES + [(256, 128)])
@pytest.mark.parametrize("decimation", [1, 2, 16])
def test_chains_on_jittered_tables(tt, trials, decimation):
    """Delay tables whose groups' classes lie zero to many channel steps apart (chains with
    in-between links, broken chains, one class): the plan is either refused or free of
    violations, and smooth tables are accepted up to the tile's class limit (16 per group, 24 with
    128 trials)."""
    rng = np.random.default_rng(75)
    accepted = 0
    for jitter in (0.0, 0.3, 1.0, 2.0):
        for ntr, cpad in ((130, 40), (64, 8), (1, 24)):
            slope = np.linspace(0.9, 0.93, cpad)
            t = np.arange(ntr)[:, None] * slope + rng.random(cpad) * 3
            t = np.floor(t + jitter * rng.random((ntr, cpad)))
            tab = np.maximum.accumulate(t, axis=0).astype(np.int32)
            ok, bad = dd.dd_tiled_plan_check(tab, decimation, tt, trials)
            assert bad == 0, (jitter, ntr, cpad)
            accepted += ok
            most = max(len(np.unique(g - g.min(1, keepdims=True), axis=0))
                       for t0 in range(0, ntr, trials)
                       for c in range(0, cpad, 8) for g in [tab[t0:t0 + trials, c:c + 8]])
            assert ok or jitter > 0 or most > (24 if trials == 128 else 16)
    assert accepted > 3


def test_128_trial_tile_on_the_workloads():
    for w in (configs.mid(nsamp=1 << 17), configs.out_of_core(nsamp=1 << 20)):
        for tab, r in list(zip(_tables(w), w.ranges))[::3]:
            assert dd.dd_tiled_plan_check(tab, r.decimation, 256, 128) == (1, 0), r


def _staged(nchans, bw, ranges, chunk, sizes):
    """Violations of the staged direct kernel's launches over the chunks of a 1500 MHz, 64 us plan,
    and which ranges it takes."""
    w = configs.mid(nsamp=1 << 15, ranges=tuple(configs.DMRange(*r) for r in ranges))
    w.nchans, w.fch1, w.foff = nchans, 1500.0, -bw / nchans
    tabs = _tables(w)
    O = oracle.overlap(tabs, w.ranges_array())
    bad, oks, T = 0, [], 0
    for n in sizes:
        for t, r in zip(tabs, w.ranges):
            ok, b = dd.dd_staged_plan_check(t, r.decimation, O, chunk, T, n)
            oks.append(ok)
            bad += b
        T += n
    return bad, oks


# coarse channels with wide DM steps: a trial tile's delays spread over up to the widest frame of
# the kernel's shared memory, and the last trial tile, of few trials, starts at the largest delay
@pytest.mark.parametrize("nchans,bw,ranges,chunk,sizes", [
    (256, 400.0, [(0.0, 1.4, 193, 1)], 8192, [8192, 8192]),
    (256, 400.0, [(0.0, 1.3, 193, 1)], 8192, [8192, 8192]),
    (64, 400.0, [(0.0, 1.4, 65, 1)], 65792, [65792, 65792, 300]),
    (64, 400.0, [(0.0, 1.2, 65, 1)], 8448, [8448, 8448, 1]),
    (64, 400.0, [(0.0, 2.4, 65, 2)], 8448, [8448, 8448, 2]),
    (64, 400.0, [(0.0, 9.0, 129, 8), (0.0, 1.25, 449, 1)], 8448, [8448, 8192, 4104, 8448]),
    (41, 400.0, [(30.0, 60.0, 66, 64)], 16384, [16384, 16384]),
    (256, 400.0, [(0.0, 0.5, 800, 1), (400.0, 1.0, 400, 2)], 16384, [16384, 16000]),
    (64, 100.0, [(0.0, 1.0, 401, 1)], 65536, [65536])])
def test_staged_copies_stay_inside_the_ring(nchans, bw, ranges, chunk, sizes):
    bad, oks = _staged(nchans, bw, ranges, chunk, sizes)
    assert all(oks)
    assert bad == 0


def test_staged_plan_refusals():
    assert _staged(64, 400.0, [(0.0, 1.8, 65, 1)], 8192, [8192]) == (0, [0])  # spread too wide
    (tab,) = _tables(configs.tiny())
    tab = tab.copy()
    tab[10, 5] = tab[0, 5] - 1  # a delay below the tile's first
    assert dd.dd_staged_plan_check(tab, 1, 2048, 8192, 0, 8192) == (0, 0)
    for args in ((3, 0, 8192, 0, 8192), (1, -1, 8192, 0, 8192), (1, 0, 8192, 0, 8193)):
        with pytest.raises(dd.DDError):
            dd.dd_staged_plan_check(tab, *args)
